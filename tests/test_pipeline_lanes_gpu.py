"""DFMA pipeline with four lanes per column (few columns, default blocking):
against the oracle at the edges of its window slots, blocks and groups, and
with NaN and Inf entries, which must reach the rows they reach with one
thread per column and no others.  Bar 1e-12 per column, as for every kernel
of the back-transformation.
"""
import numpy as np
import pytest

import oracle
from paper_1811_01277_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1811_01277_gb300 as m
    from paper_1811_01277_gb300 import build
    build.build()
    m.load()
    return m


def run(gb, n, b, hv, ht, Z, opts=None, ldz=None):
    ldz = ldz or n
    nev = Z.shape[1]
    buf = np.full((nev, ldz), 7.0)
    buf[:, :n] = Z.T
    Zt = torch.from_numpy(buf).cuda()
    wsb = gb.gb_trans_ev_workspace_bytes(n, b, nev, 0, opts)
    ws = torch.full((max(wsb, 256),), 255, dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream()
    gb.gb_trans_ev_tridi_to_band_d(n, b, nev, torch.from_numpy(hv).cuda(), torch.from_numpy(ht).cuda(), Zt, ldz, ws, wsb,
                                   st, opts)
    assert gb.gb_trans_ev_query(ws, wsb, st) == 0
    out = Zt.cpu().numpy()
    assert np.all(out[:, n:] == 7.0)
    return out[:, :n].T


@pytest.mark.parametrize("n,b,nev", [(2, 8, 1), (17, 8, 5), (18, 16, 33), (33, 32, 32), (65, 64, 31), (130, 64, 65),
                                     (257, 8, 40), (333, 32, 301), (400, 16, 100), (511, 64, 64)])
def test_parity(gb, n, b, nev):
    hv, ht = inputs.synthetic_reflectors(n, b, seed=n + b)
    Z = inputs.z_gaussian(n, nev, seed=nev)
    want = oracle.trans_ev(n, b, hv, ht, Z)
    got = run(gb, n, b, hv, ht, Z, ldz=n + 3)
    assert np.max(np.linalg.norm(got - want, axis=0) / np.linalg.norm(Z, axis=0)) <= 1e-12


def test_nonfinite_entries_reach_the_same_rows(gb):
    n, b, nev = 150, 16, 12
    hv, ht = inputs.synthetic_reflectors(n, b, seed=5)
    Z = inputs.z_gaussian(n, nev, seed=6)
    for j in range(nev):
        Z[(j * 13) % n, j] = [np.nan, np.inf, -np.inf][j % 3]
    one = {"variant": 2, "sweeps_per_tile": 16, "cols_per_block": 64}
    a, c = run(gb, n, b, hv, ht, Z), run(gb, n, b, hv, ht, Z, one)
    assert np.array_equal(np.isfinite(a), np.isfinite(c))


def test_workspace_of_more_columns_serves_fewer(gb):
    """Columns taken in chunks of 256 with a last one of 224, the workspace sized
    once for 256: n = 1000, nbw = 8, where 224 columns take 32-column blocks."""
    n, b = 1000, 8
    hv, ht = inputs.synthetic_reflectors(n, b, seed=2)
    Z = inputs.z_gaussian(n, 480, seed=4)
    want = oracle.trans_ev(n, b, hv, ht, Z)
    Zt = torch.from_numpy(np.ascontiguousarray(Z.T)).cuda()
    hvd, htd = torch.from_numpy(hv).cuda(), torch.from_numpy(ht).cuda()
    wsb = gb.gb_trans_ev_workspace_bytes(n, b, 256, 0)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream()
    for c in (0, 256):
        k = min(256, 480 - c)
        gb.gb_trans_ev_tridi_to_band_d(n, b, k, hvd, htd, Zt[c:c + k], n, ws, wsb, st)
        assert gb.gb_trans_ev_query(ws, wsb, st) == 0
    got = Zt.cpu().numpy().T
    assert np.max(np.linalg.norm(got - want, axis=0) / np.linalg.norm(Z, axis=0)) <= 1e-12
