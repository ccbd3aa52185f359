"""Bulge chase on clusters: the edges of its blocks and cluster shapes, real
and complex.  Band widths at and around the padded widths (32, 64) and the
16-row groups; orders from one reflector a sweep to several, with short last
blocks.  Checked: Q2^H B Q2 = T and T's eigenvalues (LAPACK), both to the
backward error 50 n u ||B||, which needs no agreement of roundings.
"""
import numpy as np
import pytest
import scipy.linalg

import oracle
from paper_1811_01277_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def gb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1811_01277_gb300 as m
    from paper_1811_01277_gb300 import build
    build.build()
    m.load()
    return m


SHAPES = [(b + d, b) for b in (1, 2, 15, 16, 17, 31, 32, 33, 48, 63, 64) for d in (1, b, b + 1, 3 * b + 2)]


@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
@pytest.mark.parametrize("n,b", SHAPES)
def test_chase_edges(gb, n, b, cplx):
    B = inputs.band_symmetric(n, b, seed=31 * n + b, cplx=cplx)
    dt = torch.complex128 if cplx else torch.float64
    dev = torch.device("cuda")
    AB = np.zeros((n, b + 1), dtype=B.dtype)
    for k in range(b + 1):
        AB[:n - k, k] = np.diag(B, -k)
    cnt = gb.gb_hh_count(n, b)
    d = torch.zeros(n, dtype=torch.float64, device=dev)
    e = torch.zeros(max(n - 1, 1), dtype=torch.float64, device=dev)
    hv = torch.full((max(cnt * b, 1),), np.nan, dtype=dt, device=dev)
    ht = torch.full((max(cnt, 1),), np.nan, dtype=dt, device=dev)
    wsb = (gb.gb_band_to_tridi_workspace_bytes_z if cplx else gb.gb_band_to_tridi_workspace_bytes)(n, b)
    ws = torch.empty(wsb, dtype=torch.uint8, device=dev)
    st = torch.cuda.current_stream()
    run = gb.gb_band_to_tridi_z if cplx else gb.gb_band_to_tridi_d
    run(n, b, torch.from_numpy(AB).to(dev), b + 1, d, e, hv, ht, ws, wsb, st)
    assert gb.gb_trans_ev_query(ws, wsb, st) == 0
    d, e = d.cpu().numpy(), e.cpu().numpy()[:n - 1]
    hv, ht = hv.cpu().numpy()[:cnt * b], ht.cpu().numpy()[:cnt]
    tol = 50 * n * U * max(np.linalg.norm(B, 2), 1e-300)
    lam = scipy.linalg.eigvalsh_tridiagonal(d, e) if n > 1 else d
    assert np.abs(np.sort(lam) - np.linalg.eigvalsh(B)).max() <= tol
    Q = oracle.trans_ev(n, b, hv, ht, np.eye(n, dtype=B.dtype))
    T = np.diag(d) + np.diag(e, -1) + np.diag(e, 1)
    assert np.abs(Q.conj().T @ B @ Q - T).max() <= tol


@pytest.mark.parametrize("cplx,n,b", [(False, 700, 64), (False, 500, 32), (True, 300, 64)])
def test_chase_concurrent(gb, cplx, n, b):
    """Many chases at once, so that a sweep's blocks get out of step with each
    other: every one gives the bits of a chase that runs alone."""
    dev = torch.device("cuda")
    B = inputs.band_symmetric(n, b, seed=n + b, cplx=cplx)
    AB = np.zeros((n, b + 1), dtype=B.dtype)
    for k in range(b + 1):
        AB[:n - k, k] = np.diag(B, -k)
    AB = torch.from_numpy(AB).to(dev)
    cnt = gb.gb_hh_count(n, b)
    wsb = (gb.gb_band_to_tridi_workspace_bytes_z if cplx else gb.gb_band_to_tridi_workspace_bytes)(n, b)
    run = gb.gb_band_to_tridi_z if cplx else gb.gb_band_to_tridi_d

    def buffers():
        return (torch.zeros(n, dtype=torch.float64, device=dev), torch.zeros(n - 1, dtype=torch.float64, device=dev),
                torch.zeros(cnt * b, dtype=AB.dtype, device=dev), torch.zeros(cnt, dtype=AB.dtype, device=dev),
                torch.empty(wsb, dtype=torch.uint8, device=dev))

    alone = buffers()
    run(n, b, AB, b + 1, *alone[:4], alone[4], wsb, torch.cuda.current_stream())
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(24)]
    for _ in range(6):
        many = [buffers() for _ in streams]
        torch.cuda.synchronize()
        for st, w in zip(streams, many):
            run(n, b, AB, b + 1, *w[:4], w[4], wsb, st)
        torch.cuda.synchronize()
        for st, w in zip(streams, many):
            assert gb.gb_trans_ev_query(w[4], wsb, st) == 0
            for x, y in zip(w[:4], alone[:4]):
                assert torch.equal(x, y)
