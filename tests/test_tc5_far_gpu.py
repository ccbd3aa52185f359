"""Back-transformation on tcgen05 with one reflector of a huge tau (2^15, far from
orthogonal), whose U exceeds the exponents that the folds take in one shift each
way.  The columns are all but orthogonal to it (v^H z = 2^-20), so the result
stays in range.  Bound: the oracle's own rounding of v^H z, len u ||v|| ||z||,
comes back times tau ||v||: 16 2^-53 4 2^15 = 2^-32 for ||v|| = 2, ||z|| = 1; twice
that; a wrong shift is wrong by 2^-5."""
import numpy as np
import pytest

import oracle

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


@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
@pytest.mark.parametrize("b", [16, 32, 64])
def test_far_exponents(gb, b, cplx):
    n, nev = 3 * b + 5, 130
    dt = np.complex128 if cplx else np.float64
    rng = np.random.default_rng(b)
    cnt = gb.gb_hh_count(n, b)
    hv, ht = np.zeros(cnt * b, dt), np.zeros(cnt, dt)
    v = rng.standard_normal(16) + (1j * rng.standard_normal(16) if cplx else 0)
    v[0] = 0
    v *= np.sqrt(3.0) / np.linalg.norm(v)
    v[0] = 1
    hv[:16] = v                        # the first sweep's first reflector: rows 1 .. 16
    ht[0] = 2.0 ** 15
    Z = rng.standard_normal((n, nev)) + (1j * rng.standard_normal((n, nev)) if cplx else 0)
    Z /= np.linalg.norm(Z, axis=0)
    Z[1:17] += np.outer(v, (2.0 ** -20 - v.conj() @ Z[1:17]) / 4)
    Z = np.asfortranarray(Z)
    dev, opts = torch.device("cuda"), {"variant": 4}
    Zt = torch.from_numpy(np.ascontiguousarray(Z.T)).to(dev)
    wsb = gb.gb_trans_ev_workspace_bytes(n, b, nev, cplx, opts)
    ws = torch.zeros(max(wsb, 256), dtype=torch.uint8, device=dev)
    st = torch.cuda.current_stream()
    f = gb.gb_trans_ev_tridi_to_band_z if cplx else gb.gb_trans_ev_tridi_to_band_d
    f(n, b, nev, torch.from_numpy(hv).to(dev), torch.from_numpy(ht).to(dev), Zt, n, ws, wsb, st, opts)
    assert gb.gb_trans_ev_query(ws, wsb, st) == 0
    ref = oracle.trans_ev(n, b, hv, ht, Z)
    assert np.linalg.norm(ref - Z, axis=0).max() > 0.05     # (tau v^H z ||v|| = 2^-4)
    assert np.linalg.norm(Zt.cpu().numpy().T - ref, axis=0).max() <= 2.0 ** -31
