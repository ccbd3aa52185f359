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


def tiny_column(m, size, cplx):
    """A column of m entries of about `size`, its reflector (tau, v) computed on
    the column times 2^500, and the bound on either's error: the sum of squares
    s is taken unscaled, each of its 2 m roundings up to 2^-1075, so tau and v
    are off by up to 4 (2 m 2^-1075 / s) and a few units of 2^-53."""
    g = np.random.default_rng(m)
    x = g.uniform(0.5, 1.0, m) * (np.exp(2j * np.pi * g.random(m)) if cplx else 1.0) * size
    y = x * 2.0 ** 500
    nrm = np.linalg.norm(y)
    beta = -nrm if y[0].real >= 0 else nrm
    s = (nrm * 2.0 ** -500) ** 2
    bound = 8 * m * 2.0 ** -1074 / s + 16 * U
    return x, (beta - y[0]) / beta, y[1:] / (y[0] - beta), bound


SIZES = [1e-140, 1e-150, 1e-154, 1e-155, 2e-156]


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
def test_reflector_of_a_tiny_column(gb, cplx, size):
    """H(1,0) of a band matrix whose first column below the diagonal has a
    norm around the square root of the smallest numbers."""
    n, b = 40, 16
    x, tau, v, bound = tiny_column(b, size, cplx)
    B = inputs.band_symmetric(n, b, seed=3, cplx=cplx)
    AB = np.zeros((n, b + 1), dtype=B.dtype)
    for k in range(b + 1):
        AB[:n - k, k] = np.diag(B, -k)
    AB[0, 1:] = x
    dev, st = torch.device("cuda"), torch.cuda.current_stream()
    dt = torch.complex128 if cplx else torch.float64
    cnt = gb.gb_hh_count(n, b)
    d, e = torch.zeros(n, dtype=torch.float64, device=dev), torch.zeros(n, dtype=torch.float64, device=dev)
    hv, ht = torch.zeros(cnt * b, dtype=dt, device=dev), torch.zeros(cnt, dtype=dt, device=dev)
    wsb = (gb.gb_band_to_tridi_workspace_bytes_z if cplx else gb.gb_band_to_tridi_workspace_bytes)(n, b)
    ws = torch.empty(wsb, dtype=torch.uint8, device=dev)
    run = gb.gb_band_to_tridi_z if cplx else gb.gb_band_to_tridi_d
    run(n, b, torch.from_numpy(AB).to(dev), b + 1, d, e, hv, ht, ws, wsb, st)
    assert gb.gb_trans_ev_query(ws, wsb, st) == 0
    assert abs(ht[0].item() - tau) <= bound
    assert np.abs(hv[1:b].cpu().numpy() - v).max() <= bound
