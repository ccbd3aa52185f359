"""Register-resident panel QR of full -> band, through the solvers: panel
heights at the edges of its forms (one block, clusters of 2 to 16, the
cooperative grid), panels shorter than the band at the end, band widths that
leave threads idle.  The eigenvalues come out right, with residual and
orthogonality at rounding level, only if every panel's reflectors and T do.
Bounds: max |dlambda| / ||A|| <= 1e-11, residual and orthogonality 50 n u.
"""
import ctypes

import numpy as np
import pytest

from test_chase_clusters_gpu import SIZES, tiny_column

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


# n - nbw rows in the first panel
SHAPES = [(5, 4), (66, 64), (96, 32), (97, 32), (160, 64), (193, 64), (512 + 32, 32), (513 + 32, 32), (513 + 48, 48),
          (1024 + 64, 64), (1025 + 64, 64), (1025 + 32, 32), (2049 + 20, 20), (2048 + 64, 64), (2049 + 64, 64)]


@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
@pytest.mark.parametrize("n,nbw", SHAPES)
def test_solve_through_panel_forms(gb, n, nbw, cplx):
    g = torch.Generator(device="cuda").manual_seed(7 * n + nbw)
    dt = torch.complex128 if cplx else torch.float64
    R = torch.randn(n, n, generator=g, device="cuda", dtype=dt)
    A = (0.5 * (R + R.mH)).contiguous()
    nev = min(n, 40)
    bytes_, solve = (gb.gb_solve_workspace_bytes_z, gb.gb_solve_z) if cplx else (gb.gb_solve_workspace_bytes, gb.gb_solve_d)
    wsb = bytes_(n, nev, nbw)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    ev = torch.zeros(nev, dtype=torch.float64, device="cuda")
    Z = torch.zeros(nev, n, dtype=dt, device="cuda")
    solve(n, nev, nbw, A.mT.contiguous(), n, ev, Z, n, ws, wsb, torch.cuda.current_stream())
    torch.cuda.synchronize()
    lam = torch.linalg.eigvalsh(A)
    nrm = lam.abs().max()
    assert (ev - lam[:nev]).abs().max() / nrm <= 1e-11
    V = Z.mT
    assert torch.linalg.norm(A @ V - V * ev) / torch.linalg.norm(A) <= 50 * n * U
    assert (V.mH @ V - torch.eye(nev, dtype=dt, device="cuda")).abs().max() <= 50 * n * U


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("m", [40, 600])
@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
def test_reflector_of_a_tiny_column(gb, cplx, m, size):
    """A panel's first column with a norm around the square root of the smallest
    numbers (the panel alone: one block, and a cluster)."""
    x, tau, v, bound = tiny_column(m, size, cplx)
    nb = 32
    g = np.random.default_rng(m)
    P = g.standard_normal((nb, m)) + (1j * g.standard_normal((nb, m)) if cplx else 0.0)
    P[0] = x
    Pd = torch.from_numpy(P).cuda()
    Y, t = torch.zeros_like(Pd), torch.zeros(nb, dtype=Pd.dtype, device="cuda")
    part = torch.empty(1 << 16, dtype=torch.uint8, device="cuda")
    ptr = [ctypes.c_void_p(a.data_ptr()) for a in (Pd, t, Y, part)]
    rc = gb.load().gb_test_panel_hold(ctypes.c_int(cplx), ctypes.c_int(m), ctypes.c_int(nb), *ptr,
                                      ctypes.c_longlong(10 ** 9), ctypes.c_int(-1), None,
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    assert abs(t[0].item() - tau) <= bound
    assert np.abs(Y[0, 1:].cpu().numpy() - v).max() <= bound
