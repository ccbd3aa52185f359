"""Multisection with 32, 16, 8 and 4 lanes per eigenvalue (the count of wanted
eigenvalues decides) and its FP32 first phase, through the solver: spectra
with clusters far below FP32 resolution, exact multiples, a zero matrix and
extreme scales.  Eigenvalues ascending and within 1e-11 ||A|| of LAPACK's.
"""
import pytest

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


def solve(gb, A, nev, nbw=32):
    n = A.shape[0]
    wsb = gb.gb_solve_workspace_bytes(n, nev, nbw)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    ev = torch.zeros(nev, dtype=torch.float64, device="cuda")
    Z = torch.zeros(nev, n, dtype=torch.float64, device="cuda")
    gb.gb_solve_d(n, nev, nbw, A, n, ev, Z, n, ws, wsb, torch.cuda.current_stream(), gb.GB_SOLVE_TRIDIAG_BISECT)
    torch.cuda.synchronize()
    return ev


@pytest.mark.parametrize("n,nev", [(40, 1), (300, 300), (1300, 608), (1300, 609), (1300, 1217), (2500, 2433)])
def test_lanes(gb, n, nev):
    g = torch.Generator(device="cuda").manual_seed(n + nev)
    R = torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64)
    A = 0.5 * (R + R.T)
    lam = torch.linalg.eigvalsh(A)
    ev = solve(gb, A, nev)
    assert (ev.diff() >= 0).all()
    assert (ev - lam[:nev]).abs().max() <= 1e-11 * lam.abs().max()


@pytest.mark.parametrize("kind", ["zero", "identity", "tight", "split", "huge", "tiny", "graded"])
def test_spectra(gb, kind):
    n, nev = 200, 150
    g = torch.Generator(device="cuda").manual_seed(3)
    lam = torch.linspace(-1.0, 1.0, n, dtype=torch.float64, device="cuda")
    if kind == "zero":
        lam = lam * 0.0
    elif kind == "identity":
        lam = torch.ones_like(lam)
    elif kind == "tight":      # 1e-10 apart: one FP32 value
        lam = 0.3 + 1e-10 * torch.arange(n, dtype=torch.float64, device="cuda")
    elif kind == "split":      # two clusters and one far eigenvalue
        lam = torch.cat([torch.full((100,), -1e-9, dtype=torch.float64, device="cuda"),
                         torch.full((99,), 1e-9, dtype=torch.float64, device="cuda"),
                         torch.ones(1, dtype=torch.float64, device="cuda")])
    elif kind == "huge":
        lam = lam * 1e120
    elif kind == "tiny":
        lam = lam * 1e-120
    elif kind == "graded":
        lam = torch.logspace(-14, 0, n, dtype=torch.float64, device="cuda")
    Q = torch.linalg.qr(torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64)).Q
    A = (Q * lam) @ Q.T
    A = 0.5 * (A + A.T)
    want = torch.sort(lam).values
    ev = solve(gb, A, nev)
    assert (ev.diff() >= 0).all()
    assert (ev - want[:nev]).abs().max() <= 1e-11 * max(float(want.abs().max()), 1e-300)


@pytest.mark.parametrize("n,nev", [(40, 40), (300, 1), (600, 250)])
@pytest.mark.parametrize("x", [float("nan"), float("inf"), float("-inf")])
def test_nonfinite_matrix_gives_nan(gb, n, nev, x):
    """No finite number may stand for an eigenvalue of a matrix that has none."""
    g = torch.Generator(device="cuda").manual_seed(n)
    R = torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64)
    A = 0.5 * (R + R.T)
    A[n // 2, n // 2] = x
    assert torch.isnan(solve(gb, A, nev)).all()
