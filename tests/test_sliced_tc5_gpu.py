"""Edges of the tcgen05 digit products: tiles of 128 x 64, stages of 32 and
exact sums of 128 values of k, splits, the swapped orientation of short wide
results, lower triangles and both halves of alpha / beta.

Operands are integers in [-9, 9], so every result is an integer below 2^53 and
a correct product equals the FP64 one exactly: no tolerance.
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


def ints(g, *shape):
    return torch.randint(-9, 10, shape, generator=g, device="cuda").to(torch.float64)


SHAPES = [(1, 1, 1), (128, 64, 32), (129, 65, 33), (127, 63, 31), (64, 64, 128), (65, 129, 129), (128, 128, 160),
          (64, 700, 161), (40, 300, 4100), (700, 40, 2049), (300, 1000, 64), (1000, 300, 513), (2500, 2500, 96)]


@pytest.mark.parametrize("m,n,k", SHAPES)
@pytest.mark.parametrize("ta,tb,alpha,beta", [("N", "N", 1.0, 0.0), ("T", "N", -1.0, 1.0), ("N", "T", 2.0, -3.0)])
def test_gemm_exact(gb, m, n, k, ta, tb, alpha, beta):
    g = torch.Generator(device="cuda").manual_seed(m + 10 * n + 100 * k)
    A = ints(g, *((k, m + 3) if ta == "N" else (m, k + 1)))       # column-major: (columns, leading dimension)
    B = ints(g, *((n, k + 2) if tb == "N" else (k, n + 5)))
    C = ints(g, n, m + 1)
    left = A[:, :m].T if ta == "N" else A[:, :k]
    right = B[:, :k].T if tb == "N" else B[:, :n]
    want = alpha * (left @ right) + (beta * C[:, :m].T if beta else 0.0)
    if beta == 0.0:
        C[:, :m] = float("nan")                                   # must not be read
    pad = C[:, m:].clone()
    wsb = gb.gb_dgemm_sliced_workspace_bytes(m, n, k)
    ws = torch.full((wsb,), 255, dtype=torch.uint8, device="cuda")
    gb.gb_dgemm_sliced(ta, tb, m, n, k, alpha, A, A.shape[1], B, B.shape[1], beta, C, m + 1, ws, wsb,
                       torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert torch.equal(C[:, :m].T, want)
    assert torch.equal(C[:, m:], pad)


@pytest.mark.parametrize("n", [1, 31, 64, 65, 128, 129, 200, 513])
@pytest.mark.parametrize("k", [1, 64, 130])
def test_triangles_and_symmetric_exact(gb, n, k):
    g = torch.Generator(device="cuda").manual_seed(7 * n + k)
    X, Y, C = ints(g, k, n), ints(g, k, n), ints(g, n, n)
    st = torch.cuda.current_stream()
    low = torch.ones(n, n, dtype=torch.bool, device="cuda").tril()
    # rank-2k update of the lower triangle (column-major: the transposed tensor)
    want = torch.where(low, C.T - (X.T @ Y + Y.T @ X), C.T)
    wsb = gb.gb_dsyr2k_sliced_workspace_bytes(n, k)
    ws = torch.full((wsb,), 255, dtype=torch.uint8, device="cuda")
    got = C.clone()
    gb.gb_dsyr2k_sliced(n, k, -1.0, X, n, Y, n, 1.0, got, n, ws, wsb, st)
    assert torch.equal(got.T, want)
    # symmetric times tall: only the lower triangle is read
    S = ints(g, n, n)
    S = S.tril() + S.tril(-1).T
    stored = torch.where(low, S, torch.full_like(S, float("nan"))).T.contiguous()
    wsb = gb.gb_dsymm_sliced_workspace_bytes("L", n, k)
    ws = torch.full((wsb,), 255, dtype=torch.uint8, device="cuda")
    out = torch.zeros(k, n, dtype=torch.float64, device="cuda")
    gb.gb_dsymm_sliced("L", n, k, 1.0, stored, n, X, n, 0.0, out, n, ws, wsb, st)
    assert torch.equal(out.T, S @ X.T)


@pytest.mark.parametrize("e", [-1040, -1000, 0, 970])
def test_scales_at_the_ends_of_the_range(gb, e):
    """One row of A times 2^e: normal, subnormal and large results, each the
    nearest FP64 number (scaling by a power of two commutes with rounding while
    the result is normal)."""
    m, n, k = 130, 70, 50
    g = torch.Generator(device="cuda").manual_seed(5)
    A, B = ints(g, k, m), ints(g, n, k)
    C = torch.zeros(n, m, dtype=torch.float64, device="cuda")
    As = A.clone()
    As[:, 7] = torch.ldexp(torch.ldexp(A[:, 7], torch.tensor(e // 2, device="cuda")), torch.tensor(e - e // 2, device="cuda"))
    want = (A.T @ B.T)
    want[7] = torch.ldexp(torch.ldexp(want[7], torch.tensor(e // 2, device="cuda")), torch.tensor(e - e // 2, device="cuda"))
    if e == -1040:   # subnormal operands read as zero
        want[7] = 0.0
    wsb = gb.gb_dgemm_sliced_workspace_bytes(m, n, k)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    gb.gb_dgemm_sliced("N", "N", m, n, k, 1.0, As, m, B, k, 0.0, C, m, ws, wsb, torch.cuda.current_stream())
    assert torch.equal(C.T, want)


@pytest.mark.parametrize("e", [-1018, -1010, -1000, -990, -700, -560, -530, -500, 300, 500, 600])
@pytest.mark.parametrize("form", ["gemm", "syrk", "zgemm"])
def test_both_operands_scaled(gb, form, e):
    """A and B of integers times 2^e: the product is the integers' times 2^(2 e),
    from zero (below the subnormal range, of the sum's sign or none) over exact
    subnormal and normal results to infinities; zero sums stay zeros."""
    m, n, k = (70, 70, 40) if form == "syrk" else (130, 70, 40)
    g = torch.Generator(device="cuda").manual_seed(11)
    f = 2.0 ** e
    st = torch.cuda.current_stream()
    if form == "zgemm":
        A = torch.complex(ints(g, k, m), ints(g, k, m))
        B = torch.complex(ints(g, n, k), ints(g, n, k))
        want = torch.view_as_real((A.T @ B.T).contiguous())
        As, Bs = (torch.view_as_complex(torch.view_as_real(x) * f) for x in (A, B))
        C = torch.zeros(n, m, dtype=torch.complex128, device="cuda")
        wsb = gb.gb_zgemm_sliced_workspace_bytes(m, n, k)
        ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
        gb.gb_zgemm_sliced("N", m, n, k, 1.0, As, m, Bs, k, 0.0, C, m, ws, wsb, st)
        got = torch.view_as_real(C.T.contiguous())
    elif form == "syrk":
        A = ints(g, n, k)
        A[:, 3] = 0.0                                     # a zero column of products among odd ones
        A[5] = 0.0
        want = (A @ A.T).tril()
        C = torch.zeros(n, n, dtype=torch.float64, device="cuda")
        wsb = gb.gb_dsyrk_sliced_workspace_bytes(n, k)
        ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
        gb.gb_dsyrk_sliced(n, k, 1.0, A * f, k, 0.0, C, n, ws, wsb, st)
        got = C.T.tril()
    else:
        A, B = ints(g, k, m), ints(g, n, k)
        B[5] = 0.0
        want = A.T @ B.T
        C = torch.zeros(n, m, dtype=torch.float64, device="cuda")
        wsb = gb.gb_dgemm_sliced_workspace_bytes(m, n, k)
        ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
        gb.gb_dgemm_sliced("N", "N", m, n, k, 1.0, A * f, m, B * f, k, 0.0, C, m, ws, wsb, st)
        got = C.T
    assert torch.equal(got, want * f * f)   # (each factor alone stays in the range)


@pytest.mark.parametrize("x", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("k", [40, 300, 4100])
def test_nonfinite_entries_give_nan(gb, k, x):
    """A NaN or infinity in a row of op(A) or a column of op(B) makes that row or
    column of the product NaN; every other entry is exact.  (Entries below 1/2
    beside it: nothing overflows by itself.)"""
    m, n = 140, 75
    g = torch.Generator(device="cuda").manual_seed(k)
    A, B, C = ints(g, k, m) / 32, ints(g, n, k) / 32, ints(g, n, m)
    want = C.T - A.T @ B.T
    A[k // 2, 7] = x
    B[3, k - 1] = x
    want[7] = float("nan")
    want[:, 3] = float("nan")
    wsb = gb.gb_dgemm_sliced_workspace_bytes(m, n, k)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream()
    got = C.clone()
    gb.gb_dgemm_sliced("N", "N", m, n, k, -1.0, A, m, B, k, 1.0, got, m, ws, wsb, st)
    assert torch.equal(torch.nan_to_num(got.T, nan=1e9), torch.nan_to_num(want, nan=1e9))
    got = C.clone()
    gb.gb_dgemm_sliced("N", "N", m, n, k, 0.0, A, m, B, k, 2.0, got, m, ws, wsb, st)   # alpha = 0: no product
    assert torch.equal(got, 2.0 * C)


@pytest.mark.parametrize("x", [float("nan"), float("inf")])
def test_nonfinite_entries_of_the_other_forms(gb, x):
    """The symmetric, rank-2k and complex forms: a stored entry (i, j) reaches
    rows and columns i and j, a complex one both parts."""
    n, k = 200, 50
    g = torch.Generator(device="cuda").manual_seed(9)
    st = torch.cuda.current_stream()
    S = ints(g, n, n)
    S = S.tril() + S.tril(-1).T
    X, Y, C = ints(g, k, n), ints(g, k, n), ints(g, n, n)
    want = S @ X.T
    want[[150, 20]] = float("nan")
    Sx = S.clone()
    Sx[150, 20] = x
    wsb = gb.gb_dsymm_sliced_workspace_bytes("L", n, k)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    out = torch.zeros(k, n, dtype=torch.float64, device="cuda")
    gb.gb_dsymm_sliced("L", n, k, 1.0, Sx.T.contiguous(), n, X, n, 0.0, out, n, ws, wsb, st)
    assert torch.equal(torch.nan_to_num(out.T, nan=1e9), torch.nan_to_num(want, nan=1e9))
    low = torch.ones(n, n, dtype=torch.bool, device="cuda").tril()
    want = C.T - (X.T @ Y + Y.T @ X)
    want[33] = float("nan")
    want[:, 33] = float("nan")
    want = torch.where(low, want, C.T)
    X[4, 33] = x
    wsb = gb.gb_dsyr2k_sliced_workspace_bytes(n, k)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    out = C.clone()
    gb.gb_dsyr2k_sliced(n, k, -1.0, X, n, Y, n, 1.0, out, n, ws, wsb, st)
    assert torch.equal(torch.nan_to_num(out.T, nan=1e9), torch.nan_to_num(want, nan=1e9))
    A, B = torch.complex(ints(g, k, n), ints(g, k, n)), torch.complex(ints(g, n, k), ints(g, n, k))
    want = torch.view_as_real((A.T @ B.T).contiguous())
    want[61] = float("nan")
    A[2, 61] = complex(1.0, x)
    wsb = gb.gb_zgemm_sliced_workspace_bytes(n, n, k)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    out = torch.zeros(n, n, dtype=torch.complex128, device="cuda")
    gb.gb_zgemm_sliced("N", n, n, k, 1.0, A, n, B, k, 0.0, out, n, ws, wsb, st)
    got = torch.view_as_real(out.T.contiguous())
    assert torch.equal(torch.nan_to_num(got, nan=1e9), torch.nan_to_num(want, nan=1e9))


@pytest.mark.parametrize("n", [161, 300, 2200, 2600])
def test_long_operands_exact(gb, n):
    """Operands of one chunk of k a block and (n = 2600) of several: symmetric,
    and general ones along rows and columns."""
    c = 5
    g = torch.Generator(device="cuda").manual_seed(n)
    st = torch.cuda.current_stream()
    S, B = ints(g, n, n), ints(g, c, n)
    Y = S.tril() + S.tril(-1).T
    out = torch.zeros(c, n, dtype=torch.float64, device="cuda")
    wsb = gb.gb_dsymm_sliced_workspace_bytes("L", n, c)
    ws = torch.full((wsb,), 255, dtype=torch.uint8, device="cuda")
    gb.gb_dsymm_sliced("L", n, c, 1.0, S.T.contiguous(), n, B, n, 0.0, out, n, ws, wsb, st)
    assert torch.equal(out.T, Y @ B.T)
    for ta in "NT":
        wsb = gb.gb_dgemm_sliced_workspace_bytes(n, c, n)
        ws = torch.full((wsb,), 255, dtype=torch.uint8, device="cuda")
        gb.gb_dgemm_sliced(ta, "N", n, c, n, 1.0, S, n, B, n, 0.0, out, n, ws, wsb, st)
        assert torch.equal(out.T, (S.T if ta == "N" else S) @ B.T)
