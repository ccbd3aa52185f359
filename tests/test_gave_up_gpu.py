"""Waits that run out in the products and the panel factorisation: the call
returns, the status word says GB_ERR_TIMEOUT, and nothing that was not finished
looks like a result.  The waits are made to run out by a short limit and an
arrival or copy that is left out (hooks of the library); they end by themselves
and the context stays usable.
"""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WAIT_NS = 20_000_000


@pytest.fixture(scope="module")
def gb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1811_01277_gb300 as m
    from paper_1811_01277_gb300 import build
    build.build()
    m.load()
    return m


def ptr(x):
    return ctypes.c_void_p(x.data_ptr())


@pytest.mark.parametrize("m,n,k,hold", [(130, 70, 40, 0), (130, 70, 400, 1), (2500, 2500, 96, 0), (2500, 2500, 96, 4),
                                        (300, 300, 4100, 3), (2500, 2500, 96, -1), (300, 300, 4100, -1)])
def test_product(gb, m, n, k, hold):
    g = torch.Generator(device="cuda").manual_seed(m + k)
    A = torch.randint(-9, 10, (k, m), generator=g, device="cuda").double()
    B = torch.randint(-9, 10, (n, k), generator=g, device="cuda").double()
    C = torch.full((n, m), 0.5, dtype=torch.float64, device="cuda")
    ws = torch.empty(gb.gb_dgemm_sliced_workspace_bytes(m, n, k), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = torch.cuda.current_stream()
    rc = gb.load().gb_test_sliced_hold(ctypes.c_int(m), ctypes.c_int(n), ctypes.c_int(k), ptr(A), ptr(B), ptr(C), ptr(ws),
                                       ctypes.c_longlong(WAIT_NS), ctypes.c_int(hold), ptr(status),
                                       ctypes.c_void_p(st.cuda_stream))
    torch.cuda.synchronize()
    nan = torch.isnan(C)
    assert rc == 0 and torch.equal(C[~nan], (A.T @ B.T).T[~nan])
    if hold < 0:
        assert status.item() == 0 and not nan.any()
    else:
        assert status.item() == 2 and nan.any()
        if hold == 0:
            assert nan.all()


@pytest.mark.parametrize("m,nb,hold", [(200, 32, 0), (900, 64, 5), (1500, 17, 16), (5000, 64, 3), (5000, 32, 31),
                                       (5000, 64, -1), (900, 64, -1)])
@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
def test_panel(gb, m, nb, hold, cplx):
    dt = torch.complex128 if cplx else torch.float64
    g = torch.Generator(device="cuda").manual_seed(m + nb)
    P = torch.randn(nb, m, generator=g, dtype=dt, device="cuda")
    Y = torch.zeros_like(P)
    tau = torch.zeros(nb, dtype=dt, device="cuda")
    part = torch.empty(256 + 2 * 64 * ((m + 63) // 64 + 1) * 16, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = torch.cuda.current_stream()
    rc = gb.load().gb_test_panel_hold(ctypes.c_int(cplx), ctypes.c_int(m), ctypes.c_int(nb), ptr(P), ptr(tau), ptr(Y),
                                      ptr(part), ctypes.c_longlong(WAIT_NS if hold >= 0 else 10 ** 9), ctypes.c_int(hold),
                                      ptr(status), ctypes.c_void_p(st.cuda_stream))
    torch.cuda.synchronize()
    assert rc == 0
    if hold < 0:
        assert status.item() == 0 and torch.isfinite(torch.view_as_real(P) if cplx else P).all()
    else:
        assert status.item() == 2
        assert torch.isnan(P).all() and torch.isnan(Y).all()
