"""Workloads of the eigensolver library: what its users have it do, through
its public entry points, from the smallest solves to the largest ones.

A case is a dict of plain values whose "kind" is one of

  solve     one real symmetric or complex Hermitian eigensolve (gb_solve_d, gb_solve_z)
  batched   many uneven real problems at once on 16 streams (gb_solve_batched_d)
  mixed     the mixed-precision solve, FP32 products and FP64 refinement (gb_solve_mixed_d)
  backtrans the back-transformation from tridiagonal to band form alone
            (gb_trans_ev_tridi_to_band_d / _z)
  tridiag   all eigenpairs of a tridiagonal matrix (gb_tridiag_dc_d)
  product   one FP64 matrix product on the tensor cores (gb_dgemm_sliced)

Dense matrices are symmetrised Gaussian ones, tridiagonal ones have the
entries that such matrices have after reduction (Dumitriu and Edelman's
beta-Hermite model), reflectors are random orthogonal (unitary) ones in the
bulge chase's layout.  Eigenvectors are unique up to a sign (a phase): `run`
makes the first component of each real and not negative, as a program does
that follows its eigenvectors from one call to the next.
"""
import math

import torch

import paper_1811_01277_gb300 as gb

SLOTS = 16          # streams of a batch
MIXED_STEPS = 3     # refinement steps of a mixed-precision solve


def listed():
    return [
        # the smallest solves of a batch of k-points or spins: one launch chain, latency alone counts
        {"name": "solve_180_all", "kind": "solve", "cplx": False, "n": 180, "nev": 180, "nbw": 0},
        # a plain solve of a small system, all pairs, in the band width of the small configuration
        {"name": "solve_1024_all", "kind": "solve", "cplx": False, "n": 1024, "nev": 1024, "nbw": 32},
        # a large solve for the lowest quarter of the pairs, as an SCF step asks for its occupied states
        {"name": "solve_8192_quarter", "kind": "solve", "cplx": False, "n": 8192, "nev": 2048, "nbw": 64},
        # one request of a server of complex Hermitian problems (a k-point), 30 % of the pairs, an odd size
        {"name": "solve_z_1501_30pct", "kind": "solve", "cplx": True, "n": 1501, "nev": 450, "nbw": 0},
        # a batch of uneven problems of 128 to 2048, all pairs
        {"name": "batched_24", "kind": "batched", "count": 24, "lo": 128, "hi": 2048, "mix": 512},
        # the mixed-precision solve, half of the pairs
        {"name": "mixed_2048_half", "kind": "mixed", "n": 2048, "nev": 1024, "nbw": 64},
        # the back-transformation of the large solve, alone
        {"name": "backtrans_16384", "kind": "backtrans", "cplx": False, "n": 16384, "nev": 4096, "nbw": 64},
        # the same for complex eigenvectors
        {"name": "backtrans_z_4096", "kind": "backtrans", "cplx": True, "n": 4096, "nev": 1228, "nbw": 64},
        # and for the small configuration
        {"name": "backtrans_1024", "kind": "backtrans", "cplx": False, "n": 1024, "nev": 1024, "nbw": 32},
        # a small problem of a batch, odd sizes, below the tensor-core kernels' range
        {"name": "backtrans_333", "kind": "backtrans", "cplx": False, "n": 333, "nev": 301, "nbw": 32},
        # the tridiagonal step of an all-pairs solve
        {"name": "tridiag_2500", "kind": "tridiag", "n": 2500},
        # an update C - A B of odd sizes, as a program around the solver does with its eigenvectors
        {"name": "product_3001", "kind": "product", "ta": "N", "tb": "N", "m": 3001, "n": 1777, "k": 4099},
    ]


def _size(rng, lo, hi):
    """An integer of [lo, hi], spread over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve_z", "batched", "mixed", "backtrans", "backtrans", "backtrans_z",
                       "tridiag", "product", "product"])
    if kind == "solve":
        n = _size(rng, 128, 6000)
        share = rng.choice([1.0, 0.5, 0.25]) if n <= 3000 else 0.25
        return {"kind": "solve", "cplx": False, "n": n, "nev": max(1, int(n * share)), "nbw": rng.choice([0, 32, 64])}
    if kind == "solve_z":
        n = _size(rng, 128, 2500)
        return {"kind": "solve", "cplx": True, "n": n, "nev": max(1, int(0.3 * n)), "nbw": 0}
    if kind == "batched":
        return {"kind": "batched", "count": rng.randint(6, 24), "lo": 128, "hi": _size(rng, 256, 2048),
                "mix": rng.randrange(1 << 20)}
    if kind == "mixed":
        n = _size(rng, 512, 2500)
        return {"kind": "mixed", "n": n, "nev": n // 2, "nbw": 64}
    if kind == "backtrans":
        n = _size(rng, 200, 12000)
        return {"kind": "backtrans", "cplx": False, "n": n, "nev": _size(rng, 50, min(n, 4096)),
                "nbw": rng.choice([16, 32, 64, 64])}
    if kind == "backtrans_z":
        n = _size(rng, 512, 6000)
        return {"kind": "backtrans", "cplx": True, "n": n, "nev": _size(rng, 50, min(n, 2048)),
                "nbw": rng.choice([32, 64])}
    if kind == "tridiag":
        return {"kind": "tridiag", "n": _size(rng, 100, 5000)}
    return {"kind": "product", "ta": rng.choice("NT"), "tb": rng.choice("NT"), "m": _size(rng, 32, 6000),
            "n": _size(rng, 32, 6000), "k": _size(rng, 32, 6000)}


# ---- inputs ----

def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _gen(seed):
    return torch.Generator(device=_dev()).manual_seed(int(seed) % (1 << 62))


def _randn(g, *shape, cplx=False):
    return torch.randn(*shape, generator=g, device=_dev(), dtype=torch.complex128 if cplx else torch.float64)


def _dense(g, n, cplx=False):
    """Symmetrised (Hermitian) Gaussian matrix, column-major in memory."""
    R = _randn(g, n, n, cplx=cplx)
    A = 0.5 * (R + R.mH)
    return A.mT.contiguous().mT if cplx else A


def _reflectors(g, n, b, cplx):
    """Random orthogonal (unitary) reflectors in the bulge chase's layout."""
    dev = _dev()
    sweep = torch.arange(1, n, device=dev)
    nk = (n - sweep + b - 1) // b
    first = torch.cumsum(nk, 0) - nk
    k = torch.arange(int(nk.sum()), device=dev) - torch.repeat_interleave(first, nk)
    lens = torch.clamp(n - torch.repeat_interleave(sweep, nk) - k * b, max=b)
    cnt = lens.numel()
    V = torch.rand(cnt, b, generator=g, device=dev, dtype=torch.float64).mul_(2).sub_(1)
    if cplx:
        V = torch.complex(V, torch.rand(cnt, b, generator=g, device=dev, dtype=torch.float64).mul_(2).sub_(1))
        V *= 0.5 ** 0.5
    V /= lens.to(torch.float64).sqrt()[:, None]
    V[torch.arange(b, device=dev)[None, :] >= lens[:, None]] = 0.0
    V[:, 0] = 1.0
    nrm2 = (V.real.square() + V.imag.square()).sum(1) if cplx else V.square().sum(1)
    if cplx:
        theta = (0.5 + torch.rand(cnt, generator=g, device=dev, dtype=torch.float64)) * math.pi
        tau = (1.0 - torch.polar(torch.ones_like(theta), theta)) / nrm2
    else:
        tau = 2.0 / nrm2
    return V, tau


def _tridiagonal(g, n):
    """Diagonal and couplings of a reduced Gaussian matrix of order n."""
    d = _randn(g, n)
    dof = torch.arange(n - 1, 0, -1, device=_dev(), dtype=torch.float64)
    # chi variables: square roots of Gamma(dof / 2, scale 2), through the Wilson-Hilferty cube
    x = 1.0 - 2.0 / (9.0 * dof) + _randn(g, n - 1) * (2.0 / (9.0 * dof)).sqrt()
    return d, (0.5 * dof * x.abs() ** 3).sqrt()


def _batch_sizes(case):
    """The orders of a batch's problems: one from each of `count` equal parts of the range, in random order."""
    g = torch.Generator().manual_seed(case["mix"])
    lo, hi, c = case["lo"], case["hi"], case["count"]
    u = (torch.randperm(c, generator=g).to(torch.float64) + torch.rand(c, generator=g, dtype=torch.float64)) / c
    return [min(hi, lo + int(v * (hi - lo + 1))) for v in u.tolist()]


def _bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device=_dev())


def _like(rows, cols, cplx=False):
    return torch.zeros(rows, cols, dtype=torch.complex128 if cplx else torch.float64, device=_dev())


def prepare(case, seed):
    kind, g = case["kind"], _gen(seed)
    s = {"case": dict(case)}
    if kind == "solve":
        n, nev, cplx = case["n"], case["nev"], case["cplx"]
        nbw = case["nbw"] or gb.gb_solve_default_nbw(n)
        wsb = gb.gb_solve_workspace_bytes_z(n, nev, nbw) if cplx else gb.gb_solve_workspace_bytes(n, nev, nbw)
        s.update(A=_dense(g, n, cplx), ev=torch.zeros(nev, dtype=torch.float64, device=_dev()),
                 Z=_like(nev, n, cplx), nbw=nbw, ws=_bytes(wsb), wsb=wsb)
    elif kind == "batched":
        sizes = _batch_sizes(case)
        wsb = gb.gb_solve_batched_workspace_bytes(sizes, sizes, SLOTS)
        s.update(sizes=sizes, A=[_dense(g, n) for n in sizes], Z=[_like(n, n) for n in sizes],
                 ev=[torch.zeros(n, dtype=torch.float64, device=_dev()) for n in sizes],
                 streams=[torch.cuda.Stream() for _ in range(SLOTS)], ws=_bytes(wsb), wsb=wsb)
    elif kind == "mixed":
        n, nev, nbw = case["n"], case["nev"], case["nbw"]
        wsb = gb.gb_solve_mixed_workspace_bytes(n, nev, nbw)
        s.update(A=_dense(g, n), ev=torch.zeros(nev, dtype=torch.float64, device=_dev()), Z=_like(nev, n),
                 ws=_bytes(wsb), wsb=wsb)
    elif kind == "backtrans":
        n, nev, b, cplx = case["n"], case["nev"], case["nbw"], case["cplx"]
        V, tau = _reflectors(g, n, b, cplx)
        wsb = gb.gb_trans_ev_workspace_bytes(n, b, nev, cplx)
        s.update(V=V, tau=tau, Z=_randn(g, nev, n, cplx=cplx) / math.sqrt(n), ws=_bytes(wsb), wsb=wsb)
    elif kind == "tridiag":
        n = case["n"]
        d, e = _tridiagonal(g, n)
        wsb = gb.gb_tridiag_dc_workspace_bytes(n)
        s.update(d=d, e=e, lam=torch.zeros(n, dtype=torch.float64, device=_dev()), Q=_like(n, n), ws=_bytes(wsb),
                 wsb=wsb)
    else:
        m, n, k = case["m"], case["n"], case["k"]
        wsb = gb.gb_dgemm_sliced_workspace_bytes(m, n, k)
        # column-major operands: a tensor of shape (columns, rows)
        s.update(A=_randn(g, *((k, m) if case["ta"] == "N" else (m, k))),
                 B=_randn(g, *((n, k) if case["tb"] == "N" else (k, n))), C=_randn(g, n, m), ws=_bytes(wsb), wsb=wsb)
    return s


# ---- one pass ----

def _fix_phase(Z):
    """Rows of Z (eigenvectors): first component real and not negative, in place."""
    z0 = Z[:, :1]
    if Z.is_complex():
        return Z.mul_(torch.where(z0 == 0, torch.ones_like(z0), torch.sgn(z0).conj()))
    return Z.mul_(torch.where(z0 < 0, -1.0, 1.0))


def run(s):
    case = s["case"]
    kind, st = case["kind"], torch.cuda.current_stream()
    if kind == "solve":
        n, nev = case["n"], case["nev"]
        solve = gb.gb_solve_z if case["cplx"] else gb.gb_solve_d
        solve(n, nev, s["nbw"], s["A"], n, s["ev"], s["Z"], n, s["ws"], s["wsb"], st)
        return {"ev": s["ev"], "Z": _fix_phase(s["Z"])}
    if kind == "batched":
        sizes, streams = s["sizes"], s["streams"]
        for q in streams:
            q.wait_stream(st)
        gb.gb_solve_batched_d(sizes, sizes, s["A"], sizes, s["ev"], s["Z"], sizes, s["ws"], s["wsb"], streams)
        for q in streams:
            st.wait_stream(q)
        return {"ev": s["ev"], "Z": [_fix_phase(Z) for Z in s["Z"]]}
    if kind == "mixed":
        n = case["n"]
        gb.gb_solve_mixed_d(n, case["nev"], case["nbw"], s["A"], n, s["ev"], s["Z"], n, MIXED_STEPS, s["ws"],
                            s["wsb"], st)
        return {"ev": s["ev"], "Z": _fix_phase(s["Z"])}
    if kind == "backtrans":
        n, nev = case["n"], case["nev"]
        f = gb.gb_trans_ev_tridi_to_band_z if case["cplx"] else gb.gb_trans_ev_tridi_to_band_d
        f(n, case["nbw"], nev, s["V"], s["tau"], s["Z"], n, s["ws"], s["wsb"], st)
        return {"Z": s["Z"]}
    if kind == "tridiag":
        n = case["n"]
        gb.gb_tridiag_dc_d(n, s["d"], s["e"], s["lam"], s["Q"], n, s["ws"], s["wsb"], st)
        return {"lam": s["lam"], "Q": _fix_phase(s["Q"])}
    m, n, k = case["m"], case["n"], case["k"]
    gb.gb_dgemm_sliced(case["ta"], case["tb"], m, n, k, -1.0, s["A"], s["A"].shape[1], s["B"], s["B"].shape[1], 1.0,
                       s["C"], m, s["ws"], s["wsb"], st)
    return {"C": s["C"]}


# ---- what a pass cannot do without ----

def _solve_flops(n, nev, cplx):
    """Reduction 4/3 n^3, both back-transformations 2 n^2 nev each (real flops)."""
    return (4 if cplx else 1) * (4.0 / 3.0 * n ** 3 + 4.0 * n * n * nev)


def work(case):
    kind = case["kind"]
    if kind in ("solve", "mixed"):
        n, nev, cplx = case["n"], case["nev"], case.get("cplx", False)
        el = 16 if cplx else 8
        return {"bytes": el * (n * n + n * nev) + 8 * nev, "flops": _solve_flops(n, nev, cplx)}
    if kind == "batched":
        sizes = _batch_sizes(case)
        return {"bytes": sum(16 * n * n + 8 * n for n in sizes), "flops": sum(_solve_flops(n, n, False) for n in sizes)}
    if kind == "backtrans":
        n, nev, b = case["n"], case["nev"], case["nbw"]
        el = 16 if case["cplx"] else 8
        cnt = gb.gb_hh_count(n, b)
        # four real flops for each entry of a reflector and column, 16 complex ones
        return {"bytes": el * (cnt * (b + 1) + 2 * n * nev), "flops": (4 if case["cplx"] else 1) * 2.0 * n * (n - 1) * nev}
    if kind == "tridiag":
        n = case["n"]
        return {"bytes": 8 * (n * n + 3 * n), "flops": 4.0 / 3.0 * n ** 3}
    m, n, k = case["m"], case["n"], case["k"]
    return {"bytes": 8 * (m * k + k * n + 2 * m * n), "flops": 2.0 * m * n * k}


# ---- the same in plain torch, 64 bits ----

def _eigh(A, nev):
    lam, Q = torch.linalg.eigh(A)
    return lam[:nev].clone(), _fix_phase(Q[:, :nev].mT.contiguous())


def _apply_reflectors(V, tau, Z, n, b):
    """Q2 Z by sweeps, last first; the reflectors of one sweep touch rows of their own."""
    nev = Z.shape[0]
    X = torch.zeros(n + b, nev, dtype=Z.dtype, device=Z.device)
    X[:n] = Z.mT
    end = V.shape[0]
    for s in range(n - 1, 0, -1):
        nk = (n - s + b - 1) // b
        v, t = V[end - nk:end], tau[end - nk:end]
        end -= nk
        # the rows past n are zero and stay zero: v is zero there
        x = X[s:s + nk * b].view(nk, b, nev)
        w = torch.bmm(v.conj().unsqueeze(1), x)
        x.baddbmm_((t[:, None] * v).unsqueeze(2), w, alpha=-1)
    return X[:n].mT.contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "mixed") and case["n"] > 5000:
        return None
    s = prepare(case, seed)
    if kind in ("solve", "mixed"):
        ev, Z = _eigh(s["A"], case["nev"])
        return {"ev": ev, "Z": Z}
    if kind == "batched":
        got = [_eigh(A, A.shape[0]) for A in s["A"]]
        return {"ev": [ev for ev, _ in got], "Z": [Z for _, Z in got]}
    if kind == "backtrans":
        return {"Z": _apply_reflectors(s["V"], s["tau"], s["Z"], case["n"], case["nbw"])}
    if kind == "tridiag":
        lam, Q = _eigh(torch.diag(s["d"]) + torch.diag(s["e"], 1) + torch.diag(s["e"], -1), case["n"])
        return {"lam": lam, "Q": Q}
    A, B = s["A"], s["B"]
    left = A.mT if case["ta"] == "N" else A
    right = B.mT if case["tb"] == "N" else B
    return {"C": (s["C"].mT - left @ right).mT.contiguous()}
