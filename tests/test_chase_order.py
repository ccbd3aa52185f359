"""Which stores the loads of the cluster chase (csrc/band_to_tridi.cu) meet: a
model of the blocks' loads, stores, flags and slots on the CPU.

Sweeps run on clusters of their own, so all that orders a load after a store
is what the loader waits for: O(s,k) for the O blocks of sweep s-1 up to step
k, D(s,k) for its O blocks up to step k+1 and its D blocks up to step k, and
whatever those had waited for.  (Slots carry one value each and order nothing
else.)  Every entry that a block takes from the band must have been stored
last by a block it is ordered after, and be the entry's value in the plain
chase; a store may only replace one that is there already (the slots are
filled by D blocks that had waited for it).  Values: numpy's two-sided reflections, 1e-12 ||B||.
"""
import numpy as np
import pytest

from paper_1811_01277_gb300 import inputs


def steps(n, b, s):
    return (n - s + b - 1) // b if 1 <= s < n else 0


def ordered(kind, s, k, n, b):
    """The last stored steps (O, D) of every earlier sweep that a load of
    block `kind`(s,k) is ordered after, -1 for none."""
    o, d = {}, {}
    need_o, need_d = (k, -1) if kind == "O" else (k + 1, k)
    for t in range(s - 1, 0, -1):
        # O(t, need_o) and D(t, need_d) have stored; both had waited for sweep t-1
        o[t], d[t] = min(need_o, steps(n, b, t) - 1), min(need_d, steps(n, b, t) - 1)
        need_o, need_d = max(o[t], d[t] + 1 if d[t] >= 0 else -1), d[t]
    return o, d


def run(n, b, last_row_zero, seed=0):
    """Violations of the order, and the model's matrix beside the plain one's."""
    B = inputs.band_symmetric(n, b, seed=seed + 7 * n + b)
    nrm = np.linalg.norm(B, 2)
    A = B.copy()                                # the plain chase
    W = np.tril(B)                              # the model's band: what blocks have stored
    writer = {}
    slot = {}                                   # betas and first columns, by entry
    bad = []

    def load(kind, s, k, i, j, now):
        w = writer.get((i, j))
        if w is not None:
            wk, ws, wstep = w
            o, d = ordered(kind, s, k, n, b)
            if not (o if wk == "O" else d).get(ws, -1) >= wstep:
                bad.append((kind, s, k, i, j, w))
        assert abs(W[i, j] - now[i, j]) <= 1e-12 * nrm, (kind, s, k, i, j)
        return W[i, j]

    def store(kind, s, k, i, j):
        w = writer.get((i, j))
        if w is not None and w[1] != s:
            # blocks store once their slots have come: O(s,k)'s last column from
            # D(s-1,k), D(s,k)'s last entry from D(s-1,k+1)
            seen = [ordered(kind, s, k, n, b), ordered("D", s - 1, k if kind == "O" else k + 1, n, b)]
            if not any((o if w[0] == "O" else d).get(w[1], -1) >= w[2] for o, d in seen):
                bad.append((kind, s, k, i, j, w))
        W[i, j] = A[i, j]
        writer[(i, j)] = (kind, s, k)

    for s in range(1, n):
        for k in range(steps(n, b, s)):
            r = s + k * b
            ln = min(b, n - r)
            c = s - 1 if k == 0 else r - b
            nc = 1 if k == 0 else b
            # O as it is loaded, before H(s,k-1) acts on it from the right
            now = A if k == 0 else before
            for i in range(ln):
                for j in range(nc):
                    if s > 1 and j == nc - 1:
                        got = slot[(r + i, c + j)]
                    elif s > 1 and i == b - 1 and last_row_zero:
                        got = 0.0
                    else:
                        got = load("O", s, k, r + i, c + j, now)
                    assert abs(got - now[r + i, c + j]) <= 1e-12 * nrm, (s, k, i, j)
            x = A[r:r + ln, c].copy()
            ss, alpha = float(x[1:] @ x[1:]), x[0]
            v = np.zeros(n)
            tau, beta = 0.0, alpha
            if ss != 0.0:
                beta = -np.copysign(np.sqrt(alpha * alpha + ss), alpha)
                tau = (beta - alpha) / beta
                v[r:r + ln] = x / (alpha - beta)
                v[r] = 1.0
            for i in range(ln):
                for j in range(i + 1):
                    if s > 1 and i == b - 1 and j == b - 1:
                        got = slot[(r + i, r + j)]
                    else:
                        got = load("D", s, k, r + i, r + j, A)
                    assert abs(got - A[r + i, r + j]) <= 1e-12 * nrm, (s, k, i, j)
            before = A.copy()
            A -= tau * np.outer(v, v @ A)
            A -= tau * np.outer(A @ v, v)
            # stores: O without its first column, whose head goes through a slot;
            # D without its first column, which goes through slots
            for i in range(ln):
                for j in range(1, nc):
                    store("O", s, k, r + i, c + j)
                if not last_row_zero and i > 0:
                    store("O", s, k, r + i, c)
                for j in range(1, i + 1):
                    store("D", s, k, r + i, r + j)
                slot[(r + i, r)] = A[r + i, r]
            slot[(r, c)] = beta
    return bad, A, B


SHAPES = [(b + d, b) for b in (1, 2, 3, 5, 8) for d in (1, b, 2 * b + 1, 3 * b + 2, 4 * b)]


@pytest.mark.parametrize("n,b", SHAPES)
def test_every_load_is_ordered_after_its_store(n, b):
    bad, A, B = run(n, b, last_row_zero=True)
    assert not bad
    lam = np.linalg.eigvalsh(np.diag(np.diag(A)) + np.diag(np.diag(A, -1), -1) + np.diag(np.diag(A, -1), 1))
    assert np.abs(lam - np.linalg.eigvalsh(B)).max() <= 1e-12 * np.linalg.norm(B, 2)


def test_loading_the_last_row_is_not_ordered():
    """O(s,k)'s last row, loaded from the band, meets zeros of O(s-2,k+1): a
    step beyond what O(s-1,k)'s flags imply."""
    bad, _, _ = run(24, 5, last_row_zero=False)
    assert bad and all(x[0] == "O" and x[3] == x[1] + x[2] * 5 + 4 and x[5][2] == x[2] + 1 for x in bad)
