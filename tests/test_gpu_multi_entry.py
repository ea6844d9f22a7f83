"""The sampled product with constraints of uneven lengths: numerics at the edges of a round, and a long
constraint's time beside short ones."""
import time

import numpy as np
import pytest

from paper_2403_09133_gb300 import lorads as L
from paper_2403_09133_gb300.instances import SDPInstance

pytestmark = pytest.mark.gpu


def _problem(n, lengths, diagonal, rng):
    """Constraint i has lengths[i] entries: the diagonal from row 0 on, or random ones off it."""
    con, row, col = [], [], []
    for i, k in enumerate(lengths):
        if diagonal[i]:
            r = c = np.arange(k)
        else:
            e = rng.choice(n * (n - 1) // 2, size=k, replace=False)
            r = (n - 2 - np.floor(np.sqrt(4.0 * n * (n - 1) - 7 - 8.0 * e) / 2.0 - 0.5)).astype(int)
            c = e + r + 1 - n * (n - 1) // 2 + (n - r) * (n - r - 1) // 2
        con.append(np.full(k, i)), row.append(r), col.append(c)
    con, row, col = map(np.concatenate, (con, row, col))
    assert (row <= col).all() and (col < n).all() and (row >= 0).all()
    return SDPInstance(n=n, m=len(lengths), C_row=np.arange(n), C_col=np.arange(n),
                       C_val=np.ones(n), A_con=con, A_row=row, A_col=col,
                       A_val=rng.uniform(0.5, 2.0, len(con)), b=np.ones(len(lengths)))


def _call(torch, inst, prec, r, rng):
    dt = torch.float64 if prec == L.LORADS_PREC_FP64 else torch.float32
    ld = (r + 3) // 4 * 4
    U, V = rng.standard_normal((2, inst.n, r)).astype(np.float32).astype(np.float64)
    dev = []
    for X in (U, V):
        d = torch.zeros((inst.n, ld), dtype=dt, device="cuda")
        d[:, :r] = torch.as_tensor(X)
        dev.append(d)
    q = torch.full((inst.m,), np.nan, dtype=torch.float64, device="cuda")
    return U, V, dev, q, ld


@pytest.mark.parametrize("prec", [L.LORADS_PREC_FP64, L.LORADS_PREC_MIXED])
@pytest.mark.parametrize("r", [3, 9, 20, 40])
def test_uneven_constraints(cuda, prec, r):
    """Lengths 1 to 71, odd and even, diagonal and not, in one warp and across warps."""
    rng = np.random.default_rng(r)
    lengths = [1, 2, 71, 1, 3, 8, 1, 1, 33, 32, 1, 5, 64, 2, 1, 1, 7, 1, 70, 1, 4]
    diagonal = [(i * 7) % 3 == 0 for i in range(len(lengths))]
    inst = _problem(71, lengths, diagonal, rng)
    U, V, (dU, dV), q, ld = _call(cuda, inst, prec, r, rng)
    p = L.Problem(inst)
    assert L.lorads_op_sddmm(p.handle, prec, r, ld, dU, dV, q) == 0
    got = q.cpu().numpy()
    p.close()
    want, size = np.zeros(inst.m), np.zeros(inst.m)
    for i, a, b, v in zip(inst.A_con, inst.A_row, inst.A_col, inst.A_val):
        terms = U[a] * V[b] + (U[b] * V[a] if a != b else 0.0)
        want[i] += v * terms.sum()
        size[i] += v * (np.abs(U[a] * V[b]) + (np.abs(U[b] * V[a]) if a != b else 0.0)).sum()
    # each entry's dot product rounds in T (at most 80 terms), the sums over entries in FP64
    eps = 2.0 ** -53 if prec == L.LORADS_PREC_FP64 else 2.0 ** -24
    assert (np.abs(got - want) <= 80 * eps * size + 1e-13 * size).all()


@pytest.mark.parametrize("prec", [L.LORADS_PREC_FP64, L.LORADS_PREC_MIXED])
def test_a_long_constraint_beside_short_ones(cuda, prec):
    """A trace of 2,000 entries takes as long beside constraints of one entry as alone (they shared its warp's
    rounds: 1.3 times)."""
    torch = cuda
    rng = np.random.default_rng(1)
    times = []
    for short in (0, 3000):
        inst = _problem(2000, [1] * short + [2000], [False] * short + [True], rng)
        _, _, (dU, dV), q, ld = _call(torch, inst, prec, 9, rng)
        p = L.Problem(inst)
        best = 1e9
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(20):
                assert L.lorads_op_sddmm(p.handle, prec, 9, ld, dU, dV, q) == 0
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        times.append(best)
        p.close()
    assert times[1] <= 1.15 * times[0], times
