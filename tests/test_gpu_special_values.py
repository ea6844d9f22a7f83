"""Inf and NaN in an operator's factors reach exactly the rows and columns that the definition sends them
to: each operator against a sum over the stored entries (a row without a constraint takes nothing
from the constraint part, and no row takes anything from entries it does not have)."""
import numpy as np
import pytest

from paper_2403_09133_gb300 import lorads as L
from paper_2403_09133_gb300.instances import SDPInstance

pytestmark = pytest.mark.gpu

RHO = 2.0


def _diag(rng):
    """Diagonal constraints on two thirds of the rows, a C with up to six entries per row."""
    n = 65
    rows = np.array([j for j in range(n) if j % 3 != 1])
    e = np.unique(np.sort(rng.integers(0, n, size=(3 * n, 2)), axis=1), axis=0)
    return SDPInstance(n=n, m=len(rows), C_row=e[:, 0], C_col=e[:, 1],
                       C_val=rng.standard_normal(len(e)), A_con=np.arange(len(rows)), A_row=rows,
                       A_col=rows, A_val=rng.uniform(0.5, 2.0, len(rows)), b=np.ones(len(rows)))


def _single(rng):
    """One entry per constraint, on and off the diagonal, 0 to about 20 entries per row."""
    n = 61
    e = np.unique(np.sort(rng.integers(0, n, size=(320, 2)), axis=1), axis=0)
    e = e[(e != 7).all(axis=1)]                        # row 7 carries no constraint
    e = np.concatenate([e, [[j, j] for j in range(20, 40)]])
    e = np.unique(e, axis=0)
    m = len(e)
    return SDPInstance(n=n, m=m, C_row=np.arange(n), C_col=np.arange(n), C_val=np.ones(n),
                       A_con=np.arange(m), A_row=e[:, 0], A_col=e[:, 1],
                       A_val=rng.uniform(0.5, 2.0, m), b=np.ones(m))


def _hessian(inst, W, P, gamma):
    H = np.zeros_like(P)
    for r, c, a in zip(inst.A_row, inst.A_col, inst.A_val):
        if r == c:
            H[r] += a * (a * (P[r] * W[r]).sum()) * W[r]
        else:
            q = a * ((P[r] * W[c]).sum() + (P[c] * W[r]).sum())
            H[r] += a * q * W[c]
            H[c] += a * q * W[r]
    return RHO * H + gamma * P


def _spmm(inst, w, V, gamma):
    S = np.zeros_like(V)
    for val, rows, cols in ((-np.asarray(inst.C_val), inst.C_row, inst.C_col),
                            (np.asarray(inst.A_val) * w[inst.A_con], inst.A_row, inst.A_col)):
        for r, c, a in zip(rows, cols, val):
            S[r] += a * V[c]
            if r != c:
                S[c] += a * V[r]
    return S + gamma * V if gamma != 0.0 else S


@pytest.mark.parametrize("prec", [L.LORADS_PREC_FP64, L.LORADS_PREC_MIXED])
@pytest.mark.parametrize("make", [_diag, _single])
@pytest.mark.parametrize("r", [3, 20, 40])
@pytest.mark.parametrize("where", ["V", "P"])
def test_operators_keep_special_values_to_their_entries(cuda, make, prec, r, where):
    torch = cuda
    rng = np.random.default_rng(r)
    inst = make(rng)
    dt = torch.float64 if prec == L.LORADS_PREC_FP64 else torch.float32
    ld = (r + 3) // 4 * 4
    V, P = rng.uniform(0.5, 1.5, (2, inst.n, r)).astype(np.float32).astype(np.float64)
    bad = V if where == "V" else P
    bad[4, 1], bad[7, 0], bad[33, 2] = np.inf, -np.inf, np.nan
    w = rng.standard_normal(inst.m)

    def dev(X):
        out = torch.zeros((inst.n, ld), dtype=dt, device="cuda")
        out[:, :r] = torch.as_tensor(X)
        return out

    dV, dP, dw = dev(V), dev(P), torch.as_tensor(w, device="cuda")
    H, S = torch.empty_like(dV), torch.empty_like(dV)
    p = L.Problem(inst)
    gammas = (0.0, 1.25)
    got = []
    for gamma in gammas:
        assert L.lorads_op_hessian(p.handle, prec, r, ld, RHO, gamma, dV, dP, H) == 0
        assert L.lorads_op_spmm(p.handle, prec, r, ld, dw, gamma, dV, S) == 0
        got.append((H.cpu().numpy()[:, :r].astype(float), S.cpu().numpy()[:, :r].astype(float)))
    p.close()
    # up to 20 entries of at most 40 products each, of like sign in the Hessian; FP32 4e-7 * 60
    tol = 1e-12 if prec == L.LORADS_PREC_FP64 else 3e-5
    with np.errstate(all="ignore"):
        for gamma, (gH, gS) in zip(gammas, got):
            for g, x in ((gH, _hessian(inst, V, P, gamma)), (gS, _spmm(inst, w, V, gamma))):
                assert np.array_equal(np.isnan(g), np.isnan(x))
                assert np.array_equal(np.isposinf(g), np.isposinf(x))
                assert np.array_equal(np.isneginf(g), np.isneginf(x))
                f = np.isfinite(x)
                assert np.abs(g[f] - x[f]).max() <= tol * np.abs(x[f]).max()
