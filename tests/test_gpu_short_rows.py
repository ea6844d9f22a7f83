"""Operators of the general form (a warp per row) on both sides of their short-row rules: rows of 0 to 3
entries per sub-team, at the counts where a round of one or of two entries ends.  Against the oracle."""
import numpy as np
import pytest

import oracle.lorads as OL
from oracle import SDP
from paper_2403_09133_gb300 import lorads as L
from paper_2403_09133_gb300.instances import SDPInstance

pytestmark = pytest.mark.gpu


def _instance(n, per_row, rng):
    """One entry per constraint; row j < 40 has about j entries beside a background of per_row."""
    e = [np.sort(rng.integers(0, n, size=(n * per_row // 2, 2)), axis=1)]
    for j in range(40):
        e.append(np.sort(np.stack([np.full(j, j), rng.integers(0, n, size=j)], axis=1), axis=1))
    e = np.unique(np.concatenate(e), axis=0)
    m = len(e)
    c = np.unique(np.sort(rng.integers(0, n, size=(2 * n, 2)), axis=1), axis=0)
    return SDPInstance(n=n, m=m, C_row=c[:, 0], C_col=c[:, 1], C_val=rng.standard_normal(len(c)),
                       A_con=np.arange(m), A_row=e[:, 0], A_col=e[:, 1],
                       A_val=rng.uniform(0.5, 2.0, m), b=np.ones(m))


@pytest.mark.parametrize("prec", [L.LORADS_PREC_FP64, L.LORADS_PREC_MIXED])
@pytest.mark.parametrize("r", [4, 9, 16, 20, 40, 100])
@pytest.mark.parametrize("n,per_row", [(400, 3), (150, 30), (201, 90), (7400, 40)])
def test_rows_of_uneven_lengths(cuda, prec, r, n, per_row):
    torch = cuda
    rng = np.random.default_rng(r + n)
    inst = _instance(n, per_row, rng)
    sdp = SDP.from_instance(inst)
    dt = torch.float64 if prec == L.LORADS_PREC_FP64 else torch.float32
    ld = (r + 3) // 4 * 4
    V, P = (rng.standard_normal((2, n, r)) / np.sqrt(r)).astype(np.float32).astype(np.float64)
    w = rng.standard_normal(inst.m)

    def dev(X):
        out = torch.zeros((n, ld), dtype=dt, device="cuda")
        out[:, :r] = torch.as_tensor(X)
        return out

    dV, dP, dw = dev(V), dev(P), torch.as_tensor(w, device="cuda")
    H, S = torch.full_like(dV, float("nan")), torch.full_like(dV, float("nan"))
    p = L.Problem(inst)
    assert L.lorads_op_hessian(p.handle, prec, r, ld, 7.0, 1.25, dV, dP, H) == 0
    assert L.lorads_op_spmm(p.handle, prec, r, ld, dw, 0.75, dV, S) == 0
    H, S = H.cpu().numpy(), S.cpu().numpy()
    p.close()
    # at most 140 entries a row of 200 products each, rounding growing like its root: 200 ulp in FP32
    tol = 1e-12 if prec == L.LORADS_PREC_FP64 else 200 * 2.0 ** -24
    for got, want in ((H, OL.hessian_apply(sdp, V, P, 7.0, 1.25)),
                      (S, sdp.At_times(w, V) - sdp.C_times(V) + 0.75 * V)):
        assert np.abs(got[:, :r] - want).max() <= tol * np.abs(want).max()
        assert np.all(got[:, r:] == 0.0)
