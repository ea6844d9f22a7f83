"""The FP64 operators' unit layout where test_gpu_units.py's few rows do not lead: two and four lanes per
row, which many rows take, with every count of units per lane, odd row counts, and six and seven units
per lane at eight lanes.  Against the oracle's definitions, FP64, 1e-12 of the terms' size.  And the FP32
product with diagonal constraints."""
import numpy as np
import pytest

import oracle.lorads as OL
from oracle import SDP
from paper_2403_09133_gb300 import instances as I
from paper_2403_09133_gb300 import lorads as L

pytestmark = pytest.mark.gpu

TWO, FOUR = 40001, 20001      # more rows than 38,912 and 19,456: two and four lanes stay

LAYOUTS = ([("er", TWO, ld) for ld in range(8, 33, 4)] + [("er", FOUR, ld) for ld in (36, 52, 64)] +
           [("mc", TWO, ld) for ld in (8, 20, 32)] + [("mc", FOUR, ld) for ld in (36, 52, 64)] +
           [("er", 301, ld) for ld in (84, 96, 100, 112)])


@pytest.fixture(scope="module")
def instances():
    cache = {}

    def get(kind, rows):
        if (kind, rows) not in cache:
            if kind == "er":
                inst = I.maxcut_er(rows, 3.0, seed=1)
            else:            # `rows` one-entry constraints off the diagonal
                inst = I.matrix_completion(500, 401, 2, rows, seed=1)
            cache[kind, rows] = (inst, SDP.from_instance(inst))
        return cache[kind, rows]
    return get


@pytest.mark.parametrize("kind,rows,ld", LAYOUTS)
def test_fp64_operators(cuda, instances, kind, rows, ld):
    torch = cuda
    inst, sdp = instances(kind, rows)
    assert (sdp.m if kind == "mc" else sdp.n) == rows
    r = ld - 1
    rng = np.random.default_rng(ld)
    U, V = rng.standard_normal((2, sdp.n, r)) / np.sqrt(r)
    w = rng.standard_normal(sdp.m)

    def dev(X):
        out = torch.zeros((sdp.n, ld), dtype=torch.float64, device="cuda")
        out[:, :r] = torch.as_tensor(X)
        return out

    dU, dV, dw = dev(U), dev(V), torch.as_tensor(w, device="cuda")
    q = torch.full((sdp.m,), np.nan, dtype=torch.float64, device="cuda")
    H = torch.full((sdp.n, ld), np.nan, dtype=torch.float64, device="cuda")
    S = torch.full((sdp.n, ld), np.nan, dtype=torch.float64, device="cuda")
    p = L.Problem(inst)
    assert L.lorads_op_sddmm(p.handle, L.LORADS_PREC_FP64, r, ld, dU, dV, q) == 0
    assert L.lorads_op_hessian(p.handle, L.LORADS_PREC_FP64, r, ld, 7.0, 1.25, dV, dU, H) == 0
    assert L.lorads_op_spmm(p.handle, L.LORADS_PREC_FP64, r, ld, dw, 0.75, dV, S) == 0
    torch.cuda.synchronize()
    p.close()
    for got, want in ((q.cpu().numpy(), sdp.A_of(U, V)),
                      (H.cpu().numpy()[:, :r], OL.hessian_apply(sdp, V, U, 7.0, 1.25)),
                      (S.cpu().numpy()[:, :r], sdp.At_times(w, V) - sdp.C_times(V) + 0.75 * V)):
        assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
    assert np.all(H.cpu().numpy()[:, r:] == 0.0) and np.all(S.cpu().numpy()[:, r:] == 0.0)


@pytest.mark.parametrize("rows,r", [(TWO, 9), (301, 9), (301, 40), (TWO, 20), (117001, 7)])
def test_fp32_product_with_diagonal_constraints(cuda, instances, rows, r):
    """Rows of 1 to some 12 entries of C, eight a round with few rows and four with many."""
    torch = cuda
    inst, sdp = instances("er", rows)
    ld = (r + 3) // 4 * 4
    rng = np.random.default_rng(r)
    V = (rng.standard_normal((sdp.n, r)) / np.sqrt(r)).astype(np.float32).astype(np.float64)
    w = rng.standard_normal(sdp.m)
    dV = torch.zeros((sdp.n, ld), dtype=torch.float32, device="cuda")
    dV[:, :r] = torch.as_tensor(V)
    S = torch.full_like(dV, float("nan"))
    p = L.Problem(inst)
    assert L.lorads_op_spmm(p.handle, L.LORADS_PREC_MIXED, r, ld, torch.as_tensor(w, device="cuda"),
                            0.75, dV, S) == 0
    got = S.cpu().numpy()
    p.close()
    want = sdp.At_times(w, V) - sdp.C_times(V) + 0.75 * V
    # at most some 20 terms an element, of at most its scale each: 32 roundings
    assert np.abs(got[:, :r] - want).max() <= 32 * 2.0 ** -24 * np.abs(want).max()
    assert np.all(got[:, r:] == 0.0)
