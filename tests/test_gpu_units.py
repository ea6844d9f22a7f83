"""The FP64 operators' unit layout (16-byte units dealt to 2-16 lanes per row) at the edges of its
ranges -- one unit per row, one more than a lane's eight, the widest rows, row counts that leave
part of a warp without rows, constraints of several entries -- against the oracle's definitions
(FP64: 1e-12 of the terms' size, rounding ~1e-16 times the square root of up to 512 terms); and the
launch geometry of FP64 solves on both sides of its rule."""
import numpy as np
import pytest

from oracle import SDP
import oracle.lorads as OL
from paper_2403_09133_gb300 import instances as I
from paper_2403_09133_gb300 import lorads as L

pytestmark = pytest.mark.gpu

INSTANCES = {
    "er65": lambda: I.maxcut_er(65, 5.0, seed=3),
    "mc73": lambda: I.matrix_completion(40, 33, 2, 500, seed=2),
    "theta13": lambda: I.lovasz_theta(13, I.cycle_edges(13)),
}


@pytest.mark.parametrize("name", list(INSTANCES))
@pytest.mark.parametrize("r", [1, 4, 30, 32, 33, 66, 127, 132, 256])
def test_fp64_operators(cuda, name, r):
    torch = cuda
    inst = INSTANCES[name]()
    sdp = SDP.from_instance(inst)
    ld = (r + 3) // 4 * 4
    rng = np.random.default_rng(r)
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
        assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
    assert np.all(H.cpu().numpy()[:, r:] == 0.0) and np.all(S.cpu().numpy()[:, r:] == 0.0)


@pytest.mark.parametrize("make,whole", [
    (lambda: I.maxcut_er(255, 5.0, seed=1), False), (lambda: I.maxcut_er(256, 5.0, seed=1), True),
    (lambda: I.matrix_completion(20, 19, 2, 200, seed=1), False),
    (lambda: I.matrix_completion(20, 20, 2, 200, seed=1), True)])
def test_fp64_geometry(cuda, make, whole):
    """The default geometry repeats the explicit one bit for bit."""
    inst = make()
    sms = cuda.cuda.get_device_properties(0).multi_processor_count
    out = []
    for kw in (dict(), dict(grid=sms if whole else 1)):
        p = L.Problem(inst)
        p.solve(precision=L.LORADS_PREC_FP64, max_admm_iter=20, **kw)
        out.append(p.solution())
        p.close()
    a, b = out
    assert np.array_equal(a["U_hat"], b["U_hat"]) and np.array_equal(a["y"], b["y"])
