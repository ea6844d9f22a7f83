"""The one-CTA FP64 kernel by name (grid = 1), and the library's own choice beside it: FP64 solves of these
sizes leave one CTA by default (test_geometry_rule.py), batches and grid = 1 run on it.

The steps of Algorithm 1 are compared one at a time, each from the oracle's own iterate: over whole solves
the comparison would show rounding instead.  Phase I amplifies it (the oracle on the theta SDP of n = 80
moves by 4e-2 when the constraints are only given in another order), and so does a step whose CG runs long
(the completion with n = 40 and 200 samples below takes 80 CG iterations a step; the oracle moves by
up to 8e-7 in one step when its input moves by one ulp)."""
import numpy as np
import pytest

import oracle.lorads as OL
from oracle import SDP, Params
from paper_2403_09133_gb300 import instances as I
from paper_2403_09133_gb300 import lorads as L

pytestmark = pytest.mark.gpu


def _theta(n):
    return I.lovasz_theta(n, I.erdos_renyi_edges(n, 3 * n, np.random.default_rng(1)))


STEPS = {
    "mc60": lambda: I.matrix_completion(30, 30, 2, 500, seed=3),
    "theta80": lambda: _theta(80),
    "er300": lambda: I.maxcut_er(300, 6.0, seed=3),
    "mc40": lambda: I.matrix_completion(20, 20, 2, 200, seed=1),
}


@pytest.mark.parametrize("case", list(STEPS))
@pytest.mark.parametrize("geometry", ["one", "default", "all"])
def test_single_steps_follow_the_oracle(cuda, case, geometry):
    sms = cuda.cuda.get_device_properties(0).multi_processor_count
    grid = {"one": 1, "default": 0, "all": sms}[geometry]
    inst = STEPS[case]()
    sdp = SDP.from_instance(inst)
    prm = OL.resolve_auto(sdp, Params())
    ph1 = OL.lralm(sdp, OL.initial_factor(sdp, OL.initial_rank(sdp.m, sdp.n, prm), prm.seed), prm)
    st = OL.AdmmState(U=ph1["U"].copy(), V=ph1["U"].copy(), lam=ph1["lam"].copy(),
                      rho=min(prm.h * ph1["sigma"], prm.rho_max))
    gamma = OL.penalty_gamma(sdp, prm)
    p = L.Problem(inst)
    for k in range(6):
        start = dict(n=inst.n, m=inst.m, phase=2, admm_iters=k, next_dual_test=10 ** 6, cg_iters=0,
                     hessian_applies=0, alm_outer=0, lbfgs_iters=0, rank_growths=0, reserved=0,
                     rho=st.rho, gamma=gamma, sigma=1.0, prev_d_infeas=np.nan, U=st.U, V=st.V,
                     lam=st.lam)
        G = OL.subproblem_rhs(sdp, st.V, st.lam, st.rho, gamma)
        R0 = np.linalg.norm(G - OL.hessian_apply(sdp, st.V, st.V, st.rho, gamma))
        info = OL.admm_iteration(sdp, st, prm)
        p.set_state(start)
        res = p.solve(precision=L.LORADS_PREC_FP64, phase1=0, max_admm_iter=k + 1, tol=1e-12,
                      polish=0, grid=grid)
        got = p.get_state()
        assert res["admm_iters"] == k + 1
        rel = {x: np.linalg.norm(got[x] - y) / np.linalg.norm(y)
               for x, y in (("U", st.U), ("V", st.V), ("lam", st.lam))}
        if case == "mc40":
            # both CGs stop at 1e-3 ||R_0|| on a matrix >= gamma I, so each is within
            # 1e-3 ||R_0|| / gamma of the subproblem's solution, wherever rounding takes it
            assert np.linalg.norm(got["U"] - st.U) <= 2e-3 * R0 / gamma
            assert abs(res["cg_iters"] - info["cg_u"] - info["cg_v"]) <= 16
        else:
            # the oracle moves by at most 2e-13 when its input moves by one ulp; sums of up to
            # 240 terms in another order move the input by some ten ulp
            assert max(rel.values()) <= 1e-11, rel
            assert res["cg_iters"] == info["cg_u"] + info["cg_v"]
    p.close()


def test_completion_repeats_and_recovers(cuda):
    """A whole solve of a general problem on one CTA (r = 9, ld = 12) repeats itself bit for bit and ends
    where the library's own choice does."""
    inst = I.matrix_completion(30, 30, 2, 500, seed=3)
    want = 2.0 * np.linalg.svd(inst.mc_P @ inst.mc_Q.T, compute_uv=False).sum()
    out = []
    for grid in (1, 1, 0):
        p = L.Problem(inst)
        res = p.solve(precision=L.LORADS_PREC_FP64, switch_tol=1e-3, h=5.0, tol=1e-9,
                      max_admm_iter=3000, grid=grid)
        out.append((res, p.solution()))
        p.close()
        assert abs(res["objective"] - want) <= 1e-7 * want
    (a, sa), (b, sb), _ = out
    assert a["admm_iters"] == b["admm_iters"] and a["cg_iters"] == b["cg_iters"]
    assert np.array_equal(sa["U_hat"], sb["U_hat"]) and np.array_equal(sa["y"], sb["y"])


@pytest.mark.parametrize("make", [lambda: I.matrix_completion(60, 60, 3, 1200, seed=4),
                                  lambda: I.matrix_completion(200, 200, 2, 8000, seed=3)])
def test_general_scopes_agree(cuda, make):
    """Three iterations on one CTA, on two, on the library's choice: the same CG iterations and
    objective, and the one-CTA solve repeats itself."""
    p = L.Problem(make())
    one, again, two, own = [p.solve(precision=L.LORADS_PREC_FP64, max_admm_iter=3, grid=g)
                            for g in (1, 1, 2, 0)]
    p.close()
    assert one["objective"] == again["objective"] and one["cg_iters"] == again["cg_iters"]
    for other in (two, own):
        assert abs(one["cg_iters"] - other["cg_iters"]) <= 3
        assert abs(one["objective"] - other["objective"]) <= 1e-9 * abs(one["objective"])


@pytest.mark.parametrize("case", ["er500", "mc30"])
def test_resume_on_one_cta(cuda, case):
    """A checkpoint at a multiple of 32 iterations continues on one CTA bit for bit."""
    inst = I.workload_er500() if case == "er500" else I.matrix_completion(30, 30, 2, 500, seed=3)
    kw = dict(precision=L.LORADS_PREC_FP64, tol=1e-12, grid=1)
    if case == "mc30":
        kw["h"] = 5.0
    p = L.Problem(inst)
    p.solve(max_admm_iter=96, **kw)
    ref = p.get_state()
    p.solve(max_admm_iter=64, **kw)
    st = p.get_state()
    p.close()
    q = L.Problem(inst)
    q.set_state(st)
    q.solve(max_admm_iter=96, phase1=0, **kw)
    got = q.get_state()
    q.close()
    assert ref["admm_iters"] == got["admm_iters"] == 96
    for x in ("U", "V", "lam"):
        assert np.array_equal(got[x], ref[x])


def test_static_solve_on_one_cta(cuda):
    torch = cuda
    inst = I.lovasz_theta(60, I.cycle_edges(60))
    p = L.Problem(inst)
    prm = p.params(precision=L.LORADS_PREC_FP64, max_admm_iter=200, grid=1)
    ref = L.lorads_solve(p.handle, prm)
    sol = p.solution()
    U = torch.zeros((inst.n, 64), dtype=torch.float64, device="cuda")
    y = torch.zeros(inst.m, dtype=torch.float64, device="cuda")
    got = L.lorads_solve_static(p.handle, prm, U, 64, y)
    torch.cuda.synchronize()
    p.close()
    assert got.status == ref.status and got.admm_iters == ref.admm_iters
    assert np.array_equal(U.cpu().numpy()[:, :sol["rank"]], sol["U_hat"])
    assert np.array_equal(y.cpu().numpy(), sol["y"])
