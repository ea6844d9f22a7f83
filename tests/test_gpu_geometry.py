"""Launch geometry of FP64 solves on the GPU."""
import numpy as np
import pytest

from paper_2403_09133_gb300 import instances as I
from paper_2403_09133_gb300 import lorads as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [352, 384])
@pytest.mark.parametrize("make", [lambda: I.maxcut_er(300, 6.0, seed=3),
                                  lambda: I.matrix_completion(30, 30, 2, 500, seed=3)])
def test_cta_sizes_of_the_one_cta_kernel_solve_by_default(cuda, make, threads):
    """grid = 0 with a CTA size that only the one-CTA kernel takes (384 is what an autotuned batch
    usually reports) runs there, in lorads_solve and in lorads_solve_static."""
    inst = make()
    p = L.Problem(inst)
    kw = dict(precision=L.LORADS_PREC_FP64, max_admm_iter=10, threads=threads)
    got = p.solve(**kw)
    assert got["status"] == L.LORADS_ERR_MAXITER, L.lorads_status_string(got["status"])
    U = p.solution()["U_hat"]
    one = p.solve(grid=1, **kw)
    assert one["objective"] == got["objective"]
    assert np.array_equal(p.solution()["U_hat"], U)
    st = L.lorads_solve_static(p.handle, p.params(**kw))
    p.close()
    assert st.status == L.LORADS_ERR_MAXITER and st.objective == got["objective"]
