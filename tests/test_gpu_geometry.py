"""Launch geometry of FP64 solves on the GPU."""
import threading
import time

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


@pytest.mark.parametrize("make", [lambda s: I.maxcut_er(256, 6.0, seed=s),
                                  lambda s: I.matrix_completion(30, 30, 2, 500, seed=3 + s)])
def test_callers_share_the_gpu(cuda, make):
    """Eight FP64 solves by as many threads, on a stream each, take little longer than one of them: the default
    geometry leaves room beside it.  (Grids over all SMs ran two at a time: 4.4 and 4.1 times.)"""
    torch = cuda
    count, iters = 8, 60
    probs = [L.Problem(make(s % 2)) for s in range(count)]
    streams = [torch.cuda.Stream() for _ in range(count)]
    prms = [p.params(precision=L.LORADS_PREC_FP64, max_admm_iter=iters, polish=0) for p in probs]

    def solve(i):
        assert L.lorads_solve(probs[i].handle, prms[i], streams[i]).status == L.LORADS_ERR_MAXITER

    def side_by_side(ids):
        best = 1e9
        for _ in range(3):
            ts = [threading.Thread(target=solve, args=(i,)) for i in ids]
            t0 = time.perf_counter()
            [t.start() for t in ts]
            [t.join() for t in ts]
            best = min(best, time.perf_counter() - t0)
        return best

    for i in range(count):
        solve(i)                           # assembles
    alone = max(side_by_side([0]), side_by_side([1]))      # the two instances
    together = side_by_side(range(count))
    for p in probs:
        p.close()
    assert together <= 2.5 * alone, (together, alone)
