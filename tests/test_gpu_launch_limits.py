"""Solvers on several threads whose launches of one kernel differ in shared
memory (needs a GPU): the limit set on a kernel is process-wide, so it has to be
the same for every launch.  Results are those of the solver on its own."""
import threading

import numpy as np
import pytest

from fabm_workloads import lorenz_long

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,sizes", [("fp64", [(1, 700), (30, 300), (90, 200)]),
                                             ("split", [(1, 700), (60, 300)])])
def test_threads_with_launches_of_different_size(gpu_lib, precision, sizes):
    def solve(w):
        with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params, precision=precision) as s:
            return s.solve_batch(w.y0)

    work = [lorenz_long(B, N) for B, N in sizes]
    ref = [solve(w) for w in work]
    errors = []

    def run(w, r):
        try:
            for _ in range(8):  # a new solver prepares every launch again
                if not np.array_equal(solve(w), r):
                    errors.append("results differ")
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            errors.append(repr(e))

    threads = [threading.Thread(target=run, args=a) for a in zip(work, ref)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    assert not errors, errors[:3]
