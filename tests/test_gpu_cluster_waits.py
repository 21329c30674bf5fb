"""The cluster kernel's bounded waits run out lane by lane (needs a GPU).

With limits between a few cycles and a block of steps, some lanes of a warp get
their value and others give up, each at its own time, before the warp meets the
next barrier.  Every launch has to end: the solve is right or reports
FABM_ETIMEOUT, and the solver is right again with the default limit.
"""
import numpy as np
import pytest

import oracle
from fabm_workloads import lorenz_long

pytestmark = pytest.mark.gpu
TOL_FP64 = 1e-12


def rel_err(got, ref):
    scale = np.max(np.abs(ref), axis=-2, keepdims=True)
    return float(np.max(np.abs(got - ref) / np.where(scale == 0, 1.0, scale)))


# clusters of 16, 4 and 1 CTAs; one, three and four components
@pytest.mark.parametrize("rhs,dim,B", [("lorenz", 3, 1), ("lorenz", 3, 30), ("lorenz", 3, 80), ("linear", 1, 2),
                                       ("linear", 4, 2)])
def test_waits_that_run_out_at_any_point(gpu_lib, parity, rhs, dim, B):
    N = 1300
    if rhs == "lorenz":
        w = lorenz_long(B, N)
        alpha, h, y0, params = w.alpha, w.h, w.y0, w.params
    else:
        alpha, h, y0, params = 0.8, 1e-3, np.linspace(0.5, 1.5, B * dim).reshape(B, dim), [1.0]
    ref = oracle.solve_batch(rhs, alpha, h, N, y0[:2], params=params)
    with gpu_lib.Solver(rhs, dim, alpha, h, N, params) as s:
        for limit in (16, 100, 400, 1000, 3000, 10000, 30000):
            s.set_wait_limit(limit)
            try:
                got = s.solve_batch(y0)
            except gpu_lib.FabmError as e:
                assert e.status == gpu_lib.FABM_ETIMEOUT
            else:
                parity(rel_err(got[:2], ref), TOL_FP64, f"limit {limit}")
            s.set_wait_limit(0)
            parity(rel_err(s.solve_batch(y0)[:2], ref), TOL_FP64, f"after {limit}")
