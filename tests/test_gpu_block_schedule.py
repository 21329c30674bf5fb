"""FP64 solves block by block, every point summed directly (needs a GPU): what
fabm_set_block(32) asks for, and what superblocks without room fall back to.

From N x columns = 2^19 on, consecutive blocks' history launches run two blocks
behind on two streams; below, one block behind.  The bar is the FP64 one: both
sides add the same N products per step in double.
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


def check(parity, rhs, alpha, h, params, y0, ne, got, tp=None):
    """The first, a middle and the last trajectory against the oracle."""
    idx = np.unique([0, len(y0) // 2, len(y0) - 1])
    ref = oracle.solve_batch(rhs, alpha, h, int(ne.max()), y0[idx], params=params, N_each=ne[idx],
                             traj_params=None if tp is None else tp[idx])
    for j, b in enumerate(idx):
        parity(rel_err(got[b, : ne[b] + 1], ref[j, : ne[b] + 1]), TOL_FP64, f"traj{b}")


# an odd number of blocks, the last one partial; lag 2 (first of each pair) and lag 1
@pytest.mark.parametrize("rhs,dim,alpha,h,params,B,N", [
    ("lorenz", 3, 0.98, 5e-4, (10.0, 28.0, 8 / 3), 50, 3527), ("lorenz", 3, 0.98, 5e-4, (10.0, 28.0, 8 / 3), 3, 1511),
    ("lcr", 2, [0.9, 0.8], 1e-2, (1.015, 0.55, -1.02, -0.58, 0.1), 90, 2985),
    ("lcr", 2, [0.9, 0.8], 1e-2, (1.015, 0.55, -1.02, -0.58, 0.1), 5, 1000),
    ("linear", 1, 0.7, 1e-3, (1.0,), 131, 4007), ("linear", 4, [0.6, 0.7, 0.8, 0.9], 1e-3, (1.0,), 44, 3001)])
def test_direct_sums_in_blocks_of_32(gpu_lib, parity, rhs, dim, alpha, h, params, B, N):
    y0 = 0.5 + np.linspace(-0.2, 0.2, B * dim).reshape(B, dim)
    ne = np.full(B, N, dtype=np.int64)
    ne[B // 2] = N // 2 + 1
    if B > 3:
        ne[1], ne[2] = 1, 64
    with gpu_lib.Solver(rhs, dim, alpha, h, N, params, block=32) as s:
        got = s.solve_batch(y0, N_each=ne)
        assert s.last_launch_count > 2 * (N // 32)  # kernels of every block
        assert s.block == 32 and s.last_history_kernel == "fp64"
        gpu_lib.fabm_set_history_kernel(s.handle, "auto")
        auto = s.solve_batch(y0, N_each=ne)
        assert s.last_launch_count < N // 16  # superblocks
    check(parity, rhs, alpha, h, params, y0, ne, got)
    check(parity, rhs, alpha, h, params, y0, ne, auto)


def test_no_room_for_spectra_at_lag_two(gpu_lib, parity):
    w = lorenz_long(60, 3300)
    ne = np.full(w.B, w.N, dtype=np.int64)
    with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params) as s:
        s.solve_batch(w.y0, N_each=np.full(w.B, 100))
        gpu_lib.fabm_inject_alloc_failures(1)
        try:
            got = s.solve_batch(w.y0)
        finally:
            gpu_lib.fabm_inject_alloc_failures(0)
        assert s.last_launch_count > 200
    check(parity, w.rhs, w.alpha, w.h, w.params, w.y0, ne, got)


@pytest.mark.parametrize("B,N", [(2, 6000), (150, 2000)])
def test_autotune(gpu_lib, parity, B, N):
    """Superblocks (target 0), direct sums at four CTA targets and, where it fits,
    the persistent launch are timed; the pick stays right."""
    w = lorenz_long(B, N)
    ne = np.full(B, N, dtype=np.int64)
    with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params, block=32) as s:
        rep = s.autotune(w.y0, n_probe=500)
        assert [c for _, k, c in rep if k == gpu_lib.FABM_HIST_FP64] == [0, 152, 304, 608, 1216]
        assert (gpu_lib.FABM_HIST_FP64_PERSIST in [k for _, k, _ in rep]) == (B <= 64)
        assert all(ms > 0 for ms, _, _ in rep)
        got = s.solve_batch(w.y0)
    check(parity, w.rhs, w.alpha, w.h, w.params, w.y0, ne, got)
