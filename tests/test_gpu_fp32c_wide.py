"""Compensated-fp32 history of batches too wide for SMs of its own (needs a GPU):
one chunk per CTA, beside the recurrence on the same SMs.  Ragged column groups,
one order and several, with and without forcing, at the split bar.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
TOL_SPLIT = 1e-6


def rel_err(got, ref):
    scale = np.max(np.abs(ref), axis=-2, keepdims=True)
    return float(np.max(np.abs(got - ref) / np.where(scale == 0, 1.0, scale)))


@pytest.mark.parametrize("rhs,dim,alpha,h,params,B,N", [
    ("lcr", 2, [0.9, 0.8], 1e-2, (1.015, 0.55, -1.02, -0.58, 0.1), 201, 900),
    ("lcr", 2, 0.9, 1e-2, (1.015, 0.55, -1.02, -0.58, 0.1), 203, 1100),
    ("lorenz", 3, 0.98, 5e-4, (10.0, 28.0, 8 / 3), 171, 777),
    ("linear", 1, 0.8, 1e-3, (1.0,), 1301, 650), ("manufactured", 1, 0.8, 1e-3, (0.5, 1.0, 2.0), 303, 1300)])
def test_wide_batches(gpu_lib, parity, rhs, dim, alpha, h, params, B, N):
    y0 = 0.5 + np.linspace(-0.2, 0.2, B * dim).reshape(B, dim)
    ne = np.full(B, N, dtype=np.int64)
    ne[B // 2] = N // 2 + 1
    with gpu_lib.Solver(rhs, dim, alpha, h, N, params, precision="split", history="fp32c") as s:
        got = s.solve_batch(y0, N_each=ne)
        assert s.last_history_kernel == "fp32c"
    idx = np.array([0, B // 2, B - 1])
    ref = oracle.solve_batch(rhs, alpha, h, N, y0[idx], params=params, N_each=ne[idx])
    for j, b in enumerate(idx):
        parity(rel_err(got[b, : ne[b] + 1], ref[j, : ne[b] + 1]), TOL_SPLIT, f"traj{b}")
