"""Which kernels take the steps of short solves (needs a GPU): both sides of each
rule on lengths and batch sizes, against the oracle.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
TOL_FP64 = 1e-12
PARAMS = {"linear": (1.0,), "manufactured": (0.5, 1.0, 2.0), "duffing": (0.1, 1.2, 0.7),
          "lorenz": (10.0, 28.0, 8 / 3)}


def rel_err(got, ref):
    scale = np.max(np.abs(ref), axis=-2, keepdims=True)
    return float(np.max(np.abs(got - ref) / np.where(scale == 0, 1.0, scale)))


def solve(gpu_lib, parity, rhs, dim, precision, B, N, tol, **kw):
    y0 = 0.5 + np.linspace(-0.2, 0.2, B * dim).reshape(B, dim)
    ne = np.full(B, N, dtype=np.int64)
    ne[B // 2] = N // 2 + 1
    with gpu_lib.Solver(rhs, dim, 0.9, 1e-3, N, PARAMS[rhs], precision=precision, **kw) as s:
        got = s.solve_batch(y0, N_each=ne)
        launches = s.last_launch_count
    idx = np.array([0, B // 2, B - 1])
    ref = oracle.solve_batch(rhs, 0.9, 1e-3, N, y0[idx], params=PARAMS[rhs], N_each=ne[idx])
    for j, b in enumerate(idx):
        parity(rel_err(got[b, : ne[b] + 1], ref[j, : ne[b] + 1]), tol, f"traj{b}")
    return got, launches


# launches: initial values, then one per block or superblock, and one per forcing table
@pytest.mark.parametrize("rhs,dim,B,N,launches", [
    ("linear", 1, 511, 64, 2), ("linear", 1, 512, 64, 3), ("linear", 1, 513, 65, 2), ("linear", 1, 600, 1, 2),
    ("duffing", 2, 512, 32, 2), ("duffing", 2, 513, 33, 3), ("lorenz", 3, 600, 40, 2),
    ("manufactured", 1, 4095, 128, 3), ("manufactured", 1, 4096, 128, 7)])
def test_fp64(gpu_lib, parity, rhs, dim, B, N, launches):
    assert solve(gpu_lib, parity, rhs, dim, "fp64", B, N, TOL_FP64)[1] == launches


@pytest.mark.parametrize("rhs,dim,B,N", [("linear", 1, 4861, 200), ("manufactured", 1, 4900, 97), ("lorenz", 3, 1621, 170)])
def test_fp64x2_single_chunk(gpu_lib, parity, rhs, dim, B, N):
    """From 4861 columns on a block's history is one chunk, which writes the rounded
    sums itself; they are those of a narrow batch's chunks, bit for bit (sums of about
    100 bits before the one rounding)."""
    got, _ = solve(gpu_lib, parity, rhs, dim, "fp64x2", B, N, TOL_FP64)
    y0 = 0.5 + np.linspace(-0.2, 0.2, B * dim).reshape(B, dim)
    with gpu_lib.Solver(rhs, dim, 0.9, 1e-3, N, PARAMS[rhs], precision="fp64x2") as s:
        for b in (0, B - 1):
            assert np.array_equal(got[b], s.solve_batch(y0[b : b + 1])[0])


@pytest.mark.parametrize("alpha", [0.4, 0.8, 0.95, 1.5])
def test_error_of_blocks_against_binary128(gpu_lib, parity, alpha):
    """A value takes the points of its own block of 32 one by one, 16 on average, each
    rounded to a unit of its last place: sqrt(16 / 3) 2^-53 = 2.6e-16 for mantissas of
    one, less for larger ones.  With the 32 points of the block before taken the same way
    it would be sqrt(48 / 3) 2^-53 = 4.4e-16.  2-norms over 15 trajectories; the bar is
    the first of the two and a tenth for f, the corrector and the rest of the sums."""
    N, y0 = 60, np.linspace(0.3, 1.5, 600)[:, None]
    with gpu_lib.Solver("linear", 1, alpha, 2e-3, N, [1.0]) as s:
        got = s.solve_batch(y0)[::40]
    ref = np.stack([oracle.solve_q("linear", alpha, 2e-3, N, y, params=[1.0]) for y in y0[::40]])
    parity(float(np.linalg.norm(got - ref) / np.linalg.norm(ref)), 2.8e-16)
