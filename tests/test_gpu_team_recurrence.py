"""The lane-per-column recurrence of the tensor path (teams of warps) against the
lane-per-target one (needs a GPU).

Both run the same float-float operations of a column in the same order, on the
same history partials while a block has few far segments, so their results are
equal bit for bit: every system and dimension, teams with idle lanes, a partial
last team, lengths around the edges of blocks (64) and sub-blocks (8), uneven
lengths.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rhs,dim,alpha,params,B", [
    ("const", 4, 0.7, (1.5,), 17), ("time", 3, 0.8, (), 25), ("linear", 1, 0.6, (1.2,), 65),
    ("linear", 1, 1.5, (1.2,), 65), ("linear", 3, 0.95, (0.7,), 31), ("lorenz", 3, 0.96, (10.0, 28.0, 8 / 3), 43),
    ("duffing", 2, 0.95, (0.1, 1.2, 0.9), 33), ("duffing", 2, 1.3, (0.1, 1.2, 0.9), 33),
    ("manufactured", 1, 0.8, (1.8, 1.2, 2.0), 70), ("lcr", 2, 0.9, (1.015, 0.55, -1.02, -0.58, 0.15), 40)])
@pytest.mark.parametrize("N", [1, 7, 8, 9, 63, 64, 65, 200])
def test_columns_equal_targets_bitwise(gpu_lib, rhs, dim, alpha, params, B, N):
    y0 = 1.3 * np.sin(np.arange(B * dim) + 0.4).reshape(B, dim)
    y1 = None if alpha <= 1 else 0.2 * y0
    ne = np.full(B, N, dtype=np.int64)
    ne[B // 2] = max(1, N - 5)
    out = {}
    for layout in ("columns", "targets"):
        with gpu_lib.Solver(rhs, dim, alpha, 1e-2, N, params, precision="split", history="tensor",
                            recurrence=layout) as s:
            out[layout] = s.solve_batch(y0, y1=y1, N_each=ne)
    assert np.array_equal(out["columns"], out["targets"], equal_nan=True)
