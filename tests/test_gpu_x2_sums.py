"""GPU tests of the double-double history sums' chunks (needs a GPU).

Sums that carry about 100 bits before they are rounded once to double are the
same double for any split into chunks, tiles and warps (they differ at 2^-97 of
the sum, so a rounding changes with a probability of about 2^-40 per sum), and
powers of two pass through every operation exactly.  Both are asked bit for
bit; the parity with the oracle is tested elsewhere.
"""
import numpy as np
import pytest

from fabm_workloads import duffing_sweep

pytestmark = pytest.mark.gpu


def solve(gpu_lib, alpha, N, y0, rhs="linear", params=(1.0,)):
    with gpu_lib.Solver(rhs, y0.shape[1], alpha, 1e-2, N, params, precision="fp64x2") as s:
        return s.solve_batch(y0)


# columns of a CTA full and ragged, chunks of one tile and of several, steps on SMs
# of their own (up to 16 trajectories) and not
@pytest.mark.parametrize("B,dim,N", [(2, 1, 700), (5, 1, 97), (1, 3, 4200), (16, 2, 1500), (17, 2, 1500),
                                     (61, 3, 1300), (1300, 1, 2500)])
@pytest.mark.parametrize("orders", [1, 2])
def test_sums_do_not_depend_on_the_split(gpu_lib, B, dim, N, orders):
    alpha = 0.7 if orders == 1 or dim == 1 else [0.7 + 0.1 * i for i in range(dim)]
    y0 = np.linspace(1.0, 2.0, B * dim).reshape(B, dim)
    got = solve(gpu_lib, alpha, N, y0)
    for b in {0, B // 2, B - 1}:
        wide = np.repeat(y0[b : b + 1], 40, axis=0)  # other chunks than in either
        assert np.array_equal(got[b], solve(gpu_lib, alpha, N, y0[b : b + 1])[0])
        assert np.array_equal(got[b], solve(gpu_lib, alpha, N, wide)[23])


@pytest.mark.parametrize("k", [-900, -300, 300, 900])
@pytest.mark.parametrize("B", [1, 40])
def test_scaled_by_a_power_of_two(gpu_lib, k, B):
    y0 = np.linspace(1.0, 2.0, B)[:, None]
    ref = solve(gpu_lib, 0.6, 800, y0)
    assert np.array_equal(solve(gpu_lib, 0.6, 800, np.ldexp(y0, k)), np.ldexp(ref, k))


def test_forcing_rows(gpu_lib):
    """The time-only part of f, computed a block ahead, in the last partial block
    and for trajectories of uneven length."""
    w = duffing_sweep(B=20, N=1203)
    ne = np.full(w.B, w.N, dtype=np.int64)
    ne[3], ne[7] = 1, 640
    with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params, precision="fp64x2") as s:
        got = s.solve_batch(w.y0, traj_params=w.traj_params, N_each=ne)
        for b in (0, 3, 7, 19):
            one = s.solve_batch(w.y0[b : b + 1], traj_params=w.traj_params[b : b + 1], N_each=ne[b : b + 1])
            assert np.array_equal(got[b, : ne[b] + 1], one[0, : ne[b] + 1])
