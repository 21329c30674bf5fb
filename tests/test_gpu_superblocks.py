"""GPU parity of the FP64 superblock schedule (needs a GPU): one cluster of
CTAs per trajectory and superblock of n targets, the far history by transforms
of the segments of n points.

The bar is the FP64 one, 1e-12 of the solution scale against the oracle.  Both
sum the same N products per step in double; the transforms' error is a few
units of 2^-53 of the largest term times log2(2n) <= 11, so sums of up to 10^4
terms stay below 1e-13 of the scale.
"""
import numpy as np
import pytest

import oracle
from fabm_workloads import duffing_sweep, lorenz_long, ml_scalar

pytestmark = pytest.mark.gpu
TOL_FP64 = 1e-12


def rel_err(got, ref):
    ref = np.asarray(ref)
    scale = np.max(np.abs(ref), axis=-2, keepdims=True)
    scale = np.where(scale == 0, 1.0, scale)
    return float(np.max(np.abs(np.asarray(got) - ref) / scale))


@pytest.mark.parametrize("N", [511, 512, 513, 1024, 1025, 1536, 1537, 2063])
def test_superblock_edges_scalar(gpu_lib, parity, N):
    w = ml_scalar(N)
    with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params) as s:
        got = s.solve(w.y0[0])
    parity(rel_err(got, oracle.solve(w.rhs, w.alpha, w.h, w.N, w.y0[0], params=w.params)), TOL_FP64)


# one batch size per cluster size, and one past the last
@pytest.mark.parametrize("B,N", [(1, 3500), (7, 3200), (8, 1700), (13, 1600), (14, 1601), (15, 1100),
                                 (16, 1569), (28, 1600), (29, 800), (46, 801), (47, 401), (76, 450),
                                 (77, 450), (200, 390)])
def test_cluster_sizes(gpu_lib, parity, B, N):
    w = lorenz_long(B, N)
    ne = np.full(B, N, dtype=np.int64)
    ne[B // 2] = N // 2 + 1
    with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params) as s:
        got = s.solve_batch(w.y0, N_each=ne)
    idx = np.unique([0, B // 2, B - 1])
    ref = oracle.solve_batch(w.rhs, w.alpha, w.h, N, w.y0[idx], params=w.params, N_each=ne[idx])
    for j, b in enumerate(idx):
        parity(rel_err(got[b, : ne[b] + 1], ref[j, : ne[b] + 1]), TOL_FP64, f"traj{b}")


@pytest.mark.parametrize("rhs,dim,alpha,params,B,N", [
    ("duffing", 2, 0.95, (0.1, 1.2, 0.7), 1, 3100), ("lcr", 2, [0.9, 0.8], (1.015, 0.55, -1.02, -0.58, 0.1), 9, 1700),
    ("linear", 4, 0.7, (1.0,), 1, 3100), ("linear", 4, [0.6, 0.7, 0.8, 0.9], (1.0,), 1, 1700),
    ("const", 3, 0.8, (1.5,), 60, 700), ("time", 2, 0.6, (), 20, 1700), ("linear", 2, 1.5, (1.0,), 5, 2300)])
def test_systems_and_orders(gpu_lib, parity, rhs, dim, alpha, params, B, N):
    y0 = 0.3 + np.linspace(-0.2, 0.2, B * dim).reshape(B, dim)
    y1 = None if np.max(alpha) <= 1 else np.full((B, dim), 0.25)
    with gpu_lib.Solver(rhs, dim, alpha, 1e-3, N, params) as s:
        got = s.solve_batch(y0, y1=y1)
    ref = oracle.solve_batch(rhs, alpha, 1e-3, N, y0, params=params, y1=y1)
    parity(rel_err(got, ref), TOL_FP64)


def test_values_near_overflow(gpu_lib):
    """Values above 2^900 (stored scaled in the spectra) beside ordinary ones:
    scaling y0 of the linear system by a power of two scales the solution."""
    w = ml_scalar(4000)
    big = 2.0 ** 1000
    with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params) as s:
        y = s.solve_batch([[1.0], [big], [1.0]])
    np.testing.assert_allclose(y[1] / big, y[0], rtol=1e-13)
    assert np.array_equal(y[0], y[2])


def test_nonfinite_trajectory_leaves_the_others_alone(gpu_lib):
    N = 2500
    tp = np.array([[1.0], [-500.0], [1.0]])
    with gpu_lib.Solver("linear", 1, 0.9, 0.01, N, [1.0]) as s:
        out = np.full((3, N + 1, 1), np.nan)
        with pytest.raises(gpu_lib.FabmError) as e:
            s.solve_batch(np.ones((3, 1)), traj_params=tp, out=out)
        assert e.value.status == gpu_lib.FABM_ENONFINITE and "trajectory 1" in str(e.value)
        ok = s.solve_batch(np.ones((3, 1)))
    assert np.array_equal(out[0], ok[0]) and np.array_equal(out[2], ok[2])


def test_wait_limit_is_reported_and_the_solver_recovers(gpu_lib, parity):
    w = lorenz_long(3, 2500)
    with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params) as s:
        s.set_wait_limit(16)
        with pytest.raises(gpu_lib.FabmError) as e:
            s.solve_batch(w.y0)
        assert e.value.status == gpu_lib.FABM_ETIMEOUT
        s.set_wait_limit(0)
        got = s.solve_batch(w.y0)
    parity(rel_err(got, oracle.solve_batch(w.rhs, w.alpha, w.h, w.N, w.y0, params=w.params)), TOL_FP64)


def test_no_room_for_spectra_falls_back_to_the_block_schedule(gpu_lib, parity):
    w = duffing_sweep(3, 4000)
    with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params) as s:
        s.solve_batch(w.y0, traj_params=w.traj_params, N_each=[100, 100, 100])  # no far superblock
        gpu_lib.fabm_inject_alloc_failures(1)
        try:
            got = s.solve_batch(w.y0, traj_params=w.traj_params)
        finally:
            gpu_lib.fabm_inject_alloc_failures(0)
        assert s.last_launch_count > 200  # one launch per kernel and block of 32
        again = s.solve_batch(w.y0, traj_params=w.traj_params)
        assert s.last_launch_count < 50
    ref = oracle.solve_batch(w.rhs, w.alpha, w.h, w.N, w.y0, params=w.params, traj_params=w.traj_params)
    parity(rel_err(got, ref), TOL_FP64, "blocks")
    parity(rel_err(again, ref), TOL_FP64, "superblocks")


def test_streamed_output_is_the_same(gpu_lib):
    """A pinned host output of 64 MB or more is copied superblock by superblock."""
    torch = pytest.importorskip("torch")
    w = lorenz_long(80, 40000)
    dev = torch.empty((w.B, w.N + 1, 3), dtype=torch.float64, device="cuda")
    pin = torch.empty((w.B, w.N + 1, 3), dtype=torch.float64, pin_memory=True)
    with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params) as s:
        s.solve_batch(w.y0, out=dev)
        s.solve_batch(w.y0, out=pin)
    assert torch.equal(dev.cpu(), pin)
