"""A solver's work space and cached launch graph across solves of different
shapes and failed allocations (needs a GPU).

One solver used with several batch sizes allocates some buffers anew, and an
allocation that fails (injected on the host) makes a solve take the schedule
that needs less room.  A later solve of an earlier shape gives the same bits as
before: the same launches on the same inputs.
"""
import numpy as np
import pytest

import oracle
from fabm_workloads import duffing_sweep, lorenz_long

pytestmark = pytest.mark.gpu
TOL_FP64 = 1e-12


def rel_err(got, ref):
    scale = np.max(np.abs(ref), axis=-2, keepdims=True)
    return float(np.max(np.abs(got - ref) / np.where(scale == 0, 1.0, scale)))


def test_graph_is_recorded_again_when_the_factors_move(gpu_lib):
    """Superblocks of 512 targets need longer transforms than those of 128, so the
    factors of the first solve's graph are freed by the second solve."""
    w = duffing_sweep(256, 8192)
    with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params) as s:
        first = s.solve_batch(w.y0, traj_params=w.traj_params)
        s.set_graphs(False)
        s.solve_batch(w.y0[:1], traj_params=w.traj_params[:1])
        s.set_graphs(True)
        again = s.solve_batch(w.y0, traj_params=w.traj_params)
    assert np.array_equal(first, again)


def test_failed_allocation_of_the_factors(gpu_lib):
    """The factors for 512 targets cannot be allocated (every other buffer fits):
    that solve takes the block schedule, and the next one of the first shape
    computes its factors again."""
    w = lorenz_long(30, 4000)  # superblocks of 256 targets
    with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params) as s:
        first = s.solve_batch(w.y0)
        gpu_lib.fabm_inject_alloc_failures(1)
        try:
            s.solve_batch(w.y0[:1])
        finally:
            gpu_lib.fabm_inject_alloc_failures(0)
        assert s.last_launch_count > 200  # one launch per kernel and block of 32
        again = s.solve_batch(w.y0)
    assert np.array_equal(first, again)


def test_graph_is_recorded_again_for_another_layout(gpu_lib):
    """At nine column tiles the layouts asked for leave other numbers of SMs to the
    recurrence, so the far history has 14 chunks automatically and 15 with
    "columns", in both layouts by the same kernels."""
    w = duffing_sweep(576, 2500)

    def solver(layout):
        return gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params, precision="split", history="tensor",
                              recurrence=layout)

    with solver("columns") as s:
        want = s.solve_batch(w.y0, traj_params=w.traj_params)
    with solver("auto") as s:
        s.solve_batch(w.y0, traj_params=w.traj_params)
        gpu_lib.fabm_set_recurrence_layout(s.handle, "columns")
        got = s.solve_batch(w.y0, traj_params=w.traj_params)
    assert np.array_equal(want, got)


def test_partial_spectra_are_sized_by_their_chunks(gpu_lib):
    """A wide batch's sums over segments have one chunk: 4 KB a column, where 16
    would be 1.3 GB.  All other buffers of the solve are below 0.4 GB."""
    torch = pytest.importorskip("torch")
    B, N = 20000, 400  # superblocks of 128 targets, two of them with a far history
    out = torch.empty((B, N + 1, 1), dtype=torch.float64, device="cuda")
    with gpu_lib.Solver("linear", 1, 0.9, 1e-3, N, [1.0]) as s:
        s.solve_batch(np.ones((B, 1)), N_each=np.full(B, 10), out=out)
        free = torch.cuda.mem_get_info()[0]
        s.solve_batch(np.ones((B, 1)), out=out)
        assert s.last_launch_count < 30  # superblocks
        assert free - torch.cuda.mem_get_info()[0] < 0.5e9
    ref = oracle.solve("linear", 0.9, 1e-3, N, [1.0], params=[1.0])
    assert rel_err(out[-1].cpu().numpy(), ref) <= TOL_FP64


def test_spectra_make_way_for_what_every_schedule_needs(gpu_lib, parity):
    """The spectra of an earlier solve are on the device when the staging buffer of
    a host output cannot be allocated: they are given back and the solve goes on."""
    torch = pytest.importorskip("torch")
    w = duffing_sweep(3, 4000)
    ref = oracle.solve_batch(w.rhs, w.alpha, w.h, w.N, w.y0, params=w.params, traj_params=w.traj_params)
    with gpu_lib.Solver(w.rhs, w.dim, w.alpha, w.h, w.N, w.params) as s:
        dev = torch.empty((w.B, w.N + 1, w.dim), dtype=torch.float64, device="cuda")
        s.solve_batch(w.y0, traj_params=w.traj_params, out=dev)
        gpu_lib.fabm_inject_alloc_failures(1)
        try:
            got = s.solve_batch(w.y0, traj_params=w.traj_params)
        finally:
            gpu_lib.fabm_inject_alloc_failures(0)
    parity(rel_err(got, ref), TOL_FP64, "host")
    assert np.array_equal(got, dev.cpu().numpy())


def test_fallback_gives_the_spectra_back(gpu_lib):
    """A wider batch one of whose superblock buffers cannot grow takes the block
    schedule, whose own buffers are 0.13 GB here; the spectra of the solve before
    it (0.44 GB) do not stay beside them."""
    torch = pytest.importorskip("torch")
    N, B = 20000, 700  # 32 bytes a point and column, one column
    y0 = np.ones((B + 100, 1))
    out = torch.empty((B + 100, N + 1, 1), dtype=torch.float64, device="cuda")
    with gpu_lib.Solver("linear", 1, 0.9, 1e-3, N, [1.0]) as s:
        # the buffers of the wider batch that do not depend on the schedule
        s.solve_batch(y0, N_each=np.full(B + 100, 200), out=out)
        before = torch.cuda.mem_get_info()[0]
        s.solve_batch(y0[:B], out=out[:B])
        assert before - torch.cuda.mem_get_info()[0] > 0.4e9
        gpu_lib.fabm_inject_alloc_failures(1)
        try:
            s.solve_batch(y0, N_each=np.full(B + 100, 2000), out=out)
        finally:
            gpu_lib.fabm_inject_alloc_failures(0)
        assert s.last_launch_count > 100  # one launch per kernel and block of 32
        assert before - torch.cuda.mem_get_info()[0] < 0.3e9
    ref = oracle.solve("linear", 0.9, 1e-3, 2000, [1.0], params=[1.0])
    assert rel_err(out[-1, :2001].cpu().numpy(), ref) <= TOL_FP64
