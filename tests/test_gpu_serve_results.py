"""Served results without host memory (needs a GPU): the step that would return
them reports FABM_ENOMEM, the finished requests wait, and later steps neither run
them on nor lose them.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("split", 1e-6)])
def test_finished_requests_wait_for_host_memory(gpu_lib, precision, tol):
    jobs = [("linear", 1, (1.0,), 1), ("linear", 1, (1.0,), 32), ("duffing", 2, (0.1, 1.2, 0.7), 32),
            ("lorenz", 3, (10.0, 28.0, 8 / 3), 600)]
    y0 = [1.0 + 0.1 * np.arange(d) for _, d, _, _ in jobs]
    with gpu_lib.Server(1 << 30, precision=precision) as srv:
        tickets = [srv.submit(r, d, 0.9, 1e-3, n, y, p) for (r, d, p, n), y in zip(jobs, y0)]
        srv.step()  # admission; three of the four end with the next step
        try:
            for _ in range(40):  # more steps than the short requests have rows
                gpu_lib.fabm_inject_alloc_failures(1)
                with pytest.raises(gpu_lib.FabmError) as e:
                    srv.step()
                assert e.value.status == gpu_lib.FABM_ENOMEM
                assert srv.poll(tickets[0]) == gpu_lib.FABM_REQ_RUNNING
        finally:
            gpu_lib.fabm_inject_alloc_failures(0)
        srv.step()
        assert all(srv.poll(t) == gpu_lib.FABM_REQ_DONE for t in tickets)
        for (r, d, p, n), y, t in zip(jobs, y0, tickets):
            ref = oracle.solve(r, 0.9, 1e-3, n, y, params=p)
            assert np.max(np.abs(srv.result(t) - ref) / np.max(np.abs(ref), axis=0)) <= tol
