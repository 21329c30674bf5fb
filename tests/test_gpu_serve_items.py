"""Served history with one item per warp and with four (needs a GPU): a request's
result does not depend on how many items a step has, bit for bit, whatever the
lengths of the chunks (multiples of 16 and of 512 points, and rests).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rhs,dim,params", [("linear", 1, (1.0,)), ("duffing", 2, (0.1, 1.2, 0.7)),
                                            ("lorenz", 3, (10.0, 28.0, 8 / 3))])
def test_a_crowd_leaves_results_bit_for_bit(gpu_lib, rhs, dim, params):
    lengths = [40, 96, 1100, 1575, 2600]
    y0 = 1.0 + 0.1 * np.arange(dim)

    def serve(crowd):
        with gpu_lib.Server(32 << 30, precision="split", max_slots=4096) as srv:
            tickets = [srv.submit(rhs, dim, 0.9, 1e-3, n, y0, params) for n in lengths]
            for _ in range(crowd):  # 2100 requests of 3 columns: over 6144 items from the second block on
                srv.submit("lorenz", 3, 0.8, 1e-3, 2600, [1.0, 1.0, 1.0], (10.0, 28.0, 8 / 3))
            return [srv.wait(t) for t in tickets]

    for alone, mixed in zip(serve(0), serve(2100)):
        assert np.array_equal(alone, mixed)
