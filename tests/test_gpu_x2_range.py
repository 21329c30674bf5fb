"""Double-double history sums near the end of double's range (needs a GPU).

Sums between 2^1023 and 2^1024 are finite.  A constant right-hand side scaled by a
power of two scales every sum exactly, so the solution of p = 2^1018, whose sums
pass 2^1023 from step 650 on (m^0.6 / Gamma(1.6) = 61.8 at step 800), is that of
p = 1 times 2^1018, bit for bit.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# chunks added by 32 lanes, 8 and 1 (13 chunks, and 3 at once), and a single chunk
@pytest.mark.parametrize("B", [1, 60, 400, 2000, 5000])
def test_sums_in_the_last_binade(gpu_lib, B):
    N, y0 = 800, np.zeros((B, 1))

    def solve(p0):
        with gpu_lib.Solver("const", 1, 0.6, 1e-2, N, [p0], precision="fp64x2") as s:
            return s.solve_batch(y0)

    assert np.array_equal(solve(2.0 ** 1018), np.ldexp(solve(1.0), 1018))
