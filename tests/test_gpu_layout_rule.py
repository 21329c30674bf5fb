"""Recurrence layout of one-component systems on the tensor path (needs a GPU):
the automatic choice on both sides of its limits gives the bits of either layout
(few segments, so that every layout has the same chunks), by the launches of one.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rhs,params,B,layout", [
    ("linear", (1.0,), 64, "targets"), ("linear", (1.0,), 1024, "targets"), ("linear", (1.0,), 1025, "columns"),
    ("manufactured", (0.5, 1.0, 2.0), 384, "targets"), ("manufactured", (0.5, 1.0, 2.0), 385, "columns")])
def test_automatic_layout(gpu_lib, rhs, params, B, layout):
    N = 300
    y0 = np.linspace(0.5, 1.5, B)[:, None]
    got, launches = {}, {}
    for rec in ("auto", "targets", "columns"):
        with gpu_lib.Solver(rhs, 1, 0.9, 1e-3, N, params, precision="split", history="tensor",
                            recurrence=rec) as s:
            got[rec] = s.solve_batch(y0)
            launches[rec] = s.last_launch_count
    assert launches["targets"] != launches["columns"]
    assert launches["auto"] == launches[layout]
    assert np.array_equal(got["auto"], got["targets"]) and np.array_equal(got["auto"], got["columns"])
