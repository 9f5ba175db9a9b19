"""bench.py's headline roofline entry: the FP64 operator against the integer ALU (no GPU)."""
import pytest

import bench


@pytest.mark.parametrize("kind", ["stencil", "smooth"])
def test_fp64_grid_kernels_are_held_to_the_integer_alu(kind):
    n, ms = 16777216, 0.13
    e = bench.roofline_alone(kind, ms, n, "f64", 6778.7, "measured", None)
    r = bench.integer_roof(e, kind)
    assert r["bound"] == "alu" and r["kernel"] == e["kernel"] and r["traffic"] == e["traffic"]
    assert r["achieved"] == pytest.approx(bench.INT_OPS[kind] * n / (ms / 1e3) / 1e12)
    assert r["peak"] == pytest.approx(64 * 152 * 2.07e9 / 1e12) and r["frac"] == pytest.approx(r["achieved"] / r["peak"])
    assert r["frac"] < 1.0 and r["fp64_pipe"]["fp64_issue_frac"] == e["fp64_issue_frac"]
