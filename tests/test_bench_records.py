"""Which ncu record bench.py applies to the launches it times (no GPU).

The counters of another launch give wrong bounds: a step that forms no residual runs
other kernels of the same sources, and another layout has another share of halo rows.
"""
import json

import pytest

import bench

LAYOUT = {"fused_threads": 128, "fused_rows": 128, "schedule": "grid"}


@pytest.mark.parametrize("change,found", [
    ({}, True),
    ({"residual": False}, False),
    ({"residual": None}, False),
    ({"layout": {**LAYOUT, "fused_rows": 48}}, False),
    ({"layout": {**LAYOUT, "schedule": "static"}}, False),
    ({"src_digest": "0" * 16}, False),
])
def test_a_record_describes_the_timed_launch_or_is_not_used(tmp_path, change, found):
    e = {"bytes_per_lu": 86.0, "src_digest": bench.kernel_source_digest("fused"), "residual": True,
         "layout": LAYOUT, **change}
    path = tmp_path / "traffic.json"
    path.write_text(json.dumps({"fused:fp32dev:batch64": e, "fused:fp32dev": e}))
    got = bench.profile_record("fused", "fp32dev", "batch64", LAYOUT, path=str(path))
    assert (got is not None) == found
    # nor does one workload's record describe another's launches
    assert bench.profile_record("fused", "fp32dev", "sweep257", LAYOUT, path=str(path)) is None


def test_the_bench_line_states_how_the_power_law_is_evaluated():
    """The FP32 form does not evaluate every power in FP64, and the line says what it does."""
    said = {p: bench.power_law(bench.parse_args(a)) for p, a in
            {"default": [], "fp64": ["--precision", "fp64"], "opt-in": ["--power-fp32"]}.items()}
    assert said["fp64"] == "fp64" and said["opt-in"].startswith("fp32")
    assert "float pairs" in said["default"] and "rounded" in said["default"]
