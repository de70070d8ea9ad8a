"""The benchmark scales a committed DRAM-traffic figure only to lattices that the
captured kernel steps."""
import json
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


@pytest.mark.parametrize("shape,known", [((256, 256, 256), True), ((96, 128, 200), True), ((64, 64, 64), False),
                                         ((1, 2048, 2048), False), ((64, 1, 160), False), ((24, 300, 300), False)])
def test_traffic_of_the_marching_kernel(tmp_path, monkeypatch, shape, known):
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    monkeypatch.setattr(bench, "kernel_source_hash", lambda k: "x")
    (tmp_path / "profiles" / "dram_traffic.json").write_text(
        json.dumps({"k_step_fused/f32": {"kernel_source_sha": "x", "dram_bytes_per_cell": 300.0}}))
    want = 300.0 * shape[0] * shape[1] * shape[2] if known else None
    assert bench.ncu_traffic("k_step_fused", "f32", shape) == want
