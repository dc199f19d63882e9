"""The reference arm of bench.py (the FP64 oracle on the host's cores) prints
its one JSON line for every kind of workload: one camera, the pooled cameras
(the default) and the serving cameras."""
import json

import pytest

import bench


@pytest.mark.parametrize("workload", ["c1", "c2", "c4"])
def test_reference_arm_prints_its_line(workload, monkeypatch, capsys):
    monkeypatch.setenv("GMM_REFERENCE_SECONDS", "0.2")
    bench.main(["--impl", "reference", "--workload", workload, "--steps", "1", "--warmup", "3"])
    lines = capsys.readouterr().out.strip().splitlines()
    assert len(lines) == 1
    line = json.loads(lines[0])
    assert line["impl"] == "reference" and line["metric"] == bench.METRIC
    assert line["value"] > 0 and line["steps"] == 1 and line["warmup"] == 3
    assert line["config"]["workload"].startswith(workload + ":")
