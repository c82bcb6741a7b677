"""The committed DRAM traffic that bench.py reports for a step: only for the sources and
the grouping of layers that it was captured from (CPU)."""
import json
import os
import shutil

import bench
from paper_2606_29563_gb300 import synth

WL = synth.WORKLOADS["llama8b_ragged8_b256"]


def _tree(tmp_path, monkeypatch):
    for rel in ("paper_2606_29563_gb300/csrc", "include"):
        shutil.copytree(os.path.join(bench.ROOT, rel), tmp_path / rel)
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    record = {"sources_sha256": bench.sources_sha256(),
              "step": {WL.name: {"bytes_per_layer": 10.0, "layers_per_launch": 8}},
              "decode": {WL.name: {"bytes_per_launch": 7}}}
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps(record))


def test_traffic_holds_for_the_captured_grouping_only(tmp_path, monkeypatch):
    _tree(tmp_path, monkeypatch)
    assert bench.committed_step_traffic(WL, 32, 4) == 320.0
    assert bench.committed_step_traffic(WL, 8, 1) == 80.0
    assert bench.committed_step_traffic(WL, 32, 5) is None
    assert bench.committed_step_traffic(WL, 4, 1) is None
    assert bench.committed_step_traffic(synth.WORKLOADS["llama8b_l8192_b512"], 32, 4) is None
    assert bench.committed_traffic("decode", WL.name)["bytes_per_launch"] == 7


def test_any_source_file_ends_the_record(tmp_path, monkeypatch):
    _tree(tmp_path, monkeypatch)
    names = [os.path.join("paper_2606_29563_gb300/csrc", n) for n in os.listdir(tmp_path / "paper_2606_29563_gb300/csrc")]
    assert len(names) >= 9
    for rel in names + ["include/kvec.h"]:
        text = (tmp_path / rel).read_text()
        (tmp_path / rel).write_text(text + "// other\n")
        assert bench.committed_step_traffic(WL, 32, 4) is None, rel
        assert bench.committed_traffic("decode", WL.name) is None, rel
        (tmp_path / rel).write_text(text)
    assert bench.committed_step_traffic(WL, 32, 4) == 320.0
