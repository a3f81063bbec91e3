"""The recorded DRAM traffic of the layer kernel counts only for the sources it was taken on."""
import json
import os
import shutil

import pytest

import bench

CSRC = os.path.join("paper_2606_31160_gb300", "csrc")


@pytest.mark.parametrize("changed", [None, "attention_wide.cu", "tc_common.cuh", "common.cuh", "attention_tc.cu"])
def test_a_changed_source_voids_the_record(monkeypatch, tmp_path, changed):
    shutil.copytree(os.path.join(bench.ROOT, CSRC), tmp_path / CSRC)
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    record = {"verify_layer": {"src_sha256": bench.kernel_source_hash(), "dram_bytes_per_launch": 123}}
    (tmp_path / "profiles" / "ncu_traffic.json").write_text(json.dumps(record))
    if changed:
        with open(tmp_path / CSRC / changed, "a") as f:
            f.write("// changed\n")
    assert bench.ncu_traffic() == (None if changed else 123.0)
