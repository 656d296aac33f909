"""The measured DRAM traffic that bench.py reports is dropped as soon as any source of the stage's arithmetic changes."""
import os
import shutil

import bench
from paper_1904_10070_gb300 import build


def test_stamp_covers_every_source_of_the_stage(tmp_path, monkeypatch):
    src = tmp_path / "csrc"
    shutil.copytree(build.CSRC, src)
    monkeypatch.setattr(build, "CSRC", str(src))
    note = tmp_path / "traffic.md"
    note.write_text(f"- stage_source_sha256_16: `{build.stage_tag()}`\n- dram_bytes_per_launch: `123.0`\n")
    monkeypatch.setattr(bench, "TRAFFIC_FILE", str(note))
    assert bench._traffic_per_launch() == 123.0
    for name in ("vlb_stage.cu", "vlb_node.cuh", "vlb_internal.cuh"):
        path = os.path.join(src, name)
        before = open(path).read()
        with open(path, "a") as f:
            f.write("\n")
        assert bench._traffic_per_launch() is None, name
        with open(path, "w") as f:
            f.write(before)
