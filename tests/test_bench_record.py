"""The benchmark reports profiler counts only for the very kernel that they were taken of."""
import json
import os
import re
import shutil

import bench


def _copy(tmp_path):
    os.makedirs(tmp_path / "profiles")
    shutil.copytree(os.path.join(bench.ROOT, "paper_1808_02638_gb300", "csrc"), tmp_path / "paper_1808_02638_gb300" / "csrc")
    return str(tmp_path)


def _record(root, **changes):
    rec = {"tiling": [32, 32, 1, 256], "source_sha256_16": bench.kernel_hash(root), "alu_instructions_per_cell": 1,
           "bytes_per_launch": 2}
    rec.update(changes)
    with open(os.path.join(root, "profiles", "step_uniform_2048x2048_traffic.json"), "w") as f:
        json.dump(rec, f)


def test_a_record_counts_for_its_own_tiling_and_sources_only(tmp_path):
    root = _copy(tmp_path)
    assert bench.profiled_launch((32, 32, 1, 256), root) is None   # none there
    _record(root)
    assert bench.profiled_launch((32, 32, 1, 256), root)["bytes_per_launch"] == 2
    assert bench.profiled_launch((16, 16, 1, 192), root) is None
    assert bench.profiled_launch((32, 32, 2, 256), root) is None
    _record(root, source_sha256_16="0" * 16)
    assert bench.profiled_launch((32, 32, 1, 256), root) is None


def test_every_source_of_the_kernel_is_hashed(tmp_path):
    root = _copy(tmp_path)
    _record(root)
    paths = bench.kernel_sources(root)
    names = {os.path.basename(p) for p in paths}
    assert {"claw_step_uniform_pull.cu", "claw_fixed.cuh", "claw_step.cuh", "claw_reflux.cuh", "claw_interp.cuh",
            "claw_internal.h"} <= names
    for p in paths:   # closed under inclusion
        with open(p) as f:
            src = f.read()
        assert set(re.findall(r'#include "(claw_[^"/]*)"', src)) <= names
        with open(p, "a") as f:
            f.write("// changed\n")
        assert bench.profiled_launch((32, 32, 1, 256), root) is None
        with open(p, "w") as f:
            f.write(src)
        assert bench.profiled_launch((32, 32, 1, 256), root)


def test_the_committed_record_says_what_it_was_taken_of():
    with open(os.path.join(bench.ROOT, "profiles", "step_uniform_2048x2048_traffic.json")) as f:
        rec = json.load(f)
    assert rec["bytes_per_launch"] == rec["dram_read_bytes"] + rec["dram_write_bytes"]
    assert len(rec["tiling"]) == 4 and rec["alu_instructions_per_cell"] > 0
    assert rec["source_files"] == [os.path.basename(p) for p in bench.kernel_sources()]
