"""bench.py's names for the launches of an iteration, by schedule and number, and the recorded DRAM
traffic of the two-launch form's kernels, valid while their own source is unchanged."""
import hashlib
import json

import pytest

import bench


@pytest.mark.parametrize("schedule,count,first,last", [
    (1, 1, "apg_iter", "apg_iter"), (2, 6, "fwd_scan", "node_mv_dh"), (3, 4, "fwd_scan", "node_mv_dh"),
    (4, 3, "fwd_scan", "apg_iter_bwd"), (4, 2, "tree_sweep", "lambda_apply"), (2, 2, "tree_sweep", "lambda_apply"),
    (2, 4, "merged_sweep", "node_mv_dh")])
def test_every_launch_has_its_name(schedule, count, first, last):
    names = bench.stages_of(schedule, [1.0] * count)
    assert len(names) == count and names[0] == first and names[-1] == last


def test_merged_launch_is_followed_by_the_product_of_the_transposed_pack():
    assert bench.stages_of(2, [1.0] * 4)[1:3] == ["node_mv_gt", "scan_r"]


def test_two_launch_form_has_its_own_label():
    assert bench.schedule_name(4, 2) == bench.schedule_name(2, 2) != bench.schedule_name(4, 3)
    assert bench.schedule_name(2, 4) == bench.schedule_name(2, 6)


def test_traffic_of_the_two_launch_kernels_follows_their_source(tmp_path, monkeypatch):
    src = tmp_path / "paper_1604_01074_gb300" / "csrc"
    src.mkdir(parents=True)
    (tmp_path / "profiles").mkdir()
    (src / "kernels.cu").write_bytes(b"// k")
    (src / "sweep.cuh").write_bytes(b"// s1")
    sha = hashlib.sha256(b"// s1").hexdigest()[:16]
    rec = {"kernel_sha256_16": "0", "sweep_sha256_16": sha,
           "two_launch": [{"key": "fp32_lambda_apply_21111", "dram_bytes_per_launch": 5}]}
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps(rec))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.recorded_traffic("fp32_lambda_apply_21111") == 5
    assert bench.recorded_traffic("fp32_tree_sweep_21111") is None
    assert bench.recorded_traffic("fp32_apg_iter_bwd_21111") is None
    (src / "sweep.cuh").write_bytes(b"// s2")
    assert bench.recorded_traffic("fp32_lambda_apply_21111") is None
