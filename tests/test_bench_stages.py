"""bench.py's names for the launches of an iteration, by schedule and number."""
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
