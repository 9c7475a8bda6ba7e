"""The two-launch iteration when a wait for its matrices gives up, without any GPU fault: a bound of
zero (SMPC_PIPELINE_WAIT_NS, read when a factor is created) makes each wait one test of a copy that
has just been issued; the warp records the error, lets its copy land under the normal bound and
returns, and the other launches see the error flag and exit."""
import os

import pytest

import synth
from tests import harness as H
from tests.test_gpu_two_launch import BOUND, errors, iteration_form, two_launch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [1, 2])
def test_matrix_wait_that_gives_up_reports_etimeout(precision):
    import paper_1604_01074_gb300 as smpc
    P = synth.barcelona(0, branching=(5, 5, 4), n_scenarios=100, horizon=18)
    tree, fac, _ = H.oracle_build(P)
    steps = H.closed_form_steps(fac, tree, 1e-6)
    os.environ["SMPC_PIPELINE_WAIT_NS"] = "0"
    try:
        with iteration_form("two-launch"):
            g = H.Gpu(P, steps=steps, precision=precision)
    finally:
        del os.environ["SMPC_PIPELINE_WAIT_NS"]
    try:
        for _ in range(2):  # and the next solve of the factor starts afresh
            with pytest.raises(smpc.SmpcError) as ei:
                g.solve(10)
            assert ei.value.code == smpc.SMPC_ETIMEOUT, ei.value
    finally:
        g.close()
    g = two_launch(P, steps, precision=1)  # the normal bound again
    try:
        assert g.solve(10)["iterations"] == 10
        assert errors(g.arrays(), H.oracle_run(P, steps, 10)) <= BOUND[1]
    finally:
        g.close()


def test_one_matrix_for_all_nodes_under_a_bound_of_zero():
    """Its single copy is issued before the launch waits for the previous one, so it may or may not
    have landed: the solve either times out or is the usual one."""
    import paper_1604_01074_gb300 as smpc
    P = synth.barcelona(0, branching=(5, 5, 4), n_scenarios=100, horizon=18)
    tree, fac, _ = H.oracle_build(P)
    steps = H.closed_form_steps(fac, tree, 1e-6)
    os.environ["SMPC_PIPELINE_WAIT_NS"] = "0"
    try:
        with iteration_form("two-launch"):
            g = H.Gpu(P, steps=steps, precision=1, shared_packs=1)
    finally:
        del os.environ["SMPC_PIPELINE_WAIT_NS"]
    try:
        try:
            g.solve(10)
        except smpc.SmpcError as e:
            assert e.code == smpc.SMPC_ETIMEOUT
        else:
            assert errors(g.arrays(), H.oracle_run(P, steps, 10)) <= BOUND[1]
    finally:
        g.close()
