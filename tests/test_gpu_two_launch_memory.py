"""Device memory of factors that may take the two-launch iteration: its matrices are optional,
so a factor without room for them still runs schedules 1 to 4."""
import pytest

import synth
from tests import harness as H
from tests.test_gpu_two_launch import BOUND, errors

pytestmark = pytest.mark.gpu


def _tree_242():
    P = synth.barcelona(0, branching=(10, 8, 5), n_scenarios=242)  # 5173 nodes
    tree, fac, _ = H.oracle_build(P)
    return P, H.closed_form_steps(fac, tree, 1e-6)


def test_factor_without_room_for_the_two_launch_matrices():
    """Room for the packs, and beside them either for the vectors or for the packed Lambda and
    half of the vectors: schedules 1 to 4 fit, with 27 MB to spare on either side."""
    import torch
    P, steps = _tree_242()
    n, n_v = len(P["tree"]["parent"]), 97
    H.Gpu(P, steps=steps, precision=1).close()  # what the first factor of a process loads
    g = H.Gpu(P, steps=steps, precision=1, schedule=4)
    total = g.smpc.smpc_factor_device_bytes(g.fac)
    g.close()
    packs = n * (177 * 100 + 97 * 100) * 4
    G = (n_v + 3) // 4
    lam = n * (G // 2 + 1) * G * 16 * 4
    vectors = total - packs
    assert 40e6 < vectors < lam
    R = H.oracle_run(P, steps, 10)
    torch.cuda.synchronize()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - packs - lam - vectors // 2, dtype=torch.uint8, device="cuda")
    try:
        g = H.Gpu(P, steps=steps, precision=1)
        try:
            assert g.solve(10)["iterations"] == 10
            assert errors(g.arrays(), R) <= BOUND[1]
            assert g.smpc.smpc_factor_device_bytes(g.fac) <= total
        finally:
            g.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert torch.cuda.mem_get_info()[0] > packs + lam + 2 * vectors  # given back
