"""Device memory of factors that may take the two-launch iteration: its matrices are optional,
so a factor without room for them still runs schedules 1 to 4."""
import pytest

import synth
from paper_1604_01074_gb300.shard import LibraryShard
from tests import harness as H
from tests.test_gpu_two_launch import BOUND, errors, two_launch

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


@pytest.mark.parametrize("precision,shared", [(0, 0), (1, 0), (2, 0), (1, 1)])
def test_two_launch_factor_keeps_no_packs(precision, shared):
    """Its footprint, which a server admits by, is below that of the schedules that stream packs;
    a shard adds the packs once, and both run."""
    P = synth.custom(72, 30, 56, 9, 9, synth.make_tree([4, 4], 10))
    steps = H.full_size_steps(P)
    n, n_k, n_v = len(P["tree"]["parent"]), 86, 47
    entries = (1 if shared else n) * (n_k + n_v) * n_v  # of the packs, without their padding
    size = {0: 8, 1: 4, 2: 2}[precision]
    packs = entries * (size + (4 if precision == 2 else 0))  # bfloat16 factors: float32 ones as well
    half = 0.65 * packs * n_v / (n_k + n_v)  # one half of every Lambda, with its blocks' padding
    g = H.Gpu(P, steps=steps, precision=precision, schedule=4, shared_packs=shared)
    streaming = g.smpc.smpc_factor_device_bytes(g.fac)
    g.close()
    more = 2 ** 18 + (4 * n * n_k if precision == 2 else 0)  # the sparse image and one basis; the anchor's low parts
    R = H.oracle_run(P, steps, 30)
    g = two_launch(P, steps, precision=precision, shared_packs=shared)
    try:
        own = g.smpc.smpc_factor_device_bytes(g.fac)
        assert own <= streaming - packs + half + more
        if precision == 2:
            return
        sh = [LibraryShard(g.fac, precision, 0, g.smpc.smpc_tree_info_get(g.tree)["n_chains"], g.n, g.n_x, g.n_u) for _ in range(2)]
        assert own + packs <= g.smpc.smpc_factor_device_bytes(g.fac) <= own + 1.2 * packs
        step = {k: P[k] for k in ("p", "q", "dhat", "alpha2", "eps")}
        sh[1].begin(step, 30, 0.0)
        for nu in range(30):
            sh[1].local(nu)
            sh[1].top(nu)
        sh[1].tail(30)
        sh[1].finish(30)
        assert errors([t.double().cpu().numpy() for t in (sh[1].u, sh[1].x, sh[1].y)], R) <= BOUND[precision]
        g.solve(30)
        assert errors(g.arrays(), R) <= BOUND[precision]
        for s in sh:
            s.close()
    finally:
        g.close()
