"""The two-launch iteration (tree pass, Lambda launch) a factor chooses by timing where
[Bbar; L] is sparse, against the FP64 oracle at the sizes where its layout can go wrong: one
and two block rows, odd and even counts of them, a full warp of them, the 8 x 8 blocks beyond
n_v = 128; trees of one node, one chain, late and uneven branchings, forests.  Bars as in the
other parity tests: 1e-9 (float64), 1e-4 (float32), relative to 1 + the largest entry."""
import numpy as np
import pytest

import oracle
import synth
from tests import harness as H

pytestmark = pytest.mark.gpu

BOUND = {0: 1e-9, 1: 1e-4}
LATE = synth.tree_from_fanouts_dict([[1], [1], [3], [1, 1, 1], [2, 1, 2]])
TREES = {"node": synth.make_tree([1], 1), "chain": synth.make_tree([1], 9), "late": LATE,
         "fan": synth.make_tree([3, 2], 5), "wide": synth.make_tree([70], 3)}


def _uses_sweep(g, P):
    ms = g.smpc.smpc_profile_solve(g.fac, P["p"], P["q"], P["dhat"], P["alpha2"], eps=P["eps"], iters=4)
    return len(ms) == 2


def _check(P, precision, shared, iters=40):
    tree, fac, _ = H.oracle_build(P)
    steps = oracle.jacobi_steps(fac, tree)
    R = H.oracle_run(P, steps, iters)
    g = H.Gpu(P, steps=steps, precision=precision, shared_packs=shared)
    try:
        if not _uses_sweep(g, P):
            pytest.skip("another schedule was faster here")
        info = g.solve(iters)
        u, x, y = g.arrays()
    finally:
        g.close()
    assert info["iterations"] == iters
    e = (H.relerr(u, R.u), H.relerr(x, R.x), H.relerr(y, H.stack_y(R.y)))
    assert max(e) <= BOUND[precision], e
    assert abs(info["rho_rel"] - R.rho_rel[-1]) <= BOUND[precision]


@pytest.mark.parametrize("shared", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n_x,n_u,n_e", [(1, 2, 1), (2, 4, 0), (3, 5, 0), (2, 10, 2), (4, 9, 0), (33, 66, 5),
                                         (40, 130, 3), (30, 128, 0), (31, 129, 0), (60, 196, 6)])
def test_layout_sizes(n_x, n_u, n_e, precision, shared):
    _check(synth.custom(51, n_x, n_u, max(n_e, 3), n_e, LATE), precision, shared)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", list(TREES))
def test_trees(name, precision):
    _check(synth.custom(52, 5, 11, 4, 2, TREES[name]), precision, 0)


def test_warm_start_and_early_stop():
    """A tolerance-stopped solve and a warm one: the two-launch form against schedule 1."""
    P = synth.custom(53, 5, 11, 4, 2, TREES["fan"])
    steps = H.tiny_steps(P)
    out = []
    for schedule in (1, 0):
        g = H.Gpu(P, steps=steps, schedule=schedule)
        try:
            if schedule == 0 and not _uses_sweep(g, P):
                pytest.skip("another schedule was faster here")
            a = g.solve(400, tol=1e-2)
            b = g.solve(30, warm=1)
            out.append((a["iterations"], b["iterations"], g.arrays()))
        finally:
            g.close()
    assert out[0][:2] == out[1][:2]
    for p, q in zip(out[0][2], out[1][2]):
        assert np.abs(p - q).max() <= BOUND[0] * (1 + np.abs(p).max())


@pytest.mark.parametrize("n_x,n_u,n_e", [(2, 4, 0), (3, 7, 2), (33, 66, 5), (30, 128, 0), (31, 129, 0), (65, 131, 3)])
@pytest.mark.parametrize("anchor_every,polish", [(16, 0), (3, 4), (1, 0)])
def test_bf16_per_node(n_x, n_u, n_e, anchor_every, polish):
    """bfloat16 packs, one per node: the two-launch form applies the same bfloat16 matrices to
    float32 vectors as schedule 1 and anchors in float32 in another basis, so the iterates
    agree as float32 ones do (1e-4), far inside the distance to the oracle."""
    P = synth.custom(54, n_x, n_u, max(n_e, 3), n_e, TREES["fan"] if n_x < 60 else LATE)
    tree, fac, _ = H.oracle_build(P)
    steps = oracle.jacobi_steps(fac, tree)
    out = []
    for schedule in (1, 0):
        g = H.Gpu(P, steps=steps, precision=2, schedule=schedule)
        try:
            if schedule == 0 and not _uses_sweep(g, P):
                pytest.skip("another schedule was faster here")
            info = g.smpc.smpc_solve(g.fac, P["p"], P["q"], P["dhat"], P["alpha2"], eps=P["eps"], max_iters=40, sync=1,
                                     anchor_every=anchor_every, polish_iters=polish, u=g.u, x=g.x, y=g.y)
            out.append((info["rho_rel"], g.arrays()))
        finally:
            g.close()
    assert abs(out[0][0] - out[1][0]) <= BOUND[1]
    for p, q in zip(out[0][1], out[1][1]):
        assert np.abs(p - q).max() <= BOUND[1] * (1 + np.abs(p).max())
