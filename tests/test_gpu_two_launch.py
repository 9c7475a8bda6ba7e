"""The two-launch iteration (tree pass, Lambda launch) requested by name (SMPC_ITERATION_FORM),
so that a factor that cannot run it fails the test, against the FP64 oracle: layouts, forests
with a stop per tree, general A, the ergodic average, the allocation-free entry point, graphs
and warm starts; and the networks and trees that do not take it.  Bars as in the other parity
tests: 1e-9 (float64), 1e-4 (float32), relative to 1 + the largest entry."""
import contextlib
import os

import numpy as np
import pytest

import oracle
import synth
from tests import harness as H

pytestmark = pytest.mark.gpu

BOUND = {0: 1e-9, 1: 1e-4}
LATE = synth.tree_from_fanouts_dict([[1], [1], [3], [1, 1, 1], [2, 1, 2]])


@contextlib.contextmanager
def iteration_form(name):
    os.environ["SMPC_ITERATION_FORM"] = name
    try:
        yield
    finally:
        del os.environ["SMPC_ITERATION_FORM"]


def two_launch(P, steps, **kw):
    """A factor in the two-launch form; its iterations are two launches."""
    with iteration_form("two-launch"):
        g = H.Gpu(P, steps=steps, **kw)
    try:
        assert len(g.smpc.smpc_profile_solve(g.fac, P["p"], P["q"], P["dhat"], P["alpha2"], eps=P["eps"], iters=4)) == 2
    except BaseException:
        g.close()
        raise
    return g


def errors(got, R, idx=slice(None)):
    u, x, y = got
    return max(H.relerr(u[idx], R.u), H.relerr(x[idx], R.x), H.relerr(y[idx], H.stack_y(R.y)))


@pytest.mark.parametrize("shared", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n_x,n_u,n_e", [(1, 2, 1), (2, 4, 0), (2, 10, 2), (4, 9, 0), (30, 128, 0), (31, 129, 0),
                                         (65, 131, 0)])
def test_layout_sizes(n_x, n_u, n_e, precision, shared):
    P = synth.custom(51, n_x, n_u, max(n_e, 3), n_e, LATE)
    steps = H.full_size_steps(P)
    R = H.oracle_run(P, steps, 40)
    g = two_launch(P, steps, precision=precision, shared_packs=shared)
    try:
        info = g.solve(40)
        got = g.arrays()
    finally:
        g.close()
    assert info["iterations"] == 40
    assert errors(got, R) <= BOUND[precision]
    assert abs(info["rho_rel"] - R.rho_rel[-1]) <= BOUND[precision]


def _forest(general_A=False):
    members = synth.forest_members(7, 5, max_horizon=7)
    if general_A:
        members = [synth.general_dynamics(P, 3) for P in members]
    F = synth.forest(members)
    n, n_u = len(F["tree"]["parent"]), F["net"]["n_u"]
    steps = {"s": np.zeros(n), "z": np.zeros(n), "p": np.zeros((n, n_u))}
    per = [H.tiny_steps(P) for P in members]
    for r, st in enumerate(per):
        for k in steps:
            steps[k][F["members"][r]] = st[k]
    return members, F, steps, per


@pytest.mark.parametrize("shared", [0, 1])
@pytest.mark.parametrize("general_A", [False, True])
def test_forest_stops_each_tree_on_its_own(general_A, shared):
    """Every tree stops at its own first iterate that meets the tolerance, with that iterate's
    ergodic average, as the oracle does on that tree alone."""
    members, F, steps, per = _forest(general_A)
    tol, cap = 2e-4, 4000
    g = two_launch(F, steps, shared_packs=shared)
    try:
        g.solve(cap, tol=tol, check_every=32, ergodic=1)
        got, (ub, xb) = g.arrays(), g.bars()
        its, rr = g.smpc.smpc_solve_trees(g.fac, len(members))
    finally:
        g.close()
    counts = set()
    for r, P in enumerate(members):
        tree, fac, cu = H.oracle_build(P)
        R = oracle.apg(fac, tree, cu, P["cost"], P["p"], per[r], cap, tol=tol)
        counts.add(len(R.rho_rel))
        assert its[r] == len(R.rho_rel), (r, its[r], len(R.rho_rel))
        idx = F["members"][r]
        assert errors(got, R, idx) <= BOUND[0], r
        assert max(H.relerr(ub[idx], R.ubar), H.relerr(xb[idx], R.xbar)) <= BOUND[0], r
        assert abs(rr[r] - R.rho_rel[-1]) <= BOUND[0]
    assert len(counts) > 1, counts


@pytest.mark.parametrize("general_A", [False, True])
def test_forest_fp32(general_A):
    members, F, steps, per = _forest(general_A)
    g = two_launch(F, steps, precision=1)
    try:
        g.solve(100)
        got = g.arrays()
    finally:
        g.close()
    for r, P in enumerate(members):
        assert errors(got, H.oracle_run(P, per[r], 100), F["members"][r]) <= BOUND[1], r


@pytest.mark.parametrize("precision", [0, 1])
def test_general_A_climbs_several_top_levels(precision):
    P = synth.general_dynamics(synth.custom(55, 9, 17, 5, 2, synth.make_tree([2, 3, 2], 6)), 2)
    steps = H.tiny_steps(P)
    g = two_launch(P, steps, precision=precision)
    try:
        g.solve(60)
        got = g.arrays()
    finally:
        g.close()
    assert errors(got, H.oracle_run(P, steps, 60)) <= BOUND[precision]


@pytest.mark.parametrize("precision", [0, 1])
def test_static_graph_and_warm_start(precision):
    P = synth.custom(56, 5, 11, 4, 2, synth.make_tree([3, 2], 5))
    steps = H.tiny_steps(P)
    R1 = H.oracle_run(P, steps, 50)
    y, nx = H.stack_y(R1.y), P["net"]["n_x"]
    R2 = H.oracle_run(P, steps, 30, y0=(y[:, :nx], y[:, nx:2 * nx], y[:, 2 * nx:]))
    g = two_launch(P, steps, precision=precision)
    try:
        for graph in (0, 1, 1):
            g.solve(50, use_graph=graph, check_every=16)
            assert errors(g.arrays(), R1) <= BOUND[precision]
        g.solve(30, warm=1)
        assert errors(g.arrays(), R2) <= BOUND[precision]
        g.smpc.smpc_solve_static(g.fac, P["p"], P["q"], P["dhat"], P["alpha2"], eps=P["eps"], max_iters=50, sync=1,
                                 u=g.u, x=g.x, y=g.y)
        assert errors(g.arrays(), R1) <= BOUND[precision]
    finally:
        g.close()


def _refused(P, steps, precision=0):
    import paper_1604_01074_gb300 as smpc
    with iteration_form("two-launch"), pytest.raises(smpc.SmpcError) as ei:
        H.Gpu(P, steps=steps, precision=precision)
    assert ei.value.code == smpc.SMPC_ENOTSUP


def test_dense_network_keeps_schedules_1_to_4():
    """[Bbar; L] with more entries than count as sparse."""
    P = synth.custom(57, 40, 120, 3, 0, LATE)
    P["net"] = {**P["net"], "B": np.random.default_rng(1).uniform(-0.2, 0.2, (40, 120))}
    steps = H.full_size_steps(P)
    _refused(P, steps, precision=1)
    g = H.Gpu(P, steps=steps, precision=1)
    try:
        g.solve(20)
        got = g.arrays()
    finally:
        g.close()
    assert errors(got, H.oracle_run(P, steps, 20)) <= BOUND[1]


def test_long_stem_of_top_nodes_keeps_schedules_1_to_4():
    """A branching behind 5793 single nodes: the lists of top nodes below each top node would
    have 2^24 entries and more."""
    D = 5793
    assert D * (D + 1) // 2 > 2 ** 24
    P = synth.custom(58, 1, 2, 1, 0, synth.make_tree([1, 1], 2))
    parent = np.concatenate([np.arange(-1, D - 1), [D - 1, D - 1]]).astype(np.int32)
    n = len(parent)
    stage = np.concatenate([np.arange(D), [D, D]])
    prob = np.where(stage < D, 1.0, 0.5)
    rep = lambda v: np.resize(v, (D + 1, v.shape[1]))  # noqa: E731
    P = {**P, "tree": {"parent": parent, "prob": prob, "stage": stage, "horizon": D + 1}, "dhat": rep(P["dhat"]),
         "alpha2": rep(P["alpha2"]), "eps": np.zeros((n, P["net"]["n_d"]))}
    steps = {"s": np.full(n, 1e-9), "z": np.full(n, 1e-9), "p": np.full((n, 2), 1e-9)}
    _refused(P, steps)
    g = H.Gpu(P, steps=steps)
    try:
        g.solve(2)
        got = g.arrays()
    finally:
        g.close()
    assert errors(got, H.oracle_run(P, steps, 2)) <= BOUND[0]


def test_separate_form_runs_the_launches_of_the_schedules():
    P = synth.tiny(0)
    with iteration_form("separate"):
        for precision, schedule, shared, count in ((1, 4, 0, 3), (2, 2, 1, 6)):
            g = H.Gpu(P, steps=H.tiny_steps(P), precision=precision, schedule=schedule, shared_packs=shared)
            try:
                ms = g.smpc.smpc_profile_solve(g.fac, P["p"], P["q"], P["dhat"], P["alpha2"], eps=P["eps"], iters=8)
            finally:
                g.close()
            assert len(ms) == count
        g = H.Gpu(P, steps=H.tiny_steps(P))
        try:
            assert len(g.smpc.smpc_profile_solve(g.fac, P["p"], P["q"], P["dhat"], P["alpha2"], eps=P["eps"],
                                                 iters=8)) in (1, 3, 4, 6)
        finally:
            g.close()
