"""The basis of null(E) a factor computes in: the packs of schedules 1 to 4 keep the orthonormal
one at every precision, and the two-launch form takes the reduced one only where that is well
conditioned, so no network loses digits to it."""
import numpy as np
import pytest

import oracle
import synth
from tests import harness as H
from tests.test_gpu_two_launch import BOUND, _refused, errors, two_launch

pytestmark = pytest.mark.gpu

N_X, N_U, N_E = 20, 60, 12


def _problem(kind):
    """Junctions that every actuator touches almost alike: the reduced basis has entries within
    1, but cond(L'L) near 500; or with one or two actuators per junction."""
    P = synth.custom(61, N_X, N_U, N_E, N_E, synth.make_tree([3, 2], 9))
    if kind == "alike":
        E = np.hstack([np.eye(N_E), np.random.default_rng(0).uniform(0.9, 1.0, (N_E, N_U - N_E))])
        P["net"] = {**P["net"], "E": E}
    return P


def _first_iterate(P, L, dtype):
    """u of the first iterate (w = 0: r = sums of beta over the subtrees, u = uhat + L v along the
    paths) with the matrices and vectors of basis L in dtype."""
    tree, _, cu = H.oracle_build(P)
    f64 = oracle.factor(P["net"], P["cost"])
    T = f64.L.T @ L  # beta in basis L: beta is L' times a vector of the inputs
    beta = (cu.beta @ T).astype(dtype)
    Lam = -np.linalg.inv(L.T @ P["cost"]["W_u"] @ L)
    r = beta.copy()
    for m in range(tree.n - 1, 0, -1):
        r[tree.parent[m]] += r[m]
    v = np.stack([(Lam / (2 * tree.prob[m])).astype(dtype) @ r[m] for m in range(tree.n)])
    for m in range(1, tree.n):
        v[m] += v[tree.parent[m]]
    return cu.u_hat + (v @ L.T.astype(dtype)).astype(np.float64)


def _reduced(E):
    """[-E1^{-1} E2; I] for the leading columns as E1."""
    n_e, n_u = E.shape
    return np.vstack([-np.linalg.solve(E[:, :n_e], E[:, n_e:]), np.eye(n_u - n_e)])


@pytest.mark.parametrize("schedule", [0, 1, 2, 3, 4])
def test_packs_keep_the_orthonormal_basis(schedule):
    """float32 on every schedule errs as float32 arithmetic in the orthonormal basis does (four
    times its error for other orders of summation); in the reduced basis it would not."""
    P = _problem("alike")
    tree, fac, _ = H.oracle_build(P)
    exact = _first_iterate(P, fac.L, np.float64)
    bar = 4 * np.abs(_first_iterate(P, fac.L, np.float32) - exact).max()
    assert np.abs(_first_iterate(P, _reduced(P["net"]["E"]), np.float64) - exact).max() < 1e-3 * bar
    assert np.abs(_first_iterate(P, _reduced(P["net"]["E"]), np.float32) - exact).max() > bar
    steps = H.full_size_steps(P)
    R = H.oracle_run(P, steps, 1)
    assert np.abs(R.u - exact).max() < 1e-3 * bar
    g = H.Gpu(P, steps=steps, precision=1, schedule=schedule)
    try:
        g.solve(1)
        u = g.arrays()[0]
    finally:
        g.close()
    assert np.abs(u - R.u).max() <= bar


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_two_launch_form_needs_a_well_conditioned_basis(precision):
    P = _problem("alike")
    _refused(P, H.full_size_steps(P), precision)


@pytest.mark.parametrize("shared", [0, 1])
def test_network_that_only_the_two_launch_form_can_run(shared):
    """float64 packs beyond shared memory: no better conditioned choice than the reduced basis."""
    P = synth.custom(62, 40, 150, 6, 6, synth.make_tree([3, 2], 5))
    E = np.hstack([np.eye(6), np.random.default_rng(0).uniform(0.9, 1.0, (6, 144))])
    P["net"] = {**P["net"], "E": E}
    steps = H.full_size_steps(P)
    g = H.Gpu(P, steps=steps, shared_packs=shared)
    try:
        g.solve(30)
        got = g.arrays()
    finally:
        g.close()
    assert errors(got, H.oracle_run(P, steps, 30)) <= BOUND[0]


@pytest.mark.parametrize("precision", [0, 1])
def test_shard_of_a_two_launch_factor(precision):
    """A shard runs the factor's packs, in their basis, although the factor's own solves run in
    the reduced one; both give the oracle's iterates, in either order."""
    from paper_1604_01074_gb300.shard import LibraryShard
    P = _problem("few")
    steps = H.full_size_steps(P)
    R = H.oracle_run(P, steps, 30)
    step = {k: P[k] for k in ("p", "q", "dhat", "alpha2", "eps")}
    g = two_launch(P, steps, precision=precision)
    try:
        n_chains = g.smpc.smpc_tree_info_get(g.tree)["n_chains"]
        sh = LibraryShard(g.fac, precision, 0, n_chains, g.n, g.n_x, g.n_u)  # all chains: nothing to exchange
        for _ in range(2):
            sh.begin(step, 30, 0.0)
            for nu in range(30):
                sh.local(nu)
                sh.top(nu)
            sh.tail(30)
            assert sh.finish(30)["iterations"] == 30
            assert errors([t.double().cpu().numpy() for t in (sh.u, sh.x, sh.y)], R) <= BOUND[precision]
            g.solve(30)
            assert errors(g.arrays(), R) <= BOUND[precision]
        sh.close()
    finally:
        g.close()
