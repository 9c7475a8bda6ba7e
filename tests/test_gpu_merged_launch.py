"""bfloat16 factors with one pack on schedule 2: the first three launches of an iteration as one
(tree pass) against the three launches, bit for bit: u, x, y, the residual history and with it
the stop."""
import numpy as np
import pytest

import synth
from tests import harness as H
from tests.test_gpu_two_launch import LATE, _forest, iteration_form

pytestmark = pytest.mark.gpu


def _both(P, steps, iters, tol=0.0, trees=1, **kw):
    out = []
    for form, launches in (("two-launch", 4), ("separate", 6)):
        with iteration_form(form):
            g = H.Gpu(P, steps=steps, precision=2, schedule=2, shared_packs=1, tc_width=16)
        try:
            ms = g.smpc.smpc_profile_solve(g.fac, P["p"], P["q"], P["dhat"], P["alpha2"], eps=P["eps"], iters=8)
            assert len(ms) == launches
            info = g.solve(iters, tol=tol, check_every=16, **kw)
            out.append((info["iterations"], info["history"], *g.arrays(),
                        *(g.smpc.smpc_solve_trees(g.fac, trees) if trees > 1 else ())))
        finally:
            g.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
    return out[0]


@pytest.mark.parametrize("n_x,n_u,n_e", [(4, 10, 2), (32, 64, 4), (33, 66, 5), (64, 128, 8), (65, 131, 3)])
def test_sizes(n_x, n_u, n_e):
    P = synth.custom(63, n_x, n_u, max(n_e, 3), n_e, LATE)
    _both(P, H.full_size_steps(P), 50)


def test_forest_with_a_stop_per_tree():
    members, F, steps, _ = _forest()
    out = _both(F, steps, 3000, tol=1e-3, trees=len(members))
    assert len(set(out[5])) > 1  # the trees stop at different iterations


def test_deep_tree_with_the_ergodic_average():
    P = synth.custom(64, 20, 40, 6, 6, synth.make_tree([3, 3], 24))
    _both(P, H.full_size_steps(P), 60, ergodic=1)
