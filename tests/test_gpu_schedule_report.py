"""smpc_factor_schedule: the times behind the choice, where the reported schedule itself does not
fit the network and the two-launch form reported under its number does."""
import pytest

import synth
from tests import harness as H
from tests.test_gpu_two_launch import LATE, iteration_form

pytestmark = pytest.mark.gpu

# packs of 219 to 221 KB a node: about where one no longer fits an SM beside schedule 4's vectors
SIZES = [(74, 100, 0), (75, 100, 0), (76, 100, 0)]


def _report(P, steps):
    g = H.Gpu(P, steps=steps)
    try:
        return g.smpc.smpc_factor_schedule(g.fac), len(g.smpc.smpc_profile_solve(
            g.fac, P["p"], P["q"], P["dhat"], P["alpha2"], eps=P["eps"], iters=4))
    finally:
        g.close()


def test_reported_schedule_has_its_time_when_others_have():
    seen = 0
    for n_x, n_u, n_e in SIZES:
        P = synth.custom(71, n_x, n_u, 3, n_e, LATE)
        steps = H.full_size_steps(P)
        (s, ms), launches = _report(P, steps)
        if any(ms.values()):
            assert ms[s] > 0 and ms[s] == min(t for t in ms.values() if t > 0), (n_x, n_u, s, ms)
        with iteration_form("separate"):
            try:
                (_, alone), _ = _report(P, steps)
            except Exception:  # none of schedules 1 to 4 fits
                continue
        seen += launches == 2 and any(ms.values()) and alone[4] == 0
    assert seen > 0  # sizes at which schedule 4 does not fit, some other does, and the form is chosen
