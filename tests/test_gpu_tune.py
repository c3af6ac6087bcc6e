"""The tuner times what a run does: chunks of steps with their preparation, clock and dependent launches."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import abi, synth

pytestmark = pytest.mark.gpu


def test_tuner_times_the_launches_of_a_run():
    """Small members, where launches are most of a step: the parameter-space order, which takes one launch a step
    and no fork and join, runs at three times the speed of the others, so the tuner has to find it.  Each of 64
    candidates runs whole chunks of 16 steps: 17 launches of one group and the clock, or 16 times preparation, step
    and clock."""
    specs = synth.ensemble(20, 30, 80, seed=12345, ndim=2)
    with lb.Ensemble(lb.D2Q9, specs) as e:
        e.step(7)
        before = [e.get_f(m) for m in range(20)]
        n0 = abi.lbfd_kernel_launches()
        e.tune(3)
        launches = abi.lbfd_kernel_launches() - n0
        # a warm-up chunk and 1 or 1 + 8 timed ones of every candidate
        least = 16 * 2 * 17 + 48 * 2 * 48
        most = 16 * 10 * 17 + 48 * 10 * 48
        assert least <= launches <= most
        assert e.query()[6] == lb.WALK_PARAM
        assert all(np.array_equal(before[m], e.get_f(m)) for m in range(20))
