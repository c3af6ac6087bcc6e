"""Moment-space steps with one, two and four sites per thread (the width that the buffers' start allows): the same
state bit for bit.  Two sites are updated on the packed FP32 instructions, where a product may not be fused into the
sum it enters: in the one-site form it is not."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import synth
from tests.test_gpu_buffers import _Shifted

pytestmark = pytest.mark.gpu


# 2^19 sites and more: four sites per thread on aligned buffers (D3Q19: two)
@pytest.mark.parametrize("mode,dist", [(lb.NOISE_LOCAL, lb.GAUSSIAN), (lb.NOISE_GLOBAL, lb.UNIFORM),
                                       (lb.NOISE_OFF, lb.GAUSSIAN)])
@pytest.mark.parametrize("lat,dims", [(lb.D1Q3, (1 << 19,)), (lb.D2Q5, (512, 130)), (lb.D2Q5, (1024, 512)),
                                      (lb.D2Q9, (1024, 512)), (lb.D3Q19, (64, 32, 33))])
def test_widths_agree(lat, dims, mode, dist):
    Q, N = lb.Q_OF[lat], int(np.prod(dims))
    f0 = synth.random_populations(Q, N, 40.0, 0.3, seed=N)
    states = []
    for shift in ((0, 0), (2, 2), (1, 1)):
        with _Shifted(shift, lat, dims, 0.9, 40.0, 8, noise_mode=mode, noise_dist=dist, init=lb.INIT_NONE,
                      tau_moments=[0] + [0.7 + 0.03 * a for a in range(1, Q)]) as s:
            s.set_f(f0)
            s.step(3)
            states.append(s.get_f())
    assert np.array_equal(states[0], states[1]) and np.array_equal(states[0], states[2])
