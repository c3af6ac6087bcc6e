"""Mass of long FP32 moment-space runs.

Every step rounds each site's density sum and its rest population, Q times at most half a unit of FP32 (2^-25
relative on average), in no preferred direction: over S steps and N sites the mass wanders by about sqrt(Q S / N)
2^-25 of itself.  Four times that is allowed.  A biased rounding would show as S times its mean."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import synth

pytestmark = pytest.mark.gpu

S = 1000


@pytest.mark.parametrize("lat,dims", [(lb.D1Q3, (1200,)), (lb.D2Q5, (40, 31)), (lb.D2Q9, (40, 31)),
                                      (lb.D3Q19, (12, 10, 11))])
@pytest.mark.parametrize("tau,mode", [(0.9, lb.NOISE_GLOBAL), (0.75, lb.NOISE_LOCAL)])
def test_mass_does_not_drift(lat, dims, tau, mode):
    Q, N, rho = lb.Q_OF[lat], int(np.prod(dims)), 120.0
    taus = [0] + [round(tau * (0.75 + 0.5 * ((7 * a) % Q) / Q), 4) for a in range(1, Q)]
    with lb.Simulation(lat, dims, tau, rho, 8, noise_mode=mode, tau_moments=taus, init=lb.INIT_NONE) as s:
        s.set_f(synth.random_populations(Q, N, rho, 0.2, seed=Q))
        before = s.mass()
        s.step(S)
        after = s.mass()
    assert abs(after - before) <= 4 * np.sqrt(Q * S / N) * 2.0**-25 * before
