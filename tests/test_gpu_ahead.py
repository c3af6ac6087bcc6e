"""The step kernels that draw a step's noise ahead of their loads
(k_step_ahead and k_step_twin) against the
scalar kernel asked for by name: the same state bit for bit, on rows shorter
and longer than a block, odd rows with and without a middle site, ragged last
blocks, every storage format and noise variant, and over several dependent
launches."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = [
    (lb.D2Q9, (510, 100), lb.F32), (lb.D2Q9, (1030, 520), lb.F32), (lb.D2Q9, (516, 1024), lb.F32_F16),
    (lb.D2Q9, (301, 200), lb.F32), (lb.D2Q9, (65, 801), lb.F32_BF16), (lb.D2Q9, (1, 60001), lb.F32),
    (lb.D2Q9, (3, 20011), lb.F32), (lb.D3Q19, (46, 33, 31), lb.F32), (lb.D3Q19, (258, 20, 17), lb.F32),
    (lb.D3Q19, (34, 35, 36), lb.F32_F16), (lb.D3Q19, (66, 35, 24), lb.F32_BF16), (lb.D3Q19, (47, 33, 31), lb.F32),
]


def _run(lat, dims, precision, mode, dist, n, **kw):
    Q, N = lb.Q_OF[lat], int(np.prod(dims))
    with lb.Simulation(lat, dims, 0.9, 40.0, 8, precision=precision, noise_mode=mode, noise_dist=dist,
                       init=lb.INIT_NONE, lattice_id=6, **kw) as s:
        s.set_f(synth.random_populations(Q, N, 40.0, 0.3, seed=N))
        s.step(n)
        return s.get_f()


@pytest.mark.parametrize("mode,dist", [(lb.NOISE_LOCAL, lb.GAUSSIAN), (lb.NOISE_GLOBAL, lb.UNIFORM)])
@pytest.mark.parametrize("lat,dims,precision", CASES)
def test_noise_ahead_changes_nothing(lat, dims, precision, mode, dist):
    auto = _run(lat, dims, precision, mode, dist, 5)
    scalar = _run(lat, dims, precision, mode, dist, 5, step_kernel=lb.KERNEL_SCALAR)
    assert np.array_equal(auto, scalar)
