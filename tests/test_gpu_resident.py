"""The resident kernel (csrc/resident_kernels.cuh: a small lattice stepped
many times per launch) at the edges of its rule: the largest single block and
the smallest cluster of each lattice, the largest lattice it takes and the
smallest it does not, ragged last CTAs, sides of 1 and 2, single relaxation
and the moment-space collision.  Stepped in one call or one step per call, the
state is the same bit for bit; the launches say which path ran."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import abi, synth

pytestmark = pytest.mark.gpu

# lattice, dims, precision, moment-space, launches of step(11)
CASES = [
    (lb.D1Q3, (512,), lb.F32, False, 1), (lb.D1Q3, (513,), lb.F32, False, 1), (lb.D1Q3, (16384,), lb.F32, False, 1),
    (lb.D1Q3, (16385,), lb.F32, False, 11), (lb.D2Q9, (16, 16), lb.F32, False, 1),
    (lb.D2Q9, (257, 1), lb.F32, False, 1), (lb.D2Q9, (2, 131), lb.F32_BF16, False, 1),
    (lb.D2Q9, (128, 128), lb.F32, False, 1), (lb.D2Q9, (129, 127), lb.F32_F16, False, 1),
    (lb.D2Q9, (128, 129), lb.F32, False, 11), (lb.D3Q19, (8, 16, 1), lb.F32, False, 1),
    (lb.D3Q19, (43, 3, 1), lb.F32, False, 1), (lb.D3Q19, (16, 24, 24), lb.F32, False, 1),
    (lb.D3Q19, (21, 21, 21), lb.F32, False, 11), (lb.D2Q9, (32, 64), lb.F64, False, 1),
    (lb.D2Q9, (683, 3), lb.F64, False, 11), (lb.D3Q19, (2, 1, 9), lb.F64, False, 1),
    (lb.D2Q5, (3, 3), lb.F64, True, 1), (lb.D2Q5, (81, 81), lb.F32, True, 1), (lb.D2Q5, (127, 130), lb.F32, True, 11),
    (lb.D2Q9, (61, 37), lb.F32, True, 1), (lb.D3Q19, (11, 9, 7), lb.F64, True, 1),
    (lb.D3Q19, (20, 20, 20), lb.F32, True, 1), (lb.D1Q3, (501,), lb.F32, True, 1),
]


@pytest.mark.parametrize("mode,dist", [(lb.NOISE_LOCAL, lb.GAUSSIAN), (lb.NOISE_GLOBAL, lb.UNIFORM),
                                       (lb.NOISE_OFF, lb.GAUSSIAN)])
@pytest.mark.parametrize("lat,dims,precision,mrt,launches", CASES)
def test_many_steps_equal_single_steps(lat, dims, precision, mrt, launches, mode, dist):
    Q, N = lb.Q_OF[lat], int(np.prod(dims))
    f0 = synth.random_populations(Q, N, 40.0, 0.3, seed=N)
    taus = [0] + [0.7 + 0.03 * a for a in range(1, Q)] if mrt else None
    kw = dict(precision=precision, noise_mode=mode, noise_dist=dist, init=lb.INIT_NONE, lattice_id=3, tau_moments=taus)
    with lb.Simulation(lat, dims, 0.9, 40.0, 8, **kw) as a:
        a.set_f(f0)
        n0 = abi.lbfd_kernel_launches()
        a.step(11)
        assert abi.lbfd_kernel_launches() - n0 == launches
        a.step(4)
        fa = a.get_f()
    with lb.Simulation(lat, dims, 0.9, 40.0, 8, **kw) as b:
        b.set_f(f0)
        for _ in range(15):
            b.step(1)
        fb = b.get_f()
    assert np.array_equal(fa, fb)
