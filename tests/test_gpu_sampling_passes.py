"""The separate sampling pass: few modes (kept per thread) and many (added per tile), negative and large wave
numbers on a long line, and D3Q19 above the size from which sampled steps take it."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from tests.test_gpu_fused_sampling import _check_sums

pytestmark = pytest.mark.gpu

MANY = [(1, 0, 0), (2, 1, 0), (0, 1, 1), (3, 2, 1), (-1, 0, 0), (0, -2, 1), (5, 0, 0), (0, 3, 0)]


@pytest.mark.parametrize("lat,dims,prec", [(lb.D1Q3, (4099,), lb.F32), (lb.D2Q9, (300, 261), lb.F32),
                                           (lb.D2Q9, (67, 21), lb.F32_F16), (lb.D3Q19, (33, 30, 21), lb.F32_BF16),
                                           (lb.D3Q19, (64, 64, 48), lb.F32)])
@pytest.mark.parametrize("count", [4, 5, 8])
def test_modes_kept_per_thread_and_per_tile(lat, dims, prec, count):
    # (the sums and bounds of the other sampling tests)
    modes = [(k[0] if len(dims) > 0 else 0, k[1] if len(dims) > 1 else 0, k[2] if len(dims) > 2 else 0) for k in MANY]
    modes = modes[:count]
    with lb.Simulation(lat, dims, 0.8, 30.0, 4, precision=prec, modes=modes) as s:
        fs = []
        for _ in range(2):
            s.step(5)
            fs.append(s.get_f())
            s.sample()
        _check_sums(s.observables(), fs, 30.0, modes, dims)


def test_wave_numbers_on_a_line_without_phase_table():
    modes = [(-1, 0, 0), (1100000, 0, 0), (2200000, 0, 0)]
    with lb.Simulation(lb.D1Q3, (2200001,), 0.8, 30.0, 4, modes=modes) as s:
        s.step(3)
        f = s.get_f()
        s.sample()
        _check_sums(s.observables(), [f], 30.0, modes, (2200001,))


@pytest.mark.parametrize("prec", [lb.F32, lb.F32_F16])
def test_large_d3q19_sampled_steps(prec):  # 2^22 sites and above take the pass
    dims, modes = (160, 161, 164), [(1, 0, 0), (1, 1, 1)]
    kw = dict(precision=prec, modes=modes)
    with lb.Simulation(lb.D3Q19, dims, 0.8, 30.0, 4, **kw) as plain:
        fs = [plain.get_f()]
        plain.step(4)
        fs.append(plain.get_f())
        plain.step(2)
        end = plain.get_f()
    with lb.Simulation(lb.D3Q19, dims, 0.8, 30.0, 4, sample_every=4, **kw) as s:
        s.step(6)
        np.testing.assert_array_equal(s.get_f(), end)
        _check_sums(s.observables(), fs, 30.0, modes, dims)
