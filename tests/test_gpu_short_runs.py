"""Short runs of small lattices: a launch that holds many steps is taken from the number of steps on that makes up
for its cost, and fewer steps, in one call or between two samples, are launched one by one.  The launches say which
ran; state and sums are those of single-step calls."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import abi

pytestmark = pytest.mark.gpu

# lattice, dims, precision, moment-space, the fewest steps that share a launch
CASES = [(lb.D1Q3, (300,), lb.F32, False, 2), (lb.D1Q3, (4000,), lb.F32, True, 4), (lb.D1Q3, (300,), lb.F64, False, 6),
         (lb.D2Q5, (13, 11), lb.F32, True, 2), (lb.D2Q5, (81, 81), lb.F32, True, 4), (lb.D2Q5, (127, 127), lb.F32, True, 8),
         (lb.D2Q9, (15, 17), lb.F32, False, 4), (lb.D2Q9, (61, 37), lb.F32_BF16, False, 5),
         (lb.D2Q9, (120, 120), lb.F32, True, 8), (lb.D2Q9, (20, 20), lb.F64, True, 8),
         (lb.D3Q19, (6, 6, 6), lb.F32, False, 6), (lb.D3Q19, (7, 5, 3), lb.F32, True, 6),
         (lb.D3Q19, (6, 6, 6), lb.F64, False, 8)]


def _options(lat, precision, mrt):
    taus = [0] + [0.7 + 0.03 * a for a in range(1, lb.Q_OF[lat])] if mrt else None
    return dict(precision=precision, tau_moments=taus, lattice_id=3)


def _launches(run):
    n0 = abi.lbfd_kernel_launches()
    run()
    return abi.lbfd_kernel_launches() - n0


@pytest.mark.parametrize("lat,dims,precision,mrt,least", CASES)
def test_short_calls(lat, dims, precision, mrt, least):
    kw = _options(lat, precision, mrt)
    with lb.Simulation(lat, dims, 0.9, 40.0, 8, **kw) as a, lb.Simulation(lat, dims, 0.9, 40.0, 8, **kw) as b:
        assert _launches(lambda: a.step(least)) == 1
        assert _launches(lambda: a.step(least - 1)) == least - 1
        assert _launches(lambda: a.step(least)) == 1
        assert a.kernel(least) in ("k_step_resident", abi.KERNEL_NAMES[abi.KERNEL_SMALL])
        assert a.kernel(least - 1) == a.kernel(1)
        for _ in range(3 * least - 1):
            b.step(1)
        assert np.array_equal(a.get_f(), b.get_f())


@pytest.mark.parametrize("lat,dims,precision,mrt,least", CASES)
def test_short_runs_between_samples(lat, dims, precision, mrt, least):
    kw = dict(_options(lat, precision, mrt), modes=[(1, 0, 0)])
    every = least - 1  # samples of 2 launches at 0, every, ..., then the runs between them
    with lb.Simulation(lat, dims, 0.9, 40.0, 8, sample_every=every, **kw) as a, \
            lb.Simulation(lat, dims, 0.9, 40.0, 8, **kw) as b:
        assert _launches(lambda: a.step(3 * every)) == 3 * (2 + every)
        for t in range(3 * every):
            if t % every == 0:
                b.sample()
            b.step(1)
        oa, ob = a.observables(), b.observables()
        assert oa["n_samples"] == ob["n_samples"] == 3
        for k in oa:
            assert np.array_equal(np.asarray(oa[k]), np.asarray(ob[k])), k
        assert np.array_equal(a.get_f(), b.get_f())


def test_short_calls_of_a_sampled_lattice():
    """Calls shorter than a shared launch and than the sampling interval: the sums of the separate pass."""
    kw = dict(lattice_id=3, modes=[(1, 0, 0), (0, 1, 1)])
    with lb.Simulation(lb.D3Q19, (6, 6, 6), 0.9, 40.0, 8, sample_every=4, **kw) as a, \
            lb.Simulation(lb.D3Q19, (6, 6, 6), 0.9, 40.0, 8, **kw) as b:
        for _ in range(5):
            a.step(3)
        for t in range(15):
            if t % 4 == 0:
                b.sample()
            b.step(1)
        oa, ob = a.observables(), b.observables()
        for k in oa:
            assert np.array_equal(np.asarray(oa[k]), np.asarray(ob[k])), k
        assert np.array_equal(a.get_f(), b.get_f())
