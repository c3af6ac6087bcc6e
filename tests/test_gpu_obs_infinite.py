"""FP64 observables of a state that holds an infinite population: the sums it enters are infinite, the others are
what they are without it."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import synth

pytestmark = pytest.mark.gpu


# registers (D1Q3, D2Q5, D2Q9) and tiles (D3Q19)
@pytest.mark.parametrize("lat,dims", [(lb.D1Q3, (1000,)), (lb.D2Q5, (30, 17)), (lb.D2Q9, (40, 21)), (lb.D3Q19, (9, 8, 7))])
def test_one_infinite_population(lat, dims):
    Q, N = lb.Q_OF[lat], int(np.prod(dims))
    f = synth.random_populations(Q, N, 40.0, 0.3, seed=N)
    f[1, N // 2] = np.inf
    with lb.Simulation(lat, dims, 0.9, 40.0, 8, precision=lb.F64, init=lb.INIT_NONE) as s:
        s.set_f(f)
        s.sample()
        ob = s.observables()
    rho = f.sum(0)
    # N products of FP64 numbers of one sign in any order: relative N 2^-53
    tol = dict(rtol=N * 2.0**-52, atol=0)
    np.testing.assert_allclose(ob["sum_rho"], rho.sum(), **tol)
    np.testing.assert_allclose(ob["sum_rho2"], (rho * rho).sum(), **tol)
    np.testing.assert_allclose(ob["sum_f"], f.sum(1), **tol)
    np.testing.assert_allclose(ob["sum_ff"], [[(a * b).sum() for b in f] for a in f], **tol)
