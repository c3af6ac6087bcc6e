"""Read-out of ensemble members: pieces that end inside a population and at its end, every storage format."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb

pytestmark = pytest.mark.gpu


# values of a member against a piece of 2^17 FP32, 2^18 16-bit or 2^16 FP64 values: below, equal to and above one
@pytest.mark.parametrize("precision", [lb.F32, lb.F64, lb.F32_F16, lb.F32_BF16])
@pytest.mark.parametrize("lattice,dims", [(lb.D2Q9, (7, 5)), (lb.D2Q9, (129, 131)), (lb.D2Q9, (301, 200)),
                                          (lb.D1Q3, (65536,)), (lb.D3Q19, (32, 16, 27))])
def test_members_read_out_in_pieces(lattice, dims, precision):
    specs = [{"dims": dims, "tau": 0.9, "rho_mean": 40.0 + k, "seed": 5 + k} for k in range(2)]
    ens = lb.Ensemble(lattice, specs, precision=precision)
    rng = np.random.default_rng(3)
    q = lb.Q_OF[lattice]
    for m, s in enumerate(specs):
        f = rng.uniform(0.5, 3.0, size=(q, int(np.prod(dims))))
        ens.set_f(m, f)
        sim = lb.Simulation(lattice, dims, s["tau"], s["rho_mean"], s["seed"], precision=precision)
        sim.set_f(f)
        # the same conversions of the same stored values: equal to the bit
        np.testing.assert_array_equal(ens.get_f(m), sim.get_f().reshape(q, -1))
