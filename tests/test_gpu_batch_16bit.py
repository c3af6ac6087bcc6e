"""D3Q19 members in 16-bit storage, where the last bit of an FP32 sum decides the stored value: every tile order gives
the lattice stepped alone, over enough steps for a difference to spread, in members of tens of thousands of sites."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walk", [lb.WALK_PARAM, lb.WALK_PER_TILE, lb.WALK_STRIDED])
@pytest.mark.parametrize("precision", [lb.F32_F16, lb.F32_BF16])
def test_members_equal_the_lattice_alone(precision, walk):
    dims = [(33, 40, 36), (48, 31, 40), (20, 21, 22), (70, 30, 29), (5, 64, 3)]
    specs = [{"dims": d, "tau": 0.7 + 0.1 * k, "rho_mean": 0.6 + 40.0 * k, "seed": 11 + k, "lattice_id": k}
             for k, d in enumerate(dims)]
    with lb.Ensemble(lb.D3Q19, specs, precision=precision) as e:
        e.plan(2, 8, 0, walk)
        e.step(150)
        got = [e.get_f(m) for m in range(len(dims))]
    for m, sp in enumerate(specs):
        with lb.Simulation(lb.D3Q19, sp["dims"], sp["tau"], sp["rho_mean"], sp["seed"], precision=precision,
                           lattice_id=m) as s:
            s.step(150)
            np.testing.assert_array_equal(got[m], s.get_f().reshape(19, -1))
