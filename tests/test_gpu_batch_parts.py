"""Batched members that step in parts on streams of their own: every member still equals the lattice stepped
alone, for more members than a launch takes."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb

pytestmark = pytest.mark.gpu


# 2 parts; members of a launch's limit of 112, one above it, twice it and one above that
@pytest.mark.parametrize("count", [1, 2, 112, 113, 224, 225])
def test_ensemble_parts(count):
    rng = np.random.default_rng(count)
    specs = [{"dims": (int(rng.integers(30, 70)), int(rng.integers(30, 70))), "tau": 0.8, "rho_mean": 30.0 + m,
              "seed": m, "lattice_id": m} for m in range(count)]
    specs[-1]["dims"] = (401, 380)  # above 2^17 sites in all, and most of them in one member
    ens = lb.Ensemble(lb.D2Q9, specs)
    ens.plan(2, 8, 0, lb.WALK_PARAM)
    ens.step(21)  # a captured chunk and a rest
    for m in {0, count // 2, max(count - 2, 0), count - 1}:
        sp = specs[m]
        sim = lb.Simulation(lb.D2Q9, sp["dims"], sp["tau"], sp["rho_mean"], sp["seed"], lattice_id=sp["lattice_id"])
        sim.step(21)
        np.testing.assert_array_equal(ens.get_f(m), sim.get_f().reshape(9, -1))
