"""Batched members that step in parts on streams of their own: every member still equals the lattice stepped
alone, for more members than a launch takes, and large simulations of the server while they move between streams."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from tests.test_gpu_server import _alone, _spec, _submit

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


@pytest.mark.parametrize("solo_sites", [0, 100000])
def test_server_members_move_between_streams(solo_sites):
    """Waves of different lattice types: the large simulations' order changes while they run."""
    shapes = [(lb.D3Q19, (64, 50, 40), 60), (lb.D3Q19, (50, 48, 46), 90), (lb.D2Q9, (400, 301), 70),
              (lb.D1Q3, (150000,), 50), (lb.D3Q19, (20, 21, 22), 35), (lb.D2Q9, (333, 310), 80),
              (lb.D1Q3, (140001,), 45), (lb.D2Q9, (64, 64), 100), (lb.D3Q19, (49, 48, 47), 40)]
    specs = [_spec(lat, dims, steps, k, result=lb.RESULT_F) for k, (lat, dims, steps) in enumerate(shapes)]
    with lb.Server(precision=lb.F32, hbm_budget=1 << 30, passes=4, solo_sites=solo_sites, walk=lb.WALK_PARAM) as srv:
        ids = []
        for sp in specs:
            ids.append(_submit(srv, sp))
            srv.pump(7)
        srv.drain()
        for i, sp in zip(ids, specs):
            np.testing.assert_array_equal(np.asarray(srv.result(i)).reshape(-1), _alone(sp, lb.F32).reshape(-1))
