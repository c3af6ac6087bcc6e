"""A kernel asked for by step_kernel is the one that runs, by the names of the kernels launched; the library's own
choice takes the twin kernel for rows of odd length."""
import pytest
import torch

import paper_1606_07801_gb300 as lb

pytestmark = pytest.mark.gpu


def _names(lat, dims, precision, kernel):
    with lb.Simulation(lat, dims, 0.9, 40.0, 8, precision=precision, step_kernel=kernel) as s:
        s.step(2)
        s.sync()
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            s.step(2)
            s.sync()
            torch.cuda.synchronize()
    return [e.key for e in prof.key_averages() if "k_step" in e.key]


@pytest.mark.parametrize("lat,dims,precision", [(lb.D2Q9, (301, 200), lb.F32), (lb.D2Q9, (301, 200), lb.F32_F16),
                                                (lb.D3Q19, (47, 33, 31), lb.F32)])
def test_scalar_is_k_step(lat, dims, precision):
    # (a process's first profile may come back empty)
    own = _names(lat, dims, precision, lb.KERNEL_AUTO) or _names(lat, dims, precision, lb.KERNEL_AUTO)
    if not own:
        pytest.skip("no kernel records from the profiler")
    asked = _names(lat, dims, precision, lb.KERNEL_SCALAR)
    assert all("k_step_twin" in n for n in own)
    assert asked and not any("k_step_twin" in n for n in asked)
