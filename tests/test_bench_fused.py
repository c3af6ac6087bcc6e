"""bench.py's "fused" field: by the launches of the sampled run, not by the kernel's name."""
import pytest

import bench


@pytest.mark.parametrize("launches,steps,samples,fused", [
    (22, 20, 2, True),    # a launch a step and a stage 2 a sample
    (24, 20, 2, False),   # the separate pass (D3Q19 from 2^22 sites on, FP64)
    (6, 20, 2, False),    # a small lattice: ten steps a launch
])
def test_fused_by_launches(launches, steps, samples, fused):
    assert bench.sampled_in_step(launches, steps, samples) is fused
