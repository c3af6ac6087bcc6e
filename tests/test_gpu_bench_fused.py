"""The launches that bench.py's "fused" field goes by: D3Q19 samples inside the step below 2^22 sites, by a pass of
its own from there on."""
import pytest

import bench
import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import abi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,dims,precision,fused", [(lb.D3Q19, (128, 128, 128), lb.F32, True),
                                                      (lb.D3Q19, (256, 128, 128), lb.F32, False),
                                                      (lb.D2Q9, (2048, 2048), lb.F32, True),
                                                      (lb.D2Q9, (512, 512), lb.F64, False)])
def test_sampled_run(lat, dims, precision, fused):
    with lb.Simulation(lat, dims, 0.9, 40.0, 8, precision=precision, modes=[(1, 0, 0)], sample_every=5) as s:
        n0 = abi.lbfd_kernel_launches()
        s.step(10)
        assert bench.sampled_in_step(abi.lbfd_kernel_launches() - n0, 10, 2) is fused
