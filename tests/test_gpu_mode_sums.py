"""Mode sums of the FP32 sampling pass lose nothing over the tiles of a block.

A uniform state of deviation d = 1 + 2^-21 and the wave vector 0: every site's term is d.  Sums of d over a warp are
exact in FP32 (powers of two), and so are sums of eight warps (24 bits); a sum over more tiles is not, unless it is
carried further.  So |sum d|^2 is (N d)^2 to the last bit."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb

pytestmark = pytest.mark.gpu


# one tile a block and fewer than 16, and more than 16 of them
@pytest.mark.parametrize("dims", [(32, 16, 15), (160, 160, 164), (256, 256, 160)])
@pytest.mark.parametrize("n_modes", [1, 4, 5])
def test_uniform_state(dims, n_modes):
    N = int(np.prod(dims))
    f = np.zeros((19, N))
    f[0], f[1] = 1.0, 2.0**-21
    with lb.Simulation(lb.D3Q19, dims, 0.9, 0.0, 8, precision=lb.F32_F16, init=lb.INIT_NONE,
                       modes=[(0, 0, 0)] * n_modes) as s:
        s.set_f(f)
        s.sample()
        sk = s.observables()["sum_sk"]
    assert np.all(sk == (N * (1.0 + 2.0**-21)) ** 2)
