"""Caller-owned buffers that start on any multiple of a value: the same state bit for bit as in the library's own
buffers, and the same sampled sums, in every kernel that reads vectors of a row."""
import numpy as np
import pytest
import torch

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import abi, synth
from tests.test_gpu_fused_sampling import _check_sums

pytestmark = pytest.mark.gpu

TORCH = {lb.F64: torch.float64, lb.F32: torch.float32, lb.F32_F16: torch.float16, lb.F32_BF16: torch.bfloat16}
# lattice, dims, precision, moment-space: above the smallest sizes, rows of whole vectors of four
CASES = [(lb.D1Q3, (1 << 19,), lb.F32, False), (lb.D1Q3, (1 << 19,), lb.F32_F16, False), (lb.D1Q3, (100000,), lb.F64, False),
         (lb.D2Q9, (1024, 512), lb.F32, False), (lb.D2Q9, (512, 300), lb.F32_BF16, False),
         (lb.D3Q19, (64, 32, 33), lb.F32, False), (lb.D3Q19, (128, 64, 64), lb.F32_F16, False),
         (lb.D1Q3, (1 << 19,), lb.F32, True), (lb.D3Q19, (64, 32, 33), lb.F32, True)]


class _Shifted(lb.Simulation):
    """A simulation whose buffers start `shift` values into two torch tensors."""

    def __init__(self, shift, *a, **kw):
        create, keep = abi.lbfd_create_ex, []

        def moved(o):
            n = lb.Q_OF[o.lattice] * o.dims[0] * o.dims[1] * o.dims[2]
            for k, s in enumerate(shift):
                keep.append(torch.empty(n + 8, dtype=TORCH[o.precision], device="cuda"))
                o.f_dev[k] = keep[-1].data_ptr() + s * keep[-1].element_size()
            return create(o)

        abi.lbfd_create_ex = moved
        try:
            super().__init__(*a, **kw)
        finally:
            abi.lbfd_create_ex = create
        self._keep.extend(keep)


@pytest.mark.parametrize("shift", [(1, 1), (2, 2), (0, 3), (4, 2)])
@pytest.mark.parametrize("kernel", [lb.KERNEL_AUTO, lb.KERNEL_VEC])
@pytest.mark.parametrize("lat,dims,precision,mrt", CASES)
def test_buffers_at_any_value(lat, dims, precision, mrt, kernel, shift):
    if mrt and kernel != lb.KERNEL_AUTO:
        pytest.skip("moment-space handles have one kernel")
    Q, N = lb.Q_OF[lat], int(np.prod(dims))
    modes = [(1, 0, 0), (2, 0, 0)]
    taus = [0] + [0.7 + 0.03 * a for a in range(1, Q)] if mrt else None
    kw = dict(precision=precision, tau_moments=taus, modes=modes, init=lb.INIT_NONE, step_kernel=kernel, sample_every=3)
    f0 = synth.random_populations(Q, N, 40.0, 0.3, seed=N)
    with lb.Simulation(lat, dims, 0.9, 40.0, 8, **kw) as s:
        s.set_f(f0)
        states = [s.get_f()]
        s.step(3)
        states.append(s.get_f())
        s.step(2)
        want = s.get_f()
    with _Shifted(shift, lat, dims, 0.9, 40.0, 8, **kw) as s:
        s.set_f(f0)
        s.step(5)
        ob = s.observables()
        got = s.get_f()
    assert np.array_equal(got, want)
    _check_sums(ob, states, 40.0, modes, dims)
