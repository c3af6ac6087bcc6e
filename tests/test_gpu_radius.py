"""The FP64 Box-Muller radius on the GPU over all 2^24 arguments, relative to its size (small next to u0 = 1).

Tolerance of the radius: 1.64 2^-53 (tests/test_bm64_host.py), the cosine and the product with it 2.8 2^-53, and
NumPy's logarithm (one unit, halved) and square root 1.5 2^-53 together."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import abi

pytestmark = pytest.mark.gpu


def test_radius_relative_over_all_arguments():
    k = np.arange(2**24, dtype=np.uint32)
    z = abi.lbfd_box_muller_probe(lb.F64, np.stack([k << np.uint32(8), np.zeros_like(k)], 1)).reshape(-1, 2)[:, 0]
    u = (k.astype(np.float64) + 0.5) * 2.0**-24
    want = np.sqrt(-2.0 * np.where(u > 0.5, np.log1p(u - 1.0), np.log(u))) * np.cos(np.pi * 2.0**-24)
    assert np.max(np.abs(z / want - 1.0)) <= 6 * 2.0**-53
