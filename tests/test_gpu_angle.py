"""The FP64 Box-Muller angle on the GPU over all 2^24 arguments, relative to the size of the cosine and the sine
(small next to the axes).

Tolerance: the angle 4 2^-53 (tests/test_bm64_host.py), the radius 1.64 2^-53 and the product 2^-53; NumPy's
logarithm, square root, argument, cosine and product together 4 2^-53."""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import abi

pytestmark = pytest.mark.gpu


def test_angle_relative_over_all_arguments():
    k = np.arange(2**24, dtype=np.uint32)
    r0 = np.uint32(0x12345678)
    z = abi.lbfd_box_muller_probe(lb.F64, np.stack([np.full_like(k, r0), k << np.uint32(8)], 1)).reshape(-1, 2)
    rad = np.sqrt(-2.0 * np.log((float(r0 >> 8) + 0.5) * 2.0**-24))
    turn = 4.0 * (k.astype(np.float64) + 0.5) * 2.0**-24     # quarter turns, exact
    near = np.rint(turn)
    rest = 0.5 * np.pi * (turn - near)
    c, s, q = np.cos(rest), np.sin(rest), near.astype(int) % 4
    for got, want in ((z[:, 0], np.choose(q, [c, -s, -c, s])), (z[:, 1], np.choose(q, [s, c, -s, -c]))):
        assert np.max(np.abs(got / (rad * want) - 1.0)) <= 11 * 2.0**-53
