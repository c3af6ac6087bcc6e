"""The FP64 Box-Muller pairs of csrc/bm64.cuh at the edges of its tables.

The radius takes a cell of 1024 per binade of u0 and the angle a quadrant, a
base angle and an odd remainder; the words here sit on both sides of every
cell edge of every binade, next to u0 = 0 and u0 = 1, and on both sides of
every base angle's edges.

Tolerance: the radius is formed in fixed point with 2^-56 and a square root
good to one unit in the last place (relative 2^-52), the angle factors from
three roundings of 2^-54; NumPy's reference adds as much again.  Together
below radius x 2e-15 + 1e-16.
"""
import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import abi

pytestmark = pytest.mark.gpu


def _radius_words():
    k = [np.arange(0, 4096), np.arange(2**24 - 4096, 2**24)]  # next to u0 = 0 and u0 = 1
    for e in range(25):  # K = 2 k + 1 = M 2^(e - 24), M on the cell edges
        m = (1 << 24) + (np.arange(1025) << 14)
        K = np.concatenate([(m >> (24 - e)) + d for d in (-1, 0, 1)]) | 1
        k.append((K[(K > 0) & (K < 2**25)] - 1) // 2)
    return np.unique(np.concatenate(k)).astype(np.uint32) << np.uint32(8)


def _angle_words():
    edge = np.arange(0, 2**24, 2**11, dtype=np.int64)  # base angles are 2^11 apart in k
    k = np.concatenate([edge + d for d in (-1, 0, 1, 1023, 1024)]) % 2**24
    return np.unique(k).astype(np.uint32) << np.uint32(8)


@pytest.mark.parametrize("which", ["radius", "angle"])
def test_pairs_at_table_edges(which):
    g = np.random.default_rng(3)
    r = _radius_words() if which == "radius" else _angle_words()
    other = g.integers(0, 2**32, r.size, dtype=np.uint32)
    r0, r1 = (r, other) if which == "radius" else (other, r)
    z = abi.lbfd_box_muller_probe(lb.F64, np.stack([r0, r1], 1)).reshape(-1, 2)
    u = ((r0 >> np.uint32(8)).astype(np.float64) + 0.5) * 2.0**-24
    rad = np.sqrt(-2.0 * np.where(u > 0.5, np.log1p(u - 1.0), np.log(u)))
    ang = 2.0 * (((r1 >> np.uint32(8)).astype(np.float64) + 0.5) * 2.0**-24)  # in units of pi
    near = np.rint(2.0 * ang)                 # nearest quarter turns, taken off exactly
    rest = np.pi * (ang - 0.5 * near)
    c, s, q = np.cos(rest), np.sin(rest), near.astype(int) % 4
    cos = np.choose(q, [c, -s, -c, s])
    sin = np.choose(q, [s, c, -s, -c])
    tol = rad * 2e-15 + 1e-16
    assert np.all(np.abs(z[:, 0] - rad * cos) <= tol)
    assert np.all(np.abs(z[:, 1] - rad * sin) <= tol)
