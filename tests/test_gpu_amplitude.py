"""The FP64 noise amplitude is the correctly rounded square root.

Global noise on an empty line at tau = 1 leaves f_1 = w_1 sigma T_1 alone, sigma = sqrt(rho_mean): exact
arithmetic on the drawn variates says what it is to the last bit for every rho_mean (T_+- = +-sqrt3 z^1 + sqrt2 z^2,
one product and one multiply-add, as the step forms it)."""
import math
from fractions import Fraction

import numpy as np
import pytest

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import abi

pytestmark = pytest.mark.gpu

N, SEED = 4, 77


def _rhos():
    g = np.random.default_rng(5)
    r = list(np.exp2(g.uniform(-40, 40, 2500))) + list(np.exp2(g.uniform(-990, 990, 300)))
    for edge in (2.0**-900, 2.0**900):  # where the general square root takes over
        for k in (-2, -1, 0, 1, 2):
            v = edge
            for _ in range(abs(k)):
                v = math.nextafter(v, math.inf if k > 0 else 0.0)
            r.append(v)
    return r + [0.0, 5e-324, 1e-310, 1.0, 4.0, 2.0, 1.7e308]


def test_amplitude_is_the_rounded_square_root():
    z = abi.lbfd_noise_draw(lb.F64, lb.GAUSSIAN, SEED, 0, 0, 0, N, 2)
    r3, r2 = Fraction(math.sqrt(3.0)), Fraction(math.sqrt(2.0))
    T = []
    for s in range(N):
        even = Fraction(float(r2 * Fraction(z[s, 1])))
        T.append([float(r3 * Fraction(z[s, 0]) + even), float(-r3 * Fraction(z[s, 0]) + even)])
    w = 1 / 6
    bad = []
    for rho in _rhos():
        with lb.Simulation(lb.D1Q3, (N,), 1.0, rho, SEED, precision=lb.F64, noise_mode=lb.NOISE_GLOBAL,
                           init=lb.INIT_NONE) as s:
            s.set_f(np.zeros((3, N)))
            s.step(1)
            f = s.get_f()
        ws = Fraction(w * math.sqrt(rho))
        for x in range(N):
            want = [float(ws * Fraction(t)) for t in T[x]]
            got = [f[1, (x + 1) % N], f[2, (x - 1) % N]]
            if got != want:
                bad.append((rho, x, got, want))
    assert not bad, (len(bad), bad[:3])
