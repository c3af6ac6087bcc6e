"""lbfd_obs_restore without offsets (rho_mean = 0) hands out the totals themselves, infinite ones too."""
import numpy as np

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import abi


def test_infinite_totals_without_offsets():
    Q = 9
    tt = np.arange(1.0, abi.obs_totals_count(Q, 0) + 1)
    tt[0] = tt[1] = tt[2 + 4] = np.inf
    pair = {}
    k = 2 + Q
    for i in range(Q):
        for j in range(i, Q):
            if 4 in (i, j):
                tt[k] = np.inf
            pair[i, j] = pair[j, i] = tt[k]
            k += 1
    acc = abi.lbfd_obs_restore(lb.D2Q9, 0, 0.0, 100, tt)
    assert acc[0] == np.inf and acc[1] == np.inf
    np.testing.assert_array_equal(acc[2:2 + Q], tt[2:2 + Q])
    np.testing.assert_array_equal(acc[2 + Q:].reshape(Q, Q), [[pair[i, j] for j in range(Q)] for i in range(Q)])
