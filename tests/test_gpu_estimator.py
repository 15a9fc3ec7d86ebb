"""The estimator's cluster of four slabs a leaf and its comparisons near the
thresholds: the oracle's flags bit for bit on the cells the device holds."""
import math

import numpy as np
import pytest

from gpu_common import make_pair, wind_setup
from paper_2211_12867_gb300 import inputs as I
from paper_2211_12867_gb300.icarus import FP32_MIXED, FP64

pytestmark = pytest.mark.gpu
STR = dict(x_min=(0.1, math.pi / 6, 0.0), x_max=(2.0, 5 * math.pi / 6, 2 * math.pi), stretch=True)


# more leaves than are resident at once, which are done after their gate test;
# with 6 and 10 planes the last slab is empty or short
@pytest.mark.parametrize("precision", [FP64, FP32_MIXED])
@pytest.mark.parametrize("nb0", [4, 6, 10])
def test_leaves_with_closed_gates(nb0, precision):
    g, o = make_pair(n=(8 * nb0, 64, 128), nb=(nb0, 4, 4), precision=precision, **STR)
    wind_setup(g, o)
    n = g.n_leaves(0)
    for _ in range(3):
        assert np.array_equal(g.flag_refine(), np.full(n, -1))   # no background recorded
    g.inject_cone_cme(0, t_start=100.0, **I.cme_config2(seed=0))
    o.snapshot_vbg()
    for _ in range(3):
        assert np.array_equal(g.flag_refine(dv=1e9), np.full(n, -1))
    # the gate of one cell open in every third leaf, in another slab each time
    U = g.get_state(0)
    for leaf in range(0, n, 3):
        U[leaf, 1, (leaf // 3) % nb0, 1, 2] *= 1.7
    g.set_state(0, U)
    o.set_state(g.get_state(0))
    flags = g.flag_refine()
    for k in range(n):
        o.set_padded(k, g.get_padded(0, k))
    assert np.array_equal(flags, o.flag()) and (flags[::3] >= 0).any()
