"""Contexts of several host threads: kernels of different sizes side by side."""
import math
import threading

import numpy as np
import pytest

from gpu_common import make_pair, wind_setup
from paper_2211_12867_gb300 import inputs as I
from paper_2211_12867_gb300.icarus import FP32_MIXED, FP64

pytestmark = pytest.mark.gpu
STR = dict(x_min=(0.1, math.pi / 6, 0.0), x_max=(2.0, 5 * math.pi / 6, 2 * math.pi), stretch=True)


@pytest.mark.parametrize("precision", [FP64, FP32_MIXED])
def test_flags_and_features_of_two_block_sizes(precision):
    """one context's kernels take 60 and 91 KB of shared memory, the others' 3"""
    work, errors = [], []
    for nb in ((16, 32, 32),) + ((4, 4, 4),) * 6:
        g, o = make_pair(n=(nb[0], nb[1], 2 * nb[2]), nb=nb, precision=precision, **STR)
        wind_setup(g, o)
        g.inject_cone_cme(0, t_start=100.0, **I.cme_config2(seed=0))
        work.append((g, g.flag_refine(), g.mlp_features()))

    def loop(g, flags, feat):
        try:
            for _ in range(3000):
                same = np.array_equal(g.flag_refine(), flags) and np.array_equal(g.mlp_features(), feat)
                if errors or not same:
                    assert same
                    break
        except Exception as e:
            errors.append(e)
    threads = [threading.Thread(target=loop, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
