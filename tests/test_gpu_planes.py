"""Checkpoints hold a leaf's variables one after the other, the device a cell's
side by side: the planes that go between them."""
import math
import os
import subprocess
import sys

import numpy as np
import pytest

from gpu_common import make_pair, wind_setup
from paper_2211_12867_gb300.icarus import FP32_MIXED, FP64

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
STR = dict(x_min=(0.1, math.pi / 6, 0.0), x_max=(2.0, 5 * math.pi / 6, 2 * math.pi), stretch=True)


# the smallest block, ragged ones, large ones
@pytest.mark.parametrize("precision", [FP64, FP32_MIXED])
@pytest.mark.parametrize("n,nb", [((4, 4, 4), (4, 4, 4)), ((12, 6, 10), (6, 6, 10)), ((128, 60, 180), (64, 60, 60))])
def test_planes_of_a_checkpoint(n, nb, precision, tmp_path):
    g, o = make_pair(n=n, nb=nb, precision=precision, tracer=True, **STR)
    wind_setup(g, o)
    g.set_tracer(0, np.random.default_rng(0).random(g.get_tracer(0).shape))
    g.step(2)
    path = str(tmp_path / "a.ck")
    g.save(path)
    leaves, P = g.n_leaves(0), tuple(b + 4 for b in nb)
    real = np.float32 if precision == FP32_MIXED else np.float64
    raw = np.fromfile(path, dtype=np.uint8)
    size = leaves * 9 * math.prod(P) * real().itemsize
    U = raw[-size - 4:-4].copy().view(real).reshape((leaves, 9) + P)   # four bytes: no pre-flagger parameters
    assert np.array_equal(U[:, :8, 2:-2, 2:-2, 2:-2], g.get_state(0))
    assert np.array_equal(U[:, 8, 2:-2, 2:-2, 2:-2], g.get_tracer(0).reshape(U[:, 8, 2:-2, 2:-2, 2:-2].shape))
    for k in range(leaves):
        assert np.array_equal(U[k, :8], g.get_padded(0, k))
    h, _ = make_pair(n=n, nb=nb, precision=precision, tracer=True, **STR)
    h.load(path)
    for k in range(leaves):
        assert np.array_equal(U[k, :8], h.get_padded(0, k))
    assert np.array_equal(g.get_tracer(0), h.get_tracer(0))


def test_memory_of_a_checkpoint(tmp_path):
    """saving and loading take the state once more on the host, whatever the
    number of threads"""
    code = f"""
import resource, sys
sys.path.insert(0, {HERE!r})
import conftest
from gpu_common import make_pair, wind_setup
g, o = make_pair(n=(128, 60, 180), nb=(64, 60, 180), precision=1)
wind_setup(g, o)
del o
g.step(1)
state = 2 * 68 * 64 * 184 * 32
peak = lambda: resource.getrusage(resource.RUSAGE_SELF).ru_maxrss * 1024
now = lambda: int(open('/proc/self/statm').read().split()[1]) * resource.getpagesize()
keep = bytearray(b'x') * max(peak() - now(), 1)   # fills what the set-up has given back
before = peak()
g.save({str(tmp_path / 'a.ck')!r})
g.load({str(tmp_path / 'a.ck')!r})
print((peak() - before) / state)
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, OMP_NUM_THREADS="16"))
    assert r.returncode == 0, r.stderr
    assert float(r.stdout.split()[-1]) < 2.0, r.stdout
