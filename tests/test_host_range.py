"""Host memory that the packing kernel may write itself: page-locked pieces
without a gap (the rule alone, over pieces made up here; no GPU)."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2211_12867_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "host_range.h"
// arguments: start, bytes, then (start, bytes, same address) of each piece
int main(int n, char **a) {
  auto find = [&](uintptr_t p, PinnedPiece *q) {
    for (int k = 3; k + 2 < n; k += 3) {
      const uintptr_t s = atol(a[k]);
      const size_t b = atol(a[k + 1]);
      if (p >= s && p < s + b) {
        q->start = s;
        q->bytes = b;
        q->same_address = a[k + 2][0] == '1';
        return true;
      }
    }
    return false;
  };
  printf("%d", (int)pinned_throughout(atol(a[1]), atol(a[2]), find));
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_range")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")], check=True)
    return lambda *a: subprocess.run([str(d / "main"), *map(str, a)], check=True, capture_output=True).stdout == b"1"


def test_pieces(rule):
    one = (4096, 8192, 1)
    assert rule(4096, 8192, *one) and rule(5000, 64, *one) and rule(4096, 1, *one)
    assert not rule(4096, 8193, *one) and not rule(4095, 8, *one) and not rule(12288, 8, *one)
    assert not rule(4096, 64)                                           # pageable
    assert not rule(4096, 64, 4096, 8192, 0)                            # elsewhere on the device
    assert rule(4096, 16384, 4096, 8192, 1, 12288, 8192, 1)             # two pieces side by side
    assert not rule(4096, 16384, 4096, 4096, 1, 16384, 4096, 1)         # both ends, and a gap between them
    assert not rule(4096, 16384, 4096, 8192, 1, 12288, 8192, 0)


@pytest.mark.gpu
def test_state_into_registered_memory():
    """one registered piece, and several side by side"""
    import math

    import numpy as np
    import torch
    from gpu_common import make_pair, wind_setup
    g, o = make_pair(n=(24, 8, 20), nb=(12, 8, 10), x_min=(0.1, math.pi / 6, 0.0),
                     x_max=(2.0, 5 * math.pi / 6, 2 * math.pi), stretch=True)
    wind_setup(g, o)
    plain = g.get_state(0)
    rt = torch.cuda.cudart()
    page = 65536
    for pieces in (1, 3):
        step = -(-plain.nbytes // (pieces * page)) * page
        raw = np.zeros(pieces * step + page, dtype=np.uint8)
        at = -raw.ctypes.data % page
        for k in range(pieces):
            assert int(rt.cudaHostRegister(raw.ctypes.data + at + k * step, step, 0)) == 0
        out = raw[at:at + plain.nbytes].view(np.float64).reshape(plain.shape)
        assert np.array_equal(g.get_state(0, out=out), plain) and not raw[at + plain.nbytes:].any()
        for k in range(pieces):
            assert int(rt.cudaHostUnregister(raw.ctypes.data + at + k * step)) == 0
