"""Every stage tile the library picks by itself, and the longest segments: the
grids are the smallest on which its cost model (152 SMs) takes the tile."""
import math

import numpy as np
import pytest

from gpu_common import make_pair, rel_linf, wind_setup
from paper_2211_12867_gb300.icarus import FP32_MIXED, FP64

pytestmark = pytest.mark.gpu
STR = dict(x_min=(0.1, math.pi / 6, 0.0), x_max=(2.0, 5 * math.pi / 6, 2 * math.pi), stretch=True)

# tile, cells and number of the blocks; "64": segments of 64 planes
PICKED_FP64 = [("4x32", (6, 4, 4), (1, 1, 1)), ("6x36", (10, 14, 4), (1, 2, 2)), ("8x8", (10, 6, 4), (4, 1, 2)),
               ("8x12", (10, 10, 10), (4, 2, 1)), ("8x16", (20, 24, 14), (2, 1, 2)), ("8x24", (20, 18, 18), (1, 1, 2)),
               ("8x32", (10, 6, 32), (2, 2, 2)), ("10x24", (10, 10, 22), (8, 1, 1)), ("12x12", (10, 12, 10), (8, 1, 1)),
               ("12x16", (20, 10, 14), (4, 1, 1)), ("12x20", (8, 6, 34), (1, 8, 1)), ("16x16", (10, 14, 14), (8, 1, 1)),
               ("8x12-64", (66, 18, 10), (1, 4, 12))]
PICKED_FP64_TRACER = [("8x12", (10, 4, 10), (2, 8, 1)), ("8x16", (20, 8, 14), (4, 2, 1)), ("8x24", (20, 18, 18), (1, 1, 2)),
                      ("10x24", (10, 10, 22), (8, 1, 1)), ("12x12", (10, 12, 10), (8, 1, 1)),
                      ("12x16", (20, 10, 14), (4, 1, 1)), ("12x20", (8, 6, 34), (1, 8, 1)), ("8x8-64", (66, 20, 6), (1, 4, 12))]
PICKED_FP32 = [("4x32", (6, 4, 4), (1, 1, 1)), ("6x36", (20, 14, 4), (1, 4, 1)), ("8x8", (4, 18, 4), (16, 1, 1)),
               ("8x12", (20, 6, 10), (4, 2, 2)), ("8x16", (12, 10, 14), (2, 8, 1)), ("8x24", (64, 6, 18), (2, 1, 2)),
               ("8x32", (8, 10, 32), (2, 4, 2)), ("10x24", (8, 36, 18), (2, 1, 4)), ("12x12", (10, 10, 18), (16, 1, 1)),
               ("12x16", (20, 10, 40), (2, 2, 1)), ("12x20", (24, 8, 18), (1, 10, 1)), ("16x16", (10, 14, 40), (8, 1, 1)),
               ("8x12-64", (66, 4, 10), (32, 1, 8))]
PICKED_FP32_TRACER = [("8x12", (6, 4, 10), (1, 8, 8)), ("8x16", (24, 4, 14), (8, 1, 2)), ("8x24", (64, 6, 18), (2, 1, 2)),
                      ("12x12", (6, 10, 4), (8, 4, 2)), ("12x16", (20, 10, 40), (2, 2, 1)),
                      ("12x20", (24, 8, 18), (1, 10, 1)), ("8x8-64", (66, 4, 4), (32, 10, 1))]


def _grid(nb, blocks, precision, tracer):
    g, o = make_pair(n=tuple(b * k for b, k in zip(nb, blocks)), nb=nb, precision=precision, tracer=tracer, **STR)
    wind_setup(g, o)
    if tracer:
        X = np.random.default_rng(1).random(g.get_tracer(0).shape)
        g.set_tracer(0, X * g.get_state(0)[:, 0])
        o.set_tracer(g.get_tracer(0))
    return g, o


@pytest.mark.parametrize("tracer,nb,blocks", [pytest.param(t, nb, k, id=f"{name}{'-tracer' * t}") for t, rows in
                                              ((False, PICKED_FP64), (True, PICKED_FP64_TRACER)) for name, nb, k in rows])
def test_fp64_tiles_against_the_oracle(tracer, nb, blocks):
    """the parity tests' bar of the first steps, 1e-12"""
    g, o = _grid(nb, blocks, FP64, tracer)
    g.step(2)
    o.advance(2)
    assert rel_linf(g.get_state(0), o.get_state()).max() < 1e-12
    if tracer:
        a, b = g.get_tracer(0), o.get_tracer()
        assert np.abs(a.reshape(b.shape) - b).max() < 1e-12 * np.abs(b).max()


@pytest.mark.parametrize("tracer,nb,blocks", [pytest.param(t, nb, k, id=f"{name}{'-tracer' * t}") for t, rows in
                                              ((False, PICKED_FP32), (True, PICKED_FP32_TRACER)) for name, nb, k in rows])
def test_fp32_tiles_have_the_same_bits(tracer, nb, blocks):
    states = []
    for tile in ((0, 0, 0), (8, 8, 1), (4, 32, 5)):
        g, _ = _grid(nb, blocks, FP32_MIXED, tracer)
        g.set_tile(*tile)
        g.step(3)
        states.append((g.get_state(0), g.dt()) + ((g.get_tracer(0),) if tracer else ()))
    for s in states[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(s, states[0]))


@pytest.mark.parametrize("tracer", [False, True])
@pytest.mark.parametrize("segment", [1, 5, 63, 64, 65, 66])
def test_segments_of_a_long_block(segment, tracer):
    """66 planes; the factors of at most 64 are staged at once"""
    nb, blocks = (66, 10, 14), (1, 1, 2)
    g, o = _grid(nb, blocks, FP64, tracer)
    g.set_tile(8, 8, segment)
    g.step(2)
    o.advance(2)
    assert rel_linf(g.get_state(0), o.get_state()).max() < 1e-12
    states = []
    for seg in (3, segment):
        f, _ = _grid(nb, blocks, FP32_MIXED, tracer)
        f.set_tile(12, 20, seg)
        f.step(3)
        states.append(f.get_state(0))
    assert np.array_equal(*states)
