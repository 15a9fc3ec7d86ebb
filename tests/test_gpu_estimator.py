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


def _leaf_E(U, gamma, eps):
    """largest E of a leaf's interior cells from its padded cells, every
    operation rounded on its own in the documented order"""
    msq, bsq = (U[1] * U[1] + U[2] * U[2]) + U[3] * U[3], (U[5] * U[5] + U[6] * U[6]) + U[7] * U[7]
    out = []
    for q in (U[0], (gamma - 1.0) * ((U[4] - 0.5 * msq / U[0]) - 0.5 * bsq)):
        num = den = 0.0
        c = q[2:-2, 2:-2, 2:-2]
        for d in range(3):
            lo, hi = (np.roll(q, k, axis=d)[2:-2, 2:-2, 2:-2] for k in (1, -1))
            t1, t2 = hi - c, c - lo
            d2 = t1 - t2
            s = (np.abs(t1) + np.abs(t2)) + eps * ((np.abs(hi) + 2.0 * np.abs(c)) + np.abs(lo))
            num, den = num + d2 * d2, den + s * s
        out.append(np.sqrt(np.divide(num, den, out=np.zeros_like(den), where=den > 0.0)))
    return np.maximum(*out).max()


def _check_at_the_thresholds(precision, make_state, eps=0.01):
    """Flags with every gate open at, and one ulp below, the largest E of each
    leaf: a cell refines (keeps) its leaf only above the threshold."""
    g, o = make_pair(n=(12, 24, 24), nb=(6, 8, 12), precision=precision, **STR)
    wind_setup(g, o)
    g.inject_cone_cme(0, t_start=100.0, **I.cme_config2(seed=0))
    g.set_state(0, make_state((g.n_leaves(0), 8) + g.block))
    g.ghost_fill()
    E = np.array([_leaf_E(g.get_padded(0, n), g.desc.gamma, eps) for n in range(g.n_leaves(0))])
    assert np.isfinite(E).all() and (E > 0.0).all()
    for e in E:
        for t in (e, np.nextafter(e, 0.0)):
            crit = dict(eps=eps, dv=-1e9)
            assert np.array_equal(g.flag_refine(e_refine=t, e_coarsen=t, **crit), np.where(E > t, 1, -1))
            assert np.array_equal(g.flag_refine(e_refine=1e3, e_coarsen=t, **crit), np.where(E > t, 0, -1))


# a cold stream behind the cone: the pressure is the small difference of the
# energies
@pytest.mark.parametrize("precision", [FP64, FP32_MIXED])
@pytest.mark.parametrize("p_over_e", [1e-3, 1e-5, 1e-7, 1e-8, 1e-9, 1e-10, 1e-11, 1e-12, 1e-13])
def test_thresholds_in_cold_streams(p_over_e, precision):
    def state(shape):
        rng = np.random.default_rng(5)
        U = np.zeros(shape)
        U[:, 0] = 100.0
        U[:, 1] = 800.0 * (1.0 + 0.1 * rng.random(U[:, 0].shape))
        U[:, 2:4] = 20.0 * rng.random(U[:, 2:4].shape)
        U[:, 5:8] = rng.random(U[:, 5:8].shape)
        e = 0.5 * (U[:, 1:4] ** 2).sum(1) / U[:, 0] + 0.5 * (U[:, 5:8] ** 2).sum(1)
        U[:, 4] = e * (1.0 + p_over_e / 0.5 * (1.0 + 1.5e-3 * rng.random(e.shape)))
        return U
    _check_at_the_thresholds(precision, state)


# units in which the squares of densities and pressures leave FP32's normal
# range at either end
@pytest.mark.parametrize("precision", [FP64, FP32_MIXED])
@pytest.mark.parametrize("rough", [1.0, 0.01])
@pytest.mark.parametrize("unit", [1e-30, 1e-24, 1e-22, 1e-21, 1e-20, 1e-19, 1e-18, 1e-16, 1e-12, 1e12, 1e16, 1e18, 1e19,
                                  1e20, 1e22])
def test_thresholds_in_any_unit(unit, rough, precision):
    def state(shape):
        rng = np.random.default_rng(6)
        W = 1.0 + 0.3 * rough * rng.random(shape)
        U = W.copy()
        U[:, 1:4] *= W[:, :1]
        U[:, 4] = 2.0 * W[:, 4] + 0.5 * (U[:, 1:4] ** 2).sum(1) / U[:, 0] + 0.5 * (W[:, 5:8] ** 2).sum(1)
        return U * np.where(np.arange(8) < 5, unit, math.sqrt(unit))[:, None, None, None]
    _check_at_the_thresholds(precision, state)
