"""The size-dependent paths of the kernels at the sizes where they change:
stage tiles, estimator slabs, features, training groups, physical corners and
the read-back of the state."""
import math

import numpy as np
import pytest

from gpu_common import make_pair, rel_linf, wind_setup
from oracle import mlp as M
from paper_2211_12867_gb300 import inputs as I
from paper_2211_12867_gb300.icarus import BC_OUTFLOW, BC_PERIODIC, BC_REFLECT, FP32_MIXED, FP64

from test_gpu_mlp import _grad_magnitudes

pytestmark = pytest.mark.gpu
STR = dict(x_min=(0.1, math.pi / 6, 0.0), x_max=(2.0, 5 * math.pi / 6, 2 * math.pi), stretch=True)


# blocks at and around the edges of the tiles (theta x phi): smaller than every
# tile, exact, one row or column more, several ragged tiles; 4 to 66 planes
@pytest.mark.parametrize("nb", [(4, 4, 4), (6, 8, 12), (12, 8, 16), (10, 12, 18), (4, 16, 16), (8, 18, 34),
                                (66, 10, 22)])
def test_chosen_tile_and_segment(nb):
    """FP64 against the oracle (first-step bar of the parity tests: 1e-12);
    FP32 the same bits whatever the tile."""
    n = (2 * nb[0], nb[1], 2 * nb[2])
    g, o = make_pair(n=n, nb=nb, **STR)
    wind_setup(g, o)
    g.step(2)
    o.advance(2)
    assert rel_linf(g.get_state(0), o.get_state()).max() < 1e-12
    states = []
    for tile in ((0, 0, 0), (8, 8, 0), (12, 20, 5)):
        f, p = make_pair(n=n, nb=nb, precision=FP32_MIXED, tracer=True, **STR)
        wind_setup(f, p)
        f.set_tracer(0, 0.25 * f.get_state(0)[:, 0])
        f.set_tile(*tile)
        f.step(3)
        states.append((f.get_state(0), f.get_tracer(0), f.dt()))
    for s in states[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(s, states[0]))


# four slabs of 1 to 4 planes, some of them empty; (8, 40, 96) has no room for
# its planes in shared memory
@pytest.mark.parametrize("precision", [FP64, FP32_MIXED])
@pytest.mark.parametrize("nb", [(4, 6, 8), (6, 12, 12), (10, 4, 14), (14, 8, 6), (8, 40, 96)])
def test_estimator_flags(nb, precision):
    """bit for bit the oracle's flags on the blocks the device filled, at
    thresholds between and on the values E takes"""
    g, o = make_pair(n=(2 * nb[0], nb[1], 2 * nb[2]), nb=nb, precision=precision, **STR)
    wind_setup(g, o)
    g.inject_cone_cme(0, t_start=100.0, **I.cme_config2(seed=0))
    o.snapshot_vbg()
    U = g.get_state(0)
    rng = np.random.default_rng(3)
    # faster plasma in half of the cells, rougher from leaf to leaf, some near-vacuum
    for leaf in range(len(U)):
        f = 1.0 + (0.3 if leaf % 2 else 0.003) * rng.random(U.shape[2:])
        U[leaf, :, ...] *= f
        U[leaf, 1] *= np.where(rng.random(U.shape[2:]) < 0.5, 1.4, 1.0)
        U[leaf, 4] += np.where(rng.random(U.shape[2:]) < 0.02, 1e-7, 1.0) * U[leaf, 1] ** 2 / U[leaf, 0]
    g.set_state(0, U)
    o.set_state(g.get_state(0))
    for crit in (dict(e_refine=0.1, e_coarsen=0.0125), dict(e_refine=0.01, e_coarsen=0.001, eps=0.0),
                 dict(e_refine=0.5, e_coarsen=0.2, dv=0.0), dict(e_refine=0.0, e_coarsen=0.0, dv=1e9)):
        crit = dict(dict(eps=0.01, dv=0.5), **crit)
        fg = g.flag_refine(**crit)
        for n in range(o.nleaves):
            o.set_padded(n, g.get_padded(0, n))
        assert np.array_equal(fg, o.flag(**crit)), crit


# sub-cubes of one cell to 100; the last two blocks have no room for three
# planes in shared memory
@pytest.mark.parametrize("precision", [FP64, FP32_MIXED])
@pytest.mark.parametrize("nb", [(4, 4, 4), (8, 4, 12), (12, 20, 8), (8, 40, 40), (4, 8, 180)])
def test_features(nb, precision):
    """features of the padded blocks the device read: FP64 operations on both
    sides, rounded to FP32 at the end (2^-24, doubled for a tie either way)"""
    g, o = make_pair(n=(2 * nb[0], nb[1], nb[2]), nb=nb, precision=precision, **STR)
    wind_setup(g, o)
    g.step(3)
    F = g.mlp_features()
    for n in range(o.nleaves):
        ref = M.features_from_padded(g.get_padded(0, n), 1.5)
        assert np.allclose(F[n], ref, rtol=2.0 ** -22, atol=1e-12), n


# the FP32 mode's sums in float pairs and where they give way to FP64: units in
# which densities are 1e-21, pressures 1e-5 of the energy, speeds of 0 and near
# it, near-uniform and uniform leaves
@pytest.mark.parametrize("kind", ["wind", "si", "cold", "still", "noise", "uniform"])
def test_features_of_fp32_states(kind):
    g, o = make_pair(n=(8, 24, 24), nb=(8, 12, 12), precision=FP32_MIXED, **dict(
        geometry=1, x_min=(0.0, 0.0, 0.0), x_max=(1.0, 1.0, 1.0), omega=0.0, bc_lo=(BC_OUTFLOW,) * 3,
        bc_hi=(BC_OUTFLOW,) * 3))
    rng = np.random.default_rng(4)
    a = {"noise": 2e-7, "uniform": 0.0}.get(kind, 0.1)
    W = 1.0 + a * rng.random((g.n_leaves(0), 8) + g.block)
    W[:, 1] *= 3.0
    W[:, 4] *= 0.2
    if kind == "si":
        W *= np.array([1e-21, 4e5, 4e5, 4e5, 1e-11, 5e-6, 5e-6, 5e-6])[:, None, None, None]
    if kind == "cold":
        W[:, 4] *= np.where(rng.random(W[:, 4].shape) < 0.3, 1e-4, 1.0)
    if kind == "still":
        W[:, 1] *= np.where(rng.random(W[:, 1].shape) < 0.3, 0.0, 1e-12)
        W[0, 1] = 0.0
    g.set_state(0, W, prim=True)
    F = g.mlp_features()
    for n in range(o.nleaves):
        ref = M.features_from_padded(g.get_padded(0, n), g.desc.gamma)
        # the final rounding (2^-24) and both sides' own errors, at most as much
        assert np.allclose(F[n], ref, rtol=2.0 ** -23, atol=0.0), (n, np.abs(F[n] / ref - 1).max())


# groups of 8 samples: a part of one, one, one more, a last group of 1; more
# groups than CTAs
@pytest.mark.parametrize("batch", [1, 7, 8, 9, 1217, 4096])
def test_gradient_of_a_batch(batch):
    g, _ = make_pair(n=(24, 12, 12), nb=(12, 12, 12), **STR)
    rng = np.random.default_rng(batch)
    theta = I.mlp_init(1).astype(np.float32)
    g.mlp_set_params(theta)
    X = rng.uniform(0, 0.3, (batch, 64)).astype(np.float32)
    T = (rng.random(batch) < 0.3).astype(np.float32)
    gg, loss = g.mlp_grad(X, T)
    again, loss2 = g.mlp_grad(X, T)
    assert np.array_equal(gg, again) and loss == loss2
    th, X64, T64 = theta.astype(np.float64), X.astype(np.float64), T.astype(np.float64)
    go = M.grad(th, X64, T64)
    # 1e-5 of the value plus 16 FP32 ulps of the running-error magnitude
    assert np.all(np.abs(gg - go) <= 1e-5 * np.abs(go) + 1e-6 * _grad_magnitudes(th, X64, T64))
    assert abs(loss - M.loss(th, X64, T64)) < 1e-5
    assert np.allclose(g.mlp_predict(X), M.forward(th, X64)[0], rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("batch", [1, 8, 200, 1024, 4096])
def test_batches_in_one_call(batch):
    """the steps of one call overlap their kernels: the same bits as one step a
    call (every sample the same, so that the order of the samples is none)"""
    g, _ = make_pair(n=(24, 12, 12), nb=(12, 12, 12), **STR)
    rng = np.random.default_rng(batch)
    n = min(4 * batch, 8192)
    X = np.repeat(rng.uniform(0, 1.0, (1, 64)), n, axis=0).astype(np.float32)
    theta = I.mlp_init(4).astype(np.float32)
    out = []
    for calls in (1, n // batch):
        g.mlp_set_params(theta)
        g.mlp_dataset_clear()
        g.mlp_dataset_add(X, np.ones(n, dtype=np.float32))
        for _ in range(5):
            for _ in range(calls):
                g.mlp_train(n // calls, 1, batch=batch, lr=1e-2, seed=1)
        out.append(g.mlp_get_params())
    assert np.array_equal(out[0], out[1]) and not np.array_equal(out[0], theta)


@pytest.mark.parametrize("lo,hi", [((BC_REFLECT, BC_OUTFLOW, BC_REFLECT), (BC_OUTFLOW, BC_REFLECT, BC_REFLECT)),
                                   ((BC_OUTFLOW, BC_REFLECT, BC_PERIODIC), (BC_REFLECT, BC_REFLECT, BC_PERIODIC)),
                                   ((BC_PERIODIC, BC_OUTFLOW, BC_OUTFLOW), (BC_PERIODIC, BC_OUTFLOW, BC_REFLECT))])
def test_physical_corners(lo, hi):
    """every ghost cell of a box, corners between boundaries of different
    kinds among them: copies, the same bits"""
    g, o = make_pair(n=(8, 6, 16), nb=(4, 6, 8), geometry=1, x_min=(0.0, 0.0, 0.0), x_max=(1.0, 1.0, 1.0), omega=0.0,
                     bc_lo=lo, bc_hi=hi)
    rng = np.random.default_rng(0)
    W = rng.uniform(0.5, 2.0, (g.n_leaves(0), 8) + g.block)
    g.set_state(0, W, prim=True)
    o.set_state(g.get_state(0))
    g.ghost_fill()
    o.ghost_fill()
    for n in range(o.nleaves):
        assert np.array_equal(g.get_padded(0, n), o.get_padded(n, 0)), n


@pytest.mark.parametrize("hours", [0.0, 0.7, 2.5, 4.1, 30.0])
def test_inner_boundary_with_the_cone(hours):
    """inner ghost cells while the cone opens, is open, closes and is gone:
    the oracle's mask (arc cosines) cell by cell, values to 1e-14"""
    g, o = make_pair(n=(24, 48, 96), nb=(12, 12, 12), **STR)
    wind_setup(g, o)
    cme = dict(I.cme_config2(seed=0), t_start=0.0)
    g.inject_cone_cme(0, **cme)
    o.set_cme(**cme)
    g.set_time(0, I.hours(hours))
    o.t = I.hours(hours)
    g.ghost_fill()
    o.ghost_fill()
    for n, row in enumerate(o.tree()):
        if row[1] == 0:
            a, b = g.get_padded(0, n), o.get_padded(n, 0)
            scale = np.abs(b).max(axis=(1, 2, 3), keepdims=True) + 1e-300
            assert (np.abs(a - b) / scale).max() < 1e-14, n


@pytest.mark.parametrize("precision", [FP64, FP32_MIXED])
def test_state_into_pinned_memory(precision):
    import torch
    g, o = make_pair(n=(24, 8, 20), nb=(12, 8, 10), precision=precision, **STR)
    wind_setup(g, o)
    plain = g.get_state(0)
    pinned = torch.zeros(plain.size + 8, dtype=torch.float64).pin_memory()
    got = g.get_state(0, out=pinned[:plain.size].view(plain.shape).numpy())
    assert np.array_equal(got, plain) and not pinned[plain.size:].any()


WALLS = dict(geometry=1, x_min=(0.0, 0.0, 0.0), x_max=(1.0, 1.0, 1.0), omega=0.0)


# the smallest blocks and ragged ones; all kinds of boundaries and a periodic
# direction two blocks wide
@pytest.mark.parametrize("precision", [FP64, FP32_MIXED])
@pytest.mark.parametrize("nb,kw", [
    ((4, 4, 4), STR), ((6, 4, 10), STR),
    ((4, 4, 4), dict(WALLS, bc_lo=(BC_REFLECT, BC_OUTFLOW, BC_REFLECT), bc_hi=(BC_OUTFLOW, BC_REFLECT, BC_REFLECT))),
    ((4, 6, 8), dict(WALLS, bc_lo=(BC_OUTFLOW, BC_REFLECT, BC_PERIODIC), bc_hi=(BC_REFLECT, BC_REFLECT, BC_PERIODIC))),
    ((8, 4, 6), dict(WALLS, bc_lo=(BC_PERIODIC,) * 3, bc_hi=(BC_PERIODIC,) * 3))])
def test_step_fill_of_all_levels_at_once(nb, kw, precision):
    """random trees of three levels: the bits of steps whose fills go level by
    level over every ghost cell"""
    runs = []
    for direct in (True, False):
        g, o = make_pair(n=tuple(2 * b for b in nb), nb=nb, max_level=3, max_blocks=600, precision=precision,
                         tracer=True, **kw)
        rng = np.random.default_rng(7)
        if "geometry" in kw:
            W = 1.0 + 0.2 * rng.random((g.n_leaves(0), 8) + g.block)
            g.set_state(0, W, prim=True)
        else:
            wind_setup(g, o)
        for _ in range(2):
            f = rng.random(g.n_leaves(0)) < 0.3
            f[np.argmax(g.tree(0)[:, 0])] = True   # the first leaf of the finest level
            g.set_flags(f.astype(np.int8))
            g.regrid()
        U = g.get_state(0)
        U[:, :5] *= 1.0 + 0.02 * rng.random(U[:, :1].shape)
        g.set_state(0, U)
        g.set_tracer(0, U[:, 0] * rng.random(U[:, 0].shape))
        g.set_direct_halo(direct)
        g.step(4)
        assert g.status()[0] & ~2 == 0   # floors may apply (bit 1)
        runs.append((g.tree(0), g.get_state(0), g.get_tracer(0), g.dt()))
    assert runs[0][0][:, 0].max() == 3
    for a, b in zip(*runs):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("nb,kw", [
    ((4, 4, 4), STR), ((6, 4, 10), dict(STR, bc_lo=(3, 1, 0), bc_hi=(1, 2, 0))),
    ((4, 6, 8), dict(WALLS, bc_lo=(BC_OUTFLOW, BC_REFLECT, BC_PERIODIC), bc_hi=(BC_REFLECT, BC_REFLECT, BC_PERIODIC))),
    ((8, 4, 6), dict(WALLS, bc_lo=(BC_PERIODIC,) * 3, bc_hi=(BC_PERIODIC,) * 3))])
def test_full_fill_of_a_tree(nb, kw):
    """every ghost cell of a random tree of three levels against the oracle,
    which fills level by level; 1e-13 of a variable's largest value (the bar of
    the prolonged data of the regrid tests)"""
    g, o = make_pair(n=(2 * nb[0], 2 * nb[1], nb[2]), nb=nb, max_level=3, max_blocks=600, **kw)
    rng = np.random.default_rng(11)
    if "geometry" in kw:
        g.set_state(0, 1.0 + 0.2 * rng.random((g.n_leaves(0), 8) + g.block), prim=True)
        o.set_state(g.get_state(0))
    else:
        wind_setup(g, o)
    for _ in range(2):
        f = rng.random(g.n_leaves(0)) < 0.3
        f[np.argmax(g.tree(0)[:, 0])] = True
        f = f.astype(np.int8)
        g.set_flags(f)
        g.regrid()
        o.regrid(f)
    assert np.array_equal(g.tree(0), o.tree()) and g.tree(0)[:, 0].max() == 3
    U = g.get_state(0)
    U[:, :5] *= 1.0 + 0.02 * rng.random(U[:, :1].shape)
    g.set_state(0, U)
    o.set_state(g.get_state(0))
    g.ghost_fill()
    o.ghost_fill()
    scale = np.abs(U).max(axis=(0, 2, 3, 4))[:, None, None, None] + 1e-300
    for n in range(o.nleaves):
        assert (np.abs(g.get_padded(0, n) - o.get_padded(n, 0)) / scale).max() < 1e-13, n
