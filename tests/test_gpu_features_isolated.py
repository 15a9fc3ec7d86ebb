"""Pre-flagger features of cells far below neighbours that nearly agree: the
differences cancel, and the cell's magnitude raises what is left of them."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_2211_12867_gb300.icarus import BC_PERIODIC, FP32_MIXED, FP64, Icarus

pytestmark = pytest.mark.gpu


# speeds that agree to the last bit, to FP32's and to a few FP32 bits; the cells'
# own from a little to far below; pressures likewise
@pytest.mark.parametrize("precision", [FP64, FP32_MIXED])
@pytest.mark.parametrize("var", [1, 4])
@pytest.mark.parametrize("spread", [0.0, 1e-7, 1e-6, 1e-3])
@pytest.mark.parametrize("low", [0.6, 0.3, 1e-2, 1e-4, 1e-6, 1e-9, 1e-12, 0.0])
def test_isolated_low_cells(low, spread, var, precision):
    g = Icarus(n_cells=(12, 12, 12), block=(12, 12, 12), geometry=1, x_min=(0.0, 0.0, 0.0), x_max=(1.0, 1.0, 1.0),
               bc_lo=(BC_PERIODIC,) * 3, bc_hi=(BC_PERIODIC,) * 3, precision=precision, p_floor=0.0)
    rng = np.random.default_rng(8)
    shape = (12, 12, 12)
    rho = rng.integers(4, 9, shape).astype(float)
    own = 1.0 + spread * rng.random(shape)
    i = np.indices(shape)
    own = np.where(((i % 4) == 1).all(axis=0), low, own)
    v, p = (own, np.full(shape, 0.25)) if var == 1 else (np.ones(shape), 0.25 * np.maximum(own, 1e-3))
    U = np.zeros((1, 8) + shape)
    U[0, 0], U[0, 1] = rho, rho * v
    U[0, 4] = p / (g.desc.gamma - 1.0) + 0.5 * rho * v * v
    g.set_state(0, U)
    F = g.mlp_features()[0]
    ref = M.features_from_padded(g.get_padded(0, 0), g.desc.gamma)
    # the final rounding (2^-24) and both sides' own errors, at most as much
    assert np.allclose(F, ref, rtol=2.0 ** -23, atol=0.0), np.abs(F / ref - 1).max()
