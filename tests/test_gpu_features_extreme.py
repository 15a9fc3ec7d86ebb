"""Pre-flagger features of leaves with infinite or zero values in a cell: the
infinities and NaN of the same operations in IEEE arithmetic."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_2211_12867_gb300.icarus import BC_PERIODIC, FP32_MIXED, FP64, Icarus

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [FP64, FP32_MIXED])
@pytest.mark.parametrize("v,x", [(0, 0.0), (0, -0.0), (0, np.inf), (1, np.inf), (1, -np.inf), (4, np.inf), (4, -np.inf),
                                 (5, np.inf), (0, np.nan), (4, np.nan), (1, 1e30), (4, 1e30)])
def test_one_extreme_cell(v, x, precision):
    g = Icarus(n_cells=(8, 8, 8), block=(8, 8, 8), geometry=1, x_min=(0.0, 0.0, 0.0), x_max=(1.0, 1.0, 1.0),
               bc_lo=(BC_PERIODIC,) * 3, bc_hi=(BC_PERIODIC,) * 3, precision=precision)
    U = np.zeros((1, 8, 8, 8, 8))
    U[:] = np.array([1.0, 0.1, 0.2, 0.3, 2.0, 0.1, 0.2, 0.3])[:, None, None, None]
    U[0, v, 3, 4, 5] = x
    g.set_state(0, U)
    F = g.mlp_features()[0]   # fills the ghost cells
    with np.errstate(all="ignore"):
        ref = np.asarray(M.features_from_padded(g.get_padded(0, 0), g.desc.gamma), dtype=np.float32)
    assert np.array_equal(np.isnan(F), np.isnan(ref)) and np.array_equal(np.isinf(F), np.isinf(ref))
    ok = np.isfinite(ref)
    assert np.allclose(F[ok], ref[ok], rtol=2.0 ** -22, atol=1e-12)
