"""A block of more cells than one row of CTAs a chunk would cover."""
import numpy as np
import pytest

from paper_2211_12867_gb300.icarus import BC_PERIODIC, Icarus

pytestmark = pytest.mark.gpu


def test_cfl_step_of_one_huge_block():
    """FP64, 69 million cells in a block: more chunks of cells than a grid has
    rows"""
    nb, gamma, cfl = (1020, 264, 256), 1.5, 0.8
    g = Icarus(n_cells=nb, block=nb, geometry=1, x_min=(0.0, 0.0, 0.0), x_max=(1.0, 1.0, 1.0), gamma=gamma, omega=0.0,
               cfl=cfl, bc_lo=(BC_PERIODIC,) * 3, bc_hi=(BC_PERIODIC,) * 3)
    U = np.empty((1, 8) + nb)
    u = (2.0, 0.6, -0.4, 0.2, 3.0, 0.3, 0.2, 0.1)
    for v in range(8):
        U[0, v] = u[v]
    # the last cell decides
    U[0, 1, -1, -1, -1] = 2.0
    U[0, 4, -1, -1, -1] = 4.0
    g.set_state(0, U)
    w, B = np.array([1.0, -0.2, 0.1]), np.array(u[5:])
    b2 = B @ B
    a2 = gamma * (gamma - 1.0) * (4.0 - w @ w - 0.5 * b2) / 2.0
    s = a2 + b2 / 2.0
    rate = sum((abs(w[d]) + np.sqrt(0.5 * (s + np.sqrt(s * s - 2.0 * a2 * B[d] ** 2)))) * nb[d] for d in range(3))
    assert abs(float(np.ravel(g.dt())[0]) * rate / cfl - 1.0) < 1e-13
