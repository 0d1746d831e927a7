"""Location on grids whose spacing is no power of two: elements, reference
coordinates and the cell table bit for bit, points on and one ulp beside every
grid plane included."""
import numpy as np
import pytest

import test_gpu_cell_table as case
from test_gpu_cell_table import fsi  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


# the last ones: a significand of all ones, and a spacing beyond the range of the
# reciprocal's route
@pytest.mark.parametrize("h", [(1 / 3, 0.1, 1 / 47), (3e-5, 7e4, 1.1), (1 / 24, 2.0 ** -3, 1 / 31),
                               (np.nextafter(1.0, 0), np.nextafter(0.25, 1), 1e-3),
                               (1e-170, 3e160, 0.7)])
@pytest.mark.parametrize("zero", [True, False])
def test_locate_general_spacings(fsi, oracle, h, zero):
    rng = np.random.default_rng(33)
    N = (9, 13, 6)
    x0 = (0.0, -0.0, 0.0) if zero else (0.3 * h[0], -4.7 * h[1], 1e3 * h[2])
    mesh = fsi.Mesh(N, x0=x0, h=h, device=0)
    grid = oracle.core.Grid(N, x0=x0, h=h)
    case.check(fsi, oracle, mesh, grid, case.edge_points(N, h, x0, rng))
    mesh.close()
