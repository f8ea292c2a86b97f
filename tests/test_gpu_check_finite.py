"""Block floating point: columns beyond the lattice (odd widths) do not count as saturated blocks."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_pass", [1, 2, 3])
@pytest.mark.parametrize("dirichlet", [False, True])
@pytest.mark.parametrize("nx", [255, 257])
def test_smooth_run_on_an_odd_width_stays_finite(lbm, nx, dirichlet, per_pass):
    """A smooth velocity field keeps its deviations near their initial size, far below the factor
    of 8 that saturates a block."""
    ny, dx = 256, 1.0 / 256
    lat = lbm.Lattice(nx, ny, dx, dx / 3.2, 1.0, 0.6, dirichlet=dirichlet, storage="ms_bfp", track_displacement=False)
    lat.set_step_fusion(per_pass)
    k = np.pi if dirichlet else 2 * np.pi
    x, y = (np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny
    U = np.zeros((3, 5, ny, nx))
    for c, amp in ((0, 1e-3), (1, -7e-4)):
        U[0, c] = amp * np.outer(np.sin(k * y), np.sin(k * x))
        U[1, c] = amp * k / (nx * dx) * np.outer(np.sin(k * y), np.cos(k * x))
        U[2, c] = amp * k / (ny * dx) * np.outer(np.cos(k * y), np.sin(k * x))
    lat.init(U[0], U[1], U[2], None, None)
    lat.step(600)
    assert lat.finite()
    lat.close()
