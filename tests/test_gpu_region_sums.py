"""The region kernel's mass sum beyond FP32's range: a lane's sum is FP32, a
region's is not."""
import numpy as np
import pytest

from paper_1912_09327_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(64, 64), (700, 640), (1027, 1300)])
def test_mass_beyond_fp32_range(nx, ny):
    """A fluid at rest with rho = 2e37 everywhere: a lane's mass of at most 8
    rows x 2 columns (3.2e38) stays within FP32, a region's does not.  Nothing
    in the step is unstable; it changes a density by a few 2^-24 of it and the
    compensated lane sums add as much (1e-5 covers both)."""
    from paper_1912_09327_gb300 import binding as b
    p = wl.Problem("rest", np.zeros((ny, nx), np.uint8), (True, True),
                   (0.0, 0.0), np.full((ny, nx), 2e37), np.zeros((ny, nx)),
                   np.zeros((ny, nx)))
    d = b.Domain.from_problem(p)
    d.step(1)
    _, mass = d.residual()  # raises on the instability flag
    assert mass == pytest.approx(2e37 * nx * ny, rel=1e-5)
    d.close()
