"""S_max of large grids (above 400,000 cells, where FP32 bounds choose the cells
that are evaluated) in units at the ends of the FP32 range, against the oracle:
the cell that holds the maximum must not be missed."""
import numpy as np
import pytest

from paper_2602_21911_gb300 import inputs as I

from parity import SMOOTH_TOL, check_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mass,speed,warm", [(1.0, 1.0, 0.0), (1e38, 1.0, 0.0), (1e29, 1e-29, 2.0)])
def test_units_at_the_ends_of_the_fp32_range(mass, speed, warm):
    """Densities of 0.5 to 1.2 units, the dense gas fastest; warm: the light gas slow
    and with the largest |u| + c."""
    N = 400064
    prob = dict(I.euler_wave(N, 2)[0], cfl=0.5)

    def state(x):
        r = 0.85 + 0.35 * np.sin(I.TWO_PI * x)
        p = 0.01 + warm * (1.2 - r) ** 2
        return np.stack([r, r * r * speed, (2.5 * p + 0.5 * r ** 3) * speed ** 2]) * mass
    lim = state(np.arange(N) / N)
    check_parity(prob, state((np.arange(N) + 0.5) / N), lim, lim.copy(), 3, SMOOTH_TOL)
