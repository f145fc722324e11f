"""The fixed-point Riemann problems of the flux phase and of the DET solver on
rough data, against the oracle: averages and interface data drawn
independently on periodic grids (which take the fixed-point pass at every
size), so that every interface has a Riemann problem of its own, strong
expansions among them."""
import numpy as np
import pytest

from paper_2602_21911_gb300 import inputs as I

from parity import DISC_TOL, check_parity

pytestmark = pytest.mark.gpu


def _rough(N, M, recon, solver, spread, seed):
    rng = np.random.default_rng(seed)
    prob = dict(I.euler_wave(N, M)[0], recon=recon, solver=solver, cfl=0.4)

    def states():
        r, p = np.exp(rng.uniform(-spread, spread, (2, N)))
        u = rng.uniform(-spread, spread, N)
        return np.stack([r, r * u, 2.5 * p + 0.5 * r * u * u])
    lim = states()
    return prob, states(), lim, lim.copy()


@pytest.mark.parametrize("M,recon", [(1, 0), (3, 0), (1, 1), (2, 1), (3, 1)])
@pytest.mark.parametrize("spread", [0.3, 0.6, 1.0])
def test_rough_periodic_grids(M, recon, spread):
    S, _, _ = check_parity(*_rough(40000, M, recon, 0, spread, 7 * M + recon), 2, DISC_TOL)
    assert S.status[0] == 0


@pytest.mark.parametrize("M", [1, 2, 3])
@pytest.mark.parametrize("spread", [0.3, 0.6, 1.0])
def test_rough_grids_of_the_predictor_solver(M, spread):
    S, _, _ = check_parity(*_rough(6000, M, 0, 1, spread, 50 + M), 2, DISC_TOL)
    assert S.status[0] == 0
