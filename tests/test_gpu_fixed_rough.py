"""The fixed-point Riemann problems of the flux phase and of the DET solver on
rough data, against the oracle: averages and interface data drawn
independently on periodic grids (which take the fixed-point pass at every
size), so that every interface has a Riemann problem of its own, strong
expansions among them; and jumps that leave the format on such grids."""
import numpy as np
import pytest

from paper_2602_21911_gb300 import inputs as I

from out_of_tolerance import check_exempt
from parity import DISC_TOL, check_parity, oracle_ulp_sensitivity

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


def _jumps(N, WL, WR, M, recon):
    """A periodic grid of two states: two jumps, one of them an expansion."""
    prob = dict(I.euler_wave(N, M)[0], recon=recon, cfl=0.5)
    Q = [np.array([r, r * u, 2.5 * p + 0.5 * r * u * u]) for r, u, p in (WL, WR)]
    right = (np.arange(N) >= N // 3) & (np.arange(N) < 2 * N // 3)
    avg = np.where(right[None], Q[1][:, None], Q[0][:, None])
    lim = np.where((right | np.roll(right, 1))[None], Q[1][:, None], Q[0][:, None])
    return prob, avg, lim, lim.copy()


# Runs the oracle itself does not hold: (M, recon, ratio, data) -> (the oracle's own
# response to one ulp in every average, GPU difference; the FP64 forms differ alike).
# A contact in moving gas at the interpolating degrees, its edge polynomials far
# outside the data.
ILL = {(4, 0, 30.0, 0): (4.7e-2, 5.0e-3), (2, 0, 1000.0, 0): (1.7e-2, 6.5e-2), (4, 0, 1000.0, 0): (1.1e-2, 6.4e-2),
       (2, 1, 1000.0, 0): (1.2e-2, 4.6e-2)}
ALL = [(1, 0), (2, 0), (3, 0), (4, 0), (1, 1), (2, 1), (3, 1)]


@pytest.mark.parametrize("M,recon", ALL)
@pytest.mark.parametrize("ratio", [1.2, 3.0, 30.0, 1000.0])
def test_jumps_on_periodic_grids(M, recon, ratio):
    for k, (WL, WR) in enumerate((((1.0, 0.3, 1.0), (ratio, 0.3, 1.0)), ((1.0, -0.4, ratio), (1.0, 0.5, 1.0)),
                                  ((1.0, 0.2, 1.0), (1.0 / ratio, -0.3, 1.0 / ratio)))):
        data = _jumps(101, WL, WR, M, recon)
        if (M, recon, ratio, k) in ILL:
            check_exempt(oracle_ulp_sensitivity(*data, 12), DISC_TOL, (M, recon, ratio, k))
        else:
            check_parity(*data, 12, DISC_TOL)


@pytest.mark.parametrize("M,recon", ALL)
def test_periodic_grids_take_the_fixed_point_pass(M, recon):
    """Degrees 2 and 4: the second pass is launched, as it is not by the FP64 pass of
    short open grids (nor is it at the others).  Degrees 1 and 3: five Newton steps for
    every problem."""
    from paper_2602_21911_gb300 import grprec
    counts = []
    for bc in (I.PERIODIC, I.TRANSMISSIVE):
        prob, avg, lim, lim2 = I.euler_wave(64, M, bc=bc)
        s = grprec.Solver(dict(prob, recon=recon))
        s.set_initial(avg, lim, lim2)
        s.step(1)
        n = s.launch_count()
        s.step(4)
        counts.append(s.launch_count() - n)
        stats, status = s.get_stats()
        assert status[0] == 0
        if bc == I.PERIODIC and recon == 0 and M in (1, 3):
            assert stats[0, grprec.STAT_NEWTON_MAX] == 5 and stats[0, grprec.STAT_NEWTON_SUM] % 5 == 0
    assert counts[0] == counts[1] + 4
