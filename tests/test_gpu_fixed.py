"""The fixed-point first pass of the flux phase (Euler equations, flat form)
against the oracle, at degree 2 and in short at the others: both flow directions, resting and
supersonic gas, states of very large and very small units, the ratios of
specific heats at and beyond the ends of its range, domains around the block
size, and data that leave the format and go to the second pass."""
import numpy as np
import pytest

from paper_2602_21911_gb300 import inputs as I

from parity import DISC_TOL, SMOOTH_TOL, check_parity

pytestmark = pytest.mark.gpu


def _wave(N, u, gamma=1.4, amp=0.2, mass=1.0, speed=1.0, bc=I.PERIODIC, M=2, recon=0):
    """Density wave of velocity u at p = 1, in units (mass, speed)."""
    prob, avg, lim, _ = I.euler_wave(N, M, amp=amp, gamma=gamma, bc=bc)
    prob = dict(prob, recon=recon)
    unit = np.array([[1.0], [speed], [speed * speed]]) * mass

    def state(r):
        return np.stack([r, r * u, np.full_like(r, 1.0 / (gamma - 1.0)) + 0.5 * r * u * u]) * unit
    a, g = state(avg[0]), state(lim[0])
    return prob, a, g, g.copy()


@pytest.mark.parametrize("N", [1, 2, 3, 31, 127, 128, 129])
@pytest.mark.parametrize("bc", [I.PERIODIC, I.TRANSMISSIVE])
def test_domain_sizes(N, bc):
    check_parity(*_wave(N, -0.7, bc=bc), 20, SMOOTH_TOL)


@pytest.mark.parametrize("u", [0.3, -0.3, 2.5, -2.5, 400.0])
def test_flow_directions(u):
    check_parity(*_wave(64, u), 40, SMOOTH_TOL)


@pytest.mark.parametrize("E", [2.5, 1.7320508075688772, 0.1])
def test_a_resting_density_wave_stays_at_rest_exactly(E):
    """Equal pressures give equal fluxes whatever the densities, so no momentum
    forms and no average moves (not compared with the oracle, whose own
    rounding leaves 1e-15 of momentum here)."""
    from paper_2602_21911_gb300 import grprec
    prob, a, g, _ = _wave(64, 0.0, amp=0.9)
    a[2], g[2] = E, E
    s = grprec.Solver(prob)
    s.set_initial(a, g)
    s.step(40)
    a1, g1, t = s.get_state()
    assert np.array_equal(a1, a) and np.array_equal(g1, g) and t[0] > 0


@pytest.mark.parametrize("gamma", [1.1, 1.29, 1.3, 5.0 / 3.0, 1.9, 2.0])
def test_ratios_of_specific_heats(gamma):
    check_parity(*_wave(64, 0.5, gamma=gamma), 40, SMOOTH_TOL)


@pytest.mark.parametrize("mass,speed", [(1e90, 1e20), (1e-90, 1e-20), (1e30, 1e-40), (2.0 ** -37, 2.0 ** 41)])
def test_units(mass, speed):
    check_parity(*_wave(65, -0.4, mass=mass, speed=speed), 20, SMOOTH_TOL)


@pytest.mark.parametrize("ratio", [2.0, 10.0, 1000.0])
def test_jumps_leave_the_format(ratio):
    for WL, WR in (((1.0, 0.5, 1.0), (ratio, 0.5, 1.0)), ((1.0, -0.5, ratio), (1.0, 0.5, 1.0))):
        check_parity(*I.riemann_problem(101, WL, WR, M=2), 30, DISC_TOL)


@pytest.mark.parametrize("M,recon,N", [(1, 0, 33), (3, 0, 33), (4, 0, 9800), (1, 1, 33), (2, 1, 33), (3, 1, 33)])
@pytest.mark.parametrize("u", [0.4, -0.4, -3.0])
def test_other_degrees_and_reconstructions(M, recon, N, u):
    check_parity(*_wave(N, u, amp=0.1, mass=3.0, speed=0.7, M=M, recon=recon), 12, SMOOTH_TOL)


@pytest.mark.parametrize("M,recon", [(1, 0), (3, 0), (1, 1), (2, 1), (3, 1)])
def test_riemann_problems_of_all_strengths(M, recon):
    """Expansions and compressions from weak to beyond the format's range."""
    for k, du in enumerate((0.01, 0.3, 1.0, -0.01, -0.3, -1.0)):
        prob, avg, lm, lp = I.riemann_problem(64, (1.0, -du, 1.0), (0.8 + 0.1 * k, du, 1.1), M=M, cfl=0.7)
        check_parity(dict(prob, recon=recon), avg, lm, lp, 25, DISC_TOL)


@pytest.mark.parametrize("M,recon,N", [(2, 0, 9728), (2, 0, 9729), (2, 0, 19455), (2, 0, 19456), (4, 0, 19456),
                                       (1, 0, 29183), (1, 0, 29184), (3, 0, 29184), (1, 1, 29184), (2, 1, 29184),
                                       (3, 1, 29184)])
def test_open_ends_around_the_sizes_where_the_pass_changes(M, recon, N):
    """A strong jump (into the format's second pass, and repaired) and two open
    ends, at both sides of every line of the dispatch for single domains."""
    prob, avg, lm, lp = I.riemann_problem(N, (1.0, 0.4, 1.0), (0.2, -0.5, 0.1), M=M)
    check_parity(dict(prob, recon=recon), avg, lm, lp, 6, DISC_TOL)


@pytest.mark.parametrize("M", [1, 2, 3, 4])
def test_predictor_solver_riemann_problems(M):
    """The interface problems of the DET solver: weak and strong waves, flow in
    both directions, and data that leave the format."""
    for du, ratio in ((0.0, 0.9), (0.3, 1.1), (-0.5, 0.5), (1.0, 0.8), (-3.0, 0.01)):
        prob, avg, lm, lp = I.riemann_problem(65, (1.0, -du, 1.0), (ratio, du, 1.1 * ratio), M=M, cfl=0.5)
        check_parity(dict(prob, solver=1), avg, lm, lp, 8, DISC_TOL)
    for u in (0.4, -2.5):
        p, a, lo, hi = _wave(33, u, mass=3.0, speed=0.7, M=M)
        check_parity(dict(p, solver=1), a, lo, hi, 8, SMOOTH_TOL)
