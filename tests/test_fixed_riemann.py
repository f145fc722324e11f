"""Fixed-point Riemann problems on the host (gamma = 7/5): independent left and
right states over decades, strong waves, rough data and inadmissible sides,
against quad precision and beside the FP64 path."""
import os
import platform
import subprocess

import pytest

from paper_2602_21911_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
FLUX, FLUX_BAD, TRACES, ROUGH, TRACES_BAD = range(5)


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    if platform.machine() != "x86_64":
        pytest.skip("quad precision by libquadmath: x86")
    exe = str(tmp_path_factory.mktemp("fixed") / "check")
    r = subprocess.run([B._nvcc()] + B.ARCH + ["-O2", "-std=c++17", "-I" + B.CSRC,
                                               os.path.join(HERE, "fixed_riemann_check.cu"), "-lquadmath", "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe, "20000"], capture_output=True, text=True)
    assert out.returncode == 0
    return [[float(x) for x in line.split()] for line in out.stdout.splitlines()]


def test_inadmissible_traces_are_left_to_the_general_path(lines):
    got = [x for x in lines if x[0] == TRACES_BAD]
    assert len(got) == 4
    for line in got:
        assert line[-1] == 0, line


def test_inadmissible_sides_of_a_flux_are_refused(lines):
    got = [x for x in lines if x[0] == FLUX_BAD]
    assert len(got) == 4
    for line in got:
        assert line[-1] == 0, line


def _errors_below_fp64(got):
    for kind, degree, spread, share, rms, mx, rms64, mx64, wrong in got:
        # rms below FP64's; a single result is rounded to a double of up to twice
        # its unit (2^-52 of rho a^2 / (gamma (gamma - 1)))
        assert rms <= rms64, (degree, spread, rms, rms64)
        assert mx <= max(mx64, 2.0 ** -52 * 2.0 / (1.4 * 0.4)), (degree, spread, mx, mx64)
        assert wrong == 0, (degree, spread, wrong)


def test_errors_of_the_flux_are_below_the_fp64_path(lines):
    """Strong waves among them: every problem that is taken has converged."""
    got = [x for x in lines if x[0] == FLUX]
    assert len(got) == 4 and got[0][3] > 0.9
    _errors_below_fp64(got)


@pytest.mark.parametrize("kind", [TRACES, ROUGH])
def test_errors_of_the_grp_are_below_the_fp64_path(lines, kind):
    """Of traces with independent sides and slopes up to four times their size, and
    of rough averages and interface data."""
    got = [x for x in lines if x[0] == kind]
    assert len(got) == (12 if kind == TRACES else 8) and got[0][3] > 0.4
    _errors_below_fp64([x for x in got if x[3] > 0.0])
