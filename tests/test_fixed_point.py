"""The fixed-point GRP of the flux kernel's first pass (degrees 2 and 4, equal data)
on the host: its errors against quad precision are below those of the FP64
path over the ratios of specific heats, slopes and Mach numbers it accepts, and
what it must leave to the general path (sonic fields, cut series) it leaves."""
import os
import platform
import subprocess

import pytest

from paper_2602_21911_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    if platform.machine() != "x86_64":
        pytest.skip("quad precision by libquadmath: x86")
    exe = str(tmp_path_factory.mktemp("fixed") / "check")
    r = subprocess.run([B._nvcc()] + B.ARCH + ["-O2", "-std=c++17", "-I" + B.CSRC,
                                               os.path.join(HERE, "fixed_point_check.cu"), "-lquadmath", "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe, "20000"], capture_output=True, text=True)
    assert out.returncode == 0
    return [[float(x) for x in line.split()] for line in out.stdout.splitlines()]


def test_errors_are_below_the_fp64_path(lines):
    assert len(lines) == 65
    for degree, traces, gamma, slope, share, rms, mx, rms64, mx64, wrong in lines:
        # rms below FP64's; a single result is rounded to a double of up to
        # twice its unit (2^-52 of rho a^2 / (gamma (gamma - 1)))
        assert rms <= rms64, (degree, gamma, slope, rms, rms64)
        assert mx <= max(mx64, 2.0 ** -52 * 2.0 / (gamma * (gamma - 1.0))), (degree, gamma, slope, mx, mx64)


def test_what_is_accepted(lines):
    for degree, traces, gamma, slope, share, rms, mx, rms64, mx64, wrong in lines:
        assert wrong == 0, (degree, gamma, slope)
        if 1.3 <= gamma and slope <= (0.3 if degree == 2 else 0.05):
            # (with a leading Riemann problem, the tenth or so beyond Mach 2 is left)
            assert share >= (0.99 if degree in (2, 4) and not traces else 0.9), (degree, gamma, slope, share)
