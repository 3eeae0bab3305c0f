"""The mixed form's local pseudo-time step has no error of its own common to all cells.

One Euler stage without a real-time term worth naming moves p by dtau times its residual, so the slope of the mixed
form's increments over the FP64 form's (least squares over all cells) is the mean ratio of their steps.  With cells of a
power of two everything but CFL_tau is exact; the CFL numbers are such that a single FP32 constant 1/CFL_tau would be
5e-8 to 5.8e-8 off.  Rounding errors of single cells average out over 16384 of them (1e-7/128); half of one constant's
largest rounding error, 2^-25, is the bound."""
import numpy as np
import pytest

from paper_2108_08769_gb300 import ac
from paper_2108_08769_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def increment(case, precision):
    t = ac.Tank.from_case(case, precision=precision)
    t.physical_step(1e20, -1.0, 1)
    p = t.get_state()[3]
    t.close()
    return p - case.p


@pytest.mark.parametrize("v", [0, 10, 15])
@pytest.mark.parametrize("cfl", [0.482, 0.485, 0.889, 0.941, 0.979])
def test_mean_step(monkeypatch, v, cfl):
    assert 5e-8 < abs(float(np.float32(1 / cfl)) * cfl - 1) < 6e-8
    monkeypatch.setenv("AC_TILE", str(v))
    case = W.random_two_fluid(128, 128, ratio=4.0, c0=4.0, velocity=0.5, gy=0.0)
    case.options.s_max, case.options.cfl_tau = 1, cfl
    m, f = increment(case, "mixed"), increment(case, "fp64")
    assert abs(float((m * f).sum() / (f * f).sum()) - 1) <= 2.0 ** -25
