"""The mixed form in another unit of mass: densities, pressures and beta times a power of two scale every operation of
a step exactly, but for what falls below FP32's range.  2^-66 brings the lighter fluid to 1e-20, where a product of two
densities is below it, and everything that a step adds up is not: the states agree to one FP32 rounding of each field."""
import numpy as np
import pytest

from paper_2108_08769_gb300 import ac
from paper_2108_08769_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def step(case, unit):
    t = ac.Tank(case.nx, case.ny, case.lx, case.ly, case.gx, case.gy, case.beta * unit, case.bc,
                ac.options_from(case.options, "mixed"))
    t.set_state(*(a * unit for a in case.state()))
    t.physical_step(case.dt, -1.0, 6)
    out = t.get_state()
    t.close()
    return out


@pytest.mark.parametrize("v", [0, 10, 15, 16, 19, 22, 23])
@pytest.mark.parametrize("options", ["default", "general"])
def test_mass_unit(monkeypatch, v, options):
    monkeypatch.setenv("AC_TILE", str(v))
    case = W.random_two_fluid(90, 70, ratio=1000.0, c0=20.0, bc=("slip", "noslip", "slip", "slip"))
    if options == "general":
        case.options.limiter_k = 2
    for a, b in zip(step(case, 1.0), step(case, 2.0 ** -66)):
        assert np.abs(a - b * 2.0 ** 66).max() <= 2.0 ** -23 * np.abs(a).max()
