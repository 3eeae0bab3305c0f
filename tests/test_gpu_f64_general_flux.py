"""FP64 tanks whose faces the fixed-point Osher flux does not take, all or some: they go through the FP64 formula, and
the step agrees with the oracle either way."""
import numpy as np
import pytest

import oracle
from conftest import rel_errors
from paper_2108_08769_gb300 import ac
from paper_2108_08769_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-11   # the FP64 form's bar


def agrees(case, iters=4):
    t = ac.Tank.from_case(case)
    t.physical_step(case.dt, -1.0, iters)
    got = t.get_state()
    t.close()
    ref, *_ = oracle.physical_step(case, case.state(), tol=-1.0, max_iters=iters)
    assert np.all(np.isfinite(ref[0]))
    assert max(rel_errors(got, ref)) <= TOL


@pytest.mark.parametrize("v", range(9))
def test_flow_faster_than_the_artificial_sound_speed(monkeypatch, v):
    """rho u^2/(4 beta) from 0 to some 30: taken and refused faces side by side, on every tile shape."""
    monkeypatch.setenv("AC_TILE_F64", str(v))
    agrees(W.random_two_fluid(45, 31, ratio=3.0, c0=0.15, velocity=0.5, gy=0.0))


@pytest.mark.parametrize("unit", [1e-75, 1e75])
def test_cell_sizes_outside_the_fixed_point_range(unit):
    """The same tank in another unit of length (velocities, densities and pressures as they were): no face is taken."""
    case = W.random_two_fluid(40, 24, ratio=300.0, c0=10.0)
    case.lx, case.ly = case.lx * unit, case.ly * unit
    case.gx, case.gy, case.dt = case.gx / unit, case.gy / unit, case.dt * unit
    agrees(case)
