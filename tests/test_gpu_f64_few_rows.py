"""The FP64 sweep's tiles on grids whose last tiles hold few rows of the domain (the rows past them are not computed):
every tile shape against the oracle at one row, one below, at and one above a tile's height, and the small tile's width."""
import pytest

import oracle
from conftest import rel_errors
from paper_2108_08769_gb300 import ac
from paper_2108_08769_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-11   # the FP64 form's bar
WALLS, PERIODIC = ("slip", "noslip", "slip", "transmissive"), ("periodic", "periodic", "periodic", "periodic")
GRIDS = [(33, 1, WALLS), (100, 1, ("transmissive",) * 4), (7, 2, WALLS), (8, 8, PERIODIC), (9, 7, WALLS), (17, 9, WALLS),
         (35, 15, PERIODIC), (64, 22, WALLS), (1, 5, WALLS)]


@pytest.mark.parametrize("v", range(9))
@pytest.mark.parametrize("grid", GRIDS, ids=[f"{g[0]}x{g[1]}" for g in GRIDS])
def test_against_oracle(monkeypatch, v, grid):
    nx, ny, bc = grid
    monkeypatch.setenv("AC_TILE_F64", str(v))
    case = W.random_two_fluid(nx, ny, ratio=300.0, c0=10.0, bc=bc, gy=-9.81)
    t = ac.Tank.from_case(case)
    t.physical_step(case.dt, -1.0, 5)
    assert t.tile_shape()[3] == v
    got = t.get_state()
    t.close()
    ref, *_ = oracle.physical_step(case, case.state(), tol=-1.0, max_iters=5)
    assert max(rel_errors(got, ref)) <= TOL
