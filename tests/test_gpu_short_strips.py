"""The column-strip sweep on strips of 8 and 16 rows (single tank and batch): against the oracle where a strip's row
loops meet the tank's edges (strips shorter than their four first rows, a ragged top strip, periodic y, one row), and
the batch's against the single tank's, bit for bit."""
import numpy as np
import pytest

import oracle
from conftest import rel_errors
from paper_2108_08769_gb300 import ac
from paper_2108_08769_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-5   # the mixed form's bar
GRIDS = [(61, 83, ("slip", "slip", "periodic", "periodic"), 0.0), (45, 70, ("periodic", "periodic", "slip", "noslip"), -9.81),
         (29, 17, ("slip", "noslip", "slip", "slip"), -9.81), (33, 1, ("transmissive", "slip", "slip", "slip"), -9.81),
         (57, 9, ("slip",) * 4, -9.81)]


@pytest.mark.parametrize("v,rows", [(22, 16), (23, 8)])
@pytest.mark.parametrize("grid", GRIDS, ids=[f"{g[0]}x{g[1]}" for g in GRIDS])
@pytest.mark.parametrize("limiter_k", [1, 2])
def test_against_oracle(monkeypatch, v, rows, grid, limiter_k):
    nx, ny, bc, gy = grid
    monkeypatch.setenv("AC_TILE", str(v))
    case = W.random_two_fluid(nx, ny, ratio=300.0, c0=10.0, bc=bc, gy=gy)
    case.options.limiter_k = limiter_k
    t = ac.Tank.from_case(case, precision="mixed")
    t.physical_step(case.dt, -1.0, 6)
    assert t.tile_shape()[1] == rows and t.tile_shape()[3] == v
    got = t.get_state()
    t.close()
    ref, *_ = oracle.physical_step(case, case.state(), tol=-1.0, max_iters=6)
    assert max(rel_errors(got, ref)) <= TOL


def test_batch_equals_single_tanks(monkeypatch):
    monkeypatch.setenv("AC_BATCH_TILE", "15")
    monkeypatch.setenv("AC_TILE", "22")
    cases = W.batched_tanks(count=4, nmin=20, nmax=90, seed=12) + [W.random_two_fluid(37, 19, ratio=300.0, c0=8.0)]
    b = ac.Batch.from_cases(cases)
    b.physical_step(1e-3, -1.0, 7)
    assert b.tile_shape()[1] == 16
    for k, c in enumerate(cases):
        t = ac.Tank.from_case(c, precision="mixed")
        t.physical_step(1e-3, -1.0, 7)
        for x, y in zip(b.get_state(k), t.get_state()):
            assert np.array_equal(x, y), k
        t.close()
    b.close()
