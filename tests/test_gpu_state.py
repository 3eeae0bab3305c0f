"""A state into its device form and back (ac_set_state, ac_get_state and the batch's): exact round trips at sizes off
every block size, before and after a step has moved the current buffer, and refused states that change nothing."""
import numpy as np
import pytest

from paper_2108_08769_gb300 import ac
from paper_2108_08769_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (7, 3), (33, 9), (5, 301), (300, 17)]


def same(got, want):
    # FP64 levels and zero increments: every field comes back as it was given
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_round_trip(nx, ny, precision):
    a, b = W.random_two_fluid(nx, ny, seed=1), W.random_two_fluid(nx, ny, seed=2)
    t = ac.Tank.from_case(a, precision=precision)
    same(t.get_state(), a.state())
    for k in range(3):   # the buffers rotate with every iteration
        t.physical_step(a.dt, -1.0, 1 + k)
        t.set_state(*b.state())
        same(t.get_state(), b.state())
    # and a step from the new state does not depend on what the tank did before
    t.physical_step(b.dt, -1.0, 4)
    u = ac.Tank.from_case(b, precision=precision)
    u.physical_step(b.dt, -1.0, 4)
    same(t.get_state(), u.get_state())
    t.close()
    u.close()


FAULTS = [(0, np.nan, ac.AC_ERR_NONFINITE, "rho["), (0, 0.0, ac.AC_ERR_ARG, "rho["), (1, np.inf, ac.AC_ERR_NONFINITE, "rhou["),
          (2, -np.inf, ac.AC_ERR_NONFINITE, "rhov["), (3, np.nan, ac.AC_ERR_NONFINITE, "p[")]


@pytest.mark.parametrize("form", ["fp64", "mixed", "batch"])
@pytest.mark.parametrize("field,value,code,name", FAULTS, ids=[f"{n}{v}" for _, v, _, n in FAULTS])
def test_refused_state_changes_nothing(form, field, value, code, name):
    case = W.random_two_fluid(61, 7)
    if form == "batch":
        h = ac.Batch.from_cases([case, W.random_two_fluid(9, 9)])
        put, get, step = (lambda s: h.set_state(0, *s)), (lambda: h.get_state(0)), (lambda: h.physical_step(1e-3, -1.0, 2))
    else:
        h = ac.Tank.from_case(case, precision=form)
        put, get, step = (lambda s: h.set_state(*s)), h.get_state, (lambda: h.physical_step(1e-3, -1.0, 2))
    step()
    before = get()
    bad = [a.copy() for a in case.state()]
    bad[field].flat[-1] = value
    with pytest.raises(ac.ACError) as e:
        put(bad)
    assert e.value.code == code and f"{name}{case.cells - 1}]" in str(e.value)
    same(get(), before)
    h.close()


def test_densities_outside_the_fluids_are_refused():
    case = W.random_two_fluid(20, 10, ratio=100.0)
    t = ac.Tank.from_case(case, fluids=(100.0, 1.0))
    heavy = case.rho.copy()
    heavy[3, 4] = 250.0
    with pytest.raises(ac.ACError) as e:
        t.set_state(heavy, case.rhou, case.rhov, case.p)
    assert e.value.code == ac.AC_ERR_ARG and "rho[64] = 250 lies outside" in str(e.value)
    same(t.get_state(), case.state())
    t.close()
