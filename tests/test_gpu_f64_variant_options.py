"""Every tile shape of the FP64 sweep with the options that its other tests leave at their defaults: the second limiter,
the limited pressure gradients, other stage counts, no real-time term, the global pseudo-time step and BDF3, on a grid
with tiles inside the domain, at its sides and cut off by it (two groups of rows in the 32x14 tile, short tiles in the
small ones)."""
import numpy as np
import pytest

import oracle
from conftest import rel_errors
from paper_2108_08769_gb300 import ac
from paper_2108_08769_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-11   # the FP64 form's bar
WALLS = ("slip", "noslip", "transmissive", "slip")
OPTIONS = {
    "limiter 2": dict(limiter_k=2),
    "superbee": dict(gradp="superbee"),
    "split minmod": dict(gradp="split_minmod"),
    "split superbee, limiter 2": dict(gradp="split_superbee", limiter_k=2),
    "one stage": dict(s_max=1),
    "four stages": dict(s_max=4),
    "no real time": dict(realtime=False),
    "global step": dict(local_dtau=False),
    "p row without alpha_PI": dict(alpha_pi_p_row=False),
}


def case_of(**options):
    case = W.random_two_fluid(101, 47, ratio=300.0, c0=10.0, bc=WALLS, gx=0.7)
    for name, value in options.items():
        setattr(case.options, name, value)
    return case


@pytest.mark.parametrize("v", range(9))
@pytest.mark.parametrize("name", OPTIONS)
def test_against_oracle(monkeypatch, v, name):
    monkeypatch.setenv("AC_TILE_F64", str(v))
    case = case_of(**OPTIONS[name])
    t = ac.Tank.from_case(case)
    t.physical_step(case.dt, -1.0, 4)
    assert t.tile_shape()[3] == v
    got = t.get_state()
    t.close()
    ref, *_ = oracle.physical_step(case, case.state(), tol=-1.0, max_iters=4)
    assert max(rel_errors(got, ref)) <= TOL


@pytest.mark.parametrize("v", range(9))
def test_bdf3_from_history(monkeypatch, v):
    monkeypatch.setenv("AC_TILE_F64", str(v))
    case = case_of(bdf_order=3)
    rng = np.random.default_rng(2)
    older = [tuple(a * (1 + 1e-3 * rng.standard_normal(a.shape)) for a in case.state()[:3]) for _ in range(2)]
    t = ac.Tank.from_case(case)
    for level, state in enumerate(older, start=1):
        t.set_history(level, *state)
    t.physical_step(case.dt, -1.0, 4)
    got = t.get_state()
    t.close()
    ref, *_ = oracle.physical_step(case, case.state(), tol=-1.0, max_iters=4, history=older)
    assert max(rel_errors(got, ref)) <= TOL
