"""Steps that end within their first pseudo-iterations: few kernels launched past the end, and the same states, counts
and norms as a step of that fixed number of iterations."""
import numpy as np
import pytest

from paper_2108_08769_gb300 import ac
from paper_2108_08769_gb300 import workloads as W

pytestmark = pytest.mark.gpu

COUNTS = [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 13, 16]


def test_a_tank_at_rest_launches_two_iterations(monkeypatch):
    monkeypatch.setenv("AC_TILE_F64", "0")
    case = W.random_two_fluid(20, 20)
    case.options.abs_tol = (1e300,) * 4
    t = ac.Tank.from_case(case)
    n = t.kernel_launches()
    assert t.physical_step(case.dt, 1e-3, 100)[1] == 1
    assert t.kernel_launches() - n == 1 + 2 * 4
    for k in (1, 2):
        n = t.kernel_launches()
        t.physical_step(case.dt, -1.0, k)
        assert t.kernel_launches() - n == 1 + 2 * 4
    t.close()


def test_a_batch_at_rest_launches_two_iterations_and_their_rebases(monkeypatch):
    monkeypatch.setenv("AC_BATCH_TILE", "0")
    cases = W.batched_tanks(count=4, nmin=20, nmax=40, seed=7)
    for c in cases:
        c.options.abs_tol = (1e300,) * 4
    b = ac.Batch.from_cases(cases)
    b.physical_step(1e-3, -1.0, 1)
    for tol, k in ((1e-3, 100), (-1.0, 1), (-1.0, 2)):
        n = b.kernel_launches()
        b.physical_step(1e-3, tol, k)
        assert b.kernel_launches() - n == 2 + 2 * 4 + 2 * 2
    b.close()


@pytest.mark.parametrize("form", ["fp64", "mixed", "mixed without a level", "batch", "batch without a level"])
@pytest.mark.parametrize("k", COUNTS)
def test_stopping_at_k_equals_running_k(monkeypatch, form, k):
    for name in ("AC_TILE", "AC_TILE_F64", "AC_BATCH_TILE"):
        monkeypatch.setenv(name, "0")
    cases = [W.random_two_fluid(40, 26, ratio=50.0, c0=6.0), W.random_two_fluid(23, 31, ratio=50.0, c0=6.0, seed=4)]
    for c in cases:
        if form.endswith("level"):
            c.options.gradp = "minmod"
        c.options.abs_tol = (0.0, 0.0, 0.0, 0.0)

    if form.startswith("batch"):
        def run(tol, most):
            b = ac.Batch.from_cases(cases)
            _, its, _ = b.physical_step(1e-4, tol, most)
            R = [b.residual_norms(q) for q in range(2)]
            out = list(its), [x for q in range(2) for x in b.get_state(q)]
            b.close()
            return out, max(float(np.max(r / r0)) for r, r0 in R)
    else:
        def run(tol, most):
            t = ac.Tank.from_case(cases[0], precision=form.split()[0])
            _, its = t.physical_step(1e-4, tol, most)
            R, R0 = t.residual_norms()
            out = [its], t.get_state()
            t.close()
            return out, float(np.max(R / R0))

    # (a tank's norms need not fall at once: the step may stop before k, at the first iteration below the bound)
    (_, _), ratio = run(-1.0, k)
    (its, state), _ = run(ratio * (1 + 1e-12), 1000)
    assert max(its) <= k
    (fixed, want), _ = run(-1.0, max(its))
    if len(set(its)) == 1:
        for a, w in zip(state, want):
            assert np.array_equal(a, w)
    # and a limit reached short of convergence
    (its, state), _ = run(0.0, k)
    (fixed, want), _ = run(-1.0, k)
    assert its == fixed
    for a, w in zip(state, want):
        assert np.array_equal(a, w)
