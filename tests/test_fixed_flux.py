"""The FP64 sweep's Osher flux in block fixed point (ac_fixed_flux.cuh), compiled for the CPU, where the same integer
arithmetic runs, against 60-digit decimal arithmetic.

The integers keep 57 bits or more of each quantity, so 2F should be off by its final rounding (2^-53) and by the face
states' own conditioning: the outer Gauss points' density may be 4.4 times smaller than the mean (1 - sqrt(3/5)
against 1), which multiplies the relative error of their velocity, squared in the fluxes (4.4^2 = 20).  Each component
is therefore held to 32 x 2^-53 of the sum of its terms' magnitudes.
"""
import ctypes
import os
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WRAPPER = r'''
#include "ac_fixed_flux.cuh"
extern "C" int fixed_flux(const double *s, double beta, double *F) {
    if (!acgb::fixed_flux_ok(s[0], s[1], s[2], s[3], s[4], s[5], s[6], s[7])) return 0;
    acgb::osher_flux_fixed(s[0], s[1], s[2], s[3], s[4], s[5], s[6], s[7], acgb::make_fixed_beta(beta),
                           acgb::make_fixed_scale(1.0), acgb::make_fixed_scale(1.0), F);
    return 1;
}
extern "C" void iterations(unsigned long long x, unsigned long long *out) {
    out[0] = acgb::fx::rcp61(x);
    out[1] = acgb::fx::rsqrt61(x);
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed_flux")
    (d / "w.cpp").write_text(WRAPPER)
    so = str(d / "w.so")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-shared", "-fPIC",
                    "-I" + os.path.join(ROOT, "paper_2108_08769_gb300", "csrc"), str(d / "w.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def flux(lib, states, beta):
    s = (ctypes.c_double * 8)(*states)
    F = (ctypes.c_double * 4)()
    ok = lib.fixed_flux(s, ctypes.c_double(beta), F)
    return list(F) if ok else None


def exact(states, beta):
    """2F and the sum of its terms' magnitudes, per component."""
    getcontext().prec = 60
    D = Decimal
    rL, uL, vL, pL, rR, uR, vR, pR = (D(float(x)) for x in states)
    b = D(float(beta))
    mL, nL, mR, nR = rL * uL, rL * vL, rR * uR, rR * vR
    dr, dm, dn, dq = rR - rL, mR - mL, nR - nL, (pR - pL) / b
    x = (D(3) / D(5)).sqrt()
    F = [mL + mR, mL * uL + pL + mR * uR + pR, mL * vL + mR * vR, uL + uR]
    S = [abs(mL) + abs(mR), mL * uL + abs(pL) + mR * uR + abs(pR), abs(mL * vL) + abs(mR * vR), abs(uL) + abs(uR)]
    for t, w in (((1 - x) / 2, D(5) / 18), (D(1) / 2, D(8) / 18), ((1 + x) / 2, D(5) / 18)):
        r, m, n = rL + t * dr, mL + t * dm, nL + t * dn
        u, v = m / r, n / r
        c = (u * u + 4 * b / r).sqrt()
        l4, l5, a = (u + c) / 2, (u - c) / 2, (dm - u * dr) / b
        f4 = (abs(l4) - abs(u)) * (r / c) * (l4 * a + dq)
        f5 = -(abs(l5) - abs(u)) * (r / c) * (l5 * a + dq)
        terms = ([abs(u) * dr, f4 * l4, f5 * l5], [abs(u) * dm, f4 * (u * l4 + b / r), f5 * (u * l5 + b / r)],
                 [abs(u) * dn, v * f4 * l4, v * f5 * l5], [abs(u) * dq, -f4 * l5 / r, -f5 * l4 / r])
        for k in range(4):
            F[k] -= w * sum(terms[k])
            S[k] += w * sum(abs(y) for y in terms[k])
    return F, S


def states_of(kind, rng):
    sign = lambda: rng.choice([-1.0, 1.0])  # noqa: E731
    log = lambda lo, hi: float(np.exp(rng.uniform(np.log(lo), np.log(hi))))  # noqa: E731
    if kind == "smooth":
        rL, uL, vL, pL = log(1, 1000), sign() * log(1e-3, 1), sign() * log(1e-3, 1), rng.uniform(0, 1e4)
        return [rL, uL, vL, pL, rL * (1 + 1e-2 * rng.normal()), uL * (1 + 1e-2 * rng.normal()), vL, pL + rng.normal()], 4e5
    if kind == "interface":
        return [log(0.5, 2000), sign() * log(1e-3, 3), rng.normal(), rng.uniform(0, 1e4),
                log(0.5, 2000), sign() * log(1e-3, 3), rng.normal(), rng.uniform(0, 1e4)], 4e5
    if kind == "near rest":   # hydrostatic heads with round-off motion
        p = rng.uniform(0, 1e4)
        return [1000.0, 1e-15 * rng.normal(), 1e-15 * rng.normal(), p,
                rng.choice([1.0, 1000.0]), 1e-15 * rng.normal(), 0.0, p * (1 + 2e-16 * rng.integers(-2, 3))], 4e5
    # the paper's Riemann problem 5 and its like: light against heavy, u near the artificial sound speed
    return [log(1e-3, 1e-2), rng.uniform(-1, 1), rng.normal(), 0.1, 1.0, rng.uniform(-1, 1), rng.normal(), 1.0], 1.0


@pytest.mark.parametrize("kind", ["smooth", "interface", "near rest", "riemann"])
def test_against_decimal(lib, kind):
    rng = np.random.default_rng(7)
    for _ in range(150):
        states, beta = states_of(kind, rng)
        got = flux(lib, states, beta)
        F, S = exact(states, beta)
        for k in range(4):
            assert abs(Decimal(got[k]) - F[k]) <= 32 * Decimal(2) ** -53 * S[k], (kind, k, states, got[k], F[k])


def test_mirrored_states_pass_no_mass_and_rest_stays_at_rest(lib):
    """At a wall the ghost mirrors the cell: exactly no mass and no p/beta flux.  At rest: exactly the pressure."""
    rng = np.random.default_rng(8)
    for _ in range(200):
        r, u, v, p = rng.uniform(1, 1000), rng.normal(), rng.normal(), 1e4 * rng.normal()
        F = flux(lib, [r, u, v, p, r, -u, v, p], 4e5)
        assert F[0] == 0.0 and F[2] == 0.0 and F[3] == 0.0
        assert flux(lib, [r, 0.0, 0.0, p, 1.0, 0.0, 0.0, p], 4e5) == [0.0, 2.0 * p, 0.0, 0.0]


def test_zeros_and_subnormals_count_as_zero(lib):
    """Exact zeros give exact zeros, and a subnormal velocity what a zero one gives."""
    for tiny in (0.0, -0.0, 5e-324, -1e-310):
        assert flux(lib, [3.0, tiny, tiny, 0.0, 3.0, tiny, tiny, 0.0], 10.0) == [0.0, 0.0, 0.0, 0.0]
        assert flux(lib, [3.0, tiny, 0.0, 1.5, 2.0, 0.25, tiny, 2.5], 10.0) == flux(
            lib, [3.0, 0.0, 0.0, 1.5, 2.0, 0.25, 0.0, 2.5], 10.0)


def test_refuses_what_it_cannot_represent(lib):
    good = [1.0, 0.5, 0.1, 2.0, 3.0, -0.5, 0.0, 1.0]
    assert flux(lib, good, 10.0) is not None
    for k in range(8):
        for bad in (np.inf, -np.inf, np.nan, 1e80, -1e80) + ((0.0, -1.0, 5e-324, 1e-80) if k in (0, 4) else ()):
            s = list(good)
            s[k] = bad
            assert flux(lib, s, 10.0) is None, (k, bad)


def test_reciprocal_and_square_root_iterations(lib):
    """2^61/x and 2^61/sqrt(x), x = X 2^-62: within 2^-59 of the result, at the ends of the range too."""
    getcontext().prec = 60
    rng = np.random.default_rng(9)
    out = (ctypes.c_ulonglong * 2)()
    xs = [1 << 61, (1 << 61) + 1, (1 << 62) - 1] + [int(x) for x in rng.integers(1 << 61, 1 << 62, 3000)]
    for X in xs + [x >> 1 for x in xs]:
        lib.iterations(ctypes.c_ulonglong(X), out)
        x = Decimal(X) / 2 ** 62
        if X >= 1 << 61:
            assert abs(out[0] * x / 2 ** 61 - 1) <= Decimal(2) ** -59
        assert abs(out[1] * x.sqrt() / 2 ** 61 - 1) <= Decimal(2) ** -59
