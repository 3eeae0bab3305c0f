"""What the fixed-point Osher flux (ac_fixed_flux.cuh) accepts, and its error over all of that, on the CPU.

Bound: as in test_fixed_flux.py, 32 x 2^-53 of the sum of a component's terms.  Up to rho u^2/(4 beta) = 4.8 the
difference 1 - |u|/c keeps all but 4 of its 61 bits (9 x 4.8 at an outer Gauss point: 1 - a > 1/90, squared in the
fluxes, 13 bits), so 48 bits at the least of a part whose share of the terms is that small.
"""
import ctypes
import os
import subprocess
from decimal import Decimal

import numpy as np
import pytest

from test_fixed_flux import ROOT, exact

WRAPPER = r'''
#include "ac_fixed_flux.cuh"
extern "C" int fixed_flux(const double *s, double beta, double sc, double scp, double *F) {
    const acgb::FixedBeta fb = acgb::make_fixed_beta(beta);
    if (!acgb::fixed_beta_ok(beta) || !acgb::fixed_flux_ok(s[0], s[1], s[2], s[3], s[4], s[5], s[6], s[7], fb)) return 0;
    acgb::osher_flux_fixed(s[0], s[1], s[2], s[3], s[4], s[5], s[6], s[7], fb, acgb::make_fixed_scale(sc),
                           acgb::make_fixed_scale(scp), F);
    return 1;
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed_flux_limits")
    (d / "w.cpp").write_text(WRAPPER)
    so = str(d / "w.so")
    # shifts by negative counts and the like end the process
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-shared", "-fPIC", "-fsanitize=shift-exponent", "-fsanitize-trap=all",
                    "-I" + os.path.join(ROOT, "paper_2108_08769_gb300", "csrc"), str(d / "w.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def flux(lib, states, beta, scale=1.0, scale_p=1.0):
    s = (ctypes.c_double * 8)(*states)
    F = (ctypes.c_double * 4)()
    D = ctypes.c_double
    return list(F) if lib.fixed_flux(s, D(beta), D(scale), D(scale_p), F) else None


def check(lib, states, beta, scale=1.0, scale_p=1.0):
    got = flux(lib, states, beta, scale, scale_p)
    if got is None:
        return False
    F, S = exact(states, beta)
    for k in range(4):
        f = Decimal(scale_p if k == 3 else scale)
        assert abs(Decimal(got[k]) - f * F[k]) <= 32 * Decimal(2) ** -53 * f * S[k], (k, states, beta, got[k], F[k])
    return True


def mach2(states, beta):
    return max(states[0] * states[1] ** 2, states[4] * states[5] ** 2) / (4 * beta)


def draw(rng, ratio, beta, r):
    """Faces whose faster side has rho u^2/(4 beta) = ratio: equal, mirrored and independent sides."""
    u = np.sqrt(4 * beta * ratio / r)
    sign = rng.choice([-1.0, 1.0])
    out = []
    for rR, uR in ((r, u), (r, -u), (r * 10 ** rng.uniform(-3, 0), u), (r, u * rng.uniform(-1, 1)), (r / 1000, 0.0),
                   (r * 10 ** rng.uniform(0, 3), 0.03 * u)):
        p = r * u * u * 10 ** rng.uniform(-6, 2)
        s = [r, sign * u, u * rng.normal(), p, rR, sign * uR, u * rng.normal(), p * rng.choice([1.0, 0.5, -1.0, 1 + 1e-9])]
        out += [s, s[4:] + s[:4]]
    return out


def test_speeds_far_above_the_artificial_sound_speed_are_refused_or_right(lib):
    rng = np.random.default_rng(3)
    for ratio in [1e-6, 1e-3, 0.1, 1.0, 2.0, 3.0, 3.9, 4.4, 4.9, 6.0, 30.0, 1e3, 1e4, 1e6, 1e9, 1e12]:
        for beta in (1e-6, 1.0, 4e5):
            for s in draw(rng, ratio, beta, 10 ** rng.uniform(-3, 3)):
                took, m = check(lib, s, beta), mach2(s, beta)
                assert took or m > 3.99, (m, s, beta)
                assert not took or m < 4.81, (m, s, beta)
    # a face whose mass flux came out 41 % too large
    assert flux(lib, [0.579, -7.479e5, 446.8, -2e-6, 0.579, 7.479e5, -0.0042, -415.3], 1.087e-4) is None
    assert flux(lib, [1000.0, 1e20, 0.0, 0.0, 1000.0, 1e20, 0.0, 0.0], 4e5) is None


def test_exponents_at_the_limits(lib):
    """Densities to 2^+-249, velocities and pressures to 2^249, beta to 1e+-69."""
    rng = np.random.default_rng(4)
    took = 0
    for _ in range(400):
        beta = 10.0 ** rng.uniform(-69, 69)
        rL, rR = (2.0 ** rng.uniform(-249, 249) for _ in range(2))
        if rng.random() < 0.5:
            rR = rL * 10 ** rng.uniform(-3, 3)
        u = [min(2.0 ** 249, np.sqrt(16 * beta / r)) * 2.0 ** -rng.uniform(0, 30) * rng.choice([-1, 1]) for r in (rL, rR)]
        v = [x * 2.0 ** rng.uniform(-20, 2) for x in u]
        p = [min(2.0 ** 249, beta * 2.0 ** rng.uniform(-20, 20)) * rng.choice([-1, 1]) for _ in range(2)]
        if max(abs(x) for x in v) < 2.0 ** 250:
            took += check(lib, [rL, u[0], v[0], p[0], rR, u[1], v[1], p[1]], beta)
    assert took > 300


def test_equal_pressures_or_velocities_hide_nothing(lib):
    """A jump that is exactly zero has no size: the other one keeps its bits beside it, whatever the pressures or
    velocities themselves are (flow that has all but come to rest under a large head)."""
    rng = np.random.default_rng(5)
    for k in range(300):
        rL, rR, beta = 10 ** rng.uniform(0, 3), 10 ** rng.uniform(0, 3), 10 ** rng.uniform(0, 6)
        c = np.sqrt(beta / max(rL, rR))
        p = beta * 10 ** rng.uniform(0, 12) * rng.choice([-1, 1])
        u = c * 10 ** -rng.uniform(5, 40)
        uR = [0.0, -u, 0.3 * u][k % 3]
        assert check(lib, [rL, u, u * rng.normal(), p, rR, uR, u * rng.normal(), p], beta)
        dp = beta * 10 ** -rng.uniform(10, 40)
        assert check(lib, [rL, u, c * rng.normal(), dp, rR, u, c * rng.normal(), -dp], beta)


@pytest.mark.parametrize("tiny", [0.0, -0.0, 5e-324, -5e-324, 1e-310, -2.2e-308])
def test_signed_zeros_and_subnormals_beside_a_density_jump_and_a_pressure(lib, tiny):
    """A velocity of zero of either sign, or subnormal, is a zero: at rest exactly the pressure, also where the sides'
    densities differ; and a zero or subnormal pressure or tangential velocity gives what +0 gives."""
    for rL, rR, p, v in ((1000.0, 1.0, 5.0, 0.3), (1.0, 1000.0, -7e3, -0.0), (2.0, 3.0, 1e-3, 1e3)):
        for uL, uR in ((tiny, tiny), (tiny, 0.0), (0.0, tiny), (tiny, -tiny)):
            assert flux(lib, [rL, uL, v, p, rR, uR, v, p], 4e5) == [0.0, 2.0 * p, 0.0, 0.0]
        for q in (1, 2, 3, 5, 6, 7):
            s = [rL, 0.2, 0.3, p, rR, -0.1, 0.4, 2 * p]
            s[q] = 0.0
            want = flux(lib, s, 4e5)
            s[q] = tiny
            assert flux(lib, s, 4e5) == want, (q, s)


def test_the_sign_of_a_zero_changes_no_bit(lib):
    """Random faces with some of u, v and p zero: +0, -0 and a subnormal give the same flux to the last bit."""
    rng = np.random.default_rng(6)
    for _ in range(4000):
        s = (rng.uniform(-0.5, 0.5, 8) * 2.0 ** rng.uniform(-20, 20, 8))
        s[[0, 4]] = np.abs(s[[0, 4]])
        zero = [q for q in (1, 2, 3, 5, 6, 7) if rng.random() < 0.6]
        beta = 2.0 ** rng.uniform(0, 20)
        got = []
        for tiny in (0.0, -0.0, -1e-310):
            s[zero] = tiny
            got.append(flux(lib, list(s), beta))
        assert got[0] == got[1] == got[2], (list(s), beta)


@pytest.mark.parametrize("scale,scale_p", [(128.0, 51.2e6), (0.3, 7.7e-9), (1.0 / 3e5, 1e17), (1e-60, 1e60)])
def test_factors_that_are_no_powers_of_two(lib, scale, scale_p):
    rng = np.random.default_rng(11)
    for ratio in (1e-6, 0.1, 3.0):
        for s in draw(rng, ratio, 4e5, 10 ** rng.uniform(-3, 3)):
            assert check(lib, s, 4e5, scale, scale_p)
