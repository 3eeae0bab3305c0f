"""FP64 reciprocals and square roots on the integer pipes (ac_fixed_flux.cuh), on the CPU: correctly rounded, as the
division and square root that they stand for, whatever float seed within 2 ulps they start from (the GPU's fast ones)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from test_fixed_flux import ROOT

WRAPPER = r'''
#include "ac_fixed_flux.cuh"
extern "C" void roots(const double *x, long n, double *r, double *s, double *t, double *rs, unsigned char *ok) {
    using namespace acgb::fx;
    for (long i = 0; i < n; ++i) {
        ok[i] = rcp_ok(x[i]) | (rsqrt_ok(x[i]) << 1);
        if (ok[i] & 1) r[i] = rcp(x[i]);
        if (ok[i] & 2) s[i] = sqrt_rn(x[i]), sqrt_rsqrt(x[i], t[i], rs[i]);
    }
}
'''


@pytest.fixture(scope="module", params=[-2, 0, 2], ids=lambda u: f"seed{u:+d}ulp")
def roots(request, tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed_roots")
    src = open(os.path.join(ROOT, "paper_2108_08769_gb300", "csrc", "ac_fixed_flux.cuh")).read()
    for seed in ("return 1.0f / x;", "return 1.0f / sqrtf(x);"):
        assert seed in src
        moved = f"float y = {seed[7:-1]}; uint32_t b; memcpy(&b, &y, 4); b += {request.param}; memcpy(&y, &b, 4); return y;"
        src = src.replace(seed, moved)
    (d / "ac_fixed_flux.cuh").write_text(src)
    (d / "w.cpp").write_text(WRAPPER)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-shared", "-fPIC", f"-I{d}", str(d / "w.cpp"), "-o", str(d / "w.so")],
                   check=True)
    lib = ctypes.CDLL(str(d / "w.so"))

    def call(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        out = [np.zeros_like(x) for _ in range(4)]
        ok = np.zeros(x.size, np.uint8)
        lib.roots(x.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(x.size), *(o.ctypes.data_as(ctypes.c_void_p) for o in out),
                  ok.ctypes.data_as(ctypes.c_void_p))
        return out, ok
    return call


def arguments():
    """Random bit patterns, every exponent with the mantissas at both ends and in the middle, squares and their
    neighbours (roots near a tie), reciprocals' neighbours, and what is refused."""
    rng = np.random.default_rng(10)
    bits = rng.integers(0, 1 << 64, 400_000, dtype=np.uint64)
    e = np.arange(2048, dtype=np.uint64) << np.uint64(52)
    for m in (0, 1, 2, (1 << 51) - 1, 1 << 51, (1 << 51) + 1, (1 << 52) - 2, (1 << 52) - 1):
        bits = np.concatenate([bits, e + np.uint64(m), e + np.uint64(m) + np.uint64(1 << 63)])
    x = bits.view(np.float64)
    y = rng.uniform(1, 4, 100_000)
    sq = (y * 2.0 ** -26 + np.round(y, 7)) ** 2
    return np.concatenate([x, sq, np.nextafter(sq, 0), np.nextafter(sq, 9), 1 / y, np.nextafter(1 / y, 0),
                           1.0 + np.arange(-2000, 2000) * 2.0 ** -52, 2.0 ** np.arange(-1022, 1024)])


def test_correctly_rounded(roots):
    x = arguments()
    (r, s, t, rs), ok = roots(x)
    a, b = (ok & 1) != 0, (ok & 2) != 0
    normal = np.isfinite(x) & (np.abs(x) >= 2.0 ** -1022)
    assert np.array_equal(b, normal & (x > 0))
    assert np.array_equal(a, normal & (np.abs(x) < 2.0 ** 1022))   # 1/x normal
    with np.errstate(all="ignore"):
        assert np.array_equal(r[a], 1.0 / x[a])
        assert np.array_equal(s[b], np.sqrt(x[b]))
        # root and reciprocal root together: 2^-59 and the rounding, 0.51 ulp; the check rounds its own value once more
        ulp = np.spacing(np.sqrt(x[b]))
        assert np.all(np.abs(t[b] - np.sqrt(x[b])) <= ulp)
        q = (np.longdouble(rs[b]) * np.sqrt(np.longdouble(x[b])) - 1).astype(np.float64)
        assert np.all(np.abs(q) <= 0.51 * 2.0 ** -52 + 2.0 ** -62)
