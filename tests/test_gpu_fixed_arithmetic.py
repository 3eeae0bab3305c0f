"""The integer arithmetic of the FP64 sweep as the GPU runs it (its own high products, shifts and seeds), one call per
thread: reciprocals and roots against correctly rounded ones, the Osher flux against 60-digit decimals, with the bounds
that the same code meets on the CPU."""
import ctypes
import os
import shutil
import subprocess
from decimal import Decimal

import numpy as np
import pytest

from test_fixed_flux import ROOT, exact, states_of
from test_fixed_flux_limits import draw
from test_fixed_roots import arguments

pytestmark = pytest.mark.gpu

WRAPPER = r'''
#include <cuda_runtime.h>
#include "ac_device.cuh"
using namespace acgb;
__global__ void roots(const double *x, long n, double *r, double *s, double *t, double *rs) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = Ar<double>::rcp(x[i]);
    s[i] = Ar<double>::sqrt_(x[i]);
    Ar<double>::sqrt_rsqrt(x[i], t[i], rs[i]);
}
__global__ void fluxes(const double *x, long n, const FixedBeta fb, const FixedScale sc, const FixedScale scp, double *F,
                       double *took) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double *s = x + 8 * i;
    took[i] = fixed_flux_ok(s[0], s[1], s[2], s[3], s[4], s[5], s[6], s[7], fb);
    if (took[i] != 0.0) osher_flux_fixed(s[0], s[1], s[2], s[3], s[4], s[5], s[6], s[7], fb, sc, scp, F + 4 * i);
}
extern "C" int run(const double *x, long nx, double beta, double sc, double scp, double *out, long nout) {
    double *dx = nullptr, *d = nullptr;
    cudaError_t e = cudaMalloc(&dx, nx * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&d, nout * sizeof(double));
    if (e == cudaSuccess) e = cudaMemset(d, 0, nout * sizeof(double));
    if (e == cudaSuccess) e = cudaMemcpy(dx, x, nx * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && beta == 0.0) {
        roots<<<(unsigned)((nx + 127) / 128), 128>>>(dx, nx, d, d + nx, d + 2 * nx, d + 3 * nx);
        e = cudaGetLastError();
    } else if (e == cudaSuccess) {
        const long n = nx / 8;
        fluxes<<<(unsigned)((n + 127) / 128), 128>>>(dx, n, make_fixed_beta(beta), make_fixed_scale(sc),
                                                     make_fixed_scale(scp), d, d + 4 * n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, d, nout * sizeof(double), cudaMemcpyDeviceToHost);
    cudaFree(dx);
    cudaFree(d);
    return (int)e;
}
'''


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_2108_08769_gb300 import build
    d = tmp_path_factory.mktemp("gpu_fixed")
    (d / "w.cu").write_text(WRAPPER)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-I" + os.path.join(ROOT, "paper_2108_08769_gb300", "csrc"),
                    "-shared", str(d / "w.cu"), "-o", str(d / "w.so")], check=True)
    lib = ctypes.CDLL(str(d / "w.so"))

    def call(x, nout, beta=0.0, scale=1.0, scale_p=1.0):
        x, out = np.ascontiguousarray(x, dtype=np.float64), np.zeros(nout)
        D, L, p = ctypes.c_double, ctypes.c_long, lambda a: a.ctypes.data_as(ctypes.c_void_p)
        assert lib.run(p(x), L(x.size), D(beta), D(scale), D(scale_p), p(out), L(nout)) == 0
        return out
    return call


def test_reciprocals_and_roots(run):
    x = arguments()
    r, s, t, rs = run(x, 4 * x.size).reshape(4, -1)
    with np.errstate(all="ignore"):
        # the library's functions take over past the normal range: every argument agrees
        assert np.array_equal(r, 1.0 / x, equal_nan=True)
        assert np.array_equal(s, np.sqrt(x), equal_nan=True)
        b = np.isfinite(x) & (x >= 2.0 ** -1022)
        assert np.all(np.abs(t[b] - np.sqrt(x[b])) <= np.spacing(np.sqrt(x[b])))
        assert np.all(np.abs(rs[b] * np.sqrt(x[b]) - 1) <= 4 * 2.0 ** -52)   # three roundings of the check's own


@pytest.mark.parametrize("scale,scale_p", [(1.0, 1.0), (128.0, 51.2e6), (0.3, 7.7e-9), (1.0 / 3e5, 1e17)])
def test_flux(run, scale, scale_p):
    rng = np.random.default_rng(12)
    groups = {}
    for kind in ("smooth", "interface", "near rest", "riemann"):
        for _ in range(60):
            s, beta = states_of(kind, rng)
            groups.setdefault(beta, []).append(s)
    for ratio in (1e-9, 1e-3, 0.5, 3.9, 4.4, 100.0):
        for beta in (1.0, 4e5, 3e-7):
            groups.setdefault(beta, []).extend(draw(rng, ratio, beta, 10 ** rng.uniform(-3, 3)))
    took = 0
    for beta, faces in groups.items():
        n = len(faces)
        out = run(np.array(faces).ravel(), 5 * n, beta, scale, scale_p)
        F, ok = out[:4 * n].reshape(n, 4), out[4 * n:] != 0
        took += ok.sum()
        for s, got in zip(np.array(faces)[ok], F[ok]):
            want, S = exact(list(s), beta)
            for k in range(4):
                f = Decimal(scale_p if k == 3 else scale)
                assert abs(Decimal(got[k]) - f * want[k]) <= 32 * Decimal(2) ** -53 * f * S[k], (k, s, beta)
    assert took > 350
