// ac_state.cuh -- a tank's state in and out of its device form.
//
// The host's four FP64 fields are copied as they are into the tank's scratch
// (the two state buffers that do not hold the current state), checked there,
// and converted on the device; reading back forms level + increment there and
// copies four FP64 fields.  Formed on the host, cell by cell, the records and
// their checks took 253 ms (in) and 112 ms (out) for 2048x8192 cells, ten times
// the copies themselves.  Each kernel is one pass bounded by HBM but for
// mixed_pref_kernel, whose columns are serial sums.
#pragma once

#include "ac_kernels_mixed.cuh"

namespace acgb {

// The staged fields rho, rho u, rho v, p of N cells.
struct Staged {
    double *f[4];
};
// in two scratch record buffers of a mixed tank
inline Staged staged_in(float4 *s0, float4 *s1, size_t N) {
    double *a = reinterpret_cast<double *>(s0), *b = reinterpret_cast<double *>(s1);
    return Staged{{a, a + N, b, b + N}};
}

// *bad <- 1 where a value is not finite, a density not positive or outside [lo, hi].
static __global__ void check_fields_kernel(const Staged s, size_t N, double lo, double hi, int *bad) {
    bool ok = true;
    for (size_t g = blockIdx.x * (size_t)blockDim.x + threadIdx.x; g < N; g += (size_t)gridDim.x * blockDim.x) {
        const double r = s.f[0][g];
        ok = ok && isfinite(r) && r > 0.0 && !(r < lo) && !(r > hi) && isfinite(s.f[1][g]) && isfinite(s.f[2][g]) &&
             isfinite(s.f[3][g]);
    }
    if (!ok) *bad = 1;
}

// The real-time level Q^n := Q of the FP64 form, unless the fields are bad.
static __global__ void level_from_fields_kernel(const Staged s, Staged lev, size_t N, const int *bad) {
    if (*bad) return;
    for (size_t g = blockIdx.x * (size_t)blockDim.x + threadIdx.x; g < N; g += (size_t)gridDim.x * blockDim.x)
#pragma unroll
        for (int f = 0; f < 4; ++f) lev.f[f][g] = s.f[f][g];
}

// The mixed form's levels and records of a new state (d: the current
// increments), unless the fields are bad: Q^n and p^n in FP64, their FP32 copy
// with the reference density, zero increments (without a pressure level the
// record holds p and the level zero).
static __global__ void mixed_from_fields_kernel(const Staged s, const MixedArgs a, float4 *d, int use_ref, size_t N,
                                                const int *bad) {
    if (*bad) return;
    for (size_t g = blockIdx.x * (size_t)blockDim.x + threadIdx.x; g < N; g += (size_t)gridDim.x * blockDim.x) {
        const double r = s.f[0][g], m = s.f[1][g], n = s.f[2][g], p = s.f[3][g];
        const float rec = a.plevel ? 0.0f : float(p);
        a.q64[0][g] = r;
        a.q64[1][g] = m;
        a.q64[2][g] = n;
        a.q64[3][g] = a.plevel ? p : 0.0;
        a.qn[g] = make_float4(float(r), float(m), float(n), use_ref ? float(r) : 0.0f);
        d[g] = make_float4(0.0f, 0.0f, 0.0f, rec);
        a.lev_p[g] = rec;
    }
}

// The discrete hydrostatic columns of the FP32 reference density, anchored at
// each column's top cell, one thread per column (the sum's order is the
// column's): p_ref[j] = p_ref[j+1] - (rho_ref[j] + rho_ref[j+1]) gy dy / 2.
// Eight rows' densities are in flight at a time.
static __global__ void mixed_pref_kernel(const Staged s, double *pref, int nx, int ny, double gy, double dy,
                                         const int *bad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (*bad || i >= nx) return;
    const double *rho = s.f[0];
    size_t g = (size_t)(ny - 1) * nx + i;
    double p = s.f[3][g], above = double(float(rho[g]));
    pref[g] = p;
    for (int j = ny - 2; j >= 0; j -= 8) {
        double r[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) r[k] = j - k >= 0 ? rho[(size_t)(j - k) * nx + i] : 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (j - k < 0) break;
            const double here = double(float(r[k]));
            p = __dsub_rn(p, __dmul_rn(__dmul_rn(__dmul_rn(__dadd_rn(here, above), gy), dy), 0.5));
            above = here;
            pref[(size_t)(j - k) * nx + i] = p;
        }
    }
}

// State = FP64 level + FP32 increment, into the staged fields.
static __global__ void mixed_to_fields_kernel(const MixedArgs a, const float4 *d, Staged s, size_t N) {
    for (size_t g = blockIdx.x * (size_t)blockDim.x + threadIdx.x; g < N; g += (size_t)gridDim.x * blockDim.x) {
        const float4 e = d[g];
        s.f[0][g] = a.q64[0][g] + double(e.x);
        s.f[1][g] = a.q64[1][g] + double(e.y);
        s.f[2][g] = a.q64[2][g] + double(e.z);
        s.f[3][g] = a.q64[3][g] + double(e.w);
    }
}

// Enqueue the host fields' copies and their check on `s`; *bad is cleared first.
inline cudaError_t stage_fields(const double *const f[4], const Staged &st, size_t N, double lo, double hi, int *bad,
                                int blocks, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(int), s);
    for (int k = 0; k < 4 && e == cudaSuccess; ++k)
        e = cudaMemcpyAsync(st.f[k], f[k], N * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    check_fields_kernel<<<blocks, 256, 0, s>>>(st, N, lo, hi, bad);
    return cudaGetLastError();
}

// Enqueue the conversion of the staged fields (see the kernels).
inline cudaError_t mixed_from_fields(const Staged &st, const MixedArgs &a, float4 *d, bool use_ref, double gy, double dy,
                                     const int *bad, int blocks, cudaStream_t s) {
    const size_t N = (size_t)a.nx * a.ny;
    mixed_from_fields_kernel<<<blocks, 256, 0, s>>>(st, a, d, use_ref ? 1 : 0, N, bad);
    if (use_ref)
        mixed_pref_kernel<<<(a.nx + 31) / 32, 32, 0, s>>>(st, const_cast<double *>(a.pref64), a.nx, a.ny, gy, dy, bad);
    return cudaGetLastError();
}

}  // namespace acgb
