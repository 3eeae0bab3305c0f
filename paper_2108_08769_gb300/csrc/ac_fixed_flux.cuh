// ac_fixed_flux.cuh -- the Osher flux of the FP64 sweep, and FP64
// reciprocals and square roots, on the integer pipes.
//
// GB300's FP64 unit takes 16 cycles per warp instruction (one unit an SM, so
// each of the four sub-partitions gets a turn every 64), while 64-bit integer
// adds, shifts and 64-bit high products take a sub-partition about 2, 4 and 14
// and run beside it.  So the flux, three quarters of the FP64 sweep's work, is
// evaluated in block fixed point: every quantity is a 64-bit integer and a
// binary exponent of its own or of the face's largest term of its kind, 56 bits
// or more of that term (FP64 keeps 53), and the sweep's other arithmetic keeps
// the FP64 unit busy meanwhile.  A flux takes about 1800 instructions (2900
// cycles per warp with four warps on a sub-partition, near the integer
// multiplier's rate) where the FP64 form took about 150 FP64 instructions,
// 10,000 cycles.  One pseudo-iteration of the 256x256 tank: 193 -> 87 us, of a
// 1024x512 tank 1440 -> 568 us (with the rest of the sweep thinned out to
// match, see stage_kernel); the FP64 unit is then busy 42-44 % of the cycles,
// not 80 %.  The error of 2F against 113-bit arithmetic, in units of 2^-53 of
// its terms, is 0.3-0.9 rms where the FP64 formula's is 0.7-1.7, over the faces
// that fixed_flux_ok accepts.
//
// A value is the pair (int, E): int 2^E.  "Q61" and the like: a number in
// [0, 1] scaled by 2^61.
//
// Everything is host code too (the seeds of the reciprocal and of the
// reciprocal square root come from float division there), so that the
// arithmetic is tested on the CPU.
#pragma once

#include <cstring>

#include <cmath>
#include <stdint.h>

#if defined(__CUDACC__)
#define ACFX __host__ __device__ __forceinline__
#else
#define ACFX static inline
#endif

namespace acgb {

// 8 beta and 1/(4 beta) as (63-bit mantissa, exponent); formed once on the host.
struct FixedBeta {
    uint64_t b8, ib4, tib4;   // ib4: 8/9 of 1/(4 beta) (see fx::k89); tib4: sqrt(3/5)/2 times it, at the same exponent
    int eb8, eib4;
    uint32_t most;            // most of rho u^2, as in fixed_flux_ok
};

// A positive factor of the returned flux as (63-bit mantissa in [2^62, 2^63), exponent).
struct FixedScale {
    uint64_t m;
    int e;
};
inline FixedScale make_fixed_scale(double x) {
    int e;
    const double m = frexp(x, &e);
    return FixedScale{(uint64_t)ldexp(m, 63), e - 63};
}

inline FixedBeta make_fixed_beta(double beta) {
    int e;
    const double m = frexp(beta, &e);                       // beta = m 2^e, m in [1/2, 1)
    const uint64_t mant = (uint64_t)ldexp(m, 63);           // [2^62, 2^63), exact
    FixedBeta f;
    f.b8 = mant;                                            // 8 beta = mant 2^(e - 63 + 3)
    f.eb8 = e - 60;
    // 8/9 of 1/(4 beta) = 2^(63 - e - 2) / mant is ib4 2^(61 - e - 125), ib4 = 8/9 2^125 / mant below 2^63
    f.ib4 = (uint64_t)((((unsigned __int128)1 << 127) / 9 * 2) / mant);
    f.eib4 = 61 - e - 125;
    f.tib4 = (uint64_t)(((unsigned __int128)f.ib4 * 7144393258922745604ull) >> 64);
    const double b16 = 16.0 * beta;
    uint64_t u;
    memcpy(&u, &b16, 8);
    f.most = (uint32_t)(u >> 32) + ((2u * 1023u) << 20);    // high word of 16 beta, biased as those of rho and twice u
    return f;
}

namespace fx {

constexpr uint64_t kT64 = 14288786517845491209ull; // sqrt(3/5) 2^64 (outer Gauss points at (1 -+ sqrt(3/5))/2)
constexpr uint64_t k89 = 16397105843297379214ull;  // 8/9 2^64: the weights 5/18, 8/18, 5/18 are 8/9 of 5/16, 1/2, 5/16
constexpr int64_t kOff = (int64_t)1 << 62;

ACFX uint64_t wide(uint32_t a, uint32_t b) { return (uint64_t)a * b; }

ACFX uint32_t high(uint32_t a, uint32_t b) {
#if defined(__CUDA_ARCH__)
    return __umulhi(a, b);
#else
    return (uint32_t)(wide(a, b) >> 32);
#endif
}

// a b 2^-64 for a, b <= 2^63, to within 3 units below: the product of the low words and the low halves of the
// mixed ones are left out (high products take 4 cycles, wide ones 6)
ACFX uint64_t mulu(uint64_t a, uint64_t b) {
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    return wide(ah, bh) + (high(al, bh) + high(ah, bl));   // the high halves' sum fits in 32 bits
}
// the whole high product
ACFX uint64_t mulhi(uint64_t a, uint64_t b) {
#if defined(__CUDA_ARCH__)
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
// mulu for 0 <= a <= 2^63 and a signed |b| <= 2^62: b is offset by 2^62 (signed wide products cost twice
// the unsigned ones)
ACFX int64_t smul(uint64_t a, int64_t b) { return (int64_t)mulu(a, (uint64_t)(b + kOff)) - (int64_t)(a >> 2); }
// and for both signed, |a|, |b| <= 2^62
ACFX int64_t ssmul(int64_t a, int64_t b) {
    return (int64_t)mulu((uint64_t)(a + kOff), (uint64_t)(b + kOff)) - ((a + b) >> 2) - ((int64_t)1 << 60);
}
// right shifts by any s >= 0 (64 and more: 0, or -1 for a negative x)
ACFX int64_t sar(int64_t x, int s) {
#if defined(__CUDA_ARCH__)
    int64_t r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
    return r;
#else
    return x >> (s > 63 ? 63 : s);
#endif
}
ACFX uint64_t shr(uint64_t x, int s) {
#if defined(__CUDA_ARCH__)
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
    return r;
#else
    return s > 63 ? 0 : x >> s;
#endif
}
ACFX int clz(uint64_t x) {   // x != 0
#if defined(__CUDA_ARCH__)
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}
ACFX int clz32(uint32_t x) {   // x != 0
#if defined(__CUDA_ARCH__)
    return __clz((int)x);
#else
    return __builtin_clz(x);
#endif
}
ACFX int imax(int a, int b) { return a > b ? a : b; }
// x where m = 0, -x where m = -1
ACFX int64_t neg_if(int64_t x, int m) { return (x ^ (int64_t)m) - (int64_t)m; }

ACFX uint64_t bits_of(double x) {
#if defined(__CUDA_ARCH__)
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    memcpy(&u, &x, 8);
    return u;
#endif
}

// A double as sign, 63-bit mantissa in [2^62, 2^63) and exponent.  Zeros and subnormals become positive numbers near
// 2^-1022, which vanish beside any normal number (a negative one would leave -1 behind where it is shifted far to the
// right) and which to_double makes zero again.
struct Num {
    uint64_t m;
    int e, s;   // s = -1 for a negative number, else 0
};
ACFX Num unpack(double x) {
    const uint64_t u = bits_of(x);
    const int hi = (int)(u >> 32);
    Num n;
    const int ex = (hi >> 20) & 0x7ff;
    n.s = ex == 0 ? 0 : hi >> 31;
    n.e = ex - 1085;
    n.m = ((u & 0xfffffffffffffull) | 0x10000000000000ull) << 10;
    return n;
}

ACFX double double_of(uint64_t u) {
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)u);
#else
    double d;
    memcpy(&d, &u, 8);
    return d;
#endif
}

// i 2^e times the factor f, rounded to nearest (a tie upwards in magnitude), |i| < 2^62 and the result below 2^1022;
// results below 2^-900 become zero.  In integers throughout: the conversion instruction is the FP64 unit's.
ACFX double to_double(int64_t i, int e, const FixedScale &f) {
    const int sg = (int)(i >> 63);
    const uint64_t m = (uint64_t)neg_if(i, sg);
    const int z = clz(m | 1) - 1;                        // >= 1
    uint64_t r = mulu(m << z, f.m);                      // [2^60, 2^62)
    const int up = (int)((r >> 61) ^ 1);
    r = ((r << up) + 256) >> 9;                          // [2^52, 2^53]: 53 bits, or the carry
    const int ex = e + f.e + 1147 - z - up;              // biased exponent less one: the leading bit adds it back
    const uint32_t hi = (uint32_t)(r >> 32) + ((uint32_t)ex << 20) + ((uint32_t)sg << 31);
    return ex < 123 || m == 0 ? 0.0 : double_of(((uint64_t)hi << 32) | (uint32_t)r);
}

ACFX float float_of_bits(uint32_t b) {
#if defined(__CUDA_ARCH__)
    return __uint_as_float(b);
#else
    float f;
    memcpy(&f, &b, 4);
    return f;
#endif
}
ACFX uint32_t bits_of_float(float f) {
#if defined(__CUDA_ARCH__)
    return __float_as_uint(f);
#else
    uint32_t b;
    memcpy(&b, &f, 4);
    return b;
#endif
}
ACFX float seed_rcp(float x) {
#if defined(__CUDA_ARCH__)
    return __fdividef(1.0f, x);
#else
    return 1.0f / x;
#endif
}
ACFX float seed_rsqrt(float x) {
#if defined(__CUDA_ARCH__)
    return rsqrtf(x);
#else
    return 1.0f / sqrtf(x);
#endif
}

// y0 + y0 s for y0 = Y0 2^-21 (Y0 < 2^23) and |s| < 2^-19 given as S = s 2^k, |S| < 2^63, as an integer
// scaled by 2^(k - 11 - drop): the last correction of both iterations below.
ACFX uint64_t corrected(uint32_t Y0, int64_t S, int drop) {
    const uint64_t o = (uint64_t)S + ((uint64_t)1 << 63);
    const uint64_t p = wide(Y0, (uint32_t)(o >> 32)) + (wide(Y0, (uint32_t)o) >> 32);   // Y0 (S + 2^63) 2^-32
    return (uint64_t)(((int64_t)(p - ((uint64_t)Y0 << 31))) >> drop);
}

// 2^61/x of x = X 2^-62 in [1/2, 1): a 21-bit float seed and one step of the
// geometric series 1/x = y0 (1 + e + e^2 + ...), e = 1 - x y0 (|e| < 2^-20, exact
// from the low 64 bits of X Y0).  Error below 2^-59 of the result.
ACFX uint64_t rcp61(uint64_t X) {
    const uint32_t xh = (uint32_t)(X >> 32);                                       // [2^29, 2^30)
    const float x = float_of_bits(((xh >> 6) & 0x7fffffu) | 0x3f000000u);          // x truncated to 24 bits
    const uint32_t Y0 = bits_of_float(seed_rcp(x) + 4.0f) & 0x7fffffu;             // y0 in (1, 2], scaled by 2^21
    const int64_t E = -(int64_t)(X * Y0);                                          // e 2^83
    const int32_t eh = (int32_t)(E >> 32);
    const uint32_t ea = (uint32_t)(eh < 0 ? -eh : eh);
    const int64_t S = E + (int64_t)(wide(ea, ea) >> 19);                           // (e + e^2) 2^83
    return ((uint64_t)Y0 << 40) + corrected(Y0, S, 11);                            // (.. 2^104 - 32 - 11) = 2^61
}

// 2^61/sqrt(x) of x = X 2^-62 in [1/4, 1): the same seed width and the binomial series
// 1/sqrt(x) = y0 (1 + e/2 + 3/8 e^2 + ...), e = 1 - x y0^2 (|e| < 2^-19).  Error below 2^-58 of the result.
ACFX uint64_t rsqrt61(uint64_t X) {
    const uint32_t xh = (uint32_t)(X >> 32), xl = (uint32_t)X;                     // xh in [2^28, 2^30)
    const float x = (float)(int)xh * 9.31322574615478515625e-10f;                  // 2^-30
    const uint32_t Y0 = bits_of_float(seed_rsqrt(x) + 4.0f) & 0x7fffffu;           // y0 in (1, 2], scaled by 2^21
    const uint64_t W = wide(Y0, Y0);                                               // y0^2 2^42 (45 bits)
    const uint32_t wh = (uint32_t)(W >> 32), wl = (uint32_t)W;
    // X W 2^-32, mod 2^64: (1 - e) 2^72
    const uint64_t R = wide(xh, wl) + wide(xl, wh) + (wide(xl, wl) >> 32) + ((uint64_t)(xh * wh) << 32);
    const int64_t E = -(int64_t)R;                                                 // e 2^72, |.| < 2^53
    const int32_t eh = (int32_t)(E >> 22);                                         // e 2^50
    const uint32_t ea = (uint32_t)(eh < 0 ? -eh : eh);
    const uint32_t e2 = (uint32_t)(wide(ea, ea) >> 32);                            // e^2 2^68
    const int64_t S = E + (int64_t)(12ull * e2);                      // (e/2 + 3/8 e^2) 2^73
    return ((uint64_t)Y0 << 40) + corrected(Y0, S, 1);                             // (.. 2^94 - 32 - 1) = 2^61
}


// 1/x correctly rounded, where x and 1/x are normal (rcp_ok): the quotient's rounding or one unit less, by a limit
// 8 units of 2^61 (the iteration's error) above the half, then one unit up where the remainder says so.
ACFX bool rcp_ok(double x) { return ((uint32_t)(bits_of(x) >> 52) & 0x7ff) - 1u < 2044u; }
ACFX double rcp(double x) {
    const uint64_t u = bits_of(x);
    const uint32_t hi = (uint32_t)(u >> 32);
    const uint64_t m = (u & 0xfffffffffffffull) | 0x10000000000000ull;   // [2^52, 2^53)
    uint64_t r = (rcp61(m << 9) + 248) >> 9;             // 2^105/m, in [2^52, 2^53], or one less
    const int64_t e = -(int64_t)(r * m) * 2;             // 2 (2^105 - r m), from its low 64 bits; never a tie
    r += e > (int64_t)m;
    const uint32_t ex = 2044u - ((hi >> 20) & 0x7ffu);
    return double_of(r + ((uint64_t)((ex << 20) | (hi & 0x80000000u)) << 32));
}
// Mantissa m 2^-62 in [1/4, 1) and half the (even) exponent of a positive normal x = m 2^(2h - 62) (rsqrt_ok).
struct RootArg {
    uint64_t m;
    int h;
};
ACFX bool rsqrt_ok(double x) { return (uint32_t)(bits_of(x) >> 52) - 1u < 2046u; }
ACFX RootArg root_arg(double x) {
    const uint64_t u = bits_of(x);
    const int ex = (int)(u >> 52);
    const int even = (ex & 1) ^ 1;                       // an even power of two either way
    return RootArg{((u & 0xfffffffffffffull) | 0x10000000000000ull) << (8 + even), (ex - 1021 - even) / 2};
}
// sqrt(x) and 1/sqrt(x) to within 0.51 ulp.
ACFX void sqrt_rsqrt(double x, double &s, double &rs) {
    const RootArg a = root_arg(x);
    const uint64_t y = rsqrt61(a.m);
    rs = double_of(((y + 256) >> 9) + ((uint64_t)(1022 - a.h) << 52));
    const uint64_t c = mulu(a.m * 2, y * 2);             // sqrt(x') 2^61 in [2^60, 2^61]
    s = double_of(((c + 128) >> 8) + ((uint64_t)(1021 + a.h) << 52));
}
// sqrt(x) correctly rounded, by its remainder as in rcp.
ACFX double sqrt_rn(double x) {
    const RootArg a = root_arg(x);
    uint64_t s = (mulu(a.m * 2, rsqrt61(a.m) * 2) + 112) >> 8;           // sqrt(m 2^44), in [2^52, 2^53], or one less
    const int64_t e = (int64_t)((a.m << 44) - s * s);    // below 3.1 s; (s + 1/2)^2 is s^2 + s and a quarter
    s += e > (int64_t)s;
    return double_of(s + ((uint64_t)(1021 + a.h) << 52));
}

// |x|
ACFX uint64_t mag(int64_t x) { return (uint64_t)neg_if(x, (int)(x >> 63)); }
// leading zeros beyond the second bit: x << room(x) lies in [2^61, 2^62) (x < 2^62; 61 for x = 0)
ACFX int room(uint64_t x) { return clz(x | 1) - 2; }
// 9/8 of the quadrature sum: 5/16 of the outer points' sum and half of the middle one
ACFX int64_t weighted(int64_t outer, int64_t mid) { return (outer >> 2) + (outer >> 4) + (mid >> 1); }
ACFX uint64_t weighted(uint64_t outer, uint64_t mid) { return (outer >> 2) + (outer >> 4) + (mid >> 1); }

// One Gauss point's part of the flux: what the second loop needs of it.
struct Point {
    uint64_t u;   // |u|, exponent em - er - 61 + k
    int k;
    int sg;       // sign of u (0 or -1)
    uint64_t a;   // a = |u|/c, Q61
    uint64_t c;   // 4 c 2^-ec, <= 2^63
    int ec;
    uint64_t b;   // |b|, exponent ec + k + eb
};

}  // namespace fx

// Osher flux of one face (Dumbser and Toro, 3 Gauss points on the straight
// path in Q): 2F = (mass, normal momentum, tangential momentum, p/beta flux),
// returned times sc, the last component times scp; inputs as osher_flux.
// Requires states that fixed_flux_ok accepts.
//
// |A| has the eigenvalues u (three times) and (u +- c)/2 of opposite signs,
// so with sg = sign(u) it is sg A + 2 |l| r l^T, rank one beside A itself, l
// being the acoustic speed whose sign is not u's.  On the straight path
// d(rho u) - u d(rho) is rho_L rho_R (u_R - u_L) / rho at every point.  In
// a = |u|/c, with s = (1 - a)^2, h = a (1 - a)(3 - a) and
// b = c rho_L rho_R (u_R - u_L) / rho, that is
//   |A| dQ = |u| dQ' + (r Z, m Z + G, n Z, Z - u (G - sg dp)/beta),
//   G = s b/2 + sg a dp,   Z = c (2 s dp + sg h b) / (4 beta),
// dQ' = (d rho, d(rho u), d(rho v), 0): the one difference of terms that may
// be nearly equal is 1 - a (fixed_flux_ok bounds a), and every factor but c, u,
// b and dp lies in [0, 1].  With
// r_j = (rS -+ t dr)/2 and so on, sums over the points of r Z need only the
// sum of Z and the difference of the outer points' Z.
ACFX void osher_flux_fixed(double rLd, double uLd, double vLd, double pLd, double rRd, double uRd, double vRd,
                           double pRd, const FixedBeta &fb, const FixedScale &sc, const FixedScale &scp, double F[4]) {
    using namespace fx;
    // ---- unpack; products rho u, rho v from the full mantissas ----
    const Num rL = unpack(rLd), rR = unpack(rRd), uL = unpack(uLd), uR = unpack(uRd);
    const Num vL = unpack(vLd), vR = unpack(vRd);
    const uint64_t ML = mulu(rL.m, uL.m), MR = mulu(rR.m, uR.m), NL = mulu(rL.m, vL.m), NR = mulu(rR.m, vR.m);
    const int emL = rL.e + uL.e + 64, emR = rR.e + uR.e + 64, enL = rL.e + vL.e + 64, enR = rR.e + vR.e + 64;
    // sums and differences of the two sides on common exponents, |.| < 2^62
    const int em = imax(emL, emR) + 1, en = imax(enL, enR) + 1, er = imax(rL.e, rR.e) + 1, ed = imax(uL.e, uR.e) + 2;
    const int64_t mL = neg_if((int64_t)shr(ML, em - emL), uL.s), mR = neg_if((int64_t)shr(MR, em - emR), uR.s);
    const int64_t c0 = mL + mR, DM = mR - mL;
    const int64_t nL = neg_if((int64_t)shr(NL, en - enL), vL.s), nR = neg_if((int64_t)shr(NR, en - enR), vR.s);
    const int64_t nS = nL + nR, DN = nR - nL;
    const uint64_t rLa = shr(rL.m, er - rL.e), rRa = shr(rR.m, er - rR.e);
    const uint64_t rS = rLa + rRa;                       // [2^61, 2^63)
    const int64_t DR = (int64_t)(rRa - rLa);
    const int64_t uLa = neg_if((int64_t)shr(uL.m, ed - uL.e), uL.s), uRa = neg_if((int64_t)shr(uR.m, ed - uR.e), uR.s);
    const int64_t US = uLa + uRa, DU = uRa - uLa;
    const Num pL = unpack(pLd), pR = unpack(pRd);
    const int ep = imax(pL.e, pR.e) + 2;
    const int64_t pLa = neg_if((int64_t)shr(pL.m, ep - pL.e), pL.s), pRa = neg_if((int64_t)shr(pR.m, ep - pR.e), pR.s);
    const int64_t PS = pLa + pRa, DPs = pRa - pLa;
    // jumps of p and u as signs and magnitudes in [2^61, 2^62); the point sums below are formed times sd = sign(du)
    const int sd = (int)(DU >> 63), sp = (int)(DPs >> 63) ^ sd;
    uint64_t DP = mag(DPs), du = mag(DU);
    const int kd = room(DP), ku = room(du);
    DP <<= kd;
    du <<= ku;
    // a zero jump's exponent is below all others, so that no common exponent is formed for its sake
    const int none = -16384;
    const int epd = (uint32_t)(DP >> 32) == 0 ? none : ep - kd;
    // 2 rho_L rho_R |du| in [2^62, 2^63) (or 0)
    uint64_t D = mulu(mulu(rL.m, rR.m) * 2, du * 2);     // [2^59, 2^62)
    const int kD = clz32((uint32_t)(D >> 32) | 1u) - 1;
    D <<= kD;
    int eb = (uint32_t)(du >> 32) == 0 ? none : rL.e + rR.e + (ed - ku) + 128 - kD - er;
    // ---- first loop: u, c, a, b at the Gauss points (twice the states: r' = rS -+ t dr, m' = c0 -+ t dm) ----
    const int64_t TR = neg_if((int64_t)mulhi(kT64, mag(DR)), (int)(DR >> 63));
    const int64_t TM = neg_if((int64_t)mulhi(kT64, mag(DM)), (int)(DM >> 63));
    Point q[3];
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int j = 0; j < 3; ++j) {
        const uint64_t r = j == 0 ? rS - (uint64_t)TR : (j == 1 ? rS : rS + (uint64_t)TR);
        const int64_t m = j == 0 ? c0 - TM : (j == 1 ? c0 : c0 + TM);
        const int k = clz32((uint32_t)(r >> 32)) - 2;    // -1 .. 3 (r in [2^58.8, 2^63))
        const uint64_t X = k < 0 ? r >> 1 : r << k;      // [2^61, 2^62)
        const uint64_t Y = rcp61(X) * 2;                 // 1/r' = Y 2^(k - er - 124), Y in (2^62, 2^63]
        q[j].k = k;
        q[j].sg = (int)(m >> 63);
        q[j].u = mulu(mag(m) * 2, Y);                    // < 2^62
        const int n = clz(q[j].u | 1) - 1;
        const uint64_t un = q[j].u << n;                 // [2^62, 2^63) unless u = 0
        const int eun = em - er - 61 + k - n;
        // c^2 = u^2 + 8 beta / r'
        const uint64_t f = mulu(fb.b8, Y);               // [2^60, 2^62]
        const int ef = fb.eb8 + k - er - 60;
        const uint64_t u2 = mulu(un, un);                // [2^60, 2^62)
        const int eu2 = 2 * eun + 64;
        int e2 = imax(ef, eu2) + 2;
        uint64_t M = shr(f, e2 - ef) + shr(u2, e2 - eu2);   // [2^58, 2^61]
        int sh = clz32((uint32_t)(M >> 32)) - 2;
        sh -= (e2 - sh) & 1;
        M <<= sh;                                        // [2^60, 2^62), even exponent
        e2 -= sh;
        const uint64_t R = rsqrt61(M) * 2;               // 1/c = R 2^(-93 - e2/2)
        q[j].c = mulu(M * 2, R) * 4;                     // [2^62, 2^63]
        q[j].ec = e2 / 2 - 30;
        // a = |u|/c <= 1 in Q61
        const uint64_t a = shr(mulu(un, R), imax(0, e2 / 2 - 32 - eun));
        const uint64_t one = (uint64_t)1 << 61;
        q[j].a = a < one ? a : one;
        q[j].b = mulu(q[j].c, mulu(D, Y) * 2);           // < 2^62
    }
    const int nb = room(q[0].b | q[1].b | q[2].b);
    for (int j = 0; j < 3; ++j) q[j].b <<= nb;
    eb -= nb;
    // ---- second loop: G, Z and their sums, on exponents common to the points ----
    const int ecx = imax(q[0].ec, imax(q[1].ec, q[2].ec));
    const int kx = imax(q[0].k, imax(q[1].k, q[2].k));
    const int ebx = imax(q[0].ec + q[0].k, imax(q[1].ec + q[1].k, q[2].ec + q[2].k)) + eb;
    uint64_t U[3];
    for (int j = 0; j < 3; ++j) U[j] = shr(q[j].u, kx - q[j].k);
    const int nu = room(U[0] | U[1] | U[2]), eu = em - er - 61 + kx - nu;
    for (int j = 0; j < 3; ++j) U[j] <<= nu;
    const int eg = imax(epd + 2, ebx + 1);
    const uint64_t DP4 = shr(DP, eg - 2 - epd);          // 4 |dp|
    int64_t G[3], Z[3], H[3];
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int j = 0; j < 3; ++j) {
        const int x = q[j].sg ^ sp;                      // the sign of sg sd dp
        const uint64_t b2 = shr(q[j].b, eg - 1 - (q[j].ec + q[j].k + eb));   // 2 |b|
        const uint64_t a4 = q[j].a * 4, y4 = ((uint64_t)1 << 63) - a4;  // a, y = 1 - a in Q63
        const uint64_t s = mulu(y4, y4), s2 = s * 2;     // s = y^2 in Q62, Q63
        const uint64_t t = (y4 >> 1) - s;                // a (1 - a) = y - y^2 >= 0 (s is rounded down) in Q62
        const uint64_t h2 = t * 4 + mulu(t * 2, y4) * 2; // h = t (2 + y) in Q63
        G[j] = (int64_t)(mulu(s2, b2) >> 1) + neg_if((int64_t)(mulu(a4, DP4) >> 1), x);
        const int64_t g = G[j] - neg_if((int64_t)(DP4 >> 2), x);             // G - sg dp
        const int64_t z = (int64_t)mulu(h2, b2) + neg_if((int64_t)mulu(s2, DP4), x);   // sg (2 s dp + sg h b)
        // sg is applied last, so that states mirrored in u give exactly opposite Z
        Z[j] = neg_if(sar(smul(q[j].c, z), ecx - q[j].ec), q[j].sg);    // exponent ecx + eg + 62
        H[j] = neg_if(smul(U[j] * 2, g), q[j].sg);       // u (G - sg dp), exponent eu + eg + 63
    }
    const uint64_t SU = mulu(k89 >> 1, weighted(U[0] + U[2], U[1]) * 2);
    const int64_t SG = neg_if(smul(k89 >> 1, weighted(G[0] + G[2], G[1])) * 2, sd);
    const int64_t SZ = weighted(Z[0] + Z[2], Z[1]);      // times 8/9 to come, with 1/(4 beta)
    const int64_t SH = weighted(H[0] + H[2], H[1]);
    const int64_t dz = Z[2] - Z[0];
    int64_t TZ = neg_if(smul(fb.tib4, (dz >> 2) + (dz >> 4)), sd);   // t/2 times the outer points' difference
    int64_t ZV = neg_if(smul(fb.ib4, SZ), sd);
    int ez = ecx + eg + 126 + fb.eib4;
    const int nz = room(mag(ZV) | mag(TZ));
    ZV = (int64_t)((uint64_t)ZV << nz);
    TZ = (int64_t)((uint64_t)TZ << nz);
    ez -= nz;
    const int ev = imax(eu, ez) + 1;
    const int64_t S1 = (int64_t)shr(SU, ev - eu) + sar(TZ, ev - ez), Zv = sar(ZV, ev - ez);   // |.| < 2^62
    // ---- 2F = F(Q_L) + F(Q_R) - D, each sum on the exponent of its largest term ----
    {
        const int ex = er + ev + 64, e = imax(em, ex) + 1;
        F[0] = to_double(sar(c0, e - em) - sar(ssmul(DR, S1) + (smul(rS, Zv) >> 1), e - ex), e, sc);
    }
    {
        const int eL = emL + uL.e + 64, eR = emR + uR.e + 64, ex = em + ev + 64;
        const int e = imax(imax(eL, eR), imax(ep, imax(ex, eg))) + 3;
        const int64_t t = sar(PS, e - ep) - sar(ssmul(DM, S1) + (ssmul(c0, Zv) >> 1), e - ex) - sar(SG, e - eg);
        F[1] = to_double(t + (int64_t)shr(mulu(ML, uL.m), e - eL) + (int64_t)shr(mulu(MR, uR.m), e - eR), e, sc);
    }
    {
        const int eL = emL + vL.e + 64, eR = emR + vR.e + 64, ex = en + ev + 64;
        const int e = imax(imax(eL, eR), ex) + 2;
        const int64_t l = neg_if((int64_t)shr(mulu(ML, vL.m), e - eL), uL.s ^ vL.s);
        const int64_t r = neg_if((int64_t)shr(mulu(MR, vR.m), e - eR), uR.s ^ vR.s);
        F[2] = to_double(l + r - sar(ssmul(DN, S1) + (ssmul(nS, Zv) >> 1), e - ex), e, sc);
    }
    {
        const int eh = eu + eg + 129 + fb.eib4;          // H's sum over beta, 4 ib4
        const int e = imax(ed, imax(ev, eh)) + 2;
        F[3] = to_double(sar(US, e - ed) - sar(Zv, e - ev) + sar(neg_if(smul(fb.ib4, SH), sd), e - eh), e, scp);
    }
}

// Whether osher_flux_fixed takes these states: densities within 2^-250 .. 2^250, the others below 2^250 in
// magnitude (so finite), which keeps every result far inside the range of a double (fixed_beta_ok).
ACFX bool fixed_flux_ok(double rL, double uL, double vL, double pL, double rR, double uR, double vR, double pR) {
    using namespace fx;
    const uint32_t lo = (1023u - 250u) << 20, most = (1023u + 250u) << 20;
    const uint32_t rl = (uint32_t)(bits_of(rL) >> 32) - lo, rr = (uint32_t)(bits_of(rR) >> 32) - lo;
    auto m = [](double x) { return (uint32_t)(bits_of(x) >> 32) & 0x7fffffffu; };
    auto max2 = [](uint32_t a, uint32_t b) { return a > b ? a : b; };
    return max2(rl, rr) < most - lo && max2(max2(max2(m(uL), m(uR)), max2(m(vL), m(vR))), max2(m(pL), m(pR))) < most;
}
// And whether it may run on them: besides the range, rho u^2/(4 beta) at most 4 or so on both sides.  1 - |u|/c is a
// difference of nearly equal terms where that ratio is large (an outer Gauss point's is at most 9 times the sides'
// larger one).  From 16 on the flux of p/beta is further off than in FP64 (rms in units of 2^-53 of its terms: 0.7
// and 1.3 at a ratio of 2 to 4, 3.6 and 3.0 at 16 to 32, 820 and 540 at 2^12).  The high words of doubles serve as
// their logarithms (0.09 low at most), so that the limit lies between 4.0 and 4.8.  beta is mostly rho c0^2 with c0
// ten times the velocities, and the ratio below 0.01.
ACFX bool fixed_flux_ok(double rL, double uL, double vL, double pL, double rR, double uR, double vR, double pR,
                        const FixedBeta &fb) {
    using namespace fx;
    auto q = [](double r, double u) {   // below 2^32 within the range
        return (uint32_t)(bits_of(r) >> 32) + 2u * ((uint32_t)(bits_of(u) >> 32) & 0x7fffffffu);
    };
    const uint32_t ql = q(rL, uL), qr = q(rR, uR);
    return fixed_flux_ok(rL, uL, vL, pL, rR, uR, vR, pR) && (ql > qr ? ql : qr) <= fb.most;
}
// The same for beta and the factors of the returned flux.
inline bool fixed_beta_ok(double beta) { return beta > 1e-70 && beta < 1e70; }

}  // namespace acgb
