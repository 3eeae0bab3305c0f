// ac_fixed_flux.cuh -- the Osher flux of the FP64 sweep on the integer pipes.
//
// GB300's FP64 unit takes 16 cycles per warp instruction and SM (64 per
// sub-partition), while 64-bit integer adds, shifts and 64-bit high products
// take about 2, 4 and 16 cycles per sub-partition and run beside it.  So the
// flux, three quarters of the FP64 sweep's work, is evaluated in block fixed
// point: every quantity is a 64-bit integer with at least 57 significant
// bits and a binary exponent of its own or of its face (FP64 keeps 53), and
// the sweep's other arithmetic keeps the FP64 unit busy meanwhile.  One
// pseudo-iteration of the 256x256 tank: 193 -> 118 us, of a 1024x512 tank
// 1440 -> 741 us.  The error of 2F against 113-bit arithmetic, in units of
// 2^-53 of its terms, is 0.3-0.5 rms (1.0 at most in smooth flow) where the
// FP64 formula's is 0.7-1.7 (2.9).
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
    uint64_t b8, ib4;
    int eb8, eib4;
};

inline FixedBeta make_fixed_beta(double beta) {
    int e;
    const double m = frexp(beta, &e);                       // beta = m 2^e, m in [1/2, 1)
    const uint64_t mant = (uint64_t)ldexp(m, 63);           // [2^62, 2^63), exact
    FixedBeta f;
    f.b8 = mant;                                            // 8 beta = mant 2^(e - 63 + 3)
    f.eb8 = e - 60;
    // 1/(4 beta) = 2^(63 - e - 2) / mant = ib4 2^(61 - e - 125), ib4 = 2^125 / mant in (2^62, 2^63]
    const unsigned __int128 q = ((unsigned __int128)1 << 125) / mant;
    f.ib4 = q > (((uint64_t)1 << 63) - 1) ? (((uint64_t)1 << 63) - 1) : (uint64_t)q;
    f.eib4 = 61 - e - 125;
    return f;
}

namespace fx {

constexpr uint64_t kT = 7144393258922745604ull;    // sqrt(3/5) 2^63 (outer Gauss points at (1 -+ sqrt(3/5))/2)
constexpr uint64_t kT64 = 14288786517845491209ull; // sqrt(3/5) 2^64
constexpr uint64_t kW1 = 5124095576030431004ull;   // 5/18 2^64 (their weight)
constexpr uint64_t kW2 = 8198552921648689607ull;   // 8/18 2^64 (the middle point's)
constexpr int64_t kOff = (int64_t)1 << 62;

ACFX uint64_t wide(uint32_t a, uint32_t b) { return (uint64_t)a * b; }

// a b 2^-64 for a, b <= 2^63, to within 2 units below (the product of the low words is left out)
ACFX uint64_t mulu(uint64_t a, uint64_t b) {
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    return wide(ah, bh) + ((wide(al, bh) + wide(ah, bl)) >> 32);
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

// A double as sign, 63-bit mantissa in [2^62, 2^63) and exponent; zero (and
// subnormals) as mantissa 0.
struct Num {
    uint64_t m;
    int e, s;   // s = -1 for a negative number, else 0
};
ACFX Num unpack(double x) {
    const uint64_t u = bits_of(x);
    const int hi = (int)(u >> 32);
    const int ex = (hi >> 20) & 0x7ff;
    Num n;
    n.s = hi >> 31;
    n.e = ex - 1085;
    n.m = ex == 0 ? 0 : (((u & 0xfffffffffffffull) | 0x10000000000000ull) << 10);
    return n;
}
// The same of a positive normal double (its sign and exponent known to be so).
ACFX uint64_t mantissa(double x) { return ((bits_of(x) & 0xfffffffffffffull) | 0x10000000000000ull) << 10; }

// i 2^e rounded to nearest: the conversion rounds, the exponent is added to
// the bit pattern; results below the normal range become zero, above it infinite.
ACFX double to_double(int64_t i, int e) {
    const double d = (double)i;
    const uint64_t u = bits_of(d);
    int hi = (int)(u >> 32);
    const int ex = ((hi >> 20) & 0x7ff) + e;
    uint32_t lo = (uint32_t)u;
    hi += (int)((unsigned)e << 20);
    if (ex > 2046) { hi = (i < 0 ? (int)0x80000000 : 0) | 0x7ff00000; lo = 0; }
    if (ex < 1 || i == 0) { hi = 0; lo = 0; }
#if defined(__CUDA_ARCH__)
    return __hiloint2double(hi, (int)lo);
#else
    const uint64_t r = ((uint64_t)(uint32_t)hi << 32) | lo;
    double o;
    memcpy(&o, &r, 8);
    return o;
#endif
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


// |x|
ACFX uint64_t mag(int64_t x) { return (uint64_t)neg_if(x, (int)(x >> 63)); }
// leading zeros beyond the second bit: x << room(x) lies in [2^61, 2^62) (x < 2^62; 61 for x = 0)
ACFX int room(uint64_t x) { return clz(x | 1) - 2; }

// One Gauss point's part of the flux: what the second loop needs of it.
struct Point {
    uint64_t u;   // |u|, exponent em - er - 61 + k
    int k;
    int sg;       // sign of u (0 or -1)
    uint64_t a;   // a = |u|/c, Q61
    uint64_t c;   // 4 c 2^-ec, <= 2^63
    int ec;
    int64_t b;    // d(rho u) - u d(rho), then c times it
};

}  // namespace fx

// Osher flux of one face (Dumbser and Toro, 3 Gauss points on the straight
// path in Q), returned as 2F = (mass, normal momentum, tangential momentum,
// p/beta flux); inputs as osher_flux.  Requires finite inputs and normal
// positive densities (fixed_flux_ok).
//
// |A| has the eigenvalues u (three times) and (u +- c)/2 of opposite signs,
// so with sg = sign(u) it is sg A + 2 |l| r l^T, rank one beside A itself, l
// being the acoustic speed whose sign is not u's.  In a = |u|/c, with
// s = (1 - a)^2, h = a (1 - a)(3 - a) and b = c (d(rho u) - u d(rho)), that is
//   |A| dQ = |u| dQ' + (r Z, m Z + G, n Z, Z - u (G - sg dp)/beta),
//   G = s b/2 + sg a dp,   G - sg dp = s b/2 - sg (1 - a) dp,   Z = c (2 s dp + sg h b) / (4 beta),
// dQ' = (d rho, d(rho u), d(rho v), 0): no difference of nearly equal terms
// is left, and every factor but c, u, b and dp lies in [0, 1].  With
// r_j = (rS -+ t dr)/2 and so on, sums over the points of r Z need only the
// sum of Z and the difference of the outer points' Z.
ACFX void osher_flux_fixed(double rLd, double uLd, double vLd, double pLd, double rRd, double uRd, double vRd,
                           double pRd, const FixedBeta &fb, double F[4]) {
    using namespace fx;
    // ---- unpack; products rho u, rho v from the full mantissas ----
    const Num rL = unpack(rLd), rR = unpack(rRd), uL = unpack(uLd), uR = unpack(uRd);
    const Num vL = unpack(vLd), vR = unpack(vRd);
    const uint64_t ML = mulu(rL.m, uL.m), MR = mulu(rR.m, uR.m), NL = mulu(rL.m, vL.m), NR = mulu(rR.m, vR.m);
    const int emL = rL.e + uL.e + 64, emR = rR.e + uR.e + 64, enL = rL.e + vL.e + 64, enR = rR.e + vR.e + 64;
    // sums and differences of the two sides on common exponents, |.| < 2^62
    const int em = imax(emL, emR) + 1, en = imax(enL, enR) + 1, er = imax(rL.e, rR.e) + 1;
    const int64_t mL = neg_if((int64_t)shr(ML, em - emL), uL.s), mR = neg_if((int64_t)shr(MR, em - emR), uR.s);
    const int64_t c0 = mL + mR, DM = mR - mL;
    const int64_t nL = neg_if((int64_t)shr(NL, en - enL), vL.s), nR = neg_if((int64_t)shr(NR, en - enR), vR.s);
    const int64_t nS = nL + nR, DN = nR - nL;
    const uint64_t rLa = shr(rL.m, er - rL.e), rRa = shr(rR.m, er - rR.e);
    const uint64_t rS = rLa + rRa;                       // [2^61, 2^63)
    const int64_t DR = (int64_t)(rRa - rLa);
    const Num pL = unpack(pLd), pR = unpack(pRd);
    const int ep = imax(pL.e, pR.e) + 2;
    const int64_t pLa = neg_if((int64_t)shr(pL.m, ep - pL.e), pL.s), pRa = neg_if((int64_t)shr(pR.m, ep - pR.e), pR.s);
    const int64_t PS = pLa + pRa;
    int64_t DP = pRa - pLa;                              // |.| < 2^62, then in [2^61, 2^62)
    const int kd = room(mag(DP)), epd = ep - kd;
    DP <<= kd;
    // ---- first loop: u, c, a, b at the Gauss points (twice the states: r' = rS -+ t dr, m' = c0 -+ t dm) ----
    const int drs = (int)(DR >> 63), dms = (int)(DM >> 63);
    const uint64_t DRa = mag(DR) * 2;                    // |DR|, one exponent down
    const int64_t TR = neg_if((int64_t)mulhi(kT64, DRa >> 1), drs), TM = neg_if((int64_t)mulhi(kT64, mag(DM)), dms);
    Point q[3];
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int j = 0; j < 3; ++j) {
        const uint64_t r = j == 0 ? rS - (uint64_t)TR : (j == 1 ? rS : rS + (uint64_t)TR);
        const int64_t m = j == 0 ? c0 - TM : (j == 1 ? c0 : c0 + TM);
        const int k = clz(r) - 2;                        // -1 .. 3 (r in [2^58.8, 2^63))
        const uint64_t X = k < 0 ? r >> 1 : r << k;      // [2^61, 2^62)
        const uint64_t Y = rcp61(X) * 2;                 // 1/r' = Y 2^(k - er - 124), Y in (2^62, 2^63]
        q[j].k = k;
        q[j].sg = (int)(m >> 63);
        q[j].u = mulu((uint64_t)neg_if(m, q[j].sg) * 2, Y);   // < 2^62
        const int eu = em - er - 61 + k;
        const int ku = clz(q[j].u | 1) - 1;
        const uint64_t un = q[j].u << ku;                // [2^62, 2^63) unless u = 0
        // c^2 = u^2 + 8 beta / r'
        const uint64_t f = mulu(fb.b8, Y);               // [2^60, 2^62]
        const int ef = fb.eb8 + k - er - 60;
        const uint64_t u2 = mulu(un, un);                // [2^60, 2^62)
        const int eu2 = 2 * (eu - ku) + 64;
        int e2 = imax(ef, eu2) + 2;
        uint64_t M = shr(f, e2 - ef) + shr(u2, e2 - eu2);   // [2^58, 2^61]
        int sh = clz(M) - 2;
        sh -= (e2 - sh) & 1;
        M <<= sh;                                        // [2^60, 2^62), even exponent
        e2 -= sh;
        const uint64_t R = rsqrt61(M) * 2;               // 1/c = R 2^(-93 - e2/2)
        const uint64_t C = mulu(M * 2, R);               // [2^60, 2^61]
        q[j].ec = e2 / 2 - 30;
        q[j].c = C * 4;
        // a = |u|/c <= 1 in Q61
        const int sa = imax(0, e2 / 2 - 32 - (eu - ku));
        uint64_t a = shr(mulu(un, R), sa);
        const uint64_t one = (uint64_t)1 << 61;
        q[j].a = a < one ? a : one;
        // dm - u dr in units 2^(em + 3), below 2^62
        const uint64_t P = mulu(un, DRa);                // exponent em + 2 + k - ku
        const int64_t udr = (int64_t)shr(P * 2, ku - k + 2);
        q[j].b = (DM >> 3) - neg_if(udr, q[j].sg ^ drs);
    }
    const int kb = room(mag(q[0].b) | mag(q[1].b) | mag(q[2].b));
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int j = 0; j < 3; ++j) q[j].b = smul(q[j].c, q[j].b << kb);   // exponent ec + em + 65 - kb
    const int ebm = em + 65 - kb;
    // ---- second loop: G, Z and their sums, on exponents common to the points ----
    const int ecx = imax(q[0].ec, imax(q[1].ec, q[2].ec));
    const int kx = imax(q[0].k, imax(q[1].k, q[2].k));
    uint64_t U[3];
    for (int j = 0; j < 3; ++j) U[j] = shr(q[j].u, kx - q[j].k);
    const int nu = room(U[0] | U[1] | U[2]), eu = em - er - 61 + kx - nu;
    for (int j = 0; j < 3; ++j) U[j] <<= nu;
    const int eg = imax(epd + 2, ecx + ebm + 1);
    const int64_t DP4 = sar(DP, eg - 2 - epd);           // 4 dp
    int64_t G[3], Z[3], H[3];
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int j = 0; j < 3; ++j) {
        const int64_t sdp = neg_if(DP4, q[j].sg);        // sg 4 dp
        const int64_t b2 = sar(q[j].b, eg - 1 - (q[j].ec + ebm));       // 2 b
        const uint64_t a4 = q[j].a * 4, y4 = ((uint64_t)1 << 63) - a4;  // a, 1 - a in Q63
        const uint64_t s2 = mulu(y4, y4) * 2;            // s in Q63
        const uint64_t h = mulu(mulu(a4, y4) * 8, 3 * ((uint64_t)1 << 61) - q[j].a) * 2;   // h in Q63
        const int64_t sb = smul(s2, b2 >> 1), g = sb - smul(y4, sdp >> 1);   // G - sg dp
        G[j] = sb + smul(a4, sdp >> 1);
        const int64_t z = smul(s2, sdp) + smul(h, b2);   // sg (2 s dp + sg h b)
        // sg is applied last, so that states mirrored in u give exactly opposite Z
        Z[j] = neg_if(sar(smul(q[j].c, z), ecx - q[j].ec), q[j].sg);    // exponent ecx + eg + 62
        H[j] = neg_if(smul(U[j] * 2, g), q[j].sg);       // u (G - sg dp), exponent eu + eg + 63
    }
    const uint64_t SU = mulu(kW1, U[0] + U[2]) + mulu(kW2, U[1]);
    const int64_t SG = smul(kW1, G[0] + G[2]) + smul(kW2, G[1]);
    const int64_t SZ = smul(kW1, Z[0] + Z[2]) + smul(kW2, Z[1]);
    const int64_t SH = smul(kW1, H[0] + H[2]) + smul(kW2, H[1]);
    const int eh = eu + eg + 129 + fb.eib4;              // its sum over beta
    int64_t TZ = smul(kT, smul(fb.ib4, smul(kW1, Z[2] - Z[0])));   // t/2 times the outer points' difference
    int64_t ZV = smul(fb.ib4, SZ);
    int ez = ecx + eg + 126 + fb.eib4;
    const int nz = room(mag(ZV) | mag(TZ));
    ZV <<= nz;
    TZ <<= nz;
    ez -= nz;
    const int ev = imax(eu, ez) + 1;
    const int64_t S1 = (int64_t)shr(SU, ev - eu) + sar(TZ, ev - ez), Zv = sar(ZV, ev - ez);   // |.| < 2^62
    // ---- 2F = F(Q_L) + F(Q_R) - D, each sum on the exponent of its largest term ----
    {
        const int ed = er + ev + 64, e = imax(em, ed) + 1;
        F[0] = to_double(sar(c0, e - em) - sar(ssmul(DR, S1) + (smul(rS, Zv) >> 1), e - ed), e);
    }
    {
        const int eL = emL + uL.e + 64, eR = emR + uR.e + 64, ed = em + ev + 64;
        const int e = imax(imax(eL, eR), imax(ep, imax(ed, eg))) + 3;
        const int64_t t = sar(PS, e - ep) - sar(ssmul(DM, S1) + (ssmul(c0, Zv) >> 1), e - ed) - sar(SG, e - eg);
        F[1] = to_double(t + (int64_t)shr(mulu(ML, uL.m), e - eL) + (int64_t)shr(mulu(MR, uR.m), e - eR), e);
    }
    {
        const int eL = emL + vL.e + 64, eR = emR + vR.e + 64, ed = en + ev + 64;
        const int e = imax(imax(eL, eR), ed) + 2;
        const int64_t l = neg_if((int64_t)shr(mulu(ML, vL.m), e - eL), uL.s ^ vL.s);
        const int64_t r = neg_if((int64_t)shr(mulu(MR, vR.m), e - eR), uR.s ^ vR.s);
        F[2] = to_double(l + r - sar(ssmul(DN, S1) + (ssmul(nS, Zv) >> 1), e - ed), e);
    }
    {
        const int64_t h = smul(fb.ib4, SH);
        const int e = imax(imax(uL.e, uR.e), imax(ev, eh)) + 3;
        const int64_t l = neg_if((int64_t)shr(uL.m, e - uL.e), uL.s), r = neg_if((int64_t)shr(uR.m, e - uR.e), uR.s);
        F[3] = to_double(l + r - sar(Zv, e - ev) + sar(h, e - eh), e);
    }
}

// Whether osher_flux_fixed takes these states: finite, densities positive and normal.
ACFX bool fixed_flux_ok(double rL, double uL, double vL, double pL, double rR, double uR, double vR, double pR) {
    using namespace fx;
    const uint32_t inf = 0x7ff00000u;
    const uint32_t hL = (uint32_t)(bits_of(rL) >> 32), hR = (uint32_t)(bits_of(rR) >> 32);
    const uint32_t a = (uint32_t)(bits_of(uL) >> 32) & inf, b = (uint32_t)(bits_of(uR) >> 32) & inf;
    const uint32_t c = (uint32_t)(bits_of(vL) >> 32) & inf, d = (uint32_t)(bits_of(vR) >> 32) & inf;
    const uint32_t e = (uint32_t)(bits_of(pL) >> 32) & inf, f = (uint32_t)(bits_of(pR) >> 32) & inf;
    return hL - 0x00100000u < 0x7fe00000u && hR - 0x00100000u < 0x7fe00000u && a != inf && b != inf && c != inf &&
           d != inf && e != inf && f != inf;
}

}  // namespace acgb
