// sin, cos, exp and 1/sqrt of the sampling loops with the work on the integer pipe
// (sm_103a): about 75 integer instructions for a sine / cosine pair and 60 for an
// exponential, where the FP64 versions (fp64_elem.cuh) occupy the FP64 pipe, 16
// cycles per warp instruction, for 24 and 18.
//
//   phase   q = w R: the fraction of q / 2 pi in 2^-64 turns straight from the 128-bit
//           product of R's significand with w / 2 pi (64 bits), so that q is not
//           rounded first;
//   sin, cos nearest of 1024 table angles (first quadrant stored, Q62), the rest
//           |theta| <= pi/1024 by the Taylor series to theta^5 / theta^6 (remainders
//           below 2^-70 / 2^-78), the high-order terms in 32 bits, the angles joined by
//           one complex product: absolute error below 2^-57.9;
//   exp     x log2(e) split into integer and fraction, 256 table values 2^(j/256) and
//           the series of e^rho to rho^5, rho < ln2/256 (remainder 2^-60): relative
//           error below 2^-55.7, as a significand times a power of two;
//   1/sqrt  single-precision estimate and one third-order step in FP64 (five
//           operations, error about 1 ulp).
#pragma once

#include "fxdft.cuh"

namespace pmlbie {
namespace {

// tables: cs[j] = cos, sin of 2 pi j / 1024 (digits of Q62), e2[j] = 2^(j/256) (digits
// of Q61); 6 KB read through L1 (a copy in shared memory costs the close-pair kernels
// one resident CTA per SM)
struct FxTab {
    const int4* cs;
    const int2* e2;
};
__device__ __forceinline__ FxTab fx_tables(const DeviceTables& T) { return FxTab{T.trig_fx, T.exp_fx}; }

// fraction of R w / 2 pi in units of 2^-64 turns, R >= 0
__device__ __forceinline__ u64 fx_turns(double R, FxPhase w) {
    const int hw = __double2hiint(R), e = (hw >> 20) & 0x7ff;
    const u64 m = (((u64)((unsigned)(hw & 0xfffff) | 0x100000u) << 32) | (unsigned)__double2loint(R)) << 11;
    const u64 hi = __umul64hi(m, w.W), lo = m * w.W;
    const int E = e - 1022 + w.e;            // turns = (hi, lo) 2^(E - 128)
    if (E <= 0) return (e == 0 || E < -63) ? 0ull : hi >> -E;
    return (hi << (E & 63)) | ((lo >> 1) >> (63 - (E & 63)));
}

// cos and sin (Q62) of 2 pi u / 2^64
__device__ __forceinline__ longlong2 fx_cis(u64 u, const FxTab& T) {
    const u64 v = u + (1ull << 53);
    const int j = (int)(v >> 54);                        // 0 .. 1023
    const i64 r = (i64)(u - ((u64)j << 54));             // |r| <= 2^53
    const int4 A = __ldg(T.cs + (j & 255));
    // theta = 2 pi r 2^-64 = t 2^-70
    constexpr i64 kP = 3622009729038561421ll;            // pi / 4 in Q62
    constexpr int kPl = (int)(u64)(kP & 0xffffffffll), kPh = (int)((kP - kPl) >> 32);
    const i64 t = fx_mul(r << 9, kPh, kPl);
    int th, tl;
    fx_split(t, th, tl);
    const i64 z = mul_wide(th, th) + (mul_wide(th, tl) >> 31);      // theta^2, 2^-76
    const unsigned zh = (unsigned)(z >> 28);                        // 2^-48
    // sin = theta - theta w, w = z (1/6 - z/120)
    const unsigned b = 2863311531u - (__umulhi(zh, 572662306u) >> 18);      // 2^-34
    const int wH = (int)(((u64)zh * b) >> 32);                              // 2^-50
    const i64 s = t - ((mul_wide(th, wH) + (mul_wide(tl, wH) >> 32)) >> 18);    // 2^-70
    // 1 - cos = z/2 - z eps, eps = z/24 - z^2/720
    const unsigned eps = __umulhi(zh, 2863311531u) - __umulhi(__umulhi(zh, zh), 1456u);   // 2^-52
    const i64 c = ((z >> 1) - (i64)(((u64)zh * eps) >> 24)) >> 6;           // 2^-70
    const longlong2 d = fx_cmul(fx2(-c, s), A);                             // 2^-70
    const i64 cx = ((i64)A.x << 32) + A.y + ((d.x + 128) >> 8), sx = ((i64)A.z << 32) + A.w + ((d.y + 128) >> 8);
    const int q = j >> 8;
    const i64 a = (q & 1) ? sx : cx, o = (q & 1) ? cx : sx;
    // quadrants: (c, s), (-s, c), (-c, -s), (s, -c)
    return fx2(((q + 1) & 2) ? -a : a, (q & 2) ? -o : o);
}

// e^x = m 2^(ex - 61), m in [2^61, 2^62); x clamped to |x| < 2^11
__device__ __forceinline__ i64 fx_exp(double x, const FxTab& T, int& ex) {
    const int hw = __double2hiint(x), e = min((hw >> 20) & 0x7ff, 1033);
    const u64 m = (((u64)((unsigned)(hw & 0xfffff) | 0x100000u) << 32) | (unsigned)__double2loint(x)) << 11;
    constexpr u64 kL = 13306513097844322492ull;          // log2(e) 2^63
    const u64 hi = __umul64hi(m, kL), lo = m * kL;
    const int E = e - 1021;                              // |x| log2 e = (hi, lo) 2^(E - 128)
    int ip = 0;
    u64 f;
    if (E <= 0) {
        f = (e == 0 || E < -63) ? 0ull : hi >> -E;
    } else {
        ip = (int)(hi >> (64 - E));
        f = (hi << E) | (lo >> (64 - E));
    }
    if (hw < 0) {
        ip = -ip - (f != 0);
        f = 0ull - f;
    }
    const int2 t2 = __ldg(T.e2 + (int)(f >> 56));
    // rho = (f mod 2^56) 2^-64 ln 2 = t 2^-69
    constexpr i64 kN = 3196577161300663915ll;            // ln 2 in Q62
    constexpr int kNl = (int)(u64)(kN & 0xffffffffll), kNh = (int)((kN - kNl) >> 32);
    const i64 t = fx_mul((i64)((f & ((1ull << 56) - 1)) << 5), kNh, kNl);
    const unsigned r = (unsigned)(t >> 29);                                  // 2^-40
    const unsigned a = 2863311531u + __umulhi(r, 2236962u);                  // 1/24 + rho/120, 2^-36
    const unsigned b = 2863311531u + (__umulhi(r, a) >> 10);                 // 1/6 + rho a, 2^-34
    const unsigned h = (unsigned)(((u64)r * b) >> 32);                       // rho b, 2^-42
    const i64 g = t + (i64)(((u64)r * h) >> 12);                             // rho (1/2 + rho b), 2^-70
    int th, tl, gh, gl;
    fx_split(t, th, tl);
    fx_split(g, gh, gl);
    const i64 p = t + ((mul_wide(th, gh) + ((mul_wide(th, gl) + mul_wide(tl, gh)) >> 32)) >> 6);   // 2^-69
    ex = ip;
    return ((i64)t2.x << 32) + t2.y + (fx_mul(p, t2.x, t2.y) >> 7);
}

// 1/sqrt(x), x > 0 normal; NaN for zero (a receiver on a node), denormals, x < 0, infinity
__device__ __forceinline__ double fx_rsqrt(double x) {
    const int hw = __double2hiint(x), e = (hw >> 20) - 1023;
    if ((unsigned)hw - 0x00100000u >= 0x7fe00000u) return __hiloint2double(0x7ff80000, 0);
    const unsigned mant = ((unsigned)hw << 12) | ((unsigned)__double2loint(x) >> 20);
    float y;      // estimate for the significand in [1, 4)
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(((127u + (e & 1)) << 23) | (mant >> 9))));
    const unsigned yb = __float_as_uint(y);
    const double y0 = __hiloint2double((int)((yb >> 3) + ((896 - (e >> 1)) << 20)), (int)(yb << 29));
    const double h = fma(-(x * y0), y0, 1.0);
    return fma(y0 * h, fma(h, 0.375, 0.5), y0);
}

// Principal square root R of z (z not 0) and 1/R = conj(R)/|z|, from two reciprocal
// square roots; cancellation-free on both half planes
__device__ __forceinline__ void fx_csqrt_rcp(double2 z, double2& R, double2& iR) {
    const double m2 = fma(z.x, z.x, z.y * z.y);
    const double ir = fx_rsqrt(m2);                // 1/|z|
    const double r = m2 * ir;                      // |z|
    const double u = 0.5 * (r + fabs(z.x));
    const double it = fx_rsqrt(u);
    const double t = u * it;                       // sqrt((|z| + |Re z|)/2)
    const double s = 0.5 * z.y * it;               // Im z / (2 t)
    R = z.x >= 0.0 ? c2(t, s) : c2(fabs(s), copysign(t, z.y));
    iR = c2(R.x * ir, -R.y * ir);
}

// e^{i w R} for complex R (Re R >= 0); qy = w Im R
__device__ __forceinline__ double2 fx_expi(double2 R, double qy, FxPhase w, const FxTab& T) {
    const longlong2 c = fx_cis(fx_turns(R.x, w), T);
    int ex;
    const i64 m = fx_exp(-qy, T, ex);
    int h, l;
    fx_split(m, h, l);
    return c2(fx_to_double(fx_mul(c.x, h, l), ex - 61), fx_to_double(fx_mul(c.y, h, l), ex - 61));
}

// sin(q)/q and (sin q - q cos q)/q^3 of a real phase q from its sine and cosine and iq = 1/q;
// below kSmallPhase, where the differences would magnify the rounding of sn and cs
// (absolute, about 2^-54) by 1/q and 3/q^2, their power series (terms left out below 2^-60)
constexpr double kSmallPhase = 0.5;
__device__ __forceinline__ void fx_sinc_h4(double q, double iq, double sn, double cs, double& sinc, double& h4) {
    if (fabs(q) < kSmallPhase) {
        const double x = -q * q;
        constexpr double s[8] = {1.0, 1.0 / 6, 1.0 / 120, 1.0 / 5040, 1.0 / 362880, 1.0 / 39916800, 1.0 / 6227020800.0,
                                 1.0 / 1307674368000.0};
        constexpr double h[8] = {1.0 / 3, 1.0 / 30, 1.0 / 840, 1.0 / 45360, 1.0 / 3991680, 1.0 / 518918400.0,
                                 1.0 / 93405312000.0, 1.0 / 22230464256000.0};
        sinc = s[7], h4 = h[7];
#pragma unroll
        for (int k = 6; k >= 0; --k) sinc = fma(sinc, x, s[k]), h4 = fma(h4, x, h[k]);
    } else {
        sinc = sn * iq;
        h4 = fma(-q, cs, sn) * (iq * iq * iq);
    }
}

}  // namespace
}  // namespace pmlbie
