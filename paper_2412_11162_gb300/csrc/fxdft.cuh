// Even-sequence DFTs in 64-bit block fixed point (sm_103a): the transforms of
// the FP64 sampling kernels on the integer pipe.
//
// The GB300 retires 2 FP64 operations per SM per clock, an addition costing as
// much as an FMA, so an FFT (mostly additions) in FP64 is the worst use of that
// pipe.  Here a sequence is held as 64-bit integers with one exponent, x_j = X_j
// 2^ex.  Additions are exact (two instructions); a product with a Q62 twiddle takes
// three 32 x 32 -> 64 multiply-adds.  The values start with |re| + |im| just below
// 2^59 and are shifted right only as far as the sequence can grow: after a stage
// that has combined Ns values no sum exceeds min(Ns max|y|, sum |y|), y the
// transform's input, so the shifts follow from the sequence's maximum and sum of
// magnitudes alone (T bits in all: 0 for a sequence with one large value, log2 K
// for a flat one) and nothing overflows.  A transform's error is then a few units
// of 2^-59 min(K max|x|, sum |x|), below the ~2^-52 (sum |x|^2)^(1/2) of the FP64
// transform for every such sequence.
//
// Measured (GB300), FP64 transforms -> these: modal kernels in FP64 at N = 384, M =
// 192 13.7 -> 9.2 ms, N = 128, M = 64 (8 modes) 1.77 -> 1.37 ms, field of 512 points
// at N = 512, M = 256 16.3 -> 11.3 ms; what is left there is the FP64 sampling (80 %
// of the FP64 pipe).
//
// Conversions double <-> fixed use integer operations only (the conversion
// instructions are issued to the FP64 pipe).
#pragma once

#include "device_common.cuh"

namespace pmlbie {
namespace {

using i64 = long long;
using u64 = unsigned long long;

// exponent of a sequence holding a NaN or an infinity: its values read back as NaN
constexpr int kFxNonfinite = 1 << 24;
constexpr int kFxBits = 59;      // |re| + |im| of a quantised value is below 2^kFxBits

// exponent of a quantised sequence and the bits by which its sum of |re| + |im| may
// exceed 2^kFxBits (the shift its transform needs at most)
struct FxScale {
    int ex, T;
};

// complex values in shared memory: 16 bytes, double2 before and (re, im) after
// the quantisation
__device__ __forceinline__ longlong2 fx2(i64 x, i64 y) { return make_longlong2(x, y); }
__device__ __forceinline__ longlong2 fxadd(longlong2 a, longlong2 b) { return fx2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ longlong2 fxsub(longlong2 a, longlong2 b) { return fx2(a.x - b.x, a.y - b.y); }

// x = h 2^32 + l with l signed (balanced digits), so that every partial product
// below is signed x signed
__device__ __forceinline__ void fx_split(i64 x, int& h, int& l) {
    l = (int)(u64)x;
    h = (int)(x >> 32) - (l >> 31);
}
__device__ __forceinline__ i64 mul_wide(int a, int b) { return (i64)a * (i64)b; }

// x w, w = (wh, wl) in Q62 balanced digits, |x| < 2^61: the low x low partial
// product (below half a unit) is dropped, the rest rounded
__device__ __forceinline__ i64 fx_mul(i64 x, int wh, int wl) {
    int h, l;
    fx_split(x, h, l);
    const i64 c = mul_wide(l, wh) + mul_wide(h, wl) + (1ll << 29);
    return (mul_wide(h, wh) << 2) + (c >> 30);
}
// complex product with the twiddle w = (re.h, re.l, im.h, im.l), times 2^-d (d = 0, 1, 2)
__device__ __forceinline__ longlong2 fx_cmul(longlong2 v, int4 w, int d = 0) {
    int xh, xl, yh, yl;
    fx_split(v.x, xh, xl);
    fx_split(v.y, yh, yl);
    const i64 half = 1ll << (29 + d);
    const i64 cr = mul_wide(xl, w.x) + mul_wide(xh, w.y) - mul_wide(yl, w.z) - mul_wide(yh, w.w) + half;
    const i64 ci = mul_wide(xl, w.z) + mul_wide(xh, w.w) + mul_wide(yl, w.x) + mul_wide(yh, w.y) + half;
    const i64 hr = mul_wide(xh, w.x) - mul_wide(yh, w.z);
    const i64 hi = mul_wide(xh, w.z) + mul_wide(yh, w.x);
    return fx2((hr << (2 - d)) + (cr >> (30 + d)), (hi << (2 - d)) + (ci >> (30 + d)));
}

// round(v 2^-ex) for finite v with |v| 2^-ex < 2^62
__device__ __forceinline__ i64 fx_of_double(double v, int ex) {
    const int hw = __double2hiint(v), e = (hw >> 20) & 0x7ff;
    const u64 m = ((u64)((unsigned)(hw & 0xfffff) | 0x100000u) << 32) | (unsigned)__double2loint(v);
    const int n = 1084 + ex - e;             // right shift of m 2^10, less one (the rounding bit)
    if (e == 0 || n > 63) return 0;
    const i64 r = (i64)((((m << 10) >> n) + 1) >> 1);
    return hw < 0 ? -r : r;
}

// v 2^ex as a double, correctly rounded (ties away from zero); overflow gives an
// infinity, underflow zero, a nonfinite sequence NaN
__device__ __forceinline__ double fx_to_double(i64 v, int ex) {
    if (ex == kFxNonfinite) return __hiloint2double(0x7ff80000, 0);
    if (v == 0) return 0.0;
    const u64 a = v < 0 ? 0ull - (u64)v : (u64)v;
    const int z = __clzll((i64)a);
    const u64 r = (((a << z) >> 10) + 1) >> 1;          // 53 significant bits (or 2^53)
    const int E = 1085 - z + ex;                          // biased exponent less one
    const u64 s = (u64)v & (1ull << 63);
    if (E < 0) return __longlong_as_double((i64)s);
    if (E >= 2046) return __longlong_as_double((i64)(s | (2047ull << 52)));
    return __longlong_as_double((i64)(s | (((u64)E << 52) + r)));
}
__device__ __forceinline__ double2 fx_to_double2(longlong2 v, int ex) {
    return make_double2(fx_to_double(v.x, ex), fx_to_double(v.y, ex));
}

__device__ __forceinline__ float warp_sum(float v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ i64 warp_sum(i64 v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// smallest p with v <= 2^p (v a positive normal float)
__device__ __forceinline__ int ceil_log2(float v) {
    const unsigned b = __float_as_uint(v);
    return (int)(b >> 23) - 127 + ((b & 0x7fffffu) ? 1 : 0);
}

// Quantise n complex doubles in place (one warp).  The magnitudes enter the sum by
// their high words, reread as floats relative to the largest exponent (20 mantissa
// bits, truncated: the sum is low by at most 2^-20 of itself, inside the headroom
// above the bounds).
__device__ __noinline__ FxScale fx_quantise(void* seq, int n, int lane) {
    const double2* x = reinterpret_cast<const double2*>(seq);
    unsigned top = 0;
    for (int i = lane; i < n; i += 32) {
        const double2 v = x[i];
        top = max(top, max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu));
    }
    top = __reduce_max_sync(0xffffffffu, top) >> 20;
    longlong2* o = reinterpret_cast<longlong2*>(seq);
    if (top == 0x7ff) return FxScale{kFxNonfinite, 0};
    if (top == 0) {                       // zeros (and denormals)
        for (int i = lane; i < n; i += 32) o[i] = fx2(0, 0);
        __syncwarp();
        return FxScale{0, 0};
    }
    // |re|, |im| < 2^(top - 1022)
    const int ex = (int)top - 1021 - kFxBits, base = ((int)top - 120) << 20;
    float s = 0.f;
    for (int i = lane; i < n; i += 32) {
        const double2 v = x[i];
        const int a = (int)((unsigned)__double2hiint(v.x) & 0x7fffffffu) - base;
        const int b = (int)((unsigned)__double2hiint(v.y) & 0x7fffffffu) - base;
        s += __uint_as_float((unsigned)max(a, 0) << 3) + __uint_as_float((unsigned)max(b, 0) << 3);
        o[i] = fx2(fx_of_double(v.x, ex), fx_of_double(v.y, ex));
    }
    s = warp_sum(s);
    __syncwarp();
    // the float of exponent field 120 stands for 2^(top - 1023): sum = s 2^(top - 1016)
    return FxScale{ex, max(0, ceil_log2(s) + (int)top - 1016 - ex - kFxBits)};
}

// v 2^sh, rounded when sh < 0
__device__ __forceinline__ i64 fx_shift(i64 v, int sh) {
    return sh >= 0 ? v << sh : ((v >> (-sh - 1)) + 1) >> 1;
}
__device__ __forceinline__ longlong2 fx_shift(longlong2 v, int sh) { return fx2(fx_shift(v.x, sh), fx_shift(v.y, sh)); }

// Requantise n fixed-point values x of exponent ex into y (|values| < 2^62): the
// magnitudes by their high words (rounded up) as floats built by an addition;
// im's sign changed where sy < 0.  y[n .. ny) is zeroed.
__device__ __noinline__ FxScale fx_requantise(const longlong2* x, longlong2* y, int n, int ny, int ex, bool conj,
                                              int lane) {
    float s = 0.f, m = 0.f;
    for (int i = lane; i < n; i += 32) {
        const longlong2 v = x[i];
        const unsigned a = (unsigned)abs((int)(v.x >> 32)) >> 8, b = (unsigned)abs((int)(v.y >> 32)) >> 8;
        const float t = (__uint_as_float(0x4b000000u | a) - 8388607.0f) + (__uint_as_float(0x4b000000u | b) - 8388607.0f);
        s += t;                            // |re| + |im| < t 2^40
        m = fmaxf(m, t);
    }
    s = warp_sum(s);
    m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));
    const int sh = kFxBits - 40 - ceil_log2(m);
    for (int i = lane; i < ny; i += 32) {
        longlong2 v = i < n ? fx_shift(x[i], sh) : fx2(0, 0);
        if (conj) v.y = -v.y;
        y[i] = v;
    }
    __syncwarp();
    return FxScale{ex == kFxNonfinite ? ex : ex - sh, max(0, ceil_log2(s) - ceil_log2(m))};
}

// One in-place Stockham stage of a K-point transform (one warp): every butterfly
// of the stage is read into registers before any is written back.  NB butterflies
// of radix R per lane at most.  lgNs = log2(Ns) while Ns is a power of two (radix-4
// and radix-2 stages come first), else -1.  tw[e tws] = e^{-2 pi i e / K}.  The
// inputs are scaled by 2^-d.
template <int R, int NB>
__device__ __forceinline__ void fx_stage(longlong2* x, int K, int Ns, int lgNs, int step, int d, const int4* tw,
                                         int tws, int lane) {
    const int MR = K / R;
    longlong2 v[NB][R];
    int dst[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        const int j = lane + 32 * b;
        dst[b] = -1;
        if (j >= MR) continue;
        const int jq = lgNs >= 0 ? (j >> lgNs) : j / Ns;
        const int k = j - jq * Ns;
        dst[b] = jq * Ns * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) v[b][r] = x[j + r * MR];
        if (d) v[b][0] = fx_shift(v[b][0], -d);
        if (Ns > 1) {
            const int t = k * step * tws;
#pragma unroll
            for (int r = 1; r < R; ++r) v[b][r] = fx_cmul(v[b][r], tw[r * t], d);
        } else if (d) {
#pragma unroll
            for (int r = 1; r < R; ++r) v[b][r] = fx_shift(v[b][r], -d);
        }
        if (R == 2) {
            const longlong2 p = v[b][0], q = v[b][1];
            v[b][0] = fxadd(p, q);
            v[b][1] = fxsub(p, q);
        } else if (R == 4) {
            const longlong2 t0 = fxadd(v[b][0], v[b][2]), t1 = fxsub(v[b][0], v[b][2]);
            const longlong2 t2 = fxadd(v[b][1], v[b][3]), t3 = fxsub(v[b][1], v[b][3]);
            v[b][0] = fxadd(t0, t2);
            v[b][2] = fxsub(t0, t2);
            v[b][1] = fx2(t1.x + t3.y, t1.y - t3.x);   // t1 - i t3
            v[b][3] = fx2(t1.x - t3.y, t1.y + t3.x);   // t1 + i t3
        } else {
            // w = e^{-2 pi i/3}: a + w b + w^2 c = m - i s3 (b - c), m = a - (b + c)/2
            constexpr i64 s3 = 3993837246235628775ll;  // sin(2 pi / 3) in Q62
            constexpr int s3l = (int)(u64)(s3 & 0xffffffffll), s3h = (int)((s3 - s3l) >> 32);
            const longlong2 p = v[b][0], bc = fxadd(v[b][1], v[b][2]), bm = fxsub(v[b][1], v[b][2]);
            const longlong2 m = fx2(p.x - ((bc.x + 1) >> 1), p.y - ((bc.y + 1) >> 1));
            const longlong2 q = fx2(fx_mul(bm.x, s3h, s3l), fx_mul(bm.y, s3h, s3l));
            v[b][0] = fxadd(p, bc);
            v[b][1] = fx2(m.x + q.y, m.y - q.x);
            v[b][2] = fx2(m.x - q.y, m.y + q.x);
        }
    }
    __syncwarp();
#pragma unroll
    for (int b = 0; b < NB; ++b)
        if (dst[b] >= 0) {
#pragma unroll
            for (int r = 0; r < R; ++r) x[dst[b] + r * Ns] = v[b][r];
        }
    __syncwarp();
}

// K-point FFT in place, K = 2^a 3^b <= 128 NB, of values below 2^60 whose sum is
// below 2^(60 + T); returns the bits the result was scaled down by
template <int NB>
__device__ __forceinline__ int fx_fft(longlong2* x, int K, int T, const int4* tw, int tws, int lane) {
    int rem = K, Ns = 1, lgNs = 0, cum = 0;
    while (rem > 1) {
        const int R = (rem & 3) == 0 ? 4 : ((rem & 1) == 0 ? 2 : 3);
        const int step = K / (Ns * R);
        const int d = min(32 - __clz(Ns * R - 1), T) - cum;
        if (R == 4)
            fx_stage<4, NB>(x, K, Ns, lgNs, step, d, tw, tws, lane);
        else if (R == 2)
            fx_stage<2, 2 * NB>(x, K, Ns, lgNs, step, d, tw, tws, lane);
        else
            fx_stage<3, (4 * NB + 2) / 3>(x, K, Ns, lgNs, step, d, tw, tws, lane);
        cum += d;
        Ns *= R;
        lgNs = (lgNs >= 0 && R != 3) ? lgNs + (R == 4 ? 2 : 1) : -1;
        rem /= R;
    }
    return cum;
}

// DFT of an even sequence x_0..x_{L-1} (x_k = x_{L-k}, L = 2K, K even, K <= 128
// NB) from its K+1 distinct fixed-point values, in place: x[0..K] -> X_0..X_K, one
// warp.  Real and imaginary parts are two real-even (DCT-I) transforms, each
// reduced to K values y_j = (x_j + x_{K-j})/2 - sin(pi j/K) (x_j - x_{K-j}); the two
// are packed into one complex K-point FFT z, whose even outputs are X_{2k} = z_k +
// z_{K-k}; the odd ones follow by the running sum X_{2k+1} = X_{2k-1} - I_k,
// I_k = -i (z_k - z_{K-k}) (exact in fixed point), started at X_1 = 2 sum_{j<K} x_j
// cos(pi j/K) - x_0 - x_K (its own sum, in two words; here the sum over pairs (j,
// K-j) of 2 cos(pi j/K) (x_j - x_{K-j}), to which j = 0 gives x_0 - x_K).
// sc: the quantised sequence's scale; sum |y| <= 2 sum |x|.  Returns the exponent of
// the result, |X| <= 2^60 (1 + 1/K).  tw[e tws] = e^{-2 pi i e / L}.
template <int NB>
__device__ __forceinline__ int fx_even_dft(longlong2* x, FxScale sc, int K, const int4* tw, int tws, int lane) {
    const int H = K / 2;
    longlong2 hi = fx2(0, 0);
    int2 lo = make_int2(0, 0);
    auto add = [](i64 v, i64& h, int& l) {
        h += v >> 16;
        l += (int)v & 0xffff;
    };
    for (int j = lane; j < H; j += 32) {
        const int jm = K - j;
        const longlong2 a = x[j], b = x[jm];
        const longlong2 s = fxadd(a, b), d = fxsub(a, b);
        const longlong2 h = fx2((s.x + 1) >> 1, (s.y + 1) >> 1);
        if (j == 0) {
            x[0] = h;
            add(d.x, hi.x, lo.x);            // 2 x_0 - x_0 - x_K
            add(d.y, hi.y, lo.y);
            continue;
        }
        const int4 t = tw[j * tws];      // (cos(pi j/K), -sin(pi j/K))
        const longlong2 q = fx2(fx_mul(d.x, t.z, t.w), fx_mul(d.y, t.z, t.w));
        x[j] = fxadd(h, q);
        x[jm] = fxsub(h, q);
        add(2 * fx_mul(d.x, t.x, t.y), hi.x, lo.x);
        add(2 * fx_mul(d.y, t.x, t.y), hi.y, lo.y);
    }
    __syncwarp();
    const int sh = fx_fft<NB>(x, K, sc.T, tw, 2 * tws, lane);      // <= 11
    const longlong2 X1 = fx2((warp_sum(hi.x) << (16 - sh)) + (__reduce_add_sync(0xffffffffu, lo.x) >> sh),
                             (warp_sum(hi.y) << (16 - sh)) + (__reduce_add_sync(0xffffffffu, lo.y) >> sh));
    // lane: k in [lane P, lane P + P), P = ceil(H / 32) <= 2 NB
    const int P = (H + 31) >> 5, k0 = lane * P;
    longlong2 ev[2 * NB], I[2 * NB], run = fx2(0, 0);
#pragma unroll
    for (int q = 0; q < 2 * NB; ++q) {
        const int k = k0 + q;
        if (q < P && k < H) {
            const longlong2 z = x[k], zc = x[k == 0 ? 0 : K - k];
            ev[q] = fxadd(z, zc);
            I[q] = fx2(z.y - zc.y, zc.x - z.x);
            run = fxadd(run, I[q]);
        }
    }
    const longlong2 zH = x[H];
    longlong2 incl = run;
    for (int o = 1; o < 32; o <<= 1) {
        const longlong2 v = fx2(__shfl_up_sync(0xffffffffu, incl.x, o), __shfl_up_sync(0xffffffffu, incl.y, o));
        if (lane >= o) incl = fxadd(incl, v);
    }
    longlong2 acc = fxsub(X1, fxsub(incl, run));
#pragma unroll
    for (int q = 0; q < 2 * NB; ++q) {
        const int k = k0 + q;
        if (q < P && k < H) {
            acc = fxsub(acc, I[q]);
            x[2 * k] = ev[q];
            x[2 * k + 1] = acc;
        }
    }
    if (lane == 0) x[K] = fx2(2 * zH.x, 2 * zH.y);
    __syncwarp();
    return sc.ex == kFxNonfinite ? sc.ex : sc.ex + sh;
}
// The same out of line: the close-pair kernel holds two sizes of it, and instruction
// misses cost it more than the calls (close pairs at N = 1024, M = 512 49.2 -> 48.0 ms,
// 8 low modes at N = 128 1.07 -> 1.03 ms); the far and field kernels, whose
// transforms follow a long sampling loop, are faster with it in line (field map 6.74
// against 6.98 ms).
template <int NB>
__device__ __noinline__ int fx_even_dft_call(longlong2* x, FxScale sc, int K, const int4* tw, int tws, int lane) {
    return fx_even_dft<NB>(x, sc, K, tw, tws, lane);
}

}  // namespace
}  // namespace pmlbie
