// From samples to modes in block fixed point (fxdft.cuh): the far pairs' normal
// factors and scatter, and the close pairs' convolution with the modal Laplace
// kernels (Sec. 4.1).
#pragma once

#include <type_traits>

#include "fxdft.cuh"

namespace pmlbie {
namespace {

__device__ __forceinline__ int fx_ex_add(int ex, int d) { return ex == kFxNonfinite ? ex : ex + d; }

// ---------------------------------------------------------------------------
// Far pairs.  Per pair and orientation the double layer's normal factor nd0 +
// nds sin^2(psi/2) times its column weight, and the single layer's column
// weight, as Q62 integers with an exponent (value = q 2^ex): the scatter forms
// its eight entries per mode with integer products, off the FP64 pipe.
// ---------------------------------------------------------------------------
struct FarPairFx {
    int4 nd0, nds, nd0t, ndst;
    int2 ws, wst;                // W_phi factor at the source of (l, m), (m, l)
    int en, ent, ews, ewst;
};
static_assert(sizeof(FarPairFx) == 96, "whole 16-byte units");

// x = q 2^ex with |q| < 2^62, q in balanced digits; ex from the largest exponent
__device__ __forceinline__ int2 fx_q62(double x, int ex) {
    const i64 q = fx_of_double(x, ex);
    int h, l;
    fx_split(q, h, l);
    return make_int2(h, l);
}
__device__ __forceinline__ int fx_exponent(double a, double b, double c, double d) {
    const unsigned m = max(max((unsigned)__double2hiint(a) & 0x7fffffffu, (unsigned)__double2hiint(b) & 0x7fffffffu),
                           max((unsigned)__double2hiint(c) & 0x7fffffffu, (unsigned)__double2hiint(d) & 0x7fffffffu));
    return (int)(m >> 20) - 1084;
}
__device__ __forceinline__ void fx_normal_factor(double2 nd0, double2 nds, double w, int4& q0, int4& qs, int& ex) {
    nd0 = cscale(nd0, w);
    nds = cscale(nds, w);
    ex = fx_exponent(nd0.x, nd0.y, nds.x, nds.y);
    const int2 a = fx_q62(nd0.x, ex), b = fx_q62(nd0.y, ex), c = fx_q62(nds.x, ex), d = fx_q62(nds.y, ex);
    q0 = make_int4(a.x, a.y, b.x, b.y);
    qs = make_int4(c.x, c.y, d.x, d.y);
    ex += 62;
}
// the pair's factors: wu_m, wu_l (K^ of (l, m), (m, l)) and wp_m, wp_l (S^), each
// with the trapezoid factor of the modes
__device__ __forceinline__ void far_pair_fx(const PairGeom& g, double wu_m, double wu_l, double wp_m, double wp_l,
                                            FarPairFx& o) {
    fx_normal_factor(g.nd0, g.nds, wu_m, o.nd0, o.nds, o.en);
    fx_normal_factor(g.nd0t, g.ndst, wu_l, o.nd0t, o.ndst, o.ent);
    o.ews = fx_exponent(wp_m, 0.0, 0.0, 0.0);
    o.ws = fx_q62(wp_m, o.ews);
    o.ewst = fx_exponent(wp_l, 0.0, 0.0, 0.0);
    o.wst = fx_q62(wp_l, o.ewst);
    o.ews += 62;
    o.ewst += 62;
}

// The double layer's normal factor multiplies the geometric factor g(psi) =
// e^{iq}(1 - iq) / |Delta|^3; on the M-point DFT, sin^2(psi/2) = (1 - cos psi)/2
// acts as G_n -> G_n / 2 - (G_{n-1} + G_{n+1}) / 4 (exact; G_{-1} = G_1 for even
// g, and n + 1 <= M/2 stays inside the spectrum).
__device__ __forceinline__ longlong2 sin2_mode(const longlong2* gh, int n) {
    const longlong2 gn = gh[n], gm = gh[n == 0 ? 1 : n - 1], gp = gh[n + 1];
    return fx2((2 * gn.x - gm.x - gp.x + 2) >> 2, (2 * gn.y - gm.y - gp.y + 2) >> 2);
}
// K^ of one orientation (real arithmetic when the factor is real: two physical nodes)
__device__ __forceinline__ double2 nd_mode(int4 q0, int4 qs, longlong2 g, longlong2 s2, bool real, int ex) {
    const longlong2 v = real ? fx2(fx_mul(g.x, q0.x, q0.y) + fx_mul(s2.x, qs.x, qs.y),
                                   fx_mul(g.y, q0.x, q0.y) + fx_mul(s2.y, qs.x, qs.y))
                             : fxadd(fx_cmul(g, q0), fx_cmul(s2, qs));
    return fx_to_double2(v, ex);
}

struct FarArgs {
    DeviceTables T;
    int N, M, mode_lo, mode_hi;
    double w1, w2, h;
    double2* A;     // [mode][col][row], ld 2N
    double2* raw;   // [mode][kernel][l][m]
};

// sources of a far CTA's tile (its pairs over this: targets)
constexpr int kFarTileM = 2;

// Pair of lane `lane` (< nw) of a far CTA: target l = l0 + lane % TL, source m =
// m0 + lane / TL.  Returns its flags (bit 0: (l, m) is far; bit 1: (m, l) is far;
// bit 2: the pair owns its entries, l >= m; bit 3: every pair quantity real) and,
// when a bit of 3 is set, its geometry and factors.
__device__ __forceinline__ int far_pair_setup(const FarArgs& a, int l, int m, PairGeom& g, FarPairFx& o) {
    if (!(l < a.N && m < a.N && l >= m)) return 0;
    int f = 4;
    if (l == m) return f;
    f |= (a.T.cls[(size_t)l * a.N + m] == kFar ? 1 : 0) | (a.T.cls[(size_t)m * a.N + l] == kFar ? 2 : 0);
    if (!(f & 3)) return f;
    g = grid_pair(a.T, l, m);
    if (g.d2.y == 0.0 && g.rr.y == 0.0 && g.nd0.y == 0.0 && g.nds.y == 0.0 && g.nd0t.y == 0.0 && g.ndst.y == 0.0)
        f |= 8;
    const double c4 = 0.5 / a.M;     // (1 / 4 pi)(2 pi / M)
    const double hc = a.h * c4;
    far_pair_fx(g, a.A ? hc * a.T.Wu[m] : c4, a.A ? hc * a.T.Wu[l] : c4, a.A ? hc * a.T.Wphi[m] : c4,
                a.A ? hc * a.T.Wphi[l] : c4, o);
    return f;
}

// Scatter of a CTA's spectra: thread (pair w, mode n) forms the eight entries of
// both orientations.  spec: per pair four sequences of S1 (S^a, g^a, S^b, g^b) in
// fixed point with exponents exs[4 w ..].
__device__ __forceinline__ void far_scatter(const FarArgs& a, int nw, int l0, int m0, const longlong2* spec,
                                            const int* exs, const FarPairFx* pf, const int* act) {
    const int N = a.N, S1 = a.M / 2 + 1, TM = kFarTileM, TL = nw / TM;
    const int nmodes = a.mode_hi - a.mode_lo;
    const int lg = __ffs(nw) - 1, lgl = __ffs(TL) - 1;
    const int total = nmodes << lg;
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
        const int w = idx & (nw - 1), n = idx >> lg;
        const int f = act[w];
        if (!(f & 4)) continue;
        const int l = l0 + (w & (TL - 1)), m = m0 + (w >> lgl);
        const int nn = a.mode_lo + n;
        const longlong2* b = spec + (size_t)w * 4 * S1;
        const int* ex = exs + 4 * w;
        const FarPairFx& p = pf[w];
        const bool real = (f & 8) != 0;
        longlong2 sa = fx2(0, 0), sb = sa, ga = sa, gb = sa, s2a = sa, s2b = sa;
        if (f & 3) {
            sa = b[nn];
            ga = b[S1 + nn];
            sb = b[2 * S1 + nn];
            gb = b[3 * S1 + nn];
            s2a = sin2_mode(b + S1, nn);
            s2b = sin2_mode(b + 3 * S1, nn);
        }
#pragma unroll
        for (int o = 0; o < 2; ++o) {
            if (o == 1 && l == m) break;             // the diagonal entry once
            const int tgt = o == 0 ? l : m, src = o == 0 ? m : l;
            double2 vs[2] = {c2(0.0, 0.0), c2(0.0, 0.0)}, vk[2] = {vs[0], vs[0]};
            if ((f >> o) & 1) {
                const int4 q0 = o == 0 ? p.nd0 : p.nd0t, qs = o == 0 ? p.nds : p.ndst;
                const int2 ws = o == 0 ? p.ws : p.wst;
                const int en = o == 0 ? p.en : p.ent, es = o == 0 ? p.ews : p.ewst;
                vk[0] = nd_mode(q0, qs, ga, s2a, real, fx_ex_add(ex[1], en));
                vk[1] = nd_mode(q0, qs, gb, s2b, real, fx_ex_add(ex[3], en));
                vs[0] = fx_to_double2(fx2(fx_mul(sa.x, ws.x, ws.y), fx_mul(sa.y, ws.x, ws.y)), fx_ex_add(ex[0], es));
                vs[1] = fx_to_double2(fx2(fx_mul(sb.x, ws.x, ws.y), fx_mul(sb.y, ws.x, ws.y)), fx_ex_add(ex[2], es));
            }
            if (a.A) {
                // blocks: K^a -> (t, s); -S^a -> (t, N+s); K^b -> (N+t, s); S^b -> (N+t, N+s)
                const size_t ld = 2 * (size_t)N;
                double2* col0 = a.A + (size_t)n * ld * ld + (size_t)src * ld;
                double2* col1 = col0 + (size_t)N * ld;
                col0[tgt] = vk[0];
                col1[tgt] = c2(-vs[0].x, -vs[0].y);
                col0[N + tgt] = vk[1];
                col1[N + tgt] = vs[1];
            } else {
                const size_t NN = (size_t)N * N, e = (size_t)tgt * N + src;
                a.raw[((size_t)n * 4 + 0) * NN + e] = vs[0];
                a.raw[((size_t)n * 4 + 1) * NN + e] = vk[0];
                a.raw[((size_t)n * 4 + 2) * NN + e] = vs[1];
                a.raw[((size_t)n * 4 + 3) * NN + e] = vk[1];
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Close pairs: from the samples to the modes.
//   S^_n = (1/2pi) sum_{|k| < M/2} Z^_{|n-k|} F1_k + R1_n   (K^_n with D^, F3, R3)
// The convolution is a circular one of length 2M (exact for n < M/2) of the even
// sequences z[m] = Z^_{|m|}, D^_{|m|} (|m| <= M-2) and c[k] = C_{|k|} (|k| <=
// M/2-1); all are even, so every transform is an even-sequence DFT of M+1 values,
// and the inverse of an even sequence is its forward transform divided by 2M.
// ---------------------------------------------------------------------------
struct NearShape {
    bool packed;      // both regions as real and imaginary parts of one sequence (real pairs)
    bool plain;       // far by the criterion: samples of S~ and K~ only
    bool share;       // the mirror's K^ too
    int mode_lo, nmodes;
    const double2 *Z, *D, *Dm;    // Laplace modes (and the mirror's D^), M - 1 values each
    double2 *out, *outm;          // [kernel][mode] of the pair and its mirror
};

// One CTA.  tw: 3M/2 twiddles of length 2M (e^{-2 pi i e / (2M)}); seq: the sample
// sequences of S1 = M/2 + 1 -- packed: f1, r1, f3, r3 (, the mirror's r3); general:
// the same four per region (, the mirror's r3 per region from index 8 on); plain: S~,
// K~ at 0, 2 of each region; zs: 3 sequences of S2 = M + 1 (Z^, D^, the mirror's
// D^); cv: the S and K convolution per region.  quantise(x, s) puts sequence s
// into fixed point and returns its scale (warp collective).
template <int NB, typename Q>
__device__ __forceinline__ void near_finish(const NearShape& p, int M, const int4* tw, longlong2* seq, double2* zs,
                                            double2* cv, Q quantise) {
    constexpr int NBH = (NB + 1) / 2;   // of the length-M transforms
    __shared__ int exq[10], exz[3], exc[4], exo[6];
    const int K = M / 2, S1 = K + 1, S2 = M + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    const double scale = 6.28318530717958647692 / M;
    const int mirror0 = p.packed ? 4 : 8;          // the mirror's r3
    // One warp per task, the longest first.  Phase 0: a smooth factor's transform of
    // length M followed by its modes' transform of length 2M; the Laplace modes'
    // transforms; the remainders' transforms.  Phase 1: the products' transforms.  (One
    // loop, so that each transform's code is in the kernel once.)
    const int nc = p.plain ? 0 : p.packed ? 2 : 4, nz = p.plain ? 0 : p.share ? 3 : 2;
    const int nr = p.plain ? 4 : nc + (p.share ? nc / 2 : 0);
    for (int phase = 0; phase < 2; ++phase) {
        const int ntask = phase == 0 ? nc + nz + nr : nc + (p.share ? nc / 2 : 0);
        for (int t = warp; t < ntask; t += nwarp) {
            double2* y = nullptr;         // sequence of length 2M to transform, its scale and exponent's place
            int* ey = nullptr;
            FxScale sc;
            if (phase == 0 && (t < nc || t >= nc + nz)) {
                // f1 / f3 (t < nc), r1 / r3 of the same pairs, the mirror's r3; plain: 0, 2, 4, 6
                const int u = t - nc - nz;
                const int s = t < nc ? 2 * t : p.plain ? 2 * u : u < nc ? 2 * u + 1 : mirror0 + (u - nc);
                longlong2* x = seq + s * S1;
                const int ex = fx_even_dft_call<NBH>(x, quantise(x, s), K, tw, 2, lane);
                if (lane == 0) exq[s] = ex;
                if (t < nc) {
                    // packed: F1a + i F1b and F3a - i F3b (region b's -D^ as the conjugate)
                    y = cv + t * S2;
                    ey = exc + t;
                    sc = fx_requantise(x, reinterpret_cast<longlong2*>(y), K, S2, ex, p.packed && t == 1, lane);
                }
            } else {
                if (phase == 0) {
                    const double2* src = t == nc ? p.Z : t == nc + 1 ? p.D : p.Dm;
                    y = zs + (t - nc) * S2;
                    ey = exz + (t - nc);
                    for (int i = lane; i <= M; i += 32) y[i] = i <= M - 2 ? src[i] : c2(0.0, 0.0);
                    __syncwarp();
                } else {
                    y = t < nc ? cv + t * S2 : zs + (t - nc) * S2;
                    ey = exo + t;
                }
                sc = fx_quantise(y, S2, lane);
            }
            if (y) {
                const int ex = fx_even_dft_call<NB>(reinterpret_cast<longlong2*>(y), sc, M, tw, 1, lane);
                if (lane == 0) *ey = ex;
            }
        }
        __syncthreads();
        if (phase == 1) break;
        if (p.plain) {
            for (int t = threadIdx.x; t < 4 * p.nmodes; t += blockDim.x) {
                const int k = t / p.nmodes, n = p.mode_lo + (t - k * p.nmodes);
                p.out[t] = cscale(fx_to_double2(seq[2 * k * S1 + n], exq[2 * k]), scale);
            }
            return;
        }
        // products in FP64 (their range is the product of two sequences' ranges);
        // region b's D^ is -D^ (unpacked)
        for (int i = threadIdx.x; i <= M; i += blockDim.x) {
            const longlong2* zi = reinterpret_cast<const longlong2*>(zs) + i;
            const longlong2* ci = reinterpret_cast<const longlong2*>(cv) + i;
            const double2 z = fx_to_double2(zi[0], exz[0]), d = fx_to_double2(zi[S2], exz[1]);
            const double2 dm = p.share ? fx_to_double2(zi[2 * S2], exz[2]) : c2(0.0, 0.0);
            for (int r = 0; r < nc / 2; ++r) {
                const double2 cS = fx_to_double2(ci[2 * r * S2], exc[2 * r]);
                double2 cK = fx_to_double2(ci[(2 * r + 1) * S2], exc[2 * r + 1]);
                if (r == 1) cK = c2(-cK.x, -cK.y);
                cv[2 * r * S2 + i] = cmul(z, cS);
                cv[(2 * r + 1) * S2 + i] = cmul(d, cK);
                if (p.share) zs[r * S2 + i] = cmul(dm, cK);
            }
        }
        __syncthreads();
    }
    // (1 / 2 pi) (1 / 2M) of the convolution and 2 pi / M of the modes
    const double c = 0.5 / ((double)M * M);
    const longlong2* cq = reinterpret_cast<const longlong2*>(cv);
    const longlong2* zq = reinterpret_cast<const longlong2*>(zs);
    for (int t = threadIdx.x; t < nc * p.nmodes; t += blockDim.x) {
        const int k = t / p.nmodes, n = p.mode_lo + (t - k * p.nmodes);
        const int s = 2 * k + 1, sm = mirror0 + (k >> 1);
        const double2 v = cscale(fx_to_double2(cq[k * S2 + n], exo[k]), c);
        const double2 r = fx_to_double2(seq[s * S1 + n], exq[s]);
        double2 vm = v, rm = r;
        if (p.share && (k & 1)) {
            vm = cscale(fx_to_double2(zq[(k >> 1) * S2 + n], exo[nc + (k >> 1)]), c);
            rm = fx_to_double2(seq[sm * S1 + n], exq[sm]);
        }
        if (p.packed) {
            // real parts from the convolutions, imaginary parts from the remainders
            p.out[t] = c2(v.x, r.x * scale);
            p.out[2 * p.nmodes + t] = c2(v.y, r.y * scale);
            if (p.share) {
                p.outm[t] = c2(vm.x, rm.x * scale);
                p.outm[2 * p.nmodes + t] = c2(vm.y, rm.y * scale);
            }
        } else {
            p.out[t] = c2(fma(r.x, scale, v.x), fma(r.y, scale, v.y));
            if (p.share) p.outm[t] = c2(fma(rm.x, scale, vm.x), fma(rm.y, scale, vm.y));
        }
    }
}

// Calls f with the transform size class of K points, ceil(K / 128): the
// butterflies a lane holds in registers (M <= 768, so up to 3 for K = M/2 and 6
// for K = M; 5 takes the variant of 6)
template <typename F>
static cudaError_t with_half_class(int M, F f) {
    if (M <= 256) return f(std::integral_constant<int, 1>());
    if (M <= 512) return f(std::integral_constant<int, 2>());
    return f(std::integral_constant<int, 3>());
}
template <typename F>
static cudaError_t with_full_class(int M, F f) {
    if (M <= 128) return f(std::integral_constant<int, 1>());
    if (M <= 256) return f(std::integral_constant<int, 2>());
    if (M <= 384) return f(std::integral_constant<int, 3>());
    if (M <= 512) return f(std::integral_constant<int, 4>());
    return f(std::integral_constant<int, 6>());
}

}  // namespace
}  // namespace pmlbie
