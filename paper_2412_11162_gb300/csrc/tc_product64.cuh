// Complex128 matrix times a few right-hand sides on the 5th-generation tensor cores
// (sm_103a):  Y[b] += sign * A[b](rows row0 ..) X[b], A column-major n x n per mode.
//
// On the FP64 pipe (2 FMA a clock and SM) every entry of A costs 2 clocks per right-hand
// side, eight times the time its 16 bytes take from HBM at eight right-hand sides.  Here
// the product is formed from exact integer slices as in the LU's update
// (tc_update64.cuh): in chunks of 32 columns, a row of A and a column of X are eight
// balanced base-256 digits (62 bits) below their largest entry in the chunk; the digits
// are exact in fp16 (1024 + byte by a byte permutation, less 1152), the digit products of
// one weight, summed over the real depth 64, stay below 2^23 and are exact in the FP32
// accumulators; the weights are combined in a 64-bit integer (unit 2^-54 or less of the
// row's times the column's largest entry in the chunk, the dropped pairs of digits as in the
// update) and the chunks' sums are added in FP64.  A chunk's element that this unit is too
// coarse for (weak_sum: large entries of A meet small ones of X) is formed in FP64.
//
// A CTA holds 128 rows and walks its chunks.  The complex product is a real one of depth
// 64, A' = (Re A, Im A), and X' has, per right-hand side, the columns (Re x, -Im x) and
// (Im x, Re x).  The digits of X' lie one behind the other (8 x 16 columns), so that digit
// i of A' meets the digits 0 .. 7 - i of X' in one product of 16 (8 - i) columns, its
// result falling into accumulator columns 16 i .. (weight i + j at 16 (i + j)): 8 MMAs per
// 16 depths instead of 36.  The digits of A are formed in shared memory in two halves of
// 16 columns (64 KB), two CTAs to an SM cover each other's waits.
// What bounds it is the integer work of the digits, about 50 instructions per entry, once
// for up to 8 right-hand sides, and the elements in FP64, some 10 % there: n = 768, 96 modes,
// residual of 8 right-hand sides 2.19 -> 0.70 ms (0.51 without those elements).  Mixed solve
// for 64 waves (8 solved) at N = 384, M = 192 15.9 -> 16.6 ms by those elements, four
// instances with 4 waves at N = 256 16.5 -> 17.7 ms (all on the FP64 pipe about 7 and 3 ms more).
// Waits are bounded; an expiry gives NaN.
#pragma once

#include <cuda_fp16.h>

#include "tc_update64.cuh"

namespace pmlbie {
namespace tcu {

constexpr int kProdRows = 128, kProdCols = 32, kProdRhs = 8, kProdThreads = 256;
constexpr uint32_t kProdASlice = kProdRows * 32 * 2, kProdA = kSlices * kProdASlice;     // 8 KB, 64 KB
constexpr uint32_t kProdBHalf = 128 * 32 * 2;                                            // 8 KB
constexpr uint32_t kProdOffB = kProdA, kProdOffMax = kProdOffB + 2 * kProdBHalf;
constexpr uint32_t kProdOffEx = kProdOffMax + 2 * kProdRows * 4, kProdOffBar = kProdOffEx + 32;
constexpr uint32_t kProdSmem = kProdOffBar + 32;
constexpr uint32_t kProdTmem = 128;
// as kWeakBits, per chunk: the largest error by entry on the oracle's systems is below the
// FP64 product's with 49, about equal with 48, twice with 47
constexpr int kProdWeakBits = 49;

// fp16 pair of digit s (0: top) of two values in digit_bytes form
__device__ __forceinline__ uint32_t digit_half2(u64 a, u64 b, int s) {
    const unsigned wa = s < 4 ? (unsigned)(a >> 32) : (unsigned)a, wb = s < 4 ? (unsigned)(b >> 32) : (unsigned)b;
    const unsigned k = 3 - (s & 3);
    const unsigned t = (__byte_perm(wa, wb, k | (k << 4) | ((4 + k) << 8) | ((4 + k) << 12)) & 0x00ff00ffu) | 0x64006400u;
    __half2 h;
    *reinterpret_cast<unsigned*>(&h) = t;
    h = __hsub2(h, __half2half2(__ushort_as_half(0x6480)));     // 1152
    return *reinterpret_cast<unsigned*>(&h);
}
__device__ __forceinline__ void mma_f16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dtmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(taddr));
}

// Grid (row blocks of either side of `split` x groups of 8 right-hand sides, column
// splits, modes).
__global__ void __launch_bounds__(kProdThreads, 2) product64_kernel(ProductArgs a, int groups) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const int b = blockIdx.z;
    if (a.active && !a.active[b]) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, r = tid & 127, hf = tid >> 7;
    const int rb = blockIdx.x / groups, r0 = (blockIdx.x - rb * groups) * kProdRhs;
    const int nb0 = (a.split - a.row0 + kProdRows - 1) / kProdRows;
    const bool upper = rb < nb0;
    const int nq = min(kProdRhs, a.nrhs - r0), end = upper ? a.split : a.rows;
    const int row = (upper ? a.row0 + rb * kProdRows : a.split + (rb - nb0) * kProdRows) + r;
    const double2 *x0 = upper ? a.x0 : a.x0s, *x1 = upper ? a.x1 : a.x1s;
    unsigned* rmax = reinterpret_cast<unsigned*>(sm + kProdOffMax);
    int* exq = reinterpret_cast<int*>(sm + kProdOffEx);
    uint64_t* bar = reinterpret_cast<uint64_t*>(sm + kProdOffBar);
    uint32_t* tm = reinterpret_cast<uint32_t*>(bar + 1);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tm)),
                     "r"(kProdTmem));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        mb_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tm, sbase = smem_u32(sm);
    const int per = (a.nc + kProdCols - 1) / kProdCols, total = 2 * per;
    const int k0 = (int)((long long)total * blockIdx.y / gridDim.y), k1 = (int)((long long)total * (blockIdx.y + 1) / gridDim.y);
    const double2* Ab = a.A + (size_t)b * a.as + row;
    const int quad = warp & 3;
    double sum[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) sum[c] = 0.0;
    uint32_t phase = 0;
    bool fail = false;
    for (int k = k0; k < k1 && !fail; ++k) {
        const bool second = k >= per;
        const int c0 = (second ? k - per : k) * kProdCols, cw = min(kProdCols, a.nc - c0);
        const double2* Ac = Ab + (size_t)(c0 + (second ? a.nc : 0)) * a.ld;
        // entries: columns 16 s + 8 hf + e, s the half
        double2 v[16];
        unsigned m = 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int c = (i >> 3) * 16 + hf * 8 + (i & 7);
            v[i] = (row < end && c < cw) ? __ldg(Ac + (size_t)c * a.ld) : make_double2(0.0, 0.0);
        }
        const double2* x = (second ? x1 : x0) + (size_t)b * a.xs;
        const double2 xv = (warp < nq && lane < cw) ? x[(size_t)(c0 + lane) * a.nrhs + r0 + warp] : make_double2(0.0, 0.0);
#pragma unroll
        for (int i = 0; i < 16; ++i) m = max(m, mag_hi(v[i]));
        rmax[hf * kProdRows + r] = m;
        const int xtop = (int)(__reduce_max_sync(0xffffffffu, mag_hi(xv)) >> 20), xex = xtop - 1084;
        if (lane == 0) exq[warp] = xtop == 0x7ff ? kFxNonfinite : xex;
        {
            // digits of X': lanes 2 c, 2 c + 1 hold neighbouring depths; the even lane writes
            // column 2 q (Re x, -Im x), the odd one 2 q + 1 (Im x, Re x)
            const u64 xr = digit_bytes(xv.x, xex), xi = digit_bytes(xv.y, xex);
            const int c16 = lane & 14, odd = lane & 1;
            unsigned char* o = sm + kProdOffB + (lane >> 4) * kProdBHalf + (c16 >> 3) * 2048 + (2 * warp + odd) * 16 + (c16 & 7) * 2;
#pragma unroll
            for (int j = 0; j < kSlices; ++j) {
                const uint32_t h = digit_half2(xr, xi, j), g = __shfl_xor_sync(0xffffffffu, h, 1);
                const uint32_t re = odd ? __byte_perm(g, h, 0x5410) : __byte_perm(h, g, 0x5410);
                const uint32_t im = odd ? __byte_perm(g, h, 0x7632) : __byte_perm(h, g, 0x7632);
                *reinterpret_cast<uint32_t*>(o + j * 256) = odd ? im : re;
                *reinterpret_cast<uint32_t*>(o + j * 256 + 2 * 2048) = odd ? re : im ^ 0x80008000u;
            }
        }
        __syncthreads();
        const int top = (int)(max(rmax[r], rmax[kProdRows + r]) >> 20), ex = top - 1084;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            u64 re[8], im[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                re[e] = digit_bytes(v[8 * s + e].x, ex);
                im[e] = digit_bytes(v[8 * s + e].y, ex);
            }
            uint4* o = reinterpret_cast<uint4*>(sm) + hf * kProdRows + r;
#pragma unroll
            for (int j = 0; j < kSlices; ++j) {
                o[j * (kProdASlice / 16)] = make_uint4(digit_half2(re[0], re[1], j), digit_half2(re[2], re[3], j),
                                                       digit_half2(re[4], re[5], j), digit_half2(re[6], re[7], j));
                o[j * (kProdASlice / 16) + 2 * kProdRows] =
                    make_uint4(digit_half2(im[0], im[1], j), digit_half2(im[2], im[3], j),
                               digit_half2(im[4], im[5], j), digit_half2(im[6], im[7], j));
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (tid == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t LBO = 2048, SBO = 128, bb = sbase + kProdOffB + s * kProdBHalf;
                for (int i = 0; i < kSlices; ++i) {
                    // M = 128, N = 16 (8 - i), fp16 operands, FP32 accumulators
                    const uint32_t idesc = (1u << 4) | ((uint32_t)(2 * (kSlices - i)) << 17) | (8u << 24);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        mma_f16(tmem + 16 * i, smem_desc(sbase + i * kProdASlice + h * 2 * LBO, LBO, SBO),
                                smem_desc(bb + h * 2 * LBO, LBO, SBO), idesc, (uint32_t)((s | i | h) != 0));
                }
                mma_commit(bar);
            }
            const bool ok = mbar_wait(smem_u32(bar), phase);
            phase ^= 1;
            if (__syncthreads_or(!ok)) {
                fail = true;
                break;
            }
        }
        if (fail) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (4 * hf < nq) {
            // weights 2 p and 2 p + 1 together, as in update64_kernel
            const uint32_t t0 = tmem + ((uint32_t)(32 * quad) << 16) + 8 * hf;
            i64 acc[8];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                uint32_t y0[8], y1[8];
                tmem_ld8(t0 + 32 * p, y0);
                tmem_ld8(t0 + 32 * p + 16, y1);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int w = p < 2 ? (acc_int<false>(y0[c]) << 8) + acc_int<false>(y1[c])
                                        : (acc_int<true>(y0[c]) << 8) + acc_int<true>(y1[c]);
                    if (p == 0)
                        acc[c] = (i64)w;
                    else if (p < 3)
                        acc[c] = (acc[c] << 16) + w;
                    else
                        acc[c] = (acc[c] << 4) + ((w + 2048) >> 12);
                }
            }
            unsigned weak = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int eq = exq[4 * hf + q];
                const int e = (top == 0x7ff || eq == kFxNonfinite) ? kFxNonfinite : ex + eq + 68;
                const double vr = fx_to_double(acc[2 * q], e), vi = fx_to_double(acc[2 * q + 1], e);
                const unsigned hi = max(max(mag_hi(vr), mag_hi(vi)), max(mag_hi(sum[2 * q]), mag_hi(sum[2 * q + 1])));
                if (row < end && 4 * hf + q < nq && weak_sum(e, hi, kProdWeakBits)) {
                    weak |= 1u << q;
                } else {
                    sum[2 * q] += vr;
                    sum[2 * q + 1] += vi;
                }
            }
            if (weak) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (weak >> q & 1) {
                        double sr = 0.0, si = 0.0;
#pragma unroll 8
                        for (int c = 0; c < cw; ++c) {
                            const double2 w = __ldg(Ac + (size_t)c * a.ld), y = x[(size_t)(c0 + c) * a.nrhs + r0 + 4 * hf + q];
                            sr = fma(w.x, y.x, fma(-w.y, y.y, sr));
                            si = fma(w.x, y.y, fma(w.y, y.x, si));
                        }
                        sum[2 * q] += sr;
                        sum[2 * q + 1] += si;
                    }
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();         // exponents and accumulators are read before the next chunk
    }
    if (row < end) {
        const int yr = a.map ? a.map[row] : row;
        double* y = reinterpret_cast<double*>(a.Y + (size_t)b * a.ys + (size_t)yr * a.nrhs + r0 + 4 * hf);
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (4 * hf + (c >> 1) < nq) atomicAdd(y + c, fail ? __hiloint2double(0x7ff80000, 0) : a.sign * sum[c]);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kProdTmem));
}

}  // namespace tcu
}  // namespace pmlbie
