// Trailing update of the complex128 LU on the 5th-generation tensor cores (sm_103a):
//
//   A22 <- A22 - L21 U12,   column-major, leading dimension n, depth kNB = 32.
//
// The GB300 retires 2 FP64 FMA per SM per clock (1.05 TFLOP/s), its tensor cores
// 1925 TFLOP/s in bf16, so the product is formed from exact integer slices (the
// splitting of Ozaki, Ogita, Oishi and Rump for error-free matrix products):
//
//   L21[i][k] = 2^{e_i} sum_s d_s 2^{-8 s - 6}, e_i from the row's largest entry,
//   U12[k][j] = 2^{f_j} sum_t c_t 2^{-8 t - 6}, f_j from the column's,
//
// with eight balanced base-256 digits each (|d| <= 128, exact in bf16; 62 bits below
// the row's or column's largest entry, so entries are represented to 2^-63 of it).
// Digit products are integers of at most 2^14; those of one weight s + t = q, summed
// over at most 8 pairs and the real depth 64, stay below 2^23 and are exact in the
// FP32 accumulators.  The 36 pairs with s + t <= 7 are kept; the dropped ones come to
// about 2^-59 of the row's times the column's largest entry, 2^-51 at worst (all digits
// of weight 8 at their largest and of one sign).  An element of the product is the
// combination of its eight accumulators in a 64-bit integer, in units of 2^-54 or less
// of the row's times the column's largest entry, converted to double and subtracted
// from A22.  Elements that this unit is too coarse for (weak_sum) are left as they are
// and formed in FP64 by weak64_kernel, so that every entry keeps what the FP64 dot
// product gives it.  Rows or columns holding a NaN or an infinity give NaN.
//
// The complex product is one real GEMM of depth 64 (as in tc_update.cuh): A' row 2i =
// (Re L, -Im L), row 2i + 1 = (Im L, Re L); B' = [Re U; Im U].  operand_image64_kernel
// forms, per step, the digit images of every 64-row block of L21 (8 x 16 KB) and
// 32-column block of U12 (8 x 4 KB) in the MMA's shared-memory layout (canonical
// K-major, no swizzle).  update64_kernel is persistent and warp-specialised: one CTA
// per SM walks row units (mode, 64-row block); warp 0 fetches the A' image once per
// unit and the B' images in two stages by bulk copies, warp 1 issues the 144
// tcgen05.mma (M = 128, N = 32, K = 16) of a 64 x 32 tile into one of two sets of eight
// accumulators (all 512 columns of tensor memory), warps 2-9 read them, combine, and
// update the tile in global memory (its values loaded before the accumulators are
// waited for).  Bounded waits as in tc_update.cuh; an expiry marks info[b] = -1.
//
// Measured (GB300), all updates of one factorisation, CUDA-core FP64 -> this: n = 512,
// 64 modes 28.8 -> 4.3 ms (of it the FP64 entries, 4 % of them, 1.7 ms, the operand
// images 0.35), n = 320, 32 modes 3.6 -> 1.2 ms (0.64, 0.11).  The FP64 entries are bounded
// by the FP64 pipe; the MMAs wait for the operand images next (A' is re-read from shared
// memory for every 32 columns).
#pragma once

#include "fxdft.cuh"
#include "tc_update.cuh"

namespace pmlbie {
namespace tcu {

constexpr int kSlices = 8;
constexpr int kRows64 = 64, kCols64 = 32;                       // complex tile
constexpr uint32_t kASlice = 128 * 64 * 2, kBSlice = 32 * 64 * 2;   // 16 KB, 4 KB
constexpr uint32_t kAImg64 = kSlices * kASlice, kBImg64 = kSlices * kBSlice;   // 128 KB, 32 KB
constexpr int kUpd64Threads = 320;                              // producer, MMA, 8 epilogue warps
constexpr uint32_t kOff64B = kAImg64, kOff64Bar = kOff64B + 2 * kBImg64;
constexpr uint32_t kUpd64Smem = kOff64Bar + 256;
constexpr uint32_t kIdesc64 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kCols64 >> 3) << 17) | (8u << 24);

__host__ __device__ constexpr int row_blocks64(int rem) { return (rem + kRows64 - 1) / kRows64; }
__host__ __device__ constexpr int col_blocks64(int rem) { return (rem + kCols64 - 1) / kCols64; }

// Digits of q = round(x 2^-ex), |q| < 2^62: bytes of q + 0x80...80 (below the top
// one) are the balanced digits plus 128, the top byte is the top digit
__device__ __forceinline__ u64 digit_bytes(double x, int ex) {
    return (u64)fx_of_double(x, ex) + 0x0080808080808080ull + (128ull << 56);
}
// bf16 pair of digit s (0: top) of two values
__device__ __forceinline__ uint32_t digit_pair(u64 a, u64 b, int s) {
    const unsigned da = (unsigned)(a >> (56 - 8 * s)) & 0xffu, db = (unsigned)(b >> (56 - 8 * s)) & 0xffu;
    const float fa = __uint_as_float(0x4b000000u | da) - 8388736.0f;     // byte - 128, exact
    const float fb = __uint_as_float(0x4b000000u | db) - 8388736.0f;
    return (__float_as_uint(fa) >> 16) | (__float_as_uint(fb) & 0xffff0000u);
}

// Digit images of one step.  Grid (row blocks + column blocks, batch), 256 threads.
// Four neighbouring lanes share a row of L21 (a column of U12), eight depths each.
// expo: per mode n entries, the exponent of row r at [r] and of column c at [n + c]
// (kFxNonfinite for a row or column with a NaN or an infinity).
__global__ void __launch_bounds__(256) operand_image64_kernel(int n, int k0, int nra, const double2* A,
                                                              unsigned char* img, int nca, int* expo, int* count) {
    const int b = blockIdx.y, first = k0 + 32;
    if (blockIdx.x == 0 && b == 0 && threadIdx.x == 0) *count = 0;
    const double2* a = A + (size_t)b * n * n;
    const bool rows = (int)blockIdx.x < nra;
    const int blk = rows ? blockIdx.x : blockIdx.x - nra;
    const int lines = rows ? kRows64 : kCols64;
    const int line = threadIdx.x >> 2, kg = threadIdx.x & 3;
    if (line >= lines) return;                        // whole warps
    const int idx = first + blk * lines + line;       // row of L21 or column of U12
    double2 v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int k = k0 + 8 * kg + e;
        v[e] = idx < n ? (rows ? a[(size_t)k * n + idx] : a[(size_t)idx * n + k]) : make_double2(0.0, 0.0);
    }
    unsigned m = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e)
        m = max(m, max((unsigned)__double2hiint(v[e].x) & 0x7fffffffu, (unsigned)__double2hiint(v[e].y) & 0x7fffffffu));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
    const int top = (int)(m >> 20), ex = top - 1084;  // |x| 2^-ex < 2^62
    if (kg == 0 && idx < n) expo[(size_t)b * 2 * n + (rows ? 0 : n) + idx] = top == 0x7ff ? kFxNonfinite : ex;
    u64 re[8], im[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        re[e] = digit_bytes(v[e].x, ex);
        im[e] = digit_bytes(v[e].y, ex);
    }
    // images: mode's row blocks, then its column blocks
    unsigned char* base = img + (size_t)b * ((size_t)nra * kAImg64 + (size_t)nca * kBImg64) +
                          (rows ? (size_t)blk * kAImg64 : (size_t)nra * kAImg64 + (size_t)blk * kBImg64);
#pragma unroll
    for (int s = 0; s < kSlices; ++s) {
        uint4 r, i;
        r.x = digit_pair(re[0], re[1], s), r.y = digit_pair(re[2], re[3], s);
        r.z = digit_pair(re[4], re[5], s), r.w = digit_pair(re[6], re[7], s);
        i.x = digit_pair(im[0], im[1], s), i.y = digit_pair(im[2], im[3], s);
        i.z = digit_pair(im[4], im[5], s), i.w = digit_pair(im[6], im[7], s);
        if (rows) {
            // 16-byte unit (kc, real row r): u = kc 128 + r, depths 8 kc .. 8 kc + 7
            uint4* o = reinterpret_cast<uint4*>(base + s * kASlice);
            const uint4 ni = make_uint4(i.x ^ 0x80008000u, i.y ^ 0x80008000u, i.z ^ 0x80008000u, i.w ^ 0x80008000u);
            o[kg * 128 + 2 * line] = r;
            o[(4 + kg) * 128 + 2 * line] = ni;
            o[kg * 128 + 2 * line + 1] = i;
            o[(4 + kg) * 128 + 2 * line + 1] = r;
        } else {
            uint4* o = reinterpret_cast<uint4*>(base + s * kBSlice);
            o[kg * 32 + line] = r;
            o[(4 + kg) * 32 + line] = i;
        }
    }
}

__device__ __forceinline__ void mma_bf16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dtmem),
        "l"(adesc), "l"(bdesc), "r"(kIdesc64), "r"(acc));
}
// 16 columns of this warp's 32 lanes
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
// An integer held as a float, without the FP64 pipe's conversions.  Weight q sums 64 (q + 1)
// digit products of at most 2^14: up to 2^22 for q < 4, where one magic number decodes
// both signs, up to 2^23 beyond (kWide), where the sign is taken out first.
template <bool kWide>
__device__ __forceinline__ int acc_int(uint32_t bits) {
    const float v = __uint_as_float(bits);
    if (!kWide) return __float_as_int(v + 12582912.0f) - 0x4b400000;
    const int m = __float_as_int(fabsf(v) + 8388608.0f) - 0x4b000000, sg = (int)bits >> 31;
    return (m ^ sg) - sg;
}

// A sum in units of 2^ex where 2^ex exceeds 2^-kWeakBits of the values that it meets (hi:
// the largest of their high words, signs off) has lost bits that a double would keep: the
// digits lie below the row's and the column's largest entry, and the entry itself can be
// smaller by any factor (the modal kernels of high modes fall off like (rho / rho')^n
// next to the axis).  Such entries are formed again in FP64.
// (50: the factors of the oracle's systems then are as close to P A entry by entry as in
// FP64; with 48 and 46 two and five to twenty times as far.)
constexpr int kWeakBits = 50;
__device__ __forceinline__ bool weak_sum(int ex, unsigned hi, int bits = kWeakBits) {
    return ex != kFxNonfinite && ex + bits > (int)(hi >> 20) - 1023;
}
__device__ __forceinline__ unsigned mag_hi(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
__device__ __forceinline__ unsigned mag_hi(double2 v) { return max(mag_hi(v.x), mag_hi(v.y)); }

struct Upd64Bars {
    uint64_t a_full, a_empty, b_full[2], b_empty[2], acc_full[2], acc_empty[2];
    uint32_t tmem;
    int err;
};
static_assert(sizeof(Upd64Bars) <= 256, "barrier block");

__global__ void __launch_bounds__(kUpd64Threads, 1) update64_kernel(int n, int k0, int batch, double2* A,
                                                                    const unsigned char* img, const int* expo,
                                                                    int* info, uint2* list, int* count) {
    extern __shared__ __align__(1024) unsigned char sm[];
    Upd64Bars* bar = reinterpret_cast<Upd64Bars*>(sm + kOff64Bar);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int first = k0 + 32, rem = n - first;
    const int nra = row_blocks64(rem), nca = col_blocks64(rem);
    const size_t per_mode = (size_t)nra * kAImg64 + (size_t)nca * kBImg64;
    const int U = batch * nra, G = gridDim.x;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bar->tmem)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        mb_init(&bar->a_full, 1);
        mb_init(&bar->a_empty, 1);
        for (int s = 0; s < 2; ++s) {
            mb_init(&bar->b_full[s], 1);
            mb_init(&bar->b_empty[s], 1);
            mb_init(&bar->acc_full[s], 1);
            mb_init(&bar->acc_empty[s], 8);       // one arrival per epilogue warp
        }
        bar->err = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = bar->tmem, sbase = smem_u32(sm);
    auto failed = [&] { return *reinterpret_cast<const volatile int*>(&bar->err) != 0; };

    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            int i = 0, k = 0, issued = 0;
            for (int u = blockIdx.x; u < U && ok; u += G, ++k) {
                const int b = u / nra, bx = u - b * nra;
                const unsigned char* base = img + (size_t)b * per_mode;
                if (k >= 1 && !mbar_wait(smem_u32(&bar->a_empty), (uint32_t)((k - 1) & 1))) {
                    ok = false;
                    break;
                }
                mb_expect(&bar->a_full, kAImg64);
                bulk_load(sbase, base + (size_t)bx * kAImg64, kAImg64, smem_u32(&bar->a_full));
                ++issued;
                for (int by = 0; by < nca; ++by, ++i) {
                    const int s = i & 1;
                    if (i >= 2 && !mbar_wait(smem_u32(&bar->b_empty[s]), (uint32_t)(((i >> 1) - 1) & 1))) {
                        ok = false;
                        break;
                    }
                    mb_expect(&bar->b_full[s], kBImg64);
                    bulk_load(sbase + kOff64B + s * kBImg64, base + (size_t)nra * kAImg64 + (size_t)by * kBImg64, kBImg64,
                              smem_u32(&bar->b_full[s]));
                }
            }
            if (!ok) {
                bar->err = 1;
                // copies in flight: wait (bounded) for the last issued use of every stage
                if (issued > 0) mbar_wait(smem_u32(&bar->a_full), (uint32_t)((issued - 1) & 1));
                for (int s = 0; s < 2; ++s)
                    if (i > s) mbar_wait(smem_u32(&bar->b_full[s]), (uint32_t)((((i - 1 - s) >> 1)) & 1));
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t aLBO = 16 * 128, bLBO = 4 * 128, SBO = 128;   // 128 and 32 rows of 16 bytes
            bool ok = true;
            int i = 0, k = 0;
            for (int u = blockIdx.x; u < U && ok; u += G, ++k) {
                if (failed() || !mbar_wait(smem_u32(&bar->a_full), (uint32_t)(k & 1))) {
                    ok = false;
                    break;
                }
                for (int by = 0; by < nca; ++by, ++i) {
                    const int s = i & 1;
                    if (failed() || !mbar_wait(smem_u32(&bar->b_full[s]), (uint32_t)((i >> 1) & 1)) ||
                        (i >= 2 && !mbar_wait(smem_u32(&bar->acc_empty[s]), (uint32_t)(((i >> 1) - 1) & 1)))) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t bb = sbase + kOff64B + s * kBImg64, d0 = tmem + (uint32_t)(s * 256);
                    // accumulator q: the digit pairs of weight q
                    for (int q = 0; q < kSlices; ++q)
                        for (int t = 0; t <= q; ++t) {
#pragma unroll
                            for (int h = 0; h < 4; ++h) {
                                const uint64_t ad = smem_desc(sbase + t * kASlice + h * 2 * aLBO, aLBO, SBO);
                                const uint64_t bd = smem_desc(bb + (q - t) * kBSlice + h * 2 * bLBO, bLBO, SBO);
                                mma_bf16(d0 + (uint32_t)(q * kCols64), ad, bd, (uint32_t)((t | h) != 0));
                            }
                        }
                    mma_commit(&bar->b_empty[s]);
                    mma_commit(&bar->acc_full[s]);
                    if (by == nca - 1) mma_commit(&bar->a_empty);
                }
            }
            if (!ok) bar->err = 1;
        }
    } else {
        // epilogue: lane quadrant warp & 3 (real rows 32 q ..), columns 16 h .. 16 h + 15 of
        // the tile with h = (warp - 2) / 4
        const int quad = warp & 3, h = (warp - 2) >> 2;
        const int rr = 32 * quad + lane, part = rr & 1;
        int i = 0;
        bool stop = false;
        for (int u = blockIdx.x; u < U && !stop; u += G) {
            const int b = u / nra, bx = u - b * nra;
            const int row = first + bx * kRows64 + (rr >> 1);
            const int* ef = expo + (size_t)b * 2 * n;
            const int er = row < n ? ef[row] : 0;
            double* a = reinterpret_cast<double*>(A + (size_t)b * n * n + row) + part;
            for (int by = 0; by < nca; ++by, ++i) {
                const int s = i & 1, c0 = first + by * kCols64 + 16 * h;
                double cv[16];
                int ec[16];
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const bool in = row < n && c0 + c < n;
                    cv[c] = in ? a[(size_t)(c0 + c) * n * 2] : 0.0;
                    ec[c] = in ? ef[n + c0 + c] : 0;
                }
                const bool ok = mbar_wait(smem_u32(&bar->acc_full[s]), (uint32_t)((i >> 1) & 1));
                if (!ok) bar->err = 1;
                // one decision for all 256 epilogue threads (as in tc_update.cuh)
                uint32_t any;
                asm volatile(
                    "{\n\t.reg .pred p, q;\n\t"
                    "setp.ne.u32 p, %1, 0;\n\t"
                    "bar.red.or.pred q, 1, 256, p;\n\t"
                    "selp.u32 %0, 1, 0, q;\n\t}\n"
                    : "=r"(any)
                    : "r"((uint32_t)(!ok || failed()))
                    : "memory");
                if (any) {
                    stop = true;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // digits of weights 2 p and 2 p + 1 combined: (v_2p << 8) + v_2p+1
                const uint32_t t0 = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(s * 256 + 16 * h);
                i64 acc[16];
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    uint32_t x[16], y[16];
                    tmem_ld16(t0 + (uint32_t)(2 * p * kCols64), x);
                    tmem_ld16(t0 + (uint32_t)((2 * p + 1) * kCols64), y);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        const int w = p < 2 ? (acc_int<false>(x[c]) << 8) + acc_int<false>(y[c])
                                            : (acc_int<true>(x[c]) << 8) + acc_int<true>(y[c]);
                        // unit 2^-56 of the product's scale: weights 44 - 8 q
                        if (p == 0)
                            acc[c] = (i64)w;
                        else if (p < 3)
                            acc[c] = (acc[c] << 16) + w;
                        else
                            acc[c] = (acc[c] << 4) + ((w + 2048) >> 12);
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mb_arrive(&bar->acc_empty[s]);
                unsigned weak = 0;
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    // sum of 2^-12 2^-8q 2^(e + f) v_q with q = 2^62-scaled digits: exponent er + ec + 68
                    const int ex = (er == kFxNonfinite || ec[c] == kFxNonfinite) ? kFxNonfinite : er + ec[c] + 68;
                    const double v = fx_to_double(acc[c], ex);
                    unsigned hi = max(mag_hi(cv[c]), mag_hi(v));
                    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, 1));      // the entry's other part
                    if (row < n && c0 + c < n && weak_sum(ex, hi)) weak |= 1u << c;
                    cv[c] -= v;
                }
                weak = __reduce_or_sync(0xffffffffu, weak);
                if (weak && lane == 0)
                    list[atomicAdd(count, 1)] = make_uint2((unsigned)b << 16 | weak, (unsigned)(row >> 4) << 16 | (c0 >> 4));
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    if (row < n && c0 + c < n && !(weak >> c & 1)) a[(size_t)(c0 + c) * n * 2] = cv[c];
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (failed() && tid == 0)
        for (int u = blockIdx.x; u < U; u += G) info[u / nra] = -1;
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// The columns of 16 rows that update64_kernel left as they were, in FP64: a warp takes
// one entry of the list (mode and mask of 16 columns, row / 16 and first column / 16);
// two lanes share a row, half of the depth each.  An own launch, because the entries
// lie in few row blocks: formed in the update's epilogue, one column after the other,
// they held up the CTAs that own those rows.
constexpr int kWeakThreads = 256;
__global__ void __launch_bounds__(kWeakThreads) weak64_kernel(int n, int k0, double2* A, const uint2* list,
                                                              const int* count) {
    const int lane = threadIdx.x & 31, part = lane & 1, d0 = k0 + 16 * part, total = *count;
    for (int i = (blockIdx.x * kWeakThreads + threadIdx.x) >> 5; i < total; i += gridDim.x * (kWeakThreads >> 5)) {
        const uint2 e = list[i];
        double2* m = A + (size_t)(e.x >> 16) * n * n;
        const int row = (int)(e.y >> 16) * 16 + (lane >> 1), c0 = (int)(e.y & 0xffffu) * 16;
        double2 l[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) l[k] = m[(size_t)(d0 + k) * n + min(row, n - 1)];
        for (unsigned cols = e.x & 0xffffu; cols; cols &= cols - 1) {
            double2* col = m + (size_t)(c0 + __ffs(cols) - 1) * n;
            double re = 0.0, im = 0.0;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const double2 u = col[d0 + k];
                re = fma(l[k].x, u.x, fma(-l[k].y, u.y, re));
                im = fma(l[k].x, u.y, fma(l[k].y, u.x, im));
            }
            re += __shfl_xor_sync(0xffffffffu, re, 1);
            im += __shfl_xor_sync(0xffffffffu, im, 1);
            if (row < n) reinterpret_cast<double*>(col + row)[part] -= part ? im : re;
        }
    }
}

}  // namespace tcu
}  // namespace pmlbie
