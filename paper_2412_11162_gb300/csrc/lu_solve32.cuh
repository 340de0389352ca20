// Complex64 triangular solves of the mixed path's refinement (sm_103a): L U x = b per
// mode with the factors of lu.cu (n a multiple of 32, inverted diagonal blocks, each
// step's interchanges in ptab), up to RM right-hand sides per CTA.
//
// The factors do not depend on the solve, so a producer warp streams them through shared
// memory ahead of the arithmetic: 8 columns of up to 512 rows of a block column per
// stage, one bulk copy per column, three stages, and the 32 x 32 inverse blocks in two
// more.  The 16 consumer warps hold the rows of a segment in registers for the 32
// columns of a block (a thread has one row, or two rows and half of the right-hand
// sides).  Loads issued by the consuming threads, as many as registers allow, left each
// block waiting for 16 round trips to L2 with eight right-hand sides: n = 768, 96 modes
// 1.09 ms per solve, 0.33 ms now; n = 1600, 128 modes, one right-hand side 0.71 -> 0.58 ms.
// Waits are bounded; an expiry gives NaN.
#pragma once

#include "tc_update.cuh"

namespace pmlbie {
namespace {

constexpr int kStRows = 512, kStCols = 8, kStages = 3, kStThreads = 544;
constexpr uint32_t kStDiag = 32 * 32 * 8, kStOffDiag = 128, kStOffX = kStOffDiag + 2 * kStDiag;
// the CTA's shared memory: barriers, inverse blocks, right-hand sides, stages of `rows` rows
// (small systems leave room for another CTA; large ones leave less for the stages; 0: none)
constexpr size_t kStSmemMax = 227 * 1024;
inline size_t st_smem(int n, int R, int rows) { return kStOffX + 8 * (size_t)n * R + (size_t)kStages * rows * kStCols * 8; }
inline int st_rows(int n, int R) {
    int rows = n < kStRows ? n : kStRows;
    while (rows > 0 && st_smem(n, R, rows) > kStSmemMax) rows -= 32;
    return rows;
}
struct StreamBars {
    uint64_t full[kStages], empty[kStages], dfull[2], dempty[2];
    int err;
};
static_assert(sizeof(StreamBars) <= 128, "barrier block");

template <int RM>
__global__ void __launch_bounds__(kStThreads, 1) lu_solve32_kernel(int n, int nv, int nrhs, int sr, const float2* LU, float2* B,
                                                                const int* active, const float2* dinv,
                                                                const int2* ptab) {
    using namespace tcu;
    extern __shared__ __align__(1024) unsigned char sm[];
    const int b = blockIdx.x, r0 = blockIdx.y * RM, nr = min(RM, nrhs - r0);
    if (active && !active[b]) return;
    StreamBars* bar = reinterpret_cast<StreamBars*>(sm);
    float2* sx = reinterpret_cast<float2*>(sm + kStOffX);       // [n][RM]
    float2* stage = sx + (size_t)n * RM;                        // kStages x [kStCols][sr]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nblk = n / 32;
    const float2* a = LU + (size_t)b * n * n;
    float2* x = B + (size_t)b * nv * nrhs + r0;
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) mb_init(&bar->full[s], 1), mb_init(&bar->empty[s], 16);
        for (int s = 0; s < 2; ++s) mb_init(&bar->dfull[s], 1), mb_init(&bar->dempty[s], 1);
        bar->err = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int idx = tid; idx < n * RM; idx += kStThreads) {
        const int i = idx / RM, q = idx - i * RM;
        sx[idx] = i < nv && q < nr ? x[(size_t)i * nrhs + q] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    volatile int* err = &bar->err;
    auto wait = [&](uint64_t* m, int phase) {
        if (!*err && !mbar_wait(smem_u32(m), (uint32_t)phase & 1u)) *err = 1;
    };
    // block k's rows of either sweep: below it (forward), above it (backward)
    auto first = [&](int k, int back) { return back ? 0 : 32 * (k + 1); };
    auto last = [&](int k, int back) { return back ? 32 * k : n; };

    if (warp == 16) {
        if (lane == 0) {
            int i = 0, d = 0;
            const unsigned char* db = reinterpret_cast<const unsigned char*>(dinv + (size_t)b * nblk * 2 * 1024);
            for (int t = 0; t < 2 * nblk && !*err; ++t, ++d) {
                const int back = t >= nblk, k = back ? 2 * nblk - 1 - t : t;
                if (d >= 2) wait(&bar->dempty[d & 1], (d >> 1) - 1);
                if (*err) break;
                mb_expect(&bar->dfull[d & 1], kStDiag);
                bulk_load(smem_u32(sm + kStOffDiag + (d & 1) * kStDiag), db + (size_t)(2 * k + back) * kStDiag, kStDiag,
                          smem_u32(&bar->dfull[d & 1]));
                const int end = last(k, back);
                for (int seg = first(k, back); seg < end && !*err; seg += sr) {
                    const int rows = min(sr, end - seg);
                    for (int g = 0; g < 32; g += kStCols, ++i) {
                        const int s = i % kStages;
                        if (i >= kStages) wait(&bar->empty[s], i / kStages - 1);
                        if (*err) break;
                        mb_expect(&bar->full[s], (uint32_t)rows * kStCols * 8);
                        for (int c = 0; c < kStCols; ++c)
                            bulk_load(smem_u32(stage + (s * kStCols + c) * sr), a + (size_t)(32 * k + g + c) * n + seg,
                                      (uint32_t)rows * 8, smem_u32(&bar->full[s]));
                    }
                }
            }
            // the last copies land before the CTA's memory is given back
            for (int s = 0; s < kStages; ++s)
                if (i > s) mbar_wait(smem_u32(&bar->full[s]), (uint32_t)((i - 1 - s) / kStages) & 1u);
            for (int s = 0; s < 2; ++s)
                if (d > s) mbar_wait(smem_u32(&bar->dfull[s]), (uint32_t)((d - 1 - s) >> 1) & 1u);
        }
    } else {
        constexpr int RT = RM == 1 ? 1 : RM / 2, NR = RM == 1 ? 1 : 2;      // right-hand sides and rows of a thread
        const int r = RM == 1 ? tid : 2 * (tid & 255), q0 = RM == 1 ? 0 : (tid >> 8) * RT;
        const int2* pt = ptab + (size_t)b * nblk * 64;
        int2 pn0 = make_int2(-1, -1), pn1 = pn0;            // interchanges of the next block
        if (warp < nr) pn0 = pt[lane], pn1 = pt[32 + lane];
        int i = 0, d = 0;
        for (int t = 0; t < 2 * nblk; ++t, ++d) {
            const int back = t >= nblk, k = back ? 2 * nblk - 1 - t : t, j0 = 32 * k;
            if (warp < nr) {
                if (!back) {
                    // this step's interchanges on the warp's right-hand side: slots lane, lane + 32
                    const int2 e0 = pn0, e1 = pn1;
                    if (k + 1 < nblk) pn0 = pt[(k + 1) * 64 + lane], pn1 = pt[(k + 1) * 64 + 32 + lane];
                    const float2 v0 = e0.x >= 0 ? sx[e0.y * RM + warp] : make_float2(0.f, 0.f);
                    const float2 v1 = e1.x >= 0 ? sx[e1.y * RM + warp] : make_float2(0.f, 0.f);
                    __syncwarp();
                    if (e0.x >= 0) sx[e0.x * RM + warp] = v0;
                    if (e1.x >= 0) sx[e1.x * RM + warp] = v1;
                    __syncwarp();
                }
                wait(&bar->dfull[d & 1], d >> 1);
                const float2* D = reinterpret_cast<const float2*>(sm + kStOffDiag + (d & 1) * kStDiag);
                const float2 v = sx[(j0 + lane) * RM + warp];
                float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0;
#pragma unroll
                for (int c = 0; c < 32; c += 2) {
                    const float2 x0 = make_float2(__shfl_sync(0xffffffffu, v.x, c), __shfl_sync(0xffffffffu, v.y, c));
                    const float2 x1 = make_float2(__shfl_sync(0xffffffffu, v.x, c + 1), __shfl_sync(0xffffffffu, v.y, c + 1));
                    acc0 = fma_c(acc0, D[c * 32 + lane], x0);
                    acc1 = fma_c(acc1, D[(c + 1) * 32 + lane], x1);
                }
                sx[(j0 + lane) * RM + warp] = add(acc0, acc1);
            }
            asm volatile("bar.sync 1, 512;" ::: "memory");
            if (tid == 0) mb_arrive(&bar->dempty[d & 1]);
            const int end = last(k, back);
            for (int seg = first(k, back); seg < end; seg += sr) {
                const bool in = r < min(sr, end - seg);
                float2 acc[NR][RT];
                if (in)
#pragma unroll
                    for (int e = 0; e < NR; ++e)
#pragma unroll
                        for (int q = 0; q < RT; ++q) acc[e][q] = sx[(seg + r + e) * RM + q0 + q];
                for (int g = 0; g < 32; g += kStCols, ++i) {
                    const int s = i % kStages;
                    wait(&bar->full[s], i / kStages);
                    if (in) {
                        const float2* F = stage + s * kStCols * sr + r;
                        const float2* xs = sx + (j0 + g) * RM + q0;
#pragma unroll
                        for (int c = 0; c < kStCols; ++c) {
                            float2 f[NR];
                            if constexpr (NR == 2) {
                                const float4 v = *reinterpret_cast<const float4*>(F + c * sr);
                                f[0] = make_float2(v.x, v.y), f[1] = make_float2(v.z, v.w);
                            } else {
                                f[0] = F[c * sr];
                            }
#pragma unroll
                            for (int q = 0; q < RT; ++q) {
                                const float2 xc = xs[c * RM + q];
#pragma unroll
                                for (int e = 0; e < NR; ++e) acc[e][q] = fms(acc[e][q], f[e], xc);
                            }
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mb_arrive(&bar->empty[s]);
                }
                if (in)
#pragma unroll
                    for (int e = 0; e < NR; ++e)
#pragma unroll
                        for (int q = 0; q < RT; ++q) sx[(seg + r + e) * RM + q0 + q] = acc[e][q];
            }
            asm volatile("bar.sync 1, 512;" ::: "memory");
        }
    }
    __syncthreads();
    const bool bad = *err != 0;
    for (int idx = tid; idx < nv * RM; idx += kStThreads) {
        const int i = idx / RM, q = idx - i * RM;
        if (q < nr) x[(size_t)i * nrhs + q] = bad ? make_float2(__int_as_float(0x7fc00000), 0.f) : sx[idx];
    }
}

}  // namespace
}  // namespace pmlbie
