// Self-test entry of the float-float arithmetic (ffloat.cuh, pairs of FP32 numbers):
// the selectors 20-22 of pmlbie_selftest_elementary.
#include <cmath>

#include "internal.h"
#include "ffloat.cuh"

namespace pmlbie {

namespace {

using namespace ffm;

// ---------------------------------------------------------------------------
// Self-test of the float-float elementary functions (pmlbie_selftest_elementary
// selectors 20-22): exp as mantissa x 2^E, sin / cos, 1/sqrt of the float
// pair nearest to each double, returned as doubles.
// ---------------------------------------------------------------------------
__global__ void ff_elementary_kernel(int fn, const double* x, double* out, size_t n, const float2* exp_tab,
                                     const float4* trig_tab) {
    __shared__ float4 trig[kTrigTab];
    __shared__ float2 expt[kExpTab];
    for (int i = threadIdx.x; i < kTrigTab; i += blockDim.x) trig[i] = trig_tab[i];
    for (int i = threadIdx.x; i < kExpTab; i += blockDim.x) expt[i] = exp_tab[i];
    __syncthreads();
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Tables TT{expt, trig};
    const ff v = from_double(x[i]);
    if (fn == 20) {
        int E;
        const ff m = exp_split(v, TT, E);
        out[i] = to_double(m, E);
    } else if (fn == 21) {
        ff s, c;
        sincos_ff(v, TT, s, c);
        out[2 * i] = to_double(s, 0);
        out[2 * i + 1] = to_double(c, 0);
    } else if (fn == 22) {
        out[i] = to_double(rsqrt(v), 0);
    }
}

}  // namespace

void ff_tables(std::vector<float2>& expv, std::vector<float4>& trig) {
    const double pi = 3.14159265358979323846;
    auto f2 = [](double x) {
        const float hi = (float)x;
        return make_float2(hi, (float)(x - (double)hi));
    };
    auto f4 = [&](double x, double y) {
        const float2 a = f2(x), b = f2(y);
        return make_float4(a.x, a.y, b.x, b.y);
    };
    expv.resize(kExpTab);
    for (int j = 0; j < kExpTab; ++j) expv[j] = f2(std::exp2(j / 64.0));
    trig.resize(kTrigTab);
    for (int k = 0; k < kTrigTab; ++k) trig[k] = f4(std::cos(pi * k / 256.0), std::sin(pi * k / 256.0));
}

bool ff_elementary_known(int fn) { return fn == 20 || fn == 21 || fn == 22; }

cudaError_t launch_ff_elementary(int fn, const double* x, double* out, size_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    std::vector<float4> trig;
    std::vector<float2> ex;
    ff_tables(ex, trig);
    float2* dexp = nullptr;
    float4* dtrig = nullptr;
    cudaError_t e = cudaMalloc(&dexp, sizeof(float2) * ex.size());
    if (e == cudaSuccess) e = cudaMalloc(&dtrig, sizeof(float4) * trig.size());
    if (e == cudaSuccess) e = cudaMemcpyAsync(dexp, ex.data(), sizeof(float2) * ex.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(dtrig, trig.data(), sizeof(float4) * trig.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
        ff_elementary_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(fn, x, out, n, dexp, dtrig);
        count_launch();
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (dexp) cudaFree(dexp);
    if (dtrig) cudaFree(dtrig);
    return e;
}

}  // namespace pmlbie
