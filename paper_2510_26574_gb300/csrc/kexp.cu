// Table of the engine's exponential (kexp.cuh) and its C-ABI test entry.
#include <cmath>

#include "common.cuh"
#include "kexp.cuh"

namespace kevd {

static __device__ unsigned long long g_exp2_q62[1024];

cudaError_t kexp_table(cudaStream_t s, const unsigned long long** tbl) {
    static unsigned long long host[1024];
    static bool filled = false;
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    void* addr = nullptr;
    if ((e = cudaGetSymbolAddress(&addr, g_exp2_q62)) != cudaSuccess) return e;
    *tbl = static_cast<const unsigned long long*>(addr);
    if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
    if (!filled) {
        for (int j = 0; j < 1024; ++j)
            host[j] = (unsigned long long)llroundl(ldexpl(exp2l((long double)j / 1024.0L), 62));
        filled = true;
    }
    e = cudaMemcpyToSymbolAsync(g_exp2_q62, host, sizeof(host), 0, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
    return e;
}

// (t > 0 lies outside the engine's use: CUDA's exp; NaN gives 0.)
__global__ void k_kexp(const double* __restrict__ t, int64_t n, KexpScale one, const unsigned long long* __restrict__ tbl,
                       double* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = t[i];
    out[i] = x > 0.0 ? exp(x) : x <= 0.0 ? __longlong_as_double((long long)kexp_bits(-x, one, tbl)) : 0.0;
}

}  // namespace kevd

using namespace kevd;

extern "C" int kevd_kernel_exp(const double* t, int64_t n, double* out, void* stream) {
    if (!t || !out || n < 0 || n >= ((int64_t)1 << 38)) return KEVD_EINVAL;
    if (n == 0) return KEVD_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const unsigned long long* tbl = nullptr;
    if (kexp_table(s, &tbl) != cudaSuccess) return KEVD_ECUDA;
    k_kexp<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(t, n, kexp_scale(1.0), tbl, out);
    return cudaGetLastError() == cudaSuccess ? KEVD_OK : KEVD_ECUDA;
}
