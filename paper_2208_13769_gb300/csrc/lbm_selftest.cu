// lbm_selftest.cu -- self-tests on the device.
//
// The give-up path of the bounded mbarrier wait that guards every bulk-copy
// slot of the interior kernel, without faulting or hanging anything: a barrier
// that expects two arrivals gets one, so its phase never completes, and the
// wait must return after its poll limit with the CTA (and the context) intact.
//
// The FP64 reciprocal and quotients of the kernels (rcp_j, over): the
// reciprocal's error by its residual 1 - x r, which one FMA gives to 53 bits, the
// quotients against the bits of CUDA's division.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "lbm.h"
#include "lbm_device.cuh"
#include "lbm_pipeline.cuh"

namespace {

__global__ void bounded_wait_kernel(uint32_t limit, int32_t* result) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        lbm::mbar_init(&bar, 2);
        lbm::fence_mbar_init();
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(lbm::smem_addr(&bar)) : "memory");
        // one arrival of two: phase 0 stays open; no copy is in flight, so
        // the CTA may leave with the barrier incomplete
        result[0] = lbm::mbar_wait_n(&bar, 0u, limit) ? 0 : 1;
    }
}

// the k-th pseudo-random 64-bit word of a seed (splitmix64)
__device__ uint64_t word(uint64_t seed, uint64_t k) {
    uint64_t z = seed + (k + 1) * 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// a number of random sign and mantissa, of exponent lo .. hi
__device__ double number(uint64_t w, uint64_t e, int lo, int hi) {
    const uint64_t ex = uint64_t(lo + int(e % uint64_t(hi - lo + 1)) + 1023);
    return __longlong_as_double((long long)((w & 0x800fffffffffffffull) | ex << 52));
}

// out[0]: the bits of the reciprocal's largest error in units in the last
// place; out[1]: quotients whose bits differ from the division's
__global__ void quotients_kernel(int64_t count, uint64_t seed, unsigned long long* out) {
    double worst = 0.0;
    unsigned long long differ = 0;
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < count; k += int64_t(gridDim.x) * blockDim.x) {
        const uint64_t w = word(seed, uint64_t(4 * k)), v = word(seed, uint64_t(4 * k + 1)),
                       e = word(seed, uint64_t(4 * k + 2)), f = word(seed, uint64_t(4 * k + 3));
        // J near 1 in one half, of any size in the other
        const double x = (e >> 32) & 1 ? fabs(number(w, e, -1, 0)) : number(w, e, -500, 500);
        const double r = lbm::rcp_j(x);
        const double m = __longlong_as_double((__double_as_longlong(r) & 0xfffffffffffffll) | 0x3ff0000000000000ll);
        worst = fmax(worst, fabs(fma(-x, r, 1.0)) * m * 4503599627370496.0);
        // numerators and denominators of every kind and size
        double a = number(v, f, -1023, 1024), j = (f >> 32) & 1 ? x : number(w, e, -1023, 1024);
        if (((f >> 33) & 15) == 0) a = 0.0 * (a > 0.0 ? 1.0 : -1.0);
        if (((f >> 37) & 63) == 0) j = 0.0;
        const double q = lbm::over(a, j, 1.0 / j), p = a / j;
        const bool same = __double_as_longlong(q) == __double_as_longlong(p) || (isnan(q) && isnan(p));
        differ += !same;
    }
    atomicMax(out, (unsigned long long)__double_as_longlong(worst));
    if (differ) atomicAdd(out + 1, differ);
}

}  // namespace

extern "C" lbm_status lbm_selftest_quotients(int64_t count, uint64_t seed, void* cuda_stream, double out[2]) {
    if (!out || count < 1 || count > (int64_t(1) << 30)) return LBM_E_INVALID;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    unsigned long long* d = nullptr;
    if (cudaMalloc(&d, 2 * sizeof(*d)) != cudaSuccess) {
        cudaGetLastError();
        return LBM_E_OOM;
    }
    cudaError_t e = cudaMemsetAsync(d, 0, 2 * sizeof(*d), s);
    if (e == cudaSuccess) {
        const int64_t blocks = (count + 255) / 256;
        quotients_kernel<<<unsigned(blocks < 4096 ? blocks : 4096), 256, 0, s>>>(count, seed, d);
        e = cudaGetLastError();
    }
    unsigned long long h[2] = {0, 0};
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(d);
    if (e != cudaSuccess) return LBM_E_CUDA;
    memcpy(&out[0], &h[0], sizeof(double));
    out[1] = double(h[1]);
    return LBM_OK;
}

extern "C" lbm_status lbm_selftest_bounded_wait(uint32_t polls, void* cuda_stream, int32_t* timed_out) {
    if (!timed_out || polls == 0 || polls > (1u << 22)) return LBM_E_INVALID;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    int32_t* d = nullptr;
    if (cudaMalloc(&d, sizeof(int32_t)) != cudaSuccess) {
        cudaGetLastError();
        return LBM_E_OOM;
    }
    cudaError_t e = cudaMemsetAsync(d, 0xff, sizeof(int32_t), s);
    if (e == cudaSuccess) {
        bounded_wait_kernel<<<1, 32, 0, s>>>(polls, d);
        e = cudaGetLastError();
    }
    int32_t h = -1;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(d);
    if (e != cudaSuccess) return LBM_E_CUDA;
    *timed_out = h;
    return LBM_OK;
}
