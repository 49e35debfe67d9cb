// The FP64 reciprocal of the collision (collide.cuh) against the correctly rounded quotient 1.0 / d.
#include <cuda_runtime.h>

#include <cstdint>

#include "../paper_2608_23786_gb300/csrc/collide.cuh"

namespace {

__device__ uint64_t mix(uint64_t x)  // SplitMix64
{
    x += 0x9e3779b97f4a7c15ull;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
    return x ^ (x >> 31);
}

// Of n values with exponents lo .. hi - 1, all mantissas and both signs: out[0] the largest distance to
// 1.0 / d in units in the last place, out[1] how many are not equal to it.
__global__ void k_check(uint64_t n, uint64_t seed, int lo, int hi, unsigned long long* out)
{
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint64_t r = mix(seed + i), x = 1023 + lo + mix(~r) % (uint64_t)(hi - lo);
        const double d = __longlong_as_double((long long)((r & 0x800fffffffffffffull) | x << 52));
        const long long a = __double_as_longlong(mclbm::rcp64(d)), b = __double_as_longlong(__drcp_rn(d));
        const unsigned long long ulps = a > b ? a - b : b - a;
        if (ulps != 0) {
            atomicMax(out, ulps);
            atomicAdd(out + 1, 1ull);
        }
    }
}

}  // namespace

extern "C" int rcp64_check(uint64_t n, uint64_t seed, int lo, int hi, void* d_out)
{
    k_check<<<152 * 8, 256>>>(n, seed, lo, hi, (unsigned long long*)d_out);
    const cudaError_t e = cudaGetLastError();
    return (int)(e == cudaSuccess ? cudaDeviceSynchronize() : e);
}
