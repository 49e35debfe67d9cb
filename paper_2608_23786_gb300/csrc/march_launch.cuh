// Launch of the multi-step kernel (stepper_march.cuh) for one element type.
#pragma once
#include "launch.h"
#include "stepper_march.cuh"

namespace mclbm {

template <class E, int VEC, int MODE, bool WRAP>
cudaError_t launch_march_variant(MarchArgs<E>& a, int num_sms, int64_t tiles, cudaStream_t s)
{
    constexpr bool PACK = Storage<E>::shifted && VEC % 2 == 0;
    auto kern = k_march<E, VEC, MODE, PACK, WRAP>;
    // the register split of the kernel would wait forever with fewer registers at launch
    static std::atomic<int> regs_cache{0};
    int regs = regs_cache.load(std::memory_order_relaxed);
    if (regs == 0) {
        cudaFuncAttributes fa;
        const cudaError_t e = cudaFuncGetAttributes(&fa, kern);
        if (e != cudaSuccess) return e;
        regs_cache.store(regs = fa.numRegs, std::memory_order_relaxed);
    }
    if (regs != kMarchRegs) return cudaErrorInvalidConfiguration;
    // one block per SM (its registers fill it); a small ensemble takes a block per tile
    const int64_t grid = num_sms < tiles ? num_sms : tiles;
    void* args[] = {&a};
    return cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)grid), dim3(kMarchThreads), args, 0, s);
}

template <class E, int VEC>
cudaError_t launch_march_vec(MarchArgs<E>& a, int mode, int num_sms, int64_t tiles, cudaStream_t s)
{
    const bool wrap = a.lev.g.N <= 32 * VEC;
    switch (mode) {
        case kMarchAA:
            return wrap ? launch_march_variant<E, VEC, kMarchAA, true>(a, num_sms, tiles, s)
                        : launch_march_variant<E, VEC, kMarchAA, false>(a, num_sms, tiles, s);
        case kMarchSwap:
            return wrap ? launch_march_variant<E, VEC, kMarchSwap, true>(a, num_sms, tiles, s)
                        : launch_march_variant<E, VEC, kMarchSwap, false>(a, num_sms, tiles, s);
        default:
            return wrap ? launch_march_variant<E, VEC, kMarchTrajectory, true>(a, num_sms, tiles, s)
                        : launch_march_variant<E, VEC, kMarchTrajectory, false>(a, num_sms, tiles, s);
    }
}

}  // namespace mclbm
