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
    constexpr int smem = march_smem<E, VEC, kMarchSlot<E, VEC, WRAP>>();
    if constexpr (smem > 0) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {&a};
    return cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)grid), dim3(kMarchThreads), args, smem, s);
}

template <class E, int VEC, bool WRAP>
cudaError_t launch_march_mode(MarchArgs<E>& a, int mode, int num_sms, int64_t tiles, cudaStream_t s)
{
    switch (mode) {
        case kMarchAA: return launch_march_variant<E, VEC, kMarchAA, WRAP>(a, num_sms, tiles, s);
        case kMarchSwap: return launch_march_variant<E, VEC, kMarchSwap, WRAP>(a, num_sms, tiles, s);
        default: return launch_march_variant<E, VEC, kMarchTrajectory, WRAP>(a, num_sms, tiles, s);
    }
}

}  // namespace mclbm
