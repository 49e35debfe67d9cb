// The multi-step kernel: element type __half (FP32 arithmetic), small ensembles (rows within one warp).
#include "march_launch.cuh"

namespace mclbm {

cudaError_t launch_march_f16(MarchArgs<__half>& a, int vec, int mode, int num_sms, int64_t tiles, cudaStream_t s)
{
    if (a.lev.g.N > 32 * vec) return cudaErrorInvalidValue;
    if constexpr (Q == 19)
        if (vec == 4) return launch_march_mode<__half, 4, true>(a, mode, num_sms, tiles, s);
    return launch_march_mode<__half, 2, true>(a, mode, num_sms, tiles, s);
}

}  // namespace mclbm
