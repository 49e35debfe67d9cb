// The multi-step kernel: element type __half (FP32 arithmetic).
#include "march_launch.cuh"

namespace mclbm {

cudaError_t launch_march_f16(MarchArgs<__half>& a, int mode, int num_sms, int64_t tiles, cudaStream_t s)
{
    return launch_march_vec<__half, 4>(a, mode, num_sms, tiles, s);
}

}  // namespace mclbm
