// The multi-step kernel: element type float.
#include "march_launch.cuh"

namespace mclbm {

cudaError_t launch_march_f32(MarchArgs<float>& a, int mode, int num_sms, int64_t tiles, cudaStream_t s)
{
    return launch_march_vec<float, Q == 19 ? 4 : 2>(a, mode, num_sms, tiles, s);
}

}  // namespace mclbm
