// The multi-step kernel: element type float.
#include "march_launch.cuh"

namespace mclbm {

cudaError_t launch_march_f32(MarchArgs<float>& a, int vec, int mode, int num_sms, int64_t tiles, cudaStream_t s)
{
    if (a.lev.g.N > 32 * vec) return launch_march_mode<float, Q == 19 ? 4 : 2, false>(a, mode, num_sms, tiles, s);
    return vec == 2 ? launch_march_mode<float, 2, true>(a, mode, num_sms, tiles, s)
                    : launch_march_mode<float, 4, true>(a, mode, num_sms, tiles, s);
}

}  // namespace mclbm
