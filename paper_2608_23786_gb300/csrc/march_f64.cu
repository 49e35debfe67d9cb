// The multi-step kernel: element type double, small ensembles (rows within one warp, one node per thread).
#include "march_launch.cuh"

namespace mclbm {

cudaError_t launch_march_f64(MarchArgs<double>& a, int vec, int mode, int num_sms, int64_t tiles, cudaStream_t s)
{
    if (vec != 1 || a.lev.g.N > 32) return cudaErrorInvalidValue;
    return launch_march_mode<double, 1, true>(a, mode, num_sms, tiles, s);
}

}  // namespace mclbm
