// mergepath_f32ck.cu -- keyed cooperative merge-path instantiations (float64 input), F32C precision.
#include "mergepath.cuh"

namespace pcfgb {
cudaError_t launch_mergepath_f32ck(int combo, const WalkArgs& a, int64_t npairs, cudaStream_t s)
{
    return launch_mergepath_t<float, kF32C, true>(combo, a, npairs, s);
}
}  // namespace pcfgb
