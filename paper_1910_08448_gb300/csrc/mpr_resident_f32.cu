// mpr_resident_f32.cu -- the resident sweep kernel with FP32 spins.
#include "mpr_resident.cuh"

namespace mpr {
namespace resident {

cudaError_t launch_f32(const Plan& p, bool measure, int sample, bool qhalf, const Args& a, cudaStream_t st)
{
    return go_store<float>(p, measure, sample, qhalf, a, st);
}

cudaError_t launch_stalled(const Plan& p, const Args& a, cudaStream_t st)
{
    return go_shape<float, false, 0, 2, true>(p, a, st);
}

}  // namespace resident
}  // namespace mpr
