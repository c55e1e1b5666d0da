// mpr_resident_bf16.cu -- the resident sweep kernel with BF16 spins.
#include "mpr_resident.cuh"

namespace mpr {
namespace resident {

cudaError_t launch_bf16(const Plan& p, bool measure, int sample, bool qhalf, const Args& a, cudaStream_t st)
{
    return go_store<__nv_bfloat16>(p, measure, sample, qhalf, a, st);
}

}  // namespace resident
}  // namespace mpr
