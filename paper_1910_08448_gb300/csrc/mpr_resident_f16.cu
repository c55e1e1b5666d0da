// mpr_resident_f16.cu -- the resident sweep kernel with FP16 spins.
#include "mpr_resident.cuh"

namespace mpr {
namespace resident {

cudaError_t launch_f16(const Plan& p, bool measure, int sample, bool qhalf, const Args& a, cudaStream_t st)
{
    return go_store<__half>(p, measure, sample, qhalf, a, st);
}

}  // namespace resident
}  // namespace mpr
