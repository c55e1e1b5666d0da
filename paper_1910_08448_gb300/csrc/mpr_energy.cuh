// mpr_energy.cuh -- sums of bond energies cos[q(phi_i - phi_j)] (Eq. 2) in 64-bit fixed point
// (mpr_fixed.cuh), for the energy of a state and of the measured sample.
//
// What bounds them: an FP64 cosine is about 20 instructions of a unit that issues 2 per SM and
// clock. Here an angle becomes a fraction of a turn once (about 18 integer instructions), a bond
// is the cosine of a wrapped difference (about 55), and a warp walks down a strip of columns so
// that each angle is loaded and converted once: the right neighbour comes by a shuffle, the row
// above is still in a register. Each cosine is off by at most 2^-56 and is added as a 50-bit
// fixed-point integer, so a sum does not depend on its order; FP64 enters once per strip.
#pragma once

#include "mpr_device.cuh"
#include "mpr_fixed.cuh"

namespace mpr {
namespace energy {

static __device__ const fixed::DirTable g_dirs = fixed::make_dirs();

constexpr int kThreads = 256;
constexpr int kWarpsPerBlock = kThreads / 32;
constexpr int kMaxRows = 16;   // rows a warp walks in one strip

// Rows of a strip: tall ones convert fewer rows twice, low ones give more warps a strip of a small
// grid (about 152 x 32 warps fill the device).
inline int strip_rows(long long strips, int Ly)
{
    const long long r = strips * Ly / (152 * 32);
    return r < 2 ? 2 : r > kMaxRows ? kMaxRows : (int)r;
}

// A bond's cosine (62 fraction bits) as a 50-bit fixed-point term, rounded to nearest.
__device__ __forceinline__ int64_t term(int64_t c) { return (c + (1 << 11)) >> 12; }
constexpr double kTermUnit = 0x1p-50;

// Signed angles below 7.5 in size; other values (and NaN) are the caller's FP64 case.
__device__ __forceinline__ bool in_range_signed(double x) { return fixed::in_range(fabs(x)); }
__device__ __forceinline__ uint64_t turns_signed(double x, fixed::Split k)
{
    const uint64_t t = fixed::turns(fabs(x), k);
    return __double2hiint(x) < 0 ? 0ull - t : t;
}

// Sum over the block of one value per thread, in a fixed order; valid in thread 0.
__device__ __forceinline__ double block_sum(double v)
{
    __shared__ double ws[kWarpsPerBlock];
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < kWarpsPerBlock; ++i) s += ws[i];
    return s;
}

}  // namespace energy
}  // namespace mpr
