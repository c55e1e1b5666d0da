// mpr_energy.cuh -- sums of bond energies cos[q(phi_i - phi_j)] (Eq. 2) in 64-bit fixed point
// (mpr_fixed.cuh), for the energy of a state and of the measured sample.
//
// What bounds them: integer multiplies. (An FP64 cosine is about 20 instructions of a unit that issues
// 2 per SM and clock.) A warp walks down a strip of columns: each angle is loaded once and becomes a unit
// vector once, a site's bonds are one product of its vector with the sum of its neighbours', which
// come by shuffle or are still in a register from the row above: 229 us at 4096^2 (one cosine per bond,
// of the wrapped difference of the angles, 253 us; FP64 cosines 1625 us). Each term is off by at most
// 2^-55 and is added as a 50-bit fixed-point integer, so a sum does not depend on its order; FP64
// enters once per strip.
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

// A unit vector with 62 fraction bits, and with 60 as a neighbour (four of them add up below 2^63).
struct Vec {
    int64_t c, s;
};
__device__ __forceinline__ Vec unit_of_turn(const fixed::Dir* tab, uint64_t t)
{
    Vec v;
    fixed::sincos_turn(tab, t, &v.c, &v.s);
    return v;
}
__device__ __forceinline__ Vec neighbour(Vec v, bool there)
{
    return Vec{there ? (v.c + 2) >> 2 : 0, there ? (v.s + 2) >> 2 : 0};
}

// u . h (62 and 60 fraction bits) as a 50-bit fixed-point term, rounded to nearest.
__device__ __forceinline__ int64_t term(Vec u, Vec h)
{
    const int64_t e = fixed::mulhi(fixed::split(u.c), fixed::split(h.c)) +
                      fixed::mulhi(fixed::split(u.s), fixed::split(h.s));
    return (e + (1 << 7)) >> 8;
}
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
