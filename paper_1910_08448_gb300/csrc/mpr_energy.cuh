// mpr_energy.cuh -- sums of bond energies cos[q(phi_i - phi_j)] (Eq. 2) in 64-bit fixed point
// (mpr_fixed.cuh), for the energy of a state.
//
// What bounds them: instructions, 315 per site at 64 % of the issue slots (4096^2 counters; ALU and the FMA pipe of
// the integer multiplies 59 % each, DRAM 8 %). An FP64 cosine is about 20 instructions of a unit that
// issues 2 per SM and clock. A warp walks down a strip of columns: each angle is loaded once and becomes a unit
// vector once, a site's bonds are one product of its vector with the sum of its neighbours', which
// come by shuffle or are still in a register from the row above: 213 us at 4096^2 (one cosine per bond,
// of the wrapped difference of the angles, 253 us; FP64 cosines 1625 us). A bond is off by at most 2^-55.6 (rms
// 2^-57.5, mean 1.8e-18; q = 0.3, 0.5, 1 against 113 bits) and has 56 fraction bits. Sums are exact and do not depend on their order: 64-bit integers
// within a strip, two of them beyond; the only rounding is that of the result. (With
// terms of 50 bits and sums of rounded FP64 strips the rms error of e_b was 1.1e-16 at 2 x 2, where
// FP64 cosines give 4.5e-17; now 2.4e-17, and below FP64's at every size.)
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

// u . h (62 and 60 fraction bits) with 56 fraction bits: rounded to nearest, and 2 units of 2^-58 added,
// which the two products' truncations lose on average.
__device__ __forceinline__ int64_t term(Vec u, Vec h)
{
    const int64_t e = fixed::mulhi(fixed::split(u.c), fixed::split(h.c)) +
                      fixed::mulhi(fixed::split(u.s), fixed::split(h.s));
    return (e + 4) >> 2;
}

// A bond energy in FP64 (an angle out of range) as a term; *nan is set for NaN.
__device__ __forceinline__ int64_t term_fp64(double x, bool* nan)
{
    *nan |= isnan(x);
    return __double2ll_rn(x * 0x1p56);
}

// A sum of terms, 2^32 and 1 units of 2^-56: exact. (FP64 words would be exact too, but the part adds 2 FP64 numbers
// per SM and clock: 3 us longer at 100 x 70.)
struct Sum {
    long long h;
    unsigned long long l;
    __device__ __forceinline__ void add(int64_t terms)
    {
        h += terms >> 32;
        l += (uint32_t)terms;
    }
    __device__ __forceinline__ void add(const Sum& o)
    {
        h += o.h;
        l += o.l;
    }
    __device__ __forceinline__ void add_lane(int off)   // lane ^ off's
    {
        h += __shfl_xor_sync(0xffffffffu, h, off);
        l += __shfl_xor_sync(0xffffffffu, l, off);
    }
    __device__ __forceinline__ double value() const
    {
        return (double)(h + (long long)(l >> 32)) * 0x1p-24 + (double)(uint32_t)l * 0x1p-56;
    }
};
constexpr unsigned long long kNan = ~0ull;   // in place of l: the sum is NaN (l itself stays below 2^63)

// Signed angles below 7.5 in size; other values (and NaN) are the caller's FP64 case.
__device__ __forceinline__ bool in_range_signed(double x) { return fixed::in_range(fabs(x)); }
__device__ __forceinline__ uint64_t turns_signed(double x, fixed::Split k)
{
    const uint64_t t = fixed::turns(fabs(x), k);
    return __double2hiint(x) < 0 ? 0ull - t : t;
}

// The sum over the block; valid in thread 0.
__device__ __forceinline__ Sum block_sum(Sum v)
{
    __shared__ Sum ws[kWarpsPerBlock];
#pragma unroll
    for (int off = 16; off; off >>= 1) v.add_lane(off);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int i = 1; i < kWarpsPerBlock; ++i) v.add(ws[i]);
    return v;
}

// The block's sum in its place of part; nan: a term of the thread is NaN.
__device__ __forceinline__ void store_sum(Sum v, bool nan, Sum* part)
{
    const bool any = __syncthreads_or(nan);
    v = block_sum(v);
    if (any) v.l = kNan;
    if (threadIdx.x == 0) part[blockIdx.x] = v;
}

// The sum of n blocks by one block; valid in thread 0.
__device__ __forceinline__ double final_sum(const Sum* __restrict__ part, int n)
{
    Sum s{0, 0};
    bool nan = false;
    for (int i = threadIdx.x; i < n; i += kThreads) {
        const Sum p = part[i];
        nan |= p.l == kNan;
        s.add(p);
    }
    const bool any = __syncthreads_or(nan);
    s = block_sum(s);
    return any ? (double)NAN : s.value();
}

}  // namespace energy
}  // namespace mpr
