// mpr_fixed.cuh -- sine, cosine and angles to better than FP64 accuracy in 64-bit fixed point.
//
// Why integers: this part issues 2 FP64 instructions per SM and clock against 64 32-bit integer
// multiplies and 128 other instructions, so an FP64 sincos (about 35 FP64 instructions) costs as
// much as 2000 integer ones. The angles of the method lie in a fixed range and its unit vectors
// in [-1, 1], where fixed point needs no exponents: one sincos below is about 85 integer
// instructions. Measured on the FP64-function sweeps and the FP64 energies, see mpr_sweep.cu and
// mpr_energy.cuh.
//
// Angles are fractions of a turn in an unsigned 64-bit word (2^64 = 2 pi), so sums and
// differences wrap by themselves. sin and cos come from a table of 1024 directions and the Taylor
// series of the rest (|r| <= pi / 1024, where r^6/720 is 2^-60): (c, s) of the table entry is
// rotated by r. Every product keeps the upper 64 bits of a 64 x 64 bit product up to 2.3 units
// in the last place. The error of sin and cos is below 2^-58 for a given turn, that of a turn
// below 2^-57 rad; an FP64 value near 1 is spaced by 2^-53.
//
// Host and device run the same integer code, so the CPU can check it.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#define MPR_HD __host__ __device__ __forceinline__
#else
#define MPR_HD inline
#endif

namespace mpr {
namespace fixed {

constexpr int kDirs = 1024;   // directions of the table

struct alignas(16) Dir {
    long long c, s;           // 2^62 cos, 2^62 sin
};

struct DirTable {
    Dir d[kDirs];
};

// Unsigned fixed point with 100 fraction bits, for the table only (values below 8).
constexpr unsigned __int128 mul100(unsigned __int128 a, unsigned __int128 b)
{
    const unsigned __int128 m = ~0ull;
    const unsigned __int128 al = a & m, ah = a >> 64, bl = b & m, bh = b >> 64;
    return ((ah * bh) << 28) + ((al * bh + ah * bl + ((al * bl) >> 64)) >> 36);
}

// sin and cos of the angle x (100 fraction bits, 0 <= x <= pi / 4) by their Taylor series,
// rounded to 62 fraction bits.
constexpr Dir dir_octant(unsigned __int128 x)
{
    unsigned __int128 c = (unsigned __int128)1 << 100, s = x, t = x;   // t = x^n / n!
    const unsigned __int128 x2 = mul100(x, x);
    unsigned __int128 tc = c;
    for (int n = 1; n < 16; ++n) {
        tc = mul100(tc, x2) / (unsigned)((2 * n - 1) * (2 * n));
        t = mul100(t, x2) / (unsigned)((2 * n) * (2 * n + 1));
        if (n & 1) {
            c -= tc;
            s -= t;
        } else {
            c += tc;
            s += t;
        }
    }
    const unsigned __int128 half = (unsigned __int128)1 << 37;
    return Dir{(long long)((c + half) >> 38), (long long)((s + half) >> 38)};
}

constexpr DirTable make_dirs()
{
    DirTable t{};
    // pi = 3.243F6A8885A308D313198A2E03707344... (hexadecimal), here with 100 fraction bits
    const unsigned __int128 pi =
        ((unsigned __int128)0x3243F6A888ull << 64 | 0x5A308D313198A2E0ull);
    for (int k = 0; k <= kDirs / 8; ++k) {
        const Dir o = dir_octant(pi * (unsigned)k / (unsigned)(kDirs / 2));
        // the eight reflections of the first octant
        const int q = kDirs / 4;
        t.d[k] = o;
        t.d[q - k] = Dir{o.s, o.c};
        t.d[q + k] = Dir{-o.s, o.c};
        t.d[2 * q - k] = Dir{-o.c, o.s};
        t.d[2 * q + k] = Dir{-o.c, -o.s};
        t.d[3 * q - k] = Dir{-o.s, -o.c};
        t.d[3 * q + k] = Dir{o.s, -o.c};
        if (k > 0) t.d[4 * q - k] = Dir{o.c, -o.s};
    }
    return t;
}

// ---- products -----------------------------------------------------------------------------------

// a = h * 2^32 + l with l signed, so every partial product is a signed 32 x 32 bit one.
struct Split {
    int32_t h, l;
};

MPR_HD constexpr Split split(int64_t a)
{
    // h rounded to nearest (unsigned: angles out of range pass here too, their result is not used)
    return Split{(int32_t)((uint32_t)(a >> 32) + ((uint32_t)a >> 31)), (int32_t)(uint32_t)a};
}

MPR_HD int32_t mulhi32(int32_t a, int32_t b) { return (int32_t)(((int64_t)a * b) >> 32); }
MPR_HD uint32_t umulhi32(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }

// floor(a * b / 2^64) up to 2.3 units (the low product is left out); |a.h| + |b.h| < 2^32
MPR_HD int64_t mulhi(Split a, Split b)
{
    const int32_t m = mulhi32(a.h, b.l) + mulhi32(a.l, b.h);
    return (int64_t)a.h * b.h + m;
}

MPR_HD uint64_t umulhi(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

// ---- sine and cosine ----------------------------------------------------------------------------

struct Small {
    Split cm1;   // cos r - 1, 74 fraction bits
    Split sn;    // sin r, 69 fraction bits
};

// cos r - 1 and sin r for r = rt * 2 pi / 2^64, |rt| <= 2^53.
MPR_HD Small small_angle(int64_t rt)
{
    constexpr int64_t kPi4 = 7244019458077122842ll;   // pi / 4 * 2^63
    const int64_t R = mulhi(split((int64_t)((uint64_t)rt << 9)), split(kPi4));   // r, 69 bits
    const Split r = split(R);
    const int64_t R2 = mulhi(r, r);                       // r^2, 74 bits
    const uint32_t r2 = (uint32_t)((uint64_t)R2 >> 26);   // r^2 < 2^-16.6, 48 bits
    // cos r - 1 = -r^2/2 + r^2 (r^2 (1/24 - r^2/720))
    const uint32_t a = 178956971u - umulhi32(r2, 91u);                     // 32 bits
    const uint32_t b = (uint32_t)(((uint64_t)r2 * a) >> 28);               // 52 bits
    const int64_t cm1 = (int64_t)(((uint64_t)r2 * b) >> 26) - (R2 >> 1);   // 74 bits
    // sin r = r - r (r^2 (1/6 - r^2/120))
    const uint32_t d = 2863311531u - umulhi32(r2, 2185u);                  // 34 bits
    const int32_t f = (int32_t)(((uint64_t)r2 * d + 0x80000000ull) >> 32); // 50 bits
    const int32_t r39 = (int32_t)((R + (1ll << 29)) >> 30);                // r, 39 bits
    const int64_t sn = R - (((int64_t)r39 * f) >> 20);
    return Small{split(cm1), split(sn)};
}

// (cos, sin) of t turns with 62 fraction bits.
MPR_HD void sincos_turn(const Dir* tab, uint64_t t, int64_t* c, int64_t* s)
{
    const uint32_t k = (uint32_t)((t + (1ull << 53)) >> 54) & (kDirs - 1);
    const int64_t rt = (int64_t)(t - ((uint64_t)k << 54));
    const Dir d = tab[k];
    const Small m = small_angle(rt);
    const Split C = split(d.c), S = split(d.s);
    *c = d.c + (((mulhi(C, m.cm1) >> 5) - mulhi(S, m.sn)) >> 5);
    *s = d.s + (((mulhi(S, m.cm1) >> 5) + mulhi(C, m.sn)) >> 5);
}

// ---- angles to turns ----------------------------------------------------------------------------

// q / (2 pi) with 65 fraction bits: turns of q * phi per radian of phi (q <= 1).
inline int64_t turn_factor(double q)
{
    // 2^65 / (2 pi) = 2^64 / pi as an integer and the rest, times q without rounding
    const unsigned __int128 k = ((unsigned __int128)5871781006564002452ull << 32) |
                                0xFE13ABE8u;   // 2^96 / pi, rounded down
    int e = 0;
    uint64_t m = 0;
    if (q > 0.0) {
        uint64_t u;
        memcpy(&u, &q, 8);
        e = (int)(u >> 52) - 1075;
        m = (u & 0xFFFFFFFFFFFFFull) | (1ull << 52);   // q = m * 2^e
    }
    // (k * m) >> (32 - e), k below 2^95 and m below 2^53: in two halves
    const unsigned __int128 lo = (k & 0xFFFFFFFFFFFFull) * m, hi = (k >> 48) * m;
    const unsigned __int128 p = hi + (lo >> 48);       // (k m) >> 48
    const int sh = 32 - e - 48;                        // e <= -52: sh >= 36
    return sh > 126 ? 0 : (int64_t)((p + ((unsigned __int128)1 << (sh - 1))) >> sh);
}

// An angle is in range when 0 <= x < 7.5 (never for NaN).
MPR_HD bool in_range(double x)
{
    uint64_t u;
    memcpy(&u, &x, 8);
    return (uint32_t)(u >> 32) < 0x401E0000u;
}
MPR_HD bool in_range(float x)
{
    uint32_t u;
    memcpy(&u, &x, 4);
    return u < 0x40F00000u;
}

// x with 60 fraction bits, rounded down (subnormals as 0); x in range.
MPR_HD int64_t q60(double x)
{
    uint64_t u;
    memcpy(&u, &x, 8);
    const int e = (int)(u >> 52);
    const uint64_t m = ((u << 10) | (1ull << 62)) & 0x7FFFFFFFFFFFFFFFull;   // 1.m, 62 bits below
    const uint32_t sh = (uint32_t)(1025 - e);   // out of range: any value
    return (int64_t)(m >> (sh > 63u ? 63u : sh));
}
MPR_HD int64_t q60(float x)
{
    uint32_t u;
    memcpy(&u, &x, 4);
    const int e = (int)(u >> 23);
    const uint64_t m = (uint64_t)((u & 0x007FFFFFu) | 0x00800000u) << 39;
    const uint32_t sh = (uint32_t)(129 - e);
    return (int64_t)(m >> (sh > 63u ? 63u : sh));
}

// Turns of q * x, x in range; k = split(turn_factor(q)).
template <typename F> MPR_HD uint64_t turns(F x, Split k)
{
    return (uint64_t)mulhi(split(q60(x)), k) << 3;
}

// v / 2^60 rounded to the nearest FP64 value (ties to even), 0 <= v < 2^63.
MPR_HD double to_double_q60(uint64_t v)
{
    if (v == 0) return 0.0;
#ifdef __CUDA_ARCH__
    const int z = __clzll((long long)v);
#else
    const int z = __builtin_clzll(v);
#endif
    const uint64_t n = v << z;                       // leading one at bit 63
    uint64_t m = n >> 11;                            // 53 bits
    const uint64_t rest = n & 0x7FFull;
    m += (rest > 0x400ull || (rest == 0x400ull && (m & 1))) ? 1 : 0;
    // m carries the implicit bit: adding it to the exponent field minus one places both (and a
    // mantissa that rounds up to 2^53 moves to the next exponent)
    const uint64_t u = ((uint64_t)(1023 + 3 - z - 1) << 52) + m;
    double r;
    memcpy(&r, &u, 8);
    return r;
}

// Twice the argument of (hx, hy) in turns, given t0 = that argument modulo pi as a fraction of a
// turn with 32 bits. hx, hy with 60 fraction bits, at most 4 in size and at least 2^-10 in one
// component. t0 comes from fields cut to 28 fraction bits and an FP32 arc tangent: off by 1.5e-6 rad, and by
// 2^-27.5 / |h| more in small fields (5.4e-6 rad at 2^-10). The vector is turned back by t0; what is left of
// it is num / den = tan of the rest, whose cube (2^-58 at |h| = 1, 2^-52 at 2^-10) lies below what the field's
// own last bits do to the angle there (2^-58 / |h|). The quotient is an FP32 pair: 46 bits of the rest.
MPR_HD uint64_t doubled_arg(const Dir* tab, int64_t hx, int64_t hy, int32_t t0)
{
    int64_t c0, s0;
    sincos_turn(tab, (uint64_t)(uint32_t)t0 << 32, &c0, &s0);
    const Split X = split(hx), Y = split(hy), C = split(c0), S = split(s0);
    const int64_t num = mulhi(Y, C) - mulhi(X, S);   // 58 fraction bits, below 2^42
    const int64_t den = mulhi(X, C) + mulhi(Y, S);   // 58 fraction bits, up to 2^60
    // den = dh + dl exactly but for its last 13 bits: 24 bits and a sign each (|den| may pass 2^60)
    const float dh = (float)(int32_t)((den + (1ll << 36)) >> 37) * 0x1p37f;
    const float dl = (float)(int32_t)((int64_t)((uint64_t)den << 27) >> 40) * 0x1p13f;
    const float nh = (float)(int32_t)(num >> 20) * 0x1p20f;
    const float nl = (float)(int32_t)((uint32_t)num & 0xFFFFFu);
#ifdef __CUDA_ARCH__
    float rcp;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rcp) : "f"(dh + dl));
#else
    const float rcp = 1.0f / (dh + dl);
#endif
    const float q0 = (nh + nl) * rcp;
    const float q1 = (fmaf(-q0, dh, nh) + fmaf(-q0, dl, nl)) * rcp;
    // (q0 + q1) * 2^64 / pi as an integer: the factor as an FP32 pair
    constexpr float kH = 0x1.45f306p+62f, kL = 0x1.b9391p+37f;
    const float p = q0 * kH;
    const float e = fmaf(q0, kH, -p) + fmaf(q0, kL, q1 * kH);
#ifdef __CUDA_ARCH__
    const int32_t ih = __float2int_rn(p * 0x1p-20f);
    const int32_t il = __float2int_rn(fmaf((float)ih, -0x1p20f, p) + e);
#else
    const int32_t ih = (int32_t)lrintf(p * 0x1p-20f);
    const int32_t il = (int32_t)lrintf(fmaf((float)ih, -0x1p20f, p) + e);
#endif
    return ((uint64_t)(uint32_t)t0 << 33) + (uint64_t)(((int64_t)ih << 20) + il);
}

#ifdef __CUDACC__
// The directions in shared memory, copied by all of a block's `n` threads (the caller's next
// barrier makes them visible): random reads of 16 bytes cost fewer cycles there than in L1.
__device__ __forceinline__ void load_dirs(const DirTable* src, Dir* dst, int tid, int n)
{
    const ulonglong2* s = reinterpret_cast<const ulonglong2*>(src->d);
    ulonglong2* d = reinterpret_cast<ulonglong2*>(dst);
    for (int i = tid; i < kDirs; i += n) d[i] = __ldg(s + i);
}
#endif

}  // namespace fixed
}  // namespace mpr
