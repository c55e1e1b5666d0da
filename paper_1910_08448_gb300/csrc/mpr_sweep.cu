// mpr_sweep.cu -- one colour half-sweep of the conditional hybrid Monte Carlo (Sec. 2) with FP64
// functions (X_F = D): for every prediction site of the colour, one Metropolis move with a uniform
// proposal followed by one energy-conserving over-relaxation move under Eq. 2; measured sites stay
// frozen. Fused into the same pass: the accumulation of the sampled angles (Sec. 2: averaging over
// configurations in equilibrium) and, on the black pass, the bond-energy partial sums (Sec. 2:
// e = <H>/L^2).
//
// Precision axes (Sec. 2): S = spin storage (X_S, plus FP16/BF16), E = energy accumulation (X_E).
//
// What bounds it: in FP64 arithmetic a site takes about 217 FP64 instructions (three sincos, exp,
// atan2, two divisions), and the part issues 2 of them per SM and clock: 2889 us per 4096^2 pass
// at 1.5 % of the memory rate, whatever else the kernel does. So the pass uses the FP64 unit only
// where a result needs it:
//   - unit vectors, local fields and the doubled field angle are 64-bit fixed point (mpr_fixed.cuh),
//     with smaller errors than the FP64 functions;
//   - the Metropolis test is decided from FP32 estimates whose error is bounded; a site inside the
//     bound (about 1 in 10^4) is decided by the FP64 expression;
//   - a local field below 2^-10, and a tile with an angle outside [0, 7.5) (a state set by the
//     caller), take the FP64 functions throughout.
// 4096^2, p = 0.9: 2889 -> 266 us per pass, 860 instructions per site at 68 % of the issue slots; the ALU
// (55 %) and the FMA pipe of the integer multiplies (53 %) come next. The rms error of a moved angle
// against extended precision falls from 3.6e-16 ... 8.1e-16 to 1.5e-16 ... 2.4e-16 (q 0.3 ... 1).
#include "mpr_device.cuh"
#include "mpr_fixed.cuh"
#include "mpr_internal.h"
#include "mpr_tile_f32.cuh"   // atan2_doubled

#include <type_traits>

namespace mpr {
namespace {

constexpr int kCols = 64;    // half-lattice columns per tile: 32 lanes x one site pair
constexpr int kRowWarps = 8; // 256 threads; each warp owns R rows of the tile
constexpr int kRows = 2;
constexpr int kTY = kRowWarps * kRows;
constexpr int kSW = kCols + 2;

__device__ const fixed::DirTable g_dirs = fixed::make_dirs();

// What the fixed-point path needs of q, formed once per launch.
struct FixedQ {
    int64_t k65;      // turns of q * phi per radian, 65 fraction bits
    uint64_t q64;     // q = the accepted range of the reflected angle in turns, 64 fraction bits
    uint64_t m64;     // pi / 8 / (q * 2^sh), 64 fraction bits: turns of q * phi -> phi / 16
    int sh;           // q * 2^sh in [1/2, 1); -1 for q = 1
};

FixedQ fixed_q(double q)
{
    FixedQ f;
    f.k65 = fixed::turn_factor(q);
    uint64_t u;
    memcpy(&u, &q, 8);
    const int e = (int)(u >> 52) - 1022;                      // q = m 2^-53 2^e
    const uint64_t m = (u & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    f.sh = -e;
    f.q64 = e >= 1 ? ~0ull : (e > -53 ? (m << 11) >> -e : 0ull);
    // pi * 2^114 / m
    const unsigned __int128 pi =
        ((unsigned __int128)0xC90FDAA22168Cull << 64) | 0x234C4C6628B80DC1ull;
    f.m64 = (uint64_t)(pi / m);
    return f;
}

// representative of psi modulo 2*pi in [0, 2*pi), as the method states it
__device__ __forceinline__ double wrap_rep(double psi) { return psi - kTwoPi * floor(psi / kTwoPi); }

// A staged entry of the other colour: (cos, sin) of q * phi, with 60 fraction bits or in FP64.
union Unit {
    longlong2 i;
    double2 d;
};

// Metropolis: accept if dE <= 0 or u < exp(-dE/T), in FP64.
__device__ __noinline__ bool accept_fp64(double hx, double hy, double f, double fp, double q,
                                         double T, double u)
{
    double s0, c0, sp, cp;
    sincos(q * f, &s0, &c0);
    sincos(q * fp, &sp, &cp);
    const double dE = (-(hx * cp + hy * sp)) - (-(hx * c0 + hy * s0));
    return dE <= 0.0 || u < exp(-dE / T);
}

// Over-relaxation in FP64: reflect q*phi about arg(h); keep it if it lands in [0, 2*pi*q].
__device__ __noinline__ double relax_fp64(double hx, double hy, double f1, double q)
{
    if (hx == 0.0 && hy == 0.0) return f1;
    const double r = wrap_rep(2.0 * atan2(hy, hx) - q * f1);
    return r <= kTwoPi * q ? r / q : f1;
}

// The local field of site (column j, row y, offset o) from the stored neighbours, in FP64.
template <typename S>
__device__ __noinline__ double2 field_fp64(const SweepArgs& a, int y, int j, int o)
{
    const S* __restrict__ other = static_cast<const S*>(a.other);
    const int x = 2 * j + o;
    const size_t idx = (size_t)y * a.pitch + j;
    double c[4] = {0.0, 0.0, 0.0, 0.0}, s[4] = {0.0, 0.0, 0.0, 0.0};
    if (x > 0) sincos(a.q * load_as<double>(other[idx + o - 1]), &s[0], &c[0]);
    if (x + 1 < a.Lx) sincos(a.q * load_as<double>(other[idx + o]), &s[1], &c[1]);
    if (y > 0) sincos(a.q * load_as<double>(other[idx - a.pitch]), &s[2], &c[2]);
    if (y + 1 < a.Ly) sincos(a.q * load_as<double>(other[idx + a.pitch]), &s[3], &c[3]);
    return make_double2(((c[0] + c[1]) + c[2]) + c[3], ((s[0] + s[1]) + s[2]) + s[3]);
}

// Adds a sampled angle (as stored) to its accumulator.
__device__ __forceinline__ void add_sample(const SweepArgs& a, size_t idx, double f)
{
    if (a.acc) {
        a.acc[idx] += f;
    } else {
        // Kahan: hi carries the sum, lo the (negated) lost low-order part
        const float v = (float)f;
        const float hi = a.acc_hi[idx], lo = a.acc_lo[idx];
        const float yv = v - lo;
        const float tt = hi + yv;
        a.acc_lo[idx] = (tt - hi) - yv;
        a.acc_hi[idx] = tt;
    }
}

// The block's rows in FP64 functions throughout (an angle of the tile is out of range).
template <typename S, typename E>
__device__ __noinline__ void rows_fp64(const SweepArgs& a, int j0, int y0, Unit (*nb)[kSW], E* e_out,
                                       int* n_out)
{
    const int c = a.colour, cb = c ^ 1;
    const S* __restrict__ other = static_cast<const S*>(a.other);
    S* __restrict__ own = static_cast<S*>(a.own);
    const double q = a.q;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    for (int e = tid; e < (kTY + 2) * kSW; e += 256) {
        const int r = e / kSW, cc = e - r * kSW;
        const int y = y0 - 1 + r, j = j0 - 1 + cc;
        Unit v;
        v.d = make_double2(0.0, 0.0);
        if (y >= 0 && y < a.Ly && j >= 0 && 2 * j + ((y + cb) & 1) < a.Lx)
            sincos(q * load_as<double>(other[(size_t)y * a.pitch + j]), &v.d.y, &v.d.x);
        nb[r][cc] = v;
    }
    __syncthreads();
    const bool measure = (a.flags & kMeasure) && c == 1;
    const bool sample = (a.flags & kSample) != 0;
    const bool bounded = a.width != nullptr;
    const double pw = bounded ? *a.width : 0.0;
    int n_acc = 0;
    E eacc = (E)0;
    for (int rr = 0; rr < kRows; ++rr) {
        const int ly = threadIdx.y * kRows + rr;
        const int y = y0 + ly;
        if (y >= a.Ly) break;
        const int jp = j0 + 2 * threadIdx.x;
        const int o = (y + c) & 1;
        const uint32_t mw = a.mbits[(size_t)y * a.mpitch + (jp >> 5)];
        for (int t = 0; t < 2; ++t) {
            const int j = jp + t, lj = j - j0;
            if (2 * j + o >= a.Lx) continue;
            const double2 lf = nb[ly + 1][lj + o].d, rt = nb[ly + 1][lj + o + 1].d;
            const double2 up = nb[ly][lj + 1].d, dn = nb[ly + 2][lj + 1].d;
            const double hx = ((lf.x + rt.x) + up.x) + dn.x;
            const double hy = ((lf.y + rt.y) + up.y) + dn.y;
            const size_t idx = (size_t)y * a.pitch + j;
            double f = load_as<double>(own[idx]);
            if (!((mw >> (j & 31)) & 1u)) {
                const uint4 w = pair_words((uint32_t)(jp >> 1), (uint32_t)y, a.sweep, a.problem,
                                           kTagMetropolis, (uint32_t)c, a.seed_lo, a.seed_hi);
                const double u_prop = uniform_d(t ? w.z : w.x), u_acc = uniform_d(t ? w.w : w.y);
                const double fp = bounded ? f + pw * (2.0 * u_prop - 1.0) : kTwoPi * u_prop;
                const bool inside = !bounded || (fp >= 0.0 && fp < kTwoPi);
                const bool accept = accept_fp64(hx, hy, f, fp, q, a.T, u_acc) && inside;
                n_acc += accept ? 1 : 0;
                const S st = store_from<S>(relax_fp64(hx, hy, accept ? fp : f, q));
                own[idx] = st;
                f = load_as<double>(st);
                if (sample) add_sample(a, idx, f);
            }
            if (measure) {
                double s, co;
                sincos(q * f, &s, &co);
                eacc += (E)(co * hx + s * hy);
            }
        }
    }
    *e_out = eacc;
    *n_out = n_acc;
}

// One tile of 64 half-lattice columns x 16 rows per block, tiles row-major over a 1-D grid (no
// limit on the number of tile rows).
template <typename S, typename E>
__global__ void __launch_bounds__(256, 3) sweep_kernel(const __grid_constant__ SweepArgs a,
                                                       const __grid_constant__ FixedQ fq)
{
    __shared__ Unit nb[kTY + 2][kSW];
    __shared__ fixed::Dir tab[fixed::kDirs];
    __shared__ E wsum[kRowWarps];
    constexpr int kStaged = (kTY + 2) * kSW, kPer = (kStaged + 255) / 256;

    const int c = a.colour, cb = c ^ 1;
    const int ntx = (a.Lxh + kCols - 1) / kCols;
    const int j0 = (int)(blockIdx.x % ntx) * kCols;
    const int y0 = (int)(blockIdx.x / ntx) * kTY;
    const S* __restrict__ other = static_cast<const S*>(a.other);
    S* __restrict__ own = static_cast<S*>(a.own);
    const int tid = threadIdx.y * 32 + threadIdx.x;
    // FP32 values keep their own bits through the conversion to fixed point (FP16 and BF16 are
    // FP32 values)
    using V = typename std::conditional<sizeof(S) == 8, double, float>::type;
    const fixed::Split k65 = fixed::split(fq.k65);

    // ---- the thread's entries of the other colour, its own sites and the table: loads first
    V ov[kPer];
    bool ok[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int e = tid + i * 256;
        const int r = e / kSW, cc = e - r * kSW;
        const int y = y0 - 1 + r, j = j0 - 1 + cc;
        ok[i] = e < kStaged && y >= 0 && y < a.Ly && j >= 0 && 2 * j + ((y + cb) & 1) < a.Lx;
        ov[i] = ok[i] ? load_as<V>(other[(size_t)y * a.pitch + j]) : (V)0;
    }
    const int jp = j0 + 2 * threadIdx.x;   // the thread's site pair
    V fo[kRows][2];
    uint32_t bits[kRows];   // bit t: frozen, bit 2 + t: the site exists
    bool bad = false;
#pragma unroll
    for (int rr = 0; rr < kRows; ++rr) {
        const int y = y0 + threadIdx.y * kRows + rr;
        bits[rr] = 3u;
        fo[rr][0] = fo[rr][1] = (V)0;
        if (y < a.Ly) {   // a row's pairs are padded to the pitch
            const int o = (y + c) & 1;
            bits[rr] = (a.mbits[(size_t)y * a.mpitch + (jp >> 5)] >> (jp & 31)) & 3u;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                if (2 * (jp + t) + o < a.Lx) {
                    bits[rr] |= 4u << t;
                    fo[rr][t] = load_as<V>(own[(size_t)y * a.pitch + jp + t]);
                } else {
                    bits[rr] |= 1u << t;
                }
                bad |= !fixed::in_range(fo[rr][t]);
            }
        }
    }
    fixed::load_dirs(&g_dirs, tab, tid, 256);
    __syncthreads();

    // ---- stage the other colour's unit vectors (cos q*phi, sin q*phi) with a one-site halo.
    // Entries outside the lattice stay (0, 0): that is the open boundary.
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int e = tid + i * 256;
        if (e < kStaged) {
            Unit v;
            v.i.x = v.i.y = 0;
            if (ok[i]) {
                bad |= !fixed::in_range(ov[i]);
                int64_t co, s;
                fixed::sincos_turn(tab, fixed::turns(ov[i], k65), &co, &s);
                v.i.x = (co + 2) >> 2;
                v.i.y = (s + 2) >> 2;
            }
            (&nb[0][0])[e] = v;
        }
    }
    const bool measure = (a.flags & kMeasure) && c == 1;
    int n_acc = 0;
    E eacc = (E)0;
    if (__syncthreads_or(bad)) {
        rows_fp64<S, E>(a, j0, y0, nb, &eacc, &n_acc);
    } else {
        const bool sample = (a.flags & kSample) != 0;
        const double q = a.q;
        const bool bounded = a.width != nullptr;
        const double pw = bounded ? *a.width : 0.0;   // bounded proposals: half-width
        const float Tf = (float)a.T;
        long long esum = 0;   // E = FP64: sum of u_b . h_b with 58 fraction bits (4 sites of <= 4)
#pragma unroll 1
        for (int rr = 0; rr < kRows; ++rr) {
            const int ly = threadIdx.y * kRows + rr;
            const int y = y0 + ly;
            const uint32_t b = rr ? bits[1] : bits[0];
            const int o = (y + c) & 1;
            uint4 w = make_uint4(0u, 0u, 0u, 0u);
            if ((b & 3u) != 3u)
                w = pair_words((uint32_t)(jp >> 1), (uint32_t)y, a.sweep, a.problem, kTagMetropolis,
                               (uint32_t)c, a.seed_lo, a.seed_hi);
#pragma unroll 1
            for (int t = 0; t < 2; ++t) {
                const bool upd = !((b >> t) & 1u);
                if (!upd && !(measure && ((b >> (2 + t)) & 1u))) continue;
                const int j = jp + t, lj = j - j0;
                // local field h = sum of the neighbours' unit vectors (left, right, up, down)
                const longlong2 lf = nb[ly + 1][lj + o].i, rt = nb[ly + 1][lj + o + 1].i;
                const longlong2 up = nb[ly][lj + 1].i, dn = nb[ly + 2][lj + 1].i;
                const int64_t hx = (lf.x + rt.x) + (up.x + dn.x);
                const int64_t hy = (lf.y + rt.y) + (up.y + dn.y);
                const size_t idx = (size_t)y * a.pitch + j;
                V fv = rr ? (t ? fo[1][1] : fo[1][0]) : (t ? fo[0][1] : fo[0][0]);
                if (upd) {
                    const double f = (double)fv;
                    const uint32_t wp = t ? w.z : w.x, wa = t ? w.w : w.y;
                    // Metropolis: uniform proposal 2 pi u, q times that being wp * q turns (or
                    // bounded: f + pw (2u - 1), rejected outside [0, 2 pi))
                    uint64_t tp = (uint64_t)wp * (uint32_t)(fq.q64 >> 32) +
                                  fixed::umulhi32(wp, (uint32_t)fq.q64);
                    double fp = 0.0;
                    bool inside = true;
                    const uint64_t t0 = fixed::turns(fv, k65);
                    if (bounded) {
                        fp = f + pw * (2.0 * uniform_d(wp) - 1.0);
                        inside = fp >= 0.0 && fp < kTwoPi;
                        tp = inside ? fixed::turns(fp, k65) : t0;
                    }
                    // FP32 estimates: hx, hy to 6e-8 of their size and 2^-28, the sines and cosines to
                    // 9e-7 (angle rounded to FP32 in [-pi, pi], intrinsics to 2^-21.2), so dE to
                    // 2e-6 (|hx| + |hy|) and its roundings; T |ln u| to 6e-7 of its size and
                    // 5e-7 T. Accepted iff dE < T |ln u| (which is >= 0).
                    const float hxf = (float)(int32_t)(hx >> 32) * 0x1p-28f;
                    const float hyf = (float)(int32_t)(hy >> 32) * 0x1p-28f;
                    constexpr float kTurn = 1.46291807926715968e-9f;   // 2 pi / 2^32
                    float s0, c0, sp, cp;
                    __sincosf((float)(int32_t)(t0 >> 32) * kTurn, &s0, &c0);
                    __sincosf((float)(int32_t)(tp >> 32) * kTurn, &sp, &cp);
                    const float dE = hxf * (c0 - cp) + hyf * (s0 - sp);
                    const float lu = -Tf * __logf((float)wa * 0x1p-32f);
                    const float tol = 3.5e-6f * (fabsf(hxf) + fabsf(hyf)) + 1e-6f +
                                      1e-6f * Tf + 1.5e-6f * lu;
                    const float d = lu - dE;
                    bool accept = d > tol;
                    if (inside && !accept && !(d < -tol)) {   // within the bound, u = 0, or T huge
                        if (!bounded) fp = kTwoPi * uniform_d(wp);
                        accept = accept_fp64((double)hx * 0x1p-60, (double)hy * 0x1p-60, f, fp, q,
                                             a.T, uniform_d(wa));
                    }
                    accept = accept && inside;
                    n_acc += accept ? 1 : 0;
                    // over-relaxation: reflect q*phi about arg(h); keep it if it lands in
                    // [0, 2*pi*q]
                    double fn;
                    const uint32_t ax = (uint32_t)((hx >> 32) ^ (hx >> 63));
                    const uint32_t ay = (uint32_t)((hy >> 32) ^ (hy >> 63));
                    if ((ax | ay) < (1u << 18)) {   // |hx|, |hy| < 2^-10
                        const double2 h = field_fp64<S>(a, y, j, o);
                        if (!bounded) fp = kTwoPi * uniform_d(wp);
                        fn = relax_fp64(h.x, h.y, accept ? fp : f, q);
                    } else {
                        const float d2 = f32::atan2_doubled<false>(hyf, hxf);
                        // half of it in turns, 2^32 / (4 pi) per radian
                        const int32_t th = __float2int_rn(d2 * 341782637.788f);
                        const uint64_t r =
                            fixed::doubled_arg(tab, hx, hy, th) - (accept ? tp : t0);
                        if (r <= fq.q64) {
                            const uint64_t n = fq.sh >= 0 ? r << fq.sh : r >> 1;
                            fn = fixed::to_double_q60(fixed::umulhi(n, fq.m64));
                        } else {
                            if (accept && !bounded) fp = kTwoPi * uniform_d(wp);
                            fn = accept ? fp : f;
                        }
                    }
                    const S st = store_from<S>(fn);
                    own[idx] = st;
                    fv = load_as<V>(st);
                    if (sample) add_sample(a, idx, (double)fv);
                }
                if (measure) {
                    // every bond joins a red and a black site: sum over black sites of u_b . h_b
                    int64_t co, s;
                    fixed::sincos_turn(tab, fixed::turns(fv, k65), &co, &s);
                    const int64_t e = fixed::mulhi(fixed::split(co), fixed::split(hx)) +
                                      fixed::mulhi(fixed::split(s), fixed::split(hy));
                    if (sizeof(E) == 8) esum += e;
                    else eacc += (E)e * (E)0x1p-58;
                }
            }
        }
        if (sizeof(E) == 8) eacc = (E)esum * (E)0x1p-58;
    }

    if (a.accepted) {
#pragma unroll
        for (int off = 16; off; off >>= 1) n_acc += __shfl_xor_sync(0xffffffffu, n_acc, off);
        if (threadIdx.x == 0 && n_acc) atomicAdd(a.accepted, (unsigned long long)n_acc);
    }
    if (measure) {
#pragma unroll
        for (int off = 16; off; off >>= 1) eacc += __shfl_xor_sync(0xffffffffu, eacc, off);
        if (threadIdx.x == 0) wsum[threadIdx.y] = eacc;
        __syncthreads();
        if (tid == 0) {
            E s = (E)0;
            for (int i = 0; i < kRowWarps; ++i) s += wsum[i];
            static_cast<E*>(a.epart)[blockIdx.x] = s;
        }
    }
}

template <typename S, typename E>
cudaError_t launch_typed(const SweepArgs& a, cudaStream_t st)
{
    const dim3 grid(((a.Lxh + kCols - 1) / kCols) * ((a.Ly + kTY - 1) / kTY));
    sweep_kernel<S, E><<<grid, dim3(32, kRowWarps), 0, st>>>(a, fixed_q(a.q));
    return cudaGetLastError();
}

template <typename S>
cudaError_t launch_store(const Precision& p, const SweepArgs& a, cudaStream_t st)
{
    return p.energy == 0 ? launch_typed<S, double>(a, st) : launch_typed<S, float>(a, st);
}

}  // namespace

int sweep_blocks(const Layout& L, const Precision&)
{
    return ((L.Lxh + kCols - 1) / kCols) * ((L.Ly + kTY - 1) / kTY);
}

cudaError_t launch_sweep(const Precision& p, const SweepArgs& a, cudaStream_t st)
{
    if (p.func != 0) return cudaErrorInvalidValue;   // FP32 functions: launch_sweep_f32
    switch (p.store) {
    case kF64: return launch_store<double>(p, a, st);
    case kF32: return launch_store<float>(p, a, st);
    case kF16: return launch_store<__half>(p, a, st);
    case kBF16: return launch_store<__nv_bfloat16>(p, a, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace mpr
