// mpr_aux.cu -- the non-sweep kernels of libmpr: range of the measured data, data -> spin
// mapping with the initial angles and the frozen-site bits, sample energy e_s, FP64 bond energy
// of a state, deterministic fixed-order reductions, prediction and state transfer.
//
// Every reduction writes per-block partials and sums them in a fixed order in a second kernel,
// so results do not depend on scheduling (no floating-point atomics).
#include "mpr_device.cuh"
#include "mpr_energy.cuh"
#include "mpr_internal.h"

#include <math.h>

#include <type_traits>

namespace mpr {
namespace {

constexpr int kThreads = 256;

// --------------------------------------------------------------------------------------------
// Range of the measured values: partial (min, max, count, non-finite count) per block.
// --------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) minmax_kernel(const double* __restrict__ z,
                                                          const unsigned char* __restrict__ mask,
                                                          long long N, double* __restrict__ part)
{
    double lo = INFINITY, hi = -INFINITY, n = 0.0, bad = 0.0;
    for (long long s = blockIdx.x * (long long)kThreads + threadIdx.x; s < N;
         s += (long long)gridDim.x * kThreads) {
        if (!mask[s]) continue;
        const double v = z[s];
        if (!isfinite(v)) { bad += 1.0; continue; }
        lo = fmin(lo, v);
        hi = fmax(hi, v);
        n += 1.0;
    }
    __shared__ double sh[4][kThreads];
    sh[0][threadIdx.x] = lo;
    sh[1][threadIdx.x] = hi;
    sh[2][threadIdx.x] = n;
    sh[3][threadIdx.x] = bad;
    __syncthreads();
    for (int w = kThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            sh[0][threadIdx.x] = fmin(sh[0][threadIdx.x], sh[0][threadIdx.x + w]);
            sh[1][threadIdx.x] = fmax(sh[1][threadIdx.x], sh[1][threadIdx.x + w]);
            sh[2][threadIdx.x] += sh[2][threadIdx.x + w];
            sh[3][threadIdx.x] += sh[3][threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int k = 0; k < 4; ++k) part[4 * blockIdx.x + k] = sh[k][0];
}

__global__ void minmax_final(const double* __restrict__ part, int nblk, double* __restrict__ out)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double lo = INFINITY, hi = -INFINITY, n = 0.0, bad = 0.0;
    for (int b = 0; b < nblk; ++b) {
        lo = fmin(lo, part[4 * b]);
        hi = fmax(hi, part[4 * b + 1]);
        n += part[4 * b + 2];
        bad += part[4 * b + 3];
    }
    out[0] = lo;
    out[1] = hi;
    out[2] = n;
    out[3] = bad;
}

// --------------------------------------------------------------------------------------------
// Mapping phi = 2*pi*(z - zmin)/(zmax - zmin) on measured sites, uniform initial angles on the
// prediction sites (init stream, sweep 0), packed by colour; one warp ballot per mask word.
// --------------------------------------------------------------------------------------------
template <typename S>
__global__ void __launch_bounds__(kThreads) init_kernel(Layout L, const double* __restrict__ z,
                                                        const unsigned char* __restrict__ mask,
                                                        const double* __restrict__ range,
                                                        S* __restrict__ ang0, S* __restrict__ ang1,
                                                        uint32_t* __restrict__ mb0,
                                                        uint32_t* __restrict__ mb1, uint32_t seed_lo,
                                                        uint32_t seed_hi, uint32_t problem,
                                                        int fp32_uniform)
{
    const int j = blockIdx.x * kThreads + threadIdx.x;
    if (j >= L.pitch) return;   // pitch is a multiple of 32: whole warps leave together
    const int c = blockIdx.z;
    for (int y = blockIdx.y; y < L.Ly; y += gridDim.y) {   // rows beyond the 65535 grid limit
        const int x = 2 * j + ((y + c) & 1);
        S* ang = c ? ang1 : ang0;
        uint32_t* mb = c ? mb1 : mb0;
        const size_t idx = (size_t)y * L.pitch + j;
        bool frozen = true;   // padding counts as frozen: never updated
        if (x < L.Lx) {
            const size_t s = (size_t)y * L.Lx + x;
            double phi;
            if (mask[s]) {
                const double lo = range[0], hi = range[1];
                const double t = (z[s] - lo) / (hi - lo);
                phi = kTwoPi * t;
            } else {
                frozen = false;
                const uint4 w = pair_words((uint32_t)(j >> 1), (uint32_t)y, 0u, problem, kTagInit,
                                           (uint32_t)c, seed_lo, seed_hi);
                const uint32_t wp = (j & 1) ? w.z : w.x;
                const double u = fp32_uniform ? (double)uniform_f(wp) : uniform_d(wp);
                phi = kTwoPi * u;
            }
            ang[idx] = store_from<S>(phi);
        } else {
            ang[idx] = store_from<S>(0.0);
        }
        const uint32_t bits = __ballot_sync(0xffffffffu, frozen);
        if ((threadIdx.x & 31) == 0) mb[(size_t)y * L.mpitch + (j >> 5)] = bits;
    }
}

// --------------------------------------------------------------------------------------------
// Sample energy: sum of cos[q(phi_i - phi_j)] over measured-measured bonds, in FP64 from the
// mapped values, and the number of such bonds.
// --------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) sample_energy_kernel(Layout L,
                                                                 const double* __restrict__ z,
                                                                 const unsigned char* __restrict__ mask,
                                                                 const double* __restrict__ range,
                                                                 double q, double* __restrict__ psum,
                                                                 long long* __restrict__ pcnt)
{
    const long long N = (long long)L.Lx * L.Ly;
    const double lo = range[0], hi = range[1];
    double sum = 0.0;
    long long cnt = 0;
    for (long long s = blockIdx.x * (long long)kThreads + threadIdx.x; s < N;
         s += (long long)gridDim.x * kThreads) {
        if (!mask[s]) continue;
        const int y = (int)(s / L.Lx), x = (int)(s - (long long)y * L.Lx);
        const double ps = kTwoPi * ((z[s] - lo) / (hi - lo));
        if (x + 1 < L.Lx && mask[s + 1]) {
            const double pr = kTwoPi * ((z[s + 1] - lo) / (hi - lo));
            sum += cos(q * (ps - pr));
            ++cnt;
        }
        if (y + 1 < L.Ly && mask[s + L.Lx]) {
            const double pd = kTwoPi * ((z[s + L.Lx] - lo) / (hi - lo));
            sum += cos(q * (ps - pd));
            ++cnt;
        }
    }
    __shared__ double ss[kThreads];
    __shared__ long long sc[kThreads];
    ss[threadIdx.x] = sum;
    sc[threadIdx.x] = cnt;
    __syncthreads();
    for (int w = kThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            ss[threadIdx.x] += ss[threadIdx.x + w];
            sc[threadIdx.x] += sc[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        psum[blockIdx.x] = ss[0];
        pcnt[blockIdx.x] = sc[0];
    }
}

// One block: a thread added up a chain of 1024 partials in 86 us.
__global__ void __launch_bounds__(kThreads) sample_energy_final(const double* __restrict__ psum,
                                                                const long long* __restrict__ pcnt,
                                                                int nblk, double* __restrict__ out)
{
    __shared__ double ss[kThreads];
    __shared__ long long sc[kThreads];
    double s = 0.0;
    long long n = 0;
    for (int b = threadIdx.x; b < nblk; b += kThreads) {
        s += psum[b];
        n += pcnt[b];
    }
    ss[threadIdx.x] = s;
    sc[threadIdx.x] = n;
    __syncthreads();
    for (int w = kThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            ss[threadIdx.x] += ss[threadIdx.x + w];
            sc[threadIdx.x] += sc[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = sc[0] > 0 ? -ss[0] / (double)sc[0] : 0.0;
        out[1] = (double)sc[0];
    }
}

// --------------------------------------------------------------------------------------------
// FP64 bond energy of the current state: every bond joins a red and a black site, so the bond
// sum is the sum over black sites b of (cos q phi_b, sin q phi_b) . h_b.
// --------------------------------------------------------------------------------------------
// A strip is 30 half-lattice columns x `rows` rows of one warp; lane l stands at column
// j0 - 1 + l and converts one red and one black angle per row, lanes 1 ... 30 sum the four bonds
// of their black site: red neighbours of the row by shuffle, those above and below from the red
// rows the warp keeps. A row with an angle outside [0, 7.5) (a state set by the caller) takes FP64.
// 4096^2, FP16 spins: 2305 us with five FP64 sincos per black site.
// NARROW (at most 14 half-lattice columns): a warp walks 32 / w strips side by side, w = 2^lw >= Lxh + 2 lanes
// each; rows is even there, so that every strip is at a row of the same parity (2 x 1000000: 741 us with
// a strip per warp).
template <typename S, bool NARROW>
__global__ void __launch_bounds__(kThreads) energy_kernel(Layout L, const S* __restrict__ red,
                                                          const S* __restrict__ black, double q,
                                                          int64_t k65, int rows, int lw,
                                                          energy::Sum* __restrict__ part)
{
    using V = typename std::conditional<sizeof(S) == 8, double, float>::type;
    __shared__ fixed::Dir tab[fixed::kDirs];
    fixed::load_dirs(&energy::g_dirs, tab, threadIdx.x, kThreads);
    __syncthreads();
    const fixed::Split k = fixed::split(k65);
    const int w = NARROW ? 1 << lw : 32, side = NARROW ? 32 >> lw : 1;
    const int lane = threadIdx.x & (w - 1);
    const int nsx = NARROW ? 1 : (L.Lxh + 29) / 30;
    const long long nstrips = (long long)nsx * ((L.Ly + rows - 1) / rows);
    energy::Sum sum{0, 0};
    bool nan = false;
    for (long long st = ((long long)blockIdx.x * energy::kWarpsPerBlock + (threadIdx.x >> 5)) * side;
         st < nstrips; st += (long long)gridDim.x * energy::kWarpsPerBlock * side) {
        const int sy = NARROW ? (int)st + ((threadIdx.x & 31) >> lw) : (int)(st / nsx);
        const int sx = NARROW ? 0 : (int)(st - (long long)sy * nsx);
        const int j = sx * 30 + lane - 1, y0 = sy * rows;
        const int y1 = NARROW || y0 + rows < L.Ly ? y0 + rows : L.Ly;
        // a red angle at column j of row y (0 where there is none)
        auto is_red = [&](int y) { return j >= 0 && y >= 0 && y < L.Ly && 2 * j + (y & 1) < L.Lx; };
        auto red_at = [&](int y) -> V {
            return is_red(y) ? load_as<V>(red[(size_t)y * L.pitch + j]) : (V)0;
        };
        auto unit_at = [&](int y, V f) {
            return energy::neighbour(energy::unit_of_turn(tab, fixed::turns(f, k)), is_red(y));
        };
        V fu = red_at(y0 - 1), fm = red_at(y0);
        bool oku = fixed::in_range(fu), okm = fixed::in_range(fm);
        energy::Vec uu = unit_at(y0 - 1, fu), um = unit_at(y0, fm);
        int64_t acc = 0;   // at most 16 terms of 2^58
        for (int y = y0; y < y1; ++y) {
            const V fd = red_at(y + 1);
            const bool okd = fixed::in_range(fd);
            const energy::Vec ud = unit_at(y + 1, fd);
            const int o = (y + 1) & 1;   // black: x = 2j + o, red neighbours at columns j+o-1, j+o
            const int x = 2 * j + o;
            const bool has = lane >= 1 && lane <= w - 2 && j < L.Lxh && x < L.Lx && (!NARROW || y < L.Ly);
            const V fb = has ? load_as<V>(black[(size_t)y * L.pitch + j]) : (V)0;
            const bool ok = okd && okm && oku && fixed::in_range(fb);
            if (__all_sync(0xffffffffu, ok)) {
                const energy::Vec us =
                    o ? energy::Vec{__shfl_down_sync(0xffffffffu, um.c, 1), __shfl_down_sync(0xffffffffu, um.s, 1)}
                      : energy::Vec{__shfl_up_sync(0xffffffffu, um.c, 1), __shfl_up_sync(0xffffffffu, um.s, 1)};
                const energy::Vec h{(um.c + us.c) + (uu.c + ud.c), (um.s + us.s) + (uu.s + ud.s)};
                const int64_t e = energy::term(energy::unit_of_turn(tab, fixed::turns(fb, k)), h);
                acc += has ? e : 0;
            } else {
                const V fs = o ? __shfl_down_sync(0xffffffffu, fm, 1)
                               : __shfl_up_sync(0xffffffffu, fm, 1);
                if (has) {
                    double hx = 0.0, hy = 0.0, sn, cs;
                    if (x > 0) { sincos(q * (double)(o ? fm : fs), &sn, &cs); hx += cs; hy += sn; }
                    if (x + 1 < L.Lx) { sincos(q * (double)(o ? fs : fm), &sn, &cs); hx += cs; hy += sn; }
                    if (y > 0) { sincos(q * (double)fu, &sn, &cs); hx += cs; hy += sn; }
                    if (y + 1 < L.Ly) { sincos(q * (double)fd, &sn, &cs); hx += cs; hy += sn; }
                    sincos(q * (double)fb, &sn, &cs);
                    acc += energy::term_fp64(cs * hx + sn * hy, &nan);
                }
            }
            fu = fm;
            fm = fd;
            uu = um;
            um = ud;
            oku = okm;
            okm = okd;
        }
        sum.add(acc);
    }
    energy::store_sum(sum, nan, part);
}

__global__ void __launch_bounds__(kThreads) energy_final(const energy::Sum* __restrict__ part, int n,
                                                         double* __restrict__ out)
{
    const double s = energy::final_sum(part, n);
    if (threadIdx.x == 0) *out = s;
}

// --------------------------------------------------------------------------------------------
// Prediction zhat = zmin + (zmax - zmin) * (mean phi / 2*pi) on prediction sites, z elsewhere, as
// zmin + sum * K with K = (zmax - zmin) / (2*pi*n) formed once per block: one FP64 multiply-add per
// site (and one rounding less than dividing by n and by 2*pi at every site, which took about 20
// instructions of the FP64 unit: 593 us at 4096^2, 9.4 ms at 16384^2; now 71 us at 4096^2, at 65 % of
// the DRAM rate, the FP64 unit 59 % busy). A block covers 256 columns x kPredRows rows, all of a thread's
// loads in flight before K is ready. On grids of at most 128 columns it covers 2^lw >= Lx columns and as many
// more rows, its rows interleaved over the threads (2 x 1000000: 256 columns a block leave 254 of 256
// threads idle). Grids that would make fewer blocks than two per SM take one row per thread: there the
// FP64 unit's share of a block is what the call waits for. With a range near the smallest FP64 numbers K
// would lose bits or vanish: 2^200 K then, and sums times 2^-200 (both exact).
// --------------------------------------------------------------------------------------------
constexpr int kPredRows = 8;

template <int ROWS>
__global__ void __launch_bounds__(kThreads) predict_kernel(Layout L, const double* __restrict__ z,
                                                           const unsigned char* __restrict__ mask,
                                                           const double* __restrict__ range,
                                                           const double* __restrict__ acc0,
                                                           const double* __restrict__ acc1,
                                                           const float* __restrict__ hi0,
                                                           const float* __restrict__ lo0,
                                                           const float* __restrict__ hi1,
                                                           const float* __restrict__ lo1,
                                                           int nsamples, int lw, double* __restrict__ out)
{
    __shared__ double s_k;
    const double lo = range[0], width = range[1] - lo;
    const bool tiny = width < 0x1p-900;
    if (threadIdx.x == 0) s_k = (tiny ? width * 0x1p200 : width) / (kTwoPi * (double)nsamples);
    const int x = (blockIdx.x << lw) + (threadIdx.x & ((1 << lw) - 1));
    const int ystep = kThreads >> lw;                // rows of the block side by side
    const long long rows = (long long)ROWS * ystep;
    bool first = true;
    for (long long yb = blockIdx.y * rows; yb < L.Ly; yb += gridDim.y * rows) {   // (grid limit 65535)
        const int y0 = (int)yb + (int)(threadIdx.x >> lw);
        double v[ROWS];
        bool meas[ROWS];
        // every mask byte, then every value, without a branch on the mask between the rows: with one a
        // thread's rows followed one another, 8 us longer at 64^2
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            const int y = y0 + i * ystep;
            meas[i] = x < L.Lx && y < L.Ly && mask[(size_t)y * L.Lx + x] != 0;
        }
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            const int y = y0 + i * ystep;
            const bool there = x < L.Lx && y < L.Ly;
            const size_t s = (size_t)y * L.Lx + x, idx = (size_t)y * L.pitch + (x >> 1);
            const int c = (x + y) & 1;
            if (acc0) {
                const double* const p = meas[i] ? z + s : (c ? acc1 : acc0) + idx;
                v[i] = there ? *p : 0.0;
            } else {
                // two words either way: of the value, or the sum and its compensation
                const int* const zw = reinterpret_cast<const int*>(z + s);
                const int* const p0 = meas[i] ? zw : reinterpret_cast<const int*>((c ? hi1 : hi0) + idx);
                const int* const p1 = meas[i] ? zw + 1 : reinterpret_cast<const int*>((c ? lo1 : lo0) + idx);
                const int w0 = there ? *p0 : 0, w1 = there ? *p1 : 0;
                v[i] = meas[i] ? __hiloint2double(w1, w0)
                               : (double)__int_as_float(w0) - (double)__int_as_float(w1);
            }
        }
        if (first) __syncthreads();   // s_k (every thread of the block makes the same trips)
        first = false;
        const double k = s_k;
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            const int y = y0 + i * ystep;
            if (x >= L.Lx || y >= L.Ly) continue;
            if (tiny && !meas[i]) v[i] *= 0x1p-200;
            out[(size_t)y * L.Lx + x] = meas[i] ? v[i] : fma(v[i], k, lo);
        }
    }
}

// --------------------------------------------------------------------------------------------
// State transfer between the packed colour layout and a row-major FP64 grid.
// --------------------------------------------------------------------------------------------
template <typename S>
__global__ void __launch_bounds__(kThreads) get_state_kernel(Layout L, const S* __restrict__ a0,
                                                             const S* __restrict__ a1,
                                                             double* __restrict__ out)
{
    const long long N = (long long)L.Lx * L.Ly;
    const long long s = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (s >= N) return;
    const int y = (int)(s / L.Lx), x = (int)(s - (long long)y * L.Lx);
    const size_t idx = (size_t)y * L.pitch + (x >> 1);
    out[s] = load_as<double>(((x + y) & 1) ? a1[idx] : a0[idx]);
}

template <typename S>
__global__ void __launch_bounds__(kThreads) set_state_kernel(Layout L, const double* __restrict__ in,
                                                             const unsigned char* __restrict__ mask,
                                                             S* __restrict__ a0, S* __restrict__ a1)
{
    const long long N = (long long)L.Lx * L.Ly;
    const long long s = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (s >= N || mask[s]) return;
    const int y = (int)(s / L.Lx), x = (int)(s - (long long)y * L.Lx);
    const size_t idx = (size_t)y * L.pitch + (x >> 1);
    (((x + y) & 1) ? a1 : a0)[idx] = store_from<S>(in[s]);
}

__global__ void philox_kernel(const uint32_t* __restrict__ ctr, uint32_t* __restrict__ out, int n,
                              uint32_t k0, uint32_t k1)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 c = reinterpret_cast<const uint4*>(ctr)[i];
    reinterpret_cast<uint4*>(out)[i] = philox4x32_10(c, k0, k1);
}

// Width of the bounded Metropolis proposals after one sweep: w <- w exp(a - target), with a the
// sweep's acceptance fraction over the n_pred prediction sites, kept in [1e-3, 2 pi]; the
// counter restarts at 0 for the next sweep.
// Launched as a programmatic dependent launch between two sweeps: it waits for the black pass it
// follows, then lets the next red pass be scheduled at once (that pass still waits for this
// kernel's completion before it reads the width).
__global__ void adapt_width_kernel(double* __restrict__ width, unsigned long long* __restrict__ count,
                                   long long n_pred, double target)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const double acc = n_pred > 0 ? (double)*count / (double)n_pred : target;
    *width = fmin(fmax(*width * exp(acc - target), 1e-3), 6.283185307179586);
    *count = 0ull;
}

inline int grid_for(long long n) { return (int)((n + kThreads - 1) / kThreads); }

// Folds fixed-point partial sums of sampled FP16 angles (units of 2^-24) into the FP64 sums:
// exact, as both are integer multiples of 2^-24 far below 2^53 units.
__global__ void __launch_bounds__(kThreads) fold_partials_kernel(double* __restrict__ acc,
                                                                 int* __restrict__ part,
                                                                 long long n)
{
    const long long i = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (i >= n) return;
    const int v = part[i];
    if (v) {
        acc[i] += (double)v * 0x1.0p-24;
        part[i] = 0;
    }
}

template <typename Fn>
cudaError_t dispatch_store(int store, Fn&& f)
{
    switch (store) {
    case kF64: return f(double{});
    case kF32: return f(float{});
    case kF16: return f(__half{});
    case kBF16: return f(__nv_bfloat16{});
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_minmax(const double* z, const unsigned char* mask, long long N, double* part,
                          int nblk, double* out4, cudaStream_t st)
{
    minmax_kernel<<<nblk, kThreads, 0, st>>>(z, mask, N, part);
    minmax_final<<<1, 32, 0, st>>>(part, nblk, out4);
    return cudaGetLastError();
}

cudaError_t launch_init(const Layout& L, const Precision& p, const double* z,
                        const unsigned char* mask, const double* range, void* ang0, void* ang1,
                        uint32_t* mb0, uint32_t* mb1, uint64_t seed, uint32_t problem,
                        cudaStream_t st)
{
    const dim3 grid((L.pitch + kThreads - 1) / kThreads, L.Ly < 65535 ? L.Ly : 65535, 2);
    const uint32_t klo = (uint32_t)seed, khi = (uint32_t)(seed >> 32);
    return dispatch_store(p.store, [&](auto tag) {
        using S = decltype(tag);
        init_kernel<S><<<grid, kThreads, 0, st>>>(L, z, mask, range, static_cast<S*>(ang0),
                                                  static_cast<S*>(ang1), mb0, mb1, klo, khi,
                                                  problem, p.func);
        return cudaGetLastError();
    });
}

int sample_energy_blocks(const Layout& L)
{
    const long long n = (long long)L.Lx * L.Ly;
    const long long b = (n + kThreads - 1) / kThreads;
    return (int)(b < 1024 ? b : 1024);
}

cudaError_t launch_sample_energy(const Layout& L, const double* z, const unsigned char* mask,
                                 const double* range, double q, double* part_sum,
                                 long long* part_cnt, int nblk, double* out2, cudaStream_t st)
{
    sample_energy_kernel<<<nblk, kThreads, 0, st>>>(L, z, mask, range, q, part_sum, part_cnt);
    sample_energy_final<<<1, kThreads, 0, st>>>(part_sum, part_cnt, nblk, out2);
    return cudaGetLastError();
}

// Strips of the energy kernel: 2^lw lanes (two of them neighbours' columns) x rows rows.
struct EnergyStrips {
    int lw = 5, rows;
    long long warps;   // of 32 / 2^lw strips
    explicit EnergyStrips(const Layout& L)
    {
        while (lw > 2 && (1 << (lw - 1)) >= L.Lxh + 2) --lw;
        const int nsx = (L.Lxh + 29) / 30, side = 32 >> lw;
        rows = energy::strip_rows(nsx, (L.Ly + side - 1) / side);
        if (lw < 5) rows += rows & 1;
        warps = ((long long)nsx * ((L.Ly + rows - 1) / rows) + side - 1) / side;
    }
};

int energy_blocks(const Layout& L)
{
    const long long b = (EnergyStrips(L).warps + energy::kWarpsPerBlock - 1) / energy::kWarpsPerBlock;
    return (int)(b < 152 * 6 ? b : 152 * 6);
}

cudaError_t launch_energy_fp64(const Layout& L, const Precision& p, const void* ang0,
                               const void* ang1, double q, double* part, int nblk, double* out,
                               cudaStream_t st)
{
    return dispatch_store(p.store, [&](auto tag) {
        using S = decltype(tag);
        const EnergyStrips es(L);
        energy::Sum* const sums = reinterpret_cast<energy::Sum*>(part);   // 16 bytes a block
        auto* const kern = es.lw < 5 ? energy_kernel<S, true> : energy_kernel<S, false>;
        kern<<<nblk, kThreads, 0, st>>>(L, static_cast<const S*>(ang0), static_cast<const S*>(ang1), q,
                                        fixed::turn_factor(q), es.rows, es.lw, sums);
        energy_final<<<1, kThreads, 0, st>>>(sums, nblk, out);
        return cudaGetLastError();
    });
}

cudaError_t launch_predict(const Layout& L, const Precision&, const double* z,
                           const unsigned char* mask, const double* range, const double* acc0,
                           const double* acc1, const float* hi0, const float* lo0,
                           const float* hi1, const float* lo1, int nsamples, double* out,
                           cudaStream_t st)
{
    int lw = 8;
    if (L.Lx <= 128)
        for (lw = 1; 1 << lw < L.Lx;) ++lw;
    const long long strips = (L.Ly + (kThreads >> lw) - 1) / (kThreads >> lw);   // rows of all threads
    const unsigned nx = (unsigned)((L.Lx + (1 << lw) - 1) >> lw);
    const bool few = strips * nx < (long long)kPredRows * 2 * 152;
    const long long ny = few ? strips : (strips + kPredRows - 1) / kPredRows;
    const dim3 grid(nx, (unsigned)(ny < 65535 ? ny : 65535));
    auto* const kern = few ? predict_kernel<1> : predict_kernel<kPredRows>;
    kern<<<grid, kThreads, 0, st>>>(L, z, mask, range, acc0, acc1, hi0, lo0, hi1, lo1, nsamples, lw, out);
    return cudaGetLastError();
}

cudaError_t launch_get_state(const Layout& L, const Precision& p, const void* ang0,
                             const void* ang1, double* out, cudaStream_t st)
{
    const long long N = (long long)L.Lx * L.Ly;
    return dispatch_store(p.store, [&](auto tag) {
        using S = decltype(tag);
        get_state_kernel<S><<<grid_for(N), kThreads, 0, st>>>(L, static_cast<const S*>(ang0),
                                                             static_cast<const S*>(ang1), out);
        return cudaGetLastError();
    });
}

cudaError_t launch_set_state(const Layout& L, const Precision& p, const double* in,
                             const unsigned char* mask, void* ang0, void* ang1, cudaStream_t st)
{
    const long long N = (long long)L.Lx * L.Ly;
    return dispatch_store(p.store, [&](auto tag) {
        using S = decltype(tag);
        set_state_kernel<S><<<grid_for(N), kThreads, 0, st>>>(L, in, mask, static_cast<S*>(ang0),
                                                             static_cast<S*>(ang1));
        return cudaGetLastError();
    });
}

cudaError_t launch_adapt_width(double* width, unsigned long long* count, long long n_pred,
                               double target, cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(1);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, adapt_width_kernel, width, count, n_pred, target);
}

cudaError_t launch_fold_partials(double* acc, int* part, size_t n, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    fold_partials_kernel<<<grid_for((long long)n), kThreads, 0, st>>>(acc, part, (long long)n);
    return cudaGetLastError();
}

cudaError_t launch_philox(const uint32_t* ctr, uint32_t* out, int n, uint64_t seed, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    philox_kernel<<<grid_for(n), kThreads, 0, st>>>(ctr, out, n, (uint32_t)seed,
                                                   (uint32_t)(seed >> 32));
    return cudaGetLastError();
}

}  // namespace mpr
