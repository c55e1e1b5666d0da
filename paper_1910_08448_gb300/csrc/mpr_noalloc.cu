// mpr_noalloc.cu -- mpr_bond_energy_noalloc: the bond energy of a caller-held state with no device
// allocation at all.
//
// Some callers cannot call cudaMalloc: code that works under a strict device-memory budget or a
// custom allocator that owns the whole device, and real-time loops that must not take the
// allocator's locks or synchronise. Every other entry point of this library allocates its scratch
// (reduction partials) inside a handle. This one keeps its scratch in a fixed array compiled into
// the library instead, so a call only launches kernels.
//
// Cost of that choice: the array below (32 KiB of partial sums) exists on every GPU that loads
// the library, for the life of the process, and all calls share it.
#include "mpr.h"
#include "mpr_energy.cuh"
#include "mpr_internal.h"

#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <mutex>

namespace {

constexpr int kThreads = 256;
constexpr long long kMaxSites = 1ll << 28;    // 16384 x 16384
constexpr int kPartials = 2048;               // partial sums of the first pass, at most
constexpr int kMaxDevices = 64;

// The scratch: one partial sum per block of the first pass (16 bytes). Every block of a call writes its own
// slot before the second pass reads it, so nothing has to be cleared between calls. Calls that
// overlap on the GPU (for example on two streams) use the same slots and race.
static __device__ __align__(256) mpr::energy::Sum g_bond_partials[kPartials];

// First pass: sums of cos[q(phi_s - phi_right)] and cos[q(phi_s - phi_down)] (Eq. 2, open
// boundaries). A strip is 31 columns x `rows` rows of one warp, lane 31 holding the right
// neighbours of lane 30; block b takes strips b * 8 + warp, then on by the whole grid. A row with
// an angle outside (-7.5, 7.5), its own or below it, takes FP64 cosines.
// 4096^2: 1612 us with two FP64 cosines per site on 256 blocks.
__global__ void __launch_bounds__(kThreads) bond_partials(int Lx, int Ly, int rows,
                                                          const double* __restrict__ phi, double q,
                                                          int64_t k65, mpr::energy::Sum* __restrict__ part)
{
    using namespace mpr;
    __shared__ fixed::Dir tab[fixed::kDirs];
    fixed::load_dirs(&energy::g_dirs, tab, threadIdx.x, kThreads);
    __syncthreads();
    const fixed::Split k = fixed::split(k65);
    const int lane = threadIdx.x & 31;
    const int nsx = (Lx + 30) / 31;
    const long long nstrips = (long long)nsx * ((Ly + rows - 1) / rows);
    energy::Sum sum{0, 0};
    bool nan = false;
    for (long long st = (long long)blockIdx.x * energy::kWarpsPerBlock + (threadIdx.x >> 5);
         st < nstrips; st += (long long)gridDim.x * energy::kWarpsPerBlock) {
        const int sy = (int)(st / nsx), sx = (int)(st - (long long)sy * nsx);
        const int x = sx * 31 + lane, y0 = sy * rows;
        const int y1 = y0 + rows < Ly ? y0 + rows : Ly;   // rows whose bonds the strip sums
        const bool has = x < Lx, mine = lane < 31 && has, right = mine && x + 1 < Lx;
        const double* p = phi + (size_t)y0 * Lx + x;
        double f = has ? *p : 0.0, fb = 0.0;
        energy::Vec u = energy::unit_of_turn(tab, energy::turns_signed(f, k)), ub;
        bool ok = energy::in_range_signed(f), okb;
        int64_t acc = 0;   // at most 16 terms of 2^57
        for (int y = y0; y < y1; ++y) {
            const bool below = y + 1 < Ly;
            p += Lx;
            fb = has && below ? *p : 0.0;
            okb = energy::in_range_signed(fb);
            ub = energy::unit_of_turn(tab, energy::turns_signed(fb, k));
            if (__all_sync(0xffffffffu, ok && okb)) {
                const energy::Vec ur{__shfl_down_sync(0xffffffffu, u.c, 1), __shfl_down_sync(0xffffffffu, u.s, 1)};
                const energy::Vec r = energy::neighbour(ur, right), d = energy::neighbour(ub, below);
                const int64_t e = energy::term(u, energy::Vec{r.c + d.c, r.s + d.s});
                acc += mine ? e : 0;
            } else {
                const double fr = __shfl_down_sync(0xffffffffu, f, 1);
                if (right) acc += energy::term_fp64(cos(q * (f - fr)), &nan);
                if (mine && below) acc += energy::term_fp64(cos(q * (f - fb)), &nan);
            }
            f = fb;
            u = ub;
            ok = okb;
        }
        sum.add(acc);
    }
    energy::store_sum(sum, nan, part);
}

// Second pass, one block: fixed-order sum of the partials, e_b = -sum / N_b.
__global__ void __launch_bounds__(kThreads) bond_final(const mpr::energy::Sum* __restrict__ part, int nblk,
                                                       double n_bonds, double* __restrict__ out)
{
    const double s = mpr::energy::final_sum(part, nblk);
    if (threadIdx.x == 0) *out = -s / n_bonds;
}

// Device address of g_bond_partials per device. In host code the array's name only stands for
// the symbol, so the address is looked up once per device, with that device current, and cached
// for the life of the process. It belongs to the device's primary context: after a
// cudaDeviceReset of that device the cached address is stale (see include/mpr.h).
std::mutex g_mu;
mpr::energy::Sum* g_addr[kMaxDevices] = {};

mpr_status err(mpr_status s, const char* msg)
{
    mpr::set_last_error(msg);
    return s;
}

}  // namespace

extern "C" mpr_status mpr_bond_energy_noalloc(int Lx, int Ly, const double* angles_dev, double q,
                                              double* e_bond_dev, void* stream)
{
    if (!angles_dev || !e_bond_dev) return err(MPR_ERR_INVALID_ARG, "angles or output pointer is NULL");
    if (Lx < 2 || Ly < 2) return err(MPR_ERR_INVALID_ARG, "both sides of the grid must be >= 2");
    if (!(q > 0.0 && q <= 1.0)) return err(MPR_ERR_INVALID_ARG, "q must lie in (0, 1]");
    const long long N = (long long)Lx * Ly;
    if (N > kMaxSites) {
        char buf[160];
        snprintf(buf, sizeof buf,
                 "grid of %lld sites exceeds the %lld sites (2^28) that the fixed scratch of "
                 "mpr_bond_energy_noalloc covers",
                 N, kMaxSites);
        return err(MPR_ERR_INVALID_ARG, buf);
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
        return err(MPR_ERR_CUDA, "no usable current CUDA device");
    mpr::energy::Sum* part = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (!g_addr[dev]) {
            void* p = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&p, g_bond_partials);
            if (e != cudaSuccess || !p) {
                char buf[160];
                snprintf(buf, sizeof buf, "cudaGetSymbolAddress(g_bond_partials): %s",
                         cudaGetErrorString(e));
                return err(MPR_ERR_CUDA, buf);
            }
            g_addr[dev] = static_cast<mpr::energy::Sum*>(p);
        }
        part = g_addr[dev];
    }
    // at most 152 x 6 blocks (their table copies are shared by 6 resident blocks per SM and all
    // strips of a block), as many as there are strips for their warps
    const int nsx = (Lx + 30) / 31, rows = mpr::energy::strip_rows(nsx, Ly);
    const long long strips = (long long)nsx * ((Ly + rows - 1) / rows);
    const int nblk = (int)std::min<long long>((strips + 7) / 8, 152 * 6);
    static_assert(152 * 6 <= kPartials, "one sum per block");
    const double n_bonds = (double)Lx * (Ly - 1) + (double)Ly * (Lx - 1);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    bond_partials<<<nblk, kThreads, 0, st>>>(Lx, Ly, rows, angles_dev, q,
                                            mpr::fixed::turn_factor(q), part);
    bond_final<<<1, kThreads, 0, st>>>(part, nblk, n_bonds, e_bond_dev);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        char buf[160];
        snprintf(buf, sizeof buf, "bond energy launch: %s", cudaGetErrorString(e));
        return err(MPR_ERR_CUDA, buf);
    }
    return MPR_OK;
}
