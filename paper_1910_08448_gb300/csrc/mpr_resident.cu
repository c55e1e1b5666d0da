// mpr_resident.cu -- host side of the resident sweep kernel: which lattices run resident and how
// they are laid out, the launch, and the energies of its measured sweeps.
#include "mpr_resident.h"

#include <algorithm>

#include "mpr_tile_f32.cuh"

namespace mpr {
namespace resident {
namespace {

constexpr int kCluster = 16;                 // blocks of a cluster (non-portable size)
constexpr size_t kSmem = 227 * 1024;         // shared memory of a block
constexpr int kThreads = 640;

size_t smem_of(int rows, int G, int store, bool cluster)
{
    const size_t P = 4 * (size_t)G + 8;
    return (cluster ? (size_t)4 * 4 * G * 8 : 0) + 4 * (size_t)(rows + 2) * P * 4 +
           2 * (size_t)rows * 4 * G * store_bytes(store) + 2 * (size_t)rows * G;
}

// Plan with at most `most` blocks: as few as the tallest band allows, bands of equal height but one
// row pair.
Plan bands(const Layout& L, int store, int most, bool cluster)
{
    Plan p;
    const int np = (L.Ly + 1) / 2;
    const int tall = (np + most - 1) / most;
    p.nb = (np + tall - 1) / tall;
    p.cluster = cluster;
    p.rows = 2 * tall;
    p.G = (L.Lxh + 3) / 4;
    const int groups = tall * p.G, one_role = (groups + 31) / 32 * 32;
    p.pair = 2 * one_role > kThreads;
    p.threads = std::min(kThreads, p.pair ? (groups + 31) / 32 * 32 : 2 * one_role);
    p.smem = smem_of(p.rows, p.G, store, cluster);
    if (p.smem > kSmem) p.nb = 0;
    return p;
}

// Tile (tx, ty) of a measured black pass: the thread's rows in the tile kernel's order, its warps by
// the same shuffles, the warps in order.
template <typename E>
__global__ void __launch_bounds__(256) tile_sums_kernel(const float* __restrict__ er, int Ly, int Lxh,
                                                        int G, int ntiles, E* __restrict__ part)
{
    __shared__ E ws[8];
    const int ntx = (Lxh + 127) / 128;
    const int tx = blockIdx.x % ntx, ty = blockIdx.x / ntx;
    const int rem = Lxh - tx * 128;
    const int tj = tx == ntx - 1 && rem <= 32 ? 32 : tx == ntx - 1 && rem <= 64 ? 64 : 128;
    const int per = tj / 4, rpt = tj / 32;   // lanes of a row, rows per thread
    const int lc = threadIdx.x % per, lr = threadIdx.x / per;
    const int row0 = (threadIdx.y * (32 / per) + lr) * rpt;
    const int g = tx * 32 + lc;
    const float* e = er + (size_t)blockIdx.y * Ly * G;
    E s = (E)0;
    for (int i = 0; i < rpt; ++i) {
        const int y = ty * 32 + row0 + (rpt % 2 == 0 ? i ^ 1 : i);
        if (y < Ly) s += g < G ? (E)e[(size_t)y * G + g] : (E)0;
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (threadIdx.x == 0) ws[threadIdx.y] = s;
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        E t = (E)0;
        for (int i = 0; i < 8; ++i) t += ws[i];
        part[(size_t)blockIdx.y * ntiles + blockIdx.x] = t;
    }
}

// The fixed-order sum of reduce_kernel (mpr_aux.cu), one block per sweep.
template <typename E>
__global__ void __launch_bounds__(256) sweep_sums_kernel(const E* __restrict__ part, int n,
                                                         double* __restrict__ out)
{
    __shared__ E ss[256];
    const E* p = part + (size_t)blockIdx.x * n;
    E s = (E)0;
    for (int i = threadIdx.x; i < n; i += 256) s += p[i];
    ss[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) ss[threadIdx.x] += ss[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = (double)ss[0];
}

template <typename E>
cudaError_t energies(const Layout& L, const float* er, int nsweeps, void* part, double* out,
                     cudaStream_t st)
{
    const int nt = sweep_f32_blocks(L), G = (L.Lxh + 3) / 4;
    E* p = static_cast<E*>(part);
    tile_sums_kernel<E><<<dim3(nt, nsweeps), dim3(32, 8), 0, st>>>(er, L.Ly, L.Lxh, G, nt, p);
    sweep_sums_kernel<E><<<nsweeps, 256, 0, st>>>(p, nt, out);
    return cudaGetLastError();
}

}  // namespace

Plan plan(const Layout& L, int store, int nsm)
{
    if (store == kF64 || nsm < 1) return Plan{};
    const long long sites = (long long)L.Lx * L.Ly;
    if (sites <= 128 * 128) {
        const Plan p = bands(L, store, kCluster, true);
        if (p.nb > 0) return p;
    }
    return bands(L, store, nsm, false);
}

size_t halo_bytes(const Plan& p) { return p.cluster ? 0 : (size_t)4 * p.nb * 4 * p.G * 8; }

cudaError_t launch(const Plan& p, int store, bool measure, int sample, bool qhalf, const Args& a,
                   cudaStream_t st)
{
    switch (store) {
    case kF32: return launch_f32(p, measure, sample, qhalf, a, st);
    case kF16: return launch_f16(p, measure, sample, qhalf, a, st);
    case kBF16: return launch_bf16(p, measure, sample, qhalf, a, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_energies(const Layout& L, bool e32, const float* er, int nsweeps, void* part,
                            double* out, cudaStream_t st)
{
    return e32 ? energies<float>(L, er, nsweeps, part, out, st)
               : energies<double>(L, er, nsweeps, part, out, st);
}

}  // namespace resident
}  // namespace mpr
