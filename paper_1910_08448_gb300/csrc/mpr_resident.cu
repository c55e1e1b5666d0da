// mpr_resident.cu -- host side of the resident sweep kernel: which lattices run resident and how
// they are laid out, the launch, and the energies of its measured sweeps.
#include "mpr_resident.h"

#include <algorithm>

#include "mpr_tile_f32.cuh"

namespace mpr {
namespace resident {
namespace {

constexpr int kCluster = 16;                 // blocks of a cluster (non-portable size)

// Bands of equal height but one row pair, at most `most` of them: as few as the tallest allows.
Plan bands(const Layout& L, int most)
{
    Plan p;
    const int np = (L.Ly + 1) / 2;
    const int tall = (np + most - 1) / most;
    p.nb = (np + tall - 1) / tall;
    p.rows = 2 * tall;
    p.G = (L.Lxh + 3) / 4;
    return p;
}

// fine_kernel with an exchange every `depth` passes; no plan where a band has fewer rows than that
// or its units and draws more warps than a block.
Plan fine_plan(const Layout& L, int most, bool cluster, int depth)
{
    Plan p = bands(L, most);
    p.fine = true;
    p.cluster = cluster;
    p.depth = depth;
    const int least = 2 * (((L.Ly + 1) / 2) / p.nb) - (L.Ly & 1);   // rows of the shortest band
    if (p.nb > 1 && least < depth) return Plan{};
    const int rows = p.rows + 2 * (depth - 1);
    const size_t G = (size_t)p.G, groups = (size_t)word_groups(p.rows, depth, p.G);
    const size_t warps = 2 * (((rows + 1) / 2 * 2 * G + 31) / 32) + (groups + 31) / 32;
    p.threads = 32 * (int)std::min<size_t>(warps, 64);
    p.smem = 2 * 4 * groups * 16 + (cluster ? (size_t)4 * halo_rows(depth) * 4 * G * 8 : 0) +
             4 * (size_t)(p.rows + 2 * depth) * (4 * G + 8) * 4;
    return p.threads <= kFineThreads && p.smem <= kMaxSmem ? p : Plan{};
}

Plan coarse_plan(const Layout& L, int store, int most)
{
    Plan p = bands(L, most);
    const size_t G = (size_t)p.G, n = (size_t)p.rows;
    const int groups = p.rows / 2 * p.G, one_role = (groups + 31) / 32 * 32;
    p.pair = 2 * one_role > kCoarseThreads;
    p.threads = std::min(kCoarseThreads, p.pair ? one_role : 2 * one_role);
    p.smem = 4 * (n + 2) * (4 * G + 8) * 4 + 2 * n * 4 * G * store_bytes(store) + 2 * n * G;
    // a second unit per thread only in bands taller than a pair: 5000 x 60 would leave most SMs idle and
    // take 5.7 us per pass (the tile kernel 4.1), 3500 x 600 takes 5.1 (6.0), 2300 x 1200 HDS 6.1 (9.1)
    if ((p.pair ? groups : 2 * one_role) > kCoarseThreads && p.rows == 2) return Plan{};
    return p.smem <= kMaxSmem ? p : Plan{};
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

// The sum of a sweep's n partials in a fixed order, one block per sweep: thread t adds partials t, t + 256,
// ..., then a tree (block_energy of the batched kernels adds in the same order).
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
    return launch_sums(p, nt, nsweeps, sizeof(E) == 4, out, st);
}

// A launch loads the lattice and stores it again; a run of two or three sweeps is worth that, except where the
// tile kernel's passes are short: a single column of 32-column tiles. us per call of 2 and 3 plain sweeps,
// resident / tile kernel: 64^2 25 / 21 and 25 / 24, 60 x 400 26 / 24 and 25 / 29, 60 x 20000 38 / 36 and 49 / 46 (2
// and 3 measured ones 72 / 62, 85 / 82), but 256^2 25 / 30, 777 x 523 25 / 30, 1400 x 1200 38 / 42; and 12 x 100000
// 50 / 90, whose tiles are mostly empty.
void set_least(const Layout& L, int nsm, Plan* p)
{
    if (p->nb == 0 || L.Lxh > 32) return;
    if ((L.Ly + 31) / 32 <= nsm) p->least[0] = p->nb <= kCluster ? 4 : 3;
    else if (p->pair && L.Lxh > 16) p->least[0] = p->least[1] = 4;
}

// A resident launch keeps its SMs until its last sweep, so launches of several handles take turns unless two of
// them fit side by side, where passes of the tile kernel share the device. us per run of 200 + 20 sweeps with 1 / 2
// / 3 / 4 / 8 handles on threads and streams of their own, resident and (tile kernel):
//   256^2 471 266 261 250 252 (1381 838 605 489 356): two fit (fine_kernel 80 registers, coarse_kernel 120)
//   400 x 300 589 532 552 538 549 (1403 830 605 496 364)
//   777 x 523 883 823 829 830 830 (1679 1165 797 620 493), 1024^2 1262 1175 1190 1191 1197 (1881 1328 1002 950 916)
//   1400 x 1200 2154 2101 2098 2090 2094 (2701 1649 1528 1486 1503)
// Mostly empty tiles (at most 16 half-columns) never catch up.
void set_runs(const Layout& L, int nsm, Plan* p)
{
    constexpr int kAny = 1 << 30;
    if (p->nb == 0) return;
    const int per_sm = p->threads <= (p->fine ? 352 : 256) && 2 * (p->smem + 1024) <= kMaxSmem ? 2 : 1;
    const long long sites = (long long)L.Lx * L.Ly;
    p->runs = 2 * p->nb <= per_sm * nsm || L.Lxh <= 16 ? kAny : p->fine ? 3 : sites <= 1100000 ? 2 : 1;
}

Plan any_plan(const Layout& L, int store, int nsm)
{
    // Us per plain pass, SDS, measured. One cluster while its blocks stay short of warps: exchanges
    // cost 0.25 us there and 0.5 us through L2, but 16 blocks hold little (64^2 0.49 against 0.82;
    // 128^2 0.65 against 0.78; 140^2, 840 threads, 0.87 against 0.85, sampled 1.25 against 1.10).
    // Exchanges every 4 passes while the additional rows are few (64^2: 0.49 against 0.52 every 2;
    // 128^2 in a cluster: 0.69 against 0.65; 90 x 768 on a grid: 0.89 against 0.93), else every 2.
    // coarse_kernel where the sites ask for more threads than a block has registers for (300 x 400
    // fine 1.21, coarse 1.40; 512 x 400 and wider only coarse).
    const Plan c4 = fine_plan(L, kCluster, true, 4);
    if (c4.nb > 0 && c4.threads <= 320) return c4;
    const Plan c2 = fine_plan(L, kCluster, true, 2);
    if (c2.nb > 0 && c2.threads <= 448) return c2;
    const Plan g4 = fine_plan(L, nsm, false, 4);
    if (g4.nb > 0 && g4.threads <= 544) return g4;
    const Plan g2 = fine_plan(L, nsm, false, 2);
    if (g2.nb > 0) return g2;
    return coarse_plan(L, store, nsm);
}

}  // namespace

Plan plan(const Layout& L, int store, int nsm)
{
    if (store == kF64 || nsm < 1) return Plan{};
    Plan p = any_plan(L, store, nsm);
    set_least(L, nsm, &p);
    set_runs(L, nsm, &p);
    return p;
}

size_t halo_bytes(const Plan& p)
{
    return p.cluster ? 0 : (size_t)4 * p.nb * halo_rows(p.depth) * 4 * p.G * 8;
}

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

cudaError_t launch_sums(const void* part, int n, int nsweeps, bool e32, double* out, cudaStream_t st)
{
    if (e32) sweep_sums_kernel<float><<<nsweeps, 256, 0, st>>>(static_cast<const float*>(part), n, out);
    else sweep_sums_kernel<double><<<nsweeps, 256, 0, st>>>(static_cast<const double*>(part), n, out);
    return cudaGetLastError();
}

cudaError_t launch_energies(const Layout& L, bool e32, const float* er, int nsweeps, void* part,
                            double* out, cudaStream_t st)
{
    return e32 ? energies<float>(L, er, nsweeps, part, out, st)
               : energies<double>(L, er, nsweeps, part, out, st);
}

}  // namespace resident
}  // namespace mpr
