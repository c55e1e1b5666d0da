// mpr_resident.h -- host interface of the resident sweep kernel (mpr_resident.cuh): many hybrid
// sweeps of a small or middle-sized lattice in one launch. Not part of the public ABI.
#pragma once

#include "mpr_internal.h"

namespace mpr {
namespace resident {

constexpr int kFineThreads = 768;
constexpr int kCoarseThreads = 512;
constexpr size_t kMaxSmem = 227 * 1024;   // dynamic shared memory of a block, at most

// How a lattice is laid out over the blocks of the launch.
struct Plan {
    int nb = 0;          // blocks = bands of rows (0: the lattice does not run resident)
    bool fine = false;   // fine_kernel, else coarse_kernel
    bool cluster = false;   // fine_kernel: the blocks are one cluster; else a cooperative grid
    bool pair = false;   // coarse_kernel: a unit is a row pair (else one row) of four columns
    int threads = 0;
    int rows = 0;        // rows of the tallest band
    int depth = 1;       // passes between two exchanges of boundary rows (fine_kernel: even)
    int G = 0;           // groups of four half-lattice columns in a row
    size_t smem = 0;     // dynamic shared memory of a block
    int least[2] = {2, 2};   // fewest sweeps of a run that are worth the launch: plain, measured
    int runs = 1;        // runs in flight on the device, this one included, up to which it is the quicker kernel
};

struct Args {
    int Lx, Ly, Lxh, pitch, mpitch, G, rows, depth;
    void* ang[2];
    const uint32_t* mb[2];
    double* acc[2];
    float* acc_hi[2];
    float* acc_lo[2];
    float* er;                   // measured sweeps: FP32 sums of u_b . h_b per sweep, row and group
    unsigned long long* halo;    // grid: boundary rows in flight, [parity][band][side][row][4 G]
    uint32_t epoch;              // grid: tag of the last exchange before the launch
    int nsweeps;
    uint32_t seed_lo, seed_hi, sweep;
    float qf, nl2eTf;
    PhiloxSched keys;            // round keys (k[] only)
    int* err;
    long long wait_ns;           // limit of one wait for a neighbour
};

// Rows per side of an exchange every K passes: K of the colour moved last, K - 2 of the other one.
constexpr int halo_rows(int K) { return K > 1 ? 2 * K - 2 : 1; }

// Philox groups (row pairs of four columns) of a pass, at most.
constexpr int word_groups(int rows, int K, int G) { return (rows / 2 + 2 * (K / 2)) * G; }

// Exchanges of a launch of nsweeps sweeps at most (the epoch grows by as many).
constexpr uint32_t exchanges(int nsweeps) { return 2u * (uint32_t)nsweeps + 2u; }

Plan plan(const Layout& L, int store, int nsm);
// Bytes of the halo buffer of a plan (grid only).
size_t halo_bytes(const Plan& p);
// nsweeps hybrid sweeps; sample: 0 none, 1 FP64 sums, 2 Kahan sums (only with measure).
cudaError_t launch(const Plan& p, int store, bool measure, int sample, bool qhalf, const Args& a,
                   cudaStream_t st);
// Test hook: the same launch, plain, FP32 spins, q = 1/2, in which the first band sends nothing.
cudaError_t launch_stalled(const Plan& p, const Args& a, cudaStream_t st);
// The launch was refused because the device cannot hold its blocks at once (nothing ran).
inline bool too_large(cudaError_t e)
{
    return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorInvalidClusterSize ||
           e == cudaErrorLaunchOutOfResources;
}
// out[k] = the fixed-order sum of the n partials of sweep k, a block per sweep.
cudaError_t launch_sums(const void* part, int n, int nsweeps, bool e32, double* out, cudaStream_t st);
// The raw bond sums of nsweeps measured sweeps from their row sums, in the summation order of the
// tile kernel and its reduction (bit-identical energies): out[k] for sweep k. part: nsweeps x
// tiles partials of scratch.
cudaError_t launch_energies(const Layout& L, bool e32, const float* er, int nsweeps, void* part,
                            double* out, cudaStream_t st);

cudaError_t launch_f32(const Plan& p, bool measure, int sample, bool qhalf, const Args& a, cudaStream_t st);
cudaError_t launch_f16(const Plan& p, bool measure, int sample, bool qhalf, const Args& a, cudaStream_t st);
cudaError_t launch_bf16(const Plan& p, bool measure, int sample, bool qhalf, const Args& a, cudaStream_t st);

}  // namespace resident
}  // namespace mpr
