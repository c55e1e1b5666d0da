// mpr_resident.cuh -- many hybrid sweeps of one lattice in one launch, the lattice held in shared
// memory (FP32 functions, uniform proposals). For lattices whose colour passes are too short to
// be worth a launch each.
//
// What bounds such a lattice: a chain of dependent passes. One launch per pass costs 2.3 us at
// 64^2 and 4 us at 256^2 (launch, staging from L2, one or two blocks deep in a serial chain of four
// rows per thread), where the arithmetic of a pass keeps the device busy for well under 1 us.
// Here a band of rows belongs to a block for the whole launch: unit vectors (cos, sin of q * phi)
// of both colours, the stored angles and the frozen bits stay in its shared memory, a thread owns
// one row (or a row pair) of four columns, and a pass needs only the boundary rows of the bands
// above and below. Those travel as 8-byte words, the new angle and the tag of the pass together, so
// one store and one polled load carry them and no fence is needed; between the blocks of a cluster
// they go straight into the neighbour's shared memory, between blocks of a grid through L2. A
// slot is reused only two passes later, which the neighbour's own words of the pass between imply.
// A wait is bounded: it ends with MPR_ERR_DEVICE_TIMEOUT in the error word, and every block leaves.
//
// The update is update_row of mpr_tile_f32.cuh, so states, samples and energies are the bits of
// the other FP32 kernels; a site's own sine and cosine are read back instead of computed again
// (79 instead of 89 instructions per site).
#pragma once

#include <cooperative_groups.h>

#include "mpr.h"
#include "mpr_resident.h"
#include "mpr_tile_f32.cuh"

namespace mpr {
namespace resident {
namespace {

using namespace f32;

constexpr int kMaxThreads = 640;

// Rows of one colour's unit vectors: row 0 and row rows + 1 are the neighbours' boundary rows.
struct Row {
    float* p;
    int stride;
    __device__ __forceinline__ float* operator[](int r) const { return p + r * stride; }
};
struct View {
    Row cs, sn;
};

__device__ __forceinline__ long long now_ns()
{
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Two tagged words (generic address: another block's shared memory, or global memory).
__device__ __forceinline__ void put2(unsigned long long* p, unsigned long long a, unsigned long long b)
{
    asm volatile("st.volatile.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void get2(const unsigned long long* p, unsigned long long& a,
                                     unsigned long long& b)
{
    asm volatile("ld.volatile.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ unsigned long long tagged(float v, uint32_t tag)
{
    return (unsigned long long)tag << 32 | __float_as_uint(v);
}

// Random words of the row with role ROW (0 first, 1 second of its Philox group).
template <int ROW>
__device__ __forceinline__ void row_words(const SweepArgs& a, uint32_t g, uint32_t h, RowIO& io)
{
    io.wl0 = group_call<true>(a, g, h, 0u);
    io.wl1 = group_call<true>(a, g, h, 1u);
    if constexpr (ROW == 1) io.w2 = group_call<true>(a, g, h, 2u);
}

template <typename S, bool MEASURE, int SAMPLE, int QM, bool PAIR, bool CLUSTER>
__global__ void __launch_bounds__(kMaxThreads, 1) resident_kernel(const __grid_constant__ Args A)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    namespace cg = cooperative_groups;
    const int G = A.G, P = 4 * G + 8, NR = A.rows;
    const int b = blockIdx.x, nb = gridDim.x;
    const int np = (A.Ly + 1) >> 1;                       // row pairs of the lattice
    const int h0 = (int)((long long)np * b / nb), h1 = (int)((long long)np * (b + 1) / nb);
    const int ya = 2 * h0, yb = min(2 * h1, A.Ly), nr = yb - ya;
    const int tid = threadIdx.x, T = blockDim.x;
    const float q = QM == 2 ? 0.5f : A.qf;

    // ---- shared memory
    unsigned char* sp = dsm;
    unsigned long long* mail = nullptr;   // cluster: the words of the two neighbours, [colour][side]
    if constexpr (CLUSTER) {
        mail = reinterpret_cast<unsigned long long*>(sp);
        sp += (size_t)4 * 4 * G * 8;
        for (int i = tid; i < 4 * 4 * G; i += T) mail[i] = 0ull;
    }
    const int plane = (NR + 2) * P;       // floats of one colour's cosines (then its sines)
    float* const units = reinterpret_cast<float*>(sp);
    auto view = [&](int c) {
        return View{Row{units + 2 * c * plane, P}, Row{units + (2 * c + 1) * plane, P}};
    };
    sp += (size_t)4 * plane * 4;
    S* const vals = reinterpret_cast<S*>(sp);   // the band's stored angles, row after row
    auto own = [&](int c, int r, int g) { return vals + ((size_t)(c * NR + r) * G + g) * 4; };
    sp += (size_t)2 * NR * 4 * G * sizeof(S);
    auto frozen = [&](int c, int r, int g) -> unsigned char& { return sp[(c * NR + r) * G + g]; };

    // ---- load: rows ya - 1 ... yb of both colours as unit vectors, the band's own values and bits
    for (int i = tid; i < 2 * (nr + 2) * (G + 2); i += T) {
        const int c = i / ((nr + 2) * (G + 2)), k = i - c * (nr + 2) * (G + 2);
        const int r = k / (G + 2), g = k - r * (G + 2) - 1;   // g = -1, G: the halo columns, empty
        const int y = ya - 1 + r;
        float vc[4] = {0.f, 0.f, 0.f, 0.f}, vs[4] = {0.f, 0.f, 0.f, 0.f};
        if (g >= 0 && g < G && y >= 0 && y < A.Ly) {
            Pack4<S> pk;
            load4(static_cast<const S*>(A.ang[c]) + (size_t)y * A.pitch + 4 * g, pk);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (2 * (4 * g + e) + ((y + c) & 1) < A.Lx)
                    __sincosf(q * load_as<float>(pk.s[e]), &vs[e], &vc[e]);
            if (r >= 1 && r <= nr) {
                store4(own(c, r - 1, g), pk);
                frozen(c, r - 1, g) =
                    (A.mb[c][(size_t)y * A.mpitch + (g >> 3)] >> (4 * g & 31)) & 0xFu;
            }
        }
        const View v = view(c);
        *reinterpret_cast<float4*>(&v.cs[r][4 + 4 * g]) = make_float4(vc[0], vc[1], vc[2], vc[3]);
        *reinterpret_cast<float4*>(&v.sn[r][4 + 4 * g]) = make_float4(vs[0], vs[1], vs[2], vs[3]);
    }
    if constexpr (CLUSTER) cg::this_cluster().sync();   // every block's mail is empty

    SweepArgs a{};
    a.Lx = A.Lx;
    a.Ly = A.Ly;
    a.Lxh = A.Lxh;
    a.pitch = A.pitch;
    a.mpitch = A.mpitch;
    a.qf = A.qf;
    a.nl2eTf = A.nl2eTf;
    a.ph = A.keys;
    const int NG = (h1 - h0) * G;                 // groups (row pairs of four columns) of the band
    const int NGp = (NG + 31) & ~31;              // one role of a row per warp
    const int U = PAIR ? NG : 2 * NGp;            // units of a pass
    double e_d = 0.0;   // unused: the row sums go to A.er
    float e_f = 0.0f;
    int n_acc = 0;      // unused: uniform proposals
    bool bad = false;

#pragma unroll 1
    for (int pass = 0; pass < 2 * A.nsweeps; ++pass) {
        const int c = pass & 1, cb = c ^ 1;
        const View vo = view(c), vb = view(cb);
        const uint32_t sweep = A.sweep + (uint32_t)(pass >> 1);
        a.colour = c;
        a.acc = A.acc[c];
        a.acc_hi = A.acc_hi[c];
        a.acc_lo = A.acc_lo[c];
        const uint64_t m = (uint64_t)0xCD9E8D57u * sweep;
        a.ph.a = (uint32_t)(m >> 32) ^ A.seed_lo;
        a.ph.b = (uint32_t)m;
        a.ph.c = (((uint32_t)kTagMetropolis << 1) | (uint32_t)c) ^ A.seed_hi;
        const uint32_t tag = (CLUSTER ? 0u : A.epoch) + (uint32_t)pass;   // of the pass before

        // the first unit's random words do not wait for anybody
        RowIO io;
        auto words = [&](int u) {
            if constexpr (PAIR) {
                const int pr = u / G;
                row_words<1>(a, (uint32_t)(u - pr * G), (uint32_t)(h0 + pr), io);
            } else {
                const int role = u >= NGp ? 1 : 0, w = u - role * NGp, pr = w / G;
                if (role) row_words<1>(a, (uint32_t)(w - pr * G), (uint32_t)(h0 + pr), io);
                else row_words<0>(a, (uint32_t)(w - pr * G), (uint32_t)(h0 + pr), io);
            }
        };
        if (tid < U) words(tid);

        // ---- the neighbours' boundary rows of the other colour, moved in the previous pass
        if (pass > 0) {
            for (int i = tid; i < 4 * G; i += T) {
                const int side = i >= 2 * G ? 1 : 0, j = 2 * (i - side * 2 * G);
                if (side ? b + 1 >= nb : b == 0) continue;
                const unsigned long long* p =
                    CLUSTER ? mail + (size_t)(cb * 2 + side) * 4 * G + j
                            : A.halo + ((size_t)(cb * nb + b) * 2 + side) * 4 * G + j;
                unsigned long long w0, w1;
                long long t0 = 0;
                for (int spin = 0;; ++spin) {
                    get2(p, w0, w1);
                    if ((uint32_t)(w0 >> 32) == tag && (uint32_t)(w1 >> 32) == tag) break;
                    if ((spin & 255) == 255) {
                        const long long t = now_ns();
                        if (t0 == 0) t0 = t;
                        if (t - t0 > A.wait_ns || *(volatile int*)A.err) {
                            atomicCAS(A.err, 0, (int)MPR_ERR_DEVICE_TIMEOUT);
                            bad = true;
                            break;
                        }
                    }
                }
                const int y = side ? yb : ya - 1, r = side ? nr + 1 : 0;
                float c0 = 0.f, s0 = 0.f, c1 = 0.f, s1 = 0.f;
                if (2 * j + ((y + cb) & 1) < A.Lx) __sincosf(q * __uint_as_float((uint32_t)w0), &s0, &c0);
                if (2 * j + 2 + ((y + cb) & 1) < A.Lx) __sincosf(q * __uint_as_float((uint32_t)w1), &s1, &c1);
                *reinterpret_cast<float2*>(&vb.cs[r][4 + j]) = make_float2(c0, c1);
                *reinterpret_cast<float2*>(&vb.sn[r][4 + j]) = make_float2(s0, s1);
            }
        }
        // also: this block's own rows of the other colour are complete
        if (__syncthreads_or(bad)) break;

        // ---- the units of this pass
        for (int u = tid; u < U; u += T) {
            if (u != tid) words(u);
            // one row of the unit: y = ya + r, columns 4g ... 4g + 3, role O
            auto row = [&](auto role, int pr, int g, GroupCarry& gc) {
                constexpr int O = decltype(role)::value;
                const int r = 2 * pr + (O == 0 ? c : 1 - c), y = ya + r;
                if (y >= A.Ly) return;
                Pack4<S> pk;
                load4(own(c, r, g), pk);
                io.oc = *reinterpret_cast<const float4*>(&vo.cs[r + 1][4 + 4 * g]);
                io.os = *reinterpret_cast<const float4*>(&vo.sn[r + 1][4 + 4 * g]);
                update_row<S, MEASURE, SAMPLE, true, O, false, QM, O, false>(
                    a, y, r, 4 * g, 4 * g, pk, frozen(c, r, g), vb, e_d, e_f, 0.0f, n_acc, gc, io);
                // boundary rows first: the neighbours wait for them
                const bool up = r == 0 && b > 0, dn = r == nr - 1 && b + 1 < nb;
                if (up || dn) {
                    unsigned long long w[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) w[k] = tagged(load_as<float>(pk.s[k]), tag + 1u);
                    auto send = [&](int to, int side) {
                        unsigned long long* p;
                        if constexpr (CLUSTER)
                            p = cg::this_cluster().map_shared_rank(mail, to) +
                                (size_t)(c * 2 + side) * 4 * G + 4 * g;
                        else
                            p = A.halo + ((size_t)(c * nb + to) * 2 + side) * 4 * G + 4 * g;
                        put2(p, w[0], w[1]);
                        put2(p + 2, w[2], w[3]);
                    };
                    if (up) send(b - 1, 1);
                    if (dn) send(b + 1, 0);
                }
                store4(own(c, r, g), pk);
                *reinterpret_cast<float4*>(&vo.cs[r + 1][4 + 4 * g]) =
                    make_float4(io.nc[0], io.nc[1], io.nc[2], io.nc[3]);
                *reinterpret_cast<float4*>(&vo.sn[r + 1][4 + 4 * g]) =
                    make_float4(io.ns[0], io.ns[1], io.ns[2], io.ns[3]);
                if constexpr (MEASURE) {
                    if (c == 1) A.er[((size_t)(pass >> 1) * A.Ly + y) * G + g] = io.er;
                }
                sample_row<SAMPLE>(a, (size_t)y * A.pitch + 4 * g, io.fsamp);
            };
            using First = std::integral_constant<int, 0>;
            using Second = std::integral_constant<int, 1>;
            GroupCarry gc{0u, 0u, 0u, 0u};
            carry_call0(gc, io.wl0);
            carry_call1(gc, io.wl1);
            if constexpr (PAIR) {
                const int pr = u / G, g = u - pr * G;
                row(First{}, pr, g, gc);
                row(Second{}, pr, g, gc);
            } else {
                const int role = u >= NGp ? 1 : 0, w = u - role * NGp, pr = w / G, g = w - pr * G;
                if (w < NG) {
                    if (role) row(Second{}, pr, g, gc);
                    else row(First{}, pr, g, gc);
                }
            }
        }
    }

    // ---- the band's rows back to the layout (the neighbours read their first halo rows before
    // they sent the words that the last pass here waited for)
    __syncthreads();
    for (int i = tid; i < 2 * nr * G; i += T) {
        const int c = i / (nr * G), k = i - c * nr * G, r = k / G, g = k - r * G;
        Pack4<S> pk;
        load4(own(c, r, g), pk);
        store4(static_cast<S*>(A.ang[c]) + (size_t)(ya + r) * A.pitch + 4 * g, pk);
    }
    if constexpr (CLUSTER) cg::this_cluster().sync();   // no block leaves while its mail is written
}

template <typename S, bool MEASURE, int SAMPLE, int QM, bool PAIR, bool CLUSTER>
cudaError_t go(const Plan& p, const Args& a, cudaStream_t st)
{
    auto kern = resident_kernel<S, MEASURE, SAMPLE, QM, PAIR, CLUSTER>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(p.nb);
    cfg.blockDim = dim3(p.threads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (CLUSTER) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)p.nb;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
    } else {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

template <typename S, bool MEASURE, int SAMPLE, int QM>
cudaError_t go_shape(const Plan& p, const Args& a, cudaStream_t st)
{
    if (p.cluster)
        return p.pair ? go<S, MEASURE, SAMPLE, QM, true, true>(p, a, st)
                      : go<S, MEASURE, SAMPLE, QM, false, true>(p, a, st);
    return p.pair ? go<S, MEASURE, SAMPLE, QM, true, false>(p, a, st)
                  : go<S, MEASURE, SAMPLE, QM, false, false>(p, a, st);
}

template <typename S, int QM>
cudaError_t go_mode(const Plan& p, bool measure, int sample, const Args& a, cudaStream_t st)
{
    if (!measure) return sample ? cudaErrorInvalidValue : go_shape<S, false, 0, QM>(p, a, st);
    if (sample == 0) return go_shape<S, true, 0, QM>(p, a, st);
    if (sample == 1) return go_shape<S, true, 1, QM>(p, a, st);
    return go_shape<S, true, 2, QM>(p, a, st);
}

template <typename S>
cudaError_t go_store(const Plan& p, bool measure, int sample, bool qhalf, const Args& a, cudaStream_t st)
{
    return qhalf ? go_mode<S, 2>(p, measure, sample, a, st) : go_mode<S, 0>(p, measure, sample, a, st);
}

}  // namespace
}  // namespace resident
}  // namespace mpr
