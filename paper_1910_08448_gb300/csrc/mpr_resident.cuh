// mpr_resident.cuh -- many hybrid sweeps of one lattice in one launch, the lattice held on the SMs
// (FP32 functions, uniform proposals). For lattices whose colour passes are too short to be worth a
// launch each.
//
// What bounds such a lattice: a chain of dependent passes. One launch per pass costs 2.1 us at
// 64^2 and 4 us at 777 x 523 (launch, staging from L2, one or two blocks deep in a serial chain of
// four rows per thread), where the arithmetic of a pass keeps the device busy for well under 1 us.
// Here a band of rows belongs to a block for the whole launch: unit vectors (cos, sin of q * phi)
// of both colours stay in its shared memory, and a pass needs only boundary rows of the bands above
// and below. Those travel as 8-byte words, the new angle and a tag together, so one store and one
// polled load carry them and no fence is needed; between the blocks of a cluster they go straight
// into the neighbour's shared memory, between blocks of a grid through L2. Slots alternate by
// the tag's parity: one is written again only after the neighbour's words of the exchange between,
// which imply that it was read. A wait is bounded: it ends with MPR_ERR_DEVICE_TIMEOUT in the error
// word, and every block leaves.
//
// Two kernels, by the length of a pass:
//
// fine_kernel: a thread owns two columns of a row for the whole launch, their angles and unit vectors
// in registers; other warps draw the next pass's uniforms meanwhile. A block also updates K - 1
// rows on either side of its band (same uniforms, same bits), so rows are exchanged every K passes
// only. For blocks whose sites give every thread one unit: there the length of a thread's serial
// chain is what a pass costs: with index arithmetic in the loop and four sites per thread that
// chain was 1.1 us at 64^2, now 0.49 us per pass; 256^2 0.91 (1.7 with four sites per thread and an
// exchange every pass).
//
// coarse_kernel: a thread owns four columns of a row or of a row pair (three Philox calls for eight
// sites), rows are exchanged every pass and waited for by the threads that read them, so the
// interior of the band runs on. For wider blocks, where instructions per site are what counts:
// 777 x 523 1.76 us per pass (one launch per pass 4.2), 1024^2 2.53 (3.7); sampled, the FP64
// sums loaded before the moves, 4.57 (9.5).
//
// The arithmetic is move_pair of mpr_tile_f32.cuh, so states, samples and energies are the bits of
// the other FP32 kernels; a site's own sine and cosine are kept instead of computed again.
#pragma once

#include <cooperative_groups.h>

#include "mpr.h"
#include "mpr_resident.h"
#include "mpr_tile_f32.cuh"

namespace mpr {
namespace resident {
namespace {

using namespace f32;

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

// Polls two words of a neighbour until both carry the tag; false when the wait ran out.
__device__ __forceinline__ bool wait2(const Args& A, const unsigned long long* p, uint32_t tag, float& x,
                                      float& y)
{
    long long t0 = 0;
    for (int spin = 0;; ++spin) {
        unsigned long long w0, w1;
        get2(p, w0, w1);
        x = __uint_as_float((uint32_t)w0);
        y = __uint_as_float((uint32_t)w1);
        if ((uint32_t)(w0 >> 32) == tag && (uint32_t)(w1 >> 32) == tag) return true;
        if ((spin & 255) == 255) {
            const long long t = now_ns();
            if (t0 == 0) t0 = t;
            if (t - t0 > A.wait_ns || *(volatile int*)A.err) {
                atomicCAS(A.err, 0, (int)MPR_ERR_DEVICE_TIMEOUT);
                return false;
            }
        }
    }
}

template <typename S> struct alignas(2 * sizeof(S)) Pack2 {
    S x, y;
};

// The band of rows of a block.
struct Band {
    int b, nb, ya, yb;
    __device__ __forceinline__ explicit Band(const Args& A) : b(blockIdx.x), nb(gridDim.x)
    {
        const int np = (A.Ly + 1) >> 1;   // row pairs of the lattice
        ya = 2 * (int)((long long)np * b / nb);
        yb = min(2 * (int)((long long)np * (b + 1) / nb), A.Ly);
    }
};

// Words of row `row` of the exchange with tag parity 0, in the slots of block `to`, side 0 (rows
// above its band) or 1; parity 1 lies slot_stride further.
template <bool CLUSTER>
__device__ __forceinline__ unsigned long long* slot(const Args& A, unsigned long long* mail, int to, int side,
                                                    int row)
{
    const int RS = halo_rows(A.depth);
    if constexpr (CLUSTER)
        return cooperative_groups::this_cluster().map_shared_rank(mail, to) +
               (size_t)(side * RS + row) * 4 * A.G;
    else
        return A.halo + (((size_t)to * 2 + side) * RS + row) * 4 * A.G;
}
template <bool CLUSTER> __device__ __forceinline__ size_t slot_stride(const Args& A, int nb)
{
    return (size_t)(CLUSTER ? 1 : nb) * 2 * halo_rows(A.depth) * 4 * A.G;
}

// cos and sin of q * x, (0, 0) where there is no site
__device__ __forceinline__ void unit_of(float q, float x, bool exists, float& c, float& s)
{
    __sincosf(q * x, &s, &c);
    c = exists ? c : 0.0f;
    s = exists ? s : 0.0f;
}

// The round of Philox keys and counters for colour c of sweep `sweep`.
__device__ __forceinline__ PhiloxSched pass_keys(const Args& A, uint32_t sweep, int c)
{
    PhiloxSched ph = A.keys;
    const uint64_t m = (uint64_t)0xCD9E8D57u * sweep;
    ph.a = (uint32_t)(m >> 32) ^ A.seed_lo;
    ph.b = (uint32_t)m;
    ph.c = (((uint32_t)kTagMetropolis << 1) | (uint32_t)c) ^ A.seed_hi;
    return ph;
}

// 1 + u of the proposals (x, y) and acceptances (z, w) of a unit: sites 2H, 2H + 1 of the row with
// role ROW in its Philox group, from the group's three calls (see GroupCarry).
template <int ROW, int H>
__device__ __forceinline__ float4 unit_uniforms(const uint4& w0, const uint4& w1, const uint4& w2)
{
    if constexpr (ROW == 0) {
        const uint4 w = H == 0 ? w0 : w1;
        return make_float4(one_plus_uniform_f(w.x), one_plus_uniform_f(w.z), one_plus_uniform_f(w.y),
                           one_plus_uniform_f(w.w));
    } else {
        GroupCarry gc;
        carry_call0(gc, w0);
        carry_call1(gc, w1);
        if constexpr (H == 0)
            return make_float4(one_plus_uniform_f(w2.x), one_plus_uniform_f(w2.y),
                               one_plus_low23_f(gc.a0), one_plus_low23_f(gc.a1));
        else
            return make_float4(one_plus_uniform_f(w2.z), one_plus_uniform_f(w2.w),
                               one_plus_low23_f(low3(gc.p2, w2.x)),
                               one_plus_low23_f(low3(low2(w2.y, w2.z), w2.w)));
    }
}

// STALL: test hook, the first band sends nothing (kernels of their own: the condition alone cost the others 3 %
// at 64^2).
template <typename S, bool MEASURE, int SAMPLE, int QM, bool CLUSTER, bool STALL = false>
__global__ void __launch_bounds__(kFineThreads, 1) fine_kernel(const __grid_constant__ Args A)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    const Band B(A);
    const int b = B.b, nb = B.nb, ya = B.ya, yb = B.yb, K = A.depth;   // K is even
    const int G = A.G, G2 = 2 * G, P = 4 * G + 8;
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const float q = QM == 2 ? 0.5f : A.qf;
    const float width = QM == 2 ? 3.14159265358979324f : kTwoPiF * q;
    const float inv_q = QM == 2 ? 2.0f : 1.0f / q;

    // ---- shared memory: uniforms of two passes [colour][role][group][half], cluster mail, unit
    // vectors [colour][cos, sin][row ya - K ... yb + K - 1][column]
    float4* const uni = reinterpret_cast<float4*>(dsm);
    const int NU = 4 * word_groups(A.rows, K, G);
    unsigned long long* const mail = reinterpret_cast<unsigned long long*>(uni + 2 * NU);
    const size_t nmail = CLUSTER ? 2 * slot_stride<true>(A, nb) : 0;
    float* const units = reinterpret_cast<float*>(mail + nmail);
    const int plane = (A.rows + 2 * K) * P;
    for (int i = tid; i < (int)nmail; i += T) mail[i] = 0ull;
    for (int i = tid; i < 4 * plane; i += T) units[i] = 0.0f;
    __syncthreads();

    // ---- this thread's part: a unit (row y, columns jc, jc + 1; even rows' warps first, so that a
    // warp's rows have one role) or a Philox group
    const int R0 = max(0, ya - (K - 1)), R1 = min(A.Ly, yb + (K - 1));
    const int e0 = (R0 + 1) >> 1, ne = ((R1 + 1) >> 1) - e0, o0 = R0 >> 1, no = (R1 >> 1) - o0;
    const int We = (ne * G2 + 31) >> 5, Wo = (no * G2 + 31) >> 5;
    const int P0 = R0 >> 1, nP = ((R1 + 1) >> 1) - P0;
    const bool mover = warp < We + Wo;
    int y = 0, jc = 0;
    bool unit = false;
    uint32_t dg = 0, dh = 0;
    float4* draw_to = nullptr;   // of colour 0
    if (mover) {
        const bool odd = warp >= We;
        const int idx = odd ? tid - 32 * We : tid, k = idx / G2;
        unit = k < (odd ? no : ne);
        jc = 2 * (idx - k * G2);
        y = odd ? 2 * (o0 + k) + 1 : 2 * (e0 + k);
    } else {
        const int idx = tid - 32 * (We + Wo);
        if (idx < nP * G) {
            const int pr = idx / G;
            dg = (uint32_t)(idx - pr * G);
            dh = (uint32_t)(P0 + pr);
            draw_to = uni + 2 * idx;
        }
    }
    const int above = y - ya, below = yb - 1 - y;             // rows of the band on either side
    const int dist = max(0, max(-above, -below));             // rows outside the band
    const bool mine = unit && dist == 0;
    float* const pu = units + (y - (ya - K)) * P + 4 + jc;    // column jc of the unit's row
    auto plane_of = [&](int c, int s) { return (2 * c + s) * plane; };
    auto exists = [&](int c, int row, int e) { return 2 * (jc + e) + ((row + c) & 1) < A.Lx; };
    auto put_units = [&](int c, int row, float x0, float x1, float2& cs, float2& sn) {
        unit_of(q, x0, exists(c, row, 0), cs.x, sn.x);
        unit_of(q, x1, exists(c, row, 1), cs.y, sn.y);
        float* const p = pu + (row - y) * P;
        *reinterpret_cast<float2*>(p + plane_of(c, 0)) = cs;
        *reinterpret_cast<float2*>(p + plane_of(c, 1)) = sn;
    };
    // stored angles and unit vectors of the unit's four sites, and what never changes of them
    float2 f[2] = {}, uc[2] = {}, us[2] = {};
    unsigned free_ = 0, there = 0;                            // bits 2c, 2c + 1
    const int edge = dist == K - 1 ? (above < 0 ? -1 : 1) : 0;   // toward row K, nobody's unit
    if (unit) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const Pack2<S> pk = *reinterpret_cast<const Pack2<S>*>(static_cast<const S*>(A.ang[c]) +
                                                                   (size_t)y * A.pitch + jc);
            f[c] = make_float2(load_as<float>(pk.x), load_as<float>(pk.y));
            put_units(c, y, f[c].x, f[c].y, uc[c], us[c]);
            const unsigned bits = A.mb[c][(size_t)y * A.mpitch + (jc >> 5)] >> (jc & 31);
            free_ |= (~bits & 3u) << (2 * c);
            there |= ((exists(c, y, 0) ? 1u : 0u) | (exists(c, y, 1) ? 2u : 0u)) << (2 * c);
            const int ye = y + edge;
            if (edge && ye >= 0 && ye < A.Ly) {
                const Pack2<S> pe = *reinterpret_cast<const Pack2<S>*>(static_cast<const S*>(A.ang[c]) +
                                                                       (size_t)ye * A.pitch + jc);
                float2 cs, sn;
                put_units(c, ye, load_as<float>(pe.x), load_as<float>(pe.y), cs, sn);
            }
        }
    }
    // boundary rows: where this unit's words go and come from (of the colour moved last; row
    // dist - 1, the other colour K - 1 rows further)
    const bool up = mine && above < K && b > 0, down = mine && below < K && b + 1 < nb && !(STALL && b == 0);
    unsigned long long* const to_up = slot<CLUSTER>(A, mail, up ? b - 1 : b, 1, up ? above : 0) + jc;
    unsigned long long* const to_down = slot<CLUSTER>(A, mail, down ? b + 1 : b, 0, down ? below : 0) + jc;
    const bool take = unit && dist > 0;
    const unsigned long long* const from =
        slot<CLUSTER>(A, mail, b, above < 0 ? 0 : 1, take ? dist - 1 : 0) + jc;
    const size_t parity = slot_stride<CLUSTER>(A, nb), other = (size_t)(K - 1) * 4 * G;
    const int par = y & 1;   // role of the row: its parity for colour 0, the opposite for colour 1
    const float4* const uu = uni + 2 * ((y >> 1) - P0) * G + (jc >> 1);

    // the uniforms of colour c of a sweep
    auto draw = [&](uint32_t sweep, int c) {
        const PhiloxSched ph = pass_keys(A, sweep, c);
        const uint4 w0 = pair_words(dg, dh, ph, 0u), w1 = pair_words(dg, dh, ph, 1u),
                    w2 = pair_words(dg, dh, ph, 2u);
        float4* const o = draw_to + c * NU;
        o[0] = unit_uniforms<0, 0>(w0, w1, w2);
        o[1] = unit_uniforms<0, 1>(w0, w1, w2);
        o[NU / 2] = unit_uniforms<1, 0>(w0, w1, w2);
        o[NU / 2 + 1] = unit_uniforms<1, 1>(w0, w1, w2);
    };
    if (draw_to) draw(A.sweep, 0);
    if constexpr (CLUSTER) cooperative_groups::this_cluster().sync();   // every block's mail is empty

    int n_acc = 0;            // unused: uniform proposals
    uint32_t tag = A.epoch;   // of the exchange before the current round of K passes
    int j = 0;                // pass within the round
    bool dead = false;
#pragma unroll 1
    for (int sw = 0; sw < A.nsweeps; ++sw) {
        const bool more = 2 * sw - j + K < 2 * A.nsweeps;   // another round follows this one
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (c == 0 && j == 0 && sw > 0) {
                // ---- a round begins: the neighbours' rows. Of colour 1 (moved last) distances
                // 1 ... K, of colour 0 distances 2 ... K - 1 (the row at distance 1 was moved here
                // too, after its neighbours had their last move). Nobody reads them now.
                bool bad = false;
                if (take) {
                    const unsigned long long* const p = from + (tag & 1u) * parity;
                    bad = !wait2(A, p, tag, f[1].x, f[1].y);
                    put_units(1, y, f[1].x, f[1].y, uc[1], us[1]);
                    if (dist >= 2) {
                        bad |= !wait2(A, p + other, tag, f[0].x, f[0].y);
                        put_units(0, y, f[0].x, f[0].y, uc[0], us[0]);
                    }
                    const int ye = y + edge;
                    if (edge && ye >= 0 && ye < A.Ly) {
                        float x0, x1;
                        float2 cs, sn;
                        bad |= !wait2(A, p + 4 * G, tag, x0, x1);
                        put_units(1, ye, x0, x1, cs, sn);
                    }
                }
                if (__syncthreads_or(bad)) {
                    dead = true;
                    break;
                }
            } else {
                __syncthreads();   // the other colour and this pass's uniforms are complete
            }
            if (mover) {
                float er = 0.0f;
                if (unit && dist <= K - 1 - j) {
                    const bool o = (par ^ c) != 0;   // second row of its Philox group; columns shift
                    const size_t at = (size_t)y * A.pitch + jc;
                    double2 sd{};
                    float2 sh{}, sl{};
                    if (SAMPLE && mine) {   // the sums, while the rest runs
                        if constexpr (SAMPLE == 1) sd = *reinterpret_cast<const double2*>(A.acc[c] + at);
                        if constexpr (SAMPLE == 2) {
                            sh = *reinterpret_cast<const float2*>(A.acc_hi[c] + at);
                            sl = *reinterpret_cast<const float2*>(A.acc_lo[c] + at);
                        }
                    }
                    const float4 u = uu[c * NU + (o ? NU / 2 : 0)];
                    // local fields, in the order of update_row: ((left + right) + up) + down
                    auto field = [&](const float* v) {
                        const float2 up2 = *reinterpret_cast<const float2*>(v - P);
                        const float2 mid = *reinterpret_cast<const float2*>(v);
                        const float2 dn2 = *reinterpret_cast<const float2*>(v + P);
                        const float e = v[o ? 2 : -1];
                        const float m2 = mid.x + mid.y, me = (o ? mid.y : mid.x) + e;
                        return add2(add2(make_float2(o ? m2 : me, o ? me : m2), up2), dn2);
                    };
                    const float2 hx = field(pu + plane_of(1 - c, 0)), hy = field(pu + plane_of(1 - c, 1));
                    const bool upd0 = free_ >> (2 * c) & 1u, upd1 = free_ >> (2 * c) & 2u;
                    const bool ex0 = there >> (2 * c) & 1u, ex1 = there >> (2 * c) & 2u;
                    float2 fn = move_pair<sizeof(S), true, false, QM, false>(
                        hx, hy, make_float2(u.x, u.y), make_float2(u.z, u.w), f[c], upd0, upd1, q,
                        A.nl2eTf, width, inv_q, 0.0f, n_acc, uc[c], us[c]);
                    // as stored (a frozen site's own value converts back to itself)
                    fn = make_float2(load_as<float>(store_from<S>(fn.x)), load_as<float>(store_from<S>(fn.y)));
                    f[c] = fn;
                    // rows that the neighbours need for their next round, as soon as this round is
                    // done with them
                    if (more && (up || down) && (c == 1 ? j == K - 1 : j == K - 2)) {
                        const unsigned long long w0 = tagged(fn.x, tag + 1u), w1 = tagged(fn.y, tag + 1u);
                        const size_t off = ((tag + 1u) & 1u) * parity;
                        if (c == 1) {
                            if (up) put2(to_up + off, w0, w1);
                            if (down) put2(to_down + off, w0, w1);
                        } else {   // row K + d - 1 for rows d = 1 ... K - 2 from the boundary
                            if (up && above >= 1 && above < K - 1) put2(to_up + off + other, w0, w1);
                            if (down && below >= 1 && below < K - 1) put2(to_down + off + other, w0, w1);
                        }
                    }
                    const float2 qn = mul2(splat(q), fn);
                    float2 cs, sn;
                    __sincosf(qn.x, &sn.x, &cs.x);
                    __sincosf(qn.y, &sn.y, &cs.y);
                    cs = make_float2(ex0 ? cs.x : 0.0f, ex1 ? cs.y : 0.0f);
                    sn = make_float2(ex0 ? sn.x : 0.0f, ex1 ? sn.y : 0.0f);
                    uc[c] = cs;
                    us[c] = sn;
                    *reinterpret_cast<float2*>(pu + plane_of(c, 0)) = cs;
                    *reinterpret_cast<float2*>(pu + plane_of(c, 1)) = sn;
                    if constexpr (MEASURE) {
                        const float2 e2 = fma2(cs, hx, mul2(sn, hy));
                        er = (ex0 ? e2.x : 0.0f) + (ex1 ? e2.y : 0.0f);
                    }
                    if (SAMPLE && mine) {   // frozen sites add 0
                        const float f0 = upd0 ? fn.x : 0.0f, f1 = upd1 ? fn.y : 0.0f;
                        if constexpr (SAMPLE == 1) {
                            sd.x += (double)f0;
                            sd.y += (double)f1;
                            *reinterpret_cast<double2*>(A.acc[c] + at) = sd;
                        }
                        if constexpr (SAMPLE == 2) {   // Kahan, as sample_row
                            const float y0 = f0 - sl.x, t0 = sh.x + y0, y1 = f1 - sl.y, t1 = sh.y + y1;
                            *reinterpret_cast<float2*>(A.acc_lo[c] + at) =
                                make_float2((t0 - sh.x) - y0, (t1 - sh.y) - y1);
                            *reinterpret_cast<float2*>(A.acc_hi[c] + at) = make_float2(t0, t1);
                        }
                    }
                }
                if constexpr (MEASURE) {   // the terms of four columns: (0 + 1) + (2 + 3)
                    if (c == 1) {
                        er += __shfl_xor_sync(0xffffffffu, er, 1);
                        if (mine && !(lane & 1))
                            A.er[((size_t)sw * A.Ly + y) * G + (jc >> 2)] = er;
                    }
                }
            } else if (draw_to) {   // of the next pass
                draw(A.sweep + (uint32_t)(sw + c), 1 - c);
            }
            ++j;
        }
        if (dead) break;
        if (j == K) {
            j = 0;
            ++tag;
        }
    }

    // ---- the band's rows back to the layout (the neighbours loaded their rows before they sent the
    // words of the first exchange, and every launch has one)
    if (mine) {
#pragma unroll
        for (int c = 0; c < 2; ++c)
            *reinterpret_cast<Pack2<S>*>(static_cast<S*>(A.ang[c]) + (size_t)y * A.pitch + jc) =
                Pack2<S>{store_from<S>(f[c].x), store_from<S>(f[c].y)};
    }
    if constexpr (CLUSTER) cooperative_groups::this_cluster().sync();   // no mail to a block that left
}

// The moves of one colour in four columns of row y (shared row r), whose unit vectors of the other
// colour are complete around it. O: the row's role; w0, w1, w2: the
// random words of its Philox group.
template <typename S, bool MEASURE, int QM, int O>
struct QuadRow {
    float2 fn[2], cs[2], sn[2], samp[2];
    float er;
    __device__ __forceinline__ void run(const Args& A, const View& vb, const View& vo, int r, int g,
                                        const S* stored, unsigned bits, const uint4& w0, const uint4& w1,
                                        const uint4& w2, float q, float width, float inv_q)
    {
        const int lj = 4 * g;
        float2 hx[2], hy[2];
        auto field = [&](const Row& v, float2* h) {
            const float4 u = *reinterpret_cast<const float4*>(&v[r - 1][4 + lj]);
            const float4 m = *reinterpret_cast<const float4*>(&v[r][4 + lj]);
            const float4 d = *reinterpret_cast<const float4*>(&v[r + 1][4 + lj]);
            const float e = v[r][O ? 8 + lj : 3 + lj];
            const float xy = m.x + m.y, yz = m.y + m.z, zw = m.z + m.w;
            const float2 a = O ? make_float2(xy, yz) : make_float2(e + m.x, xy);
            const float2 b = O ? make_float2(zw, m.w + e) : make_float2(yz, zw);
            h[0] = add2(add2(a, make_float2(u.x, u.y)), make_float2(d.x, d.y));
            h[1] = add2(add2(b, make_float2(u.z, u.w)), make_float2(d.z, d.w));
        };
        field(vb.cs, hx);
        field(vb.sn, hy);
        const float4 oc = *reinterpret_cast<const float4*>(&vo.cs[r][4 + lj]);
        const float4 os = *reinterpret_cast<const float4*>(&vo.sn[r][4 + lj]);
        Pack4<S> pk;
        load4(stored, pk);
        int n_acc = 0;   // unused: uniform proposals
        float ev[2];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const float4 u = t == 0 ? unit_uniforms<O, 0>(w0, w1, w2) : unit_uniforms<O, 1>(w0, w1, w2);
            const bool upd0 = !((bits >> (2 * t)) & 1u), upd1 = !((bits >> (2 * t + 1)) & 1u);
            const bool ex0 = 2 * (lj + 2 * t) + O < A.Lx, ex1 = 2 * (lj + 2 * t + 1) + O < A.Lx;
            float2 v = move_pair<sizeof(S), true, false, QM, false>(
                hx[t], hy[t], make_float2(u.x, u.y), make_float2(u.z, u.w),
                make_float2(load_as<float>(pk.s[2 * t]), load_as<float>(pk.s[2 * t + 1])), upd0, upd1, q,
                A.nl2eTf, width, inv_q, 0.0f, n_acc, t == 0 ? make_float2(oc.x, oc.y) : make_float2(oc.z, oc.w),
                t == 0 ? make_float2(os.x, os.y) : make_float2(os.z, os.w));
            v = make_float2(load_as<float>(store_from<S>(v.x)), load_as<float>(store_from<S>(v.y)));
            fn[t] = v;
            samp[t] = make_float2(upd0 ? v.x : 0.0f, upd1 ? v.y : 0.0f);   // frozen sites add 0
            const float2 qn = mul2(splat(q), v);
            __sincosf(qn.x, &sn[t].x, &cs[t].x);
            __sincosf(qn.y, &sn[t].y, &cs[t].y);
            cs[t] = make_float2(ex0 ? cs[t].x : 0.0f, ex1 ? cs[t].y : 0.0f);
            sn[t] = make_float2(ex0 ? sn[t].x : 0.0f, ex1 ? sn[t].y : 0.0f);
            if constexpr (MEASURE) {
                const float2 e2 = fma2(cs[t], hx[t], mul2(sn[t], hy[t]));
                ev[t] = (ex0 ? e2.x : 0.0f) + (ex1 ? e2.y : 0.0f);
            }
        }
        if constexpr (MEASURE) er = ev[0] + ev[1];
    }
};

template <typename S, bool MEASURE, int SAMPLE, int QM, bool PAIR, bool STALL = false>
__global__ void __launch_bounds__(kCoarseThreads, 1) coarse_kernel(const __grid_constant__ Args A)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    const Band B(A);
    const int b = B.b, nb = B.nb, ya = B.ya, yb = B.yb, nr = yb - ya;
    const int G = A.G, P = 4 * G + 8, NR = A.rows;
    const int tid = threadIdx.x, T = blockDim.x;
    const float q = QM == 2 ? 0.5f : A.qf;
    const float width = QM == 2 ? 3.14159265358979324f : kTwoPiF * q;
    const float inv_q = QM == 2 ? 2.0f : 1.0f / q;

    // ---- shared memory: unit vectors of rows ya - 1 ... yb, the band's stored angles and frozen bits
    const int plane = (NR + 2) * P;       // floats of one colour's cosines (then its sines)
    float* const units = reinterpret_cast<float*>(dsm);
    auto view = [&](int c) {
        return View{Row{units + 2 * c * plane, P}, Row{units + (2 * c + 1) * plane, P}};
    };
    S* const vals = reinterpret_cast<S*>(units + (size_t)4 * plane);
    auto own = [&](int c, int r, int g) { return vals + ((size_t)(c * NR + r) * G + g) * 4; };
    unsigned char* const fz = reinterpret_cast<unsigned char*>(vals + (size_t)2 * NR * 4 * G);
    auto frozen = [&](int c, int r, int g) -> unsigned char& { return fz[(c * NR + r) * G + g]; };
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
                unit_of(q, load_as<float>(pk.s[e]), 2 * (4 * g + e) + ((y + c) & 1) < A.Lx, vc[e], vs[e]);
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

    // unit u: four columns g of row pair pr (PAIR), or of one of its rows, whose role follows the
    // warp
    const int NG = ((nr + 1) >> 1) * G;
    const int U = PAIR ? NG : 2 * ((NG + 31) & ~31);
    auto unit_role = [](int u) { return PAIR ? 0 : (u >> 5) & 1; };
    auto unit_idx = [](int u) { return PAIR ? u : (u >> 6) * 32 + (u & 31); };
    const int pr0 = unit_idx(tid) / G, g0 = unit_idx(tid) - pr0 * G;
    const size_t parity = slot_stride<false>(A, nb);
    SweepArgs sa{};   // for sample_row
    bool bad = false;
    uint32_t tag = A.epoch;   // of the exchange before this pass (the first pass has none)
#pragma unroll 1
    for (int sw = 0; sw < A.nsweeps; ++sw) {
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            const View vo = view(c), vb = view(1 - c);
            const bool first = sw == 0 && c == 0, last = sw + 1 == A.nsweeps && c == 1;
            const PhiloxSched ph = pass_keys(A, A.sweep + (uint32_t)sw, c);
            sa.acc = A.acc[c];
            sa.acc_hi = A.acc_hi[c];
            sa.acc_lo = A.acc_lo[c];
            // the first unit's random words do not wait for anybody
            uint4 w0 = {}, w1 = {}, w2 = {};
            auto words = [&](int role, int pr, int g) {
                const uint32_t h = (uint32_t)((ya >> 1) + pr);
                w0 = pair_words((uint32_t)g, h, ph, 0u);
                w1 = pair_words((uint32_t)g, h, ph, 1u);
                if (PAIR || role) w2 = pair_words((uint32_t)g, h, ph, 2u);
            };
            if (tid < U) words(unit_role(tid), pr0, g0);
            if (__syncthreads_or(bad)) goto out;   // the band's rows of the other colour are complete
            for (int u = tid; u < U; u += T) {
                const int role = unit_role(u), idx = unit_idx(u);
                const int pr = u == tid ? pr0 : idx / G, g = u == tid ? g0 : idx - pr * G;
                if (idx >= NG) continue;
                if (u != tid) words(role, pr, g);
                auto row = [&](auto role_) {
                    constexpr int O = decltype(role_)::value;
                    const int i = 2 * pr + (O == 0 ? c : 1 - c), r = i + 1, y = ya + i;   // row i of the band
                    if (y >= A.Ly) return;
                    // a neighbour's boundary row, these four columns: read by this thread only
                    auto take = [&](int side, int rr) {
                        const unsigned long long* const p =
                            slot<false>(A, nullptr, b, side, 0) + (tag & 1u) * parity + 4 * g;
                        float x[4], vc[4], vs[4];
                        if (!wait2(A, p, tag, x[0], x[1]) || !wait2(A, p + 2, tag, x[2], x[3])) bad = true;
#pragma unroll
                        for (int e = 0; e < 4; ++e)   // that row's colour 1 - c has the parity O
                            unit_of(q, x[e], 2 * (4 * g + e) + O < A.Lx, vc[e], vs[e]);
                        *reinterpret_cast<float4*>(&vb.cs[rr][4 + 4 * g]) = make_float4(vc[0], vc[1], vc[2], vc[3]);
                        *reinterpret_cast<float4*>(&vb.sn[rr][4 + 4 * g]) = make_float4(vs[0], vs[1], vs[2], vs[3]);
                    };
                    if (!first && i == 0 && b > 0) take(0, 0);
                    if (!first && i == nr - 1 && b + 1 < nb) take(1, nr + 1);
                    [[maybe_unused]] const size_t at = (size_t)y * A.pitch + 4 * g;
                    [[maybe_unused]] double2 sd0{}, sd1{};   // FP64 sums: loaded while the moves run
                    if constexpr (SAMPLE == 1) {
                        const double2* const s = reinterpret_cast<const double2*>(sa.acc + at);
                        sd0 = s[0];
                        sd1 = s[1];
                    }
                    QuadRow<S, MEASURE, QM, O> m;
                    m.run(A, vb, vo, r, g, own(c, i, g), frozen(c, i, g), w0, w1, w2, q, width, inv_q);
                    auto send = [&](int to, int side) {
                        unsigned long long* const p =
                            slot<false>(A, nullptr, to, side, 0) + ((tag + 1u) & 1u) * parity + 4 * g;
                        put2(p, tagged(m.fn[0].x, tag + 1u), tagged(m.fn[0].y, tag + 1u));
                        put2(p + 2, tagged(m.fn[1].x, tag + 1u), tagged(m.fn[1].y, tag + 1u));
                    };
                    if (!last && i == 0 && b > 0) send(b - 1, 1);
                    if (!last && i == nr - 1 && b + 1 < nb && !(STALL && b == 0)) send(b + 1, 0);
                    Pack4<S> pk;
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        pk.s[2 * t] = store_from<S>(m.fn[t].x);
                        pk.s[2 * t + 1] = store_from<S>(m.fn[t].y);
                    }
                    store4(own(c, i, g), pk);
                    *reinterpret_cast<float4*>(&vo.cs[r][4 + 4 * g]) =
                        make_float4(m.cs[0].x, m.cs[0].y, m.cs[1].x, m.cs[1].y);
                    *reinterpret_cast<float4*>(&vo.sn[r][4 + 4 * g]) =
                        make_float4(m.sn[0].x, m.sn[0].y, m.sn[1].x, m.sn[1].y);
                    if constexpr (MEASURE) {
                        if (c == 1) A.er[((size_t)sw * A.Ly + y) * G + g] = m.er;
                    }
                    if constexpr (SAMPLE == 1) {
                        double2* const s = reinterpret_cast<double2*>(sa.acc + at);
                        s[0] = make_double2(sd0.x + (double)m.samp[0].x, sd0.y + (double)m.samp[0].y);
                        s[1] = make_double2(sd1.x + (double)m.samp[1].x, sd1.y + (double)m.samp[1].y);
                    } else if constexpr (SAMPLE != 0) {
                        const float fs[4] = {m.samp[0].x, m.samp[0].y, m.samp[1].x, m.samp[1].y};
                        sample_row<SAMPLE>(sa, at, fs);
                    }
                };
                using First = std::integral_constant<int, 0>;
                using Second = std::integral_constant<int, 1>;
                if constexpr (PAIR) {
                    row(First{});
                    row(Second{});
                } else {
                    if (role) row(Second{});
                    else row(First{});
                }
            }
            ++tag;
        }
    }
out:
    // ---- the band's rows back to the layout (the neighbours loaded their rows before they sent the
    // words of the first exchange)
    __syncthreads();
    for (int i = tid; i < 2 * nr * G; i += T) {
        const int c = i / (nr * G), k = i - c * nr * G, r = k / G, g = k - r * G;
        Pack4<S> pk;
        load4(own(c, r, g), pk);
        store4(static_cast<S*>(A.ang[c]) + (size_t)(ya + r) * A.pitch + 4 * g, pk);
    }
}

template <typename S, bool MEASURE, int SAMPLE, int QM, bool STALL = false>
cudaError_t go_shape(const Plan& p, const Args& a, cudaStream_t st)
{
    void (*kern)(const Args) = p.cluster ? fine_kernel<S, MEASURE, SAMPLE, QM, true, STALL>
                               : p.fine  ? fine_kernel<S, MEASURE, SAMPLE, QM, false, STALL>
                               : p.pair  ? coarse_kernel<S, MEASURE, SAMPLE, QM, true, STALL>
                                         : coarse_kernel<S, MEASURE, SAMPLE, QM, false, STALL>;
    // An attribute belongs to the function, and handles of other host threads launch it too: always the same
    // value, the most a plan takes. (With p.smem here, a smaller lattice's value that landed between
    // a larger one's call and its launch made that launch fail.)
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(p.nb);
    cfg.blockDim = dim3(p.threads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (p.cluster) {
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
