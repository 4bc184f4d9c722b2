// Pool-side factorisation of the gather for one query per user (bf16, head_dim 32 or 64).
//
// With a single query q per (user, group) the gathered rows are only ever used in two sums:
//     score_i  = q_u . K_u[i] + q_g . P_k[I_k[i]]            = q_u . K_u[i] + T[I_k[i]],  T = P_k q_g
//     out_g    = sum_i p_i P_v[I_v[i]]                       = sum_j w[j] P_v[j],       w[j] = sum_{i: I_v[i] = j} p_i
// (Eq. K / Eq. Kc with the user part first; q_u, q_g the user and shared slices of q).  T for all users is
// one dense product with the K pool, the output one dense product of the weight histograms w with the V pool;
// per position only two 4-byte table accesses remain instead of two gathered pool rows.  Same mathematics as
// the gathering kernels, another summation order.  It pays when histories are long compared with the pool
// (tables cost 2 x n_entries x 4 bytes per (user, group) to HBM and back) -- the caller decides.
//
// Three launches:
//   fact_table_kernel  T[r][g][j] = q_r . P_k[g][j]          m16n8k16 MMAs, fp32 out
//   fact_main_kernel   persistent CTAs over the (user, group) pairs: T row into shared memory by bulk copy, then one pass over
//                      the history: score, weight, histogram w (a buffer of its own), user-part output and row sum
//   fact_out_kernel    out[r][g][:] = (w[r][g] P_v[g] + user part) / l          MMAs, w in bf16
#include <cuda_bf16.h>
#include <math_constants.h>

#include <algorithm>
#include <type_traits>

#include "ckv_internal.h"
#include "ptx_helpers.cuh"

namespace ckv {
namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr int kMainThreads = 1024;
constexpr int64_t kSlabBytes = (int64_t)1 << 30;
constexpr size_t kMainSmem = 226 * 1024, kMainExtra = 32 * 9 * 4 + 64;  // shared memory for tables; sums and barriers
constexpr int kOutWarps = 8, kOutMT = 2, kOutRows = 16 * kOutMT, kOutCluster = 4;

__device__ __forceinline__ float bf16_bits_to_float(uint32_t b) { return __uint_as_float(b << 16); }

enum { ERR_FACT_TABLE = 128 };  // a bounded wait for a table row ran out
__device__ __forceinline__ bool table_wait(uint32_t bar, uint32_t parity)
{
    for (int i = 0; i < (1 << 22); ++i) {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}
// ------------------------------------------------------------------------------------------------ T = P_k q
// T / w rows in HBM are this many floats apart: 32-byte aligned rows, room for zero-filled bf16 pairs up to a
// multiple of 8 entries
__host__ __device__ __forceinline__ int row_floats(int n_entries) { return (n_entries + 7) & ~7; }

constexpr int kTableMT = 4;  // 16-request tiles per warp: every pool row fetched serves 64 requests

// What the main kernel needs to know of a pair, written by the table kernel (in place of a chain of three loads per pair).
struct __align__(16) PairRec {
    int64_t unit0;    // arena unit of position 0
    int32_t L, pad;
    uint4 q_head;     // the query's first eight elements (the user part meets them), bf16
};

// Rows of the tables follow the items: row = item * G + group.  The rows of the first items are written last, those of all groups
// together: the main kernel begins with them and finds them in L2 (512 users x 4 groups x 16384 entries 195 -> 192 us).
template <int D>
__global__ void __launch_bounds__(128)
    fact_table_kernel(const __grid_constant__ AttendArgs a, float* __restrict__ tw, PairRec* __restrict__ recs)
{
    constexpr int KS = D / 16, MT = kTableMT;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gl = lane >> 2, t = lane & 3;
    const int m = a.cv.n_entries, G = a.cv.n_groups, grp = blockIdx.y;
    const int j0 = blockIdx.x * 256 + warp * 64, r0 = (gridDim.z - 1 - blockIdx.z) * (16 * MT);
    if (blockIdx.x == 0 && threadIdx.x < 16 * MT && r0 + (int)threadIdx.x < a.n_items) {
        const Req rq = a.reqs[a.items[r0 + threadIdx.x].req];
        PairRec rec;
        rec.unit0 = rq.base + (int64_t)grp * rq.Lpad;
        rec.L = rq.L;
        rec.pad = 0;
        rec.q_head = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(a.queries) + ((int64_t)rq.q0 * G + grp) * D));
        recs[(int64_t)(r0 + threadIdx.x) * G + grp] = rec;
    }
    if (j0 >= m) return;
    // Which feature sits in which k-slot of the MMA is free as long as Q and the pool rows agree: a lane reads
    // D / 4 contiguous bytes of "its" rows, and k-step ks, slots (2t, 2t+1, 2t+8, 2t+9) hold features
    // (D / 4) t + 4 ks + (0, 1, 2, 3).
    constexpr int W = D / 8;  // 32-bit words per lane and row
    const uint16_t* Q = reinterpret_cast<const uint16_t*>(a.queries);
    uint32_t qa[MT][KS][4];
    bool v_lo[MT], v_hi[MT];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        const int r_lo = r0 + 16 * mt + gl, r_hi = r_lo + 8;
        v_lo[mt] = r_lo < a.n_items;
        v_hi[mt] = r_hi < a.n_items;
        const int64_t q0_lo = v_lo[mt] ? a.reqs[a.items[r_lo].req].q0 : 0, q0_hi = v_hi[mt] ? a.reqs[a.items[r_hi].req].q0 : 0;
        uint32_t q_lo[W], q_hi[W];
#pragma unroll
        for (int h = 0; h < W / 4; ++h) {
            uint4 x = make_uint4(0, 0, 0, 0), y = x;
            if (v_lo[mt])
                x = __ldg(reinterpret_cast<const uint4*>(Q + (q0_lo * G + grp) * D + 2 * W * t) + h);
            if (v_hi[mt])
                y = __ldg(reinterpret_cast<const uint4*>(Q + (q0_hi * G + grp) * D + 2 * W * t) + h);
            q_lo[4 * h] = x.x; q_lo[4 * h + 1] = x.y; q_lo[4 * h + 2] = x.z; q_lo[4 * h + 3] = x.w;
            q_hi[4 * h] = y.x; q_hi[4 * h + 1] = y.y; q_hi[4 * h + 2] = y.z; q_hi[4 * h + 3] = y.w;
        }
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
            qa[mt][ks][0] = q_lo[2 * ks];
            qa[mt][ks][1] = q_hi[2 * ks];
            qa[mt][ks][2] = q_lo[2 * ks + 1];
            qa[mt][ks][3] = q_hi[2 * ks + 1];
        }
    }
    const uint16_t* P = reinterpret_cast<const uint16_t*>(a.cv.poolK) + (int64_t)grp * m * D;
    const int ms = row_floats(m);
    // (Bound by the writing of T: 134 MB for 512 requests x 4 groups x 16384 entries in 40 us.  Storing 32 bytes per lane,
    // 128 per row, took 43; 32 requests and 256 entries per warp with the next rows prefetched 46.)
#pragma unroll 2
    for (int nt = 0; nt < 8; ++nt) {
        const int jb = j0 + 8 * nt + gl;  // pool entry whose row is this lane's B column
        const uint4* row = reinterpret_cast<const uint4*>(P + (int64_t)(jb < m ? jb : m - 1) * D + 2 * W * t);
        uint32_t pw[W];
#pragma unroll
        for (int h = 0; h < W / 4; ++h) {
            const uint4 x = __ldg(row + h);
            pw[4 * h] = x.x; pw[4 * h + 1] = x.y; pw[4 * h + 2] = x.z; pw[4 * h + 3] = x.w;
        }
        const int jc = j0 + 8 * nt + 2 * t;  // columns of the accumulator fragment
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) mma_bf16(c, qa[mt][ks], pw[2 * ks], pw[2 * ks + 1]);
            float* t_lo = tw + ((int64_t)(r0 + 16 * mt + gl) * G + grp) * ms;
            float* t_hi = t_lo + (int64_t)8 * G * ms;
            // the two columns of a lane are one aligned 8-byte store (a column past the last entry lands in the row's padding)
            if (v_lo[mt] && jc < m) *reinterpret_cast<float2*>(t_lo + jc) = make_float2(c[0], c[1]);
            if (v_hi[mt] && jc < m) *reinterpret_cast<float2*>(t_hi + jc) = make_float2(c[2], c[3]);
        }
    }
}

// ------------------------------------------------------------------------------------------------ main
constexpr int kCrowd = 3;  // lanes of a warp's first positions that share a pool entry from which on additions are combined
constexpr int kAux = 16;  // floats per (request, group): [0] row sum l, [1..8] user-part output (not normalised)

// User parts of two neighbouring positions, DU bf16 elements each (DU < 0: `d_user` of them, any number up to 8), as the
// words they are stored in.
template <int DU>
struct UserPair {
    static constexpr int W = DU < 0 ? 8 : DU == 0 ? 1 : DU;  // 32-bit words
    uint32_t w[W];
    __device__ __forceinline__ void load(const uint16_t* u, int64_t unit, int d_user)
    {
        if constexpr (DU == 1) w[0] = __ldcs(reinterpret_cast<const uint32_t*>(u + unit));
        if constexpr (DU == 2) {
            const uint2 x = __ldcs(reinterpret_cast<const uint2*>(u + unit * 2));
            w[0] = x.x; w[1] = x.y;
        }
        if constexpr (DU == 4 || DU == 8) {
#pragma unroll
            for (int h = 0; h < DU / 4; ++h) {
                const uint4 x = __ldcs(reinterpret_cast<const uint4*>(u + unit * DU) + h);
                w[4 * h] = x.x; w[4 * h + 1] = x.y; w[4 * h + 2] = x.z; w[4 * h + 3] = x.w;
            }
        }
        if constexpr (DU < 0) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {  // element e of position 0 in word e / 2, of position 1 in word 4 + e / 2
                const uint32_t x = e < d_user ? __ldg(u + unit * d_user + e) : 0u, y = e < d_user ? __ldg(u + (unit + 1) * d_user + e) : 0u;
                w[e >> 1] = e & 1 ? w[e >> 1] | x << 16 : x;
                w[4 + (e >> 1)] = e & 1 ? w[4 + (e >> 1)] | y << 16 : y;
            }
        }
    }
    __device__ __forceinline__ float at(int pos, int e) const  // element e of position pos
    {
        const int i = (DU < 0 ? 8 : DU) * pos + e;
        return i & 1 ? __uint_as_float(w[i >> 1] & 0xffff0000u) : bf16_bits_to_float(w[i >> 1] & 0xffffu);
    }
};

__device__ __forceinline__ int order_bits(float f)  // monotone in f
{
    const int i = __float_as_int(f);
    return i ^ ((i >> 31) & 0x7fffffff);
}

// Persistent: CTA c takes (item, group) pairs c, c + gridDim.x, ... of the list ordered longest history first
// (pair = item * G + group, so neighbours in the list weigh about the same).  One pass over the history: index, user
// part, T entry, weight, histogram.  The weights are taken relative to 2^0 and not to the largest score, which would
// need a pass of its own (fp32 and bf16 have the exponent range for weights of 2^-60 .. 2^60); a pair whose largest score
// turns out beyond that is worked out again relative to it.  While a pair is processed, the T row of the CTA's next pair
// is on its way into the other table buffer (one bulk copy), and every thread has two pairs of positions in flight.
// Bound by HBM: 20 bytes per position at d_u = 4 are 4 us per pair and SM at an even share of the bandwidth.  512 users,
// 4 groups, 16384 entries, 1000..16384 positions: 127 us (521 MB of DRAM traffic at 4.1 TB/s, 50 %; issue slots 40 %; a
// pair takes 18000 clocks of an SM, 9000 of them in the pass); with two passes, a block-wide maximum between them and the
// scores kept in shared memory 181 us.
template <int D, int MODE, int DU>
__global__ void __launch_bounds__(kMainThreads, 1)
    fact_main_kernel(const __grid_constant__ AttendArgs a, float* __restrict__ tw, float* __restrict__ aux,
                     const PairRec* __restrict__ recs, int n_tab)
{
    extern __shared__ __align__(128) float fsm[];
    constexpr int NU = DU < 0 ? 8 : DU;
    const int m = a.cv.n_entries, G = a.cv.n_groups, d_user = a.cv.d_user, ms = row_floats(m), tid = threadIdx.x, nt = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, n_pairs = a.n_items * G;
    float* const Ws = fsm + n_tab * (size_t)ms;      // the pair's weight histogram, all zero between pairs
    float* const red = Ws + ms;                      // [32][9] the warps' sums
    int* const smax = reinterpret_cast<int*>(red + 32 * 9);  // largest score of the pair, order_bits
    const uint32_t bar = smem_u32(smax + 4);         // [2] the table buffers' arrivals
    const uint16_t* uK = reinterpret_cast<const uint16_t*>(a.cv.userK);
    const uint16_t* uV = reinterpret_cast<const uint16_t*>(a.cv.userV);
    const uint16_t* iK = reinterpret_cast<const uint16_t*>(a.cv.idxK);
    const uint16_t* iV = reinterpret_cast<const uint16_t*>(a.cv.idxV);
    const float sc = a.scale * (MODE == CKV_SOFTMAX ? kLog2e : 0.5f);

    auto fetch_table = [&](int row, int k) {  // one thread
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar + 8 * k), "r"(4 * ms) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         smem_u32(fsm + k * (size_t)ms)),
                     "l"(tw + (int64_t)row * ms), "r"(4 * ms), "r"(bar + 8 * k)
                     : "memory");
    };
    struct Step {
        uint32_t ik, iv;
        UserPair<DU> k, v;
    };
    auto load_step = [&](Step& s, const PairRec& pr, int i) {  // positions i, i + 1 (the arena is padded: i + 1 may be read)
        if (i >= pr.L) return;
        const int64_t u = CKV_CLAMP(pr.unit0 + i, a.arena_units, a.err);
        s.ik = __ldcs(reinterpret_cast<const uint32_t*>(iK + u));
        s.iv = __ldcs(reinterpret_cast<const uint32_t*>(iV + u));
        s.k.load(uK, u, d_user);
        s.v.load(uV, u, d_user);
    };

    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar + 8) : "memory");
        *smax = INT32_MIN;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int j = tid; j < ms; j += nt) Ws[j] = 0.f;
    __syncthreads();
    int p = blockIdx.x, k = 0;
    uint32_t phase[2] = {0, 0};
    if (p >= n_pairs) return;
    PairRec cur = recs[p], nxt = recs[min(p + (int)gridDim.x, n_pairs - 1)];
    Step A, B;
    load_step(A, cur, 2 * tid);
    load_step(B, cur, 2 * (tid + nt));
    if (tid == 0) fetch_table(p, 0);
    bool ok = true;
    for (;;) {
        const float* Ts = fsm + k * (size_t)ms;
        const int p_next = p + gridDim.x;
        const bool more = p_next < n_pairs;
        const PairRec behind = recs[min(p_next + (int)gridDim.x, n_pairs - 1)];  // used a pair later
        float qu[NU > 0 ? NU : 1], ou[NU > 0 ? NU : 1];
        {
            const uint32_t w[4] = {cur.q_head.x, cur.q_head.y, cur.q_head.z, cur.q_head.w};
#pragma unroll
            for (int e = 0; e < NU; ++e)
                qu[e] = (DU >= 0 || e < d_user) ? (e & 1 ? __uint_as_float(w[e >> 1] & 0xffff0000u) : bf16_bits_to_float(w[e >> 1] & 0xffffu)) : 0.f;
        }
        ok = ok && table_wait(bar + 8 * k, phase[k]);
        phase[k] ^= 1;
        if (more && n_tab == 2 && tid == 0) {  // (its buffer was last read before the barrier behind the previous pair's pass)
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            fetch_table(p_next, k ^ 1);
        }
        float m_ref = 0.f, mx, lsum;
        for (bool again = false;; again = true) {
            mx = -CUDART_INF_F;
            lsum = 0.f;
#pragma unroll
            for (int e = 0; e < NU; ++e) ou[e] = 0.f;
            // CROWD: lanes of a warp often hit the same entry (skewed indices), and colliding additions to one address take
            // turns: they are summed by shuffles first, and one lane adds
            auto step = [&](const Step& s, int i, auto crowd) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool in = i + h < cur.L;
                    if (!decltype(crowd)::value && !in) break;
                    float pw = 0.f;
                    uint32_t j = 0x10000u + lane;
                    if (in) {
                        float d = Ts[CKV_CLAMP(h ? s.ik >> 16 : s.ik & 0xffffu, (uint32_t)m, a.err)];
#pragma unroll
                        for (int e = 0; e < NU; ++e) d = fmaf(qu[e], s.k.at(h, e), d);
                        d *= sc;
                        if constexpr (MODE == CKV_SOFTMAX) {
                            mx = fmaxf(mx, d);
                            pw = ex2(d - m_ref);
                            lsum += pw;
                        } else {  // silu(x) = x sigmoid(x) = h (1 + tanh(h)), h = x / 2
                            pw = fmaf(d, tanh_fast(d), d);
                        }
                        j = CKV_CLAMP(h ? s.iv >> 16 : s.iv & 0xffffu, (uint32_t)m, a.err);
#pragma unroll
                        for (int e = 0; e < NU; ++e) ou[e] = fmaf(pw, s.v.at(h, e), ou[e]);
                    }
                    if constexpr (decltype(crowd)::value) {
                        uint32_t peers = __match_any_sync(0xffffffffu, j);
                        uint32_t rank = __popc(peers & ((1u << lane) - 1u));
                        const bool leads = rank == 0;
                        peers &= 0xfffffffeu << lane;  // the peers above this lane
                        while (__any_sync(0xffffffffu, peers != 0)) {  // pairs, pairs of pairs, ...
                            const int nx = __ffs(peers);
                            const float t = __shfl_sync(0xffffffffu, pw, (nx - 1) & 31);
                            if (nx) pw += t;
                            peers &= __ballot_sync(0xffffffffu, !(rank & 1));
                            rank >>= 1;
                        }
                        if (in && leads) atomicAdd(&Ws[j], pw);
                    } else {
                        atomicAdd(&Ws[j], pw);
                    }
                }
            };
            if (again) {
                load_step(A, cur, 2 * tid);
                load_step(B, cur, 2 * (tid + nt));
            }
            auto pass = [&](auto crowd) {
                for (int i0 = 64 * warp; i0 < cur.L; i0 += 4 * nt) {
                    const int i = i0 + 2 * lane;
                    step(A, i, crowd);
                    load_step(A, cur, i + 4 * nt);
                    step(B, i + 2 * nt, crowd);
                    load_step(B, cur, i + 6 * nt);
                }
            };
            const uint32_t alike = __match_any_sync(0xffffffffu, 2 * tid < cur.L ? A.iv & 0xffffu : 0x10000u + lane);
            if (__reduce_max_sync(0xffffffffu, __popc(alike)) >= kCrowd) pass(std::true_type{});
            else pass(std::false_type{});
            if (MODE != CKV_SOFTMAX || again) break;
            const int wmax = __reduce_max_sync(0xffffffffu, order_bits(mx));
            if (lane == 0) atomicMax(smax, wmax);
            __syncthreads();
            const int bits = *smax;
            const float top = __int_as_float(bits ^ ((bits >> 31) & 0x7fffffff));
            if (cur.L == 0 || (top <= 60.f && top >= -60.f)) break;
            m_ref = top;  // far from 2^0: once more, relative to the largest score
            for (int j = tid; j < ms; j += nt) Ws[j] = 0.f;
            __syncthreads();
        }
        if (more) {  // the next pair's first positions travel during the write-out
            load_step(A, nxt, 2 * tid);
            load_step(B, nxt, 2 * (tid + nt));
        }
        // row sum and user-part output: warp sums, then one thread per value adds the warps' sums in fixed order.  At every
        // step of the butterfly a lane gives away half of its values and keeps the other half's sums (9 shuffles for five
        // values instead of 25).
        constexpr int NV = NU == 0 ? 1 : NU == 1 ? 2 : NU <= 3 ? 4 : NU <= 7 ? 8 : 16;  // 1 + NU values, padded
        {
            float vals[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) vals[v] = v == 0 ? lsum : v <= NU ? ou[v <= NU && NU > 0 ? v - 1 : 0] : 0.f;
            int id = 0;  // which value this lane ends up with
#pragma unroll
            for (int o = 16, n = NV; o > 0; o >>= 1) {
                if (n > 1) {
                    n >>= 1;
                    const bool up = lane & o;
#pragma unroll
                    for (int v = 0; v < NV / 2; ++v)
                        if (v < n) {
                            const float give = up ? vals[v] : vals[v + n], keep = up ? vals[v + n] : vals[v];
                            vals[v] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                        }
                    id = 2 * id + (up ? 1 : 0);
                } else {
                    vals[0] += __shfl_xor_sync(0xffffffffu, vals[0], o);
                }
            }
            constexpr int spare = 32 / NV - 1;  // the lanes of a value differ in these low bits
            if ((lane & spare) == 0 && id <= NU) red[warp * 9 + id] = vals[0];
        }
        __syncthreads();  // the histogram and the warps' sums are complete; T is dead
        if (more && n_tab == 1 && tid == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            fetch_table(p_next, 0);
        }
        // w goes back to HBM rounded to bf16 (the precision the output product takes it in), two entries per word,
        // over the head of the T row, zero up to a multiple of 8 entries; what has been read is cleared for the next pair
        {
            uint2* wrow = reinterpret_cast<uint2*>(tw + (int64_t)p * ms);
            float4* w4 = reinterpret_cast<float4*>(Ws);
            for (int j4 = tid; 4 * j4 < ms; j4 += 4 * nt) {
                float4 x[4];
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    if (4 * (j4 + h * nt) < ms) x[h] = w4[j4 + h * nt];
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    if (4 * (j4 + h * nt) < ms) {
                        wrow[j4 + h * nt] = make_uint2(pack_bf16(x[h].x, x[h].y), pack_bf16(x[h].z, x[h].w));
                        w4[j4 + h * nt] = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
            }
        }
        if (warp <= NU) {  // warp v adds up value v
            float v = lane < nt / 32 ? red[lane * 9 + warp] : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) aux[(int64_t)p * kAux + warp] = v;
        }
        if (tid == 0) *smax = INT32_MIN;
        if (!more) break;
        __syncthreads();  // the histogram is clear, the warps' sums have been read
        cur = nxt;
        nxt = behind;
        p = p_next;
        if (n_tab == 2) k ^= 1;
    }
    if (!ok && tid == 0) atomicOr(a.err, ERR_FACT_TABLE);
}

// ------------------------------------------------------------------------------------------------ out = w P_v
// A cluster of four CTAs per (32 requests, group), its 32 warps splitting the pool's entries.  What bounds it is the V pool
// out of L2 (2 MB per cluster at 16384 64-wide entries): every row fetched serves 32 requests, and the split gives every
// SM a share.  512 requests x 4 groups x 16384 entries: 27 us (2.5 TB/s of w besides), with one CTA
// per 16 requests 30, and for 100 requests the whole call takes 61 us instead of 68.  P_v rows are
// contiguous here: 32-row tiles through a two-slot cp.async ring per warp, fragments by transposing ldmatrix.
// 16-byte chunk c of tile row r sits at chunk c ^ swz(r).  The eight rows of one ldmatrix block are rows
// 8 t' + const + e (t' < 4, e < 2) here, see the k-slot order below: they must fall into eight different bank groups.
template <int D>
__device__ __forceinline__ int swz(int r)
{
    return D == 64 ? ((((r >> 3) & 3) << 1) | (r & 1)) : ((r >> 3) & 3);
}

template <int D>
__global__ void __launch_bounds__(kOutWarps * 32, 2)
    fact_out_kernel(const __grid_constant__ AttendArgs a, const float* __restrict__ tw, const float* __restrict__ aux)
{
    constexpr int NTD = D / 8, ROWB = D * 2, CPR = ROWB / 16, RPI = 32 / CPR, TILE_B = 32 * ROWB;
    extern __shared__ __align__(128) unsigned char osm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gl = lane >> 2, t = lane & 3;
    const int m = a.cv.n_entries, G = a.cv.n_groups, grp = blockIdx.y, rank = blockIdx.x % kOutCluster,
              r0 = blockIdx.x / kOutCluster * kOutRows;
    constexpr int kParts = kOutWarps * kOutCluster;
    const int span = ((m + kParts - 1) / kParts + 31) / 32 * 32;
    const int jbeg = (rank * kOutWarps + warp) * span, jend = min(m, jbeg + span);
    const uint32_t* wrow[kOutMT][2];  // the requests of this lane's fragment rows
    bool v_in[kOutMT][2];
#pragma unroll
    for (int mt = 0; mt < kOutMT; ++mt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = r0 + 16 * mt + gl + 8 * h;
            v_in[mt][h] = r < a.n_items;
            wrow[mt][h] = reinterpret_cast<const uint32_t*>(tw + ((int64_t)(v_in[mt][h] ? r : 0) * G + grp) * row_floats(m));
        }
    const char* pV = reinterpret_cast<const char*>(a.cv.poolV) + (int64_t)grp * m * ROWB;
    const uint32_t ring = smem_u32(osm) + warp * (2 * TILE_B);
    const int cr = lane / CPR, cc = lane % CPR, lr = lane & 7, lm = lane >> 3;
    // Which pool entry sits in which k-slot is free as long as w and the V rows agree: a lane reads 8 consecutive
    // weights of its requests with one 16-byte load each, and k-step b, slots (2t, 2t+1, 2t+8, 2t+9) hold
    // entries 8t + 4b + (0, 1, 2, 3) of the 32-entry chunk; the ldmatrix row addresses follow.
    uint32_t offV[2][NTD / 2];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const int r = 8 * (lr >> 1) + 4 * b + 2 * (lm & 1) + (lr & 1);  // chunk row of matrix row lr, matrix half lm & 1
#pragma unroll
        for (int jp = 0; jp < NTD / 2; ++jp) offV[b][jp] = r * ROWB + (((2 * jp + (lm >> 1)) ^ swz<D>(r)) << 4);
    }

    auto issue = [&](int jc, int slot) {  // rows jc .. jc+31 of the V pool (clamped: their weights are zero)
#pragma unroll
        for (int i = 0; i < 32 / RPI; ++i) {
            const int r = i * RPI + cr;
            const int j = min(jc + r, m - 1);
            const uint32_t dst = ring + slot * TILE_B + r * ROWB + ((cc ^ swz<D>(r)) << 4);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(pV + (int64_t)j * ROWB + cc * 16)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // weights of one 32-entry chunk: entries 8t .. 8t+7 of both requests, the bf16 pairs the main kernel stored
    // (rows start at multiples of 32 bytes and are zero-filled behind the last entry up to a multiple of 8 entries)
    auto load_w = [&](int jc, uint4 (&x)[kOutMT][2]) {
        const int j = jc + 8 * t;
#pragma unroll
        for (int mt = 0; mt < kOutMT; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                x[mt][h] = j < jend && v_in[mt][h] ? __ldg(reinterpret_cast<const uint4*>(wrow[mt][h] + (j >> 1))) : make_uint4(0, 0, 0, 0);
    };

    float o[kOutMT][NTD][4];
#pragma unroll
    for (int mt = 0; mt < kOutMT; ++mt)
#pragma unroll
        for (int j = 0; j < NTD; ++j) o[mt][j][0] = o[mt][j][1] = o[mt][j][2] = o[mt][j][3] = 0.f;
    const int nch = jbeg < jend ? (jend - jbeg + 31) / 32 : 0;
    uint4 wa[kOutMT][2], wb[kOutMT][2];
    if (nch > 0) {
        issue(jbeg, 0);
        load_w(jbeg, wa);
    }
    for (int c = 0; c < nch; ++c) {
        const int jc = jbeg + 32 * c;
        if (c + 1 < nch) {
            issue(jc + 32, (c + 1) & 1);
            load_w(jc + 32, wb);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncwarp();
        const uint32_t vt = ring + (c & 1) * TILE_B;
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int jp = 0; jp < NTD / 2; ++jp) {
                uint32_t v0, v1, v2, v3;
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(v0), "=r"(v1), "=r"(v2), "=r"(v3)
                             : "r"(vt + offV[b][jp])
                             : "memory");
#pragma unroll
                for (int mt = 0; mt < kOutMT; ++mt) {
                    const uint32_t pa[4] = {b ? wa[mt][0].z : wa[mt][0].x, b ? wa[mt][1].z : wa[mt][1].x,
                                            b ? wa[mt][0].w : wa[mt][0].y, b ? wa[mt][1].w : wa[mt][1].y};
                    mma_bf16(o[mt][2 * jp], pa, v0, v1);
                    mma_bf16(o[mt][2 * jp + 1], pa, v2, v3);
                }
            }
        __syncwarp();  // every lane is done with the slot that the next iteration refills
#pragma unroll
        for (int mt = 0; mt < kOutMT; ++mt) {
            wa[mt][0] = wb[mt][0];
            wa[mt][1] = wb[mt][1];
        }
    }

    // sum the warps' partial outputs, then the CTAs', in fixed order; add the user part, normalise, store
    __syncthreads();
    float* red = reinterpret_cast<float*>(osm);  // [kOutWarps][kOutRows][D]; the sums over the warps in [0]
#pragma unroll
    for (int mt = 0; mt < kOutMT; ++mt)
#pragma unroll
        for (int j = 0; j < NTD; ++j) {
            float* p = red + ((size_t)warp * kOutRows + 16 * mt + gl) * D + 8 * j + 2 * t;
            *reinterpret_cast<float2*>(p) = make_float2(o[mt][j][0], o[mt][j][1]);
            *reinterpret_cast<float2*>(p + 8 * D) = make_float2(o[mt][j][2], o[mt][j][3]);
        }
    __syncthreads();
    for (int x = threadIdx.x; x < kOutRows * D; x += kOutWarps * 32) {
        float v = red[x];
        for (int w = 1; w < kOutWarps; ++w) v += red[(size_t)w * kOutRows * D + x];
        red[x] = v;
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    constexpr int kMine = kOutRows * D / kOutCluster;  // elements this CTA finishes
    for (int x = rank * kMine + threadIdx.x; x < (rank + 1) * kMine; x += kOutWarps * 32) {
        const int rr = x / D, f = x - rr * D, r = r0 + rr;
        if (r >= a.n_items) continue;
        const Req rq = a.reqs[a.items[r].req];
        float v = 0.f;
        for (int c = 0; c < kOutCluster; ++c) {
            uint32_t at;
            float y;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(smem_u32(red + x)), "r"(c));
            asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(y) : "r"(at) : "memory");
            v += y;
        }
        const float* ax = aux + ((int64_t)r * G + grp) * kAux;
        if (f < a.cv.d_user) v += ax[1 + f];
        float inv;
        if (a.mode == CKV_SOFTMAX) inv = ax[0] > 0.f ? 1.0f / ax[0] : 0.f;
        else inv = rq.L > 0 ? 1.0f / (float)rq.L : 0.f;
        v *= inv;
        const int64_t oi = ((int64_t)rq.q0 * G + grp) * D + f;
        if (a.out_dtype == CKV_BF16) reinterpret_cast<__nv_bfloat16*>(a.out)[oi] = __float2bfloat16_rn(v);
        else reinterpret_cast<float*>(a.out)[oi] = v;
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");  // the others' sums have been read
}

template <int D>
cudaError_t launch_slab(const AttendArgs& a, int n_sms, float* tw, float* aux, const Launch& l)
{
    const int m = a.cv.n_entries, G = a.cv.n_groups, n_pairs = a.n_items * G;
    PairRec* recs = reinterpret_cast<PairRec*>(aux + (size_t)n_pairs * kAux);
    cudaError_t e = launch_kernel(l, fact_table_kernel<D>,
                                  dim3((m + 255) / 256, G, (a.n_items + 16 * kTableMT - 1) / (16 * kTableMT)), 128, 0, 1, a, tw, recs);
    if (e != cudaSuccess) return e;
    // two table buffers if they fit next to the histogram; two CTAs of half the threads per SM if that leaves room for both
    const size_t table = (size_t)row_floats(m) * sizeof(float);
    const int n_tab = 3 * table + kMainExtra <= kMainSmem ? 2 : 1;
    const size_t smem_main = (n_tab + 1) * table + kMainExtra;
    const int per_sm = smem_main <= kMainSmem / 2 ? 2 : 1;
    const dim3 grid((unsigned)std::min(n_pairs, per_sm * n_sms));
#define CKV_FACT_MAIN(MODE, DU) \
    launch_kernel(l, fact_main_kernel<D, MODE, DU>, grid, kMainThreads / per_sm, smem_main, 1, a, tw, aux, (const PairRec*)recs, n_tab)
#define CKV_FACT_DU(MODE)                                                                                   \
    (a.cv.d_user == 0   ? CKV_FACT_MAIN(MODE, 0) : a.cv.d_user == 1 ? CKV_FACT_MAIN(MODE, 1)                \
     : a.cv.d_user == 2 ? CKV_FACT_MAIN(MODE, 2) : a.cv.d_user == 4 ? CKV_FACT_MAIN(MODE, 4)                \
     : a.cv.d_user == 8 ? CKV_FACT_MAIN(MODE, 8) : CKV_FACT_MAIN(MODE, -1))
    e = a.mode == CKV_SOFTMAX ? CKV_FACT_DU(CKV_SOFTMAX) : CKV_FACT_DU(CKV_SILU_OVER_L);
#undef CKV_FACT_DU
#undef CKV_FACT_MAIN
    if (e != cudaSuccess) return e;
    static_assert(kOutRows * 2 == 2 * 32, "the sums take the room of the rings");
    const size_t smem_out = (size_t)kOutWarps * 2 * 32 * D * 2;
    return launch_kernel(l, fact_out_kernel<D>, dim3((unsigned)((a.n_items + kOutRows - 1) / kOutRows * kOutCluster), G),
                         kOutWarps * 32, smem_out, kOutCluster, a, (const float*)tw, (const float*)aux);
}

}  // namespace

// Whether the family takes the shape: one table and one histogram in a CTA's shared memory (so stored indices have 16 bits).
bool fact_supported(int dtype, int head_dim, int d_user, int n_entries)
{
    return dtype == CKV_BF16 && (head_dim == 32 || head_dim == 64) && d_user <= 8 &&
           2 * (size_t)row_floats(std::min(n_entries, 65536)) * sizeof(float) + kMainExtra <= kMainSmem;
}

// Items per slab: the tables take at most kSlabBytes of workspace.  (Slabs whose tables stay in L2 were no faster: the main
// kernel gained 7 %, the other two lost more to grids too small for the SMs.)
int fact_slab_items(int n_items, int n_groups, int n_entries)
{
    const int64_t row = (int64_t)row_floats(n_entries) * sizeof(float) * n_groups;
    const int64_t slabs = std::max<int64_t>(1, (n_items * row + kSlabBytes - 1) / kSlabBytes);
    return (int)std::min<int64_t>(n_items, ((n_items + slabs - 1) / slabs + 63) / 64 * 64);
}
int64_t fact_workspace_floats(int n_items, int n_groups, int n_entries)
{
    return (int64_t)fact_slab_items(n_items, n_groups, n_entries) * n_groups *
           (row_floats(n_entries) + kAux + (int)(sizeof(PairRec) / sizeof(float)));
}

cudaError_t launch_attend_fact(int D, const AttendArgs& a, int n_sms, float* ws, const Launch& l, int* launches)
{
    const int slab = fact_slab_items(a.n_items, a.cv.n_groups, a.cv.n_entries);
    float* aux = ws + (size_t)slab * a.cv.n_groups * row_floats(a.cv.n_entries);
    for (int i0 = 0; i0 < a.n_items; i0 += slab) {
        AttendArgs s = a;
        s.items = a.items + i0;
        s.n_items = std::min(slab, a.n_items - i0);
        const cudaError_t e = D == 64 ? launch_slab<64>(s, n_sms, ws, aux, l) : launch_slab<32>(s, n_sms, ws, aux, l);
        if (e != cudaSuccess) return e;
        *launches += 3;
    }
    return cudaSuccess;
}

}  // namespace ckv
