// Warp-level tensor-core gather-concat-attention kernel (bf16, head_dim 32 or 64) for a moderate
// number of queries per user (head_dim 64: also for a single query).
//
// One warp owns (work item, group, block of 16*MT queries) and walks the history chunk 32
// positions at a time with m16n8k16 MMAs: S = Q K^T, weights in registers, O += P V.
// K and V rows go from the pool into a per-warp ring of shared-memory tiles with 16-byte
// asynchronous copies, NST tiles deep, and reach the MMA register layouts through ldmatrix
// (transposing for V).  A whole row is fetched by adjacent lanes, so the L1 sees one line per
// row, and the copies in flight cost no registers: a warp keeps NST - 1 tiles outstanding
// while it computes.  The user-specific leading elements (Eq. K) are written over the head
// of each staged row.  Positions keep their order: tile row r is position p0 + r.
// A side that is not shared (sharing only keys or only values) has its full-width rows in the
// arena; they are copied into the ring in place of pool rows (cp.async loader only) and nothing is
// patched.  With visible lengths a query row only takes the positions before its own limit.
//
// What bounds it is the latency of a warp's chain, index -> row -> product -> weights -> product, against the warps that
// registers and rings admit; the L1 / shared-memory data pipe, which every gathered row crosses on the way into the ring and
// out of it, is 82 to 90 % busy with 32-wide heads, but a form that kept a group's K rows in shared memory (65 %) was 4 to 13
// % slower all the same, with 16, 20 or 24 warps.
//
// Several warps may share one (item, group, query block): `parts` of them, a power of two, take its 32-position
// tiles in turn and merge their (m, l, O) at the end, through shared memory inside a block and through distributed
// shared memory between the blocks of a cluster.  What bounds a small call is the chain index -> row -> product of
// one warp times the tiles it walks, so the tiles are spread until every SM has warps; a call needs no second launch
// and no partial results in device memory for it.
//
// Two ways to fill the ring (template parameter TMA), same results bit for bit:
//   - 16-byte cp.async copies through L1 (hot rows of skewed index distributions stay in L1, but every
//     row crosses the L1 / shared-memory data pipe on the way in and again on the way out);
//   - TMA tile::gather4 loads, four pool rows per instruction, completion on an mbarrier: the rows
//     bypass L1 and that pipe; the hardware swizzle modes are the chunk order ldmatrix wants.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <math_constants.h>

#include <type_traits>

#include "ckv_internal.h"
#include "ptx_helpers.cuh"

namespace ckv {
namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kOctavesAbove = 10.f, kSumLimit = 1.f;  // see `normalise`

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void ldsm4(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3, uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldsm4_trans(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3, uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr)
                 : "memory");
}

template <bool IDX16>
__device__ __forceinline__ int load_index(const void* base, int64_t unit)
{
    if constexpr (IDX16) return __ldg(reinterpret_cast<const uint16_t*>(base) + unit);
    else return __ldg(reinterpret_cast<const int32_t*>(base) + unit);
}

// user part of one position (d_user in {1, 2, 4, 8}: 2 to 16 bytes)
__device__ __forceinline__ uint4 load_user_part(const uint16_t* u, int64_t unit, int d_user)
{
    uint4 r = make_uint4(0, 0, 0, 0);
    switch (d_user) {
        case 1: r.x = __ldg(u + unit); break;
        case 2: r.x = __ldg(reinterpret_cast<const uint32_t*>(u + unit * 2)); break;
        case 4: {
            const uint2 w = __ldg(reinterpret_cast<const uint2*>(u + unit * 4));
            r.x = w.x;
            r.y = w.y;
            break;
        }
        case 8: r = __ldg(reinterpret_cast<const uint4*>(u + unit * 8)); break;
        default: break;
    }
    return r;
}
__device__ __forceinline__ void store_user_part(uint32_t addr, const uint4& r, int d_user)
{
    switch (d_user) {
        case 1: asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"((uint16_t)r.x) : "memory"); break;
        case 2: asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(r.x) : "memory"); break;
        case 4: asm volatile("st.shared.v2.u32 [%0], {%1,%2};" ::"r"(addr), "r"(r.x), "r"(r.y) : "memory"); break;
        case 8:
            asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(r.x), "r"(r.y), "r"(r.z), "r"(r.w)
                         : "memory");
            break;
        default: break;
    }
}

// DENSE (64-wide heads, 16 queries a warp): a ring of two slots instead of three, which leaves room for three blocks per SM.
// The deeper ring is the better one as long as the SMs are not full (see mma_shape in the host code).  (Twenty warps at
// 32-wide heads spill: 143 -> 229 us for 4096 users x 512 positions x 16 queries; three slots there: 148.)
template <int D, int MT, bool TMA, bool DENSE = false>
struct MmaCfg {
    static constexpr int ROWB = D * 2;            // bytes per row
    static constexpr int CPR = ROWB / 16;         // 16-byte chunks per row
    static constexpr int RPI = 32 / CPR;          // rows one warp-wide copy instruction covers
    static constexpr int TILE_B = 32 * ROWB;      // one K or V tile of 32 positions
    // ring depth (more resident warps beat a deeper ring, except for cp.async with 128-byte rows)
    static constexpr int NST = (D == 64 && !TMA && !DENSE) ? 3 : 2;
    static constexpr int WARPS = 4;
    // TMA: tiles on 1024-byte boundaries (the swizzle pattern follows the address), then one mbarrier per slot
    static constexpr int SMEM = WARPS * NST * 2 * TILE_B + (TMA ? 1024 + WARPS * NST * 8 : 0);
    // (two query tiles, 32-wide: 168 registers and some spills outside the loop; left to itself the compiler takes 200 to 240
    // and a third of the warps goes, 134 us instead of 117 for 3000 users x 300 positions x 20..32 queries, SiLU)
    static constexpr int MIN_BLOCKS = MT == 1 ? (D == 64 ? (TMA || DENSE ? 3 : 2) : 4) : D == 32 && MT == 2 ? 3 : 1;
};

enum { ERR_MMA_LOAD = 16 };  // a bounded wait for a TMA tile ran out
constexpr int kTmaSpinLimit = 1 << 22;

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// chunk c of tile row r sits at chunk c ^ swz(r): the eight rows of an 8x8 ldmatrix block fall into
// eight different 16-byte bank groups
template <int D>
__device__ __forceinline__ int swz(int r)
{
    return D == 64 ? (r & 7) : ((r >> 1) & 3);
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// a 32-bit word of another block of the cluster, at this block's shared-memory address `addr`
__device__ __forceinline__ float ld_cluster(uint32_t addr, uint32_t rank)
{
    uint32_t remote;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(remote) : "memory");
    return v;
}

struct TmaMaps {
    CUtensorMap K, V;
};

// VAR = false: both sides shared and no visible lengths (the hot configurations); the code for the variants is
// compiled out.  SHARED = false: one warp per unit.
template <int D, int MT, int MODE, bool IDX16, bool TMA, bool VAR, bool SHARED, bool DENSE = false>
__global__ void __launch_bounds__(128, MmaCfg<D, MT, TMA, DENSE>::MIN_BLOCKS)
    attend_mma_kernel(const __grid_constant__ AttendArgs a, int n_mb, int log_wpu, int n_cta, int* err_flag,
                      const __grid_constant__ std::conditional_t<TMA, TmaMaps, InlineTable> tab)
{
    using C = MmaCfg<D, MT, TMA, DENSE>;
    constexpr int NTD = D / 8, KS = D / 16, ROWB = C::ROWB, CPR = C::CPR, RPI = C::RPI, NST = C::NST;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    grid_dependency_wait();
    // 2^log_wpu warps of a block and the n_cta blocks of its cluster share a unit; this warp is number `part` of
    // `parts` and takes tiles part, part + parts, ... of the chunk
    if constexpr (!SHARED) {
        log_wpu = 0;
        n_cta = 1;
    }
    const int wpu = 1 << log_wpu, sub = warp & (wpu - 1), parts = wpu * n_cta;
    const uint32_t rank = n_cta > 1 ? blockIdx.x % (uint32_t)n_cta : 0;
    const int part = (int)rank * wpu + sub;
    const int64_t uid = ((int64_t)(n_cta > 1 ? blockIdx.x / (uint32_t)n_cta : blockIdx.x) * C::WARPS + warp) >> log_wpu;
    if (uid >= (int64_t)a.n_items * n_mb) return;
    const int item = (int)(uid / n_mb), mb = (int)(uid - (int64_t)item * n_mb);
    Item it;
    Req rq;
    bool from_table = false;
    if constexpr (!TMA) from_table = a.inl != 0;
    if (from_table) {
        if constexpr (!TMA) {
            const InlineReq& r = tab.r[item];
            rq = Req{(int64_t)r.base32 * 32, r.L, (r.L + 31) & ~31, r.q0, r.M, -1, 1};
            it = Item{item, 0, r.L, -1};
        }
    } else {
        it = a.items[item];
        rq = a.reqs[it.req];
    }
    const int row0 = mb * 16 * MT;
    if (row0 >= rq.M) return;
    const int grp = blockIdx.y, G = a.cv.n_groups, d_user = a.cv.d_user;
    const bool full_k = VAR && a.cv.full_k != 0, full_v = VAR && a.cv.full_v != 0;  // the side's rows are cached full width
    const bool wide_user = d_user == 1 || d_user == 2 || d_user == 4 || d_user == 8;

    uint32_t qa[MT][KS][4];
    const uint16_t* Q = reinterpret_cast<const uint16_t*>(a.queries);
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        const int r_lo = row0 + 16 * mt + g, r_hi = r_lo + 8;
        const uint16_t* q_lo = Q + ((int64_t)(rq.q0 + r_lo) * G + grp) * D;
        const uint16_t* q_hi = Q + ((int64_t)(rq.q0 + r_hi) * G + grp) * D;
        if (r_lo < rq.M) (void)CKV_CLAMP((int64_t)(rq.q0 + r_lo), a.q_rows, err_flag);
        if (r_hi < rq.M) (void)CKV_CLAMP((int64_t)(rq.q0 + r_hi), a.q_rows, err_flag);
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
            const int c = 16 * ks + 2 * t;
            qa[mt][ks][0] = r_lo < rq.M ? __ldg(reinterpret_cast<const uint32_t*>(q_lo + c)) : 0u;
            qa[mt][ks][1] = r_hi < rq.M ? __ldg(reinterpret_cast<const uint32_t*>(q_hi + c)) : 0u;
            qa[mt][ks][2] = r_lo < rq.M ? __ldg(reinterpret_cast<const uint32_t*>(q_lo + c + 8)) : 0u;
            qa[mt][ks][3] = r_hi < rq.M ? __ldg(reinterpret_cast<const uint32_t*>(q_hi + c + 8)) : 0u;
        }
    }
    // rows 8..15 of the only query tile are all padding when the user has at most 8 queries
    const bool has_hi = MT > 1 || row0 + 8 < rq.M;
    const int n_mt = (min(rq.M - row0, 16 * MT) + 15) >> 4;  // query tiles that hold queries
    // positions a query row attends: [0, lim); rows beyond the user's queries take none
    int lim[MT][2], lim_max = rq.L, lim_min = rq.L;
    if constexpr (VAR) {
        lim_max = 0;
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = row0 + 16 * mt + g + 8 * h;
                int v = 0;
                if (r < rq.M) {
                    v = a.vis ? min(max(__ldg(a.vis + rq.q0 + r), 0), rq.L) : rq.L;
                    lim_min = min(lim_min, v);
                }
                lim[mt][h] = v;
                lim_max = max(lim_max, v);
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lim_max = max(lim_max, __shfl_xor_sync(0xffffffffu, lim_max, o));
            lim_min = min(lim_min, __shfl_xor_sync(0xffffffffu, lim_min, o));
        }
    }

    float o[MT][NTD][4];
    float m_run[MT][2], l_run[MT][2];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        m_run[mt][0] = m_run[mt][1] = -CUDART_INF_F;
        l_run[mt][0] = l_run[mt][1] = 0.f;
#pragma unroll
        for (int j = 0; j < NTD; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[mt][j][e] = 0.f;
    }

    const int cr = lane / CPR, cc = lane % CPR;  // this lane's row within a copy instruction and its chunk
    const char* pK = reinterpret_cast<const char*>(a.cv.poolK) + (int64_t)grp * a.cv.n_entries * ROWB + cc * 16;
    const char* pV = reinterpret_cast<const char*>(a.cv.poolV) + (int64_t)grp * a.cv.n_entries * ROWB + cc * 16;
    const int64_t chunk0 = rq.base + (int64_t)grp * rq.Lpad + it.begin;  // the chunk's first unit
    if (it.len > 0) (void)CKV_CLAMP(chunk0 + ((it.len + 31) & ~31) - 1, a.arena_units, err_flag);  // the chunk's last (padded) unit
    const int64_t unit0 = chunk0 + 32 * part + lane;  // this lane's position of step 0
    const int stride = 32 * parts;                    // positions between two of this warp's steps
    const uint16_t* uK = reinterpret_cast<const uint16_t*>(a.cv.userK);
    const uint16_t* uV = reinterpret_cast<const uint16_t*>(a.cv.userV);
    const int end = VAR ? min(it.begin + it.len, lim_max) : it.begin + it.len;  // nothing behind the last visible position is touched
    const int n_tiles = VAR ? (end > it.begin ? (end - it.begin + 31) >> 5 : 0) : (it.len + 31) >> 5;
    const int nsteps = n_tiles > part ? (n_tiles - part + parts - 1) >> (log_wpu + (31 - __clz(n_cta))) : 0;
    const int full_end = VAR ? min(end, lim_min) : end;  // up to here every row of this warp sees every position
    // A side that is not shared: its rows are the chunk's own units in the arena, and what stands in for the pool
    // index of the position in lane l of a tile is its offset from the chunk's first unit.
    if (full_k) pK = reinterpret_cast<const char*>(a.cv.userK) + chunk0 * ROWB + cc * 16;
    if (full_v) pV = reinterpret_cast<const char*>(a.cv.userV) + chunk0 * ROWB + cc * 16;
    const float sc = a.scale * (MODE == CKV_SOFTMAX ? kLog2e : 0.5f);

    uint32_t smem0 = smem_u32(smem_raw);
    if constexpr (TMA) smem0 = (smem0 + 1023u) & ~1023u;
    const uint32_t ring = smem0 + warp * (NST * 2 * C::TILE_B);
    const uint32_t bars = smem0 + C::WARPS * (NST * 2 * C::TILE_B) + warp * (NST * 8);  // TMA only
    if constexpr (TMA) {
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < NST; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bars + 8 * i));
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
    }
    const int row_base = grp * a.cv.n_entries;  // TMA row coordinate of pool row 0 of this group
    // ldmatrix row addresses of this lane (matrix lane >> 3, row lane & 7)
    const int lr = lane & 7, lm = lane >> 3;
    uint32_t offK[KS / 2 > 0 ? KS / 2 : 1], offV[NTD / 2];
#pragma unroll
    for (int kp = 0; kp < KS / 2; ++kp) offK[kp] = lr * ROWB + (((4 * kp + lm) ^ swz<D>(lr)) << 4);
#pragma unroll
    for (int jp = 0; jp < NTD / 2; ++jp)
        offV[jp] = ((lm & 1) * 8 + lr) * ROWB + (((2 * jp + (lm >> 1)) ^ swz<D>(lr)) << 4);
    const uint32_t offU = lane * ROWB + (swz<D>(lane) << 4);  // head of this lane's row (chunk 0)

    // copies of one tile: the indices of its 32 positions sit one per lane
    auto issue = [&](int step, int idx_k, int idx_v) {
        const uint32_t kt = ring + (step % NST) * (2 * C::TILE_B), vt = kt + C::TILE_B;
        if constexpr (TMA) {
            // lanes 0..7 fetch the K tile, lanes 8..15 the V tile, four rows (positions 4j .. 4j+3) each
            const uint32_t bar = bars + 8 * (step % NST);
            if (lane == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(2 * C::TILE_B)
                             : "memory");
            __syncwarp();
            int r[4];
            const int j4 = 4 * (lane & 7);
            if constexpr (IDX16) {
                const int both = idx_k | (idx_v << 16);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int x = __shfl_sync(0xffffffffu, both, j4 + j);
                    r[j] = row_base + (lane < 8 ? (x & 0xffff) : (int)((uint32_t)x >> 16));
                }
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int xk = __shfl_sync(0xffffffffu, idx_k, j4 + j), xv = __shfl_sync(0xffffffffu, idx_v, j4 + j);
                    r[j] = row_base + (lane < 8 ? xk : xv);
                }
            }
            if (lane < 16) {
                const CUtensorMap* tm = lane < 8 ? &tab.K : &tab.V;
                const uint32_t dst = (lane < 8 ? kt : vt) + j4 * ROWB;
                asm volatile(
                    "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes "
                    "[%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(dst),
                    "l"(tm), "r"(0), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(bar)
                    : "memory");
            }
        } else {
#pragma unroll
            for (int i = 0; i < 32 / RPI; ++i) {
                const int r = i * RPI + cr;
                const uint32_t off = r * ROWB + ((cc ^ swz<D>(r)) << 4);
                // (range-checked build: a pool index below n_entries, or, for a side that is not shared, an offset
                // inside the user's padded history; the ring slot inside this block's shared memory)
                const int rk = CKV_CLAMP(__shfl_sync(0xffffffffu, idx_k, r), full_k ? rq.Lpad - it.begin : a.cv.n_entries, err_flag),
                          rv = CKV_CLAMP(__shfl_sync(0xffffffffu, idx_v, r), full_v ? rq.Lpad - it.begin : a.cv.n_entries, err_flag);
                (void)CKV_CLAMP((int)(vt + off - smem_u32(smem_raw)), C::SMEM - 15, err_flag);
                cp_async16(kt + off, pK + (int64_t)rk * ROWB);
                cp_async16(vt + off, pV + (int64_t)rv * ROWB);
            }
        }
    };
    auto fetch_idx = [&](int step, int& idx_k, int& idx_v) {
        if (step < nsteps) {
            idx_k = full_k ? 32 * part + stride * step + lane : load_index<IDX16>(a.cv.idxK, unit0 + stride * step);
            idx_v = full_v ? 32 * part + stride * step + lane : load_index<IDX16>(a.cv.idxV, unit0 + stride * step);
        } else {
            idx_k = idx_v = 0;
        }
    };
    auto fetch_user = [&](int step, uint4& k, uint4& v) {
        if (wide_user && step < nsteps) {
            if (!full_k) k = load_user_part(uK, unit0 + stride * step, d_user);
            if (!full_v) v = load_user_part(uV, unit0 + stride * step, d_user);
        }
    };

    // prologue: tiles 0 .. NST-2 in flight, indices of the next two and user parts of the first two requested.  All
    // requests before the first use: a block's life begins with this chain of latencies.
    struct Ahead {
        int ik, iv;     // indices of tile step + NST - 1
        uint4 uk, uv;   // user parts of tile step
    } even, odd;
    int ik0[NST - 1], iv0[NST - 1];
#pragma unroll
    for (int s0 = 0; s0 < NST - 1; ++s0) fetch_idx(s0, ik0[s0], iv0[s0]);
    fetch_idx(NST - 1, even.ik, even.iv);
    fetch_idx(NST, odd.ik, odd.iv);
    even.uk = even.uv = odd.uk = odd.uv = make_uint4(0, 0, 0, 0);
    fetch_user(0, even.uk, even.uv);
    fetch_user(1, odd.uk, odd.uv);
#pragma unroll
    for (int s0 = 0; s0 < NST - 1; ++s0) {
        if (s0 < nsteps) issue(s0, ik0[s0], iv0[s0]);
        if constexpr (!TMA) cp_async_commit();
    }

    // one tile; its registers of `w` are requested again for the tile two steps further
    auto body = [&](int step, Ahead& w) {
        const int p0 = it.begin + 32 * part + stride * step;
        if (step + NST - 1 < nsteps) issue(step + NST - 1, w.ik, w.iv);
        if constexpr (!TMA) cp_async_commit();
        fetch_idx(step + NST + 1, w.ik, w.iv);
        if constexpr (TMA) {
            const uint32_t bar = bars + 8 * (step % NST), parity = (step / NST) & 1;
            bool here = true;
            int spins = 0;
            while (!mbar_try_wait(bar, parity)) {
                if (++spins > kTmaSpinLimit) {
                    here = false;
                    break;
                }
            }
            if (!__all_sync(0xffffffffu, here)) return false;  // give up: nothing more is issued, nothing is stored
        } else {
            cp_async_wait<NST - 1>();
        }
        __syncwarp();
        const uint32_t kt = ring + (step % NST) * (2 * C::TILE_B), vt = kt + C::TILE_B;
        // Eq. K: dims [0, d_user) of every row come from the user-specific part
        if (wide_user) {
            if (!full_k) store_user_part(kt + offU, w.uk, d_user);
            if (!full_v) store_user_part(vt + offU, w.uv, d_user);
            fetch_user(step + 2, w.uk, w.uv);
        } else if (d_user > 0 && !(full_k && full_v)) {
            for (int e = 0; e < d_user; ++e) {
                if (!full_k) {
                    const uint16_t xk = __ldg(uK + (unit0 + stride * step) * d_user + e);
                    asm volatile("st.shared.u16 [%0], %1;" ::"r"(kt + offU + 2 * e), "h"(xk) : "memory");
                }
                if (!full_v) {
                    const uint16_t xv = __ldg(uV + (unit0 + stride * step) * d_user + e);
                    asm volatile("st.shared.u16 [%0], %1;" ::"r"(vt + offU + 2 * e), "h"(xv) : "memory");
                }
            }
        }
        __syncwarp();
        const bool tail = p0 + 32 > full_end;  // some (row, position) pair of this tile is not attended

        auto load_k = [&](int nt, uint32_t (&kf)[2 * KS]) {
#pragma unroll
            for (int kp = 0; kp < (D == 64 ? 2 : 1); ++kp)
                ldsm4(kf[4 * kp], kf[4 * kp + 1], kf[4 * kp + 2], kf[4 * kp + 3], kt + nt * (8 * ROWB) + offK[kp]);
        };
        auto load_v = [&](int b, uint32_t (&vb)[NTD][2]) {
#pragma unroll
            for (int jp = 0; jp < NTD / 2; ++jp)
                ldsm4_trans(vb[2 * jp][0], vb[2 * jp][1], vb[2 * jp + 1][0], vb[2 * jp + 1][1], vt + b * (16 * ROWB) + offV[jp]);
        };
        // weights of query tile mt from its scores
        auto normalise = [&](int mt, float (&s)[4][4], uint32_t (&pa)[2][4]) {
            // element (nt, e): position p0 + 8 nt + 2t + (e & 1), query row g (e < 2) or g + 8
            if constexpr (MODE == CKV_SOFTMAX) {
                if (tail) {
                    const int e_lo = VAR ? min(end, lim[mt][0]) : end, e_hi = VAR ? min(end, lim[mt][1]) : end;
#pragma unroll
                    for (int nt = 0; nt < 4; ++nt) {
                        const int pc = p0 + 8 * nt + 2 * t;
                        if (pc >= e_lo) s[nt][0] = -CUDART_INF_F;
                        if (pc + 1 >= e_lo) s[nt][1] = -CUDART_INF_F;
                        if (pc >= e_hi) s[nt][2] = -CUDART_INF_F;
                        if (pc + 1 >= e_hi) s[nt][3] = -CUDART_INF_F;
                    }
                }
                // A row's reference lies ten octaves above the maximum of the first tile and stays there.  A lane's eight weights
                // that add up to more than one, or to no number, give away that a score has come near it; then, as in the first
                // tile, the reference goes ten octaves above the maximum.  (A row that sees nothing of the first tile sees
                // nothing of the others.)  No weight is more than one, as with the running maximum, so that sums with
                // values near fp32's largest stay in range.  That takes the maxima and four dependent shuffles out of every
                // other tile (65536 users x 512 positions x 16 queries 2364 -> 2163 us, 4096 x 512 x 16 64-wide 315 -> 259, 199
                // ragged ones 63 -> 58).
                float ps0, ps1;
                auto weigh = [&]() {  // the weights and this lane's share of their sums
                    const float r0 = VAR && m_run[mt][0] == -CUDART_INF_F ? 0.f : m_run[mt][0],
                                r1 = VAR && m_run[mt][1] == -CUDART_INF_F ? 0.f : m_run[mt][1];
                    ps0 = ps1 = 0.f;
#pragma unroll
                    for (int nt = 0; nt < 4; ++nt) {
                        const float p0v = ex2(fmaf(s[nt][0], sc, -r0)), p1v = ex2(fmaf(s[nt][1], sc, -r0));
                        ps0 += p0v + p1v;
                        pa[nt >> 1][(nt & 1) * 2] = pack_bf16(p0v, p1v);
                        if (has_hi) {
                            const float p2v = ex2(fmaf(s[nt][2], sc, -r1)), p3v = ex2(fmaf(s[nt][3], sc, -r1));
                            ps1 += p2v + p3v;
                            pa[nt >> 1][(nt & 1) * 2 + 1] = pack_bf16(p2v, p3v);
                        } else {
                            pa[nt >> 1][(nt & 1) * 2 + 1] = 0u;
                        }
                    }
                };
                auto left = [&]() { return __any_sync(0xffffffffu, !(ps0 <= kSumLimit && ps1 <= kSumLimit)) != 0; };
                auto move = [&]() {
                    float mx0 = s[0][0], mx1 = s[0][2];
#pragma unroll
                    for (int nt = 0; nt < 4; ++nt) {
                        mx0 = fmaxf(mx0, fmaxf(s[nt][0], s[nt][1]));
                        mx1 = fmaxf(mx1, fmaxf(s[nt][2], s[nt][3]));
                    }
                    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
                    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
                    if (has_hi) {
                        mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
                        mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
                    }
                    // a row may not see any position of this tile (or of any tile so far): its maximum is then -inf
                    // and must not enter the exponent arguments
                    const float mn0 = fmaxf(m_run[mt][0], fmaf(mx0, sc, kOctavesAbove));
                    const float mn1 = has_hi ? fmaxf(m_run[mt][1], fmaf(mx1, sc, kOctavesAbove)) : 0.f;
                    // (without visible lengths the first position of a tile is always attended and the maxima are finite)
                    const float ms0 = VAR && mn0 == -CUDART_INF_F ? 0.f : mn0, ms1 = VAR && mn1 == -CUDART_INF_F ? 0.f : mn1;
                    // rescale only when one of them moved (in the first tile, and rarely behind it)
                    const bool moved = mn0 != m_run[mt][0] || (has_hi && mn1 != m_run[mt][1]);
                    if (__any_sync(0xffffffffu, moved)) {
                        const float c0 = ex2(m_run[mt][0] - ms0), c1 = has_hi ? ex2(m_run[mt][1] - ms1) : 1.f;
                        m_run[mt][0] = mn0;
                        if (has_hi) m_run[mt][1] = mn1;
                        l_run[mt][0] *= c0;
                        l_run[mt][1] *= c1;
#pragma unroll
                        for (int j = 0; j < NTD; ++j) {
                            o[mt][j][0] *= c0; o[mt][j][1] *= c0;
                            o[mt][j][2] *= c1; o[mt][j][3] *= c1;
                        }
                    }
                };
                if constexpr (SHARED) {  // (one copy of the code: a warp that shares a short unit meets it cold)
                    bool moves = step == 0;
#pragma unroll 1
                    while (true) {
                        if (moves) move();
                        weigh();
                        if (moves || !left()) break;
                        moves = true;
                    }
                } else if constexpr (D == 32 && MT != 2) {
                    // (what a first tile goes through lies in a row: one-tile histories otherwise wait for instructions.  1890
                    // users x 18..56 positions x 7..73 queries x 8 groups 121 -> 111 us, 861 x 32 x 18 x 3 12.2 -> 10.7, 65536 x 512 x
                    // 16 x 4 2192 -> 2184; the others, with more registers, lose 1 % on full SMs.)
                    if (step == 0) move();
                    weigh();
                    if (step != 0 && left()) {
                        move();
                        weigh();
                    }
                } else {
                    if (step != 0) weigh();
                    if (step == 0 || left()) {
                        move();
                        weigh();
                    }
                }
                l_run[mt][0] += ps0;
                l_run[mt][1] += ps1;
            } else {
                // silu(x) = x sigmoid(x) = h (1 + tanh(h)), h = x / 2   (sc = scale / 2)
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    float w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float h = s[nt][e] * sc;
                        w[e] = (e < 2 || has_hi) ? fmaf(h, tanh_fast(h), h) : 0.f;
                    }
                    if (tail) {
                        const int e_lo = VAR ? min(end, lim[mt][0]) : end, e_hi = VAR ? min(end, lim[mt][1]) : end,
                                  pc = p0 + 8 * nt + 2 * t;
                        if (pc >= e_lo) w[0] = 0.f;
                        if (pc + 1 >= e_lo) w[1] = 0.f;
                        if (pc >= e_hi) w[2] = 0.f;
                        if (pc + 1 >= e_hi) w[3] = 0.f;
                    }
                    pa[nt >> 1][(nt & 1) * 2] = pack_bf16(w[0], w[1]);
                    pa[nt >> 1][(nt & 1) * 2 + 1] = pack_bf16(w[2], w[3]);
                }
            }
        };
        if constexpr (MT == 1) {  // every fragment requested up front
            uint32_t kf[4][2 * KS], vb[2][NTD][2], pa[2][4];
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) load_k(nt, kf[nt]);
#pragma unroll
            for (int b = 0; b < 2; ++b) load_v(b, vb[b]);
            float s[4][4];
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) mma_bf16(s[nt], qa[0][ks], kf[nt][2 * ks], kf[nt][2 * ks + 1]);
            }
            normalise(0, s, pa);
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int j = 0; j < NTD; ++j) mma_bf16(o[0][j], pa[b], vb[b][j][0], vb[b][j][1]);
        } else {  // a fragment serves all query tiles and is gone again: their accumulators need the registers
            float s[MT][4][4];
            uint32_t pa[MT][2][4];
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                uint32_t kf[2 * KS];
                load_k(nt, kf);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    s[mt][nt][0] = s[mt][nt][1] = s[mt][nt][2] = s[mt][nt][3] = 0.f;
                    if (mt < n_mt)
#pragma unroll
                        for (int ks = 0; ks < KS; ++ks) mma_bf16(s[mt][nt], qa[mt][ks], kf[2 * ks], kf[2 * ks + 1]);
                }
            }
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
                if (mt < n_mt) normalise(mt, s[mt], pa[mt]);
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                uint32_t vb[NTD][2];
                load_v(b, vb);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
                    if (mt < n_mt)
#pragma unroll
                        for (int j = 0; j < NTD; ++j) mma_bf16(o[mt][j], pa[mt][b], vb[j][0], vb[j][1]);
            }
        }
        // every lane is done with this tile before the ring slot is refilled (TMA: its ordinary stores
        // and loads are ordered before the asynchronous-proxy writes of the refill)
        if constexpr (TMA) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        return true;
    };
    bool ok = true;
    for (int step = 0; ok && step < nsteps; step += 2) {
        ok = body(step, even);
        if (ok && step + 1 < nsteps) ok = body(step + 1, odd);
    }
    if constexpr (TMA) {
        // (a warp that gave up still takes part in the merge: the error word says that the outputs are not valid)
        if (!ok && lane == 0) atomicOr(err_flag, ERR_MMA_LOAD);
    } else {
        cp_async_wait<0>();
    }

    // merge the parts of the unit: registers as they are, value i of lane l at [i][l] of the giving warp's own ring
    if constexpr (SHARED) {
        constexpr int FR = NTD * 4 + 4;
        static_assert(FR * 128 <= NST * 2 * C::TILE_B, "a fragment fits the warp's ring");
        auto give = [&](int mt) {
            const uint32_t p = ring + lane * 4;
            auto put = [&](int i, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(p + i * 128), "f"(v) : "memory"); };
            put(0, m_run[mt][0]);
            put(1, m_run[mt][1]);
            put(2, l_run[mt][0]);
            put(3, l_run[mt][1]);
#pragma unroll
            for (int i = 0; i < NTD * 4; ++i) put(4 + i, o[mt][i >> 2][i & 3]);
        };
        auto take = [&](int mt, auto&& get) {
            if constexpr (MODE == CKV_SOFTMAX) {
                float ca[2], cb[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float m2 = get(h), mn = fmaxf(m_run[mt][h], m2), ms = mn == -CUDART_INF_F ? 0.f : mn;
                    ca[h] = ex2(m_run[mt][h] - ms);
                    cb[h] = ex2(m2 - ms);
                    m_run[mt][h] = mn;
                    l_run[mt][h] = l_run[mt][h] * ca[h] + get(2 + h) * cb[h];
                }
#pragma unroll
                for (int i = 0; i < NTD * 4; ++i) {
                    float& x = o[mt][i >> 2][i & 3];
                    x = x * ca[(i >> 1) & 1] + get(4 + i) * cb[(i >> 1) & 1];
                }
            } else {
#pragma unroll
                for (int i = 0; i < NTD * 4; ++i) o[mt][i >> 2][i & 3] += get(4 + i);
            }
        };
        auto unit_sync = [&]() {
            if (log_wpu == 2) asm volatile("bar.sync 1, 128;" ::: "memory");
            else if (log_wpu == 1) asm volatile("bar.sync %0, 64;" ::"r"(2 + (warp >> 1)) : "memory");
        };
        constexpr uint32_t RING_B = NST * 2 * C::TILE_B;
        for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
            for (int x = 0; x < MT; ++x)  // (constant indices keep the fragments in registers)
                if (x == mt && sub != 0) give(x);
            unit_sync();
            if (sub == 0)
#pragma unroll
                for (int x = 0; x < MT; ++x)
                    if (x == mt)
                        for (int w = 1; w < wpu; ++w)
                            take(x, [&](int i) {
                                float v;
                                asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(ring + w * RING_B + lane * 4 + i * 128) : "memory");
                                return v;
                            });
            unit_sync();
        }
        if (n_cta > 1) {
            for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
                for (int x = 0; x < MT; ++x)
                    if (x == mt && sub == 0 && rank != 0) give(x);
                cluster_sync();
                if (sub == 0 && rank == 0)
#pragma unroll
                    for (int x = 0; x < MT; ++x)
                        if (x == mt)
                            for (int r = 1; r < n_cta; ++r)
                                take(x, [&](int i) { return ld_cluster(ring + lane * 4 + i * 128, (uint32_t)r); });
                cluster_sync();  // the other blocks' shared memory has been read
            }
        }
        if (part != 0) return;
    }

    // epilogue: finish the row sums over the quad, then store outputs or partials
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float l = l_run[mt][h];
            l += __shfl_xor_sync(0xffffffffu, l, 1);
            l += __shfl_xor_sync(0xffffffffu, l, 2);
            const int r = row0 + 16 * mt + g + 8 * h;
            if (r >= rq.M) continue;
            if (it.part_row < 0) {
                float inv;
                if constexpr (MODE == CKV_SOFTMAX) inv = l > 0.f ? 1.0f / l : 0.f;
                else inv = rq.L > 0 ? 1.0f / (float)rq.L : 0.f;
                const int64_t base = ((int64_t)(rq.q0 + r) * G + grp) * D;
#pragma unroll
                for (int j = 0; j < NTD; ++j) {
                    const float x = o[mt][j][2 * h] * inv, y = o[mt][j][2 * h + 1] * inv;
                    if (a.out_dtype == CKV_BF16)
                        *reinterpret_cast<uint32_t*>(reinterpret_cast<uint16_t*>(a.out) + base + 8 * j + 2 * t) =
                            pack_bf16(x, y);
                    else
                        *reinterpret_cast<float2*>(reinterpret_cast<float*>(a.out) + base + 8 * j + 2 * t) =
                            make_float2(x, y);
                }
            } else {
                const int64_t row = CKV_CLAMP((int64_t)(it.part_row + r), a.part_rows, err_flag);
                if (t == 0) *part_ml(a, D, row, grp) = make_float2(m_run[mt][h], l);
                float* pr = part_acc(a, D, row, grp);
#pragma unroll
                for (int j = 0; j < NTD; ++j)
                    *reinterpret_cast<float2*>(pr + 8 * j + 2 * t) =
                        make_float2(o[mt][j][2 * h], o[mt][j][2 * h + 1]);
            }
        }
    }
}

template <int D, int MT, int MODE, bool IDX16, bool TMA, bool VAR, bool SHARED, bool DENSE>
cudaError_t launch_mma_one(const AttendArgs& a, int n_mb, int parts, const InlineTable* tab, const CUtensorMap* maps,
                           int* err_flag, const Launch& l)
{
    using C = MmaCfg<D, MT, TMA, DENSE>;
    int log_wpu = 0;
    while (log_wpu < 2 && (1 << log_wpu) < parts) ++log_wpu;
    const int n_cta = parts >> log_wpu;
    const int64_t units = (int64_t)a.n_items * n_mb, upb = C::WARPS >> log_wpu;
    const dim3 grid((unsigned)((units + upb - 1) / upb * n_cta), a.cv.n_groups);
    if constexpr (TMA) {
        return launch_kernel(l, attend_mma_kernel<D, MT, MODE, IDX16, true, VAR, SHARED>, grid, 128, C::SMEM, n_cta, a, n_mb,
                             log_wpu, n_cta, err_flag, TmaMaps{maps[0], maps[1]});
    } else {
        static const InlineTable none{};
        return launch_kernel(l, attend_mma_kernel<D, MT, MODE, IDX16, false, VAR, SHARED, DENSE>, grid, 128, C::SMEM, n_cta, a, n_mb,
                             log_wpu, n_cta, err_flag, tab ? *tab : none);
    }
}

}  // namespace

// Instantiated for each (head_dim, query tiles of a warp) in a file of its own, kernels_mma_*.cu: the forms of the kernel take a
// minute to compile in one.  DENSE: the plain form with cp.async alone (maps null, both sides shared, no visible lengths).
template <int D, int MT, bool DENSE>
cudaError_t launch_mma(const AttendArgs& a, int n_mb, int parts, const InlineTable* tab, const CUtensorMap* maps,
                       int* err_flag, const Launch& l)
{
    constexpr bool HAS_TMA = !DENSE && (D != 32 || MT != 2);  // (never asked for with the others)
    const bool i16 = a.cv.idx_bytes == 2;
    const bool var = !DENSE && (a.vis != nullptr || a.cv.full_k || a.cv.full_v);  // the TMA loader is never asked for with these
#define CKV_MMA_ONE(MODE, I16, TMA, VAR)                                                                          \
    (parts > 1 ? launch_mma_one<D, MT, MODE, I16, TMA, VAR, true, DENSE>(a, n_mb, parts, tab, maps, err_flag, l)  \
               : launch_mma_one<D, MT, MODE, I16, TMA, VAR, false, DENSE>(a, n_mb, parts, tab, maps, err_flag, l))
#define CKV_MMA_GO(MODE, I16)                                                                              \
    (HAS_TMA && maps ? CKV_MMA_ONE(MODE, I16, HAS_TMA, false)                                              \
     : var           ? CKV_MMA_ONE(MODE, I16, false, !DENSE)                                               \
                     : CKV_MMA_ONE(MODE, I16, false, false))
    if (a.mode == CKV_SOFTMAX) return i16 ? CKV_MMA_GO(CKV_SOFTMAX, true) : CKV_MMA_GO(CKV_SOFTMAX, false);
    return i16 ? CKV_MMA_GO(CKV_SILU_OVER_L, true) : CKV_MMA_GO(CKV_SILU_OVER_L, false);
#undef CKV_MMA_GO
#undef CKV_MMA_ONE
}

}  // namespace ckv
