// Prefill router (Sec. 4.3) on the tcgen05 tensor cores: I[i][g] = lowest j maximising x_i . W_g[j] + b_g[j].
//
// One CTA owns 384 positions of one group, as three blocks of 128, and every S-th share of the group's entries (S CTAs in
// a cluster share the positions when there are too few of them to fill the SMs).  The positions' inputs sit in TMEM
// (A operand, lane = position); the group's weight rows stream through a ring of shared-memory stages in tiles of 128
// entries (96 at d_in = 128; B operand, one swizzled TMA box per 64 inputs), and every tile is multiplied with all three
// blocks.  The bias is one more K = 16 step of the product, ones times the bias cut into three bf16 parts whose sum is the
// fp32 bias exactly (below 2^-100 the parts are those of 2^100 times the bias and meet 2^-100: bf16 has no room for the last
// of them there), so the read-out touches no shared memory for it.  A block has four read-out warps (thread = position =
// TMEM lane), an issuing warp and two accumulators of 64 columns (one of 96 at d_in = 128) of its own.  The read-out fetches
// an accumulator into registers, releases it at once, and keeps a running (best score, entry); the score matrix never
// leaves the SM.
// What bounds it: the turn of an accumulator, products -> commit -> read-out -> release -> products, some 800 to 1000
// clocks of latency of which the products are 160, and TMEM, which holds 384 columns of accumulators in turn; with that the
// tensor core is 82 % busy with bias and products at d_in = 64 (51 % before).  So the turn is kept short: the release is a named
// barrier of five warps (an mbarrier cost 340 clocks next to running products), the issuing warp waits for its tile
// before it, the products are issued under elect.sync from values known to be uniform (under "lane 0" the five of them
// took 380 clocks, now 200).  131072 positions x 16384 entries x 4 groups, d_in 64: 1250 us -> 880 (1250 TFLOP/s; 1197 with
// three blocks alone, 953 with the elected issue, 930 with accumulators of 128 columns and 152 registers a read-out
// thread instead of two of 64, 891 with the first tiles requested behind the inputs instead of beside them); d_in 32: 1165 ->
// 795; 10000 x 16384 x 2: 140 -> 71.  Three blocks and not two: a weight tile
// is fetched from L2 once for all of a CTA's positions, and three turns overlap.
// Every wait is bounded: a time-out raises the CTA's abort flag, the CTA drains, frees its TMEM and reports to the
// host.  The call then returns an error and its whole output is not valid: the CTA itself writes none, but others
// have, among them the first of its cluster, which takes the best entries of all of them as they stand.
#include <cuda_bf16.h>
#include <math_constants.h>

#include "ckv_internal.h"
#include "ptx_helpers.cuh"
#include "tensor_map.h"

namespace ckv {
namespace {

constexpr int kBlocks = 3, kRows = 128 * kBlocks;
constexpr int kEpiWarps = 4 * kBlocks, kIssueWarp = kEpiWarps, kLoadWarp = kIssueWarp + kBlocks;
constexpr int kThreadsRU = (kLoadWarp + 1) * 32;  // sixteen warps: 128 registers a thread
constexpr int kMaxClusterRU = 8;
constexpr uint32_t kSpin = 1u << 18, kSuspend = 4000;
constexpr float kTinyBias = 0x1p-100f;  // 0x0d80 in bf16

constexpr int kMaxStages = 8;
constexpr int kMaxAcc = 2;  // accumulators of a block
enum Bar { B_FULL = 0, B_EMPTY = kMaxStages, B_AFULL = 2 * kMaxStages, B_DRAIN = B_AFULL + kBlocks * kMaxAcc, B_COUNT };

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, const volatile int* abort_flag)
{
    for (uint32_t i = 0; i < kSpin; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
            "selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "r"(kSuspend)
            : "memory");
        if (ok) return true;
        if ((i & 31u) == 31u && *abort_flag) return false;
    }
    return false;
}
// Named barriers of an accumulator, for its block's four read-out warps and its issuing warp: "tile t has been read".  The
// read-out arrives and runs on; once a wait has run out it takes part as the issuing warp does.  Two barriers in turn: a warp that
// gives up on the next tile has arrived for this one already, and on the same barrier would count for the issuing warp, which
// then waited for good.
__device__ __forceinline__ int read_barrier(int acc, int tile) { return 1 + 2 * acc + (tile & 1); }
__device__ __forceinline__ void acc_arrive(int acc, int tile) { asm volatile("bar.arrive %0, 160;" ::"r"(read_barrier(acc, tile)) : "memory"); }
__device__ __forceinline__ void acc_sync(int acc, int tile) { asm volatile("bar.sync %0, 160;" ::"r"(read_barrier(acc, tile)) : "memory"); }
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit_to(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(acc)
        : "memory");
}
// shared-memory matrix descriptor, no swizzle: start address, leading / stride byte offsets (16-byte units), version 1
__device__ __forceinline__ uint64_t mat_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes)
{
    return (uint64_t)((addr & 0x3ffffu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) |
           ((uint64_t)(sbo_bytes >> 4) << 32) | (1ull << 46);
}
// instruction descriptor, kind::f16: fp32 accumulate, bf16 A and B, both K-major
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,"
        "%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void wait_ld32(uint32_t (&r)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                   "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                   "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}
// 16 / 32 consecutive columns of this thread's lane
__device__ __forceinline__ void st16(uint32_t taddr, const uint32_t* r)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void st8(uint32_t taddr, const uint32_t (&r)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
                 "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
__device__ __forceinline__ float max3f(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
template <int DIN>
struct RU {
    static constexpr int AN = DIN == 128 ? 96 : 64;        // columns of an accumulator
    static constexpr int ACCS = DIN == 128 ? 1 : 2;        // accumulators of a block
    static constexpr int TN = ACCS * AN;                   // entries per tile
    static constexpr int ROWB = DIN >= 64 ? 128 : 64;      // bytes of a row inside a TMA box = its swizzle span
    static constexpr int BOXES = DIN == 128 ? 2 : 1;       // boxes (of 64 inputs) per tile
    static constexpr int BOX = TN * ROWB;                  // bytes of a box
    static constexpr int TILE = BOXES * BOX;               // bytes of a weight tile
    static constexpr int STAGES = DIN == 128 ? 6 : 8;
    static constexpr int BIAS = TN * 32;                   // bytes of a tile's bias step (16 bf16 per entry)
    static constexpr int OFF_W = 0, OFF_BIAS = STAGES * TILE,
                         OFF_BEST = OFF_BIAS + STAGES * BIAS,  // [kRows] (score, entry), read by the cluster's first CTA
                         OFF_KEPT = OFF_BEST + kRows * 8,      // [8][kRows] four scores of a position's best chunk
                         OFF_BAR = OFF_KEPT + kRows * 128, OFF_ABORT = OFF_BAR + B_COUNT * 8, SMEM = OFF_ABORT + 16;
    static_assert(STAGES <= kMaxStages && SMEM <= 226 * 1024 && BOX % 1024 == 0, "shared memory");
    // TMEM: the accumulators of each block, the inputs of each block (two per column), the ones of the bias step
    static constexpr uint32_t COL_A = kBlocks * TN, COL_ONES = COL_A + kBlocks * (DIN / 2);
    static_assert(COL_ONES + 8 <= 512, "TMEM columns");
};
// Swizzled K-major operand (TMA box of ROWB-byte rows, groups of eight rows ROWB * 8 bytes apart).
template <int DIN>
__device__ __forceinline__ uint64_t swz_desc(uint32_t addr)
{
    constexpr uint64_t layout = RU<DIN>::ROWB == 128 ? 2 : 4;  // 128-byte / 64-byte swizzle
    return (uint64_t)((addr & 0x3ffffu) >> 4) | (1ull << 16) | ((uint64_t)(RU<DIN>::ROWB * 8 >> 4) << 32) | (1ull << 46) |
           (layout << 61);
}
// K-major core matrices of 16 bf16 per row, no swizzle: row r, 16-byte chunk c
__device__ __forceinline__ uint32_t step_off(int r, int c) { return (uint32_t)((r >> 3) * 256 + c * 128 + (r & 7) * 16); }

__device__ unsigned route_count[kRouteSlots];  // finished CTAs of the launch that holds the slot, zero between launches

template <int DIN>
__global__ void __launch_bounds__(kThreadsRU, 1)
    route_umma_kernel(const uint16_t* __restrict__ x, const __grid_constant__ CUtensorMap tmW, const float* __restrict__ bias,
                      int n, int m, int G, int32_t* __restrict__ out, int* flags, int slot, int n_split)
{
    using L = RU<DIN>;
    constexpr int TN = L::TN, AN = L::AN, ACCS = L::ACCS;
    extern __shared__ __align__(1024) unsigned char usm[];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t sb = s_u32(usm);
    auto bar = [&](int i) { return sb + L::OFF_BAR + 8u * (uint32_t)i; };
    volatile int* abort_flag = reinterpret_cast<volatile int*>(usm + L::OFF_ABORT);
    const int grp = blockIdx.y, split = (int)(blockIdx.x % (uint32_t)n_split);
    const int64_t row0 = (int64_t)(blockIdx.x / (uint32_t)n_split) * kRows;
    const int n_blocks = (int)min((n - row0 + 127) / 128, (int64_t)kBlocks);
    const float* bg = bias ? bias + (int64_t)grp * m : nullptr;
    // this CTA's tiles of the group's entries
    const int all_tiles = (m + TN - 1) / TN;
    const int tile0 = (int)((int64_t)all_tiles * split / n_split), n_tiles = (int)((int64_t)all_tiles * (split + 1) / n_split) - tile0;
    // a tile needs the bias step if there is a bias, or entries past the last one to rule out
    auto biased = [&](int t) { return bg != nullptr || (tile0 + t + 1) * TN > m; };

    // four read-out warps and one issuing warp per block of positions
    const int e = warp >> 2;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const int row = 128 * e + (warp & 3) * 32 + lane;  // this read-out thread's position
    // its inputs are requested before anything is set up (zero rows past the end)
    uint4 xin[DIN / 8];
    if (warp < 4 * n_blocks) {
        const uint4* xr = reinterpret_cast<const uint4*>(x + (row0 + row) * DIN);
        const bool in = row0 + row < n;
#pragma unroll
        for (int q = 0; q < DIN / 8; ++q) xin[q] = in ? __ldg(xr + q) : make_uint4(0, 0, 0, 0);
    }
    if (tid == 0) {
        for (int s = 0; s < L::STAGES; ++s) {
            bar_init(bar(B_FULL + s), 2);  // the loading warp, with the box's bytes and behind the bias step
            bar_init(bar(B_EMPTY + s), (uint32_t)n_blocks);
        }
        for (int e = 0; e < kBlocks * L::ACCS; ++e) bar_init(bar(B_AFULL + e), 1);
        bar_init(bar(B_DRAIN), kBlocks);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kIssueWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_u32(&tmem_slot)), "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp == kLoadWarp) {  // the second chunk of every bias slot stays zero (slots are whole groups of eight rows)
        for (int r = lane; r < TN * L::STAGES; r += 32)
            *reinterpret_cast<uint4*>(usm + L::OFF_BIAS + step_off(r, 1)) = make_uint4(0, 0, 0, 0);
        fence_async();
    }
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = tmem_slot;
    bool ok = true;
    float best = -CUDART_INF_F;
    int arg = 0;

    if (warp < 4 * n_blocks) {
        // the positions' inputs, once: two bf16 per column
#pragma unroll
        for (int h = 0; h < DIN / 32; ++h) {
            uint32_t v[16];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint4 w = xin[4 * h + q];
                v[4 * q] = w.x; v[4 * q + 1] = w.y; v[4 * q + 2] = w.z; v[4 * q + 3] = w.w;
            }
            st16(tmem + lane_base + L::COL_A + e * (DIN / 2) + 16 * h, v);
        }
        if (e == 0) {  // A operand of the bias step: three ones and three times kTinyBias per position
            const uint32_t ones[8] = {0x3f803f80u, 0x0d803f80u, 0x0d800d80u, 0, 0, 0, 0, 0};
            st8(tmem + lane_base + L::COL_ONES, ones);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    if (warp < kLoadWarp) {  // (the loading warp is on its way: the first tiles travel meanwhile)
        tc_before();
        asm volatile("bar.sync 15, %0;" ::"n"(kLoadWarp * 32) : "memory");
        tc_after();
    }

    if (warp < kEpiWarps) {
        // ------------------------------------------------------------ running arg-max, thread = position
        // Only the maximum of 32 columns is compared with the running best; a chunk that has a new best is kept as it is
        // in shared memory (four scores of a thread per 16-byte word, threads side by side), and the one that is left at
        // the end is searched for its first maximal column: the search in place took the ALU pipe from 45 to 67 % (1.29 ->
        // 1.20 ms of the case above).  Chunks come in increasing order of the entries and the comparison is strict, so the lowest entry wins
        // among equals; past the last entry the bias is -inf.
        uint4* const kept = reinterpret_cast<uint4*>(usm + L::OFF_KEPT) + row;
        auto look = [&](const uint32_t (&v)[32], int j0) {
            float m0 = __uint_as_float(v[0]), m1 = __uint_as_float(v[1]);
#pragma unroll
            for (int q = 2; q < 30; q += 4) {
                m0 = max3f(m0, __uint_as_float(v[q]), __uint_as_float(v[q + 1]));
                m1 = max3f(m1, __uint_as_float(v[q + 2]), __uint_as_float(v[q + 3]));
            }
            const float mx = max3f(fmaxf(m0, m1), __uint_as_float(v[30]), __uint_as_float(v[31]));
            if (mx > best) {
                best = mx;
                arg = j0;
#pragma unroll
                for (int q = 0; q < 8; ++q) kept[q * kRows] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
        };
        const uint32_t tacc = tmem + lane_base + (uint32_t)(TN * e);
        for (int t = 0; e < n_blocks && t < n_tiles; ++t) {
#pragma unroll
            for (int h = 0; h < ACCS; ++h) {
                const int acc = ACCS * e + h;
                if (ok) {
                    ok = bar_wait(bar(B_AFULL + acc), t & 1, abort_flag);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) *abort_flag = 1;
                }
                if (!ok) {
                    if (t + 1 < n_tiles) acc_sync(acc, t);
                    continue;
                }
                tc_after();
                // the whole accumulator into registers, so that it is free again before it is looked at
                uint32_t v[AN / 32][32];
#pragma unroll
                for (int c = 0; c < AN / 32; ++c) ld32(tacc + AN * h + 32 * c, v[c]);
#pragma unroll
                for (int c = 0; c < AN / 32; ++c) wait_ld32(v[c]);
                tc_before();
                if (t + 1 < n_tiles) acc_arrive(acc, t);
#pragma unroll
                for (int c = 0; c < AN / 32; ++c) look(v[c], (tile0 + t) * TN + AN * h + 32 * c);
            }
        }
        if (best > -CUDART_INF_F) {
            int first = 0;
#pragma unroll
            for (int q = 7; q >= 0; --q) {
                const uint4 w = kept[q * kRows];
                if (__uint_as_float(w.w) == best) first = 4 * q + 3;
                if (__uint_as_float(w.z) == best) first = 4 * q + 2;
                if (__uint_as_float(w.y) == best) first = 4 * q + 1;
                if (__uint_as_float(w.x) == best) first = 4 * q;
            }
            arg += first;
        }
    } else if (warp < kIssueWarp + kBlocks) {
        // ------------------------------------------------------------ MMA issue, one warp per block
        constexpr uint32_t idesc = idesc_bf16(128, AN);
        const int blk = warp - kIssueWarp;
        const uint32_t d = tmem + (uint32_t)(TN * blk), at = tmem + L::COL_A + blk * (DIN / 2), ones = tmem + L::COL_ONES;
        int s = 0;
        uint32_t par = 0;
        for (int t = 0; blk < n_blocks && t < n_tiles; ++t) {
            if (ok) {  // (the tile has usually been there for long: this wait lies before the one that paces the block)
                ok = bar_wait(bar(B_FULL + s), par, abort_flag);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) *abort_flag = 1;
            }
#pragma unroll
            for (int h = 0; h < ACCS; ++h) {
                if (t > 0) acc_sync(ACCS * blk + h, t - 1);
                if (ok && elect_one()) {
                    tc_after();
                    // (entries AN h and up of the tile: whole groups of eight rows further on)
                    const uint64_t w = swz_desc<DIN>(sb + L::OFF_W + s * L::TILE + AN * h * L::ROWB);
#pragma unroll
                    for (int ks = 0; ks < DIN / 16; ++ks)
                        mma_ts(d + AN * h, at + 8 * ks, w + (uint64_t)(((ks & 3) * 32 + (ks >> 2) * L::BOX) >> 4), idesc, ks > 0);
                    if (biased(t)) mma_ts(d + AN * h, ones, mat_desc(sb + L::OFF_BIAS + s * L::BIAS + AN * h * 32, 128, 256), idesc, 1u);
                    tc_commit_to(bar(B_AFULL + ACCS * blk + h));
                    if (h == ACCS - 1) tc_commit_to(bar(B_EMPTY + s));
                }
                __syncwarp();
            }
            if (++s == L::STAGES) {
                s = 0;
                par ^= 1;
            }
        }
        // nothing of this CTA may still run on the tensor core at teardown
        if (elect_one()) tc_commit_to(bar(B_DRAIN));
        volatile int never = 0;
        if (!bar_wait(bar(B_DRAIN), 0, &never)) *abort_flag = 1;
        __syncwarp();
    } else {
        // ------------------------------------------------------------ weight tiles, and their bias steps
        // b = hi + mid + lo, bf16 each, exactly.  Two tiles at a time: the waits, the fence and the hand-over are a chain.
        constexpr int kPer = TN / 32;
        auto load_bias = [&](int t, float (&b)[2 * kPer]) {
#pragma unroll
            for (int i = 0; i < 2 * kPer; ++i) {
                const int j = (tile0 + t) * TN + 32 * i + lane;
                b[i] = j < m ? (bg ? __ldg(bg + j) : 0.f) : -CUDART_INF_F;
            }
        };
        float nxt[2 * kPer];
        load_bias(0, nxt);
        int issued = 0, handed = 0;  // tiles whose copies have been issued / that have been handed over
        for (int t = 0; t < n_tiles; t += 2) {
            float cur[2 * kPer];
#pragma unroll
            for (int i = 0; i < 2 * kPer; ++i) cur[i] = nxt[i];
            load_bias(t + 2, nxt);
            const int n_t = min(2, n_tiles - t);
            for (int h = 0; h < n_t; ++h) {
                const int s = (t + h) % L::STAGES;
                ok = bar_wait(bar(B_EMPTY + s), (((t + h) / L::STAGES) & 1) ^ 1, abort_flag);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (lane == 0) {
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar(B_FULL + s)), "r"(L::TILE)
                                 : "memory");
#pragma unroll
                    for (int i = 0; i < L::BOXES; ++i)
                        asm volatile(
                            "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
                            "%3}], [%4];" ::"r"(sb + L::OFF_W + s * L::TILE + i * L::BOX),
                            "l"(&tmW), "r"(64 * i), "r"(grp * m + (tile0 + t + h) * TN), "r"(bar(B_FULL + s))
                            : "memory");
                }
                ++issued;
            }
            if (!ok) break;
            if (biased(t + n_t - 1)) {
#pragma unroll
                for (int i = 0; i < 2 * kPer; ++i) {
                    if (i >= kPer && n_t < 2) break;
                    const bool tiny = fabsf(cur[i]) < kTinyBias;
                    const float b = tiny ? cur[i] / kTinyBias : cur[i];
                    // (a NaN whose upper half alone would be an infinity stays one)
                    const uint32_t hi = (__float_as_uint(b) & 0xffff0000u) | (b != b ? 0x400000u : 0u);
                    const float r1 = isfinite(b) ? b - __uint_as_float(hi) : 0.f;
                    const uint32_t mid = __float_as_uint(r1) & 0xffff0000u, lo = __float_as_uint(r1 - __uint_as_float(mid));
                    *reinterpret_cast<uint4*>(usm + L::OFF_BIAS + (t + i / kPer) % L::STAGES * L::BIAS + step_off(32 * (i % kPer) + lane, 0)) =
                        tiny ? make_uint4(0, hi, (mid >> 16) | lo, 0) : make_uint4((hi >> 16) | mid, lo >> 16, 0, 0);
                }
                fence_async();
            }
            __syncwarp();
            if (lane < n_t) bar_arrive(bar(B_FULL + (t + lane) % L::STAGES));
            handed += n_t;
        }
        if (!ok && lane == 0) {
            *abort_flag = 1;
            // the copies in flight land before the CTA ends
            volatile int never = 0;
            for (int k = handed; k < issued; ++k) bar_arrive(bar(B_FULL + k % L::STAGES));
            for (int k = issued > L::STAGES ? issued - L::STAGES : 0; k < issued; ++k)
                bar_wait(bar(B_FULL + k % L::STAGES), (k / L::STAGES) & 1, &never);
        }
        __syncwarp();
    }

    tc_before();
    __syncthreads();
    tc_after();
    // (the TMEM goes back before the CTA waits for the others of its cluster: two clusters that had each other's SMs
    // to wait for could otherwise block each other)
    if (warp == kIssueWarp)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    // the CTAs of a cluster looked at different entries: the first of them, in the order of the entries, takes the best
    if (n_split > 1) {
        if (warp < kEpiWarps) {
            float* mine = reinterpret_cast<float*>(usm + L::OFF_BEST) + 2 * row;
            mine[0] = best;
            mine[1] = __int_as_float(arg);
        }
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (split == 0 && warp < kEpiWarps) {
            for (int r = 1; r < n_split; ++r) {
                uint32_t remote;
                float b2, a2;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(sb + L::OFF_BEST + 8 * row), "r"(r));
                asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(b2), "=f"(a2) : "r"(remote) : "memory");
                if (b2 > best) {
                    best = b2;
                    arg = __float_as_int(a2);
                }
            }
        }
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    if (warp < kEpiWarps && split == 0 && !*abort_flag && row0 + row < n) out[(row0 + row) * G + grp] = arg;
    report_done(slot >= 0 ? Report{flags, flags + 1, &route_count[slot]} : Report{flags}, *abort_flag != 0, gridDim.x * gridDim.y);
}

// The weights as rows of `d_in` inputs, boxes of a tile's rows and at most 64 inputs.
bool make_weight_map(int d_in, int64_t rows, int tile_rows, const void* W, CUtensorMap* map)
{
    return encode_rows(map, W, d_in, rows, d_in < 64 ? d_in : 64, tile_rows, d_in < 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
}

template <int DIN>
cudaError_t launch_t(const void* x, const void* W, const float* bias, int n, int m, int G, int32_t* out, int* flags,
                     int* slot, cudaStream_t s)
{
    CUtensorMap map;
    if (!make_weight_map(DIN, (int64_t)G * m, RU<DIN>::TN, W, &map)) return cudaErrorInvalidValue;
    // CTAs that share a block of positions: as many as shorten the run most, counting whole rounds of CTAs over the SMs and
    // sixteen tiles' time per CTA: 4 us until the first product is there and for the end, and more for the first
    // tiles, in which most chunks bring a new best (40 000 positions x 4096 entries x 4 groups: 106 us; 119 by four tiles).  A
    // cluster's CTAs have to lie side by side: of 148 SMs clusters of four fill 132, clusters of eight 120 (3359 positions x
    // 1424 entries x 2 groups 26.6 us in 18 clusters of eight, 18.9 in clusters of four).  A CTA with one or two blocks of positions
    // is done sooner, so that rounds are counted by CTAs and, twice, by blocks.  (Of 1400 shapes of 200 to 100 000
    // positions and 64 to 16384 entries this loses 0.3 % in the mean against the best number, 10 % at most; with every SM counted,
    // CTAs alone and fourteen tiles 0.9 and 47.)
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t ctas = (int64_t)((n + kRows - 1) / kRows) * G, tiles = (m + RU<DIN>::TN - 1) / RU<DIN>::TN;
    const int64_t blocks = (int64_t)((n + 127) / 128) * G;
    int split = 1;
    int64_t best = INT64_MAX;
    for (int sp = 1; sp <= kMaxClusterRU && sp <= tiles; sp *= 2) {
        const int64_t room = (int64_t)kBlocks * (sp <= 2 ? sms : sms * (sp == 4 ? 132 : 120) / 148);
        const int64_t rounds = (kBlocks * ctas * sp + room - 1) / room + 2 * ((blocks * sp + room - 1) / room);
        const int64_t cost = rounds * ((tiles + sp - 1) / sp + 16);
        if (cost < best) {
            best = cost;
            split = sp;
        }
    }
    const dim3 grid((unsigned)((n + kRows - 1) / kRows * split), (unsigned)G);
    if (ctas * split > sms) *slot = -1;  // several rounds: the report at the end of each CTA would delay the next
    return launch_kernel(Launch{s, nullptr, nullptr}, route_umma_kernel<DIN>, grid, kThreadsRU, RU<DIN>::SMEM, split,
                         (const uint16_t*)x, map, bias, n, m, G, out, flags, *slot, split);
}

}  // namespace

cudaError_t launch_route_umma(int d_in, const void* x, const void* W, const float* bias, int n, int n_entries, int G,
                              int32_t* out, int* flags, int* slot, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    switch (d_in) {
        case 32: return launch_t<32>(x, W, bias, n, n_entries, G, out, flags, slot, s);
        case 64: return launch_t<64>(x, W, bias, n, n_entries, G, out, flags, slot, s);
        default: return launch_t<128>(x, W, bias, n, n_entries, G, out, flags, slot, s);
    }
}

}  // namespace ckv
