// Prefill router (Sec. 4.3) on the tcgen05 tensor cores: I[i][g] = lowest j maximising x_i . W_g[j] + b_g[j].
//
// One CTA owns 256 positions of one group, as two blocks of 128, and every S-th share of the group's entries (S CTAs in
// a cluster share the positions when there are too few of them to fill the SMs).  The positions' inputs sit in TMEM
// (A operand, lane = position); the group's weight rows stream through a ring of shared-memory stages in tiles of 128
// entries (B operand, one swizzled TMA box per tile), and every tile is multiplied with both blocks.  The bias is one
// more K = 16 step of the product, ones times the bias cut into three bf16 parts whose sum is the fp32 bias exactly (below
// 2^-100 the parts are those of 2^100 times the bias and meet 2^-100: bf16 has no room for the last of them there), so
// the read-out touches no shared memory.  One thread per block issues the products into three 128-column TMEM
// accumulators in turn; two groups of four warps, one per block (thread = position = TMEM lane), fetch their accumulator
// into registers, release it at once, and keep a running (best score, entry); the score matrix never leaves the SM.
// What bounds it: a product takes 64 clocks (five per block and tile at d_in = 64), but every barrier operation next to
// running products takes its thread about 200, so an issuing thread spends 1150 clocks on a step (225 on the stage, 340 on
// the accumulator, 430 in the products, 130 in the commits), and two of them set the pace.  Measured on 131072 positions
// x 16384 entries x 4 groups, d_in = 64: 1.23 ms (895 TFLOP/s), with one issuing thread 1.73; with A and the bias in
// shared memory, whose fetch competed with the B operand for its 128 bytes per clock, 2.04.  Four issuing threads leave
// the read-out 128 registers (spills: 1.34 ms); four accumulators of 96 columns, each with its own issuing thread and
// read-out group: 1.41.
// Every wait is bounded: a time-out raises the CTA's abort flag, the CTA drains, frees its TMEM and reports through
// the error word.  The call then returns an error and its whole output is not valid: the CTA itself writes none, but others
// have, among them the first of its cluster, which takes the best entries of all of them as they stand.
#include <cuda_bf16.h>
#include <math_constants.h>

#include "ckv_internal.h"
#include "tensor_map.h"

namespace ckv {
namespace {

constexpr int kRows = 256, kTileN = 128, kAcc = 3;
constexpr int kEpiWarps = 8, kIssueWarp = kEpiWarps, kIssuers = 2, kLoadWarp = kIssueWarp + kIssuers, kBiasWarp = kLoadWarp + 1;
constexpr int kThreadsRU = (kBiasWarp + 1) * 32;  // twelve warps: 168 registers for a read-out thread's 128 columns
constexpr int kMaxClusterRU = 8;
constexpr uint32_t kSpin = 1u << 18, kSuspend = 4000;
constexpr float kTinyBias = 0x1p-100f;  // 0x0d80 in bf16
enum { ERR_ROUTE = 64 };

// A step k is (tile, block); it uses accumulator k mod 3.  With two blocks an accumulator goes from one block to the
// other, so that its uses are told apart by barriers per step mod 6: each has one waiting role, which meets every phase.
constexpr int kMaxStages = 8, kAccBars = 2 * kAcc;
enum Bar { B_FULL = 0, B_EMPTY = kMaxStages, B_AFULL = 2 * kMaxStages, B_AEMPTY = B_AFULL + kAccBars, B_DRAIN = B_AEMPTY + kAccBars, B_COUNT };

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __noinline__ bool bar_wait(uint32_t bar, uint32_t parity, const volatile int* abort_flag)
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
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit_to(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc)
        : "memory");
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
__device__ __forceinline__ float max3f(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
template <int DIN>
struct RU {
    static constexpr int ROWB = DIN >= 64 ? 128 : 64;      // bytes of a row inside a TMA box = its swizzle span
    static constexpr int BOXES = DIN == 128 ? 2 : 1;       // boxes (of 64 inputs) per tile
    static constexpr int BOX = kTileN * ROWB;              // bytes of a box
    static constexpr int TILE = BOXES * BOX;               // bytes of a weight tile
    static constexpr int STAGES = DIN == 128 ? 5 : 8;
    static constexpr int BIAS = kTileN * 32;               // bytes of a tile's bias step (16 bf16 per entry)
    static constexpr int OFF_W = 0, OFF_BIAS = STAGES * TILE, OFF_ONES = OFF_BIAS + STAGES * BIAS,
                         OFF_BEST = OFF_ONES + 128 * 32,   // [kRows] (score, entry), read by the cluster's first CTA
                         OFF_BAR = OFF_BEST + kRows * 8, OFF_ABORT = OFF_BAR + B_COUNT * 8, SMEM = OFF_ABORT + 16;
    static_assert(STAGES <= kMaxStages && SMEM <= 226 * 1024, "shared memory");
    static constexpr uint32_t COL_A = kAcc * kTileN;       // TMEM columns of the inputs, DIN / 2 per block
    static_assert(COL_A + 2 * (DIN / 2) <= 512, "TMEM columns");
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
    extern __shared__ __align__(1024) unsigned char usm[];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sb = s_u32(usm);
    auto bar = [&](int i) { return sb + L::OFF_BAR + 8u * (uint32_t)i; };
    volatile int* abort_flag = reinterpret_cast<volatile int*>(usm + L::OFF_ABORT);
    const int grp = blockIdx.y, split = (int)(blockIdx.x % (uint32_t)n_split);
    const int64_t row0 = (int64_t)(blockIdx.x / (uint32_t)n_split) * kRows;
    const int n_blocks = n - row0 > 128 ? 2 : 1;
    const float* bg = bias ? bias + (int64_t)grp * m : nullptr;
    // this CTA's tiles of the group's entries
    const int all_tiles = (m + kTileN - 1) / kTileN;
    const int tile0 = (int)((int64_t)all_tiles * split / n_split), n_tiles = (int)((int64_t)all_tiles * (split + 1) / n_split) - tile0;
    // a tile needs the bias step if there is a bias, or entries past the last one to rule out
    auto biased = [&](int t) { return bg != nullptr || (tile0 + t + 1) * kTileN > m; };

    if (tid == 0) {
        for (int s = 0; s < L::STAGES; ++s) {
            bar_init(bar(B_FULL + s), 2);  // the loading thread (with the box's bytes) and the bias warp
            bar_init(bar(B_EMPTY + s), (uint32_t)n_blocks);
        }
        for (int e = 0; e < kAccBars; ++e) {
            bar_init(bar(B_AFULL + e), 1);
            bar_init(bar(B_AEMPTY + e), 128);
        }
        bar_init(bar(B_DRAIN), kIssuers);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kIssueWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_u32(&tmem_slot)), "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp == kBiasWarp) {
        // A operand of the bias step: three ones and three times kTinyBias per position; and the second chunk of every
        // bias slot stays zero
        for (int r = lane; r < 128; r += 32) {
            *reinterpret_cast<uint4*>(usm + L::OFF_ONES + step_off(r, 0)) = make_uint4(0x3f803f80u, 0x0d803f80u, 0x0d800d80u, 0);
            *reinterpret_cast<uint4*>(usm + L::OFF_ONES + step_off(r, 1)) = make_uint4(0, 0, 0, 0);
        }
        for (int r = lane; r < kTileN * L::STAGES; r += 32)  // (slots are whole groups of eight rows, one behind the other)
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

    // four read-out warps and one issuing thread per block of positions
    const int e = warp >> 2;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const int row = 128 * e + (warp & 3) * 32 + lane;  // this read-out thread's position
    if (warp < 4 * n_blocks) {
        // the positions' inputs, once: two bf16 per column (zero rows past the end)
        const uint4* xr = reinterpret_cast<const uint4*>(x + (row0 + row) * DIN);
        const bool in = row0 + row < n;
#pragma unroll
        for (int h = 0; h < DIN / 32; ++h) {
            uint32_t v[16];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint4 w = in ? __ldg(xr + 4 * h + q) : make_uint4(0, 0, 0, 0);
                v[4 * q] = w.x; v[4 * q + 1] = w.y; v[4 * q + 2] = w.z; v[4 * q + 3] = w.w;
            }
            st16(tmem + lane_base + L::COL_A + e * (DIN / 2) + 16 * h, v);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    tc_before();
    __syncthreads();
    tc_after();

    if (warp < kEpiWarps) {
        // ------------------------------------------------------------ running arg-max, thread = position
        for (int t = 0; e < n_blocks && t < n_tiles; ++t) {
            const int k = n_blocks * t + e, b = k % kAccBars;
            ok = bar_wait(bar(B_AFULL + b), (k / kAccBars) & 1, abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_after();
            const uint32_t tacc = tmem + lane_base + (uint32_t)(kTileN * (k % kAcc));
            const int j0 = (tile0 + t) * kTileN;
            // the whole accumulator into registers, so that it is free again before it is looked at
            uint32_t v[kTileN / 32][32];
#pragma unroll
            for (int c = 0; c < kTileN / 32; ++c) ld32(tacc + 32 * c, v[c]);
#pragma unroll
            for (int c = 0; c < kTileN / 32; ++c) wait_ld32(v[c]);
            tc_before();
            bar_arrive(bar(B_AEMPTY + b));
            // Only the maximum of 32 columns is compared with the running best (a new best gets rare quickly); they are
            // searched for their first maximal column only then.  Entries come in increasing order and the comparison
            // is strict, so the lowest entry wins among equals; past the last entry the bias is -inf.
#pragma unroll
            for (int c = 0; c < kTileN / 32; ++c) {
                float m0 = __uint_as_float(v[c][0]), m1 = __uint_as_float(v[c][1]);
#pragma unroll
                for (int q = 2; q < 30; q += 4) {
                    m0 = max3f(m0, __uint_as_float(v[c][q]), __uint_as_float(v[c][q + 1]));
                    m1 = max3f(m1, __uint_as_float(v[c][q + 2]), __uint_as_float(v[c][q + 3]));
                }
                const float mx = max3f(fmaxf(m0, m1), __uint_as_float(v[c][30]), __uint_as_float(v[c][31]));
                if (mx > best) {
                    best = mx;
                    int first = 31;
#pragma unroll
                    for (int q = 30; q >= 0; --q) first = __uint_as_float(v[c][q]) == mx ? q : first;
                    arg = j0 + 32 * c + first;
                }
            }
        }
        if (!ok) *abort_flag = 1;
    } else if (warp < kIssueWarp + kIssuers) {
        // ------------------------------------------------------------ MMA issue, one thread per block
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_bf16(128, kTileN);
            const uint64_t ones = mat_desc(sb + L::OFF_ONES, 128, 256);
            const int blk = warp - kIssueWarp;
            for (int t = 0; blk < n_blocks && t < n_tiles; ++t) {
                const int k = n_blocks * t + blk, s = t % L::STAGES, kp = k - kAcc;  // kp: the accumulator's use before
                ok = bar_wait(bar(B_FULL + s), (t / L::STAGES) & 1, abort_flag) &&
                     (kp < 0 || bar_wait(bar(B_AEMPTY + kp % kAccBars), (kp / kAccBars) & 1, abort_flag));
                if (!ok) break;
                tc_after();
                const uint64_t w = swz_desc<DIN>(sb + L::OFF_W + s * L::TILE);
                const uint32_t d = tmem + (uint32_t)(kTileN * (k % kAcc)), at = tmem + L::COL_A + blk * (DIN / 2);
#pragma unroll
                for (int ks = 0; ks < DIN / 16; ++ks)
                    mma_ts(d, at + 8 * ks, w + (uint64_t)(((ks & 3) * 32 + (ks >> 2) * L::BOX) >> 4), idesc, ks > 0);
                if (biased(t)) mma_ss(d, ones, mat_desc(sb + L::OFF_BIAS + s * L::BIAS, 128, 256), idesc, 1u);
                tc_commit_to(bar(B_AFULL + k % kAccBars));
                tc_commit_to(bar(B_EMPTY + s));
            }
            if (!ok) *abort_flag = 1;
            // nothing of this CTA may still run on the tensor core at teardown
            tc_commit_to(bar(B_DRAIN));
            volatile int never = 0;
            if (!bar_wait(bar(B_DRAIN), 0, &never)) *abort_flag = 1;
        }
        __syncwarp();
    } else if (warp == kLoadWarp) {
        // ------------------------------------------------------------ weight tiles
        if (lane == 0) {
            int s = 0, issued = 0;
            uint32_t pe = 1;
            for (int t = 0; t < n_tiles; ++t) {
                ok = bar_wait(bar(B_EMPTY + s), pe, abort_flag);
                if (!ok) break;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar(B_FULL + s)), "r"(L::TILE)
                             : "memory");
#pragma unroll
                for (int h = 0; h < L::BOXES; ++h)
                    asm volatile(
                        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
                        "[%4];" ::"r"(sb + L::OFF_W + s * L::TILE + h * L::BOX),
                        "l"(&tmW), "r"(64 * h), "r"(grp * m + (tile0 + t) * kTileN), "r"(bar(B_FULL + s))
                        : "memory");
                ++issued;
                if (++s == L::STAGES) {
                    s = 0;
                    pe ^= 1;
                }
            }
            if (!ok) {
                *abort_flag = 1;
                // the copies in flight land before the CTA ends: every stage's last fill has its bytes (a stage whose
                // bias arrival is missing times out here, with its bytes long there)
                volatile int never = 0;
                for (int k = issued > L::STAGES ? issued - L::STAGES : 0; k < issued; ++k)
                    bar_wait(bar(B_FULL + k % L::STAGES), (k / L::STAGES) & 1, &never);
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ bias steps: b = hi + mid + lo, bf16 each, exactly
        // two tiles at a time: the wait, the fence and the hand-over are a chain, and one per tile would set the pace
        constexpr int kPer = kTileN / 32;
        auto load_bias = [&](int t, float (&b)[2 * kPer]) {
#pragma unroll
            for (int i = 0; i < 2 * kPer; ++i) {
                const int j = (tile0 + t) * kTileN + 32 * i + lane;
                b[i] = j < m ? (bg ? __ldg(bg + j) : 0.f) : -CUDART_INF_F;
            }
        };
        float nxt[2 * kPer];
        load_bias(0, nxt);
        for (int t = 0; t < n_tiles; t += 2) {
            float cur[2 * kPer];
#pragma unroll
            for (int i = 0; i < 2 * kPer; ++i) cur[i] = nxt[i];
            load_bias(t + 2, nxt);
            const int n_t = min(2, n_tiles - t);
            for (int h = 0; h < n_t; ++h)
                ok = ok && bar_wait(bar(B_EMPTY + (t + h) % L::STAGES), (((t + h) / L::STAGES) & 1) ^ 1, abort_flag);
            ok = __all_sync(0xffffffffu, ok);
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
        }
        if (!ok) *abort_flag = 1;
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
    if (tid == 0 && *abort_flag) *reinterpret_cast<volatile int*>(flags) = ERR_ROUTE;
    if (slot >= 0) report_done(Report{flags, flags + 1, &route_count[slot]}, gridDim.x * gridDim.y);
}

// The weights as rows of `d_in` inputs, boxes of 128 rows and at most 64 inputs.
bool make_weight_map(int d_in, int64_t rows, const void* W, CUtensorMap* map)
{
    return encode_rows(map, W, d_in, rows, d_in < 64 ? d_in : 64, kTileN, d_in < 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
}

template <int DIN>
cudaError_t launch_t(const void* x, const void* W, const float* bias, int n, int m, int G, int32_t* out, int* flags,
                     int slot, cudaStream_t s)
{
    CUtensorMap map;
    if (!make_weight_map(DIN, (int64_t)G * m, W, &map)) return cudaErrorInvalidValue;
    // CTAs per position block: as many as shorten the run most, counting whole waves of CTAs over the SMs and about
    // four tiles' time for setting one up
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t ctas = (int64_t)((n + kRows - 1) / kRows) * G, tiles = (m + kTileN - 1) / kTileN;
    int split = 1;
    int64_t best = INT64_MAX;
    for (int sp = 1; sp <= kMaxClusterRU && sp <= tiles; sp *= 2) {
        const int64_t cost = (ctas * sp + sms - 1) / sms * ((tiles + sp - 1) / sp + 4);
        if (cost < best) {
            best = cost;
            split = sp;
        }
    }
    const dim3 grid((unsigned)((n + kRows - 1) / kRows * split), (unsigned)G);
    if (ctas * split > sms) slot = -1;  // several rounds: the report at the end of each CTA would delay the next
    return launch_kernel(Launch{s, nullptr, nullptr}, route_umma_kernel<DIN>, grid, kThreadsRU, RU<DIN>::SMEM, split,
                         (const uint16_t*)x, map, bias, n, m, G, out, flags, slot, split);
}

}  // namespace

cudaError_t launch_route_umma(int d_in, const void* x, const void* W, const float* bias, int n, int n_entries, int G,
                              int32_t* out, int* flags, int slot, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    switch (d_in) {
        case 32: return launch_t<32>(x, W, bias, n, n_entries, G, out, flags, slot, s);
        case 64: return launch_t<64>(x, W, bias, n, n_entries, G, out, flags, slot, s);
        default: return launch_t<128>(x, W, bias, n, n_entries, G, out, flags, slot, s);
    }
}

}  // namespace ckv
