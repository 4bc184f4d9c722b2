// tcgen05 gather-concat-attention kernel (bf16, head_dim 32) for many queries per user.
//
// Persistent: one CTA per SM holds three workers, and every worker walks its own static round-robin share of the work
// units, where a unit is (work item = history chunk of one user, group, block of up to 128 queries).  The history chunk
// is processed in tiles of 64 positions.  A worker is (warp-specialised, 6 warps of the CTA's 18)
//   four normalisation warps: thread i owns TMEM lane i, query row i of the block (turned by whole warps, see block_turn)
//   one issuing warp: the score MMAs and the weighted-sum MMAs
//   one producer warp: gathers pool rows into the worker's ring of shared-memory stages with 16-byte cp.async, patches
//     the user-specific leading elements (Eq. K), publishes the tile one tile later, and stages Q with a unit's first
//     tile.  (A side that is not shared -- sharing only keys or only values -- is copied from the user's full-width
//     rows instead.)
// Workers share nothing but the SM: no merge between them, no hand-over, every barrier has one waiting role that meets
// its phases in order.
//
// A worker has two score buffers in TMEM; the weights of a tile are written over the head of the scores they were
// computed from (32 columns of bf16 pairs over 64 columns of fp32):
//   S_i  = Q K_tile^T                 UMMA 128 x 64 x 32, A = Q smem, B = K tile smem (K-major)
//   P_i  = exp2(S_i c - m) | silu     tcgen05.ld -> math -> bf16 -> tcgen05.st, in place
//   O   += P_i V_tile                 UMMA 128 x 32 x 64, A = P from TMEM, B = V tile (MN-major)
// The issuing thread issues the weighted sum of step t, then the scores of step t + 2 (into the buffer the weighted sum
// has just read): the tensor core runs one thread's instructions in order, so the buffer needs no completion hand-off in
// between, and the scores of step t + 1 are there while step t is normalised.
//
// What bounds it: the special-function unit (one ex2 or tanh per score, 16 per clock per SM).  The normalisation of a
// tile is a chain of dependent work for its warp (wait for the scores, TMEM load, arithmetic, TMEM store, publish; at a
// unit's end the last weighted sum, the accumulator read-out, the store), and three workers fill each other's gaps: of the
// 1900 clocks of a tile (SiLU; 2150 softmax) a warp spends 1530 in the arithmetic, whose share of the unit is 512, 105 on
// the wait for the scores, 120 on the TMEM loads.  Registers (65536 / 20 warps = 96 a thread, enough for one
// 32-column chunk of scores at a time) and TMEM (3 x (2 x 64 + 32) = 480 columns) admit no fourth.  An SM of busy
// workers takes 0.36 us per 64 positions and 1.2 us per unit, the special-function unit busy 79 % of the time.
// With the three groups on one unit instead (its tiles dealt out in turn, accumulators merged through shared memory at its
// end) a unit cost 5 us plus 0.45 us per 128 positions; three workers took 1024 users x 1024 positions x 100 queries x 8 groups
// from 490 to 386 us, 2048 users x 4096 x 128 (SiLU) from 2.88 to 2.57 ms, 64 causal self-attentions of 200..1500 positions from
// 283 to 148 us.  The issuing warp walks its loop as a whole and an elected thread issues, with operands known to be
// uniform: under "lane 0" each product and commit waited for its operands' way into uniform registers (357 us, 2.47 ms, 127
// us).  With the swizzled tiles and the arithmetic left out that no row needs, both below, 354 us, 2.43 ms, 107 us.
// (Measured and not kept: scores in pieces of sixteen columns with the next tile's requested ahead, and a unit's read-out put
// off behind the next unit's first tile, 548 us and 3.27 ms: with the registers that takes the arithmetic no longer
// overlaps itself.)
//
// Softmax bookkeeping.  The reference m of a row lies ten octaves above the largest of the first 32 scores of the unit's
// first tile and stays fixed.  The row sum l is added up by the row's thread in fp32, chunk by chunk, and a chunk's share of
// it also tells when a score has come near the reference (32 weights above one, in sum); only then is the reference moved, O
// and the row sum rescaled (TMEM read-modify-write) and the chunk worked out again.  So no weight is more than one, as with
// the running maximum, and sums with values near fp32's largest stay in range.
//
// Shared-memory tiles hold rows of 64 bytes one behind the other, 16-byte chunk c of row r at chunk c ^ (r / 2 mod 4): the
// 64-byte swizzle of the UMMA layouts, K-major for Q and K, MN-major for V.  A copied row then lies in one 64-byte
// piece.  With the layout without swizzle (chunk c of row r at 128 c + 16 (r mod 8)) its four chunks fell on the same
// banks, where a row's chunks, which leave the L1 together, were written one after the other (2048 users x 4096 positions x 128
// queries, SiLU: 2.47 -> 2.41 ms; 512 x 512 x 64 104 -> 98 us).
//
// Every wait in this kernel is bounded: on time-out the CTA records an error code, raises a
// CTA-wide abort flag that ends every other wait, drains its own copies, frees its TMEM and
// returns.
#include <cuda_bf16.h>
#include <math_constants.h>

#include <type_traits>

#include "ckv_internal.h"
#include "ptx_helpers.cuh"

namespace ckv {
namespace {

constexpr int D = 32;
constexpr int TH = 64;                   // positions per tile = one step: one score MMA, normalisation, weighted sum
constexpr int NW = 3;                    // workers
constexpr int NS = 7;                    // K/V stages of a worker (at most)
constexpr int kGroupThreads = 128;       // normalisation threads of a worker
constexpr int kIssueWarp0 = 4 * NW;      // warps 12..14 issue the MMAs of worker 0..2; warp 12 owns the TMEM allocation
constexpr int kProducerWarp0 = kIssueWarp0 + NW;
constexpr int kThreads = (kProducerWarp0 + NW) * 32;  // 576
constexpr int kTileQ = 128 * D * 2;      // 8 KB
constexpr int kTileK = TH * D * 2;       // 4 KB
constexpr int kTileV = TH * D * 2;       // 4 KB
constexpr int kGroupB = 8 * D * 2;       // bytes of a group of eight rows of any tile
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColWorker = 2 * TH + D;  // worker b: S_i (and P_i over its head) at kColWorker b + 64 i, O behind them
static_assert(kColWorker * NW <= kTmemCols, "TMEM columns");
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kOctavesAbove = 10.f;    // of a row's reference above the maximum it is set by
constexpr float kSumLimit = 1.f;         // a chunk's sum beyond it gives away a score near the reference
constexpr uint32_t kSpinLimit = 1u << 18;  // polls of a wait before the CTA gives up
constexpr uint32_t kSuspendNs = 4000;      // how long one poll may stay suspended in hardware (longer hints wake later)

// barrier slots (8 bytes each) of a worker
enum { BAR_FULL = 0, BAR_EMPTY = NS, BAR_QEMPTY = 2 * NS, BAR_SFULL = BAR_QEMPTY + 2, BAR_PREADY = BAR_SFULL + 2,
       BAR_DRAIN = BAR_PREADY + 2, BAR_COUNT };

// dynamic shared memory map, DUB = bytes of a user part: per worker two Q blocks, the K stages, the V stages, and a ring
// of what the producer has requested from the compressed cache, tile by tile
template <int DUB>
struct Map {
    static constexpr int STAGES = DUB >= 8 ? NS - 1 : NS;
    static constexpr int META = 256 + 2 * TH * DUB, META_SLOTS = 4;  // K indices, V indices, K user parts, V user parts
    static constexpr int Q = 0, K = 2 * kTileQ, V = K + STAGES * kTileK, M = V + STAGES * kTileV, WORKER = M + META_SLOTS * META;
    static constexpr int BAR = NW * WORKER, ABORT = BAR + NW * BAR_COUNT * 8, BYTES = ABORT + 32;
    static_assert(BYTES <= 231424, "shared memory of one CTA");
};

// error codes OR-ed into the context's device error word: which role gave up (bits 0..3); bits 8..11 carry the
// site code of the first wait that ran out (see SITE_*)
enum { ERR_NORMALISE = 1, ERR_MMA = 2, ERR_DRAIN = 4, ERR_PRODUCER = 8 };

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait on a phase parity.  Returns false on time-out or when the CTA is aborting.
// A wait that runs out (rather than being ended by the abort flag) leaves its site code in the word behind the flag;
// the first one stays, and the kernel reports it in bits 8.. of the error word.
enum { SITE_SFULL = 1, SITE_OFULL, SITE_PREV, SITE_TILE, SITE_PREADY, SITE_STAGE, SITE_QBUF, SITE_DRAIN };
__device__ __forceinline__ void note_site(const volatile int* abort_flag, int site)
{
    atomicCAS(const_cast<int*>(abort_flag) + 1, 0, site);
}
__device__ __noinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const volatile int* abort_flag, int site)
{
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
            "selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "r"(kSuspendNs)
            : "memory");
        if (ok) return true;
        if ((i & 31u) == 31u && *abort_flag) return false;
    }
    note_site(abort_flag, site);
    return false;
}
// One poll, without waiting.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// The bounded wait with its first poll inline: most waits of the issuing threads find their phase complete.
__device__ __forceinline__ bool mbar_wait_fast(uint32_t bar, uint32_t parity, const volatile int* abort_flag, int site)
{
    return mbar_test(bar, parity) || mbar_wait(bar, parity, abort_flag, site);
}
// 16-byte copy global -> shared; src_bytes = 0 fills the destination with zeros instead.
// Pool rows go through L1 (with skewed indices the hot rows then stop hammering a few L2 lines
// from every SM at once); rows that are read once bypass it.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async16_once(uint32_t dst, const void* src, uint32_t src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem]
__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc)
        : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(acc)
        : "memory");
}

// Shared-memory matrix descriptor of a tile of 64-byte rows, 64-byte swizzle: start address, 512 bytes from one group of
// eight rows to the next (in 16-byte units; the other offset has no meaning here), descriptor version 1 of sm_100.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr)
{
    return (uint64_t)((addr & 0x3ffffu) >> 4) | (1ull << 16) | ((uint64_t)(kGroupB >> 4) << 32) | (1ull << 46) | (4ull << 61);
}
// Instruction descriptor for kind::f16: fp32 accumulate, bf16 A and B.
__host__ __device__ constexpr uint32_t make_idesc(int M, int N, bool b_mn_major)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

// 32 consecutive columns of this thread's TMEM lane.  The load is asynchronous: its registers
// hold the data only after tmem_wait_ld32 on the same array.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
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
// Waits for every tcgen05.ld of this thread.  Naming the registers as in/out operands keeps the
// compiler from scheduling their consumers ahead of the wait.
__device__ __forceinline__ void tmem_wait_ld32(uint32_t (&r)[32])
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
__device__ __forceinline__ uint32_t tmem_ld1(uint32_t taddr)
{
    uint32_t r;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r) : : "memory");
    return r;
}
__device__ __forceinline__ void tmem_st1(uint32_t taddr, uint32_t r)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "r"(r) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,"
        "%30,%31,%32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
        "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
        "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

__device__ __forceinline__ float max3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Two fp32 operations in one instruction (packed pairs): the normalisation is short of issue slots, not of FMA lanes.
// (d0, d1) = (a0, a1) * b + c
__device__ __forceinline__ void fma2_scalar(float& d0, float& d1, float a0, float a1, float b, float c)
{
    asm("{\n.reg .b64 ra, rb, rc, rd;\nmov.b64 ra, {%2, %3};\nmov.b64 rb, {%4, %4};\nmov.b64 rc, {%5, %5};\n"
        "fma.rn.f32x2 rd, ra, rb, rc;\nmov.b64 {%0, %1}, rd;\n}\n"
        : "=f"(d0), "=f"(d1)
        : "f"(a0), "f"(a1), "f"(b), "f"(c));
}
// (d0, d1) = (a0, a1) * (b0, b1) + (c0, c1)
__device__ __forceinline__ void fma2(float& d0, float& d1, float a0, float a1, float b0, float b1, float c0, float c1)
{
    asm("{\n.reg .b64 ra, rb, rc, rd;\nmov.b64 ra, {%2, %3};\nmov.b64 rb, {%4, %5};\nmov.b64 rc, {%6, %7};\n"
        "fma.rn.f32x2 rd, ra, rb, rc;\nmov.b64 {%0, %1}, rd;\n}\n"
        : "=f"(d0), "=f"(d1)
        : "f"(a0), "f"(a1), "f"(b0), "f"(b1), "f"(c0), "f"(c1));
}
// (d0, d1) += (a0, a1)
__device__ __forceinline__ void add2(float& d0, float& d1, float a0, float a1)
{
    asm("{\n.reg .b64 ra, rd;\nmov.b64 rd, {%0, %1};\nmov.b64 ra, {%2, %3};\nadd.rn.f32x2 rd, rd, ra;\n"
        "mov.b64 {%0, %1}, rd;\n}\n"
        : "+f"(d0), "+f"(d1)
        : "f"(a0), "f"(a1));
}
// (d0, d1) = (a0, a1) * b
__device__ __forceinline__ void mul2_scalar(float& d0, float& d1, float a0, float a1, float b)
{
    asm("{\n.reg .b64 ra, rb, rd;\nmov.b64 ra, {%2, %3};\nmov.b64 rb, {%4, %4};\nmul.rn.f32x2 rd, ra, rb;\n"
        "mov.b64 {%0, %1}, rd;\n}\n"
        : "=f"(d0), "=f"(d1)
        : "f"(a0), "f"(a1), "f"(b));
}

// byte offset of (row r, 16-byte chunk c) inside a Q, K or V tile
__device__ __forceinline__ uint32_t tile_off(int r, int c) { return (uint32_t)(r * (D * 2) + ((c ^ ((r >> 1) & 3)) << 4)); }

// Inside a tile the producer places position 32 c + 4 q + i (q < 8, i < 4) in row
// 32 c + 8 i + q: a lane's four 16-byte copies of a 32-position block then fall into different shared-memory banks.
// Attention does not depend on the order of positions; only the tail mask has to know which
// position a score column belongs to.
__device__ __forceinline__ int pos_of_col(int c, int e) { return 32 * c + 4 * (e & 7) + (e >> 3); }

// ---- normalisation of one 128 x 64 score tile by the worker's four warps (thread = query row = TMEM lane) ----

// Multiplies this thread's row of O (32 columns) by f.
__device__ __noinline__ void rescale_row(uint32_t tO, float f)
{
    uint32_t o[32];
    tmem_ld32(tO, o);
    tmem_wait_ld32(o);
#pragma unroll
    for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * f);
    tmem_st32(tO, o);
}

// Multiplies the 32 weights (16 columns of bf16 pairs) this thread wrote for the first chunk of the current tile by f, a power of two: exact unless a weight drops below the smallest bf16.
__device__ __noinline__ void rescale_weights(uint32_t tP, float f)
{
    for (int c = 0; c < 16; ++c) {
        const uint32_t w = tmem_ld1(tP + c);
        tmem_st1(tP + c, pack_bf16(__uint_as_float(w << 16) * f, __uint_as_float(w & 0xffff0000u) * f));
    }
}

// The weights of one 32-column chunk once more (returns their sum), from scores the caller has put into local memory (only used on
// the rare path that moves a row's reference; kept out of line so that it costs the common path nothing).
template <bool TAIL>
__device__ __noinline__ float rewrite_weights(uint32_t tP, const uint32_t* cur, float sc, float nm, int valid, int c)
{
    uint32_t p[16];
    float sum = 0.f;
#pragma unroll
    for (int e = 0; e < 32; e += 2) {
        float x0 = fmaf(__uint_as_float(cur[e]), sc, nm), x1 = fmaf(__uint_as_float(cur[e + 1]), sc, nm);
        if (TAIL) {
            if (pos_of_col(c, e) >= valid) x0 = -CUDART_INF_F;
            if (pos_of_col(c, e + 1) >= valid) x1 = -CUDART_INF_F;
        }
        const float e0 = ex2(x0), e1 = ex2(x1);
        sum += e0 + e1;
        p[e >> 1] = pack_bf16(e0, e1);
    }
    tmem_st16(tP, p);
    return sum;
}

__device__ __noinline__ void zero_weights(uint32_t tP)
{
    const uint32_t p[16] = {};
    tmem_st16(tP, p);
}

// Largest exponent argument of one 32-column chunk (rare path only, like rewrite_weights).
template <bool TAIL>
__device__ __noinline__ float chunk_max(const uint32_t* cur, float sc, float nm, int valid, int c)
{
    float mx = -CUDART_INF_F;
#pragma unroll
    for (int e = 0; e < 32; ++e) {
        const float x = fmaf(__uint_as_float(cur[e]), sc, nm);
        if (!TAIL || pos_of_col(c, e) < valid) mx = fmaxf(mx, x);
    }
    return mx;
}

// Softmax weights of one 32-column chunk (c = 0, 1) of a 128 x 64 score tile: p = exp2(s c - m) as bf16
// pairs written over the head of the scores (columns 0..31 of the buffer; chunk 1 of the scores, columns 32..63,
// is still to be read when chunk 0's weights land on columns 0..15, and chunk 1's weights
// land on columns 16..31, whose scores have been consumed).  The chunk's weights are added to the row sum l.  With `first`
// (the unit's first tile) chunk 0 sets the row's reference m from its 32 scores (column 0 is the tile's position 0, always a
// real one).  A chunk whose sum gives away a score near the reference moves it up by some
// octaves and is written again from its scores, read once more; what O holds so far
// (`have_o`; wait_prev() waits for the previous step's MMAs) and, for chunk 1, the weights of chunk 0 are
// multiplied by the same factor.  Returns false if that wait ran out.
// `valid` counts the real positions of the tile (1..64); column e of chunk c holds position
// pos_of_col(c, e) of the tile.  TAIL = true (the last tile of a history, at most once per unit) masks the
// columns beyond.
// VIS (visible lengths): `valid` differs from thread to thread and may be zero or negative (the row sees nothing
// of this tile); a row's reference is then set by the first chunk in which it sees a position.
template <bool TAIL, bool VIS, typename WaitPrev>
__device__ __forceinline__ bool softmax_chunk(const uint32_t (&cur)[32], int c, uint32_t tS, uint32_t tO, float sc,
                                              int valid, bool first, bool have_o, float& m_ref, float& l, WaitPrev&& wait_prev)
{
    if ((c == 0 && first) || (VIS && m_ref == -CUDART_INF_F)) {
        float t0 = -CUDART_INF_F, t1 = -CUDART_INF_F;
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
            float x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                x[i] = (TAIL && pos_of_col(c, e + i) >= valid) ? -CUDART_INF_F : __uint_as_float(cur[e + i]);
            t0 = max3(t0, x[0], x[1]);
            t1 = max3(t1, x[2], x[3]);
        }
        m_ref = fmaf(fmaxf(t0, t1), sc, kOctavesAbove);
    }
    float nm = -m_ref;
    float ls0 = 0.f, ls1 = 0.f;  // this chunk's share of the row sum
    uint32_t p[16];
#pragma unroll
    for (int e = 0; e < 32; e += 2) {
        float x0, x1;
        fma2_scalar(x0, x1, __uint_as_float(cur[e]), __uint_as_float(cur[e + 1]), sc, nm);
        if (TAIL) {
            if (pos_of_col(c, e) >= valid) x0 = -CUDART_INF_F;
            if (pos_of_col(c, e + 1) >= valid) x1 = -CUDART_INF_F;
        }
        const float e0 = ex2(x0), e1 = ex2(x1);
        add2(ls0, ls1, e0, e1);
        p[e >> 1] = pack_bf16(e0, e1);
    }
    // A sum beyond one (or one that is not a number) means some weight of this row is beyond 2^-5, while a sum of 32 weights
    // ten octaves down is 2^-5 at most.  That costs one comparison here instead of a running maximum over the arguments.
    if (!__any_sync(0xffffffffu, !(ls0 + ls1 <= kSumLimit))) {
        tmem_st16(tS + 16 * c, p);
    } else {
        // rare: some row of this warp came near its reference and its weights may have overflowed.  Nothing of this
        // chunk has been written yet, so its scores are still in TMEM: move the reference, bring what was
        // accumulated and written before into the new scale, and work the chunk out again from there.
        uint32_t again[32];
        tmem_ld32(tS + 32 * c, again);
        tmem_wait_ld32(again);
        const float mx = chunk_max<TAIL>(again, sc, nm, valid, c);
        const float moved = mx > -5.f ? m_ref + (ceilf(mx) + kOctavesAbove) : m_ref;
        // (by what the reference moved, rounding included; a row that sees nothing has no finite one)
        const float f = moved != m_ref ? ex2(m_ref - moved) : 1.f;
        m_ref = moved;
        nm = -m_ref;
        tc_wait_st();
        l *= f;
        if (have_o) {
            if (!wait_prev()) return false;
            tc_fence_after();
            rescale_row(tO, f);
        }
        if (c == 1) rescale_weights(tS, f);
        ls0 = rewrite_weights<TAIL>(tS + 16 * c, again, sc, nm, valid, c);
        ls1 = 0.f;
        tc_wait_st();
    }
    l += ls0 + ls1;
    return true;
}

// p = silu(x) = x sigmoid(x) = h (1 + tanh(h)), h = x / 2, as bf16 pairs over the head of the scores like the
// softmax weights   (sc = scale / 2)
template <bool TAIL>
__device__ __forceinline__ void silu_chunk(const uint32_t (&cur)[32], int c, uint32_t tS, float sc, int valid)
{
    uint32_t p[16];
#pragma unroll
    for (int e = 0; e < 32; e += 2) {
        float h0, h1, w0, w1;
        mul2_scalar(h0, h1, __uint_as_float(cur[e]), __uint_as_float(cur[e + 1]), sc);
        fma2(w0, w1, h0, h1, tanh_fast(h0), tanh_fast(h1), h0, h1);
        if (TAIL) {
            if (pos_of_col(c, e) >= valid) w0 = 0.f;
            if (pos_of_col(c, e + 1) >= valid) w1 = 0.f;
        }
        p[e >> 1] = pack_bf16(w0, w1);
    }
    tmem_st16(tS + 16 * c, p);
}

// Blocks of fewer than 97 query rows leave warps of their worker without a row.  Those skip the arithmetic, and tile row r of
// the block is query row (r - 32 turn) mod 128, so that the rows of an SM's workers, and of a worker's units one after the
// other, fall to different quarters of the SM, whose special-function units are what is short.  512 users x 512 positions x 8
// groups: 64 queries 98.6 -> 91.3 us (SiLU 92 -> 80.5), 96 queries 101.2 -> 96.0; 300 x 1000 x 150 210 -> 191.
__device__ __forceinline__ int block_turn(int worker, int unit, int rows)
{
    const int warps = (rows + 31) >> 5;
    return warps > 3 ? 0 : ((warps == 2 ? 2 * worker : worker) + unit) & 3;
}

// The user-specific leading elements of one row (DUB = 2 d_user bytes), on their way from the request ring to a tile.
template <int DUB> struct UserPart;
template <> struct UserPart<0> {};
template <> struct UserPart<2> {
    uint16_t v;
    __device__ __forceinline__ void take(const unsigned char* p) { v = *reinterpret_cast<const uint16_t*>(p); }
    __device__ __forceinline__ void store(unsigned char* p) const { *reinterpret_cast<uint16_t*>(p) = v; }
};
template <> struct UserPart<4> {
    uint32_t v;
    __device__ __forceinline__ void take(const unsigned char* p) { v = *reinterpret_cast<const uint32_t*>(p); }
    __device__ __forceinline__ void store(unsigned char* p) const { *reinterpret_cast<uint32_t*>(p) = v; }
};
template <> struct UserPart<8> {
    uint2 v;
    __device__ __forceinline__ void take(const unsigned char* p) { v = *reinterpret_cast<const uint2*>(p); }
    __device__ __forceinline__ void store(unsigned char* p) const { *reinterpret_cast<uint2*>(p) = v; }
};
template <> struct UserPart<16> {
    uint4 v;
    __device__ __forceinline__ void take(const unsigned char* p) { v = *reinterpret_cast<const uint4*>(p); }
    __device__ __forceinline__ void store(unsigned char* p) const { *reinterpret_cast<uint4*>(p) = v; }
};

// One work unit of a worker's share, decoded from its Work record.
struct Unit {
    Work wk;
    int grp;
    int row0;        // first query row of the block
    int n_tiles;     // > 0: tiles to process; 0: empty history (zero output rows)
    int last_valid;  // real positions in the last tile
};

__device__ __forceinline__ Work load_work(const Work* p)
{
    static_assert(sizeof(Work) == 48, "Work is read as three 16-byte words");
    union {
        Work w;
        uint4 q[3];
    } u;
    const uint4* src = reinterpret_cast<const uint4*>(p);
    u.q[0] = __ldg(src);
    u.q[1] = __ldg(src + 1);
    u.q[2] = __ldg(src + 2);
    return u.w;
}

// A worker's units.  Worker k = x + gridDim.x b (worker b of block x) takes one unit of every run of NW gridDim.x
// consecutive ones, number k of the even runs and number k from the end of the odd ones, so that units in order of falling
// cost come out even.  Every role walks an identical copy, so stage and buffer indices need no communication.  The record
// of the following unit is always in flight while the current one is processed.
// Unit w stands for (work record, group) = (w / G, w % G), a record for every (item, query block) that exists.
// KEEP_EMPTY: also stop at units with an empty history (the role that writes their zero rows).
template <bool KEEP_EMPTY, bool VIS>
struct Units {
    const Work* works;
    const int32_t* vmax;       // VIS: per record the largest visible length of its rows
    uint32_t n_groups, n_work, run, k;  // the host keeps n_work + 2 run below 2^32
    uint32_t base;             // first unit of the run behind the current one
    bool odd;                  // that run is an odd one
    uint32_t w_nxt, grp_nxt;   // the unit taken from it
    int vmax_nxt;
    Unit u;
    Work nxt;                  // its record (valid if w_nxt < n_work)
    bool valid;
    __device__ __forceinline__ void request()
    {
        w_nxt = base + (odd ? run - 1 - k : k);
        base += run;
        odd = !odd;
        if (w_nxt >= n_work) return;  // (a later run lies behind the end altogether)
        const uint32_t i = w_nxt / n_groups;
        grp_nxt = w_nxt - i * n_groups;
        nxt = load_work(works + i);
        if constexpr (VIS) vmax_nxt = __ldg(vmax + i);
    }
    __device__ __forceinline__ void next()
    {
        valid = false;
        while (w_nxt < n_work) {
            u.wk = nxt;
            u.grp = (int)grp_nxt;
            u.row0 = u.wk.row0;
            // with visible lengths nothing behind the block's largest limit is touched (every role decodes the same)
            int len = u.wk.len;
            if constexpr (VIS) len = min(len, max(vmax_nxt - u.wk.begin, 0));
            request();
            u.n_tiles = (len + TH - 1) / TH;
            u.last_valid = len - (u.n_tiles - 1) * TH;
            if (u.n_tiles > 0 || KEEP_EMPTY) {
                valid = true;
                return;
            }
        }
    }
    __device__ __forceinline__ void init(const AttendArgs& a, int64_t n_work_, int worker)
    {
        works = a.works;
        if constexpr (VIS) vmax = a.vmax;
        n_groups = (uint32_t)a.cv.n_groups;
        n_work = (uint32_t)n_work_;
        run = NW * gridDim.x;
        k = blockIdx.x + gridDim.x * (uint32_t)worker;
        base = 0;
        odd = false;
        request();
        next();
    }
};

// VIS: visible lengths (a.vis, a.vmax); the plain instantiations carry none of that code.
template <int MODE, int DUB, bool VIS>
__global__ void __launch_bounds__(kThreads, 1) attend_umma_kernel(const AttendArgs a, int64_t n_work, int* err_flag)
{
    using L = Map<DUB>;
    constexpr int NS = L::STAGES;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint32_t tmem_base_slot;

    // (the warp number as a value known to be uniform: tensor-core and TMEM instructions take theirs from uniform registers)
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t sbase = smem_u32(smem);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::ABORT);
    const int G = a.cv.n_groups;

    if (tid == 0) {
        for (int b = 0; b < NW; ++b) {
            const uint32_t bar0 = sbase + L::BAR + b * (BAR_COUNT * 8);
            for (int i = 0; i < BAR_COUNT; ++i)  // (full: lane 0 of the producer; empty: the commit behind a weighted sum)
                mbar_init(bar0 + 8 * i, i == BAR_PREADY || i == BAR_PREADY + 1 ? kGroupThreads : 1);
        }
        abort_flag[0] = 0;  // raised by the first role that gives up
        abort_flag[1] = 0;  // site of the first wait that ran out
        abort_flag[2] = 0;  // never raised: the flag of the teardown wait, which must not be cut short
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kIssueWarp0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_slot;
    const int b = warp < kIssueWarp0 ? warp >> 2 : warp < kProducerWarp0 ? warp - kIssueWarp0 : warp - kProducerWarp0;  // worker
    const uint32_t bar0 = sbase + L::BAR + b * (BAR_COUNT * 8), wbase = sbase + b * L::WORKER;
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    const uint32_t tS0 = tmem + kColWorker * b, tO0 = tS0 + 2u * TH;  // lane 0 of the score buffers and the accumulator

    if (warp < kIssueWarp0) {
        // --------------------------------------------------------------- normalisation
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tSl = tS0 + lane_base, tO = tO0 + lane_base;
        const float sc = a.scale * (MODE == CKV_SOFTMAX ? kLog2e : 0.5f);
        int cnt = 0;    // tiles normalised
        int stage = 0, sphase = 0;  // stage of the tile last normalised and the parity of its release: cnt - 1 in units of NS
        bool ok = true;
        uint32_t sa[32];  // one 32-column chunk of a tile's scores
        int seq = 0;      // units with tiles begun
        Units<true, VIS> un;
        un.init(a, n_work, b);
        for (; un.valid && ok; un.next()) {
            const Unit& u = un.u;
            const int rows = min(u.wk.M - u.row0, kGroupThreads);
            const int quarter = ((warp & 3) - block_turn(b, seq, rows)) & 3;
            const int r = u.row0 + 32 * quarter + lane;
            if (r < u.wk.M) (void)CKV_CLAMP((int64_t)(u.wk.q0 + r), a.q_rows, err_flag);
            const int64_t out_base = ((int64_t)(u.wk.q0 + r) * G + u.grp) * D;
            if (u.n_tiles == 0) {  // empty history, or a chunk behind every row's visible length: zero rows
                if (r < u.wk.M) {
                    if (u.wk.part_row >= 0) {  // (only with visible lengths) an empty partial result
                        const int64_t pr = CKV_CLAMP((int64_t)(u.wk.part_row + r), a.part_rows, err_flag);
                        *part_ml(a, D, pr, u.grp) = make_float2(-CUDART_INF_F, 0.f);
                        float4* dst = reinterpret_cast<float4*>(part_acc(a, D, pr, u.grp));
                        for (int q4 = 0; q4 < 8; ++q4) dst[q4] = make_float4(0.f, 0.f, 0.f, 0.f);
                    } else if (a.out_dtype == CKV_BF16) {
                        uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<uint16_t*>(a.out) + out_base);
                        for (int q4 = 0; q4 < 4; ++q4) dst[q4] = make_uint4(0, 0, 0, 0);
                    } else {
                        float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(a.out) + out_base);
                        for (int q4 = 0; q4 < 8; ++q4) dst[q4] = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
                continue;
            }
            ++seq;
            if (32 * quarter >= rows) {  // no row of this warp is a query row: it keeps step, and leaves its weights as they are
                for (int j = 0; j < u.n_tiles; ++j) {
                    ok = mbar_wait_fast(bar(BAR_SFULL + (cnt & 1)), (cnt >> 1) & 1, abort_flag, SITE_SFULL);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    mbar_arrive(bar(BAR_PREADY + (cnt & 1)));
                    if (cnt > 0 && ++stage == NS) {
                        stage = 0;
                        sphase ^= 1;
                    }
                    ++cnt;
                }
                continue;
            }
            // positions this thread's query row attends: [0, lim); a thread without a row goes by the block's last one, so
            // that it asks for no masking of its own
            int lim = u.wk.L;
            if constexpr (VIS) lim = min(max(__ldg(a.vis + u.wk.q0 + min(r, u.row0 + rows - 1)), 0), u.wk.L);
            float m_ref = -CUDART_INF_F, l = 0.f;
            for (int j = 0; j < u.n_tiles && ok; ++j) {
                const int valid = j == u.n_tiles - 1 ? u.last_valid : TH;  // real positions of the tile
                const int i = cnt & 1;                                     // buffer of this step
                const uint32_t tS = tSl + (uint32_t)TH * i;
                ok = mbar_wait_fast(bar(BAR_SFULL + i), (cnt >> 1) & 1, abort_flag, SITE_SFULL);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                // (softmax, only taken when a row's reference moves) the previous step's weighted sum must have
                // finished before O is rescaled: it is what releases that step's stage
                auto wait_prev = [&]() {
                    bool w = mbar_wait(bar(BAR_EMPTY + stage), sphase, abort_flag, SITE_PREV);
                    return __all_sync(0xffffffffu, w);
                };
                // real (and, with visible lengths, attended) positions of this thread's row in the tile
                int valid_r = valid;
                bool tail = valid < TH;
                if constexpr (VIS) {
                    valid_r = min(valid, lim - (u.wk.begin + j * TH));
                    tail = __any_sync(0xffffffffu, valid_r < TH);
                }
                // One 32-column chunk at a time: the other workers' warps on this sub-partition cover the TMEM load.
                if (tail) {  // end of a history or of some row's visible positions: masked columns
#pragma unroll 1
                    for (int c = 0; c < 2 && ok; ++c) {
                        // seen by no row of this warp (64 causal self-attentions of 200..1500 positions 125.5 -> 107 us)
                        if (__all_sync(0xffffffffu, valid_r <= 32 * c)) {
                            zero_weights(tS + 16 * c);
                            continue;
                        }
                        tmem_ld32(tS + 32 * c, sa);
                        tmem_wait_ld32(sa);
                        if constexpr (MODE == CKV_SOFTMAX)
                            ok = softmax_chunk<true, VIS>(sa, c, tS, tO, sc, valid_r, j == 0, j > 0, m_ref, l, wait_prev);
                        else
                            silu_chunk<true>(sa, c, tS, sc, valid_r);
                    }
                } else {
#pragma unroll 1
                    for (int c = 0; c < 2 && ok; ++c) {
                        tmem_ld32(tS + 32 * c, sa);
                        tmem_wait_ld32(sa);
                        if constexpr (MODE == CKV_SOFTMAX)
                            ok = softmax_chunk<false, VIS>(sa, c, tS, tO, sc, valid, j == 0, j > 0, m_ref, l, wait_prev);
                        else
                            silu_chunk<false>(sa, c, tS, sc, valid);
                    }
                }
                if (!ok) break;
                tc_wait_st();
                tc_fence_before();
                mbar_arrive(bar(BAR_PREADY + i));
                if (cnt > 0 && ++stage == NS) {
                    stage = 0;
                    sphase ^= 1;
                }
                ++cnt;
            }
            if (!ok) break;

            // ---- the unit's epilogue: O is complete with the last tile's weighted sum (its stage's release)
            ok = mbar_wait(bar(BAR_EMPTY + stage), sphase, abort_flag, SITE_OFULL);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            tmem_ld32(tO, sa);
            tmem_wait_ld32(sa);
            tc_fence_before();  // (the next unit overwrites O behind these warps' next hand-over)
            if (r < u.wk.M) {
                auto o = [&](int e) { return __uint_as_float(sa[e]); };
                if (u.wk.part_row < 0) {
                    float inv;
                    if constexpr (MODE == CKV_SOFTMAX) inv = l > 0.f ? 1.0f / l : 0.f;
                    else inv = 1.0f / (float)u.wk.L;
                    if (a.out_dtype == CKV_BF16) {
                        uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<uint16_t*>(a.out) + out_base);
#pragma unroll
                        for (int q4 = 0; q4 < 4; ++q4) {
                            uint4 v;
                            v.x = pack_bf16(o(8 * q4 + 0) * inv, o(8 * q4 + 1) * inv);
                            v.y = pack_bf16(o(8 * q4 + 2) * inv, o(8 * q4 + 3) * inv);
                            v.z = pack_bf16(o(8 * q4 + 4) * inv, o(8 * q4 + 5) * inv);
                            v.w = pack_bf16(o(8 * q4 + 6) * inv, o(8 * q4 + 7) * inv);
                            dst[q4] = v;
                        }
                    } else {
                        float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(a.out) + out_base);
#pragma unroll
                        for (int q4 = 0; q4 < 8; ++q4)
                            dst[q4] = make_float4(o(4 * q4) * inv, o(4 * q4 + 1) * inv, o(4 * q4 + 2) * inv, o(4 * q4 + 3) * inv);
                    }
                } else {
                    const int64_t pr = CKV_CLAMP((int64_t)(u.wk.part_row + r), a.part_rows, err_flag);
                    *part_ml(a, D, pr, u.grp) = make_float2(m_ref, l);
                    float4* dst = reinterpret_cast<float4*>(part_acc(a, D, pr, u.grp));
#pragma unroll
                    for (int q4 = 0; q4 < 8; ++q4)
                        dst[q4] = make_float4(o(4 * q4), o(4 * q4 + 1), o(4 * q4 + 2), o(4 * q4 + 3));
                }
            }
        }
        tc_wait_ld();
        if (!ok) {
            *abort_flag = 1;
            if (lane == 0) atomicOr(err_flag, ERR_NORMALISE);
        }
    } else if (warp < kProducerWarp0) {
        // --------------------------------------------------------------------- MMA issue
        // One warp, and its loop paces the worker: it is a chain of dependent instructions, so everything that can be
        // kept out of it is (descriptors are a constant plus an offset, waits poll once inline before they call).  The
        // whole warp walks it and an elected thread issues.
        constexpr uint32_t idesc_s = make_idesc(128, TH, false), idesc_pv = make_idesc(128, D, true);
        const uint64_t dq0 = smem_desc(wbase + L::Q), dk0 = smem_desc(wbase + L::K), dv0 = smem_desc(wbase + L::V);
        auto at = [](uint64_t d, uint32_t byte_off) { return d + (uint64_t)(byte_off >> 4); };  // no carry out of the address field
        auto arrived = [&](uint32_t bar, uint32_t parity, int site) {
            const bool here = mbar_wait_fast(bar, parity, abort_flag, site);
            return __all_sync(0xffffffffu, here) != 0;
        };
        Units<false, VIS> un;
        un.init(a, n_work, b);
        int cnt = 0, done = 0;    // steps whose scores / weighted sum have been issued; at most two apart
        int s = 0, par = 0;       // stage of step cnt and the phase parity of its tile
        int pv_s = 0;             // stage of step `done`
        uint32_t acc0 = 0, acc1 = 0;  // of the steps in flight, oldest first: O already holds earlier tiles of the unit
        int useq = 0;             // units begun
        bool ok = true;
        // O += P_i V for step `done`, once the normalisation warps have written P_i
        auto issue_pv = [&]() {
            const int i = done & 1;
            if (!arrived(bar(BAR_PREADY + i), (done >> 1) & 1, SITE_PREADY)) return false;
            if (elect_one()) {
                tc_fence_after();
                const uint64_t dv = at(dv0, (uint32_t)pv_s * kTileV);
#pragma unroll
                for (int kk = 0; kk < TH / 16; ++kk)  // sixteen positions per instruction
                    umma_ts(tO0, tS0 + (uint32_t)TH * i + 8 * kk, at(dv, kk * 2 * kGroupB), idesc_pv, kk > 0 ? 1u : acc0);
                tc_commit(bar(BAR_EMPTY + pv_s));
            }
            __syncwarp();
            acc0 = acc1;
            if (++pv_s == NS) pv_s = 0;
            ++done;
            return true;
        };
        for (; ok && un.valid; un.next(), ++useq) {
            const uint64_t dq = at(dq0, (uint32_t)(useq & 1) * kTileQ);
            const int n_tiles = __shfl_sync(0xffffffffu, un.u.n_tiles, 0);
            for (int j = 0; j < n_tiles; ++j) {
                // buffer i still holds the weights of step cnt - 2: its weighted sum goes first (and before the wait
                // for the tile: at a unit's end the normalisation warps wait for exactly this weighted sum).  The tensor
                // core runs this warp's instructions in order, so the scores below need not wait for it to finish.
                if (cnt - done == 2) ok = issue_pv();
                if (ok) ok = arrived(bar(BAR_FULL + s), par, SITE_TILE);
                if (!ok) break;
                const int i = cnt & 1;
                if (elect_one()) {
                    tc_fence_after();
                    const uint64_t dk = at(dk0, (uint32_t)s * kTileK);
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks)
                        umma_ss(tS0 + (uint32_t)TH * i, at(dq, ks * 32), at(dk, ks * 32), idesc_s, ks > 0 ? 1u : 0u);
                    tc_commit(bar(BAR_SFULL + i));
                    if (j == n_tiles - 1) tc_commit(bar(BAR_QEMPTY + (useq & 1)));
                }
                __syncwarp();
                (cnt == done ? acc0 : acc1) = j > 0 ? 1u : 0u;
                if (++s == NS) {
                    s = 0;
                    par ^= 1;
                }
                ++cnt;
            }
        }
        while (ok && done < cnt) ok = issue_pv();
        if (lane == 0 && !ok) {
            *abort_flag = 1;
            atomicOr(err_flag, ERR_MMA);
        }
        __syncwarp();
        // nothing of this worker may still be running on the tensor core at teardown
        if (elect_one()) tc_commit(bar(BAR_DRAIN));
        if (!mbar_wait(bar(BAR_DRAIN), 0, abort_flag + 2, SITE_DRAIN)) atomicOr(err_flag, ERR_DRAIN);
        __syncwarp();
    } else {
        // --------------------------------------------------------------------- producer
        // Lane (q = lane / 4, chunk = lane % 4) copies chunk `chunk` of the pool rows of positions 32 rb + 4 q + i
        // (rb < 2, i < 4) into tile rows 32 rb + 8 i + q, and patches the user-specific leading elements of tile rows
        // 32 rb + lane.  A tile is published one tile later, when its copies have had time to land (or as soon as there
        // is no free stage to copy into).  Its indices and user parts are contiguous streams of the arena: they come
        // into shared memory with asynchronous copies of their own, two tiles ahead (held in registers instead they
        // cost the warp a stall of a memory latency per tile, wherever the compiler moves a register).
        const int q = lane >> 2, chunk = lane & 3;
        const int patch_pos = 4 * (lane & 7) + (lane >> 3);  // position (inside a 32-block) held by row `lane`
        const uint32_t kv_lane = tile_off(q, chunk);
        const int64_t pool_stride = (int64_t)a.cv.n_entries * (D * 2);
        const char* poolK0 = reinterpret_cast<const char*>(a.cv.poolK) + chunk * 16;
        const char* poolV0 = reinterpret_cast<const char*>(a.cv.poolV) + chunk * 16;
        const uint16_t* Q = reinterpret_cast<const uint16_t*>(a.queries);
        // A side that is not shared (sharing only keys or only values): its rows are the tile's own units in the
        // arena, the position inside the tile stands in for the pool index, and nothing is patched.
        const bool full_k = a.cv.full_k != 0, full_v = a.cv.full_v != 0;
        const char* rowsK0 = reinterpret_cast<const char*>(a.cv.userK) + chunk * 16;
        const char* rowsV0 = reinterpret_cast<const char*>(a.cv.userV) + chunk * 16;
        Units<false, VIS> un;
        un.init(a, n_work, b);
        bool ok = true;
        struct Tile {
            int valid;               // real positions; 0: no tile
            int grp, q_rows;         // q_rows >= 0: first tile of a unit with that many query rows in its block
            int64_t q_row, unit0;    // first query row; arena unit of the tile's position 0
        };
        int j = 0, mslot = 0;  // tile of the unit that is requested next, and its slot of the request ring
        const uint32_t meta0 = wbase + L::M;
        unsigned char* const metap = smem + b * L::WORKER + L::M;
        auto request = [&]() {
            Tile t;
            t.valid = t.grp = 0;
            t.q_rows = -1;
            t.q_row = t.unit0 = 0;
            if (un.valid) {
                const Unit& u = un.u;
                const int pos0 = u.wk.begin + j * TH, room = u.wk.Lpad - pos0;  // (the arena is padded to 32 positions per user)
                t.grp = u.grp;
                t.unit0 = u.wk.base + (int64_t)u.grp * u.wk.Lpad + pos0;
                (void)CKV_CLAMP(t.unit0, a.arena_units, err_flag);
                t.valid = j == u.n_tiles - 1 ? u.last_valid : TH;
                if (j == 0) {
                    t.q_rows = u.wk.M - u.row0;
                    t.q_row = u.wk.q0 + u.row0;
                }
                const uint32_t dst = meta0 + mslot * L::META;
#pragma unroll
                for (int k = 0; k < (16 + 8 * DUB + 31) / 32; ++k) {
                    const int c = lane + 32 * k;  // 16-byte chunk of the slot
                    const char* src;
                    int pos;
                    bool want;
                    if (c < 16) {
                        pos = 8 * (c & 7);
                        src = reinterpret_cast<const char*>(c < 8 ? a.cv.idxK : a.cv.idxV) + (t.unit0 + pos) * 2;
                        want = c < 8 ? !full_k : !full_v;
                    } else {
                        const int side = c - 16 >= 4 * DUB, off = 16 * (c - 16 - (side ? 4 * DUB : 0));
                        pos = off / (DUB > 0 ? DUB : 1);
                        src = reinterpret_cast<const char*>(side ? a.cv.userV : a.cv.userK) + t.unit0 * DUB + off;
                        want = (side ? !full_v : !full_k) && c < 16 + 8 * DUB;
                    }
                    if (want && pos < room) cp_async16_once(dst + 16 * c, src, 16u);
                }
                if (++j == u.n_tiles) {
                    j = 0;
                    un.next();
                }
            }
            mslot = (mslot + 1) & (L::META_SLOTS - 1);
            return t;
        };
        Tile t0 = request(), t1 = request();
        cp_async_commit();
        cp_async_wait<0>();
        __syncwarp();
        int p_valid = 0, p_s = 0, p_m = 0;  // the tile whose copies are in flight: positions, stage, request slot
        auto publish = [&]() {  // its copies have landed: patch, and hand it to the issuing thread
            UserPart<DUB> xk[2], xv[2];
            if constexpr (DUB > 0) {
#pragma unroll
                for (int rb = 0; rb < 2; ++rb) {
                    const unsigned char* up = metap + p_m * L::META + 256 + (32 * rb + patch_pos) * DUB;
                    xk[rb].take(up);
                    xv[rb].take(up + TH * DUB);
                }
            }
            __syncwarp();       // a row's chunks were copied by four lanes of this warp
            if constexpr (DUB > 0) {
                unsigned char *kt = smem + b * L::WORKER + L::K + p_s * kTileK + tile_off(lane, 0),
                              *vt = smem + b * L::WORKER + L::V + p_s * kTileV + tile_off(lane, 0);
#pragma unroll
                for (int rb = 0; rb < 2; ++rb) {
                    if (32 * rb + patch_pos < p_valid) {  // zero rows beyond the history stay zero
                        if (!full_k) xk[rb].store(kt + rb * 4 * kGroupB);
                        if (!full_v) xv[rb].store(vt + rb * 4 * kGroupB);
                    }
                }
            }
            fence_proxy_async();  // by the writing threads themselves: a fence on the reading side alone is not enough
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(BAR_FULL + p_s));
            p_valid = 0;
        };
        int s = 0, useq = 0, m = 0;
        uint32_t par = 1;  // parity of the release of stage s that the next copy into it waits for (the first round passes)
        bool stage_free = true;  // of stage s, as seen an iteration ago
        while (t0.valid > 0) {
            // a free stage, and for a unit's first tile the Q block of the unit before the last
            bool free = stage_free && (t0.q_rows < 0 || mbar_test(bar(BAR_QEMPTY + (useq & 1)), ((useq >> 1) & 1) ^ 1));
            if (!__all_sync(0xffffffffu, free)) {
                if (p_valid > 0) {
                    cp_async_wait<0>();
                    publish();
                }
                ok = mbar_wait(bar(BAR_EMPTY + s), par, abort_flag, SITE_STAGE) &&
                     (t0.q_rows < 0 || mbar_wait(bar(BAR_QEMPTY + (useq & 1)), ((useq >> 1) & 1) ^ 1, abort_flag, SITE_QBUF));
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
            }
            if (t0.q_rows >= 0) {  // stage the unit's Q block (rows beyond M are zero)
                const uint32_t qdst = wbase + L::Q + (useq & 1) * kTileQ + kv_lane;
                const uint16_t* qsrc = Q + ((t0.q_row + q) * G + t0.grp) * D + chunk * 8;
                const int turn = block_turn(b, useq, min(t0.q_rows, kGroupThreads));
#pragma unroll 2
                for (int rr = 0; rr < 16; ++rr) {  // tile rows 8 rr + q
                    const int r8 = 8 * ((rr - 4 * turn) & 15);  // of the block's query row r8 + q
                    const bool in = r8 + q < t0.q_rows;
                    cp_async16_once(qdst + kGroupB * rr, in ? qsrc + (int64_t)r8 * G * D : Q, in ? 16u : 0u);
                }
                ++useq;
            }
            const char* pk = full_k ? rowsK0 + t0.unit0 * (D * 2) : poolK0 + t0.grp * pool_stride;
            const char* pv = full_v ? rowsV0 + t0.unit0 * (D * 2) : poolV0 + t0.grp * pool_stride;
            const uint32_t kdst = wbase + L::K + s * kTileK + kv_lane, vdst = wbase + L::V + s * kTileV + kv_lane;
            uint2 xk[2], xv[2];  // pool rows of this lane's positions 32 rb + 4 q .. + 3
#pragma unroll
            for (int rb = 0; rb < 2; ++rb) {
                const int p4 = 32 * rb + 4 * q;
                xk[rb] = xv[rb] = make_uint2(p4 | ((p4 + 1) << 16), (p4 + 2) | ((p4 + 3) << 16));
                if (!full_k) xk[rb] = *reinterpret_cast<const uint2*>(metap + m * L::META + 2 * p4);
                if (!full_v) xv[rb] = *reinterpret_cast<const uint2*>(metap + m * L::META + 128 + 2 * p4);
            }
            auto copies = [&](auto tail) {
#pragma unroll
                for (int it = 0; it < 8; ++it) {  // position 32 rb + 4 q + i -> tile row 32 rb + 8 i + q   (rb = it / 4, i = it % 4)
                    const int i = it & 3, pos = 32 * (it >> 2) + 4 * q + i;
                    uint32_t jk = __byte_perm(i < 2 ? xk[it >> 2].x : xk[it >> 2].y, 0, i & 1 ? 0x4432 : 0x4410),
                             jv = __byte_perm(i < 2 ? xv[it >> 2].x : xv[it >> 2].y, 0, i & 1 ? 0x4432 : 0x4410);
                    uint32_t nb = 16u;
                    if (decltype(tail)::value && pos >= t0.valid) jk = jv = nb = 0;  // rows behind the history are zero
                    // (range-checked build: pool indices below n_entries, destinations inside the stage)
                    (void)CKV_CLAMP((int)(kGroupB * it + kv_lane), kTileK - 15, err_flag);
                    (void)CKV_CLAMP((int)(kGroupB * it + kv_lane), kTileV - 15, err_flag);
                    cp_async16(kdst + kGroupB * it, pk + (size_t)CKV_CLAMP(jk, (uint32_t)(full_k ? TH : a.cv.n_entries), err_flag) * (D * 2), nb);
                    cp_async16(vdst + kGroupB * it, pv + (size_t)CKV_CLAMP(jv, (uint32_t)(full_v ? TH : a.cv.n_entries), err_flag) * (D * 2), nb);
                }
            };
            if (t0.valid == TH) copies(std::false_type{});
            else copies(std::true_type{});
            Tile t2 = request();
            cp_async_commit();
            const int s_cur = s;
            if (++s == NS) {
                s = 0;
                par ^= 1;
            }
            stage_free = mbar_test(bar(BAR_EMPTY + s), par);
            if (p_valid > 0) {
                cp_async_wait<1>();  // the copies of the tile before, and the requests of the tile behind this one
                publish();
            } else {
                cp_async_wait<1>();
                __syncwarp();
            }
            p_valid = t0.valid;
            p_s = s_cur;
            p_m = m;
            m = (m + 1) & (L::META_SLOTS - 1);
            t0 = t1;
            t1 = t2;
        }
        cp_async_wait<0>();
        if (ok && p_valid > 0) publish();
        if (!ok) {
            *abort_flag = 1;
            if (lane == 0) atomicOr(err_flag, ERR_PRODUCER);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (tid == 0 && abort_flag[1] != 0) atomicOr(err_flag, abort_flag[1] << 8);
    if (warp == kIssueWarp0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

}  // namespace

bool umma_supported(int dtype, int head_dim, int d_user, int idx_bytes)
{
    return dtype == CKV_BF16 && head_dim == D && idx_bytes == 2 &&
           (d_user == 0 || d_user == 1 || d_user == 2 || d_user == 4 || d_user == 8);
}

namespace {

// vmax[i] = largest visible length (clamped to the history) among the rows of work record i.  One warp per record.
__global__ void vis_block_max_kernel(const Work* __restrict__ works, int n_works, const int32_t* __restrict__ vis,
                                     int32_t* __restrict__ vmax)
{
    const int i = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (i >= n_works) return;
    const Work w = works[i];
    int m = 0;
    for (int r = w.row0 + (threadIdx.x & 31); r < min(w.M, w.row0 + 128); r += 32)
        m = max(m, min(max(__ldg(vis + w.q0 + r), 0), w.L));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) vmax[i] = m;
}

}  // namespace

cudaError_t launch_vis_block_max(const AttendArgs& a, int32_t* vmax, cudaStream_t s)
{
    if (a.n_works == 0) return cudaSuccess;
    vis_block_max_kernel<<<(a.n_works + 3) / 4, 128, 0, s>>>(a.works, a.n_works, a.vis, vmax);
    return cudaGetLastError();
}

cudaError_t launch_attend_umma(const AttendArgs& a, int n_sms, int* err_flag, const Launch& l)
{
    if (a.n_works == 0) return cudaSuccess;
    const int64_t n_work = (int64_t)a.n_works * a.cv.n_groups;
    if (n_work + 2 * NW * (int64_t)n_sms >= (int64_t)1 << 32) return cudaErrorInvalidValue;  // the kernel counts units in 32 bits
    const unsigned grid = (unsigned)(n_work < n_sms ? n_work : n_sms);
    auto go = [&](auto kernel, int smem_bytes) {
        return launch_kernel(l, kernel, grid, kThreads, smem_bytes, 1, a, n_work, err_flag);
    };
    const bool sm = a.mode == CKV_SOFTMAX, vis = a.vis != nullptr;
    if (vis && a.vmax == nullptr) return cudaErrorInvalidValue;
#define CKV_UMMA_GO(DUB)                                                                                          \
    (vis ? (sm ? go(attend_umma_kernel<CKV_SOFTMAX, DUB, true>, Map<DUB>::BYTES)                                  \
               : go(attend_umma_kernel<CKV_SILU_OVER_L, DUB, true>, Map<DUB>::BYTES))                             \
         : (sm ? go(attend_umma_kernel<CKV_SOFTMAX, DUB, false>, Map<DUB>::BYTES)                                 \
               : go(attend_umma_kernel<CKV_SILU_OVER_L, DUB, false>, Map<DUB>::BYTES)))
    switch (a.cv.full_k && a.cv.full_v ? 0 : a.cv.d_user) {  // the user-specific width of the shared side(s)
        case 0: return CKV_UMMA_GO(0);
        case 1: return CKV_UMMA_GO(2);
        case 2: return CKV_UMMA_GO(4);
        case 4: return CKV_UMMA_GO(8);
        case 8: return CKV_UMMA_GO(16);
    }
#undef CKV_UMMA_GO
    return cudaErrorInvalidValue;
}

}  // namespace ckv
