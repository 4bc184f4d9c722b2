// Internal declarations shared by the host side of the library and its kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "ckv.h"
#include "report.cuh"

namespace ckv {

// One request row of an attend plan: where the user's compressed history lives in the
// arena and which query rows belong to it.
struct Req {
    int64_t base;      // first arena unit of the user; unit(g, i) = base + g * Lpad + i
    int32_t L;         // history length
    int32_t Lpad;      // L rounded up to a multiple of 32
    int32_t q0;        // first query row
    int32_t M;         // number of query rows
    int32_t part0;     // first partial-result row block (split requests), else -1
    int32_t n_chunks;  // history chunks this request was cut into (>= 1)
};

// One unit of kernel work: a contiguous chunk of one request's history, for every group.
struct Item {
    int32_t req;
    int32_t begin;     // first position of the chunk
    int32_t len;       // positions in the chunk (0 only for an empty history)
    int32_t part_row;  // first row of this chunk's partial results, or -1: write `out`
};

// A whole request as a kernel argument: short request lists travel with the launch instead of through tables in
// device memory (no upload, nothing to wait for).  Arena units are handed out in multiples of 32, Lpad is L rounded up.
struct InlineReq {
    uint32_t base32;   // Req::base / 32
    int32_t L, q0, M;
};
constexpr int kInlineReqs = 224;  // with AttendArgs just under the 4 KB of kernel arguments that every launch can take
struct InlineTable {
    InlineReq r[kInlineReqs];
};

// A block of up to 128 query rows of an Item, merged with its request row, for kernels that read their work list once per unit
// with plain 16-byte loads (48 bytes, 16-byte aligned).
struct Work {
    int64_t base;      // Req::base
    int32_t L, Lpad;   // Req::L, Req::Lpad
    int32_t q0, M;     // Req::q0, Req::M
    int32_t begin, len, part_row;  // Item::begin, Item::len, Item::part_row
    int32_t row0;      // first query row of the block
    int32_t pad[2];
};

// Everything a kernel needs to find the compressed cache and the pool.
struct CacheView {
    const void* poolK;   // [G][m][D] rows, first d_user slots zero
    const void* poolV;
    const void* idxK;    // arena, idx_bytes per unit
    const void* idxV;
    const void* userK;   // arena, d_user elements per unit
    const void* userV;
    int32_t n_groups;
    int32_t n_entries;
    int32_t d_user;      // user-specific elements per unit of a shared side
    int32_t idx_bytes;   // 2 or 4
    // Sharing only keys or only values: a side that is not shared has no pool and no indices (poolX, idxX
    // null); its userX array holds the full head_dim-wide row of every unit.
    int32_t full_k;
    int32_t full_v;
};

struct AttendArgs {
    CacheView cv;
    const Req* reqs;
    const Item* items;
    const Work* works;     // tcgen05 family only: one per (item, block of 128 queries)
    int32_t n_works;
    int32_t n_items;
    int32_t inl;           // the requests are kernel arguments (InlineTable), one unsplit item each; reqs and items are null
    const void* queries;   // [Q][G][D]
    const int32_t* vis;    // null, or per query row the number of leading history positions it attends [Q]
    const int32_t* vmax;   // tcgen05 family with visible lengths: largest limit per work record
    void* out;             // [Q][G][D]
    float* partials;       // [part rows][G][D] accumulators, behind them [part rows][G] (m, l)
    int32_t out_dtype;     // ckv_dtype
    int32_t mode;          // ckv_mode
    float scale;
    // What the range-checked build (-DCKV_BOUNDS) compares against; unused otherwise.
    int64_t arena_units;   // units the arena arrays hold
    int64_t q_rows;        // rows of `queries` and `out`
    int64_t part_rows;     // rows of `partials`
    int* err;              // device error word (the context's)
};

#ifdef __CUDACC__
// Where the partial result of (part row, group) stands: rows on 16-byte boundaries, so that they move four floats at a time.
__device__ __forceinline__ float* part_acc(const AttendArgs& a, int D, int64_t row, int g)
{
    return a.partials + (row * a.cv.n_groups + g) * D;
}
__device__ __forceinline__ float2* part_ml(const AttendArgs& a, int D, int64_t row, int g)
{
    return reinterpret_cast<float2*>(a.partials + a.part_rows * a.cv.n_groups * D) + row * a.cv.n_groups + g;
}
#endif

// How a launcher launches: stream, the access-policy window over the pool (null: none) as a launch attribute, and the
// context's record of which kernels have been allowed how much dynamic shared memory (the permission belongs to the
// device the context sits on, so it is asked for once per context and kernel, not once per launch).
struct SmemGrants {
    static constexpr int kMax = 48;
    const void* fn[kMax];
    size_t bytes[kMax];
    int n = 0;
};
struct Launch {
    cudaStream_t s;
    const cudaAccessPolicyWindow* window;
    SmemGrants* grants;
    bool early = false;  // programmatic launch: the blocks may be set up while the stream's previous kernel still runs
                         // (the kernel waits for that one's memory itself, grid_dependency_wait)
};
inline cudaError_t grant_smem(SmemGrants* g, const void* fn, size_t bytes)
{
    if (bytes <= 48 * 1024) return cudaSuccess;
    int i = 0;
    if (g) {
        while (i < g->n && g->fn[i] != fn) ++i;
        if (i < g->n && g->bytes[i] >= bytes) return cudaSuccess;
    }
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && g && i < SmemGrants::kMax) {
        g->fn[i] = fn;
        g->bytes[i] = bytes;
        if (i == g->n) ++g->n;
    }
    return e;
}
// cluster: thread blocks per cluster along x (1: none)
template <typename... P, typename... A>
cudaError_t launch_kernel(const Launch& l, void (*fn)(P...), dim3 grid, int threads, size_t smem, int cluster, A&&... args)
{
    cudaError_t e = grant_smem(l.grants, (const void*)fn, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at[3];
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = smem;
    c.stream = l.s;
    c.attrs = at;
    if (cluster > 1) {
        at[c.numAttrs].id = cudaLaunchAttributeClusterDimension;
        at[c.numAttrs].val.clusterDim.x = (unsigned)cluster;
        at[c.numAttrs].val.clusterDim.y = at[c.numAttrs].val.clusterDim.z = 1;
        ++c.numAttrs;
    }
    if (l.window) {
        at[c.numAttrs].id = cudaLaunchAttributeAccessPolicyWindow;
        at[c.numAttrs].val.accessPolicyWindow = *l.window;
        ++c.numAttrs;
    }
    if (l.early) {
        at[c.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[c.numAttrs].val.programmaticStreamSerializationAllowed = 1;
        ++c.numAttrs;
    }
    return cudaLaunchKernelEx(&c, fn, std::forward<A>(args)...);
}

// ---- kernels_pack.cu
cudaError_t launch_pool_layout(int dtype, int G, int m, int d_shared, int D, const void* src,
                               void* dst, cudaStream_t s);
// One user of a put: where its positions start in the [P][G] inputs and its 32-position tiles among those of the batch.
struct PutUser {
    int64_t pos0;
    int32_t tile0, L;
};
constexpr int kInlinePuts = 224;  // users whose table travels as a kernel argument
struct PutTable {
    PutUser u[kInlinePuts];
};
// Packs n users' [P][G] indices and [P][G][d_user] user parts into arena units and validates the index range.  The users
// come from `table` (device memory) or, if that is null, from *inl; the arena arrays and the sides' widths from `cv`
// (head_dim D).  report.done becomes null if the kernel does not report (here and below).
cudaError_t launch_pack(int dtype, int G, int n_entries, int idx_bytes, int n_users, const PutUser* table,
                        const PutTable* inl, int64_t total_tiles, int64_t arena_base, const int32_t* idxK,
                        const int32_t* idxV, const void* userK, const void* userV, const CacheView& cv, int D,
                        Report& report, cudaStream_t s);
// Writes a user's units for L_old + L_new positions at arena unit dst_base: the first L_old positions copied from
// the units at old_base (same arena), the rest packed from the new [L_new][G] indices and [L_new][G][d_user] parts.  dst_base = old_base (and
// Lpad_tot = Lpad_old): the new positions are written behind the old ones, in place.
cudaError_t launch_append(int dtype, int G, int n_entries, int idx_bytes, int64_t old_base, int L_old,
                          int Lpad_old, int64_t dst_base, int L_new, int Lpad_tot, const int32_t* idxK,
                          const int32_t* idxV, const void* userK, const void* userV, const CacheView& cv, int D,
                          Report& report, cudaStream_t s);
cudaError_t launch_materialize(int dtype, int D, const CacheView& cv, int64_t base, int L, int Lpad,
                               void* K_out, void* V_out, cudaStream_t s);

// *bad_flag (host-mapped int) becomes 1 if any of the n_units stored K or V indices is >= n_entries (idxK or idxV may be
// null: that side is not checked).
cudaError_t launch_check_indices(int idx_bytes, int n_entries, const void* idxK, const void* idxV, int64_t n_units,
                                 int* bad_flag, cudaStream_t s);

// ---- kernels_simt.cu : CUDA-core family (any number of queries, best for few)
// tab: the requests when a.inl is set.  wide: blocks of more warps (few blocks, each with a history to itself)
cudaError_t launch_attend_simt(int dtype, int D, int max_M, bool wide, const AttendArgs& a, const InlineTable* tab,
                               const Launch& l);
// Merges the partial results of split requests into `out`.
cudaError_t launch_combine(int D, int max_M, const AttendArgs& a, const int32_t* split_reqs, int n_split, const Launch& l);

// ---- kernels_mma.cu, attend_mma.cuh, kernels_mma_*.cu : warp-level tensor-core family (bf16, head_dim 32 or 64, d_user <= 8)
bool mma_supported(int dtype, int head_dim, int d_user);  // d_user of the shared side(s)
// big: every resident warp has some twenty tiles of 32 positions x 16 queries to do
int mma_queries_per_warp(int head_dim, int max_M, bool big);
// tensor_maps: null = fill the staging ring with cp.async copies; else the two maps of make_pool_tensor_maps =
// fill it with TMA gathers (err_flag: device int, OR-ed with a code if a bounded wait for a tile ran out).
// parts: warps that share one (item, group, query block), a power of two up to kMmaMaxParts; more than four lie in a
// cluster of thread blocks.  tab: the requests when a.inl is set (cp.async loader only).  dense: more resident warps with
// shallower rings (head_dim 64, 16 queries a warp, the plain form with cp.async; ignored elsewhere).
constexpr int kMmaMaxParts = 32;
cudaError_t launch_attend_mma(int head_dim, int max_M, int queries_per_warp, int parts, bool dense, const AttendArgs& a, const InlineTable* tab,
                              const void* tensor_maps, int* err_flag, const Launch& l);
int mma_warps_per_sm(int head_dim, int queries_per_warp, bool dense = false);
bool make_pool_tensor_maps(int head_dim, int64_t rows, const void* poolK, const void* poolV, void* maps_out);

// ---- kernels_fact.cu : pool-side factorisation for one query per user (bf16, head_dim 32 or 64, d_user <= 8)
bool fact_supported(int dtype, int head_dim, int d_user, int n_entries);
// Floats of workspace for a list of n_items requests.
int64_t fact_workspace_floats(int n_items, int n_groups, int n_entries);
// a.items: one unsplit item per request with a query.  Adds the kernels launched to *launches.
cudaError_t launch_attend_fact(int head_dim, const AttendArgs& a, int n_sms, float* ws, const Launch& l, int* launches);

// ---- kernels_route.cu : prefill router, fused scores + row arg-max (bf16, d_in 32 / 64 / 128)
bool route_supported(int d_in);
// out[i][g] = lowest entry j maximising x_i . W[g][j] + bias[g][j]; x [n][d_in], W [G][n_entries][d_in] bf16 (device),
// bias [G][n_entries] fp32 or null, out [n][G] int32.
cudaError_t launch_route(int d_in, const void* x, const void* W, const float* bias, int n, int n_entries, int G,
                         int32_t* out, cudaStream_t s);

// ---- kernels_route_umma.cu : the same router on tcgen05 (TMEM accumulators, warp-specialised)
// flags: two host-mapped ints.  flags[0] becomes non-zero if a bounded wait inside the kernel ran out (`out` is not
// valid then, whether written or not).  If *slot is in [0, kRouteSlots), and no other launch uses it at the time, flags[1] becomes 1
// at its end; where the kernel does not report (several rounds of blocks) *slot becomes -1.
constexpr int kRouteSlots = 64;
cudaError_t launch_route_umma(int d_in, const void* x, const void* W, const float* bias, int n, int n_entries, int G,
                              int32_t* out, int* flags, int* slot, cudaStream_t s);

// kernels_route.cu, the same for few positions (route_few says which calls that is): the entries shared by the warps of a
// cluster.  flags, slot: as above, flags[0] stays 0.
bool route_few(int d_in, const void* x, const void* W, int n, int n_entries, int G);
cudaError_t launch_route_few(int d_in, const void* x, const void* W, const float* bias, int n, int n_entries, int G,
                             int32_t* out, int* flags, int* slot, cudaStream_t s);

// out[i][g][c] = x_i . W[g][c] + bias[g][c] (bf16 in and out, fp32 sums); W [G][d_out][d_in], bias [G][d_out] or null.
bool project_supported(int d_in, int d_out, int n_groups);
cudaError_t launch_project(int d_in, int d_out, int G, const void* x, const void* W, const float* bias, int64_t n,
                           void* out, cudaStream_t s);

// ---- kernels_umma.cu : tcgen05 family (bf16, head_dim 32, d_user in {0, 1, 2, 4, 8}, 16-bit stored indices)
bool umma_supported(int dtype, int head_dim, int d_user, int idx_bytes);
// err_flag: device int, OR-ed with a non-zero code if a bounded wait inside the kernel ran out.
// Persistent: one CTA per SM (n_sms of them at most).
cudaError_t launch_attend_umma(const AttendArgs& a, int n_sms, int* err_flag, const Launch& l);
// Fills vmax (one int per work record) from a.vis; a.works as for the attend.
cudaError_t launch_vis_block_max(const AttendArgs& a, int32_t* vmax, cudaStream_t s);

}  // namespace ckv
