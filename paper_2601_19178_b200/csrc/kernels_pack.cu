// Data-movement kernels: pool row layout, compressed-cache packing with index
// validation, and the test-only full-width materialisation (Eq. Kc + Eq. K).
// All of them copy bits; none does arithmetic on values.
#include <algorithm>

#include "ckv_internal.h"

namespace ckv {
namespace {

// dst[g][j][c] = c < d_user ? 0 : src[g][j][c - d_user]      (rows padded to the head width)
template <typename E>
__global__ void pool_layout_kernel(const E* __restrict__ src, E* __restrict__ dst, int64_t rows,
                                   int d_shared, int D)
{
    const int d_user = D - d_shared;
    const int64_t total = rows * D;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / D;
        const int c = (int)(t - r * D);
        dst[t] = c < d_user ? E(0) : src[r * d_shared + (c - d_user)];
    }
}

// The two sides of a cache entry (K and V) are stored alike but may differ in width: a shared side keeps a pool
// index and d_user user-specific elements per unit, a side that is not shared (sharing only keys or only values)
// keeps the whole head_dim-wide row and no index.
struct SideDst {
    void* idx;     // arena indices, null for a side that is not shared
    void* user;    // arena user parts / full rows
    int width;     // elements per unit in `user`
    int vec;       // bytes per unit if they can be moved from the caller's array as one word, else 0
    int vec_arena; // the same between units of the arena
};
// A unit's user part is one word if its size is a power of two of 4 to 16 bytes and the caller's array is aligned to it
// (the arena is: units start at multiples of the size).
inline int vec_bytes(int bytes, const void* src)
{
    return (bytes == 4 || bytes == 8 || bytes == 16) && (uintptr_t)src % (uintptr_t)bytes == 0 ? bytes : 0;
}
inline SideDst side_dst(bool full, const void* idx, const void* user, int d_user, int D, int elem, const void* src)
{
    const int width = full ? D : d_user;
    return SideDst{full ? nullptr : const_cast<void*>(idx), const_cast<void*>(user), width, vec_bytes(width * elem, src),
                   vec_bytes(width * elem, nullptr)};
}

// `bytes` bytes of one unit: one access where they are a word of 4 to 16 bytes (aligned on both sides, see vec_bytes),
// else element by element
template <typename E>
__device__ __forceinline__ void copy_user(E* dst, const E* src, int width, int vec, bool real)
{
    switch (vec) {
        case 4: *reinterpret_cast<uint32_t*>(dst) = real ? __ldg(reinterpret_cast<const uint32_t*>(src)) : 0u; return;
        case 8:
            *reinterpret_cast<uint2*>(dst) = real ? __ldg(reinterpret_cast<const uint2*>(src)) : make_uint2(0, 0);
            return;
        case 16:
            *reinterpret_cast<uint4*>(dst) = real ? __ldg(reinterpret_cast<const uint4*>(src)) : make_uint4(0, 0, 0, 0);
            return;
    }
    for (int c = 0; c < width; ++c) dst[c] = real ? __ldg(src + c) : E(0);
}

// Returns whether the index was out of range (an entry of the pool is stored in its place).
template <typename E, typename I>
__device__ __forceinline__ bool store_unit(const SideDst& d, int64_t dst, const int32_t* idx_src, const E* user_src,
                                           int64_t src, bool real, int n_entries)
{
    bool bad = false;
    int32_t j = d.idx && real ? __ldg(idx_src + src) : 0;
    if (d.width > 0)
        copy_user<E>(reinterpret_cast<E*>(d.user) + dst * d.width, user_src + src * d.width, d.width, d.vec, real);
    if (d.idx) {  // padding: a valid row index (and zeros)
        bad = j < 0 || j >= n_entries;
        reinterpret_cast<I*>(d.idx)[dst] = (I)(bad ? 0 : j);
    }
    return bad;
}

// One warp per tile of 32 positions of one user, every group of them: the inputs are [position][group], the arena is
// [group][position], so a lane reads its position's groups one after the other out of the same few sectors and every
// store of the warp is contiguous.  A warp takes a run of consecutive tiles: one search in the user table for all of
// them.  Bound by DRAM traffic.  The whole call for 65536 users of 512 positions and 4 groups takes 5.5 ms, 15.6 with one
// thread per unit and a search each; 512 users of 1000..16384 positions 228 us, before 498; one user 23 us, before 41.
template <typename E, typename I>
__global__ void __launch_bounds__(256) pack_kernel(int G, int n_entries, int n_users, const PutUser* __restrict__ table,
                                                   int64_t total_tiles, int64_t arena_base, const int32_t* __restrict__ idxK,
                                                   const int32_t* __restrict__ idxV, const E* __restrict__ userK,
                                                   const E* __restrict__ userV, SideDst dK, SideDst dV, Report report,
                                                   const __grid_constant__ PutTable inl)
{
    const PutUser* tab = table ? table : inl.u;
    const int lane = threadIdx.x & 31;
    const int64_t n_warps = (int64_t)gridDim.x * (blockDim.x / 32), w = blockIdx.x * (int64_t)(blockDim.x / 32) + (threadIdx.x >> 5);
    const int64_t t0 = total_tiles * w / n_warps, t1 = total_tiles * (w + 1) / n_warps;
    int u = 0, hi = n_users;  // last user whose first tile is <= t0
    while (hi - u > 1) {
        const int mid = (u + hi) >> 1;
        if (tab[mid].tile0 <= t0) u = mid; else hi = mid;
    }
    PutUser e = tab[u];
    bool bad = false;
    for (int64_t t = t0; t < t1; ++t) {
        while (u + 1 < n_users && tab[u + 1].tile0 <= t) e = tab[++u];
        const int i = (int)(32 * (t - e.tile0)) + lane, Lpad = (e.L + 31) & ~31;
        const int64_t dst = arena_base + 32 * (int64_t)e.tile0 * G + i, src = (e.pos0 + i) * G;
        const bool real = i < e.L;
#pragma unroll 4
        for (int g = 0; g < G; ++g) {
            bad |= store_unit<E, I>(dK, dst + (int64_t)g * Lpad, idxK, userK, src + g, real, n_entries);
            bad |= store_unit<E, I>(dV, dst + (int64_t)g * Lpad, idxV, userV, src + g, real, n_entries);
        }
    }
    report_done(report, bad, gridDim.x);
}

template <typename E, typename I>
__device__ __forceinline__ void copy_unit(const SideDst& d, int64_t dst, int64_t src)
{
    E* du = reinterpret_cast<E*>(d.user);
    copy_user<E>(du + dst * d.width, du + src * d.width, d.width, d.vec_arena, true);
    if (d.idx) reinterpret_cast<I*>(d.idx)[dst] = reinterpret_cast<I*>(d.idx)[src];
}

// Append: units of one user with L_old + L_new positions at arena unit `dst_base`; position i < L_old is copied
// from the user's old units, the rest comes from the new [L_new][G] inputs (range-checked like pack_kernel).  With
// dst_base = old_base (the new positions fit the old padding) only positions from L_old on are written.
template <typename E, typename I>
__global__ void append_kernel(int G, int n_entries, int64_t old_base, int L_old, int Lpad_old,
                              int64_t dst_base, int L_new, int Lpad_tot, const int32_t* __restrict__ idxK,
                              const int32_t* __restrict__ idxV, const E* __restrict__ userK,
                              const E* __restrict__ userV, SideDst dK, SideDst dV, Report report)
{
    const int first = dst_base == old_base ? L_old : 0, n = Lpad_tot - first;
    const int64_t total = (int64_t)G * n;
    bool bad = false;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int g = (int)(t / n);
        const int i = first + (int)(t - (int64_t)g * n);
        const int64_t dst = dst_base + (int64_t)g * Lpad_tot + i;
        if (i < L_old) {
            const int64_t src = old_base + (int64_t)g * Lpad_old + i;
            copy_unit<E, I>(dK, dst, src);
            copy_unit<E, I>(dV, dst, src);
        } else {
            const int64_t src = (int64_t)(i - L_old) * G + g;
            const bool real = i < L_old + L_new;
            bad |= store_unit<E, I>(dK, dst, idxK, userK, src, real, n_entries);
            bad |= store_unit<E, I>(dV, dst, idxV, userV, src, real, n_entries);
        }
    }
    report_done(report, bad, gridDim.x);
}

template <typename E, typename I>
__global__ void materialize_kernel(int G, int n_entries, int D, CacheView cv, int64_t base, int L, int Lpad,
                                   E* __restrict__ K_out, E* __restrict__ V_out)
{
    const E* poolK = reinterpret_cast<const E*>(cv.poolK);
    const E* poolV = reinterpret_cast<const E*>(cv.poolV);
    const I* idxK = reinterpret_cast<const I*>(cv.idxK);
    const I* idxV = reinterpret_cast<const I*>(cv.idxV);
    const E* userK = reinterpret_cast<const E*>(cv.userK);
    const E* userV = reinterpret_cast<const E*>(cv.userV);
    const int duk = cv.full_k ? D : cv.d_user, duv = cv.full_v ? D : cv.d_user;
    const int64_t total = (int64_t)L * G * D;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(t % D);
        const int64_t ig = t / D;
        const int g = (int)(ig % G);
        const int64_t i = ig / G;
        const int64_t unit = base + (int64_t)g * Lpad + i;
        K_out[t] = c < duk ? userK[unit * duk + c] : poolK[((int64_t)g * n_entries + (int64_t)idxK[unit]) * D + c];
        V_out[t] = c < duv ? userV[unit * duv + c] : poolV[((int64_t)g * n_entries + (int64_t)idxV[unit]) * D + c];
    }
}

// Range check of stored indices that did not go through pack_kernel (imported blobs).
template <typename I>
__global__ void check_indices_kernel(const I* __restrict__ a, const I* __restrict__ b, int64_t n, uint32_t n_entries,
                                     int* bad_flag)
{
    bool bad = false;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        bad |= (a && (uint32_t)a[i] >= n_entries) || (b && (uint32_t)b[i] >= n_entries);
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) *reinterpret_cast<volatile int*>(bad_flag) = 1;
}

inline int grid_for(int64_t total, int block)
{
    int64_t g = (total + block - 1) / block;
    if (g < 1) g = 1;
    if (g > 148 * 32) g = 148 * 32;
    return (int)g;
}

}  // namespace

cudaError_t launch_pool_layout(int dtype, int G, int m, int d_shared, int D, const void* src,
                               void* dst, cudaStream_t s)
{
    const int64_t rows = (int64_t)G * m;
    const int grid = grid_for(rows * D, 256);
    if (dtype == CKV_BF16)
        pool_layout_kernel<uint16_t><<<grid, 256, 0, s>>>((const uint16_t*)src, (uint16_t*)dst, rows,
                                                          d_shared, D);
    else
        pool_layout_kernel<uint32_t><<<grid, 256, 0, s>>>((const uint32_t*)src, (uint32_t*)dst, rows,
                                                          d_shared, D);
    return cudaGetLastError();
}

// Beyond this many blocks a kernel takes so long that a synchronise costs nothing in comparison.
constexpr int kMaxReporting = 1024;

cudaError_t launch_pack(int dtype, int G, int n_entries, int idx_bytes, int n_users, const PutUser* table,
                        const PutTable* inl, int64_t total_tiles, int64_t arena_base, const int32_t* idxK,
                        const int32_t* idxV, const void* userK, const void* userV, const CacheView& cv, int D,
                        Report& report, cudaStream_t s)
{
    if (total_tiles == 0) return cudaSuccess;
    // two warps per block while that leaves SMs without a block, then eight; at most 16 blocks of eight per SM
    const int block = total_tiles <= 148 * 8 ? 64 : 256, wpb = block / 32;
    const int grid = (int)std::min<int64_t>((total_tiles + wpb - 1) / wpb, 148 * 16);
    if (grid > kMaxReporting) report.done = nullptr;
    static const PutTable none{};
    const PutTable& pt = inl ? *inl : none;
    const int es = dtype == CKV_BF16 ? 2 : 4;
    const SideDst dK = side_dst(cv.full_k, cv.idxK, cv.userK, cv.d_user, D, es, userK);
    const SideDst dV = side_dst(cv.full_v, cv.idxV, cv.userV, cv.d_user, D, es, userV);
#define CKV_PACK(E, I)                                                                                         \
    pack_kernel<E, I><<<grid, block, 0, s>>>(G, n_entries, n_users, table, total_tiles, arena_base, idxK, idxV, \
                                             (const E*)userK, (const E*)userV, dK, dV, report, pt)
    if (dtype == CKV_BF16) {
        if (idx_bytes == 2) CKV_PACK(uint16_t, uint16_t); else CKV_PACK(uint16_t, int32_t);
    } else {
        if (idx_bytes == 2) CKV_PACK(uint32_t, uint16_t); else CKV_PACK(uint32_t, int32_t);
    }
#undef CKV_PACK
    return cudaGetLastError();
}

cudaError_t launch_append(int dtype, int G, int n_entries, int idx_bytes, int64_t old_base, int L_old,
                          int Lpad_old, int64_t dst_base, int L_new, int Lpad_tot, const int32_t* idxK,
                          const int32_t* idxV, const void* userK, const void* userV, const CacheView& cv, int D,
                          Report& report, cudaStream_t s)
{
    const int64_t total = (int64_t)G * (Lpad_tot - (dst_base == old_base ? L_old : 0));
    if (total == 0) return cudaSuccess;
    const int grid = grid_for(total, 256);
    if (grid > kMaxReporting) report.done = nullptr;
    const int es = dtype == CKV_BF16 ? 2 : 4;
    const SideDst dK = side_dst(cv.full_k, cv.idxK, cv.userK, cv.d_user, D, es, userK);
    const SideDst dV = side_dst(cv.full_v, cv.idxV, cv.userV, cv.d_user, D, es, userV);
#define CKV_APPEND(E, I)                                                                                       \
    append_kernel<E, I><<<grid, 256, 0, s>>>(G, n_entries, old_base, L_old, Lpad_old, dst_base, L_new,        \
                                             Lpad_tot, idxK, idxV, (const E*)userK, (const E*)userV, dK, dV,  \
                                             report)
    if (dtype == CKV_BF16) {
        if (idx_bytes == 2) CKV_APPEND(uint16_t, uint16_t); else CKV_APPEND(uint16_t, int32_t);
    } else {
        if (idx_bytes == 2) CKV_APPEND(uint32_t, uint16_t); else CKV_APPEND(uint32_t, int32_t);
    }
#undef CKV_APPEND
    return cudaGetLastError();
}

cudaError_t launch_materialize(int dtype, int D, const CacheView& cv, int64_t base, int L, int Lpad,
                               void* K_out, void* V_out, cudaStream_t s)
{
    if (L == 0) return cudaSuccess;
    const int grid = grid_for((int64_t)L * cv.n_groups * D, 256);
#define CKV_MAT(E, I)                                                                            \
    materialize_kernel<E, I><<<grid, 256, 0, s>>>(cv.n_groups, cv.n_entries, D, cv, base, L, Lpad, \
                                                  (E*)K_out, (E*)V_out)
    if (dtype == CKV_BF16) {
        if (cv.idx_bytes == 2) CKV_MAT(uint16_t, uint16_t); else CKV_MAT(uint16_t, int32_t);
    } else {
        if (cv.idx_bytes == 2) CKV_MAT(uint32_t, uint16_t); else CKV_MAT(uint32_t, int32_t);
    }
#undef CKV_MAT
    return cudaGetLastError();
}

cudaError_t launch_check_indices(int idx_bytes, int n_entries, const void* idxK, const void* idxV, int64_t n_units,
                                 int* bad_flag, cudaStream_t s)
{
    if (n_units == 0) return cudaSuccess;
    const int grid = grid_for(n_units, 256);
    if (idx_bytes == 2)
        check_indices_kernel<uint16_t><<<grid, 256, 0, s>>>((const uint16_t*)idxK, (const uint16_t*)idxV, n_units,
                                                            (uint32_t)n_entries, bad_flag);
    else
        check_indices_kernel<int32_t><<<grid, 256, 0, s>>>((const int32_t*)idxK, (const int32_t*)idxV, n_units,
                                                           (uint32_t)n_entries, bad_flag);
    return cudaGetLastError();
}

}  // namespace ckv
