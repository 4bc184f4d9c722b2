// Dispatch of the warp-level tensor-core attention kernel (attend_mma.cuh) and the tensor maps of its TMA loader.
#include "ckv_internal.h"
#include "tensor_map.h"

namespace ckv {

template <int D, int MT, bool DENSE>
cudaError_t launch_mma(const AttendArgs& a, int n_mb, int parts, const InlineTable* tab, const CUtensorMap* maps,
                       int* err_flag, const Launch& l);

bool mma_supported(int dtype, int head_dim, int d_user)
{
    return dtype == CKV_BF16 && (head_dim == 32 || head_dim == 64) && d_user <= 8;
}

// Queries a warp holds.  One 16-query tile gathers a row for every tile of a user's queries, but leaves registers for more
// warps (16 an SM at 32-wide heads, 12 with two tiles, 8 with three) and starts and merges sooner; more tiles pay only when
// every resident warp has `big` amounts of work: 200 users x 1000 positions, 64-wide, 20..32 queries 64 us with two tiles, 75
// with one (40 queries: 105 either way); 32-wide, 3000 users x 300 positions x 4 groups, SiLU / softmax, 32 queries 119 / 145
// us with two tiles, 133 / 152 with one, 33..47 queries 168 / 222 with three, 193 / 217 with one.
int mma_queries_per_warp(int D, int max_M, bool big)
{
    if (!big || max_M <= 16) return 16;
    return D == 64 || max_M <= 32 ? 32 : 48;
}

// warps of the kernel that are resident on an SM
int mma_warps_per_sm(int D, int queries_per_warp, bool dense)
{
    if (dense) return 12;
    return D == 64 ? 8 : queries_per_warp == 16 ? 16 : queries_per_warp == 32 ? 12 : 8;
}

cudaError_t launch_attend_mma(int D, int max_M, int queries_per_warp, int parts, bool dense, const AttendArgs& a, const InlineTable* tab,
                              const void* tensor_maps, int* err_flag, const Launch& l)
{
    if (a.n_items == 0) return cudaSuccess;
    const CUtensorMap* maps = reinterpret_cast<const CUtensorMap*>(tensor_maps);
    if (maps && D == 32 && queries_per_warp == 32) queries_per_warp = 16;  // (no such form with the TMA loader; the same bits)
    const int n_mb = (max_M + queries_per_warp - 1) / queries_per_warp;
    if (D == 64) {
        if (dense && queries_per_warp == 16 && !maps && !a.vis && !a.cv.full_k && !a.cv.full_v)
            return launch_mma<64, 1, true>(a, n_mb, parts, tab, maps, err_flag, l);
        return queries_per_warp == 16 ? launch_mma<64, 1, false>(a, n_mb, parts, tab, maps, err_flag, l)
                                      : launch_mma<64, 2, false>(a, n_mb, parts, tab, maps, err_flag, l);
    }
    return queries_per_warp == 16   ? launch_mma<32, 1, false>(a, n_mb, parts, tab, maps, err_flag, l)
           : queries_per_warp == 32 ? launch_mma<32, 2, false>(a, n_mb, parts, tab, maps, err_flag, l)
                                    : launch_mma<32, 3, false>(a, n_mb, parts, tab, maps, err_flag, l);
}

// Tensor maps of the K and the V pool ([n_groups * n_entries] rows of head_dim bf16) for tile::gather4: a box of
// one row, hardware swizzle of the row's 16-byte chunks (128-byte rows: chunk ^ (row & 7); 64-byte rows:
// chunk ^ ((row >> 1) & 3)).  maps_out: 2 x 128 bytes, 64-byte aligned.  false if the driver cannot encode them.
bool make_pool_tensor_maps(int D, int64_t rows, const void* poolK, const void* poolV, void* maps_out)
{
    if ((D != 32 && D != 64) || rows < 1 || rows > INT32_MAX) return false;
    CUtensorMap* maps = reinterpret_cast<CUtensorMap*>(maps_out);
    const void* src[2] = {poolK, poolV};
    for (int i = 0; i < 2; ++i)
        if (!encode_rows(&maps[i], src[i], D, rows, D, 1, D == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                         CU_TENSOR_MAP_L2_PROMOTION_NONE))
            return false;
    return true;
}

}  // namespace ckv
