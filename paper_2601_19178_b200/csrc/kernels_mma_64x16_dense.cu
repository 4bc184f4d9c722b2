// Warp-level tensor-core attention, 64-wide heads, 16 queries per warp, twelve warps on an SM.
#include "attend_mma.cuh"

namespace ckv {
template cudaError_t launch_mma<64, 1, true>(const AttendArgs&, int, int, const InlineTable*, const CUtensorMap*, int*, const Launch&);
}  // namespace ckv
