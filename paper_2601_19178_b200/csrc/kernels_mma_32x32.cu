// Warp-level tensor-core attention, 32-wide heads, 32 queries per warp.
#include "attend_mma.cuh"

namespace ckv {
template cudaError_t launch_mma<32, 2, false>(const AttendArgs&, int, int, const InlineTable*, const CUtensorMap*, int*, const Launch&);
}  // namespace ckv
