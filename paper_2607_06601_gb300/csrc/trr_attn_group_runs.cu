// trr_attn_group_runs.cu - the kernels of trr_decode_attn with a KV head and its query group per warp,
// for caches whose splits may have more tiles than a warp plans at once.
#include "trr_row.cuh"

namespace trr {
TRR_ROW_FAMILY(, kGroup, false, true)
}  // namespace trr
