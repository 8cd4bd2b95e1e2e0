// trr_attn_group_step_runs.cu - the kernels of trr_decode_step with a KV head and its query group per warp,
// for caches whose splits may have more tiles than a warp plans at once.
#include "trr_row.cuh"

namespace trr {
TRR_ROW_FAMILY(, kGroup, true, true)
}  // namespace trr
