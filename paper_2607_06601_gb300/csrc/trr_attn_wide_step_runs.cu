// trr_attn_wide_step_runs.cu - the kernels of trr_decode_step with a KV head and 8 / (d/G) heads of its query
// group per warp, for groups wider than that,
// for caches whose splits may have more tiles than a warp plans at once.
#include "trr_row.cuh"

namespace trr {
TRR_ROW_FAMILY(, kWide, true, true)
}  // namespace trr
