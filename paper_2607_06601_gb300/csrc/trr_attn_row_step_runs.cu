// trr_attn_row_step_runs.cu - the kernels of trr_decode_step with one query head per warp,
// for caches whose splits may have more tiles than a warp plans at once.
#include "trr_row.cuh"

namespace trr {
TRR_ROW_FAMILY(, kRow, true, true)
}  // namespace trr
