// trr_attn_row_runs.cu - the kernels of trr_decode_attn with one query head per warp (one mode per query),
// for caches whose splits may have more tiles than a warp plans at once.
#include "trr_row.cuh"

namespace trr {
TRR_ROW_FAMILY(, kRow, false, true)
}  // namespace trr
