// trr_attn_row_heads_runs.cu - the kernels of trr_decode_attn with one query head per warp (a mode per head),
// for caches whose splits may have more tiles than a warp plans at once.
#include "trr_row.cuh"

namespace trr {
TRR_ROW_FAMILY(, kHeads, false, true)
}  // namespace trr
