// cg_tc_tiles.cu -- tensor-core encode of block-uniform tiles (one range per 16 tokens x block,
// Sec. 4.3 with T_b = 16 from Sec. 4.2); the kernel is in cg_tc_rows.cuh.
#include "cg_tc_rows.cuh"

namespace cg {

// The shapes of the row encoder (it takes the same rows; only the ranges differ): below 64 tokens
// a call fills less than half of a 128-row MMA tile.
bool tc_tile_encode_eligible(const RowArgs& a) { return tc_row_encode_eligible(a); }

cudaError_t tc_launch_tile_encode(const RowArgs& a, cudaStream_t st) { return launch_rows_any<true>(a, st); }

}  // namespace cg
