// cg_tc_rows.cu -- tensor-core encode of block-uniform rows and KIVI value rows (one range per
// block of a token); the kernel is in cg_tc_rows.cuh.
#include "cg_tc_rows.cuh"

namespace cg {

bool tc_row_encode_eligible(const RowArgs& a) {
    if (a.d != kD || a.none_mode) return false;
    if (!(a.blk == 32 || a.blk == 64 || a.blk == 128)) return false;
    if (a.t_count < 64) return false;
    const int64_t rows = (int64_t)a.L * 2 * a.B * a.H * a.T_x;
    if (rows + 128 >= (int64_t)1 << 31) return false;
    if ((reinterpret_cast<uintptr_t>(a.x) & 15u) || (reinterpret_cast<uintptr_t>(a.codes) & 15u)) return false;
    return tmap_encode_fn() != nullptr;
}

cudaError_t tc_launch_row_encode(const RowArgs& a, cudaStream_t st) { return launch_rows_any<false>(a, st); }

}  // namespace cg
