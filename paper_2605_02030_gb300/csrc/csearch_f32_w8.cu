// Cooperative search kernel for float traversal rows, 8 distance warps per query.
#include "csearch_inst.cuh"

namespace uhnsw_dev {

cudaError_t launch_csearch_f32_w8(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st) {
  return claunch_shape<float, 8>(sh, a, grid, smem, st);
}

int csearch_regs_f32_w8(WarpShape sh) { return cregs_shape<float, 8>(sh); }

}  // namespace uhnsw_dev
