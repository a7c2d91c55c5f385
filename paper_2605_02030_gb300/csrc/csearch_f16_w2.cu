// Cooperative search kernel for __half traversal rows, 2 distance warps per query.
#include "csearch_inst.cuh"

namespace uhnsw_dev {

cudaError_t launch_csearch_f16_w2(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st) {
  return claunch_shape<__half, 2>(sh, a, grid, smem, st);
}

int csearch_regs_f16_w2(WarpShape sh) { return cregs_shape<__half, 2>(sh); }

}  // namespace uhnsw_dev
