// Cooperative search kernel for __nv_bfloat16 traversal rows, 4 distance warps per query.
#include "csearch_inst.cuh"

namespace uhnsw_dev {

cudaError_t launch_csearch_bf16_w4(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st) {
  return claunch_shape<__nv_bfloat16, 4>(sh, a, grid, smem, st);
}

int csearch_regs_bf16_w4(WarpShape sh) { return cregs_shape<__nv_bfloat16, 4>(sh); }

}  // namespace uhnsw_dev
