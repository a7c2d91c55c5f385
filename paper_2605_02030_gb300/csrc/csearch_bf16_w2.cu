// Cooperative search kernel for __nv_bfloat16 traversal rows, 2 distance warps per query.
#include "csearch_inst.cuh"

namespace uhnsw_dev {

cudaError_t launch_csearch_bf16_w2(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st) {
  return claunch_shape<__nv_bfloat16, 2>(sh, a, grid, smem, st);
}

int csearch_regs_bf16_w2(WarpShape sh) { return cregs_shape<__nv_bfloat16, 2>(sh); }

}  // namespace uhnsw_dev
