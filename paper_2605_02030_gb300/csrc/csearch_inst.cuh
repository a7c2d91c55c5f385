// Instantiation of the cooperative search kernel for one storage type and one
// number of distance warps: the team shapes of the warp kernel's defaults and
// of the block-per-query form (pick_warp_shape, pick_block_shape).
#pragma once

#include <atomic>

#include "coop_kernels.cuh"
#include "launch.h"

namespace uhnsw_dev {

// Rows per team and round.
template <int CPL>
struct CoopRows {
  static constexpr int value = CPL <= 4 ? 2 : 1;
};

template <typename T, int TEAM, int CPL, int NW>
auto csearch_kernel(bool most) {
  constexpr int U = CoopRows<CPL>::value;
  auto kern = uhnsw_csearch_kernel<T, TEAM, CPL, U, NW, false>;
  if constexpr (coop_has_many<T, TEAM, CPL, NW>())
    if (most) kern = uhnsw_csearch_kernel<T, TEAM, CPL, U, NW, true>;
  return kern;
}

template <typename T, int TEAM, int CPL, int NW>
cudaError_t claunch_one(bool most, const QueryArgs& a, int grid, size_t smem, cudaStream_t st) {
  return launch_search_kernel(csearch_kernel<T, TEAM, CPL, NW>(most), grid, (NW + 1) * 32, smem, a, st);
}

// Resident blocks per SM that the registers allow, asked of the runtime once (0: it
// failed, as it does where the kernel's first load finds no device memory; the next
// call asks again).
template <typename T, int TEAM, int CPL, int NW, bool MOST>
int cregs_one() {
  static std::atomic<int> known{0};
  int blocks = known.load(std::memory_order_relaxed);
  if (blocks > 0) return blocks;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &blocks, csearch_kernel<T, TEAM, CPL, NW>(MOST), (NW + 1) * 32, 0) != cudaSuccess)
    return 0;
  known.store(blocks, std::memory_order_relaxed);
  return blocks;
}

// Calls CALL(T, TEAM, CPL, NW) for the compiled shape.  (4 x 3, 16 x 1 and 32 x
// 1 serve 16-bit rows; only FP32 rows reach 32 x 16.)
#define UHNSW_CSHAPE_SWITCH(T, SH, NW, CALL)                        \
  do {                                                              \
    constexpr bool k16 = sizeof(T) == 2;                            \
    switch ((SH).team * 1000 + (SH).cpl) {                          \
      case 8001: return CALL(T, 8, 1, NW);                          \
      case 8002: return CALL(T, 8, 2, NW);                          \
      case 16002: return CALL(T, 16, 2, NW);                        \
      case 32002: return CALL(T, 32, 2, NW);                        \
      case 32004: return CALL(T, 32, 4, NW);                        \
      case 32008: return CALL(T, 32, 8, NW);                        \
      case 4003: if constexpr (k16) return CALL(T, 4, 3, NW);       \
        break;                                                      \
      case 16001: if constexpr (k16) return CALL(T, 16, 1, NW);     \
        break;                                                      \
      case 32001: if constexpr (k16) return CALL(T, 32, 1, NW);     \
        break;                                                      \
      case 32016: if constexpr (!k16) return CALL(T, 32, 16, NW);   \
        break;                                                      \
    }                                                               \
  } while (0)

#define CLAUNCH_CALL(T, TEAM, CPL, NW) claunch_one<T, TEAM, CPL, NW>(sh.most, a, grid, smem, st)
#define CREGS_CALL(T, TEAM, CPL, NW) \
  (sh.most ? cregs_one<T, TEAM, CPL, NW, true>() : cregs_one<T, TEAM, CPL, NW, false>())

template <typename T, int NW>
cudaError_t claunch_shape(WarpShape sh, const QueryArgs& a, int grid, size_t smem, cudaStream_t st) {
  UHNSW_CSHAPE_SWITCH(T, sh, NW, CLAUNCH_CALL);
  return cudaErrorInvalidValue;
}
template <typename T, int NW>
int cregs_shape(WarpShape sh) {
  UHNSW_CSHAPE_SWITCH(T, sh, NW, CREGS_CALL);
  return 0;
}

}  // namespace uhnsw_dev
