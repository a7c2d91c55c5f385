// Host-side launch interfaces of the device code (one translation unit per
// storage type keeps the build parallel).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "warp_kernels.cuh"

namespace uhnsw_dev {

// Warp-per-query kernel: TEAM lanes per row, CPL 16-byte chunks per lane,
// U rows per team loaded per round; kWarpsPerBlock warps (queries) per block.
struct WarpShape {
  int team, cpl, u;
  bool most = false;  // warp kernel: the form for 32 warps per SM, not 24; cooperative
                      // kernel: the form for more queries than are resident
};
constexpr int kWarpsPerBlock = 2;
// The warp kernel's team shape for rows of `chunks` 16-byte chunks.
// team_pref 0: the narrowest compiled team that covers the row; else the
// first covering shape with exactly that many lanes.  `few`: the batch has
// fewer queries than the GPU has warp slots (kWarpSlots per SM).
bool pick_warp_shape(uhnsw_dtype dt, int chunks, int team_pref, bool few, WarpShape* out);
cudaError_t launch_wsearch(uhnsw_dtype dt, WarpShape sh, const QueryArgs& a, int grid,
                           size_t smem, cudaStream_t st);
int wsearch_occupancy(uhnsw_dtype dt, WarpShape sh, size_t smem);

// Launches a search kernel; one that follows another of its chain (a.chain) may
// start before that one's end.
template <typename K>
cudaError_t launch_search_kernel(K kern, int grid, int threads, size_t smem, const QueryArgs& a,
                                 cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute early = {};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &early;
  cfg.numAttrs = (a.chain & 2) ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

// Cooperative kernel (coop_kernels.cuh): one query per block, kCoopWarps[i]
// distance warps and one merge warp.
constexpr int kCoopForms = 3;
constexpr int kCoopWarps[kCoopForms] = {2, 4, 8};
// The block-per-query form's team shape where the caller asks for that form:
// the first compiled shape that covers rows of `chunks` 16-byte chunks (false:
// none does).
bool pick_block_shape(uhnsw_dtype dt, int chunks, WarpShape* out);
cudaError_t launch_csearch(uhnsw_dtype dt, int warps, WarpShape sh, const QueryArgs& a, int grid,
                           size_t smem, cudaStream_t st);
// Resident blocks per SM with `smem` bytes of shared memory per block (0: does
// not fit).
int csearch_occupancy(uhnsw_dtype dt, int warps, WarpShape sh, size_t smem);

// Verification only (verify_kernels.cuh): one block per query.
cudaError_t launch_verify(const QueryArgs& a, int num_sms, cudaStream_t st);

// Beam buckets of a bucketed persistent search (ascending bounds).
struct BeamBuckets {
  int n;
  int bound[8];
};
// Query routes (graph x verification p form) and sort bins (bucket x route).
constexpr int kRoutes = 8;
constexpr int kBins = 8 * kRoutes;
// Bucket scratch: ws[2 kBins] counts and cursors, then info[16], then the order.
constexpr int kBucketInfo = 2 * kBins;
constexpr int kBucketOrder = kBucketInfo + 16;
// Groups the query indices by beam bucket, and by route inside a bucket, into
// `order` and writes {first slot, count} per bucket into info[2b], info[2b+1].
cudaError_t launch_bucketing(const QueryArgs& a, const BeamBuckets& bb, int32_t* ws,
                             int32_t* order, int32_t* info, cudaStream_t st);

cudaError_t launch_convert(const float* src, void* dst, uhnsw_dtype dt, int64_t count,
                           cudaStream_t st);
cudaError_t launch_inexact_count(const float* src, const void* dst, uhnsw_dtype dt, int64_t count,
                                 unsigned long long* bad, cudaStream_t st);

// Idealized-recall curves (idealized.cu).
cudaError_t launch_base_p(const float* p, int64_t nq, float gp0, float gp1, float cutoff,
                          float* out, cudaStream_t st);
cudaError_t launch_recall_curve(const int64_t* ids_k, const int64_t* ids_t, int64_t nq, int K,
                                int T, int32_t* counts, cudaStream_t st);
// Exhaustive search: ws holds nslices x nq x k 8-byte keys.  nslices is at most
// exact_workspace_slices of the same k; more than kExactMergeKeys / k are refused
// (cudaErrorInvalidValue): the merge holds a query's keys in shared memory.
constexpr int kExactMergeKeys = 8192;
int exact_workspace_slices(int64_t n, int64_t nq, int k, int num_sms);
cudaError_t launch_exact(const float* base, int64_t n, int d, int d_pad, const float* q,
                         const float* p, int64_t nq, int k, int nslices, int num_sms, void* ws,
                         int64_t* out_ids, float* out_dist, cudaStream_t st);

// per-storage-type entry points (defined in wsearch_<type>.cu and csearch_<type>_w<warps>.cu)
cudaError_t launch_wsearch_f32(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                               cudaStream_t st);
int wocc_f32(WarpShape sh, size_t smem);
cudaError_t launch_csearch_f32_w2(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st);
int csearch_regs_f32_w2(WarpShape sh);
cudaError_t launch_csearch_f32_w4(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st);
int csearch_regs_f32_w4(WarpShape sh);
cudaError_t launch_csearch_f32_w8(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st);
int csearch_regs_f32_w8(WarpShape sh);
cudaError_t launch_wsearch_f16(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                               cudaStream_t st);
int wocc_f16(WarpShape sh, size_t smem);
cudaError_t launch_csearch_f16_w2(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st);
int csearch_regs_f16_w2(WarpShape sh);
cudaError_t launch_csearch_f16_w4(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st);
int csearch_regs_f16_w4(WarpShape sh);
cudaError_t launch_csearch_f16_w8(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st);
int csearch_regs_f16_w8(WarpShape sh);
cudaError_t launch_wsearch_bf16(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                               cudaStream_t st);
int wocc_bf16(WarpShape sh, size_t smem);
cudaError_t launch_csearch_bf16_w2(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st);
int csearch_regs_bf16_w2(WarpShape sh);
cudaError_t launch_csearch_bf16_w4(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st);
int csearch_regs_bf16_w4(WarpShape sh);
cudaError_t launch_csearch_bf16_w8(WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                                 cudaStream_t st);
int csearch_regs_bf16_w8(WarpShape sh);

}  // namespace uhnsw_dev
