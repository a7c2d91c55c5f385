// Verification-only kernel launch and the storage conversion kernel.
#include <cuda_runtime.h>

#include "launch.h"
#include "verify_kernels.cuh"

namespace uhnsw_dev {

template <int NW>
cudaError_t launch_verify_warps(const QueryArgs& a, cudaStream_t st) {
  const VerifyLayout L(a.d_pad, a.k_max, a.vcap, NW);
  auto kern = uhnsw_verify_kernel<NW>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L.total);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)a.nq, (NW + 1) * 32, L.total, st>>>(a);
  return cudaGetLastError();
}

// Warps per query, us of back-to-back calls of queries x candidates (128
// dimensions, the last column 960; Algorithm 1 with K = 10):
//               1 x 300   456 x 300   3,000 x 200   3,000 x 500   10,000 x 90   3,000 x 500   3,000 x 24
//                 exact       exact         exact         exact         exact   Algorithm 1  Algorithm 1
//   8 warps          43          50            99           169           214            78          240
//   4 warps          49          56            79           159           123            49          142
//   2 warps          66          70            75           166           119            38           93
// Eight while all queries are resident at once (3 blocks of 9 warps an SM): the
// steps of one query are then what takes the time.  Past that, two for up to
// 256 candidates between two barriers of Algorithm 1 (the exact mode has
// none): more warps find few rows to sum.  Two as well for up to 64 short
// rows: in steps of 32 or 64 none of them would be dropped.  Around the line, two
// and four warps, exact mode, 128 dimensions: 3,000 queries x 200 81 and 83 us, 256
// 95 and 94, 300 108 and 108, 512 171 and 165; 8,000 x 200 197 and 190.  From 457
// queries to about a thousand four are faster on both sides of it (600 x 200: 32 and
// 23; 960 dimensions 163 and 102).
cudaError_t launch_verify(const QueryArgs& a, int num_sms, cudaStream_t st) {
  if (a.cand_t <= 64 && a.d_pad <= 256) return launch_verify_warps<2>(a, st);
  if (a.nq <= 3 * (int64_t)num_sms) return launch_verify_warps<8>(a, st);
  int span = a.cand_t;
  if (a.mode == UHNSW_VERIFY_PAPER) span = a.kappa > a.k_max ? a.kappa : a.k_max;
  return span <= 256 ? launch_verify_warps<2>(a, st) : launch_verify_warps<4>(a, st);
}

// FP32 master rows -> FP16 / BF16 traversal rows (round to nearest even).
__global__ void convert_kernel(const float* __restrict__ src, void* dst, int dt, int64_t count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float x = src[i];
    if (dt == UHNSW_F16) reinterpret_cast<__half*>(dst)[i] = __float2half_rn(x);
    else reinterpret_cast<__nv_bfloat16*>(dst)[i] = __float2bfloat16_rn(x);
  }
}

// Counts the elements whose FP16 / BF16 copy differs from the FP32 value.
__global__ void inexact_kernel(const float* __restrict__ src, const void* dst, int dt,
                               int64_t count, unsigned long long* bad) {
  unsigned long long mine = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float back = dt == UHNSW_F16 ? __half2float(reinterpret_cast<const __half*>(dst)[i])
                                       : __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(dst)[i]);
    mine += back != src[i];
  }
  if (mine) atomicAdd(bad, mine);
}

cudaError_t launch_inexact_count(const float* src, const void* dst, uhnsw_dtype dt, int64_t count,
                                 unsigned long long* bad, cudaStream_t st) {
  int64_t blocks = (count + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  if (blocks < 1) blocks = 1;
  inexact_kernel<<<(unsigned)blocks, 256, 0, st>>>(src, dst, (int)dt, count, bad);
  return cudaGetLastError();
}

cudaError_t launch_convert(const float* src, void* dst, uhnsw_dtype dt, int64_t count,
                           cudaStream_t st) {
  int64_t blocks = (count + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  if (blocks < 1) blocks = 1;
  convert_kernel<<<(unsigned)blocks, 256, 0, st>>>(src, dst, (int)dt, count);
  return cudaGetLastError();
}

bool pick_block_shape(uhnsw_dtype dt, int chunks, WarpShape* out) {
  static const WarpShape f32[] = {{8, 1, 0},  {16, 2, 0}, {32, 2, 0},
                                  {32, 4, 0}, {32, 8, 0}, {32, 16, 0}};
  static const WarpShape f16[] = {{8, 1, 0},  {16, 1, 0}, {32, 1, 0},
                                  {32, 2, 0}, {32, 4, 0}, {32, 8, 0}};
  const WarpShape* list = dt == UHNSW_F32 ? f32 : f16;
  for (int i = 0; i < 6; ++i)
    if (list[i].team * list[i].cpl >= chunks) {
      *out = list[i];
      return true;
    }
  return false;
}

// Beam ef' of a query exactly as the search kernels derive it.
__device__ __forceinline__ int query_beam(bool direct, int k, int ef, int t) {
  int tt = direct ? k : (t > 0 ? t : ef);
  if (tt < k) tt = k;
  return max(ef, tt);
}

__device__ __forceinline__ int beam_bucket(const BeamBuckets& bb, int efp) {
  for (int b = 0; b < bb.n; ++b)
    if (efp <= bb.bound[b]) return b;
  return bb.n - 1;  // beyond every bound: the query fails validation there
}

// Code route of a query: graph slot (with the same rule as the search
// kernels' route_query) and the p form of its verification (none for a
// direct query, then p = 0.5, p = 1.5, general p).  Queries of one route run
// the same instructions, so grouping them keeps the code that the warps of an
// SM execute at the same time small.
__device__ __forceinline__ int query_route(float p, float cutoff, float gp0, float gp1) {
  const int slot = p == gp0 ? 0 : p == gp1 ? 1 : (p <= cutoff ? 0 : 1);
  const bool direct = p == (slot == 0 ? gp0 : gp1);
  const int form = direct ? 0 : p == 0.5f ? 1 : p == 1.5f ? 2 : 3;
  return slot * 4 + form;
}

__device__ __forceinline__ int query_bin(const BeamBuckets& bb, const float* p, const int32_t* k,
                                         const int32_t* ef, const int32_t* tq, int64_t i,
                                         int k_max, int ef_default, int t, float cutoff, float gp0,
                                         float gp1) {
  const bool direct = p[i] == gp0 || p[i] == gp1;
  const int b = beam_bucket(bb, query_beam(direct, k ? k[i] : k_max, ef ? ef[i] : ef_default,
                                           tq ? tq[i] : t));
  return b * kRoutes + query_route(p[i], cutoff, gp0, gp1);
}

// Counting sort of the query indices by (beam bucket, route): counts, then
// slots.  ws[0..64): counts per bin, ws[64..128): cursors; info[2b] = first
// slot of bucket b, info[2b+1] = its count.
__global__ void bucket_count_kernel(const float* p, const int32_t* k, const int32_t* ef,
                                    const int32_t* tq, int64_t nq,
                                    int k_max, int ef_default, int t, float cutoff, float gp0,
                                    float gp1, BeamBuckets bb, int32_t* ws) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nq;
       i += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&ws[query_bin(bb, p, k, ef, tq, i, k_max, ef_default, t, cutoff, gp0, gp1)], 1);
}

__global__ void bucket_scatter_kernel(const float* p, const int32_t* k, const int32_t* ef,
                                      const int32_t* tq, int64_t nq, int k_max, int ef_default, int t, float cutoff,
                                      float gp0, float gp1, BeamBuckets bb, int32_t* ws,
                                      int32_t* order, int32_t* info) {
  if (blockIdx.x == 0 && threadIdx.x < bb.n) {
    const int b = threadIdx.x;
    int first = 0, cnt = 0;
    for (int j = 0; j < b * kRoutes; ++j) first += ws[j];
    for (int j = b * kRoutes; j < (b + 1) * kRoutes; ++j) cnt += ws[j];
    info[2 * b] = first;
    info[2 * b + 1] = cnt;
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nq;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int bin = query_bin(bb, p, k, ef, tq, i, k_max, ef_default, t, cutoff, gp0, gp1);
    int base = 0;
    for (int j = 0; j < bin; ++j) base += ws[j];
    const int pos = atomicAdd(&ws[kBins + bin], 1);
    order[base + pos] = (int32_t)i;
  }
}

cudaError_t launch_bucketing(const QueryArgs& a, const BeamBuckets& bb, int32_t* ws,
                             int32_t* order, int32_t* info, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(ws, 0, 2 * kBins * sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  int64_t blocks = (a.nq + 255) / 256;
  if (blocks > 1024) blocks = 1024;
  bucket_count_kernel<<<(unsigned)blocks, 256, 0, st>>>(a.p, a.k, a.ef, a.tq, a.nq, a.k_max,
                                                         a.ef_default, a.t, a.cutoff, a.gp[0],
                                                         a.gp[1], bb, ws);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  bucket_scatter_kernel<<<(unsigned)blocks, 256, 0, st>>>(a.p, a.k, a.ef, a.tq, a.nq, a.k_max,
                                                           a.ef_default, a.t, a.cutoff, a.gp[0],
                                                           a.gp[1], bb, ws, order, info);
  return cudaGetLastError();
}

bool pick_warp_shape(uhnsw_dtype dt, int chunks, int team_pref, bool few, WarpShape* out) {
  // The first covering shape of each list is the default.  For 128-dimension
  // FP16 rows (1M x 128, p ~ U(0.5, 2], ef 52, width 2, 10,000-query batches
  // on two streams) two rows per team and round measured 8 % faster than
  // three (1.37 vs 1.49 ms per batch) and one row 6 % slower.  A batch too
  // small to fill the GPU's warps (`few`) is bound by each query's own
  // latency: there three rows per round keep more loads in flight (2,000 to
  // 3,600 queries, ef 52 at width 2 and ef 128: 0.92 to 0.98 of the time with
  // two rows; batches whose queries are all resident run the cooperative
  // kernel, which has its own number of rows).  Rows of 12 chunks (96 FP16 dimensions) take 4 lanes x 3
  // chunks, which leaves no lane on a zeroed chunk: 3.5 % faster than
  // 8 x 2 at 10M x 96, ef 512.  The shape never changes a result.
  static const WarpShape f32[] = {{8, 1, 4},  {8, 2, 2},  {16, 2, 4}, {32, 2, 2},
                                  {32, 4, 2}, {32, 8, 1}, {32, 16, 1}};
  static const WarpShape f16[] = {{8, 1, 4},  {4, 3, 2},  {8, 2, 2},  {16, 2, 2},
                                  {32, 2, 2}, {32, 4, 2}, {32, 8, 1}, {32, 16, 1}};
  static const WarpShape f16_few[] = {{8, 1, 4},  {4, 3, 2},  {8, 2, 3},  {16, 2, 2},
                                      {32, 2, 2}, {32, 4, 2}, {32, 8, 1}, {32, 16, 1}};
  const WarpShape* list = dt == UHNSW_F32 ? f32 : few ? f16_few : f16;
  const int cnt = dt == UHNSW_F32 ? (int)(sizeof(f32) / sizeof(f32[0]))
                                  : (int)(sizeof(f16) / sizeof(f16[0]));
  static_assert(sizeof(f16) == sizeof(f16_few), "the two 16-bit lists have one length");
  for (int i = 0; i < cnt; ++i)
    if (list[i].team * list[i].cpl >= chunks && (team_pref == 0 || list[i].team == team_pref)) {
      *out = list[i];
      return true;
    }
  return false;
}

cudaError_t launch_wsearch(uhnsw_dtype dt, WarpShape sh, const QueryArgs& a, int grid, size_t smem,
                           cudaStream_t st) {
  switch (dt) {
    case UHNSW_F32: return launch_wsearch_f32(sh, a, grid, smem, st);
    case UHNSW_F16: return launch_wsearch_f16(sh, a, grid, smem, st);
    case UHNSW_BF16: return launch_wsearch_bf16(sh, a, grid, smem, st);
  }
  return cudaErrorInvalidValue;
}

int wsearch_occupancy(uhnsw_dtype dt, WarpShape sh, size_t smem) {
  switch (dt) {
    case UHNSW_F32: return wocc_f32(sh, smem);
    case UHNSW_F16: return wocc_f16(sh, smem);
    case UHNSW_BF16: return wocc_bf16(sh, smem);
  }
  return 0;
}

cudaError_t launch_csearch(uhnsw_dtype dt, int warps, WarpShape sh, const QueryArgs& a, int grid,
                           size_t smem, cudaStream_t st) {
  using Fn = cudaError_t (*)(WarpShape, const QueryArgs&, int, size_t, cudaStream_t);
  static const Fn fn[3][kCoopForms] = {
      {launch_csearch_f32_w2, launch_csearch_f32_w4, launch_csearch_f32_w8},
      {launch_csearch_f16_w2, launch_csearch_f16_w4, launch_csearch_f16_w8},
      {launch_csearch_bf16_w2, launch_csearch_bf16_w4, launch_csearch_bf16_w8}};
  for (int i = 0; i < kCoopForms; ++i)
    if (kCoopWarps[i] == warps) return fn[(int)dt][i](sh, a, grid, smem, st);
  return cudaErrorInvalidValue;
}

int csearch_occupancy(uhnsw_dtype dt, int warps, WarpShape sh, size_t smem) {
  using Fn = int (*)(WarpShape);
  static const Fn fn[3][kCoopForms] = {
      {csearch_regs_f32_w2, csearch_regs_f32_w4, csearch_regs_f32_w8},
      {csearch_regs_f16_w2, csearch_regs_f16_w4, csearch_regs_f16_w8},
      {csearch_regs_bf16_w2, csearch_regs_bf16_w4, csearch_regs_bf16_w8}};
  constexpr size_t kSmSmem = 228 * 1024, kBlockReserve = 1024, kBlockMax = 227 * 1024;
  if (smem > kBlockMax) return 0;
  for (int i = 0; i < kCoopForms; ++i)
    if (kCoopWarps[i] == warps) {
      const int by_smem = (int)(kSmSmem / (smem + kBlockReserve));
      const int by_regs = fn[(int)dt][i](sh);
      return by_smem < by_regs ? by_smem : by_regs;
    }
  return 0;
}

}  // namespace uhnsw_dev
