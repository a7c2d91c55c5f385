// Exhaustive L_p k-NN over the FP32 master copy: for every query, the k base
// rows with the smallest (S, id), S = sum_j |x_j - q_j|^p (the exact answer
// that recall is measured against, Section 4.1.2).
//
// Pass 1 (exact_slice_kernel): a block of 4 warps scores its slice of the rows
// in tiles of 128, WQ warps of it different queries (4 a warp) on the same
// rows, 4 / WQ groups of warps different rows of the tile.  Each lane sums RPL
// = WQ rows for the 4 queries of its warp.  A query belongs to one warp of a
// group, so the p form is a uniform branch, and the warp keeps the query's
// top-k list by itself; the groups' lists are merged at the end.  Pass 2
// (exact_merge_kernel) merges the per-slice lists.
//
// What bounds it: a general-p term costs one lg2 and one ex2, which the SFU
// issues at 16 and 32 a clock and SM (21.3 a clock for the pair): 38 ms for
// all terms of 1,001 queries on 1M x 128, and 36.1 ms measured, since a part of
// them is skipped (81.6 ms with one term at a time on tiles shared by one row a
// thread; unit vectors of 96 dimensions, where little is skipped, take 33.3 ms,
// 0.86 of the SFU rate).  The rest of a term is 1.5 paired FP32 instructions, two
// rows at a time, behind that.  Rows are staged
// transposed (row stride 132 floats: a dimension's 128 rows are one
// conflict-free 16-byte read per lane, and the transposing stores of 16 rows x 2
// chunks hit 32 banks), the next 16 dimensions in registers while the current
// ones are summed.  After every 16 dimensions a query is skipped for the rest
// of the tile once all the warp's rows have passed its k-th sum, and the tile
// ends once no query is left: sums never decrease, so no answer changes.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "coop_kernels.cuh"
#include "launch.h"

namespace uhnsw_dev {

constexpr int kExTR = 128;     // rows per tile
constexpr int kExDC = 16;      // dimensions per chunk
constexpr int kExWarps = 4;
constexpr int kExBlock = kExWarps * 32;
constexpr int kExQW = 4;       // queries per warp
constexpr int kExStride = kExTR + 4;
// Blocks per SM asked of the register allocator: 5 (102 registers) against 6
// with spills, 36.1 and 41.8 ms for 1,001 queries on 1M x 128; 4 for up to 8
// queries (one query: 0.37 against 0.55 ms).
template <int WQ>
constexpr int kExPerSm = WQ == 4 ? 5 : 4;

struct ExactSmem {
  int tile, qsm, top, buf, nk, sk, total;
  __host__ __device__ ExactSmem(int k) {
    int o = 0;
    tile = o; o += 2 * kExDC * kExStride * 4;
    qsm = o; o += 2 * kExWarps * kExQW * kExDC * 4;
    top = o; o += kExWarps * kExQW * k * 8;
    buf = o; o += kExWarps * kExTR * 8;
    nk = o; o += kExWarps * kExTR * 8;
    sk = o; o += kExWarps * (kExTR + 32) * 8;
    total = o;
  }
};

// acc + |x - q|^p for RPL rows of one dimension, rows in pairs (p = 2: the
// square is rounded before it is added).
template <int PM, int RPL>
__device__ __forceinline__ void exact_terms(float (&acc)[RPL], const float (&x)[RPL], float q,
                                            float p) {
  if constexpr (RPL == 1) {
    const float a = fabsf(x[0] - q);
    acc[0] = __fadd_rn(acc[0], PM == kPOne   ? a
                               : PM == kPTwo ? __fmul_rn(a, a)
                                             : hw_ex2(p * hw_lg2(a)));
  } else {
    const uint64_t q2 = f2_pack(q, q), p2 = f2_pack(p, p);
#pragma unroll
    for (int r = 0; r < RPL; r += 2) {
      const uint64_t d = f2_sub(f2_pack(x[r], x[r + 1]), q2);
      uint64_t s = f2_pack(acc[r], acc[r + 1]);
      float lo, hi;
      f2_unpack(d, lo, hi);
      lo = fabsf(lo);
      hi = fabsf(hi);
      if (PM == kPTwo) {
        lo = __fmul_rn(lo, lo);
        hi = __fmul_rn(hi, hi);
      } else if (PM != kPOne) {
        f2_unpack(f2_mul(f2_pack(hw_lg2(lo), hw_lg2(hi)), p2), lo, hi);
        lo = hw_ex2(lo);
        hi = hw_ex2(hi);
      }
      s = f2_add(s, f2_pack(lo, hi));
      f2_unpack(s, acc[r], acc[r + 1]);
    }
  }
}

// The first ND dimensions of a chunk (8 or 16).
template <int PM, int RPL, int ND>
__device__ __forceinline__ void exact_chunk(float (&acc)[RPL], const float* tile, const float* q,
                                            float p) {
#pragma unroll 2
  for (int j0 = 0; j0 < ND; j0 += 4) {
    const float4 qv = *reinterpret_cast<const float4*>(q + j0);
    const float qj[4] = {qv.x, qv.y, qv.z, qv.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float x[RPL];
      const float* t = tile + (j0 + j) * kExStride;
      if constexpr (RPL == 4) {
        const float4 v = *reinterpret_cast<const float4*>(t);
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
      } else if constexpr (RPL == 2) {
        const float2 v = *reinterpret_cast<const float2*>(t);
        x[0] = v.x; x[1] = v.y;
      } else {
        x[0] = *t;
      }
      exact_terms<PM, RPL>(acc, x, qj[j], p);
    }
  }
}

template <int RPL, int ND>
__device__ __forceinline__ void exact_chunk_mode(float (&acc)[RPL], const float* tile,
                                                 const float* q, float p, int pm) {
  if (pm == kPGeneral) exact_chunk<kPGeneral, RPL, ND>(acc, tile, q, p);
  else if (pm == kPOne) exact_chunk<kPOne, RPL, ND>(acc, tile, q, p);
  else exact_chunk<kPTwo, RPL, ND>(acc, tile, q, p);
}

// HALF: the rows end in the middle of their last chunk (they are padded to 8).  The
// other half is left out: half a chunk's work (3,000 queries x 30,000 x 20 1,478 ->
// 1,345 us, 4,000 x 200 950 -> 913), and terms that are 0 for p > 0 alone.
template <int WQ, bool HALF>
__global__ void __launch_bounds__(kExBlock, kExPerSm<WQ>) exact_slice_kernel(
    const float* __restrict__ base, int64_t n, int d_pad, const float* __restrict__ q, int d,
    const float* __restrict__ p, int64_t nq, int k, int64_t rows_per_slice, unsigned long long* part) {
  constexpr int RPL = WQ;                 // rows per lane
  constexpr int GROUPS = kExWarps / WQ;   // row groups of a tile
  constexpr int GR = 32 * RPL;            // rows of a group per tile
  extern __shared__ __align__(16) unsigned char smem[];
  const ExactSmem L(k);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int group = warp / WQ, wq = warp % WQ;
  float* tile = reinterpret_cast<float*>(smem + L.tile);
  float* qsm = reinterpret_cast<float*>(smem + L.qsm);
  unsigned long long* top = reinterpret_cast<unsigned long long*>(smem + L.top) + warp * kExQW * k;
  unsigned long long* buf = reinterpret_cast<unsigned long long*>(smem + L.buf) + warp * kExTR;
  unsigned long long* nk = reinterpret_cast<unsigned long long*>(smem + L.nk) + warp * kExTR;
  unsigned long long* sk = reinterpret_cast<unsigned long long*>(smem + L.sk) + warp * (kExTR + 32);
  const float kInf = __int_as_float(0x7f800000);

  const int64_t q0 = (int64_t)blockIdx.y * (WQ * kExQW);
  const int64_t slice = blockIdx.x;
  const int64_t r0 = slice * rows_per_slice;
  const int64_t r1 = min(n, r0 + rows_per_slice);
  float pq[kExQW], thr_d[kExQW];
  int pm[kExQW], thr_i[kExQW], tn[kExQW];
#pragma unroll
  for (int u = 0; u < kExQW; ++u) {
    const int64_t qi = q0 + wq * kExQW + u;
    pq[u] = qi < nq ? p[qi] : 1.0f;
    pm[u] = qi >= nq ? -1 : pq[u] == 1.0f ? kPOne : pq[u] == 2.0f ? kPTwo : kPGeneral;
    thr_d[u] = kInf;
    thr_i[u] = INT_MAX;
    tn[u] = 0;
  }
  // staging: 2 lanes take 8 dimensions of a row, a warp 16 rows at a time
  float4 xs[4];
  float xq[2];
  auto fetch = [&](int64_t t0, int c0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e = i * kExWarps + warp;  // (16-row block, half of the chunk)
      const int r = (e >> 1) * 16 + (lane >> 1), j = c0 + (e & 1) * 8 + (lane & 1) * 4;
      xs[i] = t0 + r < r1 && j < d_pad
                  ? __ldg(reinterpret_cast<const float4*>(base + (t0 + r) * d_pad + j))
                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int e = i * kExBlock + tid, qq = e / kExDC, j = c0 + e % kExDC;
      xq[i] = qq < WQ * kExQW && q0 + qq < nq && j < d ? __ldg(q + (q0 + qq) * d + j) : 0.f;
    }
  };
  auto store = [&](int b) {
    float* tb = tile + b * kExDC * kExStride;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e = i * kExWarps + warp;
      const int r = (e >> 1) * 16 + (lane >> 1), j = (e & 1) * 8 + (lane & 1) * 4;
      tb[(j + 0) * kExStride + r] = xs[i].x;
      tb[(j + 1) * kExStride + r] = xs[i].y;
      tb[(j + 2) * kExStride + r] = xs[i].z;
      tb[(j + 3) * kExStride + r] = xs[i].w;
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int e = i * kExBlock + tid;
      if (e < WQ * kExQW * kExDC) qsm[b * kExWarps * kExQW * kExDC + e] = xq[i];
    }
  };

  int b = 0;
  fetch(r0, 0);
  for (int64_t t0 = r0; t0 < r1; t0 += kExTR) {
    const int64_t my0 = t0 + group * GR;
    float acc[kExQW][RPL];
    bool live[kExQW];
#pragma unroll
    for (int u = 0; u < kExQW; ++u) {
      live[u] = pm[u] >= 0 && my0 < r1;
#pragma unroll
      for (int r = 0; r < RPL; ++r) acc[u][r] = 0.f;
    }
    for (int c0 = 0; c0 < d_pad; c0 += kExDC) {
      store(b);
      // (the buffer written two chunks ago is free: its readers passed this barrier since)
      if (!__syncthreads_or(live[0] || live[1] || live[2] || live[3])) {
        b ^= 1;
        break;
      }
      if (c0 + kExDC < d_pad) fetch(t0, c0 + kExDC);
      const float* tb = tile + b * kExDC * kExStride + group * GR + lane * RPL;
      const float* qb = qsm + (b * kExWarps + wq) * kExQW * kExDC;
#pragma unroll
      for (int u = 0; u < kExQW; ++u) {
        if (!live[u]) continue;
        const float* qu = qb + u * kExDC;
        if (HALF && c0 + kExDC > d_pad) exact_chunk_mode<RPL, kExDC / 2>(acc[u], tb, qu, pq[u], pm[u]);
        else exact_chunk_mode<RPL, kExDC>(acc[u], tb, qu, pq[u], pm[u]);
        float least = acc[u][0];
#pragma unroll
        for (int r = 1; r < RPL; ++r) least = fminf(least, acc[u][r]);
        live[u] = __any_sync(kFull, !(least > thr_d[u]));
      }
      b ^= 1;
    }
    if (t0 + kExTR < r1) fetch(t0 + kExTR, 0);
#pragma unroll
    for (int u = 0; u < kExQW; ++u) {
      if (!live[u]) continue;
      int c = 0;
#pragma unroll
      for (int r = 0; r < RPL; ++r) {
        const int64_t row = my0 + lane * RPL + r;
        const bool in = row < r1 && pair_lt(acc[u][r], (int32_t)row, thr_d[u], thr_i[u]);
        const unsigned ball = __ballot_sync(kFull, in);
        if (in) buf[c + __popc(ball & lanemask_lt())] = make_key(acc[u][r], (uint32_t)row);
        c += __popc(ball);
      }
      if (c == 0) continue;
      __syncwarp();
      int at;
      tn[u] = coop_merge(top + u * k, tn[u], k, buf, c, kNoKey, 0, nk, sk, &at);
      if (tn[u] == k) {
        const unsigned long long last = top[u * k + k - 1];
        thr_d[u] = key_dist(last);
        thr_i[u] = (int)key_id(last);
      }
      __syncwarp();
    }
  }
  if (GROUPS > 1) {
    // the groups' lists of a query into one of them: each group takes its share of
    // the queries (1,000 x 8, 60 queries, k 1: 33 us by the first group alone, 21 now)
    __shared__ int gn[kExWarps][kExQW];
#pragma unroll
    for (int u = 0; u < kExQW; ++u)
      if (lane == 0) gn[warp][u] = tn[u];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kExQW; ++u) {
      if (u % GROUPS != group) continue;
      for (int w = wq; w < kExWarps; w += WQ) {
        if (w == warp) continue;
        const unsigned long long* other =
            reinterpret_cast<unsigned long long*>(smem + L.top) + (w * kExQW + u) * k;
        for (int e = 0; e < gn[w][u]; e += kExTR) {
          int at;
          tn[u] = coop_merge(top + u * k, tn[u], k, other + e, min(kExTR, gn[w][u] - e), kNoKey, 0,
                             nk, sk, &at);
          __syncwarp();
        }
      }
    }
  }
#pragma unroll
  for (int u = 0; u < kExQW; ++u) {
    const int64_t qi = q0 + wq * kExQW + u;
    if (qi >= nq || u % GROUPS != group) continue;
    for (int j = lane; j < k; j += 32)
      part[(slice * nq + qi) * k + j] = j < tn[u] ? top[u * k + j] : kNoKey;
  }
}

// Merge of the per-slice lists of one query: survivors are the entries not
// after the smallest per-slice k-th entry; each survivor's rank among them is
// its output position.
__global__ void exact_merge_kernel(const unsigned long long* part, int nslices, int64_t nq, int k,
                                   int64_t* out_ids, float* out_dist, const float* p) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(smem);
  __shared__ int cnt;
  __shared__ unsigned long long least[32];
  const int64_t qi = blockIdx.x;
  if (qi >= nq) return;
  const int tid = threadIdx.x;
  unsigned long long bound = kNoKey;
  for (int s = tid; s < nslices; s += blockDim.x) {
    const unsigned long long x = part[((int64_t)s * nq + qi) * k + (k - 1)];
    bound = x < bound ? x : bound;
  }
  bound = warp_min_key(bound);
  if ((tid & 31) == 0) least[tid >> 5] = bound;
  if (tid == 0) cnt = 0;
  __syncthreads();
  for (int w = 0; w < (int)blockDim.x / 32; ++w) bound = least[w] < bound ? least[w] : bound;
  for (int e = tid; e < nslices * k; e += blockDim.x) {
    const int s = e / k, j = e - s * k;
    const unsigned long long x = part[((int64_t)s * nq + qi) * k + j];
    if (x != kNoKey && x <= bound) keys[atomicAdd(&cnt, 1)] = x;
  }
  __syncthreads();
  const int m = cnt;
  const double inv_p = 1.0 / (double)p[qi];
  for (int e = tid; e < m; e += blockDim.x) {
    const unsigned long long x = keys[e];
    int r = 0;
    for (int j = 0; j < m; ++j) r += keys[j] < x;
    if (r < k) {
      out_ids[qi * k + r] = key_id(x);
      out_dist[qi * k + r] = (float)pow((double)key_dist(x), inv_p);
    }
  }
  for (int j = m + tid; j < k; j += blockDim.x) {
    out_ids[qi * k + j] = -1;
    out_dist[qi * k + j] = __int_as_float(0x7f800000);
  }
}

namespace {
// Warps of a block that take different queries: 16, 8 or 4 queries per block.
// Eight for lists of up to 128 where one tile at a time would give an SM less
// than 14 blocks of 16 (a warp's merges, four queries one after the other, are then
// what takes the time): 3,000 x 32, 250 queries, k 10: 48 us with eight and 75 with
// sixteen; 1,000 x 8, 4,000 queries, k 32: 126, 148; 1,165 x 16, 2,139 queries, k
// 10: 78, 101; past it 1,500 x 60, 3,000 queries: 215, 188; k 256 on 1,000 x 8, 600
// queries: 192, 173.  Four where two blocks an SM are not reached otherwise
// (1,089 x 134, 144 queries: 74 -> 44 us; 1,083 x 146, 57 queries: 82 -> 61).
int exact_wq(int64_t n, int64_t nq, int k, int num_sms) {
  const int64_t tiles = (n + kExTR - 1) / kExTR;
  auto blocks = [&](int wq) { return tiles * ((nq + wq * kExQW - 1) / (wq * kExQW)); };
  int wq = nq > 8 ? 4 : nq > 4 ? 2 : 1;
  if (wq == 4 && blocks(4) < (k <= 128 ? 14 : 2) * (int64_t)num_sms) wq = 2;
  if (wq == 2 && blocks(2) < 2 * (int64_t)num_sms) wq = 1;
  return wq;
}
}  // namespace

int exact_workspace_slices(int64_t n, int64_t nq, int k, int num_sms) {
  const int wq = exact_wq(n, nq, k, num_sms);
  const int64_t qb = (nq + wq * kExQW - 1) / (wq * kExQW);
  const int64_t slots = (int64_t)(wq == 4 ? kExPerSm<4> : kExPerSm<1>) * num_sms;
  // as many blocks along the rows as fill whole rounds of the GPU best; more
  // rounds only where fewer leave over 4 % of it idle and a slice keeps 16 tiles:
  // every slice fills its own list, and the merge takes a list per slice (3,000 x
  // 32, 2,500 queries: k 10 4 slices 198 us, 19 slices 284; k 200 818 and 2,521)
  const int64_t tiles = (n + kExTR - 1) / kExTR;
  const int64_t cap = std::max<int64_t>(1, std::min<int64_t>(kExactMergeKeys / k, tiles));
  int64_t best = 1;
  double fill = 0.0;
  for (int64_t s = 1; s <= cap && (s * qb <= 8 * slots || s == 1); ++s) {
    const int64_t blocks = s * qb, rounds = (blocks + slots - 1) / slots;
    if (s > 1 && rounds > 1 && (tiles + s - 1) / s < 16) break;
    const double f = (double)blocks / (double)(rounds * slots);
    if (f > fill + 0.04) {
      best = s;
      fill = f;
    }
    if (s >= slots) break;
  }
  return (int)best;
}

template <int WQ>
static cudaError_t launch_slices(const float* base, int64_t n, int d, int d_pad, const float* q,
                                 const float* p, int64_t nq, int k, int nslices,
                                 unsigned long long* part, cudaStream_t st) {
  const ExactSmem L(k);
  auto kern = d_pad % kExDC ? exact_slice_kernel<WQ, true> : exact_slice_kernel<WQ, false>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L.total);
  if (e != cudaSuccess) return e;
  int64_t rows = (n + nslices - 1) / nslices;
  rows = (rows + kExTR - 1) / kExTR * kExTR;
  const dim3 grid(nslices, (unsigned)((nq + WQ * kExQW - 1) / (WQ * kExQW)));
  kern<<<grid, kExBlock, L.total, st>>>(base, n, d_pad, q, d, p, nq, k, rows, part);
  return cudaGetLastError();
}

cudaError_t launch_exact(const float* base, int64_t n, int d, int d_pad, const float* q,
                         const float* p, int64_t nq, int k, int nslices, int num_sms, void* ws,
                         int64_t* out_ids, float* out_dist, cudaStream_t st) {
  if (nslices < 1 || nslices * (int64_t)k > kExactMergeKeys) return cudaErrorInvalidValue;
  unsigned long long* part = static_cast<unsigned long long*>(ws);
  const int wq = exact_wq(n, nq, k, num_sms);
  cudaError_t e = wq == 4   ? launch_slices<4>(base, n, d, d_pad, q, p, nq, k, nslices, part, st)
                  : wq == 2 ? launch_slices<2>(base, n, d, d_pad, q, p, nq, k, nslices, part, st)
                            : launch_slices<1>(base, n, d, d_pad, q, p, nq, k, nslices, part, st);
  if (e != cudaSuccess) return e;
  const int msm = nslices * k * 8;
  if (msm > 40 * 1024) {  // (48 KB less the kernel's own arrays need no attribute)
    e = cudaFuncSetAttribute(exact_merge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, msm);
    if (e != cudaSuccess) return e;
  }
  exact_merge_kernel<<<(unsigned)nq, 128, msm, st>>>(part, nslices, nq, k, out_ids, out_dist, p);
  return cudaGetLastError();
}

}  // namespace uhnsw_dev
