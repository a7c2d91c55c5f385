// Verification of given candidate lists (uhnsw_verify; Algorithm 1, lines 6-10):
// one block per query, NW warps that sum candidate rows and one more that keeps
// the top-k list.
//
// The NW warps take 8 NW candidates a step, two per team of 8 lanes: a lane
// reads four 32-dimension groups of both rows before it sums any, so that the
// work on one row overlaps the loads and reductions of the other.  Meanwhile
// the merge warp folds the step before into the list, and a step is one
// barrier long; a candidate is dropped against the k-th sum of two steps ago,
// which only costs terms.  Every lane sums the same elements in the same order
// as lp_sum_team_staged (element j = 32 g + 4 lane + e), so the sums are the
// searches' bit for bit.
//
// What bounds it: the rows' bytes (768 MB for 5,003 queries x 300 candidates of
// 128 dimensions, 113 us at the measured copy rate) and, for few queries, the
// chain of steps.  One warp per query and a merge after every 8 candidates took
// 291 us for those 5,003 queries and 137 us for one: 38 steps each, in a grid
// of 1.2 times the resident warps.  Now 164 us back to back (4.7 TB/s of rows;
// 0.20 ms on a cold L2) and 43 us.
// 64 registers (1,024 threads an SM) without spills: 56 registers spill and one
// block less per SM (68 registers) hides less latency (5,003 queries, 4 warps: 165
// us, 178, 175).
#pragma once

#include "coop_kernels.cuh"

namespace uhnsw_dev {

struct VerifyLayout {
  int qs, cv, top, vk, nk, sk, total;
  __host__ __device__ VerifyLayout(int d_pad, int k_max, int vcap, int warps) {
    const int wave = warps * 8, keys = (wave + 63) / 64 * 64;
    int o = 0;
    qs = o; o += align16(d_pad * 4);
    top = o; o += align16(k_max * 8);
    vk = o; o += 2 * wave * 8;
    nk = o; o += keys * 8;
    sk = o; o += (keys + 32) * 8;
    cv = o; o += align16(vcap * 4);
    total = o;
  }
};

// L_p sums of two candidates (ids ida, idb; -1 = none) by one team of 8
// lanes.  A candidate is tested against thr after every vgroups groups and
// after its last; done = finished below thr (S = its sum), g = groups
// accumulated.  Dropped or absent candidates take no further SFU work.
template <int PM>
__device__ __forceinline__ void lp_sum_pair(const float* __restrict__ base32, int d, int d_pad,
                                            const float* qs, float p, int32_t ida, int32_t idb,
                                            float thr, unsigned tmask, int lane8, int vgroups,
                                            bool& doneA, float& SA, int& gA, bool& doneB,
                                            float& SB, int& gB) {
  const int G = (d + 31) >> 5;
  bool liveA = ida >= 0, liveB = idb >= 0;
  float accA = 0.f, accB = 0.f;
  int until_test = vgroups;
  gA = gB = 0;
  SA = SB = 0.f;
  const float* ra = base32 + (int64_t)(ida >= 0 ? ida : 0) * d_pad;
  const float* rb = base32 + (int64_t)(idb >= 0 ? idb : 0) * d_pad;
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int g0 = 0; g0 < G && (liveA || liveB); g0 += 4) {
    float4 xa[4], xb[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = (g0 + u) * 32 + lane8 * 4;
      const bool in = j < d_pad;
      xa[u] = (liveA && in) ? __ldg(reinterpret_cast<const float4*>(ra + j)) : z;
      xb[u] = (liveB && in) ? __ldg(reinterpret_cast<const float4*>(rb + j)) : z;
    }
    // (fully unrolled: no break, so that xa / xb stay in registers)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int g = g0 + u;
      if (g < G) {
        const int j = g * 32 + lane8 * 4;
        const float4 qq = j < d_pad ? *reinterpret_cast<const float4*>(qs + j) : z;
        if (liveA) {
          accA = add_terms4<PM>(accA, xa[u], qq, p);
          gA = g + 1;
        }
        if (liveB) {
          accB = add_terms4<PM>(accB, xb[u], qq, p);
          gB = g + 1;
        }
        if (--until_test == 0 || g + 1 == G) {
          until_test = vgroups;
          float ta = accA, tb = accB;
          ta += __shfl_xor_sync(tmask, ta, 1);
          tb += __shfl_xor_sync(tmask, tb, 1);
          ta += __shfl_xor_sync(tmask, ta, 2);
          tb += __shfl_xor_sync(tmask, tb, 2);
          ta += __shfl_xor_sync(tmask, ta, 4);
          tb += __shfl_xor_sync(tmask, tb, 4);
          if (liveA) {
            if (ta > thr) liveA = false;
            else SA = ta;
          }
          if (liveB) {
            if (tb > thr) liveB = false;
            else SB = tb;
          }
        }
      }
    }
  }
  doneA = liveA;
  doneB = liveB;
}

// What the warps of a block share besides the layout's arrays.  Steps are
// numbered through all ranges of a query; step s writes thr[s & 1].
struct VerifyShared {
  float thr[2];  // k-th sum as of the merge in that step (+inf: list not full)
  int tn;        // length of the list
  int stop;      // Algorithm 1: the overlap test passed
  int terms;
  int valid[2][12];  // valid candidates of each warp's share
};

// Verifies the candidates C[i0 .. i1) (none dropped with no_drop) and folds
// them into top[0 .. tn), a list of at most k (the merge warp's tn is the
// one that counts).  `step` numbers the barriers.
template <int PM, int NW>
__device__ __forceinline__ void verify_range(const QueryArgs& a, const float* qs, float p,
                                             const uint32_t* C, int i0, int i1, int k,
                                             bool no_drop, unsigned long long* top, int& tn,
                                             unsigned long long* vk, unsigned long long* nk,
                                             unsigned long long* sk, VerifyShared& sh, int& step,
                                             int& terms) {
  constexpr int WAVE = NW * 8;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float kInf = __int_as_float(0x7f800000);
  const int steps = (i1 - i0 + WAVE - 1) / WAVE + 1;  // the last one only merges
  for (int s = 0; s < steps; ++s) {
    if (warp == NW) {
      if (s > 0) {
        int at;
        tn = coop_merge(top, tn, k, vk + ((step + 1) & 1) * WAVE, WAVE,
                        tn == k ? top[k - 1] : kNoKey, 0, nk, sk, &at);
      }
      if (lane == 0) sh.thr[step & 1] = tn == k ? key_dist(top[k - 1]) : kInf;
    } else if (s + 1 < steps) {
      const int team = lane >> 3, lane8 = lane & 7;
      const unsigned tmask = 0xffu << (team * 8);
      const float thr = no_drop ? kInf : sh.thr[(step + 1) & 1];
      // neighbouring teams of all warps take neighbouring candidates first
      const int ia = i0 + s * WAVE + warp * 4 + team, ib = ia + NW * 4;
      const int32_t ida = ia < i1 ? (int32_t)chk_idx((int64_t)C[ia], a.n, 2, a.err) : -1;
      const int32_t idb = ib < i1 ? (int32_t)chk_idx((int64_t)C[ib], a.n, 2, a.err) : -1;
      bool dA, dB;
      float SA, SB;
      int gA, gB;
      lp_sum_pair<PM>(a.base32, a.d, a.d_pad, qs, p, ida, idb, thr, tmask, lane8, a.vgroups, dA,
                      SA, gA, dB, SB, gB);
      if (lane8 == 0) {
        unsigned long long* o = vk + (step & 1) * WAVE + warp * 4 + team;
        o[0] = dA ? make_key(SA, (uint32_t)ida) : kNoKey;
        o[NW * 4] = dB ? make_key(SB, (uint32_t)idb) : kNoKey;
        terms += min(gA * 32, a.d) + min(gB * 32, a.d);
      }
    }
    __syncthreads();
    ++step;
  }
}

// Exact mode takes all of C as one range, Algorithm 1 the first K, then batches
// of kappa until the overlap test passes.  Returns the number of candidates
// verified.
template <int PM, int NW>
__device__ __forceinline__ int verify_run(const QueryArgs& a, const float* qs, float p,
                                          const uint32_t* C, int t, int k,
                                          unsigned long long* top, unsigned long long* vk,
                                          unsigned long long* nk, unsigned long long* sk,
                                          VerifyShared& sh, int& terms) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool paper = a.mode == UHNSW_VERIFY_PAPER;
  const int kappa = a.kappa > 0 ? a.kappa : k;
  int tn = 0, step = 0, i = 0;
  while (i < t) {
    const int bend = !paper ? t : i == 0 ? min(k, t) : (int)min((int64_t)i + kappa, (int64_t)t);
    const bool batch = i > 0;
    if (batch && warp == NW) {
      for (int j = lane; j < tn; j += 32) top[j] |= 1ull;  // mark R
      __syncwarp();
    }
    verify_range<PM, NW>(a, qs, p, C, i, bend, k, paper && !batch, top, tn, vk, nk, sk, sh, step,
                         terms);
    i = bend;
    if (batch) {
      if (warp == NW) {
        int ov = 0;
        for (int j = lane; j < tn; j += 32) {
          ov += (int)(top[j] & 1ull);
          top[j] &= ~1ull;
        }
        ov = (int)__reduce_add_sync(kFull, (unsigned)ov);
        if (lane == 0) sh.stop = (float)ov / (float)k >= a.tau;
        __syncwarp();
      }
      __syncthreads();
      if (sh.stop) break;
    }
  }
  if (warp == NW && lane == 0) sh.tn = tn;
  return i;
}

template <int NW>
__global__ void __launch_bounds__((NW + 1) * 32, 1024 / ((NW + 1) * 32)) uhnsw_verify_kernel(const QueryArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ VerifyShared sh;
  constexpr int THREADS = (NW + 1) * 32;
  const VerifyLayout L(a.d_pad, a.k_max, a.vcap, NW);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if ((uint32_t)L.total > dynamic_smem_bytes()) {
    if (tid == 0) set_error(a.err, UHNSW_ECAPACITY);
    return;
  }
  const int64_t qi = blockIdx.x;
  const float p = a.p[qi];
  const int k = a.k_max;
  if (!(p > 0.f) || !(p <= 2.f)) {
    coop_invalid<NW>(a, qi);
    return;
  }
  float* qs = reinterpret_cast<float*>(smem + L.qs);
  uint32_t* cv = reinterpret_cast<uint32_t*>(smem + L.cv);
  unsigned long long* top = reinterpret_cast<unsigned long long*>(smem + L.top);
  const float kInf = __int_as_float(0x7f800000);
  for (int j = tid; j < a.d_pad; j += THREADS) qs[j] = j < a.d ? a.q[qi * a.d + j] : 0.f;
  if (tid == 0) {
    sh.thr[1] = kInf;  // what step 0 reads
    sh.terms = 0;
  }
  // the valid candidate slots, in order
  int tv = 0;
  const int32_t* row = a.cand + qi * a.cand_t;
  for (int b0 = 0, h = 0; b0 < a.cand_t; b0 += THREADS, h ^= 1) {
    const int j = b0 + tid;
    const int32_t c = j < a.cand_t ? row[j] : -1;
    const bool keep = c >= 0 && c < a.n;
    const unsigned ball = __ballot_sync(kFull, keep);
    if (lane == 0) sh.valid[h][warp] = __popc(ball);
    __syncthreads();
    const int cnt = lane <= NW ? sh.valid[h][lane] : 0;
    const int before = (int)__reduce_add_sync(kFull, lane < warp ? (unsigned)cnt : 0u);
    if (keep)
      cv[chk_idx(tv + before + __popc(ball & lanemask_lt()), a.vcap, 6, a.err)] = (uint32_t)c;
    tv += (int)__reduce_add_sync(kFull, (unsigned)cnt);
  }
  __syncthreads();
  unsigned long long* vk = reinterpret_cast<unsigned long long*>(smem + L.vk);
  unsigned long long* nk = reinterpret_cast<unsigned long long*>(smem + L.nk);
  unsigned long long* sk = reinterpret_cast<unsigned long long*>(smem + L.sk);
  int np, terms = 0;
  switch (pmode_of(p)) {
    case kPOne: np = verify_run<kPOne, NW>(a, qs, p, cv, tv, k, top, vk, nk, sk, sh, terms); break;
    case kPTwo: np = verify_run<kPTwo, NW>(a, qs, p, cv, tv, k, top, vk, nk, sk, sh, terms); break;
    case kPHalf: np = verify_run<kPHalf, NW>(a, qs, p, cv, tv, k, top, vk, nk, sk, sh, terms); break;
    case kPThreeHalves:
      np = verify_run<kPThreeHalves, NW>(a, qs, p, cv, tv, k, top, vk, nk, sk, sh, terms);
      break;
    default: np = verify_run<kPGeneral, NW>(a, qs, p, cv, tv, k, top, vk, nk, sk, sh, terms); break;
  }
  __syncthreads();
  const int tn = sh.tn;
  for (int j = tid; j < k; j += THREADS) {
    const bool have = j < tn;
    a.out_ids[qi * k + j] = have ? (int64_t)key_id(top[j]) : -1;
    a.out_dist[qi * k + j] = have ? root_p(key_dist(top[j]), p) : kInf;
  }
  if (a.stats) {
    if (terms) atomicAdd(&sh.terms, terms);
    __syncthreads();
    if (tid == 0) put_stats(a, qi, 0, np, sh.terms, 0, 0, 0, 0, 0);
  }
}

}  // namespace uhnsw_dev
