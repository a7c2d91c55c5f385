// HNSW construction on the GPU (the index construction behind Section 2.2's
// graphs: G1 under L1, G2 under L2, G0.5 under the L0.5 sum of U-HNSW-E, and
// the L1.5 graph of a fixed-p comparison).
//
// The published HNSW insertion, applied to batches of nodes at once:
//   - nodes are inserted in id order; node 0 is the first entry point;
//   - a batch [s, e) searches the graph of nodes [0, s): a block per new
//     node runs the greedy descent (beam 1) above the node's level, then at
//     each level from min(top, level) down to 0 a beam search of width
//     efConstruction whose entry set is the whole result of the level above,
//     and keeps at most M links chosen by the neighbour heuristic (a
//     candidate is kept only if strictly nearer to the new node than to every
//     link already kept);
//   - the reverse links go to a per-row incoming buffer; after the batch, a
//     block per touched row appends them, or, past the row's cap (2M at layer
//     0, M above), re-selects the row with the heuristic over its old links
//     and the incoming ones, ordered by (distance, id);
//   - the entry point moves to the first node of a new top level.
// Nodes of one batch do not link to each other directly; batches grow with
// the graph (1/16 of the nodes already inserted, at most 65,536), so that a
// node's batch is a small part of the graph it searches.  Results depend on
// the batch schedule, not on thread timing: the incoming links of a row are
// sorted before they are used, so the graph is the same on every run.
//
// Layout on the device: FP32 rows [n][d_pad]; layer 0 as [n][2M] int32 and
// the upper levels as [rows][M] int32 with the row of (v, level l) at
// up_off[v] + l - 1 (the search index's layout), -1 padded.  Every loop is
// bounded; an index or capacity problem sets an error word that the host
// reads at the end.

#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <new>
#include <vector>

#include "uhnsw.h"
#include "uhnsw_internal.h"
#include "coop_kernels.cuh"

namespace uhnsw_dev {
namespace {

constexpr int kBuildWarps = 4;   // warps per block of the reverse-link kernel
constexpr int kInCap = 128;      // incoming links buffered per row and batch

struct BuildArgs {
  const float* X;          // [n][d_pad]
  const int32_t* lv;       // [n] levels
  const int32_t* up_off;   // [n] first upper row of the node, -1 if none
  const int32_t* up_owner; // [rows] node of each upper row
  int32_t* ell0;           // [n][M0]
  int32_t* up_adj;         // [rows][M]
  int32_t* inc_cnt;        // [n + rows] incoming links of this batch
  int32_t* inc;            // [n + rows][kInCap]
  int32_t* touched;        // rows with incoming links, then their count at touched_n
  int32_t* touched_n;
  int32_t* err;            // [0] error code, [1] dropped incoming links
  int64_t n, rows;
  int32_t d_pad, metric, M, M0, efc;
  float bp;                // the p of metric 5
};

__device__ __forceinline__ const int32_t* adj_row(const BuildArgs& a, int32_t v, int l, int* deg) {
  if (l == 0) {
    *deg = a.M0;
    return a.ell0 + chk_idx(v, a.n, 23, a.err) * a.M0;
  }
  *deg = a.M;
  const int32_t r = a.up_off[chk_idx(v, a.n, 24, a.err)];
  if (r < 0) {
    *deg = 0;
    return a.up_adj;
  }
  return a.up_adj + chk_idx((int64_t)r + l - 1, a.rows, 25, a.err) * a.M;
}

// Queues the reverse link (row r <- u) for the batch's second phase.
__device__ __forceinline__ void push_incoming(const BuildArgs& a, int64_t r, int32_t u) {
  const int pos = atomicAdd(&a.inc_cnt[r], 1);
  if (pos == 0) {
    const int t = atomicAdd(a.touched_n, 1);
    a.touched[chk_idx(t, a.n + a.rows, 26, a.err)] = (int32_t)r;
  }
  if (pos < kInCap) a.inc[r * kInCap + pos] = u;
  else atomicAdd(&a.err[1], 1);  // dropped: the row had more incoming links than the buffer
}

// Phase 1 of a batch: one block of NW + 1 warps per new node, with the step of
// the cooperative search (coop_kernels.cuh): NW warps sum the rows of a step,
// the last merges W, and every warp picks the next parent.  An insertion is a
// chain of about efConstruction such steps, and the schedule runs about 150
// batches one after the other for 50,000 nodes, so the chain is what bounds
// the build.  Eight, four or two distance warps are taken by the size of the
// batch, the most with which all its nodes are resident at once; two past that
// (one warp per node, without the step's overlap, took 1.5 times as long at
// 1M x 128 and 2.1 times at 60k x 960).  Rows are summed by teams of 8 lanes,
// 4 elements a lane and group of 32, two rows at a time.

// acc + the base-metric terms of four elements, added in order.
template <int METRIC>
__device__ __forceinline__ float build_terms(float acc, const float4& x, const float4& y, float bp) {
  const float t[4] = {x.x - y.x, x.y - y.y, x.z - y.z, x.w - y.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float v = fabsf(t[e]);
    if (METRIC == UHNSW_BASE_L1) acc = __fadd_rn(acc, v);
    else if (METRIC == UHNSW_BASE_L05) acc = __fadd_rn(acc, sqrtf(v));
    else if (METRIC == UHNSW_BASE_L15) acc = fmaf(v, sqrtf(v), acc);
    else if (METRIC == UHNSW_BASE_LP) acc = __fadd_rn(acc, __powf(v, bp));
    else acc = fmaf(v, v, acc);
  }
  return acc;
}

// Sums of rows ra and rb against y (shared or global) by a team of 8 lanes,
// four 32-element groups of both rows loaded before they are summed.
template <int METRIC>
__device__ __forceinline__ void build_dist2(const float* __restrict__ ra,
                                            const float* __restrict__ rb, const float* y, int d_pad,
                                            int lt, float bp, float& sa, float& sb) {
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  sa = sb = 0.f;
  for (int j0 = lt * 4; j0 < d_pad; j0 += 128) {
    float4 xa[4], xb[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int j = j0 + 32 * g;
      xa[g] = j < d_pad ? __ldg(reinterpret_cast<const float4*>(ra + j)) : z;
      xb[g] = j < d_pad ? __ldg(reinterpret_cast<const float4*>(rb + j)) : z;
    }
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int j = j0 + 32 * g;
      if (j < d_pad) {
        const float4 yy = *reinterpret_cast<const float4*>(y + j);
        sa = build_terms<METRIC>(sa, xa[g], yy, bp);
        sb = build_terms<METRIC>(sb, xb[g], yy, bp);
      }
    }
  }
#pragma unroll
  for (int off = 1; off < 8; off <<= 1) {
    sa += __shfl_xor_sync(kFull, sa, off);
    sb += __shfl_xor_sync(kFull, sb, off);
  }
}
__device__ __forceinline__ void build_dist2_metric(int metric, const float* ra, const float* rb,
                                                   const float* y, int d_pad, int lt, float bp,
                                                   float& sa, float& sb) {
  switch (metric) {
    case UHNSW_BASE_L1: build_dist2<1>(ra, rb, y, d_pad, lt, bp, sa, sb); break;
    case UHNSW_BASE_L2: build_dist2<2>(ra, rb, y, d_pad, lt, bp, sa, sb); break;
    case UHNSW_BASE_L05: build_dist2<3>(ra, rb, y, d_pad, lt, bp, sa, sb); break;
    case UHNSW_BASE_L15: build_dist2<4>(ra, rb, y, d_pad, lt, bp, sa, sb); break;
    default: build_dist2<5>(ra, rb, y, d_pad, lt, bp, sa, sb); break;
  }
}

// Neighbour heuristic by a block of G warps over the ascending candidates
// W[0 .. nw): a candidate is kept only if its distance to the base point is
// below its distance to every candidate already kept; at most m kept.  G
// candidates at a time: each warp checks one against those kept so far, and
// the survivors are taken in order, each first checked against those just
// taken.  Lane j of every warp ends with kept[i] = the (32 i + j)-th; returns
// their number.  state: [2][G] shared ints.
template <int G, int KC>
__device__ __forceinline__ int block_select(const BuildArgs& a, const unsigned long long* W, int nw,
                                            int m, uint32_t (&kept)[KC], int32_t* state) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, team = lane >> 3, lt = lane & 7;
  auto kept_row = [&](int j) {
    uint32_t v = __shfl_sync(kFull, kept[0], j & 31);
#pragma unroll
    for (int c = 1; c < KC; ++c) {
      const uint32_t w = __shfl_sync(kFull, kept[c], j & 31);
      if (j >> 5 == c) v = w;
    }
    return a.X + chk_idx(v, a.n, 22, a.err) * a.d_pad;
  };
  int r = 0, ph = 0;
  for (int i0 = 0; i0 < nw && r < m; i0 += G) {
    const int i = i0 + warp;
    const unsigned long long x = i < nw ? W[i] : kNoKey;
    const float dc = key_dist(x);
    const float* xc = a.X + chk_idx(i < nw ? key_id(x) : 0, a.n, 21, a.err) * a.d_pad;
    bool keep = i < nw;
    for (int j0 = 0; j0 < r && keep; j0 += 8) {
      const float* ra = kept_row(min(j0 + team, r - 1));
      const float* rb = kept_row(min(j0 + 4 + team, r - 1));
      float sa, sb;
      build_dist2_metric(a.metric, ra, rb, xc, a.d_pad, lt, a.bp, sa, sb);
      keep = !__any_sync(kFull, !(dc < sa) || !(dc < sb));
    }
    if (lane == 0) state[ph * G + warp] = keep;
    __syncthreads();
    unsigned mask = __ballot_sync(kFull, lane < G && state[ph * G + min(lane, G - 1)] != 0);
    ph ^= 1;
    while (mask && r < m) {
      const uint32_t id = key_id(W[i0 + __ffs(mask) - 1]);
#pragma unroll
      for (int c = 0; c < KC; ++c)
        if (r == 32 * c + lane) kept[c] = id;
      ++r;
      mask &= mask - 1;
      if (!mask || r >= m) break;
      bool still = (mask >> warp) & 1u;
      if (still) {
        const float* xs = a.X + chk_idx(id, a.n, 22, a.err) * a.d_pad;
        float sa, sb;
        build_dist2_metric(a.metric, xs, xs, xc, a.d_pad, lt, a.bp, sa, sb);
        still = dc < sa;
      }
      if (lane == 0) state[ph * G + warp] = still;
      __syncthreads();
      mask = __ballot_sync(kFull, lane < G && state[ph * G + min(lane, G - 1)] != 0);
      ph ^= 1;
    }
  }
  return r;
}

struct BuildInsertLayout {
  int qv, W, tab, ck0, ck1, nk, sk, wl, cnt, pub, total;
  __host__ __device__ BuildInsertLayout(int d_pad, int efc, int hb, int slots, int warps) {
    const int keys = (slots + 63) / 64 * 64;
    int o = 0;
    qv = o; o += align16(d_pad * 4);
    W = o; o += align16(efc * 8);
    tab = o; o += (1 << hb) * 4;
    ck0 = o; o += keys * 8;
    ck1 = o; o += keys * 8;
    nk = o; o += keys * 8;
    sk = o; o += (keys + 32) * 8;
    wl = o; o += warps * 32 * 4;
    cnt = o; o += align16(2 * warps * 4);
    pub = o; o += 2 * (int)sizeof(CoopPub);
    total = o;
  }
};

template <int NW>
__global__ void __launch_bounds__((NW + 1) * 32, (NW >= 8 ? 1 : NW >= 4 ? 4 : 7))
    build_insert_kernel(const BuildArgs a, int64_t s, int32_t ep, int32_t top, int hb) {
  constexpr int THREADS = (NW + 1) * 32;
  extern __shared__ __align__(16) unsigned char smem[];
  const int spw = (a.M0 + NW - 1) / NW, total = spw * NW, keys = (total + 63) / 64 * 64;
  const BuildInsertLayout L(a.d_pad, a.efc, hb, total, NW + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int team = lane >> 3, lt = lane & 7;
  const bool merger = warp == NW;
  float* qv = reinterpret_cast<float*>(smem + L.qv);
  unsigned long long* W = reinterpret_cast<unsigned long long*>(smem + L.W);
  int32_t* tab = reinterpret_cast<int32_t*>(smem + L.tab);
  unsigned long long* nk = reinterpret_cast<unsigned long long*>(smem + L.nk);
  unsigned long long* sk = reinterpret_cast<unsigned long long*>(smem + L.sk);
  uint32_t* wl = reinterpret_cast<uint32_t*>(smem + L.wl) + warp * 32;
  int32_t* fresh_of = reinterpret_cast<int32_t*>(smem + L.cnt);
  CoopPub* pub = reinterpret_cast<CoopPub*>(smem + L.pub);
  auto ckbuf = [&](int i) {
    return reinterpret_cast<unsigned long long*>(smem + (i ? L.ck1 : L.ck0));
  };
  const int64_t u = s + blockIdx.x;
  const int H = 1 << hb;
  for (int j = tid; j < a.d_pad; j += THREADS) qv[j] = a.X[u * a.d_pad + j];
  for (int j = tid; j < 2 * keys; j += THREADS)
    ckbuf(j >= keys)[j >= keys ? j - keys : j] = kNoKey;
  __syncthreads();

  // this warp's slots [b, b + 32) of a step (lane i: link v, -1: none), those
  // not seen at this level summed into out, the others emptied
  auto sum_slots = [&](int b, int32_t v, bool filter, unsigned long long* out) {
    const int cnt = min(32, spw - b);
    unsigned long long* o = out + warp * spw + b;
    const bool fresh = v >= 0 && v < a.n && (!filter || hash_insert(tab, hb, v, a.err));
    const unsigned mask = __ballot_sync(kFull, fresh);
    const int nf = __popc(mask);
    if (fresh) wl[__popc(mask & lanemask_lt())] = (uint32_t)v;
    if (lane >= nf && lane < cnt) o[lane] = kNoKey;
    __syncwarp();
    for (int i0 = 0; i0 < nf; i0 += 8) {
      const int ia = i0 + team, ib = ia + 4;
      const uint32_t da = wl[min(ia, nf - 1)], db = wl[min(ib, nf - 1)];
      float sa, sb;
      build_dist2_metric(a.metric, a.X + chk_idx(da, a.n, 20, a.err) * a.d_pad,
                         a.X + chk_idx(db, a.n, 20, a.err) * a.d_pad, qv, a.d_pad, lt, a.bp, sa,
                         sb);
      if (lt == 0 && ia < nf) o[ia] = make_key(sa, da);
      if (lt == 0 && ib < nf) o[ib] = make_key(sb, db);
    }
    __syncwarp();
    return nf;
  };
  // one step's share of this warp: the links of node v at level l
  auto expand = [&](int32_t v, int l, bool filter, unsigned long long* out) {
    int deg = 0;
    const int32_t* row = adj_row(a, v, l, &deg);
    int nf = 0;
    for (int b = 0; b < spw; b += 32) {
      const int f = warp * spw + b + lane;
      nf += sum_slots(b, b + lane < spw && f < deg ? row[f] : -1, filter, out);
    }
    return nf;
  };

  // beam 1 down to the node's own level
  int ph = 0;
  if (warp == 0) sum_slots(0, lane == 0 ? ep : -1, false, ckbuf(0));
  __syncthreads();
  unsigned long long curk = ckbuf(0)[0];
  const int lu = a.lv[u];
  const int64_t max_steps = ((int64_t)top + 1) * (a.n + 16);
  int64_t step = 0;
  for (int l = top; l > lu; ++step) {
    if (step >= max_steps) {  // (never: every step is nearer, or a level lower)
      if (tid == 0) set_error(a.err, UHNSW_ECAPACITY);
      break;
    }
    ph ^= 1;
    if (!merger) expand((int32_t)key_id(curk), l, false, ckbuf(ph));
    __syncthreads();
    unsigned long long mn = kNoKey;
    for (int b = lane; b < total; b += 32) mn = ckbuf(ph)[b] < mn ? ckbuf(ph)[b] : mn;
    mn = warp_min_key(mn);
    if (mn < curk) curk = mn;
    else --l;
  }
  if (tid == 0) W[0] = curk;
  int nw = 1;
  for (int l = min(top, lu); l >= 0; --l) {
    // SEARCH-LAYER of width efConstruction from the entry set W
    __syncthreads();
    for (int j = tid; j < H / 4; j += THREADS)
      reinterpret_cast<int4*>(tab)[j] = make_int4(kEmpty, kEmpty, kEmpty, kEmpty);
    for (int j = tid; j < 2 * keys; j += THREADS)
      ckbuf(j >= keys)[j >= keys ? j - keys : j] = kNoKey;
    __syncthreads();
    for (int j = tid; j < nw; j += THREADS) hash_insert(tab, hb, (int32_t)key_id(W[j]), a.err);
    if (merger) {
      if (lane == 0) {
        pub[0].uk[0] = W[0];
        pub[0].pos[0] = 0;
        pub[0].bn = nw;
        pub[0].last = kNoKey;
      }
      __syncwarp();
      coop_merge_step(W, a.efc, 1, ckbuf(0), 0, &pub[0], &pub[1], 0, 0, nk, sk);
    }
    __syncthreads();
    ph = 1;
    int hcount = nw, nWp = 0, jn = 0;
    uint32_t par = 0;
    int npar = coop_select(ckbuf(ph), total, &pub[ph], 1, a.efc, nWp, jn, par);
    for (int64_t st = 0; npar > 0; ++st) {
      if (st >= a.n + 16) {
        if (tid == 0) set_error(a.err, UHNSW_ECAPACITY);
        break;
      }
      if (merger)
        coop_merge_step(W, a.efc, 1, ckbuf(ph), total, &pub[ph], &pub[ph ^ 1], nWp, jn, nk, sk);
      if (hcount > (H >> 1)) {
        __syncthreads();
        hcount = pub[ph ^ 1].bn;
        for (int j = tid; j < H / 4; j += THREADS)
          reinterpret_cast<int4*>(tab)[j] = make_int4(kEmpty, kEmpty, kEmpty, kEmpty);
        __syncthreads();
        for (int j = tid; j < hcount; j += THREADS)
          hash_insert(tab, hb, (int32_t)key_id(W[j]), a.err);
        __syncthreads();
      }
      if (!merger) {
        const int nf = expand((int32_t)__shfl_sync(kFull, par, 0), l, true, ckbuf(ph ^ 1));
        if (lane == 0) fresh_of[(ph ^ 1) * NW + warp] = nf;
      }
      __syncthreads();
      ph ^= 1;
      hcount += (int)__reduce_add_sync(kFull, lane < NW ? (unsigned)fresh_of[ph * NW + lane] : 0u);
      npar = coop_select(ckbuf(ph), total, &pub[ph], 1, a.efc, nWp, jn, par);
    }
    nw = pub[ph].bn;
    for (int j = tid; j < nw; j += THREADS) W[j] &= ~1ull;
    __syncthreads();

    uint32_t kept[2] = {0, 0};
    const int r = block_select<NW + 1, 2>(a, W, nw, a.M, kept, reinterpret_cast<int32_t*>(nk));
    int deg = 0;
    int32_t* row = const_cast<int32_t*>(adj_row(a, (int32_t)u, l, &deg));
    if (warp == 0) {
      for (int j = lane; j < deg; j += 32) {
        const int32_t v = (int32_t)(j < 32 ? kept[0] : kept[1]);  // (M <= 64 links)
        row[j] = j < r ? v : -1;
        if (j >= r) continue;
        const int32_t off = l == 0 ? 0 : a.up_off[v];
        if (off < 0) {  // a level-l link to a node below level l
          set_error(a.err, UHNSW_EINVAL);
          continue;
        }
        const int64_t rid = l == 0 ? (int64_t)v : a.n + (int64_t)off + l - 1;
        push_incoming(a, chk_idx(rid, a.n + a.rows, 29, a.err), (int32_t)u);
      }
    }
  }
}

// Phase 2 of a batch: one block per row that received links; a row past its
// cap is re-selected by all its warps, others only take the new links.
struct BuildReverseLayout {
  int qv, ui, key, sorted, state, total;
  __host__ __device__ BuildReverseLayout(int d_pad, int M0) {
    const int ucap = M0 + kInCap;
    int o = 0;
    qv = o; o += align16(d_pad * 4);
    ui = o; o += align16(ucap * 4);
    key = o; o += align16(ucap * 8);
    sorted = o; o += align16(ucap * 8);
    state = o; o += 2 * kBuildWarps * 4;
    total = o;
  }
};

__global__ void __launch_bounds__(kBuildWarps * 32) build_reverse_kernel(const BuildArgs a) {
  constexpr int THREADS = kBuildWarps * 32;
  extern __shared__ __align__(16) unsigned char smem[];
  const BuildReverseLayout L(a.d_pad, a.M0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, team = lane >> 3, lt = lane & 7;
  float* qv = reinterpret_cast<float*>(smem + L.qv);
  uint32_t* ui = reinterpret_cast<uint32_t*>(smem + L.ui);
  unsigned long long* key = reinterpret_cast<unsigned long long*>(smem + L.key);
  unsigned long long* sorted = reinterpret_cast<unsigned long long*>(smem + L.sorted);
  const int total = *a.touched_n;
  for (int t = blockIdx.x; t < total; t += gridDim.x) {
    const int64_t r = a.touched[chk_idx(t, a.n + a.rows, 27, a.err)];
    const bool l0 = r < a.n;
    const int64_t v = l0 ? r : a.up_owner[chk_idx(r - a.n, a.rows, 28, a.err)];
    const int cap = l0 ? a.M0 : a.M;
    int32_t* row = l0 ? a.ell0 + r * a.M0 : a.up_adj + (r - a.n) * a.M;
    const int nin = min(a.inc_cnt[r], kInCap);
    // old links (compact, -1 after the last)
    int ne = 0;
    for (int b0 = 0; b0 < cap; b0 += 32) {
      const int j = b0 + lane;
      ne += __popc(__ballot_sync(kFull, j < cap && row[j] >= 0));
    }
    const int nu = ne + nin;
    // incoming links sorted by id, so that the row does not depend on the
    // order in which the warps of phase 1 pushed them
    for (int j = tid; j < nin; j += THREADS) key[j] = (uint32_t)a.inc[r * kInCap + j];
    __syncthreads();
    for (int j = tid; j < nu; j += THREADS) {
      if (j < ne) {
        ui[j] = (uint32_t)row[j];
      } else {
        const unsigned long long x = key[j - ne];
        int rank = 0;
        for (int i = 0; i < nin; ++i) rank += key[i] < x;
        ui[ne + rank] = (uint32_t)x;
      }
    }
    __syncthreads();
    if (nu <= cap) {
      for (int j = ne + tid; j < nu; j += THREADS) row[j] = (int32_t)ui[j];
    } else {
      for (int j = tid; j < a.d_pad; j += THREADS) qv[j] = a.X[v * a.d_pad + j];
      __syncthreads();
      for (int i0 = warp * 8; i0 < nu; i0 += kBuildWarps * 8) {
        const int ia = i0 + team, ib = ia + 4;
        const uint32_t da = ui[min(ia, nu - 1)], db = ui[min(ib, nu - 1)];
        float sa, sb;
        build_dist2_metric(a.metric, a.X + chk_idx(da, a.n, 20, a.err) * a.d_pad,
                           a.X + chk_idx(db, a.n, 20, a.err) * a.d_pad, qv, a.d_pad, lt, a.bp, sa,
                           sb);
        if (lt == 0 && ia < nu) key[ia] = make_key(sa, da);
        if (lt == 0 && ib < nu) key[ib] = make_key(sb, db);
      }
      __syncthreads();
      // order by (distance, id)
      for (int j = tid; j < nu; j += THREADS) {
        const unsigned long long x = key[j];
        int rank = 0;
        for (int i = 0; i < nu; ++i) rank += key[i] < x;
        sorted[rank] = x;
      }
      __syncthreads();
      uint32_t kept[4] = {0, 0, 0, 0};  // (caps of up to 128 links)
      const int rs = block_select<kBuildWarps, 4>(a, sorted, nu, cap, kept,
                                                  reinterpret_cast<int32_t*>(smem + L.state));
      if (warp == 0)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int j = 32 * c + lane;
          if (j < cap) row[j] = j < rs ? (int32_t)kept[c] : -1;
        }
    }
    if (tid == 0) a.inc_cnt[r] = 0;
    __syncthreads();
  }
}

}  // namespace
}  // namespace uhnsw_dev

extern "C" int uhnsw_build_graph_gpu(const float* base, int64_t n, int32_t d, int32_t metric,
                                     int32_t M, int32_t ef_construction, const int32_t* levels,
                                     uhnsw_built** out) {
  uhnsw_internal::clear_error();
  if (!out) return uhnsw_internal::fail(UHNSW_EINVAL, "uhnsw_build_graph_gpu: out is NULL");
  *out = nullptr;
  if (metric < UHNSW_BASE_L1 || metric > UHNSW_BASE_L15)
    return uhnsw_internal::fail(UHNSW_EINVAL, "uhnsw_build_graph_gpu: metric must be 1, 2, 3 or 4");
  return uhnsw_internal::build_graph_gpu(base, n, d, metric, 0.f, M, ef_construction, levels, out);
}

int uhnsw_internal::build_graph_gpu(const float* base, int64_t n, int32_t d, int32_t metric,
                                    float bp, int32_t M, int32_t ef_construction,
                                    const int32_t* levels, uhnsw_built** out) {
  using namespace uhnsw_dev;
  using uhnsw_internal::fail;
  if (!base || !levels || n < 1 || n > INT32_MAX / 2 || d < 1 || d > UHNSW_MAX_DIM)
    return fail(UHNSW_EINVAL, "uhnsw_build_graph_gpu: bad base/levels/n/d");
  if (M < 2 || 2 * M > UHNSW_MAX_DEGREE || ef_construction < 1 || ef_construction > 512)
    return fail(UHNSW_EINVAL, "uhnsw_build_graph_gpu: need 2 <= M <= %d, 1 <= efc <= 512",
                UHNSW_MAX_DEGREE / 2);
  std::vector<int32_t> up_off(n, -1), up_owner;
  int32_t top = 0;
  for (int64_t v = 0; v < n; ++v) {
    if (levels[v] < 0 || levels[v] >= UHNSW_MAX_LEVELS)
      return fail(UHNSW_EINVAL, "uhnsw_build_graph_gpu: level of node %lld is %d", (long long)v,
                  levels[v]);
    if (levels[v] > 0) {
      up_off[v] = (int32_t)up_owner.size();
      for (int l = 0; l < levels[v]; ++l) up_owner.push_back((int32_t)v);
    }
  }
  const int64_t rows = (int64_t)up_owner.size();
  const int32_t M0 = 2 * M;
  const int32_t d_pad = (d + 7) / 8 * 8;
  const int32_t efc = ef_construction;
  int hb = 11;
  while ((1 << hb) < 4 * (efc + M0)) ++hb;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return fail(UHNSW_ECUDA, "uhnsw_build_graph_gpu: %s", cudaGetErrorString(e));
  const size_t smem2 = (size_t)BuildReverseLayout(d_pad, M0).total;

  // device buffers
  float* X = nullptr;
  int32_t *lv = nullptr, *doff = nullptr, *downer = nullptr, *ell0 = nullptr, *up_adj = nullptr;
  int32_t *inc_cnt = nullptr, *inc = nullptr, *touched = nullptr, *scal = nullptr;
  auto release = [&]() {
    cudaFree(X); cudaFree(lv); cudaFree(doff); cudaFree(downer); cudaFree(ell0);
    cudaFree(up_adj); cudaFree(inc_cnt); cudaFree(inc); cudaFree(touched); cudaFree(scal);
  };
  const int64_t nr = n + rows;
  e = cudaMalloc(&X, (size_t)n * d_pad * 4);
  if (e == cudaSuccess) e = cudaMalloc(&lv, n * 4);
  if (e == cudaSuccess) e = cudaMalloc(&doff, n * 4);
  if (e == cudaSuccess) e = cudaMalloc(&downer, std::max<int64_t>(rows, 1) * 4);
  if (e == cudaSuccess) e = cudaMalloc(&ell0, (size_t)n * M0 * 4);
  if (e == cudaSuccess) e = cudaMalloc(&up_adj, (size_t)std::max<int64_t>(rows, 1) * M * 4);
  if (e == cudaSuccess) e = cudaMalloc(&inc_cnt, nr * 4);
  if (e == cudaSuccess) e = cudaMalloc(&inc, (size_t)nr * kInCap * 4);
  if (e == cudaSuccess) e = cudaMalloc(&touched, nr * 4);
  if (e == cudaSuccess) e = cudaMalloc(&scal, 64);
  if (e != cudaSuccess) {
    release();
    return fail(UHNSW_EOOM, "uhnsw_build_graph_gpu: device memory: %s", cudaGetErrorString(e));
  }
  e = cudaMemset(X, 0, (size_t)n * d_pad * 4);
  if (e == cudaSuccess)
    e = cudaMemcpy2D(X, (size_t)d_pad * 4, base, (size_t)d * 4, (size_t)d * 4, n,
                     cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(lv, levels, n * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(doff, up_off.data(), n * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess && rows)
    e = cudaMemcpy(downer, up_owner.data(), rows * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(ell0, 0xff, (size_t)n * M0 * 4);
  if (e == cudaSuccess) e = cudaMemset(up_adj, 0xff, (size_t)std::max<int64_t>(rows, 1) * M * 4);
  if (e == cudaSuccess) e = cudaMemset(inc_cnt, 0, nr * 4);
  if (e == cudaSuccess) e = cudaMemset(scal, 0, 64);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(build_reverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem2);
  int occ2 = 0;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ2, build_reverse_kernel,
                                                      kBuildWarps * 32, smem2);
  // the insertion's forms, most warps first, and the batch sizes up to which
  // all blocks are resident
  struct Form {
    void (*kern)(BuildArgs, int64_t, int32_t, int32_t, int);
    int warps, hb;
    size_t smem;
    int64_t cap;
  } forms[3] = {{build_insert_kernel<8>, 8, 13, 0, 0},
                {build_insert_kernel<4>, 4, 12, 0, 0},
                {build_insert_kernel<2>, 2, 11, 0, 0}};
  for (Form& f : forms) {
    f.hb = std::max(f.hb, hb);
    const int slots = (M0 + f.warps - 1) / f.warps * f.warps;
    f.smem = BuildInsertLayout(d_pad, efc, f.hb, slots, f.warps + 1).total;
    int occ = 0;
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)f.smem);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, f.kern, (f.warps + 1) * 32, f.smem);
    f.cap = (int64_t)occ * sms;
  }
  if (e != cudaSuccess || occ2 < 1 || forms[2].cap < 1) {
    release();
    return fail(UHNSW_ECUDA, "uhnsw_build_graph_gpu: setup: %s",
                e != cudaSuccess ? cudaGetErrorString(e) : "kernel does not fit");
  }

  BuildArgs a;
  a.X = X;
  a.lv = lv;
  a.up_off = doff;
  a.up_owner = downer;
  a.ell0 = ell0;
  a.up_adj = up_adj;
  a.inc_cnt = inc_cnt;
  a.inc = inc;
  a.touched = touched;
  a.touched_n = scal + 8;
  a.err = scal;
  a.n = n;
  a.rows = rows;
  a.d_pad = d_pad;
  a.metric = metric;
  a.bp = bp;
  a.M = M;
  a.M0 = M0;
  a.efc = efc;

  int32_t ep = 0, cur_top = levels[0];
  int64_t s = 1;
  while (s < n && e == cudaSuccess) {
    const int64_t b = std::max<int64_t>(1, std::min<int64_t>(65536, s / 16));
    const int64_t end = std::min(n, s + b);
    const int64_t warps = end - s;
    const Form& form = warps <= forms[0].cap ? forms[0] : warps <= forms[1].cap ? forms[1] : forms[2];
    form.kern<<<(unsigned)warps, (form.warps + 1) * 32, form.smem>>>(a, s, ep, cur_top, form.hb);
    e = cudaGetLastError();
    if (e != cudaSuccess) break;
    const int64_t grid2 = std::min<int64_t>(warps * M * 2, (int64_t)occ2 * sms);
    build_reverse_kernel<<<(unsigned)std::max<int64_t>(grid2, 1), kBuildWarps * 32, smem2>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) break;
    e = cudaMemsetAsync(a.touched_n, 0, 4);
    for (int64_t u = s; u < end; ++u)
      if (levels[u] > cur_top) {
        cur_top = levels[u];
        ep = (int32_t)u;
      }
    s = end;
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  int32_t hs[2] = {0, 0};
  if (e == cudaSuccess) e = cudaMemcpy(hs, scal, 8, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) {
    release();
    return fail(UHNSW_ECUDA, "uhnsw_build_graph_gpu: %s", cudaGetErrorString(e));
  }
  if (hs[0] != 0) {
    release();
    return fail(hs[0], "uhnsw_build_graph_gpu: device error %d", hs[0]);
  }
  try {
    std::vector<int32_t> h0((size_t)n * M0), hu((size_t)std::max<int64_t>(rows, 1) * M);
    e = cudaMemcpy(h0.data(), ell0, h0.size() * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(hu.data(), up_adj, hu.size() * 4, cudaMemcpyDeviceToHost);
    release();
    if (e != cudaSuccess)
      return fail(UHNSW_ECUDA, "uhnsw_build_graph_gpu: download: %s", cudaGetErrorString(e));
    *out = uhnsw_internal::make_built(n, M, M0, levels, ep, cur_top, h0.data(), up_off.data(),
                                      hu.data());
    if (!*out) return fail(UHNSW_EOOM, "uhnsw_build_graph_gpu: out of host memory");
  } catch (const std::bad_alloc&) {
    release();
    return fail(UHNSW_EOOM, "uhnsw_build_graph_gpu: out of host memory");
  }
  return UHNSW_OK;
}
