// What the search kernels share: their arguments, the routing of a query and
// the shared-memory layout of the warp kernel (Section 3.1, Algorithm 1).
//
// Per query, both kernels (warp_kernels.cuh: one warp per query;
// coop_kernels.cuh: one block per query):
//   1. route: p == 1 / p == 2 search G1 / G2 for the K nearest directly;
//      otherwise p <= cutoff -> G1 (L1), else G2 (squared L2);
//   2. greedy descent from the entry point through the upper levels (beam 1);
//   3. layer-0 best-first search with beam ef' (HNSW SEARCH-LAYER);
//   4. C = the first t beam entries (ascending base distance);
//   5. verification: exact (top-K by (S, id) over C, a candidate abandoned
//      once its partial sum exceeds the running K-th S) or Algorithm 1's
//      batches of kappa with the |R_new n R| / K >= tau stop;
//   6. distances S^(1/p), ascending (distance, id), padded with -1 / +inf.
//
// Layer 0 keeps the result set W as one sorted shared-memory list of ef'
// (distance, id) entries with an "expanded" bit.  With a strict total order
// this is the same search as HNSW's two heaps: every unexpanded member of W
// sits in the candidate heap, every other heap member is worse than W's
// furthest entry, so the heap's next pop is W's best unexpanded entry, and the
// heap search stops exactly when W has none left.  Expanding one entry per step
// (search_width 1) therefore reproduces the sequential HNSW order; its
// neighbours are merged into W in one step, which equals inserting them one by
// one into a bounded W (both keep the best ef' of the union).
//
// The visited set is an open-addressing table in shared memory.  When its load
// passes one half it is cleared and refilled with the ids currently in W.  A
// node forgotten this way can be evaluated again, but it cannot re-enter W: it
// was either rejected or evicted while W was full, and W's furthest entry only
// improves afterwards.  So W, the expansion order and the result are exactly
// those of an unbounded visited set; only extra distance evaluations are paid.
#pragma once

#include <climits>
#include <type_traits>

#include "device_common.cuh"

namespace uhnsw_dev {

struct GraphDev {
  const int32_t* ell0;   // [n][deg0] layer-0 links, -1 padded
  const int32_t* up_row; // [n] first upper-level row of the node, -1 if it is only on layer 0
  const int32_t* up_adj; // [rows][deg], -1 padded; row of (v, level l) = up_row[v] + l - 1
  int32_t up_rows;
  int32_t entry;
  int32_t top_level;
  int32_t deg0;
  int32_t deg;
};

__host__ __device__ inline int align16(int x) { return (x + 15) & ~15; }

// Dynamic shared-memory carve-up (byte offsets), identical on host and device.
struct SmemLayout {
  int stage, qs, bd0, bi0, bd1, bi1, hash, cd, ci, sd, si, td0, ti0, td1, ti1, cv, total;
  SmemLayout() = default;
  __host__ __device__ SmemLayout(int d_pad, int ef_cap, int hash_bits, int cmax, int k_max,
                                 int vcap, int stage_bytes = 0) {
    int o = 0;
    qs = o; o += align16(d_pad * 4);
    bd0 = o; o += align16(ef_cap * 4);
    bi0 = o; o += align16(ef_cap * 4);
    bd1 = o; o += align16(ef_cap * 4);
    bi1 = o; o += align16(ef_cap * 4);
    // The visited table lives during the search, the staged verification rows
    // after it: they share one region.
    const int hash_bytes = align16((hash_bits > 0 ? (1 << hash_bits) : 0) * 4);
    hash = o;
    stage = o;
    o += hash_bytes > align16(stage_bytes) ? hash_bytes : align16(stage_bytes);
    cd = o; o += align16(cmax * 4);
    ci = o; o += align16(cmax * 4);
    sd = o; o += align16(cmax * 4);
    si = o; o += align16(cmax * 4);
    td0 = o; o += align16(k_max * 4);
    ti0 = o; o += align16(k_max * 4);
    td1 = o; o += align16(k_max * 4);
    ti1 = o; o += align16(k_max * 4);
    cv = o; o += align16(vcap * 4);
    total = o;
  }
};

struct QueryArgs {
  const float* base32;  // FP32 master copy [n][d_pad]
  const void* trav;     // traversal copy [n][d_pad] in the kernel's element type
  int64_t n;
  int32_t d, d_pad;
  GraphDev g[2];        // graph slots: G1 (L1) and G2 (squared L2), or G0.5 and G1
  int32_t gmetric[2];   // base metric of each slot (uhnsw_base_metric)
  float gp[2];          // the p of each slot's base metric
  const float* q;       // [nq][d]
  const float* p;       // [nq]
  const int32_t* k;     // [nq] or null (k_max)
  const int32_t* ef;    // [nq] or null (ef_default)
  int64_t nq;
  int32_t k_max, ef_default, ef_cap;
  int32_t t;            // 0 => ef
  int32_t kappa;        // 0 => k
  float tau, cutoff;
  const int32_t* tq;    // [nq] per-query t, or null (t)
  const float* tauq;    // [nq] per-query tau (0 => 0.92), or null (tau)
  int32_t mode;         // uhnsw_verify_mode
  int32_t width;        // beam entries expanded per step
  int32_t hash_bits;    // visited table holds 1 << hash_bits slots
  int32_t cmax;         // capacity of the per-step candidate buffers
  int32_t vcap;         // capacity of the candidate list C (verification-only launch)
  int64_t* out_ids;     // [nq][k_max]
  float* out_dist;      // [nq][k_max]
  int32_t* stats;       // [nq][UHNSW_NSTATS] or null
  int32_t* queue_head;  // persistent launch: next query slot; null => blockIdx.x only
  const int32_t* qorder;   // bucketed launch: query of each slot, grouped by beam bucket
  const int32_t* qbucket;  // bucketed launch: {first slot, slot count} of this bucket
  int32_t* err;         // sticky device error word
  const int32_t* cand;  // verification-only launch: [nq][cand_t]
  int32_t cand_t;
  int32_t trav_exact;   // 1: the traversal copy holds every FP32 value exactly
  int32_t stage_bytes;  // warp kernel: per-warp staging buffer for cp.async row copies
  int32_t sb;           // warp kernel: traversal rows staged per batch
  int32_t sv;           // warp kernel: FP32 rows staged per verification batch (multiple of 4)
  SmemLayout lay;       // warp kernel: one warp's shared memory
  int32_t chain;        // launches that may run at once (see chain_begin): 1 = a next one
                        // follows, 2 = one is before this
  int32_t vgroups;      // warp kernels' verification: 32-dimension groups between two drop
                        // tests (>= 1); the cooperative kernel tests after every four
};

// Routing of a query (Algorithm 1, lines 1-5): the graph slot it searches,
// whether it is answered directly (p is that graph's own base p), the slot's
// base metric and its p.  p <= cutoff selects the first slot.
struct Route {
  int slot;
  bool direct;
  int metric;
  float bp;
};
__device__ __forceinline__ Route route_query(const QueryArgs& a, float p) {
  const int slot = p == a.gp[0] ? 0 : p == a.gp[1] ? 1 : (p <= a.cutoff ? 0 : 1);
  const float bp = a.gp[slot];
  return Route{slot, p == bp, a.gmetric[slot], bp};
}

// t and tau of query qi (per-query arrays when given).
__device__ __forceinline__ int query_t(const QueryArgs& a, int64_t qi) {
  return a.tq ? a.tq[qi] : a.t;
}
__device__ __forceinline__ float query_tau(const QueryArgs& a, int64_t qi) {
  if (!a.tauq) return a.tau;
  const float v = a.tauq[qi];
  return v != 0.f ? v : 0.92f;
}

// The distance a direct query returns: the base sum's root S^(1/bp).
__device__ __forceinline__ float base_root(int metric, float bp, float s) {
  return metric == UHNSW_BASE_L1    ? s
         : metric == UHNSW_BASE_L2  ? sqrtf(s)
         : metric == UHNSW_BASE_L05 ? (float)((double)s * (double)s)
         : metric == UHNSW_BASE_L15 ? root_p(s, 1.5f)
                                    : root_p(s, bp);
}

__device__ __forceinline__ uint32_t dynamic_smem_bytes() {
  uint32_t r;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(r));
  return r;
}

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned r;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(r));
  return r;
}

// The launches of a bucketed search take different queries and depend on each
// other in nothing, so each may start as soon as every block of the one before
// has started, on the slots that its finished blocks leave: its last queries,
// up to a third of a launch, no longer run on an idle GPU.  Block 0 ends only
// when the launch before has, so that the stream's next work waits for all.
// Queries of mixed ef, ms one after the other and chained: 10,000 of 100k x 960
// BF16 14.2 and 12.6; 1M x 128 FP16, 10,000 11.0 and 7.7, 4,000 7.9 and 3.6, 30
// 1.58 and 0.85.
__device__ __forceinline__ void chain_begin(const QueryArgs& a) {
  if (a.chain & 1) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void chain_end(const QueryArgs& a) {
  if ((a.chain & 2) && blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Per-query counters; the caller lets exactly one thread of the query call it.
__device__ __forceinline__ void put_stats(const QueryArgs& a, int64_t qi, int nb, int np,
                                          int terms, int nexp, int nres, int status, int graph,
                                          int nadj) {
  if (!a.stats) return;
  int32_t* st = a.stats + qi * UHNSW_NSTATS;
  st[UHNSW_STAT_NB] = nb;
  st[UHNSW_STAT_NP] = np;
  st[UHNSW_STAT_TERMS] = terms;
  st[UHNSW_STAT_EXPANSIONS] = nexp;
  st[UHNSW_STAT_RESETS] = nres;
  st[UHNSW_STAT_STATUS] = status;
  st[UHNSW_STAT_GRAPH] = graph;
  st[UHNSW_STAT_ADJ] = nadj;
}

}  // namespace uhnsw_dev
