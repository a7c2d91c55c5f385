// Cooperative form of the query kernel (same algorithm and result as the warp
// kernel in warp_kernels.cuh, Section 3.1 / Algorithm 1), for launches that
// cannot fill the GPU with one warp per query: NW warps compute the distances
// of one query's step and one more warp keeps its beam.
//
// What bounds such a launch is the chain of dependent operations of each
// query's search, so a step here is one barrier long.  Between two barriers
// the distance warps read the parents' links, filter them through the visited
// table and sum the fresh rows, each warp its own share of the links; the
// merge warp meanwhile folds the candidates of the step before into W.  After
// the barrier every warp picks the next parents for itself from the new
// candidates and what the merge warp published of W (its first unexpanded
// entries and the last ones that can be pushed out), so nobody waits for the
// merge: the order of expansions is exactly the warp kernel's.
//
// W and the candidates are 64-bit keys (distance bits, id, expanded flag),
// which order like (distance, id): distances are sums of non-negative terms,
// whose bits order like their values (a NaN sorts last).  W is kept in place:
// a merge moves the entries behind the first new one, from the end down.
//
// Each row is summed by the same lanes in the same order as in the warp
// kernel, and each L_p sum by the same 8-lane teams, so the two kernels
// return identical ids and distances.
#pragma once

#include "query_kernels.cuh"
#include "warp_kernels.cuh"

namespace uhnsw_dev {

constexpr unsigned long long kNoKey = ~0ull;
constexpr int kMaxWidth = 8;

__device__ __forceinline__ unsigned long long make_key(float d, uint32_t id) {
  return ((unsigned long long)__float_as_uint(d) << 32) | (id << 1);
}
__device__ __forceinline__ uint32_t key_id(unsigned long long k) { return (uint32_t)k >> 1; }
__device__ __forceinline__ float key_dist(unsigned long long k) {
  return __uint_as_float((uint32_t)(k >> 32));
}
__device__ __forceinline__ unsigned long long warp_min_key(unsigned long long k) {
  const unsigned hi = (unsigned)(k >> 32);
  const unsigned mh = __reduce_min_sync(kFull, hi);
  const unsigned ml = __reduce_min_sync(kFull, hi == mh ? (unsigned)k : 0xffffffffu);
  return ((unsigned long long)mh << 32) | ml;
}

// What the merge warp tells the others about W.
struct CoopPub {
  unsigned long long uk[2 * kMaxWidth];  // the first 2 width unexpanded entries, kNoKey past the last
  unsigned long long wl[kMaxWidth];      // wl[j]: the entry that j + 1 smaller new ones push out
  int pos[2 * kMaxWidth];                // positions of uk (INT_MAX past the last)
  unsigned long long last;               // W's last entry if W is full, else kNoKey
  int bn;                                // length of W
  int pad;
};

struct CoopLayout {
  int qs, W, tab, ck0, ck1, nk, sk, wl, cnt, pub, td, vs, total;
  // d_ext: query floats kept (the row padded to the team's chunks); slots:
  // candidate slots of a step; warps: all warps of the block
  __host__ __device__ CoopLayout(int d_ext, int ef_cap, int hash_bits, int slots, int k_max,
                                 int warps) {
    const int most = slots > warps * 4 ? slots : warps * 4;
    const int keys = (most + 63) / 64 * 64;
    int o = 0;
    qs = o; o += align16(d_ext * 4);
    W = o; o += align16(ef_cap * 8);
    // the visited table during the search, the candidate ids C after it
    const int tb = (1 << hash_bits) * 4;
    tab = o; o += align16(tb > ef_cap * 4 ? tb : ef_cap * 4);
    ck0 = o; o += align16(keys * 8);
    ck1 = o; o += align16(keys * 8);
    nk = o; o += align16(keys * 8);
    sk = o; o += align16((keys + 32) * 8);
    wl = o; o += align16(warps * 32 * 4);
    cnt = o; o += align16(2 * warps * 4);
    pub = o; o += 2 * (int)sizeof(CoopPub);
    td = o; o += align16(k_max * 8);
    vs = o; o += 32;
    total = o;
  }
};

// coop_merge for m <= 32 new keys nk and a list of n <= 32 NC entries, which
// the lanes hold: each new key finds its place in L by search, each entry its
// shift by counting the new keys before it.  Lane i returns the place of key i.
template <int NC>
__device__ __forceinline__ void coop_merge_small(unsigned long long* L, int n, int cap,
                                                 const unsigned long long* nk, int m, int flagged,
                                                 int* at) {
  const int lane = threadIdx.x & 31;
  const unsigned long long mine = lane < m ? nk[lane] : kNoKey;
  unsigned long long x[NC];
  int c[NC], place = 0, rank = 0;
#pragma unroll
  for (int u = 0; u < NC; ++u) {
    x[u] = 32 * u + lane < n ? L[32 * u + lane] : kNoKey;
    c[u] = 0;
  }
#pragma unroll
  for (int h = NC * 16; h > 0; h >>= 1)
    if (place + h <= n && L[place + h - 1] < mine) place += h;
  if (place < n && L[place] < mine) ++place;
#pragma unroll 4
  for (int i = 0; i < m; ++i) {
    const unsigned long long y = nk[i];
    rank += y < mine;
#pragma unroll
    for (int u = 0; u < NC; ++u) c[u] += y < x[u];
  }
  __syncwarp();
#pragma unroll
  for (int u = 0; u < NC; ++u) {
    const int j = 32 * u + lane;
    if (j < n && c[u] > 0 && j + c[u] < cap) L[j + c[u]] = x[u];
  }
  place += rank;
  if (lane < m && place < cap) L[place] = mine | (rank < flagged ? 1ull : 0ull);
  *at = (int)__reduce_min_sync(kFull, lane < m && rank == flagged ? (unsigned)place : (unsigned)INT_MAX);
  __syncwarp();
}

// Merges the keys below `limit` among in[0 .. total) into the ascending list
// L[0 .. n) in place, keeping the first `cap`; the `flagged` smallest of them
// enter with the expanded flag.  One warp; nk / sk are scratch (sk holds at
// least 32 entries past the last new key).  Returns the length of the merged
// list; *at receives the position of the first new entry without the flag
// (INT_MAX if none).
//
// The new keys are sorted by counting (m of them, few after the limit), each
// entry of L finds its shift c by a search without branches, four chunks of L
// at a time so that the searches overlap, and the places of the new keys
// follow from where c steps: key i stands before the first entry whose c
// exceeds i.  Chunks are taken from the end down, so that entries move in
// place, and the walk stops below the first new key.
__device__ __forceinline__ int coop_merge(unsigned long long* L, int n, int cap,
                                          const unsigned long long* in, int total,
                                          unsigned long long limit, int flagged,
                                          unsigned long long* nk, unsigned long long* sk, int* at) {
  const int lane = threadIdx.x & 31;
  int m = 0;
  for (int b = 0; b < total; b += 64) {
    const unsigned long long x0 = b + lane < total ? in[b + lane] : kNoKey;
    const unsigned long long x1 = b + 32 + lane < total ? in[b + 32 + lane] : kNoKey;
    const unsigned b0 = __ballot_sync(kFull, x0 < limit);
    const unsigned b1 = __ballot_sync(kFull, x1 < limit);
    const int m0 = m + __popc(b0);
    if (x0 < limit) nk[m + __popc(b0 & lanemask_lt())] = x0;
    if (x1 < limit) nk[m0 + __popc(b1 & lanemask_lt())] = x1;
    m = m0 + __popc(b1);
  }
  *at = INT_MAX;
  if (m == 0) return n;
  __syncwarp();
  if (m <= 32 && n <= 128) {
    if (n <= 64) coop_merge_small<2>(L, n, cap, nk, m, flagged, at);
    else coop_merge_small<4>(L, n, cap, nk, m, flagged, at);
    return min(cap, n + m);
  }
  for (int i = lane; i < m; i += 32) {
    const unsigned long long x = nk[i];
    int r = 0;
#pragma unroll 4
    for (int j = 0; j < m; ++j) r += nk[j] < x;
    sk[r] = x;
  }
  sk[m + lane] = kNoKey;
  __syncwarp();
  int* place = reinterpret_cast<int*>(nk);
  // up to 32 of them at a time, the smallest first
  for (int s0 = 0; s0 < m; s0 += 32) {
    const int mm = min(32, m - s0);
    const unsigned long long* ks = sk + s0;
    int top = 1;
    while (top < mm) top <<= 1;
    top >>= 1;
    int above = mm;  // c of the entry behind the chunk
    int b = n > 0 ? (n - 1) & ~127 : -128;
    for (; b >= 0 && above > 0; b -= 128) {
      unsigned long long x[4];
      int c[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = b + 32 * u + lane;
        x[u] = j < n ? L[j] : kNoKey;
        c[u] = 0;
      }
      for (int h = top; h > 0; h >>= 1) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (b + 32 * u < n) c[u] += ks[c[u] + h - 1] < x[u] ? h : 0;
        }
      }
#pragma unroll
      for (int u = 3; u >= 0; --u) {
        if (b + 32 * u < n) {
          const int j = b + 32 * u + lane;
          c[u] += ks[c[u]] < x[u];
          if (j >= n) c[u] = mm;
          int next = __shfl_down_sync(kFull, c[u], 1);
          if (lane == 31) next = above;
          if (j < n) {
            for (int i = c[u]; i < next; ++i) place[i] = j + 1;
            if (c[u] > 0 && j + c[u] < cap) L[j + c[u]] = x[u];
          }
          above = __shfl_sync(kFull, c[u], 0);
        }
      }
      __syncwarp();
    }
    if (lane < above) place[lane] = 0;  // before every entry of L
    __syncwarp();
    const int pos = lane < mm ? place[lane] + lane : 0;
    if (lane < mm && pos < cap) L[pos] = ks[lane] | (s0 + lane < flagged ? 1ull : 0ull);
    if (flagged >= s0 && flagged < s0 + mm) *at = __shfl_sync(kFull, pos, flagged - s0);
    n = min(cap, n + mm);
    __syncwarp();
  }
  return n;
}

// The merge warp's part of a step: the candidates in[] into W, the parents
// just picked (the first nWp of pub.uk and the jn smallest candidates) marked
// expanded, and the new state of W published.
__device__ __forceinline__ void coop_merge_step(unsigned long long* W, int cap, int width,
                                                const unsigned long long* in, int total,
                                                const CoopPub* pi, CoopPub* po, int nWp, int jn,
                                                unsigned long long* nk, unsigned long long* sk) {
  const int lane = threadIdx.x & 31;
  const int bn = pi->bn;
  if (lane < nWp) W[pi->pos[lane]] |= 1ull;
  // a candidate behind a full W's last entry cannot enter it
  const unsigned long long limit = pi->last;
  int at = 0;
  const int nbn = coop_merge(W, bn, cap, in, total, limit, jn, nk, sk, &at);
  // entries before both the next old unexpanded one and the first new one
  // without the flag are expanded (positions of old ones only grow)
  const int want = 2 * width;
  int found = 0;
  for (int b = min(pi->pos[nWp], at); b < nbn && found < want; b += 32) {
    const int j = b + lane;
    const unsigned long long x = j < nbn ? W[j] : 1ull;
    const bool open = !(x & 1ull);
    const unsigned ball = __ballot_sync(kFull, open);
    const int r = found + __popc(ball & lanemask_lt());
    if (open && r < want) {
      po->uk[r] = x;
      po->pos[r] = j;
    }
    found += __popc(ball);
  }
  if (lane < want && lane >= found) {
    po->uk[lane] = kNoKey;
    po->pos[lane] = INT_MAX;
  }
  if (lane < width) {
    const int e = cap - 1 - lane;
    po->wl[lane] = e < 0 ? 0ull : e < nbn ? W[e] : kNoKey;
  }
  if (lane == 0) {
    po->bn = nbn;
    po->last = nbn == cap ? W[cap - 1] : kNoKey;
  }
}

// The next parents, picked by every warp for itself: the first `width`
// unexpanded entries of W merged with the candidates ck[0 .. total), in key
// order.  An entry is one of W's first cap exactly if fewer than cap entries
// precede it: pos[i] + (new ones before it) for an old one; for a new one
// with jn new ones before it, if it precedes wl[jn].  Returns their number;
// lane j < that number holds parent j in par; nWp and jn count the old and
// the new ones.  ck is filled with kNoKey up to a multiple of 64.
__device__ __forceinline__ int coop_select(const unsigned long long* ck, int total,
                                           const CoopPub* pub, int width, int cap, int& nWp,
                                           int& jn, uint32_t& par) {
  const int lane = threadIdx.x & 31;
  unsigned long long x0 = ck[lane], x1 = ck[lane + 32];
  if (width == 1 && total <= 64) {
    const unsigned long long u = pub->uk[0], w0 = pub->wl[0];
    const unsigned long long c = warp_min_key(x0 < x1 ? x0 : x1);
    // (an unexpanded entry of W keeps its place: no candidate precedes it)
    nWp = u < c;
    jn = !nWp && c < w0;
    par = key_id(nWp ? u : c);
    return nWp + jn;
  }
  nWp = jn = 0;
  int npar = 0;
  unsigned long long lo = 0, c = kNoKey;
  bool scan = true;
  for (;;) {
    if (scan) {
      unsigned long long mn = kNoKey;
      for (int b = lane; b < total; b += 64) {
        if (b >= 64) {
          x0 = ck[b];
          x1 = ck[b + 32];
        }
        if (x0 >= lo && x0 < mn) mn = x0;
        if (x1 >= lo && x1 < mn) mn = x1;
      }
      if (total > 64) {
        x0 = ck[lane];
        x1 = ck[lane + 32];
      }
      c = warp_min_key(mn);
      scan = false;
    }
    const unsigned long long u = pub->uk[nWp];
    if (u == kNoKey && c == kNoKey) break;
    unsigned long long pick;
    if (u < c) {
      if (pub->pos[nWp] + jn >= cap) break;
      pick = u;
      ++nWp;
    } else {
      if (!(c < pub->wl[jn])) break;
      pick = c;
      lo = c + 1;
      scan = true;
      ++jn;
    }
    if (lane == npar) par = key_id(pick);
    if (++npar == width) break;
  }
  return npar;
}

// Base distances of the rows ids[0 .. nf) by one distance warp, as keys into
// out[0 .. nf).  TEAM lanes per row, CPL 16-byte chunks per lane, U rows per
// team and round; chunk order and team butterfly as in warp_dist.  A lane
// whose chunk lies past the row adds nothing (the warp kernel adds zeros).
template <typename T, int TEAM, int CPL, int U, bool QREG, int METRIC>
__device__ __forceinline__ void coop_dist(const T* __restrict__ rows, int d_pad, const float* qs,
                                          const uint64_t (&qv)[QREG ? CPL : 1][Elems16<T>::n / 2],
                                          const uint32_t* ids, int nf, unsigned long long* out,
                                          float bp) {
  constexpr int VEC = Elems16<T>::n;
  constexpr int NT = 32 / TEAM;
  const int lane = threadIdx.x & 31;
  const int team = lane / TEAM, lt = lane % TEAM;
  const int R = d_pad / VEC;
  for (int r0 = 0; r0 < nf; r0 += NT * U) {
    uint4 buf[U][CPL];
    uint32_t id[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = r0 + u * NT + team;
      id[u] = ids[min(i, nf - 1)];
      const uint4* row = reinterpret_cast<const uint4*>(rows + (int64_t)id[u] * d_pad);
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const int ch = lt + c * TEAM;
        buf[u][c] = make_uint4(0u, 0u, 0u, 0u);
        if (i < nf && ch < R) buf[u][c] = __ldg(row + ch);
      }
    }
    uint64_t acc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) acc[u] = 0;  // (+0.0f, +0.0f)
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const int ch = lt + c * TEAM;
      if (ch < R) {
        if constexpr (QREG) {
#pragma unroll
          for (int u = 0; u < U; ++u) chunk_partial<T, METRIC>(buf[u][c], qv[c], acc[u], bp);
        } else {
          uint64_t q[VEC / 2];
          const ulonglong2* qp = reinterpret_cast<const ulonglong2*>(qs + ch * VEC);
#pragma unroll
          for (int e = 0; e < VEC / 4; ++e) {
            const ulonglong2 v = qp[e];
            q[2 * e] = v.x;
            q[2 * e + 1] = v.y;
          }
#pragma unroll
          for (int u = 0; u < U; ++u) chunk_partial<T, METRIC>(buf[u][c], q, acc[u], bp);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float s = f2_hsum(acc[u]);
#pragma unroll
      for (int off = TEAM / 2; off > 0; off >>= 1) s += __shfl_xor_sync(kFull, s, off, TEAM);
      const int i = r0 + u * NT + team;
      if (lt == 0 && i < nf) out[i] = make_key(s, id[u]);
    }
  }
}

template <typename T, int TEAM, int CPL, int U, bool QREG>
__device__ __forceinline__ void coop_dist_metric(
    int metric, float bp, const T* rows, int d_pad, const float* qs,
    const uint64_t (&qv)[QREG ? CPL : 1][Elems16<T>::n / 2], const uint32_t* ids, int nf,
    unsigned long long* out) {
  switch (metric) {
    case UHNSW_BASE_L1: coop_dist<T, TEAM, CPL, U, QREG, 1>(rows, d_pad, qs, qv, ids, nf, out, bp); break;
    case UHNSW_BASE_L2: coop_dist<T, TEAM, CPL, U, QREG, 2>(rows, d_pad, qs, qv, ids, nf, out, bp); break;
    case UHNSW_BASE_L05: coop_dist<T, TEAM, CPL, U, QREG, 3>(rows, d_pad, qs, qv, ids, nf, out, bp); break;
    case UHNSW_BASE_L15: coop_dist<T, TEAM, CPL, U, QREG, 4>(rows, d_pad, qs, qv, ids, nf, out, bp); break;
    default: coop_dist<T, TEAM, CPL, U, QREG, 5>(rows, d_pad, qs, qv, ids, nf, out, bp); break;
  }
}

// L_p sum of base row `id` by a team of 8 lanes, element order as in
// lp_sum_team_staged; four 32-dimension groups are loaded before they are summed,
// and the partial sum is tested against thr after each four.
__device__ __forceinline__ bool coop_lp_sum(const float* __restrict__ row, int d, int d_pad,
                                            const float* qs, float p, int pm, float thr,
                                            unsigned tmask, int lane8, float& S, int& groups) {
  const int G = (d + 31) >> 5;
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  float acc = 0.f;
  for (int g0 = 0; g0 < G; g0 += 4) {
    float4 x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = (g0 + u) * 32 + lane8 * 4;
      x[u] = j < d_pad ? __ldg(reinterpret_cast<const float4*>(row + j)) : z;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = (g0 + u) * 32 + lane8 * 4;
      if (g0 + u < G) {
        const float4 q = j < d_pad ? *reinterpret_cast<const float4*>(qs + j) : z;
        switch (pm) {
          case kPOne: acc = add_terms4<kPOne>(acc, x[u], q, p); break;
          case kPTwo: acc = add_terms4<kPTwo>(acc, x[u], q, p); break;
          case kPHalf: acc = add_terms4<kPHalf>(acc, x[u], q, p); break;
          case kPThreeHalves: acc = add_terms4<kPThreeHalves>(acc, x[u], q, p); break;
          default: acc = add_terms4<kPGeneral>(acc, x[u], q, p); break;
        }
      }
    }
    groups = min(g0 + 4, G);
    float tot = acc;
    tot += __shfl_xor_sync(tmask, tot, 1);
    tot += __shfl_xor_sync(tmask, tot, 2);
    tot += __shfl_xor_sync(tmask, tot, 4);
    S = tot;
    if (tot > thr) return false;
  }
  return true;
}

template <int NW>
__device__ __forceinline__ void coop_invalid(const QueryArgs& a, int64_t qi) {
  for (int j = threadIdx.x; j < a.k_max; j += (NW + 1) * 32) {
    a.out_ids[qi * a.k_max + j] = -1;
    a.out_dist[qi * a.k_max + j] = __int_as_float(0x7f800000);
  }
  if (threadIdx.x == 0) put_stats(a, qi, 0, 0, 0, 0, 0, UHNSW_EINVAL, 0, 0);
}

template <typename T, int TEAM, int CPL, int U, int NW, bool MANY>
__device__ void coop_query(const QueryArgs& a, int64_t qi, unsigned char* smem,
                           const CoopLayout& L) {
  constexpr int VEC = Elems16<T>::n;
  constexpr int THREADS = (NW + 1) * 32;
  constexpr bool QREG = CPL * VEC <= 16;
    constexpr bool AHEAD = NW >= 8;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool merger = warp == NW;
  const float kInf = __int_as_float(0x7f800000);
  float* qs = reinterpret_cast<float*>(smem + L.qs);
  unsigned long long* W = reinterpret_cast<unsigned long long*>(smem + L.W);
  int32_t* tab = reinterpret_cast<int32_t*>(smem + L.tab);
  unsigned long long* nk = reinterpret_cast<unsigned long long*>(smem + L.nk);
  unsigned long long* sk = reinterpret_cast<unsigned long long*>(smem + L.sk);
  uint32_t* wl = reinterpret_cast<uint32_t*>(smem + L.wl) + warp * 32;
  CoopPub* pub = reinterpret_cast<CoopPub*>(smem + L.pub);
  auto ckbuf = [&](int i) {
    return reinterpret_cast<unsigned long long*>(smem + (i ? L.ck1 : L.ck0));
  };

  const float p = a.p[qi];
  const int k = a.k ? a.k[qi] : a.k_max;
  const int ef = a.ef ? a.ef[qi] : a.ef_default;
  const Route rt = route_query(a, p);
  const bool direct = rt.direct;
  const int tq = query_t(a, qi);
  int tt = direct ? k : (tq > 0 ? tq : ef);
  if (tt < k) tt = k;
  const int cap = max(ef, tt);
  const GraphDev g = rt.slot == 0 ? a.g[0] : a.g[1];
  const bool ok = (p > 0.f) && (p <= 2.f) && k >= 1 && k <= a.k_max && ef >= 1 && tq >= 0 &&
                  cap <= a.ef_cap && g.ell0 != nullptr && a.width * g.deg0 <= a.cmax &&
                  g.deg <= a.cmax;
  if (!ok) {
    coop_invalid<NW>(a, qi);
    return;
  }
  const int d_ext = TEAM * CPL * VEC;
  for (int j = tid; j < d_ext; j += THREADS) qs[j] = j < a.d ? a.q[qi * a.d + j] : 0.f;
  const int hb = a.hash_bits, H = 1 << hb;
  for (int j = tid; j < H / 4; j += THREADS)
    reinterpret_cast<int4*>(tab)[j] = make_int4(kEmpty, kEmpty, kEmpty, kEmpty);
  __syncthreads();
  uint64_t qv[QREG ? CPL : 1][VEC / 2];
  if constexpr (QREG) {
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const ulonglong2* qp =
          reinterpret_cast<const ulonglong2*>(qs + (lane % TEAM + c * TEAM) * VEC);
#pragma unroll
      for (int e = 0; e < VEC / 4; ++e) {
        const ulonglong2 v = qp[e];
        qv[c][2 * e] = v.x;
        qv[c][2 * e + 1] = v.y;
      }
    }
  }
  const T* trav = reinterpret_cast<const T*>(a.trav);
  const int spw = a.cmax / NW;  // slots of one distance warp
  const int total = spw * NW, keys = (total + 63) / 64 * 64;
  for (int j = tid; j < 2 * keys; j += THREADS)  // the slots past `total` stay empty
    ckbuf(j >= keys)[j >= keys ? j - keys : j] = kNoKey;
  int nb = 1, nadj = 0, nexp = 0, nres = 0;
  int32_t* fresh_of = reinterpret_cast<int32_t*>(smem + L.cnt);  // [2][NW]: rows each warp found fresh
  // descent: upper row of each slot's candidate, one half for each parity of the hop
  int32_t* up_of = reinterpret_cast<int32_t*>(nk);

  // With many distance warps (`ahead`), the links of the parents that
  // will be next if this step's candidates are all behind them are read one
  // step early (they are next in 77 % of the steps at 1M x 128, ef 64).
  const bool ahead = AHEAD && spw <= 32;
  const int slot = warp * spw + lane;  // (ahead)
  const int slot_par = slot / g.deg0, slot_link = slot - slot_par * g.deg0;
  int32_t vnext = -1;                  // the early link of this slot
  uint32_t par_next = kIdMask;         // lane j: the parent vnext belongs to (kIdMask: none)

  // This warp's slots [b, b + 32) of a step, lane i holding slot b + i's link v
  // (-1: none): the fresh ones (layer0: those the visited table has not seen)
  // are summed into the first of them, the others emptied; returns their number.
  auto sum_slots = [&](int b, int32_t v, bool layer0, unsigned long long* out) {
    const int cnt = min(32, spw - b);
    unsigned long long* o = out + warp * spw + b;
    const bool fresh = v >= 0 && (!layer0 || hash_insert(tab, hb, v, a.err));
    const unsigned mask = __ballot_sync(kFull, fresh);
    const int nf = __popc(mask);
    if (fresh) wl[__popc(mask & lanemask_lt())] = (uint32_t)chk_idx(v, a.n, 1, a.err);
    if (lane >= nf && lane < cnt) o[lane] = kNoKey;
    __syncwarp();
    coop_dist_metric<T, TEAM, CPL, U, QREG>(rt.metric, rt.bp, trav, a.d_pad, qs, qv, wl, nf, o);
    __syncwarp();
    return nf;
  };

  // greedy descent from the entry point through the upper levels (beam 1)
  int ph = 0;
  __syncthreads();
  if (warp == 0) sum_slots(0, lane == 0 ? g.entry : -1, false, ckbuf(0));
  __syncthreads();
  unsigned long long curk = ckbuf(0)[0];
  int level = g.top_level;
  int32_t row = level >= 1 ? g.up_row[chk_idx(g.entry, a.n, 3, a.err)] : -1;
  bool early = false;  // vnext holds this hop's links
  const int64_t max_steps = ((int64_t)g.top_level + 1) * (a.n + 1) + 16;
  for (int64_t step = 0; level >= 1; ++step) {
    if (row < 0 || step >= max_steps) {  // a node above its own level, or a cycle
      if (tid == 0) set_error(a.err, row < 0 ? UHNSW_EINVAL : UHNSW_ECAPACITY);
      early = false;
      break;
    }
    ph ^= 1;
    if (!merger) {
      const int32_t* adj = g.up_adj + chk_idx((int64_t)row + level - 1, g.up_rows, 4, a.err) * g.deg;
      int nf = 0;
      for (int b = 0; b < spw; b += 32) {
        const int f = slot + b;
        int32_t v = -1;
        if (b + lane < spw && f < g.deg) v = early ? vnext : adj[f];
        if (ahead) {
          // if no link is nearer, the next hop is the same node a level below
          vnext = -1;
          if (lane < spw) {
            if (level > 1) {
              if (f < g.deg) vnext = adj[f - g.deg];
            } else if (f < g.deg0) {
              vnext = g.ell0[chk_idx(key_id(curk), a.n, 5, a.err) * g.deg0 + f];
            }
          }
        }
        const int32_t ur = v >= 0 ? g.up_row[chk_idx(v, a.n, 3, a.err)] : -1;
        nf += sum_slots(b, v, false, ckbuf(ph));
        const unsigned val = __ballot_sync(kFull, v >= 0);
        if (v >= 0)
          up_of[(ph ? total : 0) + warp * spw + b + __popc(val & lanemask_lt())] = ur;
      }
      if (lane == 0) fresh_of[ph * NW + warp] = nf;
    }
    __syncthreads();
    unsigned long long mn = kNoKey;
    int at = 0;
    for (int b = lane; b < total; b += 32) {
      const unsigned long long x = ckbuf(ph)[b];
      if (x < mn) {
        mn = x;
        at = b;
      }
    }
    nadj += 1;
    nb += (int)__reduce_add_sync(kFull, lane < NW ? (unsigned)fresh_of[ph * NW + lane] : 0u);
    const unsigned long long best = warp_min_key(mn);
    early = false;
    if (best < curk) {
      curk = best;
      at = __shfl_sync(kFull, at, __ffs(__ballot_sync(kFull, mn == best)) - 1);
      row = up_of[(ph ? total : 0) + at];
    } else {
      --level;
      early = ahead;
    }
  }

  // MANY: a warp that is done with the rows of its own links, and the merge warp after
  // its merge, takes rounds of the other warps' rows (posted: how many rows a warp
  // has, -1 before it knows; cursor: the next one to take; [2][NW] each, by the
  // step's parity, in the merge warp's link buffer, which has no other use).  A row's
  // key has its place whoever sums it, so that the candidates are the same.
  volatile int* posted = reinterpret_cast<volatile int*>(smem + L.wl) + NW * 32;
  int* cursor = reinterpret_cast<int*>(smem + L.wl) + NW * 32 + 2 * NW;
  if (MANY && tid < 2 * NW) {
    posted[tid] = -1;
    cursor[tid] = 0;
  }

  // layer-0 search from W = {cur}; its first parent is cur
  if (tid == 0) {
    hash_insert(tab, hb, (int32_t)key_id(curk), a.err);
    W[0] = curk | 1ull;
  }
  __syncthreads();
  int npar = 1, nWp = 0, jn = 0, hcount = 1;
  uint32_t par = key_id(curk);
  if (early && lane == 0) par_next = par;
  for (int64_t step = 0;; ++step) {
    if (step >= max_steps) {
      if (tid == 0) set_error(a.err, UHNSW_ECAPACITY);
      break;
    }
    nexp += npar;
    nadj += npar;
    if (merger) {
      if (step == 0) {
        CoopPub& po = pub[ph ^ 1];
        if (lane < 2 * a.width) {
          po.uk[lane] = kNoKey;
          po.pos[lane] = INT_MAX;
        }
        if (lane < a.width) {
          const int e = cap - 1 - lane;
          po.wl[lane] = e < 0 ? 0ull : e < 1 ? W[0] : kNoKey;
        }
        if (lane == 0) {
          po.bn = 1;
          po.last = cap == 1 ? W[0] : kNoKey;
        }
      } else {
        coop_merge_step(W, cap, a.width, ckbuf(ph), total, &pub[ph], &pub[ph ^ 1], nWp, jn, nk, sk);
      }
    }
    if (hcount > (H >> 1)) {
      // the table is past half full: refill it with W once the merge is done
      __syncthreads();
      hcount = pub[ph ^ 1].bn;
      for (int j = tid; j < H / 4; j += THREADS)
        reinterpret_cast<int4*>(tab)[j] = make_int4(kEmpty, kEmpty, kEmpty, kEmpty);
      __syncthreads();
      for (int j = tid; j < hcount; j += THREADS)
        hash_insert(tab, hb, (int32_t)key_id(W[j]), a.err);
      ++nres;
      __syncthreads();
    }
    if constexpr (MANY) {
      unsigned long long* out = ckbuf(ph ^ 1);
      const int at = (ph ^ 1) * NW;
      if (!merger) {
        const bool in = lane < spw && slot < npar * g.deg0;
        const int j = in ? slot / g.deg0 : 0;
        const uint32_t mine = __shfl_sync(kFull, par, j);
        const int32_t v =
            in ? g.ell0[chk_idx(mine, a.n, 5, a.err) * g.deg0 + (slot - j * g.deg0)] : -1;
        const bool fresh = v >= 0 && hash_insert(tab, hb, v, a.err);
        const unsigned mask = __ballot_sync(kFull, fresh);
        const int nf = __popc(mask);
        if (fresh) wl[__popc(mask & lanemask_lt())] = (uint32_t)chk_idx(v, a.n, 1, a.err);
        if (lane >= nf && lane < spw) out[warp * spw + lane] = kNoKey;
        __syncwarp();
        if (lane == 0) {
          fresh_of[at + warp] = nf;
          posted[ph * NW + warp] = -1;  // (the next step's)
          cursor[ph * NW + warp] = 0;
          __threadfence_block();
          posted[at + warp] = nf;
        }
        __syncwarp();
      }
      for (int i = 0; i < NW; ++i) {
        const int w = (warp + i) % NW;
        int n = lane == 0 ? posted[at + w] : 0;
        n = __shfl_sync(kFull, n, 0);
        __threadfence_block();
        const uint32_t* ids = reinterpret_cast<const uint32_t*>(smem + L.wl) + w * 32;
        constexpr int kRound = U * (32 / TEAM);
        while (n > 0) {
          int c = lane == 0 ? atomicAdd(&cursor[at + w], kRound) : 0;
          c = __shfl_sync(kFull, c, 0);
          if (c >= n) break;
          coop_dist_metric<T, TEAM, CPL, U, QREG>(rt.metric, rt.bp, trav, a.d_pad, qs, qv, ids + c,
                                                  min(kRound, n - c), out + w * spw + c);
        }
      }
    } else if (!merger) {
      unsigned long long* out = ckbuf(ph ^ 1);
      int nf = 0;
      if (ahead) {
        const uint32_t mine = __shfl_sync(kFull, par, slot_par & 31);
        const uint32_t was = __shfl_sync(kFull, par_next, slot_par & 31);
        int32_t v = -1;
        if (lane < spw && slot_par < npar)
          v = mine == was ? vnext : g.ell0[chk_idx(mine, a.n, 5, a.err) * g.deg0 + slot_link];
        // the parents after these, if no candidate of this step is nearer
        par_next = step > 0 && lane < a.width ? key_id(pub[ph].uk[nWp + lane]) : kIdMask;
        const uint32_t then = __shfl_sync(kFull, par_next, slot_par & 31);
        vnext = -1;
        if (lane < spw && slot_par < a.width && then != kIdMask)
          vnext = g.ell0[chk_idx(then, a.n, 5, a.err) * g.deg0 + slot_link];
        nf = sum_slots(0, v, true, out);
      } else {
        for (int b = 0; b < spw; b += 32) {
          const int f = slot + b;
          const bool in = b + lane < spw && f < npar * g.deg0;
          const int j = in ? f / g.deg0 : 0;
          const uint32_t mine = __shfl_sync(kFull, par, j);
          const int32_t v =
              in ? g.ell0[chk_idx(mine, a.n, 5, a.err) * g.deg0 + (f - j * g.deg0)] : -1;
          nf += sum_slots(b, v, true, out);
        }
      }
      if (lane == 0) fresh_of[(ph ^ 1) * NW + warp] = nf;
    }
    __syncthreads();
    ph ^= 1;
    const int m = (int)__reduce_add_sync(kFull, lane < NW ? (unsigned)fresh_of[ph * NW + lane] : 0u);
    npar = coop_select(ckbuf(ph), total, &pub[ph], a.width, cap, nWp, jn, par);
    nb += m;
    hcount += m;
    // no parent: no candidate of the last step can enter W either
    if (npar == 0) break;
  }
  const int bn = pub[ph].bn;

  // candidate set, verification and output (as warp_query)
  const bool reduced = !std::is_same<T, float>::value && !a.trav_exact;
  const int nc = (direct && reduced) ? bn : min(tt, bn);
  int64_t* oid = a.out_ids + qi * a.k_max;
  float* odist = a.out_dist + qi * a.k_max;
  if (direct && !reduced) {
    for (int j = tid; j < a.k_max; j += THREADS) {
      const bool have = j < k && j < bn;
      const unsigned long long x = have ? W[j] : 0ull;
      oid[j] = have ? (int64_t)key_id(x) : -1;
      odist[j] = have ? base_root(rt.metric, rt.bp, key_dist(x)) : kInf;
    }
    if (tid == 0) put_stats(a, qi, nb, 0, 0, nexp, nres, 0, rt.slot + 1, nadj);
    return;
  }
  uint32_t* C = reinterpret_cast<uint32_t*>(tab);
  unsigned long long* top = reinterpret_cast<unsigned long long*>(smem + L.td);
  int* vs = reinterpret_cast<int*>(smem + L.vs);  // [0] top length, [1] terms
  unsigned long long* vk = ckbuf(0);
  for (int j = tid; j < nc; j += THREADS) C[j] = key_id(W[j]);
  if (tid == 0) vs[1] = 0;
  __syncthreads();
  constexpr int NVT = THREADS / 8;
  const int team = tid >> 3, lane8 = tid & 7;
  const unsigned tmask = 0xffu << (lane & ~7);
  const int pm = pmode_of(p);
  const bool paper = !direct && a.mode == UHNSW_VERIFY_PAPER;
  const int kappa = a.kappa > 0 ? a.kappa : k;
  const float tau = query_tau(a, qi);
  int tn = 0, np = 0, terms = 0;
  for (int i = 0; i < nc;) {
    const int bend = !paper ? nc : i == 0 ? min(k, nc) : i + min(kappa, nc - i);  // (kappa may be INT_MAX)
    const bool batch = i > 0;
    if (batch) {
      for (int j = tid; j < tn; j += THREADS) top[j] |= 1ull;  // mark R
      __syncthreads();
    }
    for (int w0 = i; w0 < bend; w0 += NVT) {
      const float thr = (paper && !batch) || tn < k ? kInf : key_dist(top[k - 1]);
      const int c = w0 + team;
      unsigned long long key = kNoKey;
      if (c < bend) {
        const uint32_t id = (uint32_t)chk_idx(C[c], a.n, 2, a.err);
        float S = 0.f;
        int groups = 0;
        if (coop_lp_sum(a.base32 + (int64_t)id * a.d_pad, a.d, a.d_pad, qs, p, pm, thr, tmask,
                        lane8, S, groups))
          key = make_key(S, id);
        terms += lane8 == 0 ? min(groups * 32, a.d) : 0;
      }
      if (lane8 == 0) vk[team] = key;
      np += min(NVT, bend - w0);
      __syncthreads();
      if (warp == 0) {
        int at;
        const int n = coop_merge(top, tn, k, vk, NVT, tn == k ? top[k - 1] : kNoKey, 0, nk, sk, &at);
        if (lane == 0) vs[0] = n;
      }
      __syncthreads();
      tn = vs[0];
    }
    i = bend;
    if (batch) {
      int ov = 0;
      for (int j = lane; j < tn; j += 32) ov += (int)(top[j] & 1ull);
      ov = (int)__reduce_add_sync(kFull, (unsigned)ov);
      __syncthreads();
      for (int j = tid; j < tn; j += THREADS) top[j] &= ~1ull;
      __syncthreads();
      if ((float)ov / (float)k >= tau) break;
    }
  }
  for (int j = tid; j < a.k_max; j += THREADS) {
    const bool have = j < k && j < tn;
    oid[j] = have ? (int64_t)key_id(top[j]) : -1;
    odist[j] = have ? root_p(key_dist(top[j]), p) : kInf;
  }
  if (a.stats) {
    if (terms) atomicAdd(&vs[1], terms);
    __syncthreads();
    if (tid == 0) put_stats(a, qi, nb, np, vs[1], nexp, nres, 0, rt.slot + 1, nadj);
  }
}

// Blocks per SM asked of the register allocator where all queries are resident.
// Eight distance warps serve launches of at most one block per SM and take the
// registers they want: at 72 registers (3 blocks) the spills cost 2,403 against
// 1,779 cycles a merge.
template <int CPL, int NW>
struct CoopMinBlocks {
  static constexpr int value = NW >= 8    ? 1
                               : NW >= 4  ? (CPL <= 4 ? 4 : 2)
                               : CPL <= 3 ? 7
                               : CPL <= 4 ? 5
                                          : 3;
};

// The form for more queries than are resident (MANY), for rows whose sums are what
// a step takes: the warps of a block share a step's rows.  A link is fresh or not by
// chance, and a distance warp that finds few fresh ones, or the merge warp once it has
// merged, waited for the slowest (the barrier was 7.7 of the 17.7 cycles between two
// instructions of a warp at 200k x 200 FP32).  Two distance warps for rows of two chunks a lane and FP32 rows of four, four
// for longer ones (coop_warps in the host code).  10,000 queries, ms: this form;
// without the sharing; two distance warps without it; and the kernel before the
// cooperative one (four warps per query, each summing and merging in turn):
//   1M x 960 BF16, ef 512, k 100                         75.5, 107, 129, 103
//   the same rows, mixed k and ef, one launch            31.1, 43.9, 52.8, 52.8
//   the same, launches queued on two streams             31.9, 45.1, 54.0, 41.2
//   200k x 960 FP16, ef 64 and 300                       6.6, 6.6, 7.8, 10.8; 20.6, 19.6, 20.3, 37.4
//   100k x 800 FP32, ef 64 and 300                       11.4, 13.8, 20.7; 34.8, 43.1, 60.2
//   200k x 200 FP32, ef 64 and 300                       3.7, 4.2, 4.4, 3.6; 17.3, 19.9, 21.6, 17.9
// The 1M x 960 form then reads DRAM at 4.18 TB/s, 0.97 of the rate of random rows of
// that length.
// A block per SM more than CoopMinBlocks asks (72 registers) for 16-bit rows of four
// chunks: with four blocks the first row takes 83.5 ms.  Resident queries keep the
// registers of CoopMinBlocks (300 to 600 queries took 1.05 to 1.18 times as long).
template <typename T, int TEAM, int CPL, int NW>
constexpr bool coop_has_many() {
  constexpr bool f32 = std::is_same<T, float>::value;
  return TEAM == 32 &&
         (NW == 4 ? CPL == 8 || (CPL == 4 && !f32) : NW == 2 && (CPL == 2 || (CPL == 4 && f32)));
}
template <int CPL, int NW, bool MANY>
constexpr int kCoopBlocks = !MANY || NW == 2 ? CoopMinBlocks<CPL, NW>::value : CPL == 4 ? 5 : 4;

// One block of NW + 1 warps per query; a.queue_head set = persistent.
template <typename T, int TEAM, int CPL, int U, int NW, bool MANY>
__global__ void __launch_bounds__((NW + 1) * 32, (kCoopBlocks<CPL, NW, MANY>))
    uhnsw_csearch_kernel(const QueryArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int next;
  const CoopLayout L(TEAM * CPL * Elems16<T>::n, a.ef_cap, a.hash_bits, a.cmax, a.k_max, NW + 1);
  chain_begin(a);
  const bool fits = (uint32_t)L.total <= dynamic_smem_bytes();
  if (!fits && threadIdx.x == 0) set_error(a.err, UHNSW_ECAPACITY);
  int64_t qi = blockIdx.x;
  while (fits) {
    if (a.queue_head) {
      if (threadIdx.x == 0) {
        const int slot = atomicAdd(a.queue_head, 1);
        next = !a.qbucket ? slot : (slot < a.qbucket[1] ? a.qorder[a.qbucket[0] + slot] : (int)a.nq);
      }
      __syncthreads();
      qi = next;
    }
    if (qi >= a.nq) break;
    coop_query<T, TEAM, CPL, U, NW, MANY>(a, qi, smem, L);
    __syncthreads();
    if (!a.queue_head) break;
  }
  chain_end(a);
}

}  // namespace uhnsw_dev
