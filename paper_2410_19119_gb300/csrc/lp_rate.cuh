// Device code of the rating and approval steps, shared by the kernels of
// lp.cu (a launch per step) and lp_small.cu (all rounds of a small level in
// one launch). Included by exactly these two; everything has internal linkage.
#pragma once
#include <algorithm>

#include "decode.cuh"
#include "select.cuh"

namespace tp {

namespace {

enum Mode { M_LP = 0, M_FAV = 1, M_REBAL = 2 };

constexpr int kSmallLog = 7;   // 128 slots
constexpr int kMidSmallLog = 9;  // 512 slots: mid tier, degree <= kMidSplit = 256
constexpr int kMidLog = 10;    // 1024 slots: mid tier, degree <= 512
constexpr int kHugeLog = 11;   // 2048 slots: one 1000-neighbour chunk of a hub
constexpr int kMidWarps = 4;

struct RateCtx {
  GView g;
  const uint8_t *tier;
  const int32_t *label;
  const int64_t *lw;
  int64_t cap;
  int64_t nlabels;
  uint64_t rk;
  const uint64_t *rk_dev;  // if set, the round key is read here (replayed round graphs)
  int32_t S, s;
  int32_t slack;  // warp tiers: table slots per neighbour (power of two)
  // M_LP outputs
  int32_t *mv_u, *mv_t, *mv_o;
  int64_t *mv_g;
  int64_t *in_w;
  unsigned long long *counters;
  // M_FAV output
  int32_t *fav;
  // M_REBAL (batched graphs: rb_best and blk_of hold one entry per graph)
  int32_t blk;
  int64_t *rb_loss;
  int32_t *rb_t;
  long long *rb_best;
  const int32_t *blk_of;
  // labels are blocks: how many (one graph; batched graphs have seg.k), and
  // the most of any graph (0: labels are clusters)
  int32_t k, kmax;
  // batched graphs (seg.gid == null: one graph)
  SegLp seg;
  // lists and global tables
  const int32_t *list;
  int64_t list_n;
  int32_t *tkeys;
  int64_t *tvals;
  int32_t *tlist, *tcount;  // filled slots per huge table
  const int64_t *toff;
  const int32_t *tcap;
  int64_t tbase;  // slot offset of this tier's tables inside tkeys/tvals
  const int64_t *chunk_start;
  int64_t n_chunks;
  const int64_t *seg_start;  // huge tables: prefix of segment counts
  int64_t n_segs;
  // lane tier in LP mode: this round's buckets (null: hash every vertex);
  // sub-round s holds bucket[bucket_off[s * nb] .. bucket_off[(s + 1) * nb])
  const int32_t *bucket;
  const int64_t *bucket_off;
  int64_t bucket_nb;
  int32_t lane_win;  // vertices of a warp's window (32 .. kLaneWin)
  // per listed vertex: record start << 8 | record length (compressed graphs)
  const uint64_t *bucket_rec;
  // quiet[u] == *epoch: u's last rating found no label better than its own and
  // no neighbour has moved since, so it need not be rated (k_rate_lane_quiet)
  uint8_t *quiet;
  const int32_t *epoch;
  // this round's sub-round + 1 of every vertex (null: hash on the fly)
  const uint8_t *sub_byte;
  // bucket mode of the warp/block tiers: this tier's list positions grouped
  // by sub-round (null: scan the whole list and test each vertex)
  const int32_t *bpos;
  const int64_t *boff;  // this tier's S + 1 offsets into bpos
  // huge tier in bucket mode: prefix of chunk / segment counts over bpos and
  // the items (hub position << 32 | chunk or segment index)
  const int64_t *hc_pre, *hs_pre, *hc_item, *hs_item;
  // all tiers' buckets (rate_tiers slices them per tier)
  const int32_t *tb_pos;
  const int64_t *tb_off;
  int64_t tb_base[LpWork::kTiers];
};

// Range of list entries (bucket mode: of bpos) a tier kernel walks.
__device__ __forceinline__ void tier_range(const RateCtx &c, int64_t &b, int64_t &e) {
  if (c.bpos) b = c.boff[c.s], e = c.boff[c.s + 1];
  else b = 0, e = c.list_n;
}
// List position of entry k and whether its vertex is active this sub-round.
template <int MODE>
__device__ __forceinline__ bool tier_entry(const RateCtx &c, int64_t k, int64_t &pos, int64_t &u);

__device__ __forceinline__ int64_t node_w(const GView &g, int64_t u) { return g.vw ? g.vw[u] : 1; }

__device__ __forceinline__ uint64_t rk_of(const RateCtx &c) { return c.rk_dev ? *c.rk_dev : c.rk; }

// Batched graphs: u's number inside its own graph, its cap, and the
// favourite key of a vertex without favourite (one per graph).
__device__ __forceinline__ int64_t local_id(const RateCtx &c, int64_t u) {
  return c.seg.gid ? u - c.seg.vb[c.seg.gid[u]] : u;
}
__device__ __forceinline__ int64_t cap_of(const RateCtx &c, int64_t u) {
  return c.seg.gid ? c.seg.cap[c.seg.gid[u]] : c.cap;
}
__device__ __forceinline__ int32_t no_fav(const RateCtx &c, int64_t u) {
  return (int32_t)(c.g.n + (c.seg.gid ? c.seg.gid[u] : 0));
}

// Blocks of u's graph: labels lb .. lb + k - 1 (direct tables, rebalancing).
__device__ __forceinline__ int32_t block_range(const RateCtx &c, int64_t u, int32_t &lb) {
  if (!c.seg.gid) {
    lb = 0;
    return c.k;
  }
  const int32_t g = c.seg.gid[u];
  lb = (int32_t)c.seg.lb[g];
  return c.seg.k[g];
}

template <int MODE>
__device__ __forceinline__ bool active(const RateCtx &c, int64_t u) {
  if (MODE == M_LP)
    return c.sub_byte ? c.sub_byte[u] == c.s + 1
                      : sub_round_of(hstep(rk_of(c), (uint64_t)local_id(c, u)), c.S) == c.s;
  if (MODE == M_FAV) return c.label[u] == u && c.lw[u] == node_w(c.g, u);
  return c.label[u] == (c.blk_of ? c.blk_of[c.seg.gid[u]] : c.blk);
}

template <int MODE>
__device__ __forceinline__ bool tier_entry(const RateCtx &c, int64_t k, int64_t &pos, int64_t &u) {
  pos = c.bpos ? c.bpos[k] : k;
  u = c.list[pos];
  return c.bpos ? true : active<MODE>(c, u);
}

// The tie order of vertex u: tie_of(k, x) is the tie hash of label x as u's
// graph numbers it (its label base folded into the additive constant, so
// (x - base) + gamma costs one add, as x + gamma does for one graph).
struct TieKey {
  uint64_t hv, add;
};
__device__ __forceinline__ uint32_t tie_of(const TieKey &k, int32_t x) {
  return (uint32_t)(mix64(k.hv ^ ((uint64_t)(int64_t)x + k.add)) >> 32);
}
template <int MODE>
__device__ __forceinline__ TieKey tie_key(const RateCtx &c, int64_t u) {
  if (MODE == M_REBAL) return TieKey{0, 0};
  int64_t vb = 0, lb = 0;
  if (c.seg.gid) {
    const int32_t g = c.seg.gid[u];
    vb = c.seg.vb[g];
    lb = c.seg.lb[g];
  }
  return TieKey{hstep(hstep(rk_of(c), (uint64_t)(u - vb)), kTagTie), kGamma - (uint64_t)lb};
}
// The lane tier decides batched graphs at compile time (SEG), so the one-graph
// kernels carry no per-graph lookups in their tight register budget.
template <bool SEG>
__device__ __forceinline__ int64_t lane_cap(const RateCtx &c, int64_t u) {
  return SEG ? c.seg.cap[c.seg.gid[u]] : c.cap;
}
template <int MODE, bool SEG>
__device__ __forceinline__ TieKey lane_tie_key(const RateCtx &c, int64_t u) {
  if (SEG) return tie_key<MODE>(c, u);
  return TieKey{hstep(hstep(rk_of(c), (uint64_t)u), kTagTie), kGamma};
}

__device__ __forceinline__ uint32_t slot_of(int32_t x, int logcap) {
  return ((uint32_t)x * 0x9E3779B1u) >> (32 - logcap);
}

// Adds w to the rating of label x (open addressing, linear probing); V is
// int64_t, or uint32_t where ratings are counts (unit weights).
template <class V>
__device__ __forceinline__ void tbl_add(int32_t *keys, V *vals, int logcap, int32_t x, int64_t w,
                                        int32_t *err) {
  uint32_t mask = (1u << logcap) - 1u, h = slot_of(x, logcap);
  for (uint32_t probe = 0; probe <= mask; ++probe, h = (h + 1) & mask) {
    int32_t k = *(volatile int32_t *)&keys[h];
    if (k == -1) {
      int32_t prev = atomicCAS(&keys[h], -1, x);
      k = prev == -1 ? x : prev;
    }
    if (k == x) {
      if constexpr (sizeof(V) == 8) atomicAdd((unsigned long long *)&vals[h], (unsigned long long)w);
      else atomicAdd((unsigned int *)&vals[h], (unsigned int)w);
      return;
    }
  }
  latch_error(err, TP_ERR_CORRUPT);  // more distinct labels than the degree allows
}

struct Best {
  int64_t r;
  uint32_t t;
  int32_t x;
  int64_t rown;
  __device__ __forceinline__ void init() { r = -1, t = 0xffffffffu, x = INT32_MAX, rown = 0; }
};

__device__ __forceinline__ void warp_reduce_best(Best &b) {
  warp_best(b.r, b.t, b.x);
  b.rown = warp_max(b.rown);
}

// Per-warp buffer of mover records, flushed with one atomic per 32 movers.
struct MoverBuf {
  int32_t *u, *t, *o;
  int64_t *gain;
  int cnt;
};

__device__ __forceinline__ void flush_movers(const RateCtx &c, MoverBuf &mb) {
  __syncwarp();
  if (mb.cnt == 0) return;
  unsigned long long base = 0;
  if (lane_id() == 0) base = atomicAdd(c.counters, (unsigned long long)mb.cnt);
  base = __shfl_sync(kFull, base, 0);
  int l = lane_id();
  if (l < mb.cnt) {
    c.mv_u[base + l] = mb.u[l];
    c.mv_t[base + l] = mb.t[l];
    c.mv_o[base + l] = mb.o[l];
    c.mv_g[base + l] = mb.gain[l];
  }
  mb.cnt = 0;
  __syncwarp();
}

// Acts on the (warp-uniform) decision for vertex u.
template <int MODE>
__device__ __forceinline__ void finalize_warp(const RateCtx &c, const Best &b, int64_t u, int64_t cu,
                                              MoverBuf *mb) {
  int lane = lane_id();
  if (MODE == M_LP) {
    if (b.r > b.rown) {
      if (lane == 0) {
        mb->u[mb->cnt] = (int32_t)u;
        mb->t[mb->cnt] = b.x;
        mb->o[mb->cnt] = c.label[u];
        mb->gain[mb->cnt] = b.r - b.rown;
        atomicAdd((unsigned long long *)&c.in_w[b.x], (unsigned long long)cu);
      }
      if (++mb->cnt == 32) flush_movers(c, *mb);
    }
  } else if (MODE == M_FAV) {
    if (lane == 0) c.fav[u] = b.r > 0 ? b.x : no_fav(c, u);
  } else {
    int32_t lb;
    const int32_t k = block_range(c, u, lb);
    int32_t blk = c.blk;
    long long *best = c.rb_best;
    if (c.seg.gid) {
      const int32_t g = c.seg.gid[u];
      blk = c.blk_of[g];
      best += g;
    }
    const int64_t cap = cap_of(c, u);
    int32_t tz = -1;
    if (b.r <= 0) {  // no admissible neighbouring block: smallest admissible block
      for (int32_t base = 0; base < k && tz < 0; base += 32) {
        int32_t t = lb + base + lane;
        bool ok = base + lane < k && t != blk && c.lw[t] + cu <= cap;
        unsigned m = __ballot_sync(kFull, ok);
        if (m) tz = lb + base + __ffs(m) - 1;
      }
    }
    if (lane == 0) {
      int32_t tt = b.r > 0 ? b.x : tz;
      c.rb_t[u] = tt;
      if (tt >= 0) {
        int64_t loss = b.rown - (b.r > 0 ? b.r : 0);
        c.rb_loss[u] = loss;
        atomicMin(best, (long long)loss);
      }
    }
  }
}

// Adds the labels of u's neighbours to a warp's table: add(label, weight).
// CSR rows are read 128 entries a step, all loads of a kind issued before the
// first is used, so a row costs two round trips (entries, then labels) per
// 128 neighbours. SHORT: rows of up to 32 are common (the small tier), and take
// one load without the other three's tests, which cost a level of 524 288
// vertices of degree 12 with wide weights an eighth (4.4 against 3.9 ms); where
// rows are long this test costs 1-2%.
template <bool COMP, bool SHORT = false, class F>
__device__ __forceinline__ void warp_labels(const RateCtx &c, int64_t u, F &&add,
                                            const ZipNbr *z = nullptr) {
  if constexpr (COMP) {
    warp_neighbours<true>(
        c.g, u, -1,
        [&](bool has, int32_t v, int64_t w, int64_t) {
          if (has) add(c.label[v], w);
        },
        z);
  } else {
    const int64_t b = c.g.xadj[u], e = c.g.xadj[u + 1];
    if (SHORT && e - b <= 32) {
      const int64_t i = b + lane_id();
      if (i < e) {
        const int32_t v = __ldcs(c.g.adj + i);
        const int64_t w = c.g.ew ? __ldcs(c.g.ew + i) : 1;
        add(c.label[v], w);
      }
      return;
    }
    for (int64_t i = b + lane_id(); i - lane_id() < e; i += 128) {
      int32_t v[4], x[4];
      int64_t w[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const bool in = i + 32 * r < e;
        v[r] = in ? __ldcs(c.g.adj + i + 32 * r) : -1;
        w[r] = in && c.g.ew ? __ldcs(c.g.ew + i + 32 * r) : 1;
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) x[r] = v[r] >= 0 ? c.label[v[r]] : -1;
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (x[r] >= 0) add(x[r], w[r]);
    }
  }
}

// Picks u's label from a warp's filled table: slot(i, x, R) gives the label
// (negative: none) and rating of slot i < cap. The scan takes two passes: the
// top rating among the other labels (and the own rating), then the tie order
// among the labels at that rating only, so tie hashes are formed for tied
// candidates alone; in LP mode a vertex whose top rating does not beat its
// own cannot move and skips the second pass.
template <int MODE, class Slot>
__device__ __forceinline__ Best pick_warp(const RateCtx &c, int64_t u, int64_t cu, int cap,
                                          Slot &&slot) {
  const int lane = lane_id();
  const int32_t own = c.label[u];
  const int64_t capu = cap_of(c, u);
  int64_t rmax = -1, rown = 0;
  for (int i = lane; i < cap; i += 32) {
    int32_t x;
    int64_t R;
    slot(i, x, R);
    if (x < 0) continue;
    if (x == own) rown = R;
    else rmax = R > rmax ? R : rmax;
  }
  rmax = warp_max(rmax);
  rown = warp_max(rown);
  Best b;
  b.init();
  b.rown = rown;
  if (rmax >= 0 && (MODE != M_LP || rmax > rown)) {
    const TieKey hv = tie_key<MODE>(c, u);
    // the best label ignoring the cap: the top-rated one first in tie order
    for (int i = lane; i < cap; i += 32) {
      int32_t x;
      int64_t R;
      slot(i, x, R);
      if (x < 0 || x == own || R != rmax) continue;
      const uint32_t t = MODE == M_REBAL ? 0u : tie_of(hv, x);
      if (better(rmax, t, x, b.r, b.t, b.x)) b.r = rmax, b.t = t, b.x = x;
    }
    warp_best(b.r, b.t, b.x);
    // the winner is full: the best admissible label instead (for a move it
    // must also improve on the own rating)
    if (MODE != M_FAV && b.x != INT32_MAX && c.lw[b.x] + cu > capu) {
      b.init();
      for (int i = lane; i < cap; i += 32) {
        int32_t x;
        int64_t R;
        slot(i, x, R);
        if (x < 0 || x == own) continue;
        if (MODE == M_LP && R <= rown) continue;
        const uint32_t t = MODE == M_REBAL ? 0u : tie_of(hv, x);
        if (better(R, t, x, b.r, b.t, b.x) && c.lw[x] + cu <= capu) b.r = R, b.t = t, b.x = x;
      }
      warp_best(b.r, b.t, b.x);
      b.rown = rown;
    }
  }
  return b;
}

// Rates vertex u with one warp; the hash table must be empty on entry and is
// empty again on exit.
template <bool COMP, int MODE, class V, bool SHORT = false>
__device__ __forceinline__ void rate_vertex_warp(const RateCtx &c, int64_t u, int32_t *keys,
                                                 V *vals, int logcap, MoverBuf *mb,
                                                 const ZipNbr *z = nullptr) {
  // every lane adds its neighbour's label to the table (shared-memory
  // atomics are far cheaper than grouping equal labels across lanes first)
  warp_labels<COMP, SHORT>(c, u, [&](int32_t x, int64_t w) {
    tbl_add<V>(keys, vals, logcap, x, w, c.g.err);
  }, z);
  __syncwarp();
  __threadfence_block();
  const int cap = 1 << logcap;
  const int64_t cu = node_w(c.g, u);
  const Best b = pick_warp<MODE>(c, u, cu, cap, [&](int i, int32_t &x, int64_t &R) {
    x = keys[i];
    R = (int64_t)vals[i];
  });
  for (int i = lane_id(); i < cap; i += 32) keys[i] = -1, vals[i] = 0;
  __syncwarp();
  finalize_warp<MODE>(c, b, u, cu, mb);
}

// Degree of u, and (compressed) the layout of its record for the decoder.
template <bool COMP>
__device__ __forceinline__ int64_t row_degree(const GView &g, int64_t u, ZipNbr &z) {
  if (!COMP) return g.xadj[u + 1] - g.xadj[u];
  z = zip_nbr(g, u);
  return z.deg;
}

// Warp tiers: the table of a degree-d vertex uses the first 2^lc slots,
// the least power of two >= slack * d (at least 32, at most 2^maxlog); only
// those are scanned and cleared.
__device__ __forceinline__ int table_log(const RateCtx &c, int64_t d, int maxlog) {
  int lc = 5;
  while (lc < maxlog && ((int64_t)1 << lc) < c.slack * d) ++lc;
  return lc;
}

// Shared memory per warp: table keys + values, then the mover buffer.
template <int LOG, class V = int64_t>
struct WarpSmem {
  int32_t keys[1 << LOG];
  V vals[1 << LOG];
  int32_t mu[32], mt[32], mo[32];
  int64_t mg[32];
};

template <int LOG, class V>
__device__ __forceinline__ void init_table(WarpSmem<LOG, V> &w) {
  for (int i = lane_id(); i < (1 << LOG); i += 32) w.keys[i] = -1, w.vals[i] = 0;
  __syncwarp();
}

// ---------------------------------------------------------------- lane tier
// Low-degree vertices, one lane per vertex, so a warp keeps 32
// neighbourhoods in flight. Each warp step:
//   1. takes a window of up to 128 active vertices (this sub-round's bucket
//      list, or a scan of 256-vertex slabs) and rates it as four batches of
//      32 in list order;
//   2. per batch, every lane loads its compressed record at once (five
//      16-byte groups; the next batch's records are prefetched to L2
//      meanwhile) and decodes it a 32-bit word at a time into its column of
//      shared memory; the gaps are then summed into neighbour ids while the
//      label gathers are issued, all of them before the first is used (CSR:
//      the adjacency entries directly);
//   3. the labels are sorted with Batcher's odd-even merge network of 16 or
//      32 elements (picked per batch), so equal labels form runs whose
//      lengths (summed weights) are the ratings;
//   4. only the candidates tied at the top rating are hashed for the tie
//      order; the cap is checked for the winner only, with a scan over all
//      admissible candidates when the winner is full;
//   5. the window's movers are collected in shared memory and written out
//      with one atomic per window.
constexpr int kLaneWarps = 8;
constexpr int kLaneBlocksPerSM = 3;
constexpr int kLaneWin = 128;             // vertices per warp step
constexpr int kLaneQueue = kLaneWin + 32;  // slab scans append 32 at a time

struct LaneCand {
  int32_t r;
  uint32_t t;
  int32_t x;
};

__device__ __forceinline__ bool lane_better(const LaneCand &a, const LaneCand &b) {
  return better(a.r, a.t, a.x, b.r, b.t, b.x);
}

// Record range of a compressed lane-tier vertex: from the bucket list when
// it carries the ranges (coalesced with the vertex ids), else the offsets.
__device__ __forceinline__ void lane_record(const GView &g, const uint64_t *rec, int64_t pos,
                                            int32_t u, uint64_t &b, uint64_t &e) {
  if (rec) {
    const uint64_t r = rec[pos];
    b = r >> 8;
    e = b + (r & 255u);
  } else {
    b = off_at(g, u);
    e = off_at(g, u + 1);
  }
}

template <bool COMP>
__device__ __forceinline__ void lane_prefetch(const GView &g, const uint64_t *rec, int64_t pos,
                                              int64_t u) {
  if (COMP) {
    uint64_t b, e;
    lane_record(g, rec, pos, (int32_t)u, b, e);
    prefetch_l2(g.bytes + b);
    prefetch_l2(g.bytes + e);
  } else {
    const int64_t b = g.xadj[u], e = g.xadj[u + 1];
    if (e > b) {
      prefetch_l2(g.adj + b);
      prefetch_l2(g.adj + e - 1);
    }
  }
}

// Batcher's odd-even merge sort of a[0..N), ascending (63 comparators for 16
// elements, 191 for 32), registers only. The network
// is generated by template recursion so every index is a constant.
template <class T>
__device__ __forceinline__ void cmp_swap(T &x, T &y) {
  const T lo = min(x, y), hi = max(x, y);
  x = lo;
  y = hi;
}

// Merges the two sorted halves of the subsequence a[LO], a[LO + R], ...
template <int LO, int N, int R, class T>
__device__ __forceinline__ void oem_merge(T (&a)[kLaneMaxDeg]) {
  constexpr int M = 2 * R;
  if constexpr (M < N) {
    oem_merge<LO, N, M>(a);
    oem_merge<LO + R, N, M>(a);
#pragma unroll
    for (int i = LO + R; i + R < LO + N; i += M) cmp_swap(a[i], a[i + R]);
  } else {
    cmp_swap(a[LO], a[LO + R]);
  }
}

// N: 8, 16 or 32. (A network of 24, 32 without its last quarter, fits half of
// the batches of a mesh of average degree 16, but a further size beside the
// others cost the compressed kernel 15.0 -> 18.5 ms over 80 launches and the
// CSR kernel 3.36 -> 3.93 ms for a round of 2^24 vertices.)
template <int LO, int N, class T>
__device__ __forceinline__ void oem_sort_range(T (&a)[kLaneMaxDeg]) {
  if constexpr (N > 1) {
    oem_sort_range<LO, N / 2>(a);
    oem_sort_range<LO + N / 2, N / 2>(a);
    oem_merge<LO, N, 1>(a);
  }
}

template <int N, class T>
__device__ __forceinline__ void oem_sort(T (&a)[kLaneMaxDeg]) {
  oem_sort_range<0, N>(a);
}

// Mover records of one batch.
struct BatchMovers {
  int32_t u[32], t[32], o[32], g[32];
};

// Mover records of one warp's window, written out with one atomic per window.
struct LaneMovers {
  int32_t u[kLaneWin], t[kLaneWin], o[kLaneWin], g[kLaneWin];
};

// Emits the favourite (two-hop mode) or queues the move of this lane's
// vertex in the warp's buffer (nmv records so far, warp-uniform).
template <int MODE, class Movers>
__device__ __forceinline__ void emit_lane(const RateCtx &c, bool has, int32_t u, int32_t own,
                                          int32_t rown, int64_t cu, const LaneCand &best,
                                          Movers &mb, int &nmv) {
  if (MODE == M_FAV) {
    if (has) c.fav[u] = best.r > 0 ? best.x : no_fav(c, u);
  } else {
    const bool mv = has && best.r > rown;
    const unsigned mm = __ballot_sync(kFull, mv);
    if (mv) {
      const int at = nmv + __popc(mm & lanemask_lt());
      mb.u[at] = u;
      mb.t[at] = best.x;
      mb.o[at] = own;
      mb.g[at] = best.r - rown;
      atomicAdd((unsigned long long *)&c.in_w[best.x], (unsigned long long)cu);
    }
    nmv += __popc(mm);
  }
}

// LIVE: labels change while the kernel runs (k_lp_small), so they are not read
// through the read-only path.
template <bool LIVE>
__device__ __forceinline__ int32_t load_label(const int32_t *p) {
  return LIVE ? *p : __ldg(p);
}

// Labels below this fit a 32-bit sort key with the slot (weighted lane tier).
constexpr int64_t kLaneKeyLabels = ((int64_t)1 << 27) - 1;

// Rates one batch: this lane's vertex u with deg neighbours (compressed:
// already decoded into the column; CSR: adjacency from xadj[u]) and emits
// the favourite, or queues the move in the warp's window buffer (nmv
// records so far, warp-uniform). N >= the largest degree of the batch.
// WIDE (weighted): labels beyond kLaneKeyLabels, sorted with the weights in
// 64-bit keys.
// QUIET: vertices without a better label are marked quiet.
template <bool COMP, int MODE, bool W, int N, bool SEG, bool LIVE = false, bool WIDE = false,
          bool QUIET = false, class Movers>
__device__ __forceinline__ void lane_batch(const RateCtx &c, bool has, int32_t u, int deg,
                                           uint32_t *col, uint32_t *wcol, uint8_t *cnt,
                                           Movers &mb, int &nmv) {
  const int32_t own = has ? c.label[u] : -1;
  int32_t rown = 0, rmax = 0;
  int32_t *ccol = reinterpret_cast<int32_t *>(col);
  if constexpr (W) {  // weighted levels are CSR; candidates listed in the column
    const int64_t b = has ? c.g.xadj[u] : 0;
    const int32_t *adj = c.g.adj + b;
    const int64_t *ew = c.g.ew + b;
    int ncand = 0;
    uint32_t run = 0;
    // one sorted entry: label x (INT32_MAX: padding), its weight, and whether
    // it is the last of its label
    auto step = [&](int32_t x, uint32_t wt, bool end) {
      run += wt;
      const bool real = end && x != INT32_MAX;
      const bool cand = real && x != own;
      ccol[ncand * 32] = x;
      wcol[ncand * 32] = run;
      rown = real && !cand ? (int32_t)run : rown;
      rmax = cand ? max(rmax, (int32_t)run) : rmax;
      ncand += cand;
      run = end ? 0u : run;
    };
    if constexpr (WIDE) {  // label << 32 | weight; padding: label INT32_MAX, weight 0
      uint64_t a[kLaneMaxDeg];
#pragma unroll
      for (int i = 0; i < N; ++i)
        a[i] = i < deg ? ((uint64_t)(uint32_t)load_label<LIVE>(c.label + __ldcs(adj + i)) << 32) |
                             (uint32_t)__ldcs(ew + i)
                       : (uint64_t)INT32_MAX << 32;
      oem_sort<N>(a);
#pragma unroll
      for (int i = 0; i < N; ++i)
        step((int32_t)(a[i] >> 32), (uint32_t)a[i],
             i + 1 == N || (int32_t)(a[i + 1] >> 32) != (int32_t)(a[i] >> 32));
    } else {
      // label << 5 | slot, the weights apart in the lane's column: a comparator
      // of the sort is two instructions instead of six on 64-bit pairs
      uint32_t a[kLaneMaxDeg], wt[kLaneMaxDeg];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        a[i] = i < deg ? (uint32_t)load_label<LIVE>(c.label + __ldcs(adj + i)) << 5 | (uint32_t)i
                       : 0xffffffffu;
        wcol[i * 32] = i < deg ? (uint32_t)__ldcs(ew + i) : 0u;
      }
      oem_sort<N>(a);
#pragma unroll
      for (int i = 0; i < N; ++i) wt[i] = a[i] == 0xffffffffu ? 0u : wcol[(a[i] & 31u) * 32];
#pragma unroll
      for (int i = 0; i < N; ++i)
        step(a[i] == 0xffffffffu ? INT32_MAX : (int32_t)(a[i] >> 5), wt[i],
             i + 1 == N || a[i + 1] >> 5 != a[i] >> 5);
    }
    const int64_t cu = has ? node_w(c.g, u) : 1;
    LaneCand best{-1, 0xffffffffu, INT32_MAX};
    if (MODE == M_FAV ? rmax > 0 : rmax > rown) {
      const TieKey hv = lane_tie_key<MODE, SEG>(c, u);
      const int64_t capu = lane_cap<SEG>(c, u);
      // the best candidate overall is tied at the top rating
      LaneCand b1{-1, 0xffffffffu, INT32_MAX};
      for (int k = 0; k < ncand; ++k) {
        if ((int32_t)wcol[k * 32] != rmax) continue;
        const int32_t x = ccol[k * 32];
        const LaneCand cand{rmax, tie_of(hv, x), x};
        if (lane_better(cand, b1)) b1 = cand;
      }
      if (MODE == M_FAV || c.lw[b1.x] + cu <= capu) {
        best = b1;
      } else {
        // the winner is full: the best admissible candidate that improves
        for (int k = 0; k < ncand; ++k) {
          const int32_t r = (int32_t)wcol[k * 32];
          const int32_t x = ccol[k * 32];
          if (r <= rown || x == b1.x) continue;
          const LaneCand cand{r, tie_of(hv, x), x};
          if (lane_better(cand, best) && c.lw[x] + cu <= capu) best = cand;
        }
      }
    }
    if (QUIET && has && rmax <= rown) c.quiet[u] = (uint8_t)*c.epoch;
    emit_lane<MODE>(c, has, u, own, rown, cu, best, mb, nmv);
  } else if constexpr (COMP) {
    // compressed, unit weights: the sorted runs become a list of (label,
    // rating) candidates in the lane's column; the decoder already keeps the
    // ALU pipe busy, and listing takes fewer instructions than walking the
    // runs when many labels tie (the first rounds)
    int32_t a[kLaneMaxDeg];
    {
      // raw values -> neighbour ids (first: signed offset from u, then gaps)
      const uint32_t nmax = (uint32_t)(c.g.n - 1);
      int32_t prev = u;
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const uint32_t v = col[i * 32];
        int32_t x = i == 0 ? ((v & 1u) ? u - (int32_t)(v >> 1) : u + (int32_t)(v >> 1))
                           : prev + (int32_t)v;
        // streams are validated on creation; the clamp only keeps a
        // corrupted one from reading out of bounds
        x = (int32_t)min((uint32_t)x, nmax);
        prev = x;
        a[i] = i < deg ? load_label<LIVE>(c.label + x) : INT32_MAX;
      }
    }
    oem_sort<N>(a);
    // branch-free run scan: every position writes slot ncand, which only
    // advances past a candidate (later writes overwrite the others)
    int ncand = 0, start = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const bool end = i + 1 == N || a[i + 1] != a[i];
      const int32_t run = i + 1 - start;
      const bool real = end && a[i] != INT32_MAX;
      const bool cand = real && a[i] != own;
      ccol[ncand * 32] = a[i];
      cnt[ncand * 32] = (uint8_t)run;
      rown = real && !cand ? run : rown;
      rmax = cand ? max(rmax, run) : rmax;
      ncand += cand;
      start = end ? i + 1 : start;
    }
    const int64_t cu = has ? node_w(c.g, u) : 1;
    LaneCand best{-1, 0xffffffffu, INT32_MAX};
    if (MODE == M_FAV ? rmax > 0 : rmax > rown) {
      const TieKey hv = lane_tie_key<MODE, SEG>(c, u);
      const int64_t capu = lane_cap<SEG>(c, u);
      // the best candidate overall is tied at the top rating
      LaneCand b1{-1, 0xffffffffu, INT32_MAX};
      for (int k = 0; k < ncand; ++k) {
        if ((int32_t)cnt[k * 32] != rmax) continue;
        const int32_t x = ccol[k * 32];
        const LaneCand cand{rmax, tie_of(hv, x), x};
        if (lane_better(cand, b1)) b1 = cand;
      }
      if (MODE == M_FAV || c.lw[b1.x] + cu <= capu) {
        best = b1;
      } else {
        // the winner is full: the best admissible candidate that improves
        for (int k = 0; k < ncand; ++k) {
          const int32_t r = (int32_t)cnt[k * 32];
          const int32_t x = ccol[k * 32];
          if (r <= rown || x == b1.x) continue;
          const LaneCand cand{r, tie_of(hv, x), x};
          if (lane_better(cand, best) && c.lw[x] + cu <= capu) best = cand;
        }
      }
    }
    if (QUIET && has && rmax <= rown) c.quiet[u] = (uint8_t)*c.epoch;
    emit_lane<MODE>(c, has, u, own, rown, cu, best, mb, nmv);
  } else {
    // CSR, unit weights: the labels are sorted with the own label as padding (its
    // count is corrected below), then one register pass finds the own
    // rating, the top rating among other labels, how many labels share it
    // and the first two of them
    int32_t a[kLaneMaxDeg];
    {
      const int64_t b = has ? c.g.xadj[u] : 0;
#pragma unroll
      for (int i = 0; i < N; ++i) a[i] = i < deg ? load_label<LIVE>(c.label + __ldcs(c.g.adj + b + i)) : own;
    }
    oem_sort<N>(a);
    int start = 0, ntop = 0;
    int32_t x1 = 0, x2 = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const bool end = i + 1 == N || a[i + 1] != a[i];
      const int32_t run = i + 1 - start;
      const bool isown = a[i] == own;
      rown = end && isown ? run : rown;
      const bool cand = end && !isown;
      const bool gt = cand && run > rmax, eq = cand && run == rmax;
      x2 = eq && ntop == 1 ? a[i] : x2;
      x1 = gt ? a[i] : x1;
      ntop = gt ? 1 : ntop + (eq ? 1 : 0);
      rmax = gt ? run : rmax;
      start = end ? i + 1 : start;
    }
    rown -= N - deg;  // the padding counted as own label
    const int64_t cu = has ? node_w(c.g, u) : 1;
    const bool go = MODE == M_FAV ? rmax > 0 : rmax > rown;
    TieKey hv{0, 0};
    bool have_hv = false;
    LaneCand b1{rmax, 0u, x1};
    if (go && ntop >= 2) {
      hv = lane_tie_key<MODE, SEG>(c, u);
      have_hv = true;
      const LaneCand c1{rmax, tie_of(hv, x1), x1}, c2{rmax, tie_of(hv, x2), x2};
      b1 = lane_better(c1, c2) ? c1 : c2;
    }
    const bool many = go && ntop >= 3;
    bool full = false;
    const int64_t capu = go && MODE != M_FAV ? lane_cap<SEG>(c, u) : 0;
    if (go && MODE != M_FAV) full = c.lw[b1.x] + cu > capu;
    // rare: three or more labels tied at the top, or the winner is full;
    // the sorted labels go to this lane's column and the runs are walked
    if (__any_sync(kFull, many || full)) {
#pragma unroll
      for (int i = 0; i < N; ++i) ccol[i * 32] = a[i];
      if (many || full) {
        if (!have_hv) hv = lane_tie_key<MODE, SEG>(c, u);
        const int own_run = rown + (N - deg);  // the own label's entries, padding included
        LaneCand bb{-1, 0xffffffffu, INT32_MAX};
        for (int i = 0; i < N;) {
          const int32_t x = ccol[i * 32];
          if (x == own) {
            i += own_run;
            continue;
          }
          int j = i + 1;
          while (j < N && ccol[j * 32] == x) ++j;
          const int32_t r = j - i;
          i = j;
          if (many && !full) {  // the best of the top-tied labels
            if (r != rmax) continue;
          } else {  // the best admissible label that improves
            if (r <= rown) continue;
          }
          const LaneCand cand{r, tie_of(hv, x), x};
          if (lane_better(cand, bb) && (!full || MODE == M_FAV || c.lw[x] + cu <= capu))
            bb = cand;
        }
        if (!full) {
          b1 = bb;
          if (MODE != M_FAV) full = c.lw[b1.x] + cu > capu;
          if (full) {  // the top-tied winner is full: look again for an admissible one
            bb = LaneCand{-1, 0xffffffffu, INT32_MAX};
            for (int i = 0; i < N;) {
              const int32_t x = ccol[i * 32];
              if (x == own) {
                i += own_run;
                continue;
              }
              int j = i + 1;
              while (j < N && ccol[j * 32] == x) ++j;
              const int32_t r = j - i;
              i = j;
              if (r <= rown) continue;
              const LaneCand cand{r, tie_of(hv, x), x};
              if (lane_better(cand, bb) && c.lw[x] + cu <= capu) bb = cand;
            }
          }
        }
        if (full) b1 = bb;
      }
    }
    LaneCand best{-1, 0xffffffffu, INT32_MAX};
    if (go) best = b1;
    if (QUIET && has && rmax <= rown) c.quiet[u] = (uint8_t)*c.epoch;
    emit_lane<MODE>(c, has, u, own, rown, cu, best, mb, nmv);
    return;
  }
}

// ---------------------------------------------------------------- approval
struct ApproveCtx {
  const int32_t *mv_u, *mv_t, *mv_o;
  const int64_t *mv_g;
  int8_t *mv_ok;
  int64_t *in_w;
  int32_t *ccnt, *cfill, *ctarget, *cbig;
  // contested movers grouped by target: index, gain and vertex side by side, so
  // the select reads a segment straight through
  int32_t *cseg, *cseg_u;
  int64_t *cseg_g;
  int64_t *cbase;
  // [0] movers [1] contested targets [2] contested pool [3] targets of more than 32 movers
  unsigned long long *counters;
  int32_t *label;
  int64_t *lw;
  int64_t cap;
  const int64_t *vw;
  bool narrow;  // all vertex weights together fit 31 bits
  // batched graphs: graph of every label and every graph's cap (null: one graph)
  const int32_t *lgid;
  const int64_t *gcap;
};

__device__ __forceinline__ int64_t vwt(const ApproveCtx &a, int64_t u) { return a.vw ? a.vw[u] : 1; }
// Mover i's place in its target's segment.
__device__ __forceinline__ void put_contested(const ApproveCtx &a, int64_t i, int32_t t) {
  const int64_t at = a.cbase[t] + atomicAdd(&a.cfill[t], 1);
  a.cseg[at] = (int32_t)i;
  a.cseg_u[at] = a.mv_u[i];
  a.cseg_g[at] = a.mv_g[i];
}
__device__ __forceinline__ int64_t target_cap(const ApproveCtx &a, int32_t t) {
  return a.lgid ? a.gcap[a.lgid[t]] : a.cap;
}

// One contested target with at most 32 movers, by a warp: every mover's
// inclusive weight prefix in (gain desc, vertex asc) order, from all pairs.
__device__ __forceinline__ void approve_small(const ApproveCtx &a, int64_t base, int cnt,
                                              int64_t rem) {
  const int lane = lane_id();
  const bool in = lane < cnt;
  const int32_t i = in ? a.cseg[base + lane] : 0;
  const int64_t g = in ? a.cseg_g[base + lane] : 0;
  const int32_t u = in ? a.cseg_u[base + lane] : 0;
  const int64_t w = in ? vwt(a, u) : 0;
  int64_t pre = 0;
  for (int q = 0; q < cnt; ++q) {
    const int64_t gq = __shfl_sync(kFull, g, q), wq = __shfl_sync(kFull, w, q);
    const int32_t uq = __shfl_sync(kFull, u, q);
    if (gq > g || (gq == g && uq <= u)) pre += wq;
  }
  if (in && pre <= rem) a.mv_ok[i] = 1;
}

// C: the nt contested targets (and among them the nbig of more than 32 movers,
// listed apart), shared out over nblk blocks (this is number blk): each approves the longest fitting prefix of its movers in
// (gain desc, vertex asc) order. Few movers (the usual case of clustering)
// take a warp per target, more a block with the radix select.
__device__ void approve_targets(const ApproveCtx &a, int64_t nt, int64_t nbig, int blk, int nblk) {
  const int nwarp = blockDim.x >> 5;
  for (int64_t j = (int64_t)blk * nwarp + (threadIdx.x >> 5); j < nt; j += (int64_t)nblk * nwarp) {
    const int32_t t = a.ctarget[j];
    const int32_t cnt = a.ccnt[t];
    if (cnt > 32 || cnt == 0) continue;  // (0: a block is done with it already)
    const int64_t rem = target_cap(a, t) - a.lw[t];
    if (rem >= 0) approve_small(a, a.cbase[t], cnt, rem);
    __syncwarp();
    if (lane_id() == 0) a.ccnt[t] = 0, a.cfill[t] = 0;
  }
  for (int64_t j = blk; j < nbig; j += nblk) {
    const int32_t t = a.cbig[j];
    const int64_t base = a.cbase[t], cnt = a.ccnt[t];
    __syncthreads();  // every thread has read ccnt, and the previous target is done with
    const int64_t rem = target_cap(a, t) - a.lw[t];
    auto item = [&](int64_t q, uint64_t &hi, uint32_t &lo, int64_t &w) {
      const int32_t u = a.cseg_u[base + q];
      hi = ~(uint64_t)a.cseg_g[base + q];
      lo = (uint32_t)u;
      w = vwt(a, u);
    };
    if (rem >= 0) {  // (else nothing can enter: mv_ok is 0 already)
      uint64_t khi;
      uint32_t klo;
      block_select(cnt, rem, a.narrow, item, khi, klo);
      for (int64_t q = threadIdx.x; q < cnt; q += blockDim.x) {
        uint64_t hi;
        uint32_t lo;
        int64_t w;
        item(q, hi, lo, w);
        if (hi < khi || (hi == khi && lo < klo)) a.mv_ok[a.cseg[base + q]] = 1;
      }
    }
    if (threadIdx.x == 0) a.ccnt[t] = 0, a.cfill[t] = 0;
  }
}

ApproveCtx approve_ctx(tp_graph *g, const LpState &st, LpWork &w) {
  ApproveCtx a;
  a.mv_u = w.mv_u.get();
  a.mv_o = w.mv_o.get();
  a.mv_t = w.mv_t.get();
  a.mv_g = w.mv_g.get();
  a.mv_ok = w.mv_ok.get();
  a.in_w = w.in_w.get();
  a.ccnt = w.ccnt.get();
  a.cfill = w.cfill.get();
  a.cseg = w.cseg.get();
  a.cseg_u = w.cseg_u.get();
  a.cseg_g = w.cseg_g.get();
  a.ctarget = w.ctarget.get();
  a.cbig = w.cbig.get();
  a.cbase = w.cbase.get();
  a.counters = (unsigned long long *)w.counters.get();
  a.label = st.label;
  a.lw = st.lw;
  a.cap = st.cap;
  a.vw = g->unit_vw ? nullptr : g->vw.get();
  a.narrow = g->total_vw >= 0 && g->total_vw < ((int64_t)1 << 31);
  a.lgid = st.seg.gid ? st.seg.lgid : nullptr;
  a.gcap = st.seg.cap;
  return a;
}

}  // namespace

}  // namespace tp
