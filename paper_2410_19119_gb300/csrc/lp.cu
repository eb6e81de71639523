// Size-constrained label propagation on the GPU (Algorithm 1 of the paper,
// made synchronous and deterministic), its two-hop packing and rebalancing.
//
// Rating (Section "Rating Maps", Algorithm 2): a vertex's ratings R[C[v]] +=
// w(u,v) accumulate in a hash table. The paper's split into a first phase
// with small per-thread tables and a second phase for "bumped" high-degree
// vertices becomes five degree tiers, each a different kernel:
//   lane  (deg <= tier_lane):  one lane per vertex, labels sorted in
//          registers (no table at all);
//   small (deg <= tier_small): one warp per vertex, shared table of up to
//          128 slots;
//   mid   (deg <= tier_mid):   one warp per vertex, shared table of up to
//          1024 slots (both warp tiers fill and scan only the least power of
//          two >= table_slack * degree slots, at least 32);
//   big   (deg <= 10000):      one block per vertex, shared table of 2048 to
//          16384 slots by its degree;
//   huge  (deg > 10000):       one block per chunk of 1000 neighbours (the
//          compressed format's independently decodable chunks) aggregates in
//          a shared table and flushes into the vertex's global table with
//          atomics (the paper's "hash tables as flush buffers" against
//          contention); blocks then scan that table in segments and one
//          block per vertex combines the segments' results.
// Where the labels are at most 1024 blocks (refinement, rebalancing) the tiers
// above lane count in one counter per block instead of a hash table. Levels of
// one graph that fit a thread-block cluster run all their rounds in one launch
// (lp_small.cu).
// The tier only decides where the sums are formed; integer sums commute and
// the argmax uses a total order, so the result is tier-independent.
//
// Approval: movers add their weight to in_w[target] with atomics. Targets
// whose weight plus in_w fits approve every mover; for the others a warp (up
// to 32 movers) or a block per target runs a weighted radix select over the
// key (gain desc, vertex asc) and approves exactly the longest fitting prefix.
#include <algorithm>
#include <memory>
#include <mutex>

#include "lp_rate.cuh"

namespace tp {

namespace {

// Small tier: one warp per listed vertex (c.list), or, in rebalancing mode
// (c.list == nullptr), every vertex of the small and lane tiers, filtered in
// 32-vertex slabs.
template <bool COMP, int MODE, class V>
__global__ void k_rate_small(RateCtx c) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  WarpSmem<kSmallLog, V> &ws =
      reinterpret_cast<WarpSmem<kSmallLog, V> *>(smem_raw)[threadIdx.x >> 5];
  init_table(ws);
  MoverBuf mb{ws.mu, ws.mt, ws.mo, ws.mg, 0};
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  if (c.list) {
    int64_t kb, ke;
    tier_range(c, kb, ke);
    for (int64_t k = kb + gw; k < ke; k += nw) {
      int64_t i, u;
      if (tier_entry<MODE>(c, k, i, u)) {
        ZipNbr z;
        const int64_t d = row_degree<COMP>(c.g, u, z);
        rate_vertex_warp<COMP, MODE, V, true>(c, u, ws.keys, ws.vals, table_log(c, d, kSmallLog), &mb, &z);
      }
    }
  } else {
    for (int64_t base = gw * 32; base < c.g.n; base += nw * 32) {
      int64_t u = base + lane_id();
      bool act = u < c.g.n && (c.tier[u] == TIER_SMALL || c.tier[u] == TIER_LANE) &&
                 active<MODE>(c, u);
      unsigned am = __ballot_sync(kFull, act);
      while (am) {
        int j = __ffs(am) - 1;
        am &= am - 1;
        const int64_t v = base + j;
        ZipNbr z;
        const int64_t d = row_degree<COMP>(c.g, v, z);
        rate_vertex_warp<COMP, MODE, V, true>(c, v, ws.keys, ws.vals, table_log(c, d, kSmallLog), &mb, &z);
      }
    }
  }
  if (MODE == M_LP) flush_movers(c, mb);
}

template <bool W>
__host__ __device__ constexpr int lane_warps() { return W ? 4 : kLaneWarps; }

// LONG: some compressed records exceed the 80-byte window (skewed graphs), or
// (weighted) labels beyond kLaneKeyLabels; separate instantiations keep the
// common kernels free of those paths.
template <bool COMP, int MODE, bool W, bool LONG = false, bool SEG = false>
__global__ void __launch_bounds__(lane_warps<W>() * 32, W ? 1 : kLaneBlocksPerSM)
    k_rate_lane(RateCtx c) {
  static_assert(!(COMP && W), "weighted levels are CSR");
  constexpr int WARPS = lane_warps<W>();
  // per lane: staged record words, then candidate labels
  __shared__ uint32_t lab_all[WARPS][kLaneMaxDeg][32];
  __shared__ uint32_t aux_all[WARPS][W ? kLaneMaxDeg : 1][32];  // candidate ratings (weighted)
  __shared__ uint8_t cnt_all[WARPS][COMP && !W ? kLaneMaxDeg : 1][32];  // candidate ratings
  __shared__ int32_t queue_all[WARPS][kLaneQueue];
  __shared__ LaneMovers movers_all[WARPS];
  const int lane = lane_id(), w = threadIdx.x >> 5;
  uint32_t *col = &lab_all[w][0][lane];
  uint32_t *wcol = &aux_all[w][0][lane];
  int32_t *queue = queue_all[w];
  LaneMovers &mb = movers_all[w];
  uint8_t *cnt = &cnt_all[w][0][lane];
  // warps and list positions fit 32 bits (lists hold < 2^31 vertex ids)
  const int32_t gw = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int32_t nw = (int32_t)((gridDim.x * blockDim.x) >> 5);
  // bucket mode: this sub-round's lane-tier vertices come as a list
  const bool list_mode = MODE == M_LP && c.bucket != nullptr;
  int32_t bcount = 0, bnext = gw * c.lane_win;
  const int32_t *blist = c.bucket;
  const uint64_t *brec = COMP ? c.bucket_rec : nullptr;
  int64_t base = (int64_t)gw * 256;
  int j8 = 0, pending = 0;  // slab scan position; queued vertices (warp-uniform)
  if (list_mode) {
    const int64_t bstart = c.bucket_off[(int64_t)c.s * c.bucket_nb];
    bcount = (int32_t)(c.bucket_off[(int64_t)(c.s + 1) * c.bucket_nb] - bstart);
    blist += bstart;
    if (brec) brec += bstart;
    base = c.g.n;  // no slab scan
  }
  for (;;) {
    int take, wstart = 0;
    if (list_mode) {
      if (bnext >= bcount) break;
      wstart = bnext;
      take = bcount - bnext < c.lane_win ? bcount - bnext : c.lane_win;
      // never step past the end (keeps bnext below 2^31)
      bnext = bcount - bnext > nw * c.lane_win ? bnext + nw * c.lane_win : bcount;
    } else {
      // fill the queue, 32 vertices of the current 256-vertex slab at a time
      while (pending < kLaneWin && base < c.g.n) {
        const int64_t v = base + 32 * j8 + lane;
        const bool act = v < c.g.n && c.tier[v] == TIER_LANE && active<MODE>(c, v);
        const unsigned m = __ballot_sync(kFull, act);
        if (act) queue[pending + __popc(m & lanemask_lt())] = (int32_t)v;
        pending += __popc(m);
        if (++j8 == 8) j8 = 0, base += (int64_t)nw * 256;
      }
      if (pending == 0) break;
      __syncwarp();
      take = pending < kLaneWin ? pending : kLaneWin;
    }
    // batches of 32 in list order: vertices close in the list are close in
    // the graph, so a batch's records and label gathers share cache lines
    // (grouping a window by degree instead was measured slower)
    const int32_t *win = list_mode ? blist + wstart : queue;
    const uint64_t *wrec = list_mode && brec ? brec + wstart : nullptr;
    int nmv = 0;  // movers of this window so far (warp-uniform)
    for (int q = 0; q < take; q += 32) {
      const bool has = q + lane < take;
      const int32_t u = has ? win[q + lane] : 0;
      if (q + 32 + lane < take) lane_prefetch<COMP>(c.g, wrec, q + 32 + lane, win[q + 32 + lane]);
      int deg = 0;
      if (has) {
        if (COMP) {
          uint64_t rb, re;
          lane_record(c.g, wrec, q + lane, u, rb, re);
          // records beyond the 80-byte window (rare except on skewed graphs)
          // take the decoder that loads further groups
          if (LONG && __any_sync(__activemask(), (re - (rb & ~(uint64_t)15)) > 80))
            deg = lane_decode<true>(c.g, rb, re, col);
          else
            deg = lane_decode<false>(c.g, rb, re, col);
        } else {
          deg = min((int)(c.g.xadj[u + 1] - c.g.xadj[u]), kLaneMaxDeg);
        }
      }
      const unsigned maxdeg = __reduce_max_sync(kFull, (unsigned)deg);
      constexpr bool WIDE = W && LONG;
      if (W && maxdeg <= 8)  // coarse levels of meshes
        lane_batch<COMP, MODE, W, 8, SEG, false, WIDE>(c, has, u, deg, col, wcol, cnt, mb, nmv);
      else if (maxdeg <= 16)
        lane_batch<COMP, MODE, W, 16, SEG, false, WIDE>(c, has, u, deg, col, wcol, cnt, mb, nmv);
      else
        lane_batch<COMP, MODE, W, kLaneMaxDeg, SEG, false, WIDE>(c, has, u, deg, col, wcol, cnt, mb, nmv);
    }
    __syncwarp();
    if (nmv) {  // the window's movers, coalesced
      unsigned long long basep = 0;
      if (lane == 0) basep = atomicAdd(c.counters, (unsigned long long)nmv);
      basep = __shfl_sync(kFull, basep, 0);
      for (int i = lane; i < nmv; i += 32) {
        c.mv_u[basep + i] = mb.u[i];
        c.mv_t[basep + i] = mb.t[i];
        c.mv_o[basep + i] = mb.o[i];
        c.mv_g[basep + i] = mb.g[i];
      }
      __syncwarp();
    }
    if (!list_mode) {  // slab scans: move the vertices beyond the window to the front
      const int left = pending - take;
      const int32_t t = lane < left ? queue[take + lane] : 0;
      __syncwarp();
      if (lane < left) queue[lane] = t;
      __syncwarp();
      pending = left;
    }
  }
}

// Lane tier with quiet vertices left out. A vertex whose rating found no label
// better than its own moves in no later sub-round, whatever the tie order and
// the label weights, until a neighbour moves; k_wake forgets the marks of the
// neighbours of every moved vertex. In refinement the interior of every block
// is quiet after the first round, which leaves a tenth of a mesh to rate. A
// warp's window of the list is filtered into a queue of list positions, so the
// batches stay full.
template <bool COMP, bool W>
__global__ void __launch_bounds__(lane_warps<W>() * 32, W ? 1 : kLaneBlocksPerSM)
    k_rate_lane_quiet(RateCtx c) {
  constexpr int WARPS = lane_warps<W>();
  __shared__ uint32_t lab_all[WARPS][kLaneMaxDeg][32];
  __shared__ uint32_t aux_all[WARPS][W ? kLaneMaxDeg : 1][32];
  __shared__ uint8_t cnt_all[WARPS][COMP && !W ? kLaneMaxDeg : 1][32];
  __shared__ int32_t queue_all[WARPS][64];
  __shared__ BatchMovers movers_all[WARPS];
  const int lane = lane_id(), w = threadIdx.x >> 5;
  uint32_t *col = &lab_all[w][0][lane];
  uint32_t *wcol = &aux_all[w][0][lane];
  uint8_t *cnt = &cnt_all[w][0][lane];
  int32_t *queue = queue_all[w];
  BatchMovers &mb = movers_all[w];
  const int64_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = (gridDim.x * blockDim.x) >> 5;
  const int64_t bstart = c.bucket_off[(int64_t)c.s * c.bucket_nb];
  const int64_t bcount = c.bucket_off[(int64_t)(c.s + 1) * c.bucket_nb] - bstart;
  const int32_t *blist = c.bucket + bstart;
  const uint64_t *brec = COMP ? c.bucket_rec + bstart : nullptr;
  const int epoch = *c.epoch;
  int64_t win = gw * c.lane_win;  // this window's start; at: next position in it
  int at = 0, pending = 0;
  for (;;) {
    while (pending < 32 && win < bcount) {
      const int64_t p = win + at + lane;
      const bool act = at + lane < c.lane_win && p < bcount && c.quiet[blist[p]] != epoch;
      const unsigned m = __ballot_sync(kFull, act);
      if (act) queue[pending + __popc(m & lanemask_lt())] = (int32_t)p;
      pending += __popc(m);
      at += 32;
      if (at >= c.lane_win) at = 0, win += nw * c.lane_win;
    }
    if (pending == 0) break;
    __syncwarp();
    const int take = min(pending, 32);
    const bool has = lane < take;
    const int32_t p = has ? queue[lane] : 0;
    const int32_t rest = take + lane < pending ? queue[take + lane] : 0;
    __syncwarp();
    if (take + lane < pending) queue[lane] = rest;
    pending -= take;
    const int32_t u = has ? blist[p] : 0;
    int deg = 0, nmv = 0;
    if (has) {
      if (COMP) {
        uint64_t rb, re;
        lane_record(c.g, brec, p, u, rb, re);
        deg = lane_decode<false>(c.g, rb, re, col);
      } else {
        deg = min((int)(c.g.xadj[u + 1] - c.g.xadj[u]), kLaneMaxDeg);
      }
    }
    const unsigned maxdeg = __reduce_max_sync(kFull, (unsigned)deg);
    if (maxdeg <= 16)
      lane_batch<COMP, M_LP, W, 16, false, false, false, true>(c, has, u, deg, col, wcol, cnt, mb, nmv);
    else
      lane_batch<COMP, M_LP, W, kLaneMaxDeg, false, false, false, true>(c, has, u, deg, col, wcol, cnt, mb, nmv);
    __syncwarp();
    if (nmv) {
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(c.counters, (unsigned long long)nmv);
      base = __shfl_sync(kFull, base, 0);
      if (lane < nmv) {
        c.mv_u[base + lane] = mb.u[lane];
        c.mv_t[base + lane] = mb.t[lane];
        c.mv_o[base + lane] = mb.o[lane];
        c.mv_g[base + lane] = mb.g[lane];
      }
      __syncwarp();
    }
  }
}

// The neighbours of every moved vertex are quiet no longer: low-degree movers
// by a thread each, mid ones by a warp, the others by the block. Where a
// sub-round moved so many that little would stay quiet, or a hub of more than
// kWakeMost neighbours, the epoch advances instead (once a sub-round: counters[4]),
// which ends all marks. (A warp for every hub: a mesh of 2^22 vertices with one
// joined to every eighth refined in 9.4 ms and with one joined to all clustered,
// compressed, in 32, where rating everything took 4.9 and 7.3.)
constexpr int64_t kWakeMost = 65536;  // 64 steps of the block, about as many us
template <bool COMP>
__global__ void __launch_bounds__(256) k_wake(GView g, const uint8_t *tier,
                                              unsigned long long *counters, const int32_t *mv_u,
                                              const int8_t *mv_ok, int64_t limit, uint8_t *quiet,
                                              int32_t *epoch) {
  __shared__ int32_t big[256], n_big;
  const int64_t nm = (int64_t)counters[0];
  if (nm > limit) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *epoch += 1;
    return;
  }
  const int w = threadIdx.x >> 5;
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x; i0 < nm;
       i0 += (int64_t)gridDim.x * blockDim.x) {
    if (threadIdx.x == 0) n_big = 0;
    __syncthreads();
    const int64_t i = i0 + threadIdx.x;
    const bool in = i < nm && mv_ok[i];
    const int32_t u = in ? mv_u[i] : 0;
    const uint8_t t = in ? tier[u] : TIER_LANE;
    if (in && (t == TIER_LANE || t == TIER_SMALL))
      thread_neighbours<COMP>(g, u, [&](int32_t v, int64_t) { quiet[v] = 0; });
    if (t == TIER_BIG || t == TIER_HUGE) {
      const int64_t d = COMP ? zip_nbr(g, u).deg : g.xadj[u + 1] - g.xadj[u];
      if (d <= kWakeMost) big[atomicAdd(&n_big, 1)] = u;
      else if (atomicExch(&counters[4], 1ull) == 0) atomicAdd(epoch, 1);
    }
    __syncwarp();
    for (unsigned q = __ballot_sync(kFull, t == TIER_MID); q; q &= q - 1)
      warp_neighbours<COMP>(g, __shfl_sync(kFull, u, __ffs(q) - 1), -1,
                            [&](bool has, int32_t v, int64_t, int64_t) {
                              if (has) quiet[v] = 0;
                            });
    __syncthreads();
    const int nb = n_big;
    for (int k = 0; k < nb; ++k) {
      const int32_t b = big[k];
      if constexpr (COMP) {  // a chunk is decoded by one warp, a record below the threshold whole
        const ZipNbr z = zip_nbr(g, b);
        for (int64_t j = (w + k) & 7; j < z.nchunks; j += 8)
          warp_neighbours<true>(
              g, b, z.nchunks > 1 ? j : -1,
              [&](bool has, int32_t v, int64_t, int64_t) {
                if (has) quiet[v] = 0;
              },
              &z);
      } else {
        const int64_t e = g.xadj[b + 1];
        for (int64_t x = g.xadj[b] + threadIdx.x; x < e; x += 4 * 256) {
          int32_t v[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) v[r] = x + 256 * r < e ? g.adj[x + 256 * r] : -1;
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (v[r] >= 0) quiet[v[r]] = 0;
        }
      }
    }
    __syncthreads();  // big is listed anew
  }
}

// Mid tier: one warp per listed vertex, its table of up to 2^LOG slots in
// shared memory (V: uint32_t counts at unit weights, int64_t sums otherwise;
// the smaller tables leave room for more warps per SM).
template <bool COMP, int MODE, int LOG, class V>
__global__ void k_rate_list(RateCtx c) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int32_t mu[kMidWarps][32], mt[kMidWarps][32], mo[kMidWarps][32];
  __shared__ int64_t mg[kMidWarps][32];
  const int w = threadIdx.x >> 5;
  WarpSmem<LOG, V> &ws = reinterpret_cast<WarpSmem<LOG, V> *>(smem_raw)[w];
  init_table(ws);
  MoverBuf mb{mu[w], mt[w], mo[w], mg[w], 0};
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int64_t kb, ke;
  tier_range(c, kb, ke);
  for (int64_t k = kb + gw; k < ke; k += nw) {
    int64_t i, u;
    if (!tier_entry<MODE>(c, k, i, u)) continue;
    ZipNbr z;
    const int64_t d = row_degree<COMP>(c.g, u, z);
    rate_vertex_warp<COMP, MODE, V>(c, u, ws.keys, ws.vals, table_log(c, d, LOG), &mb, &z);
  }
  if (MODE == M_LP) flush_movers(c, mb);
}

// Few labels (refinement and rebalancing: the k blocks of the vertex's graph,
// at most kDirectMax): a rating is one counter per block, indexed by the
// label, so there is nothing to hash, and a vertex clears and scans k
// counters instead of up to 16384 slots. One warp per listed vertex of degree
// <= kBigTinySplit; the block and hub kernels take the same tables (DIR).
constexpr int kDirectMax = 1024;
constexpr int kDirectWarps = 4;

template <bool COMP, int MODE, class V>
__global__ void __launch_bounds__(32 * kDirectWarps) k_rate_direct(RateCtx c, int kmax) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int32_t mu[kDirectWarps][32], mt[kDirectWarps][32], mo[kDirectWarps][32];
  __shared__ int64_t mg[kDirectWarps][32];
  const int w = threadIdx.x >> 5, lane = lane_id();
  V *vals = reinterpret_cast<V *>(smem_raw) + (size_t)w * kmax;
  for (int i = lane; i < kmax; i += 32) vals[i] = 0;
  __syncwarp();
  MoverBuf mb{mu[w], mt[w], mo[w], mg[w], 0};
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int64_t kb, ke;
  tier_range(c, kb, ke);
  for (int64_t q = kb + gw; q < ke; q += nw) {
    int64_t pos, u;
    if (!tier_entry<MODE>(c, q, pos, u)) continue;
    int32_t lb;
    const int32_t k = block_range(c, u, lb);
    warp_labels<COMP>(c, u, [&](int32_t x, int64_t wt) {
      const uint32_t i = (uint32_t)(x - lb);
      if (i < (uint32_t)k) atomicAdd(&vals[i], (V)wt);
    });
    __syncwarp();
    const int64_t cu = node_w(c.g, u);
    const Best b = pick_warp<MODE>(c, u, cu, k, [&](int i, int32_t &x, int64_t &R) {
      R = (int64_t)vals[i];
      x = R ? lb + i : -1;  // weights are positive: a block with a neighbour has a rating
    });
    for (int i = lane; i < k; i += 32) vals[i] = 0;
    __syncwarp();
    finalize_warp<MODE>(c, b, u, cu, &mb);
  }
  if (MODE == M_LP) flush_movers(c, mb);
}

// ---------------------------------------------------------------- big tier
// One block per listed vertex: its ratings are summed in a shared-memory
// hash table of 2^logc >= 1.5 deg slots (keys, then 32-bit counts for unit
// weights or 64-bit sums), so no rating touches global memory. A compressed
// neighbourhood (one chunk below the chunking threshold) is decoded by the
// whole block: every thread takes a slice of the record's bytes, assembles
// the values whose last byte lies in its slice (reading back into the
// previous slice for the first bytes of a value), and two block scans give
// each value its index and the sum of the gaps before it.
constexpr int kBlockThreads = 256;
constexpr int kBlockTinyLog = 11;   // 2048 slots: degrees up to kBigTinySplit = 1024
constexpr int kBlockMidLog = 12;    // 4096 slots: degrees up to kBigMidSplit = 2048
constexpr int kBlockSmallLog = 13;  // 8192 slots: degrees up to kBigSplit = 4096
constexpr int kBlockBigLog = 14;    // 16384 slots: degrees up to 10000
// Record staging and decoded values for a compressed vertex of degree <= dmax:
// at most 5 bytes per neighbour (+ alignment slack), 4 bytes per value.
__host__ __device__ constexpr size_t block_stage_bytes(int64_t dmax) {
  return ((size_t)(5 * dmax + 64) + 15) & ~(size_t)15;
}
__host__ __device__ constexpr size_t block_vbuf_bytes(int64_t dmax) { return (size_t)4 * dmax; }
__host__ __device__ constexpr int64_t block_max_deg(int lg) {
  return lg == kBlockTinyLog    ? kBigTinySplit
         : lg == kBlockMidLog   ? kBigMidSplit
         : lg == kBlockSmallLog ? kBigSplit
                                : kChunkThreshold;
}

// Block-wide exclusive sum of one int64 per thread; returns this thread's
// prefix and sets total. red holds kBlockThreads / 32 + 1 entries.
__device__ __forceinline__ int64_t block_excl_sum(int64_t v, int64_t *red, int64_t &total) {
  const int lane = lane_id(), w = threadIdx.x >> 5;
  const int64_t inc = warp_incl_scan(v);
  if (lane == 31) red[w] = inc;
  __syncthreads();
  if (w == 0) {
    const int64_t x = lane < kBlockThreads / 32 ? red[lane] : 0;
    const int64_t xi = warp_incl_scan(x);
    if (lane < kBlockThreads / 32) red[lane] = xi - x;
    if (lane == kBlockThreads / 32 - 1) red[kBlockThreads / 32] = xi;
  }
  __syncthreads();
  const int64_t r = red[w] + inc - v;
  total = red[kBlockThreads / 32];
  __syncthreads();
  return r;
}

// Block-wide exclusive sum of one uint32 per thread (same contract as
// block_excl_sum).
__device__ __forceinline__ uint32_t block_excl_sum32(uint32_t v, int64_t *red, uint32_t &total) {
  int64_t t;
  const int64_t r = block_excl_sum((int64_t)v, red, t);
  total = (uint32_t)t;
  return (uint32_t)r;
}

// Decodes one chunk [cb, ce) of u's neighbourhood (count values: the first
// a signed offset from u, then gaps) with the whole block and calls f(v)
// for every neighbour. The chunk's bytes are copied into shared memory
// (stage: at least ce - cb + 32 bytes, 16-byte aligned) with 16-byte loads;
// then (1) every thread counts the value ends (bytes without the
// continuation bit) in its slice of the bytes, (2) a block scan gives each
// thread the index of its first value and every thread writes the values
// ending in its slice to vbuf (count entries), each assembled without
// branches from its last byte and up to four preceding continuation bytes,
// (3) a block scan over the values turns them into neighbour ids, and (4)
// f(count) is called by every thread once the ids are in vbuf.
template <class F>
__device__ __forceinline__ void block_decode_range(const GView &g, int64_t u, uint64_t cb,
                                                   uint64_t ce, int64_t count, uint8_t *stage,
                                                   uint32_t *vbuf, int64_t *red, F &&f) {
  const uint64_t ws = cb & ~(uint64_t)15;
  const int off = (int)(cb - ws), L = (int)(ce - cb);
  const int ngroups = (off + L + 15) >> 4;
  const uint4 *src = reinterpret_cast<const uint4 *>(g.bytes + ws);
  for (int k = threadIdx.x; k < ngroups; k += kBlockThreads)
    reinterpret_cast<uint4 *>(stage)[k] = __ldcs(src + k);
  __syncthreads();
  const uint8_t *by = stage + off;
  const int K = (L + kBlockThreads - 1) / kBlockThreads;
  const int lo = min((int)threadIdx.x * K, L), hi = min((int)(threadIdx.x + 1) * K, L);
  uint32_t ends = 0;
  for (int p = lo; p < hi; ++p) ends += !(by[p] & 0x80u);
  uint32_t nval;
  uint32_t idx = block_excl_sum32(ends, red, nval);
  const int cnt = (int)min((int64_t)nval, count);
  if (threadIdx.x == 0 && (int64_t)nval != count) latch_error(g.err, TP_ERR_CORRUPT);
  // the four bytes before the slice (continuation bytes of a value ending in it)
  uint32_t win = 0;  // byte p-1 in bits 0..7, p-2 in 8..15, ...
#pragma unroll
  for (int d = 4; d >= 1; --d) win = (win << 8) | (lo - d >= 0 ? by[lo - d] : 0u);
  for (int p = lo; p < hi; ++p) {
    const uint32_t b0 = by[p];
    // continuation bytes directly before p: k = 0..4
    const uint32_t stop = ~win & 0x80808080u;
    const int k = stop ? (__ffs(stop) - 8) >> 3 : 4;
    // payloads of bytes p-1 .. p-4 packed 7 bits apart, p-1 lowest
    uint32_t pk = (win & 0x7fu) | ((win >> 1) & 0x3f80u) | ((win >> 2) & 0x1fc000u) |
                  ((win >> 3) & 0xfe00000u);
    // value = bytes p-k .. p, earliest byte lowest: reverse the k packed payloads
    uint32_t v = b0 & 0x7fu;
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      const bool take = d < k;
      v = take ? (v << 7) | (pk & 0x7fu) : v;
      pk >>= 7;
    }
    if (!(b0 & 0x80u)) {
      if ((int)idx < cnt) vbuf[idx] = v;
      ++idx;
    }
    win = (win << 8) | b0;
  }
  __syncthreads();
  // ids: id_0 = u + signed offset, id_i = id_(i-1) + gap_i
  const int P = (cnt + kBlockThreads - 1) / kBlockThreads;
  const int a0 = min((int)threadIdx.x * P, cnt), a1 = min((int)(threadIdx.x + 1) * P, cnt);
  uint32_t part = 0;
  for (int i = max(a0, 1); i < a1; ++i) part += vbuf[i];
  uint32_t gtot;
  uint32_t run = block_excl_sum32(part, red, gtot);
  const uint32_t c0 = vbuf[0];
  const int64_t id0 = (c0 & 1u) ? u - (int64_t)(c0 >> 1) : u + (int64_t)(c0 >> 1);
  __syncthreads();  // vbuf[0] read by every thread before it is overwritten
  const int64_t nmax = g.n - 1;
  for (int i = a0; i < a1; ++i) {
    if (i > 0) run += vbuf[i];
    // streams are validated on creation; the clamp only keeps a corrupted
    // one from reading out of bounds
    vbuf[i] = (uint32_t)min(max(id0 + (int64_t)run, (int64_t)0), nmax);
  }
  __syncthreads();
  f(cnt);  // the ids are in vbuf[0 .. cnt)
  __syncthreads();  // stage and vbuf are reused
}

template <class V>
__device__ __forceinline__ void blk_add(int32_t *keys, V *vals, int logc, int32_t x, V w,
                                        int32_t *err) {
  const uint32_t mask = (1u << logc) - 1u;
  uint32_t h = slot_of(x, logc);
  for (uint32_t probe = 0; probe <= mask; ++probe, h = (h + 1) & mask) {
    int32_t k = keys[h];
    if (k == -1) {
      const int32_t prev = atomicCAS(&keys[h], -1, x);
      k = prev == -1 ? x : prev;
    }
    if (k == x) {
      atomicAdd(&vals[h], w);
      return;
    }
  }
  latch_error(err, TP_ERR_CORRUPT);
}

// Block-wide maxima of two values; the results are in every thread.
__device__ __forceinline__ void block_max2(int64_t &a, int64_t &b, int64_t *red) {
  a = warp_max(a);
  b = warp_max(b);
  const int lane = lane_id(), w = threadIdx.x >> 5;
  __shared__ int64_t rb[kBlockThreads / 32];
  if (lane == 0) red[w] = a, rb[w] = b;
  __syncthreads();
  int64_t x = lane < kBlockThreads / 32 ? red[lane] : INT64_MIN;
  int64_t y = lane < kBlockThreads / 32 ? rb[lane] : INT64_MIN;
  a = warp_max(x);
  b = warp_max(y);
  __syncthreads();
}

// Block-wide best (rating order) and own rating; the result is in every thread.
__device__ __forceinline__ void block_reduce_best(Best &b, Best *wb) {
  warp_reduce_best(b);
  const int lane = lane_id(), w = threadIdx.x >> 5;
  if (lane == 0) wb[w] = b;
  __syncthreads();
  b = lane < kBlockThreads / 32 ? wb[lane] : Best{-1, 0xffffffffu, INT32_MAX, 0};
  warp_reduce_best(b);
  __syncthreads();
}

// V: uint32_t where all edge weights together fit, else 64 bits (32-bit shared
// atomics are native, and the smaller tables leave room for more blocks).
// DIR: a counter per block of the vertex's graph (kmax: most of any graph)
// instead of the hash table.
template <bool COMP, int MODE, class V, bool DIR>
__global__ void __launch_bounds__(kBlockThreads) k_rate_block(RateCtx c, int maxlog, int kmax) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const size_t slots = DIR ? (size_t)((kmax + 3) & ~3) : (size_t)1 << maxlog;
  int32_t *keys = reinterpret_cast<int32_t *>(smem_raw);
  V *vals = reinterpret_cast<V *>(smem_raw + (DIR ? 0 : sizeof(int32_t) * slots));
  // compressed: the record's bytes (at most 5 per neighbour, + alignment),
  // then its decoded values
  uint8_t *stage = reinterpret_cast<uint8_t *>(vals + slots);
  uint32_t *vbuf = reinterpret_cast<uint32_t *>(stage + block_stage_bytes(block_max_deg(maxlog)));
  __shared__ int64_t red[kBlockThreads / 32 + 1];
  __shared__ Best wb[kBlockThreads / 32];
  __shared__ int32_t mu[32], mt[32], mo[32];
  __shared__ int64_t mg[32];
  const int tid = threadIdx.x;
  int64_t kb, ke;
  tier_range(c, kb, ke);
  for (int64_t k = kb + blockIdx.x; k < ke; k += gridDim.x) {
    int64_t i, u;
    if (!tier_entry<MODE>(c, k, i, u)) continue;  // uniform over the block
    ZipNbr z;
    const int64_t d = row_degree<COMP>(c.g, u, z);  // one chunk: below the chunking threshold
    int logc = 5;
    while (logc < maxlog && ((int64_t)1 << logc) < d + d / 2) ++logc;
    int32_t lb = 0;
    const int cap = DIR ? block_range(c, u, lb) : 1 << logc;
    for (int k = tid; k < cap; k += kBlockThreads) {
      if (!DIR) keys[k] = -1;
      vals[k] = 0;
    }
    __syncthreads();
    auto add = [&](int32_t x, V w) {
      if constexpr (DIR) {
        if ((uint32_t)(x - lb) < (uint32_t)cap) atomicAdd(&vals[x - lb], w);
      } else {
        blk_add<V>(keys, vals, logc, x, w, c.g.err);
      }
    };
    auto slot_label = [&](int k) -> int32_t {
      if constexpr (DIR) return vals[k] ? lb + k : -1;
      else return keys[k];
    };
    if (COMP) {
      block_decode_range(c.g, u, z.data, z.end, z.deg, stage, vbuf, red, [&](int cnt) {
        for (int e = tid; e < cnt; e += kBlockThreads) add(c.label[vbuf[e]], (V)1);
      });
    } else {
      // four entries a thread and step, their loads together
      const int64_t b = c.g.xadj[u];
      for (int64_t e0 = tid; e0 < d; e0 += 4 * kBlockThreads) {
        int32_t v[4], x[4];
        V w[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int64_t e = e0 + r * kBlockThreads;
          v[r] = e < d ? __ldcs(c.g.adj + b + e) : -1;
          w[r] = e < d && c.g.ew ? (V)__ldcs(c.g.ew + b + e) : (V)1;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) x[r] = v[r] >= 0 ? c.label[v[r]] : -1;
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (x[r] >= 0) add(x[r], w[r]);
      }
    }
    __syncthreads();
    // the top rating among the other labels and the own rating, then the tie
    // order among the top-rated labels only (as in the warp tiers)
    const int32_t own = c.label[u];
    const int64_t cu = node_w(c.g, u), capu = cap_of(c, u);
    int64_t rmax = -1, rown = 0;
    for (int k = tid; k < cap; k += kBlockThreads) {
      const int32_t x = slot_label(k);
      if (x < 0) continue;
      const int64_t R = (int64_t)vals[k];
      if (x == own) rown = R;
      else rmax = R > rmax ? R : rmax;
    }
    block_max2(rmax, rown, red);
    Best b;
    b.init();
    b.rown = rown;
    const bool rate = rmax >= 0 && (MODE != M_LP || rmax > rown);  // uniform over the block
    const TieKey hv = rate ? tie_key<MODE>(c, u) : TieKey{0, 0};
    if (rate) {
      for (int k = tid; k < cap; k += kBlockThreads) {
        const int32_t x = slot_label(k);
        if (x < 0 || x == own || (int64_t)vals[k] != rmax) continue;
        const uint32_t t = MODE == M_REBAL ? 0u : tie_of(hv, x);
        if (better(rmax, t, x, b.r, b.t, b.x)) b.r = rmax, b.t = t, b.x = x;
      }
      block_reduce_best(b, wb);
    }
    // the winner is full: the best admissible label instead (it must improve
    // on the own rating to matter)
    if (rate && MODE != M_FAV && b.x != INT32_MAX && c.lw[b.x] + cu > capu) {
      const int64_t rown = b.rown;
      b.init();
      for (int k = tid; k < cap; k += kBlockThreads) {
        const int32_t x = slot_label(k);
        if (x < 0 || x == own) continue;
        const int64_t R = (int64_t)vals[k];
        if (MODE == M_LP && R <= rown) continue;
        const uint32_t t = MODE == M_REBAL ? 0u : tie_of(hv, x);
        if (better(R, t, x, b.r, b.t, b.x) && c.lw[x] + cu <= capu) b.r = R, b.t = t, b.x = x;
      }
      block_reduce_best(b, wb);
      b.rown = rown;
    }
    if (tid < 32) {
      MoverBuf mb{mu, mt, mo, mg, 0};
      finalize_warp<MODE>(c, b, u, cu, &mb);
      if (MODE == M_LP) flush_movers(c, mb);
    }
    __syncthreads();
  }
}

// Huge tier, phase 1: one block per (vertex, chunk of 1000 neighbours; the
// compressed format's independently decodable chunks) sums the chunk's
// ratings in a shared-memory table and adds them into the vertex's global
// table (the paper's rating maps as flush buffers against contention).
constexpr int kHugeStage = (5 * kChunkSize + 64 + 15) & ~15;  // one chunk's bytes + alignment
template <bool COMP, int MODE, class V, bool DIR>
__global__ void __launch_bounds__(kBlockThreads) k_rate_huge_chunks(RateCtx c) {
  static_assert(kDirectMax <= 1 << kHugeLog, "a counter per block fits the chunk's table");
  __shared__ int32_t keys[DIR ? 1 : 1 << kHugeLog];
  __shared__ V vals[1 << kHugeLog];
  __shared__ __align__(16) uint8_t stage[COMP ? kHugeStage : 16];
  __shared__ uint32_t vbuf[COMP ? kChunkSize : 1];
  __shared__ int64_t red[kBlockThreads / 32 + 1];
  __shared__ int64_t s_vi;
  __shared__ int32_t claimed[1 << kHugeLog];
  __shared__ int32_t s_nclaim, s_base;
  const int tid = threadIdx.x;
  for (int k = tid; k < (1 << kHugeLog); k += kBlockThreads) {
    if (!DIR) keys[k] = -1;
    vals[k] = 0;
  }
  __syncthreads();
  // bucket mode: this sub-round's chunk items; else every chunk, skipping
  // inactive hubs (the hub of an item found by binary search)
  const int64_t ib = c.bpos ? c.hc_pre[c.boff[c.s]] : 0;
  const int64_t ie = c.bpos ? c.hc_pre[c.boff[c.s + 1]] : c.n_chunks;
  for (int64_t item = ib + blockIdx.x; item < ie; item += gridDim.x) {
    int64_t i, j;
    if (c.bpos) {
      const int64_t it = c.hc_item[item];
      i = it >> 32;
      j = it & 0xffffffffLL;
    } else {
      if (tid == 0) {  // vertex index: last i with chunk_start[i] <= item
        int64_t lo = 0, hi = c.list_n - 1;
        while (lo < hi) {
          const int64_t mid = (lo + hi + 1) / 2;
          if (c.chunk_start[mid] <= item) lo = mid;
          else hi = mid - 1;
        }
        s_vi = lo;
      }
      __syncthreads();
      i = s_vi;
      j = item - c.chunk_start[i];
      __syncthreads();  // s_vi is rewritten by the next item
    }
    const int64_t u = c.list[i];
    if (!c.bpos && !active<MODE>(c, u)) continue;  // uniform over the block
    int32_t lb = 0;
    const int32_t nblk = DIR ? block_range(c, u, lb) : 0;
    auto add = [&](int32_t x, V w) {
      if constexpr (DIR) {
        if ((uint32_t)(x - lb) < (uint32_t)nblk) atomicAdd(&vals[x - lb], w);
      } else {
        blk_add<V>(keys, vals, kHugeLog, x, w, c.g.err);
      }
    };
    if (COMP) {
      const ZipNbr z = zip_nbr(c.g, u);
      uint64_t cb, ce;
      int64_t cnt;
      zip_chunk(c.g, z, j, cb, ce, cnt);
      block_decode_range(c.g, u, cb, ce, cnt, stage, vbuf, red, [&](int n) {
        for (int e = tid; e < n; e += kBlockThreads) add(c.label[vbuf[e]], (V)1);
      });
    } else {
      // the chunk's entries (at most four a thread), their loads together
      static_assert(kChunkSize <= 4 * kBlockThreads, "one step per chunk");
      const int64_t b = c.g.xadj[u] + j * kChunkSize;
      const int64_t e = min(b + kChunkSize, c.g.xadj[u + 1]);
      int32_t v[4], x[4];
      V w[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int64_t q = b + tid + r * kBlockThreads;
        v[r] = q < e ? __ldcs(c.g.adj + q) : -1;
        w[r] = q < e && c.g.ew ? (V)__ldcs(c.g.ew + q) : (V)1;
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) x[r] = v[r] >= 0 ? c.label[v[r]] : -1;
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (x[r] >= 0) add(x[r], w[r]);
    }
    __syncthreads();
    int32_t *tk = c.tkeys + c.tbase + c.toff[i];
    int64_t *tv = c.tvals + c.tbase + c.toff[i];
    int32_t *tl = c.tlist + (c.tbase + c.toff[i]) / 2;
    const int lc = c.tcap[i];
    if (tid == 0) s_nclaim = 0;
    __syncthreads();
    // every thread inserts its kFlush shared slots together: each probe
    // step issues all pending key loads, then all claims (atomicCAS), so a
    // thread waits for one round trip per step instead of one per label
    constexpr int kFlush = (1 << kHugeLog) / kBlockThreads;
    {
      const uint32_t mask = (1u << lc) - 1u;
      int32_t lab[kFlush];
      int64_t w[kFlush];
      uint32_t h[kFlush], probes[kFlush];
      bool pend[kFlush];
#pragma unroll
      for (int q = 0; q < kFlush; ++q) {
        const int k = tid + q * kBlockThreads;
        w[q] = (int64_t)vals[k];
        if constexpr (DIR) {
          lab[q] = w[q] ? lb + k : -1;
        } else {
          lab[q] = keys[k];
          keys[k] = -1;
        }
        vals[k] = 0;
        pend[q] = lab[q] >= 0;
        h[q] = pend[q] ? slot_of(lab[q], lc) : 0;
        probes[q] = 0;
      }
      for (;;) {
        bool any = false;
#pragma unroll
        for (int q = 0; q < kFlush; ++q) any |= pend[q];
        if (!any) break;
        int32_t cur[kFlush], prev[kFlush];
#pragma unroll
        for (int q = 0; q < kFlush; ++q) cur[q] = pend[q] ? *(volatile int32_t *)&tk[h[q]] : 0;
#pragma unroll
        for (int q = 0; q < kFlush; ++q)
          prev[q] = pend[q] && cur[q] == -1 ? atomicCAS(&tk[h[q]], -1, lab[q]) : 0;
#pragma unroll
        for (int q = 0; q < kFlush; ++q) {
          if (!pend[q]) continue;
          const int32_t kk = cur[q] == -1 ? (prev[q] == -1 ? lab[q] : prev[q]) : cur[q];
          if (kk == lab[q]) {
            atomicAdd((unsigned long long *)&tv[h[q]], (unsigned long long)w[q]);
            if (cur[q] == -1 && prev[q] == -1) claimed[atomicAdd(&s_nclaim, 1)] = (int32_t)h[q];
            pend[q] = false;
          } else if (++probes[q] > mask) {
            latch_error(c.g.err, TP_ERR_CORRUPT);  // more distinct labels than the table holds
            pend[q] = false;
          } else {
            h[q] = (h[q] + 1) & mask;
          }
        }
      }
    }
    __syncthreads();
    // the slots this chunk filled join the hub's list with one counter update
    if (tid == 0 && s_nclaim) s_base = atomicAdd(c.tcount + i, s_nclaim);
    __syncthreads();
    for (int j = tid; j < s_nclaim; j += kBlockThreads) tl[s_base + j] = claimed[j];
    __syncthreads();
  }
}

// Huge tier, phase 2: one block per vertex scans its global table.
static_assert(2 * sizeof(Best) == kSegBestBytes, "segment results are two Best records");

// Huge tier, phase 2: every (vertex, segment of 4096 table slots) is scanned
// by its own block for its best label ignoring the cap (with the own
// rating) and for its best admissible label; it then clears its slots.
// Admissibility is checked only for a label that beats the thread's best
// admissible one so far, so few label weights are read.
template <int MODE>
__global__ void __launch_bounds__(kBlockThreads) k_rate_huge_scan(RateCtx c, Best *seg_best) {
  __shared__ Best wb[kBlockThreads / 32];
  __shared__ int64_t s_vi;
  const int64_t ib = c.bpos ? c.hs_pre[c.boff[c.s]] : 0;
  const int64_t ie = c.bpos ? c.hs_pre[c.boff[c.s + 1]] : c.n_segs;
  for (int64_t item = ib + blockIdx.x; item < ie; item += gridDim.x) {
    int64_t i, sg;
    if (c.bpos) {
      const int64_t it = c.hs_item[item];
      i = it >> 32;
      sg = it & 0xffffffffLL;
    } else {
      if (threadIdx.x == 0) {  // vertex index: last i with seg_start[i] <= item
        int64_t lo = 0, hi = c.list_n - 1;
        while (lo < hi) {
          const int64_t mid = (lo + hi + 1) / 2;
          if (c.seg_start[mid] <= item) lo = mid;
          else hi = mid - 1;
        }
        s_vi = lo;
      }
      __syncthreads();
      i = s_vi;
      sg = item - c.seg_start[i];
      __syncthreads();
    }
    const int64_t u = c.list[i];
    if (!c.bpos && !active<MODE>(c, u)) continue;
    const int32_t own = c.label[u];
    const int64_t cu = node_w(c.g, u), capu = cap_of(c, u);
    const TieKey hv = tie_key<MODE>(c, u);
    // a table filled to an eighth or more is read in slot order (8192 slots
    // per segment); a sparser one through its list of filled slots (4096
    // list entries per segment)
    const int64_t filled = c.tcount[i], cap = (int64_t)1 << c.tcap[i];
    const bool dense = 8 * filled >= cap;
    const int64_t s0 = sg << kSegLog;
    const int64_t s1 = dense ? min(2 * (s0 + ((int64_t)1 << kSegLog)), cap)
                             : min(s0 + ((int64_t)1 << kSegLog), filled);
    int32_t *tk = c.tkeys + c.tbase + c.toff[i];
    int64_t *tv = c.tvals + c.tbase + c.toff[i];
    const int32_t *tl = c.tlist + (c.tbase + c.toff[i]) / 2;
    Best b, a;
    b.init();
    a.init();
    // kScanBatch slots per thread and step, every load of a step issued
    // before the first is used (list entries, then keys, then values), so a
    // thread waits for one round trip per step instead of one per slot
    constexpr int kScanBatch = 8;
    for (int64_t j0 = (dense ? 2 * s0 : s0) + threadIdx.x; j0 < s1;
         j0 += (int64_t)kBlockThreads * kScanBatch) {
      int32_t sl[kScanBatch], xs[kScanBatch];
      int64_t Rs[kScanBatch];
#pragma unroll
      for (int q = 0; q < kScanBatch; ++q) {
        const int64_t j = j0 + (int64_t)q * kBlockThreads;
        sl[q] = j < s1 ? (dense ? (int32_t)j : tl[j]) : -1;
      }
#pragma unroll
      for (int q = 0; q < kScanBatch; ++q) xs[q] = sl[q] >= 0 ? tk[sl[q]] : -1;
#pragma unroll
      for (int q = 0; q < kScanBatch; ++q) Rs[q] = xs[q] >= 0 ? tv[sl[q]] : 0;
#pragma unroll
      for (int q = 0; q < kScanBatch; ++q) {
        const int32_t x = xs[q];
        if (x < 0) continue;
        const int64_t R = Rs[q];
        tk[sl[q]] = -1;
        tv[sl[q]] = 0;
        if (x == own) {
          b.rown = R;
          continue;
        }
        const uint32_t t = MODE == M_REBAL ? 0u : tie_of(hv, x);
        if (better(R, t, x, b.r, b.t, b.x)) b.r = R, b.t = t, b.x = x;
        if (MODE != M_FAV && better(R, t, x, a.r, a.t, a.x) && c.lw[x] + cu <= capu)
          a.r = R, a.t = t, a.x = x;
      }
    }
    block_reduce_best(b, wb);
    if (MODE != M_FAV) block_reduce_best(a, wb);
    if (threadIdx.x == 0) {  // the hub's segment sg, where the decision reads it
      const int64_t q = c.seg_start[i] + sg;
      seg_best[2 * q] = b;
      seg_best[2 * q + 1] = a;
    }
  }
}

// Huge tier, phase 3: one block per vertex combines its segments: the best
// label if it is admissible, else the best admissible one; then it acts on
// the decision.
template <int MODE>
__global__ void __launch_bounds__(kBlockThreads) k_rate_huge_decide(RateCtx c, const Best *seg_best) {
  __shared__ Best wb[kBlockThreads / 32];
  __shared__ int32_t mu[32], mt[32], mo[32];
  __shared__ int64_t mg[32];
  int64_t kb, ke;
  tier_range(c, kb, ke);
  for (int64_t k = kb + blockIdx.x; k < ke; k += gridDim.x) {
    int64_t i, u;
    if (!tier_entry<MODE>(c, k, i, u)) continue;
    const int64_t cu = node_w(c.g, u);
    Best b, a;
    b.init();
    a.init();
    for (int64_t q = c.seg_start[i] + threadIdx.x; q < c.seg_start[i + 1]; q += kBlockThreads) {
      const Best o = seg_best[2 * q], oa = seg_best[2 * q + 1];
      if (better(o.r, o.t, o.x, b.r, b.t, b.x)) b.r = o.r, b.t = o.t, b.x = o.x;
      b.rown = max(b.rown, o.rown);
      if (better(oa.r, oa.t, oa.x, a.r, a.t, a.x)) a.r = oa.r, a.t = oa.t, a.x = oa.x;
    }
    block_reduce_best(b, wb);
    block_reduce_best(a, wb);
    if (MODE != M_FAV && b.x != INT32_MAX && c.lw[b.x] + cu > cap_of(c, u)) {
      // the winner is full: the best admissible label (for a move it must
      // also improve on the own rating, which finalize_warp checks)
      a.rown = b.rown;
      b = a;
    }
    if (threadIdx.x == 0) c.tcount[i] = 0;  // the segments cleared the table
    if (threadIdx.x < 32) {
      MoverBuf mb{mu, mt, mo, mg, 0};
      finalize_warp<MODE>(c, b, u, cu, &mb);
      if (MODE == M_LP) flush_movers(c, mb);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- approval
// A: targets that fit take every mover; the others become contested and
// count their movers (the first one also lists the target).
__global__ void k_approve_fit(ApproveCtx a) {
  int64_t nm = (int64_t)a.counters[0];
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nm;
       i += (int64_t)gridDim.x * blockDim.x) {
    int32_t t = a.mv_t[i];
    bool fits = a.lw[t] + a.in_w[t] <= target_cap(a, t);
    a.mv_ok[i] = fits;
    if (!fits && atomicAdd(&a.ccnt[t], 1) == 0) {
      unsigned long long j = atomicAdd(&a.counters[1], 1ull);
      a.ctarget[j] = t;
    }
  }
}

// A2: every contested target reserves its segment of the contested list.
__global__ void k_approve_alloc(ApproveCtx a) {
  int64_t nt = (int64_t)a.counters[1];
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nt;
       j += (int64_t)gridDim.x * blockDim.x) {
    const int32_t t = a.ctarget[j], c = a.ccnt[t];
    a.cbase[t] = (int64_t)atomicAdd(&a.counters[2], (unsigned long long)c);
    if (c > 32) a.cbig[atomicAdd(&a.counters[3], 1ull)] = t;
  }
}

// B: contested movers are grouped by target.
__global__ void k_approve_scatter(ApproveCtx a) {
  int64_t nm = (int64_t)a.counters[0];
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nm;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (a.mv_ok[i]) continue;
    put_contested(a, i, a.mv_t[i]);
  }
}

// 1024 threads: the movers into a hub's cluster can be 1e5 and more, one
// block's work (with 256 threads and the gains behind two index loads such a
// segment took 0.19 ms).
constexpr int kContestedThreads = 1024;
__global__ void __launch_bounds__(kContestedThreads) k_approve_contested(ApproveCtx a) {
  approve_targets(a, (int64_t)a.counters[1], (int64_t)a.counters[3], (int)blockIdx.x, (int)gridDim.x);
}

// D: apply approved moves and reset the per-target counters. The grid covers
// the largest possible mover count, so every mover has its own thread and
// the dependent loads of different movers overlap.
__global__ void k_apply(ApproveCtx a) {
  int64_t nm = (int64_t)a.counters[0];
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nm;
       i += (int64_t)gridDim.x * blockDim.x) {
    int32_t t = a.mv_t[i];
    if (a.mv_ok[i]) {
      int32_t u = a.mv_u[i];
      int64_t w = vwt(a, u);
      int32_t own = a.mv_o[i];  // labels change only here, so this is still u's label
      a.label[u] = t;
      atomicAdd((unsigned long long *)&a.lw[t], (unsigned long long)w);
      atomicAdd((unsigned long long *)&a.lw[own], (unsigned long long)(-w));
    }
    a.in_w[t] = 0;
  }
}

__global__ void k_init_singletons(const int64_t *vw, int64_t n, int32_t *label, int64_t *lw) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    label[u] = (int32_t)u;
    lw[u] = vw ? vw[u] : 1;
  }
}

// ---------------------------------------------------------------- tier dispatch
// Algorithmic bytes one round of rating must move for the vertices of one
// tier (level 0, unit weights): the tier's share of the adjacency stream and
// its offsets, one 4-byte label gather per adjacency entry, the own label
// and one 8-byte label-weight read per vertex.
double tier_round_bytes(const tp_graph *g, int64_t n_t, int64_t e_t) {
  double adj = g->compressed
                   ? (double)g->nbytes * (g->m2 ? (double)e_t / (double)g->m2 : 0.0) +
                         (double)n_t * (g->off_is64 ? 8.0 : 4.0)
                   : 4.0 * (double)e_t + 8.0 * (double)n_t;
  return adj + 4.0 * (double)e_t + 12.0 * (double)n_t;
}

// Entries in the tiers above the small one from which their kernels go side by
// side: a fork and join cost about 10 us of launches per sub-round. With against
// without, clustering: R-MAT with 1.3e6 such entries 0.58, 4e6 0.60, 2.4e7 0.65,
// a mesh with 1.8e6 0.88, a uniform random graph with 6e6 in one tier 1.05.
constexpr int64_t kForkEntries = (int64_t)1 << 19;

template <int MODE>
void rate_tiers(tp_graph *g, RateCtx c, const tp_params &p, cudaStream_t s,
                TierStreams *side = nullptr) {
  build_tiers(g, p, s);
  ensure_hub_tables(g, s);
  TierCache &T = g->tiers;
  c.g = view(g);
  c.tier = T.tier.get();
  {  // table slots per neighbour: a power of two in 1..8
    const int32_t sl = std::max(1, std::min(8, p.table_slack));
    c.slack = 1;
    while (c.slack < sl) c.slack <<= 1;
  }
  c.tkeys = T.tkeys.get();
  c.tvals = T.tvals.get();
  c.tlist = T.tlist.get();
  c.tcount = T.tcount.get();
  const int sms = num_sms();
  const bool comp = g->compressed;
  const bool prof = MODE == M_LP && prof_active();
  // bucket mode (M_LP with this round's tier buckets): tier t walks its
  // sub-round's positions only
  auto bucketed = [&](RateCtx &m, int t) {
    if (MODE == M_LP && c.tb_pos) {
      m.bpos = c.tb_pos + c.tb_base[t];
      m.boff = c.tb_off + (int64_t)t * (c.S + 1);
    } else {
      m.bpos = nullptr;
      m.boff = nullptr;
    }
  };
  const double per_launch = MODE == M_LP && c.S > 0 ? 1.0 / c.S : 0.0;
  const int64_t n_lane = MODE == M_REBAL ? 0 : T.count[TIER_LANE];
  const int64_t n_small = T.count[TIER_SMALL] + (MODE == M_REBAL ? T.count[TIER_LANE] : 0);
  const bool fork = side && !prof &&
                    T.edges[TIER_MID] + T.edges[TIER_BIG] + T.edges[TIER_HUGE] >= kForkEntries &&
                    side->make();
  cudaStream_t s_mid = fork ? side->st[0] : s, s_big = fork ? side->st[1] : s,
               s_big2 = fork ? side->st[2] : s, s_huge = fork ? side->st[3] : s;
  if (fork) side->begin(s);
  if (n_lane > 0) {
    if (prof) prof_begin(PF_RATE_LANE, s);
    constexpr int LM = MODE == M_REBAL ? M_LP : MODE;
    // windows of this launch's list: full where every warp gets one, shorter
    // ones spread a small list over the warps (a coarse level of 4e4 lane
    // vertices: four batches in series on 40 warps took 65 us, one each on 156
    // warps 27). From the host: a value in a register of the compressed kernel
    // costs it a tenth of its speed.
    auto lane_window = [&](int64_t warps) {
      const int64_t list = (n_lane + std::max(c.S, 1) - 1) / std::max(c.S, 1);
      c.lane_win = (int32_t)std::min<int64_t>(kLaneWin, ((list + warps - 1) / warps + 31) & ~31ll);
    };
    if (g->unit_ew) {
      unsigned blocks = (unsigned)std::min<int64_t>(
          (g->n + 256 * kLaneWarps - 1) / (256 * kLaneWarps), (int64_t)sms * kLaneBlocksPerSM);
      lane_window((int64_t)blocks * kLaneWarps);
      // batched graphs are CSR unions
      if (MODE == M_LP && c.quiet && comp) launch(k_rate_lane_quiet<true, false>, blocks, 32 * kLaneWarps, 0, s, c);
      else if (MODE == M_LP && c.quiet) launch(k_rate_lane_quiet<false, false>, blocks, 32 * kLaneWarps, 0, s, c);
      else if (comp && T.lane_long) launch(k_rate_lane<true, LM, false, true>, blocks, 32 * kLaneWarps, 0, s, c);
      else if (comp) launch(k_rate_lane<true, LM, false>, blocks, 32 * kLaneWarps, 0, s, c);
      else if (c.seg.gid) launch(k_rate_lane<false, LM, false, false, true>, blocks, 32 * kLaneWarps, 0, s, c);
      else launch(k_rate_lane<false, LM, false>, blocks, 32 * kLaneWarps, 0, s, c);
    } else {  // weighted levels are CSR
      constexpr int WW = lane_warps<true>();
      unsigned blocks =
          (unsigned)std::min<int64_t>((g->n + 256 * WW - 1) / (256 * WW), (int64_t)sms * 16);
      lane_window((int64_t)blocks * WW);
      // labels are vertices or, in refinement, block numbers
      const bool wide = g->n > kLaneKeyLabels || c.nlabels > kLaneKeyLabels;
      if (MODE == M_LP && c.quiet) launch(k_rate_lane_quiet<false, true>, blocks, 32 * WW, 0, s, c);
      else if (c.seg.gid && wide) launch(k_rate_lane<false, LM, true, true, true>, blocks, 32 * WW, 0, s, c);
      else if (c.seg.gid) launch(k_rate_lane<false, LM, true, false, true>, blocks, 32 * WW, 0, s, c);
      else if (wide) launch(k_rate_lane<false, LM, true, true>, blocks, 32 * WW, 0, s, c);
      else launch(k_rate_lane<false, LM, true>, blocks, 32 * WW, 0, s, c);
    }
    TP_LAUNCH_CHECK();
    if (prof) prof_end(PF_RATE_LANE, s, per_launch * tier_round_bytes(g, n_lane, T.edges[TIER_LANE]));
  }
  // sums in 32 bits wherever all edge weights of the graph together fit
  // (compressed levels have unit weights)
  const bool narrow = g->unit_ew || ew_sum_bound(g) < ((int64_t)1 << 31);
  // few labels: direct tables for every tier above the small one, and for the
  // small one where k counters are no more than its largest hash table
  const bool direct = MODE != M_FAV && c.kmax > 0 && c.kmax <= kDirectMax;
  auto run_direct = [&](const int32_t *list, int64_t cnt, int t, cudaStream_t s) {
    RateCtx m = c;
    m.list = list;
    m.list_n = cnt;
    bucketed(m, t);
    constexpr int DM = MODE == M_FAV ? M_LP : MODE;
    const unsigned blocks =
        (unsigned)std::min<int64_t>((cnt + kDirectWarps - 1) / kDirectWarps, (int64_t)sms * 16);
    const size_t sm = (size_t)c.kmax * kDirectWarps * (narrow ? 4 : 8);
    if (comp) launch(k_rate_direct<true, DM, uint32_t>, blocks, 32 * kDirectWarps, sm, s, m, c.kmax);
    else if (narrow) launch(k_rate_direct<false, DM, uint32_t>, blocks, 32 * kDirectWarps, sm, s, m, c.kmax);
    else launch(k_rate_direct<false, DM, unsigned long long>, blocks, 32 * kDirectWarps, sm, s, m, c.kmax);
    TP_LAUNCH_CHECK();
  };
  if (n_small > 0) {
    if (prof) prof_begin(PF_RATE_SMALL, s);
    if (MODE != M_REBAL && direct && c.kmax <= 1 << kSmallLog) {
      run_direct(T.small.get(), T.n_small, 0, s);
    } else {
      int wpb = p.warps_per_block >= 1 && p.warps_per_block <= 16 ? p.warps_per_block : 8;
      size_t sm = (narrow ? sizeof(WarpSmem<kSmallLog, uint32_t>) : sizeof(WarpSmem<kSmallLog>)) * wpb;
      RateCtx m = c;
      int64_t items = g->n;
      if (MODE != M_REBAL) {
        m.list = T.small.get();
        m.list_n = T.n_small;
        items = T.n_small;
        bucketed(m, 0);
      } else {
        m.list = nullptr;
      }
      const int64_t per_warp = MODE != M_REBAL ? 1 : 32;  // list entries / vertices per warp step
      unsigned blocks = (unsigned)std::min<int64_t>((items + per_warp * wpb - 1) / (per_warp * wpb),
                                                    (int64_t)sms * 16);
      if (comp) launch(k_rate_small<true, MODE, uint32_t>, blocks, 32 * wpb, sm, s, m);
      else if (narrow) launch(k_rate_small<false, MODE, uint32_t>, blocks, 32 * wpb, sm, s, m);
      else launch(k_rate_small<false, MODE, int64_t>, blocks, 32 * wpb, sm, s, m);
      TP_LAUNCH_CHECK();
    }
    if (prof) prof_end(PF_RATE_SMALL, s, per_launch * tier_round_bytes(g, T.count[TIER_SMALL], T.edges[TIER_SMALL]));
  }
  if (T.n_mid + T.n_mid2 > 0) {
    cudaStream_t s = s_mid;
    if (prof) prof_begin(PF_RATE_MID, s);
    auto run = [&](const int32_t *list, int64_t cnt, int t, bool big_tables) {
      if (!cnt) return;
      if (direct) return run_direct(list, cnt, t, s);
      RateCtx m = c;
      m.list = list;
      m.list_n = cnt;
      bucketed(m, t);
      const unsigned blocks =
          (unsigned)std::min<int64_t>((cnt + kMidWarps - 1) / kMidWarps, (int64_t)sms * 16);
#define TP_MID(LG, V)                                                                         \
  do {                                                                                        \
    const size_t sm = sizeof(WarpSmem<LG, V>) * kMidWarps;                                    \
    if (comp) launch(k_rate_list<true, MODE, LG, V>, blocks, 32 * kMidWarps, sm, s, m);      \
    else launch(k_rate_list<false, MODE, LG, V>, blocks, 32 * kMidWarps, sm, s, m);          \
  } while (0)
      if (big_tables) {
        if (narrow) TP_MID(kMidLog, uint32_t);
        else TP_MID(kMidLog, int64_t);
      } else {
        if (narrow) TP_MID(kMidSmallLog, uint32_t);
        else TP_MID(kMidSmallLog, int64_t);
      }
#undef TP_MID
      TP_LAUNCH_CHECK();
    };
    run(T.mid.get(), T.n_mid, 1, false);
    run(T.mid2.get(), T.n_mid2, 2, true);
    if (prof) prof_end(PF_RATE_MID, s, per_launch * tier_round_bytes(g, T.n_mid + T.n_mid2, T.edges[TIER_MID]));
  }
  if (T.n_big0 + T.n_big1 + T.n_big + T.n_big2 > 0) {
    if (prof) prof_begin(PF_RATE_BIG, s);
    auto run = [&](const int32_t *list, int64_t cnt, int maxlog, int t, cudaStream_t s) {
      if (!cnt) return;
      RateCtx m = c;
      m.list = list;
      m.list_n = cnt;
      bucketed(m, t);
      const size_t table = direct ? (size_t)((c.kmax + 3) & ~3) * (narrow ? 4 : 8)
                                  : ((size_t)1 << maxlog) * (sizeof(int32_t) + (narrow ? 4 : 8));
      const size_t sm = table + (comp ? block_stage_bytes(block_max_deg(maxlog)) +
                                            block_vbuf_bytes(block_max_deg(maxlog))
                                      : 0);
      const int per_sm = std::max(1, std::min(8, (int)((size_t)(228 * 1024) / (sm + 2048))));
      const unsigned blocks = (unsigned)std::min<int64_t>(cnt, (int64_t)sms * per_sm);
      constexpr int DM = MODE == M_FAV ? M_LP : MODE;
#define TP_BLK(CM, V)                                                                            \
  do {                                                                                           \
    if (direct) launch(k_rate_block<CM, DM, V, true>, blocks, kBlockThreads, sm, s, m, maxlog, c.kmax); \
    else launch(k_rate_block<CM, MODE, V, false>, blocks, kBlockThreads, sm, s, m, maxlog, 0);   \
  } while (0)
      if (comp) TP_BLK(true, uint32_t);
      else if (narrow) TP_BLK(false, uint32_t);
      else TP_BLK(false, unsigned long long);
#undef TP_BLK
      TP_LAUNCH_CHECK();
    };
    if (T.n_big0 && direct) run_direct(T.big0.get(), T.n_big0, 3, s_big);
    else run(T.big0.get(), T.n_big0, kBlockTinyLog, 3, s_big);
    run(T.big1.get(), T.n_big1, kBlockMidLog, 4, s_big);
    run(T.big.get(), T.n_big, kBlockSmallLog, 5, s_big2);
    run(T.big2.get(), T.n_big2, kBlockBigLog, 6, s_big2);
    if (prof) prof_end(PF_RATE_BIG, s, per_launch * tier_round_bytes(g, T.n_big0 + T.n_big1 + T.n_big + T.n_big2, T.edges[TIER_BIG]));
  }
  if (T.n_huge > 0) {
    cudaStream_t s = s_huge;
    if (prof) prof_begin(PF_RATE_HUGE, s);
    RateCtx m = c;
    m.list = T.huge.get();
    m.list_n = T.n_huge;
    bucketed(m, 7);
    m.toff = T.huge_toff.get();
    m.tcap = T.huge_tcap.get();
    m.tbase = 0;
    m.chunk_start = T.huge_chunk_start.get();
    m.n_chunks = T.n_huge_chunks;
    const unsigned blocks = (unsigned)std::max<int64_t>(
        1, std::min<int64_t>(T.n_huge_chunks, (int64_t)sms * 6));
    constexpr int DM = MODE == M_FAV ? M_LP : MODE;
#define TP_HUGE(CM, V)                                                                           \
  do {                                                                                           \
    if (direct) launch(k_rate_huge_chunks<CM, DM, V, true>, blocks, kBlockThreads, 0, s, m);     \
    else launch(k_rate_huge_chunks<CM, MODE, V, false>, blocks, kBlockThreads, 0, s, m);         \
  } while (0)
    if (comp) TP_HUGE(true, uint32_t);
    else if (narrow) TP_HUGE(false, uint32_t);
    else TP_HUGE(false, unsigned long long);
#undef TP_HUGE
    TP_LAUNCH_CHECK();
    m.seg_start = T.huge_seg_start.get();
    m.n_segs = T.n_huge_segs;
    Best *seg_best = reinterpret_cast<Best *>(T.huge_seg_best.get());
    const unsigned sb = (unsigned)std::max<int64_t>(1, std::min<int64_t>(T.n_huge_segs, (int64_t)sms * 8));
    launch(k_rate_huge_scan<MODE>, sb, kBlockThreads, 0, s, m, seg_best);
    const unsigned db = (unsigned)std::max<int64_t>(1, std::min<int64_t>(T.n_huge, (int64_t)sms * 4));
    launch(k_rate_huge_decide<MODE>, db, kBlockThreads, 0, s, m, (const Best *)seg_best);
    TP_LAUNCH_CHECK();
    if (prof) prof_end(PF_RATE_HUGE, s, per_launch * tier_round_bytes(g, T.n_huge, T.edges[TIER_HUGE]));
  }
  if (fork) side->end(s);
}

template <class K>
void set_smem_limits(K kernel, size_t bytes) {
  TP_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
}

void configure_kernels_once() {
  size_t small16 = sizeof(WarpSmem<kSmallLog>) * 16;
#define TP_CFG_MID(M, LG, V)                                                       \
  set_smem_limits(k_rate_list<true, M, LG, V>, sizeof(WarpSmem<LG, V>) * kMidWarps); \
  set_smem_limits(k_rate_list<false, M, LG, V>, sizeof(WarpSmem<LG, V>) * kMidWarps);
#define TP_CFG_MODE(M)                                              \
  set_smem_limits(k_rate_small<true, M, uint32_t>, small16);        \
  set_smem_limits(k_rate_small<false, M, uint32_t>, small16);       \
  set_smem_limits(k_rate_small<false, M, int64_t>, small16);        \
  TP_CFG_MID(M, kMidSmallLog, uint32_t)                             \
  TP_CFG_MID(M, kMidSmallLog, int64_t)                              \
  TP_CFG_MID(M, kMidLog, uint32_t)                                  \
  TP_CFG_MID(M, kMidLog, int64_t)

  TP_CFG_MODE(M_LP)
  TP_CFG_MODE(M_FAV)
  TP_CFG_MODE(M_REBAL)
#undef TP_CFG_MODE
#undef TP_CFG_MID
  // the largest dynamic shared memory: weighted CSR with 16384 slots, or
  // compressed with 16384 slots and the record staging
  const size_t blk = std::max(((size_t)1 << kBlockBigLog) * (sizeof(int32_t) + 8),
                              ((size_t)1 << kBlockBigLog) * (sizeof(int32_t) + 4) +
                                  block_stage_bytes(kChunkThreshold) +
                                  block_vbuf_bytes(kChunkThreshold));
#define TP_CFG_BLOCK(M)                                   \
  set_smem_limits(k_rate_block<true, M, uint32_t, false>, blk);            \
  set_smem_limits(k_rate_block<false, M, uint32_t, false>, blk);           \
  set_smem_limits(k_rate_block<false, M, unsigned long long, false>, blk);
  TP_CFG_BLOCK(M_LP)
  TP_CFG_BLOCK(M_FAV)
  TP_CFG_BLOCK(M_REBAL)
#undef TP_CFG_BLOCK
  // direct tables: the record staging of compressed graphs dominates
  const size_t dir = (size_t)kDirectMax * 4 + block_stage_bytes(kChunkThreshold) +
                     block_vbuf_bytes(kChunkThreshold);
  set_smem_limits(k_rate_block<true, M_LP, uint32_t, true>, dir);
  set_smem_limits(k_rate_block<true, M_REBAL, uint32_t, true>, dir);
}

void configure_kernels() {
  static std::once_flag once;
  std::call_once(once, configure_kernels_once);
}

// A3: the lane-tier vertices of one round grouped by sub-round, in ascending
// vertex order inside every sub-round. Block b owns vertices
// [b * kBucketSpan, (b + 1) * kBucketSpan); pass 0 writes its count per
// sub-round to cnt[s * nblocks + b], an exclusive scan turns the counts into
// offsets, pass 1 writes every vertex at its offset plus its rank inside the
// block (chunks of 32 vertices in order, ballot ranks inside a chunk).
constexpr int kBucketSpan = 2048;
constexpr int kBucketChunks = kBucketSpan / 32;

// Pass 0 hashes every vertex once and keeps its sub-round + 1 in sub_byte
// (every rating tier tests it instead of hashing again) and counts the lane
// tier; pass 1 lists the lane tier. Lanes of a 32-vertex chunk with the
// same sub-round are grouped with one match instruction.
// With offsets (compressed graphs), pass 1 also stores each listed vertex's
// record start << 8 | record length in rec (lane-tier records are <= 65 bytes).
// Batched graphs (gid non-null): a vertex hashes its number inside its graph.
__global__ void __launch_bounds__(256) k_bucket(const uint8_t *tier, int64_t n, uint64_t rk_in,
                                                const uint64_t *rk_dev, int32_t S, bool fill,
                                                int64_t *cnt, int32_t *bucket, uint8_t *sub_byte,
                                                const uint32_t *o32, const uint64_t *o64,
                                                uint64_t *rec, const int32_t *gid,
                                                const int64_t *vb) {
  __shared__ int32_t chunk_cnt[kBucketChunks][32];  // [chunk][sub-round], S <= 32
  const int lane = lane_id(), w = threadIdx.x >> 5;
  const int64_t nblocks = gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * kBucketSpan;
  for (int i = threadIdx.x; i < kBucketChunks * 32; i += blockDim.x) (&chunk_cnt[0][0])[i] = 0;
  __syncthreads();
  const uint64_t rk = fill ? 0 : (rk_dev ? *rk_dev : rk_in);
  int32_t sub_of[kBucketChunks / 8];
  for (int q = 0; q < kBucketChunks / 8; ++q) {
    const int chunk = w + 8 * q;
    const int64_t u = lo + 32 * chunk + lane;
    int32_t sub = -1;
    if (u < n) {
      if (fill) {
        sub = tier[u] == TIER_LANE ? (int32_t)sub_byte[u] - 1 : -1;
      } else {
        // every vertex's sub-round is kept (the other tiers test it); only
        // the lane tier is listed
        const int64_t lu = gid ? u - vb[gid[u]] : u;
        const int32_t sr = sub_round_of(hstep(rk, (uint64_t)lu), S);
        sub_byte[u] = (uint8_t)(sr + 1);
        sub = tier[u] == TIER_LANE ? sr : -1;
      }
    }
    sub_of[q] = sub;
    const unsigned peers = __match_any_sync(kFull, sub);
    if (sub >= 0 && (peers & lanemask_lt()) == 0) chunk_cnt[chunk][sub] = __popc(peers);
  }
  __syncthreads();
  if (!fill) {
    for (int32_t k = threadIdx.x; k < S; k += blockDim.x) {
      int64_t t = 0;
      for (int ch = 0; ch < kBucketChunks; ++ch) t += chunk_cnt[ch][k];
      cnt[(int64_t)k * nblocks + blockIdx.x] = t;
    }
    return;
  }
  // exclusive prefix over the chunks of this block, per sub-round
  if (threadIdx.x < S) {
    const int k = threadIdx.x;
    int32_t run = 0;
    for (int ch = 0; ch < kBucketChunks; ++ch) {
      const int32_t c = chunk_cnt[ch][k];
      chunk_cnt[ch][k] = run;
      run += c;
    }
  }
  __syncthreads();
  for (int q = 0; q < kBucketChunks / 8; ++q) {
    const int chunk = w + 8 * q;
    const int32_t sub = sub_of[q];
    const unsigned peers = __match_any_sync(kFull, sub);
    if (sub >= 0) {
      const int64_t pos = cnt[(int64_t)sub * nblocks + blockIdx.x] + chunk_cnt[chunk][sub] +
                          __popc(peers & lanemask_lt());
      const int64_t u = lo + 32 * chunk + lane;
      bucket[pos] = (int32_t)u;
      if (rec) {
        const uint64_t b = o32 ? o32[u] : o64[u], e = o32 ? o32[u + 1] : o64[u + 1];
        rec[pos] = b << 8 | (e - b);
      }
    }
  }
}

// The lists of the warp and block tiers lie side by side (TierCache::lists):
// start[t] .. start[t + 1] is list t.
struct TierRanges {
  int64_t start[LpWork::kTiers + 1];
  __device__ __forceinline__ int tier(int64_t k) const {
    int t = 0;
#pragma unroll
    for (int i = 1; i < LpWork::kTiers; ++i) t += k >= start[i];
    return t;
  }
};

// Tier buckets: every list's vertices per sub-round (from sub_byte), all lists
// in one launch.
__global__ void k_tier_count(const int32_t *lists, TierRanges r, const uint8_t *sub_byte, int32_t S,
                             int64_t *cnt) {
  __shared__ int32_t sc[LpWork::kTiers * 32];
  for (int i = threadIdx.x; i < LpWork::kTiers * 32; i += blockDim.x) sc[i] = 0;
  __syncthreads();
  const int64_t n = r.start[LpWork::kTiers];
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&sc[r.tier(k) * 32 + sub_byte[lists[k]] - 1], 1);
  __syncthreads();
  for (int i = threadIdx.x; i < LpWork::kTiers * 32; i += blockDim.x)
    if (sc[i])
      atomicAdd((unsigned long long *)&cnt[(i >> 5) * S + (i & 31)], (unsigned long long)sc[i]);
}

// Offsets of every tier's sub-rounds (one block): off[t * (S + 1) + s].
__global__ void k_tier_offsets(const int64_t *cnt, int32_t S, int tiers, int64_t *off, int64_t *cur) {
  if (threadIdx.x >= tiers) return;
  const int t = threadIdx.x;
  int64_t run = 0;
  for (int s = 0; s < S; ++s) {
    const int64_t c = cnt[t * S + s];  // cnt and cur may be the same array
    off[t * (S + 1) + s] = run;
    cur[t * S + s] = run;
    run += c;
  }
  off[t * (S + 1) + S] = run;
}

// Scatters every list's positions into its sub-round buckets: each block counts
// its slice of the lists per tier and sub-round, reserves the ranges with one
// atomic each, then places its entries (the order inside a bucket does not
// matter).
constexpr int kTierSlice = 4096;
__global__ void k_tier_scatter(const int32_t *lists, TierRanges r, const uint8_t *sub_byte,
                               int32_t S, int64_t *cur, int32_t *pos) {
  __shared__ int32_t sc[LpWork::kTiers * 32];
  __shared__ int64_t base[LpWork::kTiers * 32];
  const int64_t n = r.start[LpWork::kTiers];
  for (int64_t lo = (int64_t)blockIdx.x * kTierSlice; lo < n; lo += (int64_t)gridDim.x * kTierSlice) {
    const int64_t hi = min(lo + kTierSlice, n);
    for (int i = threadIdx.x; i < LpWork::kTiers * 32; i += blockDim.x) sc[i] = 0;
    __syncthreads();
    for (int64_t k = lo + threadIdx.x; k < hi; k += blockDim.x)
      atomicAdd(&sc[r.tier(k) * 32 + sub_byte[lists[k]] - 1], 1);
    __syncthreads();
    for (int i = threadIdx.x; i < LpWork::kTiers * 32; i += blockDim.x) {
      base[i] = sc[i] ? (int64_t)atomicAdd((unsigned long long *)&cur[(i >> 5) * S + (i & 31)],
                                           (unsigned long long)sc[i])
                      : 0;
      sc[i] = 0;
    }
    __syncthreads();
    for (int64_t k = lo + threadIdx.x; k < hi; k += blockDim.x) {
      const int t = r.tier(k), i = t * 32 + sub_byte[lists[k]] - 1;
      pos[r.start[t] + base[i] + atomicAdd(&sc[i], 1)] = (int32_t)(k - r.start[t]);
    }
    __syncthreads();
  }
}

// Huge tier: chunk and segment counts of the hubs in bucket order.
__global__ void k_huge_counts(const int32_t *bpos, int64_t nh, const int64_t *chunk_start,
                              const int64_t *seg_start, int64_t *hc, int64_t *hs) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nh;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = bpos[k];
    hc[k] = chunk_start[p + 1] - chunk_start[p];
    hs[k] = seg_start[p + 1] - seg_start[p];
  }
}

// Huge tier: the items of every hub (warp per hub), hub position << 32 | index.
__global__ void k_huge_items(const int32_t *bpos, int64_t nh, const int64_t *pre,
                             int64_t *item) {
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t k = gw; k < nh; k += nw) {
    const int64_t p = bpos[k];
    for (int64_t j = pre[k] + lane_id(); j < pre[k + 1]; j += 32) item[j] = p << 32 | (j - pre[k]);
  }
}

}  // namespace

// Buckets the warp and block tiers' lists of this round by sub-round.
static void tier_buckets(tp_graph *g, LpWork &w, int32_t S, cudaStream_t stream) {
  TierCache &T = g->tiers;
  const int64_t lens[LpWork::kTiers] = {T.n_small, T.n_mid, T.n_mid2, T.n_big0,
                                        T.n_big1,  T.n_big, T.n_big2, T.n_huge};
  int64_t total = 0;
  TierRanges r;
  for (int t = 0; t < LpWork::kTiers; ++t) r.start[t] = w.tb_base[t] = total, total += lens[t];
  r.start[LpWork::kTiers] = total;
  w.tb_valid = false;
  if (total == 0) return;
  if ((int64_t)w.tb_pos.n < total) w.tb_pos.alloc(total, stream);
  if ((int64_t)w.tb_off.n < LpWork::kTiers * 33) {
    w.tb_off.alloc(LpWork::kTiers * 33, stream);
    w.tb_cur.alloc(LpWork::kTiers * 32, stream);
  }
  TP_CUDA(cudaMemsetAsync(w.tb_cur.get(), 0, sizeof(int64_t) * LpWork::kTiers * S, stream));
  const int sms = num_sms();
  launch(k_tier_count, grid_for(total, 256, (int64_t)sms * 4), 256, 0, stream, T.lists.get(), r,
         w.bucket_sub.get(), S, w.tb_cur.get());
  launch(k_tier_offsets, 1, 32, 0, stream, w.tb_cur.get(), S, LpWork::kTiers, w.tb_off.get(),
         w.tb_cur.get());
  launch(k_tier_scatter, grid_for(total, kTierSlice, (int64_t)sms * 4), 256, 0, stream, T.lists.get(), r,
         w.bucket_sub.get(), S, w.tb_cur.get(), w.tb_pos.get());
  TP_LAUNCH_CHECK();
  if (T.n_huge) {
    const int64_t nh = T.n_huge;
    if ((int64_t)w.hc_pre.n < nh + 1) {
      w.hc_pre.alloc(nh + 1, stream);
      w.hs_pre.alloc(nh + 1, stream);
    }
    if ((int64_t)w.hc_item.n < std::max<int64_t>(T.n_huge_chunks, 1))
      w.hc_item.alloc(std::max<int64_t>(T.n_huge_chunks, 1), stream);
    if ((int64_t)w.hs_item.n < std::max<int64_t>(T.n_huge_segs, 1))
      w.hs_item.alloc(std::max<int64_t>(T.n_huge_segs, 1), stream);
    const int32_t *hp = w.tb_pos.get() + w.tb_base[7];
    launch(k_huge_counts, grid_for(nh, 256), 256, 0, stream, hp, nh, T.huge_chunk_start.get(),
           T.huge_seg_start.get(), w.hc_pre.get(), w.hs_pre.get());
    exclusive_scan_i64(w.hc_pre.get(), w.hc_pre.get(), nh, stream);
    exclusive_scan_i64(w.hs_pre.get(), w.hs_pre.get(), nh, stream);
    launch(k_huge_items, grid_for(nh * 32, 256), 256, 0, stream, hp, nh, w.hc_pre.get(),
           w.hc_item.get());
    launch(k_huge_items, grid_for(nh * 32, 256), 256, 0, stream, hp, nh, w.hs_pre.get(),
           w.hs_item.get());
    TP_LAUNCH_CHECK();
  }
  w.tb_valid = true;
}

void lp_bucket(tp_graph *g, LpWork &w, uint64_t rk, int32_t S, const tp_params &p,
               cudaStream_t stream, const uint64_t *rk_dev, bool tiers, const SegLp *seg) {
  const int32_t *gid = seg ? seg->gid : nullptr;
  const int64_t *vb = seg ? seg->vb : nullptr;
  build_tiers(g, p, stream);
  w.bucket_S = 0;
  if (S > 32) return;
  const int64_t nblocks = (g->n + kBucketSpan - 1) / kBucketSpan;
  if (!w.bucket.get()) w.bucket.alloc(std::max<int64_t>(w.n, 1), stream);
  if (!w.bucket_sub.get()) w.bucket_sub.alloc(std::max<int64_t>(w.n, 1), stream);
  if ((int64_t)w.bucket_off.n < S * nblocks + 1) w.bucket_off.alloc(S * nblocks + 1, stream);
  const bool zrec = g->compressed != 0;
  if (zrec && !w.bucket_rec.get()) w.bucket_rec.alloc(std::max<int64_t>(w.n, 1), stream);
  const uint32_t *o32 = zrec && !g->off_is64 ? g->off32.get() : nullptr;
  const uint64_t *o64 = zrec && g->off_is64 ? g->off64.get() : nullptr;
  uint64_t *rec = zrec ? w.bucket_rec.get() : nullptr;
  launch(k_bucket, (unsigned)nblocks, 256, 0, stream, g->tiers.tier.get(), g->n, rk, rk_dev, S,
         false, w.bucket_off.get(), w.bucket.get(), w.bucket_sub.get(), o32, o64, rec, gid, vb);
  exclusive_scan_i64(w.bucket_off.get(), w.bucket_off.get(), S * nblocks, stream);
  launch(k_bucket, (unsigned)nblocks, 256, 0, stream, g->tiers.tier.get(), g->n, rk, rk_dev, S,
         true, w.bucket_off.get(), w.bucket.get(), w.bucket_sub.get(), o32, o64, rec, gid, vb);
  TP_LAUNCH_CHECK();
  w.bucket_S = S;
  w.bucket_nblocks = nblocks;
  w.tb_valid = false;
  if (tiers) tier_buckets(g, w, S, stream);
}

bool TierStreams::make() {
  if (made) return st[0] != nullptr;
  made = true;
  bool ok = cudaEventCreateWithFlags(&forked, cudaEventDisableTiming) == cudaSuccess;
  for (int i = 0; i < kN && ok; ++i)
    ok = cudaStreamCreateWithFlags(&st[i], cudaStreamNonBlocking) == cudaSuccess &&
         cudaEventCreateWithFlags(&joined[i], cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    (void)cudaGetLastError();
    for (int i = 0; i < kN; ++i) {
      if (st[i]) cudaStreamDestroy(st[i]);
      st[i] = nullptr;
    }
  }
  return ok;
}

void TierStreams::begin(cudaStream_t s) {
  TP_CUDA(cudaEventRecord(forked, s));
  open = true;
  for (int i = 0; i < kN; ++i) TP_CUDA(cudaStreamWaitEvent(st[i], forked, 0));
}

void TierStreams::end(cudaStream_t s) {
  for (int i = 0; i < kN; ++i) {
    TP_CUDA(cudaEventRecord(joined[i], st[i]));
    TP_CUDA(cudaStreamWaitEvent(s, joined[i], 0));
  }
  open = false;
}

TierStreams::~TierStreams() {
  for (int i = 0; i < kN; ++i) {
    if (open && st[i]) cudaStreamSynchronize(st[i]);
    if (joined[i]) cudaEventDestroy(joined[i]);
    if (st[i]) cudaStreamDestroy(st[i]);
  }
  if (forked) cudaEventDestroy(forked);
}

void LpWork::init(int64_t n_vertices, int64_t n_labels, cudaStream_t s) {
  if (n_vertices <= n && n_labels <= nlabels) return;
  n = std::max(n, n_vertices);
  nlabels = std::max(nlabels, n_labels);
  size_t L = (size_t)std::max<int64_t>(nlabels, 1), N = (size_t)std::max<int64_t>(n, 1);
  in_w.alloc(L, s);
  ccnt.alloc(L, s);
  cfill.alloc(L, s);
  cbase.alloc(L, s);
  ctarget.alloc(L, s);
  cbig.alloc(L, s);
  mv_u.alloc(N, s);
  mv_t.alloc(N, s);
  mv_o.alloc(N, s);
  mv_g.alloc(N, s);
  mv_ok.alloc(N, s);
  cseg.alloc(N, s);
  cseg_u.alloc(N, s);
  cseg_g.alloc(N, s);
  counters.alloc(5, s);
  TP_CUDA(cudaMemsetAsync(in_w.get(), 0, L * 8, s));
  TP_CUDA(cudaMemsetAsync(ccnt.get(), 0, L * 4, s));
  TP_CUDA(cudaMemsetAsync(cfill.get(), 0, L * 4, s));
  TP_CUDA(cudaMemsetAsync(counters.get(), 0, 5 * 8, s));
}

// The approval of one sub-round: the same five kernels and counter reset on
// every sub-round of a level (only the data differs).
constexpr int kApproveKernels = 5;
// wake (nullable): the graph whose quiet vertices the moves wake, S its
// sub-rounds. Marks pay while a round moves few vertices: beyond an eighth
// of the vertices (a mesh vertex wakes 16, movers side by side the same ones)
// hardly any would last.
void launch_approval(const ApproveCtx &a, int64_t wn, int64_t *counters, cudaStream_t stream,
                     const tp_graph *wake = nullptr, LpWork *w = nullptr, int32_t S = 1) {
  const unsigned blocks = (unsigned)num_sms() * 4;
  const unsigned wide = grid_for(std::max<int64_t>(wn, 1), 256, (int64_t)num_sms() * 64);
  launch(k_approve_fit, wide, 256, 0, stream, a);
  launch(k_approve_alloc, (unsigned)num_sms(), 256, 0, stream, a);
  launch(k_approve_scatter, blocks, 256, 0, stream, a);
  launch(k_approve_contested, (unsigned)num_sms() * 2, kContestedThreads, 0, stream, a);
  launch(k_apply, wide, 256, 0, stream, a);
  if (wake) {
    const int64_t limit = wake->n / (8 * (int64_t)S);
    const unsigned wb = grid_for(std::max<int64_t>(limit, 1), 256);
    const uint8_t *tier = wake->tiers.tier.get();
    unsigned long long *cnt = (unsigned long long *)counters;
    if (wake->compressed)
      launch(k_wake<true>, wb, 256, 0, stream, view(wake), tier, cnt, a.mv_u, a.mv_ok, limit,
             w->quiet.get(), w->epoch.get());
    else
      launch(k_wake<false>, wb, 256, 0, stream, view(wake), tier, cnt, a.mv_u, a.mv_ok, limit,
             w->quiet.get(), w->epoch.get());
  }
  TP_LAUNCH_CHECK();
  TP_CUDA(cudaMemsetAsync(counters, 0, 5 * sizeof(int64_t), stream));
}

// Records the approval of a level's sub-rounds into a CUDA graph on a
// private stream, so each sub-round replays it with one launch. Returns null
// (callers then launch directly) if capturing is not possible.
struct ApprovalGraph {
  cudaStream_t cs = nullptr;
  cudaGraphExec_t exec = nullptr;
  ApprovalGraph(const ApproveCtx &a, int64_t wn, int64_t *counters, const tp_graph *wake,
                LpWork *w, int32_t S) {
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) {
      (void)cudaGetLastError();
      cs = nullptr;
      return;
    }
    if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      (void)cudaGetLastError();
      return;
    }
    capture_counting(true);
    bool ok = true;
    try {
      launch_approval(a, wn, counters, cs, wake, w, S);
    } catch (...) {
      ok = false;
    }
    capture_counting(false);
    cudaGraph_t graph = nullptr;
    if (cudaStreamEndCapture(cs, &graph) != cudaSuccess || !ok || !graph) {
      (void)cudaGetLastError();
      if (graph) cudaGraphDestroy(graph);
      return;
    }
    if (cudaGraphInstantiate(&exec, graph, 0) != cudaSuccess) {
      (void)cudaGetLastError();
      exec = nullptr;
    }
    cudaGraphDestroy(graph);
  }
  ~ApprovalGraph() {
    if (exec) cudaGraphExecDestroy(exec);
    if (cs) cudaStreamDestroy(cs);
  }
};

void lp_subround(tp_graph *g, const LpState &st, LpWork &w, uint64_t rk, int32_t S, int32_t s,
                 const tp_params &p, cudaStream_t stream, cudaGraphExec_t approval,
                 const uint64_t *rk_dev) {
  configure_kernels();
  RateCtx c{};
  c.label = st.label;
  c.lw = st.lw;
  c.cap = st.cap;
  c.nlabels = st.nlabels;
  c.seg = st.seg;
  c.k = st.k;
  c.kmax = st.kmax;
  c.rk = rk;
  c.rk_dev = rk_dev;
  c.S = S;
  c.s = s;
  c.mv_u = w.mv_u.get();
  c.mv_o = w.mv_o.get();
  c.mv_t = w.mv_t.get();
  c.mv_g = w.mv_g.get();
  c.in_w = w.in_w.get();
  c.counters = (unsigned long long *)w.counters.get();
  if (w.bucket_S == S) {
    if (w.quiet_on) c.quiet = w.quiet.get(), c.epoch = w.epoch.get();
    c.bucket = w.bucket.get();
    c.bucket_off = w.bucket_off.get();
    c.bucket_nb = w.bucket_nblocks;
    c.bucket_rec = g->compressed ? w.bucket_rec.get() : nullptr;
    c.sub_byte = w.bucket_sub.get();
    if (w.tb_valid) {
      c.tb_pos = w.tb_pos.get();
      c.tb_off = w.tb_off.get();
      for (int t = 0; t < LpWork::kTiers; ++t) c.tb_base[t] = w.tb_base[t];
      c.hc_pre = w.hc_pre.get();
      c.hs_pre = w.hs_pre.get();
      c.hc_item = w.hc_item.get();
      c.hs_item = w.hs_item.get();
    }
  }
  rate_tiers<M_LP>(g, c, p, stream, &w.streams);
  prof_begin(PF_APPROVE, stream);
  if (approval) {
    TP_CUDA(cudaGraphLaunch(approval, stream));
    count_launches(kApproveKernels + (w.quiet_on ? 1 : 0));
  } else {
    launch_approval(approve_ctx(g, st, w), w.n, w.counters.get(), stream, w.quiet_on ? g : nullptr, &w,
                    S);
  }
  prof_end(PF_APPROVE, stream, 0.0);
}

// Round key of round *r (then r advances): the first node of a replayed
// round graph.
__global__ void k_round_key(uint64_t seed, uint64_t tag, uint64_t a, uint64_t b0, int32_t *r,
                            uint64_t *rk) {
  *rk = round_key(seed, tag, a, b0 + (uint64_t)*r);
  *r += 1;
}

__global__ void k_set_i32(int32_t *p, int32_t v) { *p = v; }

// Small levels: a whole LP round (round key, bucketing, every sub-round's
// rating and approval) is recorded once as a CUDA graph on a private stream
// and replayed once per round on the caller's stream, the round key coming
// from device memory. Levels above this size launch directly (their kernels
// are long enough to hide launch costs, and their bucket scan would allocate
// inside the graph).
constexpr int64_t kRoundGraphMaxN = (int64_t)1 << 19;

bool lp_rounds_graph(tp_graph *g, const LpState &st, LpWork &w, uint64_t seed, uint64_t tag,
                     uint64_t a, uint64_t b0, int32_t rounds, int32_t S, const tp_params &p,
                     cudaStream_t stream) {
  configure_kernels();
  build_tiers(g, p, stream);  // synchronises; must not run while capturing
  ensure_hub_tables(g, stream);  // nor may the tables be allocated inside the capture
  const int64_t nblocks = (g->n + kBucketSpan - 1) / kBucketSpan;
  if (S > 32 || S * nblocks > 2048) return false;
  if (!w.bucket.get()) w.bucket.alloc(std::max<int64_t>(w.n, 1), stream);
  if (!w.bucket_sub.get()) w.bucket_sub.alloc(std::max<int64_t>(w.n, 1), stream);
  if ((int64_t)w.bucket_off.n < S * nblocks + 1) w.bucket_off.alloc(S * nblocks + 1, stream);
  if (g->compressed && !w.bucket_rec.get()) w.bucket_rec.alloc(std::max<int64_t>(w.n, 1), stream);
  Buf<int32_t> d_r(1, stream);
  Buf<uint64_t> d_rk(1, stream);
  TP_CUDA(cudaMemsetAsync(d_r.get(), 0, sizeof(int32_t), stream));
  cudaStream_t cs = nullptr;
  if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  struct StreamGuard {
    cudaStream_t s;
    ~StreamGuard() { cudaStreamDestroy(s); }
  } sg{cs};
  if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  capture_counting(true);
  bool ok = true;
  try {
    launch(k_round_key, 1u, 1u, 0, cs, seed, tag, a, b0, d_r.get(), d_rk.get());
    lp_bucket(g, w, 0, S, p, cs, d_rk.get(), false, &st.seg);
    for (int32_t s = 0; s < S; ++s) lp_subround(g, st, w, 0, S, s, p, cs, nullptr, d_rk.get());
    w.bucket_S = 0;
  } catch (...) {
    ok = false;
  }
  const uint64_t kernels = capture_counting(false);
  cudaGraph_t graph = nullptr;
  if (cudaStreamEndCapture(cs, &graph) != cudaSuccess || !ok || !graph) {
    (void)cudaGetLastError();
    if (graph) cudaGraphDestroy(graph);
    return false;
  }
  cudaGraphExec_t exec = nullptr;
  const bool inst = cudaGraphInstantiate(&exec, graph, 0) == cudaSuccess;
  cudaGraphDestroy(graph);
  if (!inst) {
    (void)cudaGetLastError();
    return false;
  }
  struct ExecGuard {
    cudaGraphExec_t e;
    ~ExecGuard() { cudaGraphExecDestroy(e); }
  } eg{exec};
  for (int32_t r = 0; r < rounds; ++r) {
    TP_CUDA(cudaGraphLaunch(exec, stream));
    count_launches(kernels);
  }
  return true;
}

void lp_rounds(tp_graph *g, const LpState &st, LpWork &w, uint64_t seed, uint64_t tag, uint64_t a,
               uint64_t b0, int32_t rounds, int32_t S, const tp_params &p, cudaStream_t stream) {
  if (rounds <= 0) return;
  if (p.use_graphs && g->n <= std::min<int64_t>(p.graph_n, kRoundGraphMaxN) && !prof_active() &&
      lp_rounds_small(g, st, w, seed, tag, a, b0, rounds, S, p, stream))
    return;
  if (p.use_graphs && g->n <= std::min<int64_t>(p.graph_n, kRoundGraphMaxN) && !prof_active() &&
      lp_rounds_graph(g, st, w, seed, tag, a, b0, rounds, S, p, stream))
    return;
  build_tiers(g, p, stream);
  const TierCache &T = g->tiers;
  // quiet vertices: one graph, most entries in the lane tier, and so few
  // sub-rounds that the epoch (one step each at most) fits its byte. In
  // clustering nearly every vertex moves in the first two rounds, which go
  // without (labels are vertices then: kmax is 0), and the rounds after them
  // cost more with the marks than they save in small levels and few rounds.
  // Meshes of degree 16, with marks against without, CSR / compressed: 6e5
  // vertices, 5 rounds 1.00 (none) / 1.11, 8 rounds 1.12 / 1.14; 2^21, 6 rounds
  // 0.99 / 0.99, 8 rounds 0.94 / 0.96; 2^23, 5 rounds 1.00 (none) / 0.95, 6
  // rounds 0.95 / 0.91, 12 rounds 0.74 / 0.75; 2^24 and CSR, 3 rounds 1.11, 5
  // rounds 1.01. In refinement the marks pay from two rounds on: 6e5 vertices
  // 0.94 / 0.96, five rounds 0.89 / 0.90; 2^23 0.73 / 0.75 and 0.53 / 0.56.
  const int32_t quiet_from = st.kmax ? 0 : 2;
  // A single round rates every vertex once, so marks are of no use in it.
  const int32_t quiet_least = st.kmax ? 2 : g->compressed && g->n >= ((int64_t)1 << 22) ? 5 : 6;
  const bool quiet_ok = !st.seg.gid && S <= 32 && (int64_t)rounds * S < 250 && rounds >= quiet_least &&
                        (st.kmax || g->n >= ((int64_t)1 << 21)) && !T.lane_long && !prof_active() &&
                        5 * T.edges[TIER_LANE] >= 4 * g->m2 && g->n <= kLaneKeyLabels &&
                        st.nlabels <= kLaneKeyLabels;
  std::unique_ptr<ApprovalGraph> ag;
  for (int32_t r = 0; r < rounds; ++r) {
    const bool quiet = quiet_ok && r >= quiet_from;
    if (quiet && !w.quiet_on) {
      if ((int64_t)w.quiet.n < g->n) w.quiet.alloc(g->n, stream);
      if (!w.epoch.get()) w.epoch.alloc(1, stream);
      TP_CUDA(cudaMemsetAsync(w.quiet.get(), 0, g->n, stream));
      launch(k_set_i32, 1, 1, 0, stream, w.epoch.get(), 1);
    }
    if (!ag || quiet != w.quiet_on) {
      w.quiet_on = quiet;
      ag.reset(new ApprovalGraph(approve_ctx(g, st, w), w.n, w.counters.get(), quiet ? g : nullptr, &w, S));
    }
    uint64_t rk = round_key(seed, tag, a, b0 + (uint64_t)r);
    lp_bucket(g, w, rk, S, p, stream, nullptr, true, &st.seg);
    for (int32_t s = 0; s < S; ++s) lp_subround(g, st, w, rk, S, s, p, stream, ag->exec);
    w.bucket_S = 0;
    w.tb_valid = false;
  }
  w.quiet_on = false;
}

// ---------------------------------------------------------------- two-hop packing
namespace {

__global__ void k_fav_init(int32_t *fav, int64_t n) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x)
    fav[u] = -2;
}

__global__ void k_th_flags(const int32_t *fav, int64_t n, int32_t *flag) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x)
    flag[u] = fav[u] >= 0;
}

__global__ void k_th_gather(const int32_t *fav, const int32_t *flag, const int64_t *pos, int64_t n,
                            uint64_t *keys, uint64_t *vals) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x)
    if (flag[u]) {
      keys[pos[u]] = (uint64_t)fav[u];
      vals[pos[u]] = (uint64_t)u;
    }
}

// weights in sorted order and run-start markers
__global__ void k_th_prep(const uint64_t *keys, const uint64_t *vals, const int64_t *vw, int64_t m,
                          int64_t *wt, int64_t *rs) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    wt[i] = vw ? vw[vals[i]] : 1;
    rs[i] = (i == 0 || keys[i] != keys[i - 1]) ? i : -1;
  }
}

// bins, straddlers and group heads (batched graphs: a group lies in one
// graph, whose U is gU[gid[vertex]])
__global__ void k_th_heads(const int64_t *excl, const int64_t *rs, const int64_t *wt, int64_t m,
                           int64_t U_one, const uint64_t *vals, const int32_t *gid,
                           const int64_t *gU, int64_t *head) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t U = gid ? gU[gid[vals[i]]] : U_one;
    int64_t P = excl[i] - excl[rs[i]];
    int64_t bin = P / U;
    bool str = P + wt[i] > (bin + 1) * U;
    bool h = false;
    if (!str) {
      if (i == rs[i]) h = true;
      else {
        int64_t Pp = excl[i - 1] - excl[rs[i - 1]];
        int64_t binp = Pp / U;
        bool strp = Pp + wt[i - 1] > (binp + 1) * U;
        h = strp || binp != bin;
      }
    }
    head[i] = str ? -2 : (h ? i : -1);
  }
}

__global__ void k_th_assign(const int64_t *head_raw, const int64_t *head_scan,
                            const uint64_t *vals, int64_t m, int32_t *C) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (head_raw[i] == -2) continue;  // straddler stays alone
    C[vals[i]] = (int32_t)vals[head_scan[i]];
  }
}

}  // namespace

void favourites(tp_graph *g, const int32_t *C, const int64_t *Wc, uint64_t rk, int32_t *fav,
                const tp_params &p, cudaStream_t s, const SegLp *seg) {
  configure_kernels();
  launch(k_fav_init, grid_for(g->n, 256), 256, 0, s, fav, g->n);
  TP_LAUNCH_CHECK();
  RateCtx c{};
  c.label = C;
  c.lw = Wc;
  c.rk = rk;
  c.fav = fav;
  if (seg) c.seg = *seg;
  rate_tiers<M_FAV>(g, c, p, s);
}

void two_hop(tp_graph *g, int32_t *C, const int64_t *Wc, int64_t U, uint64_t seed, int32_t level,
             const tp_params &p, cudaStream_t s, const SegLp *seg) {
  int64_t n = g->n;
  if (n == 0) return;
  const bool sg = seg && seg->gid;
  Buf<int32_t> fav(n, s), flag(n, s);
  favourites(g, C, Wc, round_key(seed, kTagTwoHop, (uint64_t)level, 0), fav.get(), p, s, seg);
  launch(k_th_flags, grid_for(n, 256), 256, 0, s, fav.get(), n, flag.get());
  TP_LAUNCH_CHECK();
  Buf<int64_t> pos(n + 1, s);
  exclusive_scan_i32_to_i64(flag.get(), pos.get(), n, s);
  int64_t m = read_scalar(pos.get() + n, s);
  if (m == 0) return;
  Buf<uint64_t> keys(m, s), vals(m, s);
  launch(k_th_gather, grid_for(n, 256), 256, 0, s, fav.get(), flag.get(), pos.get(), n, keys.get(),
                                                 vals.get());
  TP_LAUNCH_CHECK();
  // keys: favourites (vertex ids) and the no-favourite key n (per graph:
  // n + graph), so no group spans two graphs
  radix_sort_pairs(keys.get(), vals.get(), m,
                   bits_for((uint64_t)n + (sg ? (uint64_t)seg->ngraphs : 0)), s);
  Buf<int64_t> wt(m, s), rs(m, s), excl(m + 1, s), head(m, s), hs(m, s);
  launch(k_th_prep, grid_for(m, 256), 256, 0, s, keys.get(), vals.get(),
                                               g->unit_vw ? nullptr : g->vw.get(), m, wt.get(),
                                               rs.get());
  TP_LAUNCH_CHECK();
  inclusive_max_scan_i64(rs.get(), rs.get(), m, s);
  exclusive_scan_i64(wt.get(), excl.get(), m, s);
  launch(k_th_heads, grid_for(m, 256), 256, 0, s, excl.get(), rs.get(), wt.get(), m, U, vals.get(),
         sg ? seg->gid : nullptr, sg ? seg->cap : nullptr, head.get());
  TP_LAUNCH_CHECK();
  inclusive_max_scan_i64(head.get(), hs.get(), m, s);
  launch(k_th_assign, grid_for(m, 256), 256, 0, s, head.get(), hs.get(), vals.get(), m, C);
  TP_LAUNCH_CHECK();
}

void lp_cluster(tp_graph *g, int64_t U, const tp_params &p, int32_t level, int32_t *d_cluster,
                cudaStream_t s, cudaEvent_t ev_begin, cudaEvent_t ev_end, const SegLp *seg) {
  int64_t n = g->n;
  if (n == 0) return;
  Buf<int64_t> Wc(n, s);
  launch(k_init_singletons, grid_for(n, 256), 256, 0, s, g->unit_vw ? nullptr : g->vw.get(), n,
                                                       d_cluster, Wc.get());
  TP_LAUNCH_CHECK();
  LpState st{d_cluster, Wc.get(), n, U};
  if (seg) {  // labels are vertices: a label's graph and base are its vertex's
    st.seg = *seg;
    st.seg.lgid = seg->gid;
    st.seg.lb = seg->vb;
  }
  {
    LpWork w;  // gone before the packing's buffers are made
    w.init(n, n, s);
    prof_scope(level == 0 && !seg);
    if (ev_begin) TP_CUDA(cudaEventRecord(ev_begin, s));
    lp_rounds(g, st, w, p.seed, kTagCluster, (uint64_t)level, 0, p.cluster_rounds, p.sub_rounds, p, s);
    if (ev_end) TP_CUDA(cudaEventRecord(ev_end, s));
    prof_scope(false);
  }
  if (p.two_hop) two_hop(g, d_cluster, Wc.get(), U, p.seed, level, p, s, seg ? &st.seg : nullptr);
  release_hub_tables(g, s);
}

void lp_refine(tp_graph *g, int32_t k, int64_t l_max, const tp_params &p, int32_t level,
               int32_t *d_part, int64_t *d_B, cudaStream_t s, const SegLp *seg) {
  if (g->n == 0) return;
  LpWork w;
  w.init(g->n, k, s);
  LpState st{d_part, d_B, k, l_max};
  st.k = k;
  st.kmax = seg ? seg->kmax : k;
  if (seg) st.seg = *seg;
  lp_rounds(g, st, w, p.seed, kTagRefine, (uint64_t)level, 0, p.refine_rounds, p.sub_rounds, p, s);
  release_hub_tables(g, s);
}

// ---------------------------------------------------------------- rebalancing
namespace {

__global__ void k_find_over(const int64_t *B, int32_t k, int64_t l_max, int32_t *out) {
  __shared__ int32_t best;
  if (threadIdx.x == 0) best = INT32_MAX;
  __syncthreads();
  for (int32_t b = threadIdx.x; b < k; b += blockDim.x)
    if (B[b] > l_max) atomicMin(&best, b);
  __syncthreads();
  if (threadIdx.x == 0) out[0] = best == INT32_MAX ? -1 : best;
}

__global__ void k_rb_pick(const int32_t *part, int32_t blk, const int32_t *rb_t,
                          const int64_t *rb_loss, const long long *best, int64_t n, int32_t *best_u) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x)
    if (part[u] == blk && rb_t[u] >= 0 && rb_loss[u] == *best) atomicMin(best_u, (int32_t)u);
}

__global__ void k_rb_apply(int32_t *part, int64_t *B, const int64_t *vw, const int32_t *rb_t,
                           const int32_t *best_u) {
  int32_t u = *best_u;
  if (u == INT32_MAX) return;
  int32_t t = rb_t[u], b = part[u];
  int64_t w = vw ? vw[u] : 1;
  B[b] -= w;
  B[t] += w;
  part[u] = t;
}

}  // namespace

void rebalance_moves(tp_graph *g, int32_t k, int64_t l_max, int32_t *d_part, int64_t *d_B,
                     int *balanced, const tp_params &p, cudaStream_t s) {
  configure_kernels();
  int64_t n = g->n;
  Buf<int32_t> small(4, s);  // [0] overloaded block [1] best vertex
  Buf<long long> best(1, s);
  Buf<int32_t> rb_t(std::max<int64_t>(n, 1), s);
  Buf<int64_t> rb_loss(std::max<int64_t>(n, 1), s);
  *balanced = 1;
  for (;;) {
    launch(k_find_over, 1, 256, 0, s, d_B, k, l_max, small.get());
    TP_LAUNCH_CHECK();
    int32_t blk = read_scalar(small.get(), s);
    if (blk < 0) return;
    long long init_best = INT64_MAX;
    int32_t init_u = INT32_MAX;
    TP_CUDA(cudaMemcpyAsync(best.get(), &init_best, sizeof(init_best), cudaMemcpyHostToDevice, s));
    TP_CUDA(cudaMemcpyAsync(small.get() + 1, &init_u, sizeof(init_u), cudaMemcpyHostToDevice, s));
    RateCtx c{};
    c.label = d_part;
    c.lw = d_B;
    c.cap = l_max;
    c.blk = blk;
    c.k = c.kmax = k;
    c.rb_loss = rb_loss.get();
    c.rb_t = rb_t.get();
    c.rb_best = best.get();
    rate_tiers<M_REBAL>(g, c, p, s);
    launch(k_rb_pick, grid_for(n, 256), 256, 0, s, d_part, blk, rb_t.get(), rb_loss.get(), best.get(),
                                                 n, small.get() + 1);
    launch(k_rb_apply, 1, 1, 0, s, d_part, d_B, g->unit_vw ? nullptr : g->vw.get(), rb_t.get(),
                               small.get() + 1);
    TP_LAUNCH_CHECK();
    int32_t bu = read_scalar(small.get() + 1, s);
    if (bu == INT32_MAX) {
      *balanced = 0;
      return;
    }
  }
}

namespace {

// Batched rebalancing, step 1 (one block per graph of the union): the
// smallest overloaded block of every graph still rebalancing, or -1; resets
// the graph's best loss and vertex and counts the graphs with one.
__global__ void k_find_over_seg(const int64_t *B, SegLp seg, const int32_t *graphs, int64_t ng,
                                const int32_t *stuck, int32_t *blk_of, long long *best,
                                int32_t *best_u, int32_t *n_over) {
  __shared__ int32_t bmin;
  for (int64_t j = blockIdx.x; j < ng; j += gridDim.x) {
    const int32_t i = graphs[j];
    if (threadIdx.x == 0) bmin = INT32_MAX;
    __syncthreads();
    const int64_t lb = seg.lb[i], cap = seg.cap[i];
    if (!stuck[i])
      for (int32_t b = threadIdx.x; b < seg.k[i]; b += blockDim.x)
        if (B[lb + b] > cap) atomicMin(&bmin, b);
    __syncthreads();
    if (threadIdx.x == 0) {
      const bool over = bmin != INT32_MAX;
      blk_of[i] = over ? (int32_t)(lb + bmin) : -1;
      best[i] = INT64_MAX;
      best_u[i] = INT32_MAX;
      if (over) atomicAdd(n_over, 1);
    }
    __syncthreads();
  }
}

// Step 2: per graph, the smallest vertex among those of least loss.
__global__ void k_rb_pick_seg(const int32_t *part, const int32_t *gid, const int32_t *blk_of,
                              const int32_t *rb_t, const int64_t *rb_loss, const long long *best,
                              int64_t n, int32_t *best_u) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    const int32_t g = gid[u], blk = blk_of[g];
    if (blk >= 0 && part[u] == blk && rb_t[u] >= 0 && rb_loss[u] == best[g])
      atomicMin(&best_u[g], (int32_t)u);
  }
}

// Step 3 (one thread per graph): make the move, or retire a graph without one.
__global__ void k_rb_apply_seg(const int32_t *graphs, int64_t ng, const int32_t *blk_of,
                               const int32_t *best_u, const int32_t *rb_t, const int64_t *vw,
                               int32_t *part, int64_t *B, int32_t *stuck) {
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < ng;
       j += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = graphs[j];
    if (blk_of[i] < 0) continue;
    const int32_t u = best_u[i];
    if (u == INT32_MAX) {
      stuck[i] = 1;
      continue;
    }
    const int32_t t = rb_t[u], b = part[u];
    const int64_t w = vw ? vw[u] : 1;
    B[b] -= w;
    B[t] += w;
    part[u] = t;
  }
}

}  // namespace

void rebalance_moves_seg(tp_graph *g, const SegLp &seg, const int32_t *d_graphs, int64_t ng,
                         int32_t *d_part, int64_t *d_B, const tp_params &p, cudaStream_t s) {
  configure_kernels();
  const int64_t n = g->n, G = seg.ngraphs;
  if (n == 0 || ng == 0) return;
  Buf<int32_t> blk_of(G, s), best_u(G, s), stuck(G, s), n_over(1, s);
  Buf<long long> best(G, s);
  Buf<int32_t> rb_t(n, s);
  Buf<int64_t> rb_loss(n, s);
  TP_CUDA(cudaMemsetAsync(stuck.get(), 0, G * sizeof(int32_t), s));
  const unsigned gb = (unsigned)std::min<int64_t>(ng, (int64_t)num_sms() * 8);
  for (;;) {
    TP_CUDA(cudaMemsetAsync(n_over.get(), 0, sizeof(int32_t), s));
    launch(k_find_over_seg, gb, 128, 0, s, d_B, seg, d_graphs, ng, stuck.get(), blk_of.get(),
           best.get(), best_u.get(), n_over.get());
    TP_LAUNCH_CHECK();
    if (read_scalar(n_over.get(), s) == 0) return;
    RateCtx c{};
    c.label = d_part;
    c.lw = d_B;
    c.seg = seg;
    c.kmax = seg.kmax;
    c.blk_of = blk_of.get();
    c.rb_loss = rb_loss.get();
    c.rb_t = rb_t.get();
    c.rb_best = best.get();
    rate_tiers<M_REBAL>(g, c, p, s);
    launch(k_rb_pick_seg, grid_for(n, 256), 256, 0, s, d_part, seg.gid, blk_of.get(), rb_t.get(),
           rb_loss.get(), best.get(), n, best_u.get());
    launch(k_rb_apply_seg, grid_for(ng, 256), 256, 0, s, d_graphs, ng, blk_of.get(), best_u.get(),
           rb_t.get(), g->unit_vw ? nullptr : g->vw.get(), d_part, d_B, stuck.get());
    TP_LAUNCH_CHECK();
  }
}

}  // namespace tp
