// Cluster contraction (Section "Contraction" of the paper): every cluster
// becomes a coarse vertex, w'(a,b) sums the weights of the fine edges between
// clusters a and b, intra-cluster edges vanish.
//
// GPU form: coarse ids are ranks of the non-empty labels (mark + exclusive
// scan, so ids are deterministic where the paper's atomic counters are not).
// The fine vertices are listed by coarse vertex, and a warp (or a block) per
// coarse vertex walks its members' rows once and sums the weights per
// neighbouring cluster in a shared-memory hash table; the distinct neighbours
// are sorted there and written out. Tables come in four sizes (256 and 1024
// slots a warp, 4096 and 16384 a block): a coarse vertex starts with the size
// that its members' entries suggest and moves to the next if its distinct
// neighbours overflow it, so nothing depends on the guess. The few beyond the
// largest table (coarse vertices of hubs) emit every inter-cluster entry as
// the key a*n' + b, which the library's LSD radix sort and a run-length
// reduction turn into their rows. (Sorting all entries took five passes over
// them; a mesh merges about 17 entries into one.) Weights are summed in 32
// bits where all edge weights together fit or every edge weighs one (a table's
// coarse vertex has no more than 40 960 entries).
#include <algorithm>
#include <memory>

#include "decode.cuh"

namespace tp {

namespace {

__global__ void k_mark(const int32_t *C, int64_t n, int32_t *flag) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x)
    flag[C[u]] = 1;
}

// Coarse id of every vertex, its place among the cluster's members, the
// cluster's weight, members and entries (compressed graphs: bytes of the
// records, no fewer than entries; it only picks the first table size). A warp
// whose 32 vertices share a cluster adds once (2^26 vertices in one cluster: 46
// ms of the 48.6 that the contraction took went into the queue on one word).
__global__ void k_map(GView g, const int32_t *C, const int64_t *rank, int32_t *map, int64_t *cvw,
                      int32_t *place, int32_t *mcnt, unsigned long long *ent) {
  for (int64_t u0 = (int64_t)blockIdx.x * blockDim.x; u0 < g.n;
       u0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = u0 + threadIdx.x;
    const bool in = u < g.n;
    const int32_t a = in ? (int32_t)rank[C[u]] : -1;
    const int64_t w = in && g.vw ? g.vw[u] : 0;
    const int64_t e = !in ? 0
                      : g.compressed ? (int64_t)(off_at(g, u + 1) - off_at(g, u))
                                     : g.xadj[u + 1] - g.xadj[u];
    if (in) map[u] = a;
    const int32_t a0 = __shfl_sync(kFull, a, 0);
    if (__all_sync(kFull, a == a0)) {
      const int64_t ws = g.vw ? warp_sum(w) : 0, es = warp_sum(e);
      int32_t at = 0;
      if (lane_id() == 0 && a0 >= 0) {
        at = atomicAdd(&mcnt[a0], 32);
        if (g.vw) atomicAdd((unsigned long long *)&cvw[a0], (unsigned long long)ws);
        if (es) atomicAdd(&ent[a0], (unsigned long long)es);
      }
      at = __shfl_sync(kFull, at, 0);
      if (in) place[u] = at + lane_id();
    } else if (in) {
      place[u] = atomicAdd(&mcnt[a], 1);
      if (g.vw) atomicAdd((unsigned long long *)&cvw[a], (unsigned long long)w);
      atomicAdd(&ent[a], (unsigned long long)e);
    }
  }
}

// Batched graphs: coarse offset of every graph (the rank of its first vertex).
__global__ void k_seg_rank(const int64_t *rank, const int64_t *voff, int64_t nseg, int64_t *coff) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= nseg;
       i += (int64_t)gridDim.x * blockDim.x)
    coff[i] = rank[voff[i]];
}

__global__ void k_members(const int32_t *map, const int32_t *place, const int64_t *mstart,
                          int64_t n, int32_t *members) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x)
    members[mstart[map[u]] + place[u]] = (int32_t)u;
}

// ---------------------------------------------------------------- table sizes
// Size 0 and 1: a warp's table of 256 / 1024 slots; 2 and 3: a block's of 4096
// / 16384; 4: keys and the radix sort. A table takes up to agg_fill distinct
// neighbours; a coarse vertex starts with a size whose fill is no less than a
// fifth of its entries (meshes merge far more than that into one, skewed
// graphs less and move up).
constexpr int kAggSizes = 4;
__host__ __device__ constexpr int agg_log(int size) { return size == 0 ? 8 : size == 1 ? 10 : size == 2 ? 12 : 14; }
__host__ __device__ constexpr int agg_fill(int size) { return size == 0 ? 192 : size == 1 ? 768 : size == 2 ? 2816 : 10240; }
__host__ __device__ constexpr int64_t agg_start(int size) {
  return size == 0 ? 1024 : size == 1 ? 4096 : size == 2 ? 14336 : 40960;
}

// Lists every coarse vertex under its first size, its weight where members
// weigh one each, and adds up the entries of those that start in a table (rows:
// no fewer than the tables write). A member counts for an entry at least: a
// table's warp or block walks the members, and one cluster of 2^26 vertices
// without edges was a warp's walk of 2.0 s (now 4.5 ms). lists: kAggSizes + 1
// lists of nc entries, cnt: their lengths.
__global__ void __launch_bounds__(256)
    k_agg_classes(const unsigned long long *ent, const int32_t *mcnt, int64_t nc, int64_t *cvw,
                  int32_t *lists, int32_t *cnt, unsigned long long *rows) {
  __shared__ int64_t part[8], part0[8];
  int64_t mine = 0, low = 0;
  for (int64_t a0 = (int64_t)blockIdx.x * blockDim.x; a0 < nc;
       a0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = a0 + threadIdx.x;
    int cl = -1;
    if (a < nc) {
      const int64_t e = max((int64_t)ent[a], (int64_t)mcnt[a]);
      cl = 0;
      while (cl < kAggSizes && e > agg_start(cl)) ++cl;
      if (cl < kAggSizes) mine += (int64_t)ent[a];
      if (cl == 0) low += (int64_t)ent[a];
      if (cvw) cvw[a] = mcnt[a];
    }
    const unsigned peers = __match_any_sync(kFull, cl);
    if (cl >= 0) {
      const int leader = __ffs(peers) - 1;
      int32_t base = 0;
      if (lane_id() == leader) base = atomicAdd(&cnt[cl], __popc(peers));
      base = __shfl_sync(peers, base, leader);
      lists[(int64_t)cl * nc + base + __popc(peers & lanemask_lt())] = (int32_t)a;
    }
  }
  mine = warp_sum(mine);
  low = warp_sum(low);
  if (lane_id() == 0) part[threadIdx.x >> 5] = mine, part0[threadIdx.x >> 5] = low;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) mine += part[w], low += part0[w];
    if (mine) atomicAdd(&rows[0], (unsigned long long)mine);
    if (low) atomicAdd(&rows[1], (unsigned long long)low);
  }
}

// Inter-cluster entries among those of every (n / kRowSamples)-th vertex's row
// (its first chunk), a warp each: out[0] of out[1].
constexpr int64_t kRowSamples = 1024;
template <bool COMP>
__global__ void k_row_sample(GView g, const int32_t *map, unsigned long long *out) {
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (i >= kRowSamples) return;
  const int64_t u = g.n / kRowSamples * i;
  const int32_t a = map[u];
  int64_t cut = 0, all = 0;
  warp_neighbours<COMP>(g, u, 0, [&](bool has, int32_t v, int64_t, int64_t) {
    all += has;
    cut += has && map[v] != a;
  });
  cut = warp_sum(cut);
  all = warp_sum(all);
  if (lane_id() == 0 && all) {
    atomicAdd(&out[1], (unsigned long long)all);
    if (cut) atomicAdd(&out[0], (unsigned long long)cut);
  }
}

struct AggCtx {
  GView g;
  const int32_t *map, *members;
  const int64_t *mstart;
  int64_t nc;
  int32_t *lists, *cnt;        // per size: coarse vertices still to do, how many
  unsigned long long *cursor;  // entries written so far
  int64_t room;                // entries that fit; the cursor counts on beyond them
  int32_t *out_key;            // neighbours of every coarse vertex, sorted, at toff
  void *out_val;
  int64_t *toff, *deg;
  unsigned long long *max_w;
};

// Adds w to label x's slot. Returns 0: added, 1: added in a slot it claimed,
// 2: no slot left.
template <class V>
__device__ __forceinline__ int agg_add(int32_t *keys, V *vals, int logc, int32_t x, V w) {
  const uint32_t mask = (1u << logc) - 1u;
  uint32_t h = ((uint32_t)x * 0x9E3779B1u) >> (32 - logc);
  for (uint32_t probe = 0; probe <= mask; ++probe, h = (h + 1) & mask) {
    int32_t k = *(volatile int32_t *)&keys[h];
    int claimed = 0;
    if (k == -1) {
      const int32_t prev = atomicCAS(&keys[h], -1, x);
      claimed = prev == -1;
      k = claimed ? x : prev;
    }
    if (k == x) {
      atomicAdd(&vals[h], w);
      return claimed;
    }
  }
  return 2;
}

// A compressed record of more bytes than this has more than kLaneMaxDeg
// neighbours (header and VarInts of at most ten and five bytes).
constexpr uint64_t kLaneRecordMost = 10 + 5 * kLaneMaxDeg;
constexpr uint64_t kLaneRecordShort = 65;  // fits lane_decode's first window

// This lane's member of those from m on, and where its row lies (entries, or
// bytes of the record).
struct AggMember {
  int32_t u;
  uint64_t b, e;
};
template <bool COMP>
__device__ __forceinline__ AggMember agg_member(const AggCtx &c, int64_t m, int64_t mend) {
  AggMember r{0, 0, 0};
  if (m + lane_id() < mend) {
    r.u = c.members[m + lane_id()];
    r.b = COMP ? off_at(c.g, r.u) : (uint64_t)c.g.xadj[r.u];
    r.e = COMP ? off_at(c.g, r.u + 1) : (uint64_t)c.g.xadj[r.u + 1];
  }
  return r;
}

// A warp's inter-cluster entries on their way to the table (compressed graphs,
// which are meshes here: skewed ones are decoded first). Most entries of a mesh
// lie inside the cluster (about two in three), so those that do not are queued
// and added 32 at a time with every lane busy: adding them where they were
// found ran the probing code for a third of the lanes, 16 times a row batch,
// unrolled beyond the instruction cache (mesh of 4.2 M vertices: 0.70 -> 0.60
// ms). CSR levels, with more entries between clusters, fewer instructions per
// entry and more warps, are faster adding directly (R-MAT 2^22: 1.7 against 2.0 ms).
constexpr int kAggStep = 4;  // entries a lane has in flight
template <class V>
struct AggQueue {
  int32_t x[32 + 32 * kAggStep];
  V w[32 + 32 * kAggStep];
};

// One warp sums the rows of members m, m + step, ... (32 at a time) of coarse
// vertex a into the table; fill() tells the distinct neighbours so far (of the
// warp or the block), add_fill(k) counts k more. Rows of up to 32 entries are
// walked a lane each (compressed: decoded into the lane's column), several
// entries in flight; row(u, entries) takes the longer ones and says whether
// the table held. Returns whether it held throughout.
template <bool COMP, class V, class Fill, class AddFill, class Row>
__device__ __forceinline__ bool agg_rows(const AggCtx &c, int32_t a, int64_t m, int64_t mend,
                                         int64_t step, int32_t *keys, V *vals, int logc,
                                         uint32_t *col, AggQueue<V> *qu, int limit,
                                         AggMember first, Fill fill, AddFill add_fill, Row row) {
  constexpr int U = kAggStep;
  const int lane = lane_id();
  int nq = 0;  // queued entries
  // adds queued entries 32 at a time, down to fewer than `keep`; whether the table holds
  auto drain = [&](int keep) -> bool {
    __syncwarp();
    int at = 0;
    for (; nq - at >= keep; at += 32) {
      const int i = at + lane;
      const int res = i < nq ? agg_add<V>(keys, vals, logc, qu->x[i], qu->w[i]) : 0;
      const unsigned claimed = __ballot_sync(kFull, res == 1);
      if (claimed) add_fill(__popc(claimed));
      if (__any_sync(kFull, res == 2) || fill() > limit) return false;
    }
    if (at) {  // the rest to the front
      const bool mine = at + lane < nq;
      const int32_t mx = mine ? qu->x[at + lane] : 0;
      const V mw = mine ? qu->w[at + lane] : V(0);
      __syncwarp();
      if (mine) qu->x[lane] = mx, qu->w[lane] = mw;
      nq = max(nq - at, 0);
    }
    return true;
  };
  for (AggMember mem = first; m < mend; m += step, mem = agg_member<COMP>(c, m, mend)) {
    const bool in = m + lane < mend;
    const int32_t u = mem.u;
    int deg = 0;
    int64_t b = 0;
    bool wide = false;
    if (in) {
      if (COMP) {
        const uint64_t rb = mem.b, re = mem.e;
        if (re - rb <= kLaneRecordShort) deg = lane_decode<false, true>(c.g, rb, re, col);
        else if (re - rb <= kLaneRecordMost) deg = lane_decode<true, true>(c.g, rb, re, col);
        else deg = kLaneMaxDeg + 1;
      } else {
        b = (int64_t)mem.b;
        deg = (int)min((int64_t)(mem.e - mem.b), (int64_t)kLaneMaxDeg + 1);
      }
      wide = deg > kLaneMaxDeg;
      if (wide) deg = 0;
    }
    const unsigned wides = __ballot_sync(kFull, wide);
    const int most = (int)__reduce_max_sync(kFull, (unsigned)deg);
    int32_t prev = u;
    for (int i0 = 0; i0 < most; i0 += U) {
      int32_t x[U];
      V w[U];
#pragma unroll
      for (int r = 0; r < U; ++r) {
        const int i = i0 + r;
        x[r] = -1;
        w[r] = 1;
        if (i < deg) {
          if (COMP) {
            const uint32_t v = col[i * 32];
            prev = i == 0 ? ((v & 1u) ? u - (int32_t)(v >> 1) : u + (int32_t)(v >> 1))
                          : prev + (int32_t)v;
            prev = (int32_t)min((uint32_t)prev, (uint32_t)(c.g.n - 1));
            x[r] = prev;
          } else {
            x[r] = c.g.adj[b + i];
            if (c.g.ew) w[r] = (V)c.g.ew[b + i];
          }
        }
      }
#pragma unroll
      for (int r = 0; r < U; ++r) x[r] = x[r] >= 0 ? c.map[x[r]] : a;
      if constexpr (COMP) {
#pragma unroll
        for (int r = 0; r < U; ++r) {
          const unsigned m = __ballot_sync(kFull, x[r] != a);
          if (m == 0) continue;
          if (x[r] != a) {
            const int at = nq + __popc(m & lanemask_lt());
            qu->x[at] = x[r];
            qu->w[at] = w[r];
          }
          nq += __popc(m);
        }
        if (nq >= 32 && !drain(32)) return false;
      } else {
        unsigned claimed = 0;
        bool full = false;
#pragma unroll
        for (int r = 0; r < U; ++r)
          if (x[r] != a) {
            const int res = agg_add<V>(keys, vals, logc, x[r], w[r]);
            claimed += res == 1;
            full |= res == 2;
          }
        claimed = __reduce_add_sync(kFull, claimed);
        if (claimed) add_fill((int)claimed);
        if (__any_sync(kFull, full) || fill() > limit) return false;
      }
    }
    for (unsigned q = wides; q; q &= q - 1)
      if (!row(__shfl_sync(kFull, u, __ffs(q) - 1))) return false;
  }
  return !COMP || nq == 0 || drain(1);
}

// A long row, or of a CSR row the pieces of 128 entries number first, first +
// step, ..., by a warp, 128 entries in flight (compressed: a decoder's step).
template <bool COMP, class V, class Fill, class AddFill>
__device__ __forceinline__ bool agg_long_row(const AggCtx &c, int32_t a, int32_t u, int first,
                                             int step, int32_t *keys, V *vals, int logc, int limit,
                                             Fill fill, AddFill add_fill) {
  const int lane = lane_id();
  bool bad = false;
  auto settle = [&](unsigned claimed, bool full) {
    claimed = __reduce_add_sync(kFull, claimed);
    if (claimed) add_fill((int)claimed);
    bad = __any_sync(kFull, full) || fill() > limit;
  };
  if constexpr (COMP) {
    warp_neighbours<true>(c.g, u, -1, [&](bool has, int32_t v, int64_t, int64_t) {
      if (bad) return;
      const int32_t x = has ? c.map[v] : a;
      const int res = x != a ? agg_add<V>(keys, vals, logc, x, (V)1) : 0;
      settle(res == 1, res == 2);
    });
  } else {
    const int64_t e = c.g.xadj[u + 1];
    for (int64_t i0 = c.g.xadj[u] + 128 * first; i0 < e && !bad; i0 += 128 * (int64_t)step) {
      int32_t x[4];
      V w[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int64_t i = i0 + 32 * r + lane;
        x[r] = i < e ? c.g.adj[i] : -1;
        w[r] = i < e && c.g.ew ? (V)c.g.ew[i] : (V)1;
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) x[r] = x[r] >= 0 ? c.map[x[r]] : a;
      unsigned claimed = 0;
      bool full = false;
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (x[r] != a) {
          const int res = agg_add<V>(keys, vals, logc, x[r], w[r]);
          claimed += res == 1;
          full |= res == 2;
        }
      settle(claimed, full);
    }
  }
  return !bad;
}

// Ascending bitonic sort of a[0 .. n2) (a power of two) by nt threads, t this
// one's number; sync separates the steps.
template <class Sync>
__device__ __forceinline__ void bitonic(uint64_t *a, int n2, int t, int nt, Sync sync) {
  for (int k = 2; k <= n2; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = t; i < n2 / 2; i += nt) {
        const int lo = 2 * i - (i & (j - 1)), hi = lo + j;
        const uint64_t x = a[lo], y = a[hi];
        if ((x > y) == ((lo & k) == 0)) a[lo] = y, a[hi] = x;
      }
      sync();
    }
}

// Sizes 0 and 1: a warp per coarse vertex.
template <bool COMP, int SIZE, class V>
struct AggWarp {
  union {
    uint64_t items[SIZE == 0 ? 256 : 1024];        // neighbour << 32 | slot, once the rows are done
    uint32_t col[COMP ? kLaneMaxDeg * 32 : 1];     // decoded records
  };
  int32_t keys[1 << agg_log(SIZE)];
  V vals[1 << agg_log(SIZE)];
  AggQueue<V> queue[COMP ? 1 : 0];
};
__host__ __device__ constexpr int agg_warps(int size) { return size == 0 ? 8 : 4; }

template <bool COMP, int SIZE, class V>
__global__ void __launch_bounds__(32 * agg_warps(SIZE), SIZE == 0 && !COMP ? 6 : 3)
    k_agg_warp(AggCtx c) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int L = agg_log(SIZE), SLOTS = 1 << L;
  using Warp = AggWarp<COMP, SIZE, V>;
  Warp &s = reinterpret_cast<Warp *>(smem)[threadIdx.x >> 5];
  const int lane = lane_id();
  V *out_val = static_cast<V *>(c.out_val);
  for (int i = lane; i < SLOTS; i += 32) s.keys[i] = -1, s.vals[i] = 0;
  __syncwarp();
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t cnt = c.cnt[SIZE];
  unsigned long long most = 0;
  // the next coarse vertex's list entry, members and their rows are loaded
  // while this one is summed, sorted and written: its own chain of dependent
  // loads (entry, range, member, offset, record) would leave the warp waiting
  const int32_t *list = c.lists + (int64_t)SIZE * c.nc;
  int32_t a_next = gw < cnt ? list[gw] : 0;
  int64_t m0_next = 0, m1_next = 0;
  if (gw < cnt) m0_next = c.mstart[a_next], m1_next = c.mstart[a_next + 1];
  AggMember mem_next = agg_member<COMP>(c, m0_next, m1_next);
  for (int64_t q = gw; q < cnt; q += nw) {
    const int32_t a = a_next;
    const int64_t m0 = m0_next, m1 = m1_next;
    const AggMember mem = mem_next;
    const bool more = q + nw < cnt;
    if (more) a_next = list[q + nw];
    int n_fill = 0;
    auto fill = [&] { return n_fill; };
    auto add_fill = [&](int k) { n_fill += k; };
    const bool ok = agg_rows<COMP, V>(
        c, a, m0, m1, 32, s.keys, s.vals, L, s.col + lane, s.queue, agg_fill(SIZE), mem, fill, add_fill,
        [&](int32_t u) {
          return agg_long_row<COMP, V>(c, a, u, 0, 1, s.keys, s.vals, L, agg_fill(SIZE), fill, add_fill);
        });
    __syncwarp();
    m0_next = more ? c.mstart[a_next] : 0;
    m1_next = more ? c.mstart[a_next + 1] : 0;
    if (!ok) {  // to the next size
      mem_next = agg_member<COMP>(c, m0_next, m1_next);
      if (lane == 0)
        c.lists[(int64_t)(SIZE + 1) * c.nc + atomicAdd(&c.cnt[SIZE + 1], 1)] = a;
      for (int i = lane; i < SLOTS; i += 32) s.keys[i] = -1, s.vals[i] = 0;
      __syncwarp();
      continue;
    }
    // the occupied slots, sorted by neighbour
    int d = 0;
    for (int i = lane; i < SLOTS; i += 32) {
      const int32_t k = s.keys[i];
      const unsigned m = __ballot_sync(kFull, k >= 0);
      if (k >= 0) s.items[d + __popc(m & lanemask_lt())] = (uint64_t)(uint32_t)k << 32 | (uint32_t)i;
      d += __popc(m);
    }
    __syncwarp();
    unsigned long long base = 0;
    if (lane == 0) {
      base = d ? atomicAdd(c.cursor, (unsigned long long)d) : 0ull;  // (used after the sort)
      c.deg[a] = d;
    }
    mem_next = agg_member<COMP>(c, m0_next, m1_next);
    if (d <= 32) {  // in registers
      uint64_t x = lane < d ? s.items[lane] : ~0ull;
#pragma unroll
      for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
          const uint64_t y = __shfl_xor_sync(kFull, x, j);
          const bool up = ((lane & k) == 0) == ((lane & j) == 0);
          x = up ? (x < y ? x : y) : (x < y ? y : x);
        }
      base = __shfl_sync(kFull, base, 0);
      if (lane < d && (int64_t)base + d <= c.room) {
        const V w = s.vals[(uint32_t)x];
        c.out_key[base + lane] = (int32_t)(x >> 32);
        out_val[base + lane] = w;
        most = w > most ? w : most;
      }
    } else {
      int n2 = 64;
      while (n2 < d) n2 <<= 1;
      for (int i = d + lane; i < n2; i += 32) s.items[i] = ~0ull;
      __syncwarp();
      bitonic(s.items, n2, lane, 32, [] { __syncwarp(); });
      base = __shfl_sync(kFull, base, 0);
      const int fit = (int64_t)base + d <= c.room ? d : 0;
      for (int i = lane; i < fit; i += 32) {
        const uint64_t x = s.items[i];
        const V w = s.vals[(uint32_t)x];
        c.out_key[base + i] = (int32_t)(x >> 32);
        out_val[base + i] = w;
        most = w > most ? w : most;
      }
    }
    if (lane == 0) c.toff[a] = (int64_t)base;
    if (COMP && mem_next.e > mem_next.b) prefetch_l2(c.g.bytes + mem_next.b);
    __syncwarp();
    for (int i = lane; i < SLOTS; i += 32) s.keys[i] = -1, s.vals[i] = 0;
    __syncwarp();
  }
  most = warp_max(most);
  if (lane == 0 && most) atomicMax(c.max_w, most);
}

// Sizes 2 and 3: a block per coarse vertex, its warps taking 32 members each
// in turn.
constexpr int64_t kAggDecodeDeg = 1024;  // compressed graphs beyond this degree are decoded first
constexpr int64_t kSortZip = (int64_t)1 << 23;  // (from this many entries on)
constexpr int kAggThreads = 256;
constexpr int kAggWide = 256;
// The largest table with 64-bit sums has half the slots.
template <class V>
__host__ __device__ constexpr int agg_block_log(int size) {
  return size == 3 && sizeof(V) == 8 ? 13 : agg_log(size);
}
template <class V>
__host__ __device__ constexpr int agg_block_fill(int size) {
  return size == 3 && sizeof(V) == 8 ? 4096 : agg_fill(size);
}
template <class V>
__host__ __device__ constexpr int agg_block_items(int size) {
  return size == 2 ? 4096 : sizeof(V) == 8 ? 4096 : 10240;
}
template <bool COMP, class V>
__host__ __device__ constexpr size_t agg_block_smem(int size) {
  return ((size_t)1 << agg_block_log<V>(size)) * (4 + sizeof(V)) + 8 * (size_t)agg_block_items<V>(size) +
         (COMP && size == 2 ? (size_t)4 * kLaneMaxDeg * kAggThreads : 0);
}

template <bool COMP, int SIZE, class V>
__global__ void __launch_bounds__(kAggThreads, SIZE == 2 ? 3 : 1) k_agg_block(AggCtx c) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int L = agg_block_log<V>(SIZE), SLOTS = 1 << L, FILL = agg_block_fill<V>(SIZE);
  constexpr int ITEMS = agg_block_items<V>(SIZE);
  uint64_t *items = reinterpret_cast<uint64_t *>(smem);
  V *vals = reinterpret_cast<V *>(items + ITEMS);
  int32_t *keys = reinterpret_cast<int32_t *>(vals + SLOTS);
  // columns of decoded records: their own, or where the items will be (the
  // largest table leaves no room beside it; items are listed after the rows)
  uint32_t *cols = SIZE == 2 ? reinterpret_cast<uint32_t *>(keys + SLOTS)
                             : reinterpret_cast<uint32_t *>(items);
  static_assert(8 * ITEMS >= 4 * kLaneMaxDeg * kAggThreads, "columns fit where the items go");
  __shared__ int32_t s_fill, s_fail, s_d, s_wide, s_next;
  __shared__ AggQueue<V> queue[COMP ? kAggThreads / 32 : 1];
  __shared__ int32_t wide[kAggWide];  // long rows, shared out over the warps after the others
  __shared__ unsigned long long s_base;
  const int tid = threadIdx.x, lane = lane_id(), w = tid >> 5;
  V *out_val = static_cast<V *>(c.out_val);
  const int64_t cnt = c.cnt[SIZE];
  unsigned long long most = 0;
  for (int64_t q = blockIdx.x; q < cnt; q += gridDim.x) {
    const int32_t a = c.lists[(int64_t)SIZE * c.nc + q];
    const int64_t m0 = c.mstart[a] + 32 * w, m1 = c.mstart[a + 1];
    for (int i = tid; i < SLOTS; i += kAggThreads) keys[i] = -1, vals[i] = 0;
    if (tid == 0) s_fill = 0, s_fail = 0, s_d = 0, s_wide = 0, s_next = 0;
    __syncthreads();
    auto fill = [&] { return __shfl_sync(kFull, *(volatile int32_t *)&s_fill, 0); };
    auto add_fill = [&](int k) {
      if (lane == 0) atomicAdd(&s_fill, k);
      __syncwarp();
    };
    bool ok = agg_rows<COMP, V>(
        c, a, m0, m1, kAggThreads, keys, vals, L, cols + (size_t)w * kLaneMaxDeg * 32 + lane,
        queue + (COMP ? w : 0), FILL, agg_member<COMP>(c, m0, m1), fill, add_fill, [&](int32_t u) {
          int at = 0;
          if (lane == 0) {
            at = atomicAdd(&s_wide, 1);
            if (at < kAggWide) wide[at] = u;
          }
          at = __shfl_sync(kFull, at, 0);
          return at < kAggWide ||
                 agg_long_row<COMP, V>(c, a, u, 0, 1, keys, vals, L, FILL, fill, add_fill);
        });
    __syncthreads();
    const int nwide = min(s_wide, kAggWide);
    if (COMP) {  // a record is decoded by one warp
      while (ok) {
        int i = 0;
        if (lane == 0) i = atomicAdd(&s_next, 1);
        i = __shfl_sync(kFull, i, 0);
        if (i >= nwide) break;
        ok = agg_long_row<COMP, V>(c, a, wide[i], 0, 1, keys, vals, L, FILL, fill, add_fill);
      }
    } else {  // every warp takes its pieces of each row
      for (int i = 0; i < nwide && ok; ++i)
        ok = agg_long_row<COMP, V>(c, a, wide[i], (w + i) % (kAggThreads / 32), kAggThreads / 32, keys,
                                   vals, L, FILL, fill, add_fill);
    }
    if (!ok && lane == 0) s_fail = 1;
    __syncthreads();
    if (s_fail || s_fill > FILL) {  // uniform: to the next size
      if (tid == 0)
        c.lists[(int64_t)(SIZE + 1) * c.nc + atomicAdd(&c.cnt[SIZE + 1], 1)] = a;
      __syncthreads();
      continue;
    }
    for (int i = tid; i < SLOTS; i += kAggThreads) {
      const int32_t k = keys[i];
      const unsigned m = __ballot_sync(kFull, k >= 0);
      int32_t base = 0;
      if (lane == 0 && m) base = atomicAdd(&s_d, __popc(m));
      base = __shfl_sync(kFull, base, 0);
      if (k >= 0) items[base + __popc(m & lanemask_lt())] = (uint64_t)(uint32_t)k << 32 | (uint32_t)i;
    }
    __syncthreads();
    const int d = s_d;
    int n2 = 64;
    while (n2 < d) n2 <<= 1;
    if (n2 <= ITEMS) {
      for (int i = d + tid; i < n2; i += kAggThreads) items[i] = ~0ull;
      __syncthreads();
      bitonic(items, n2, tid, kAggThreads, [] { __syncthreads(); });
    } else {
      // more than 8192: the first 8192 and the rest (below 2048) sorted apart,
      // then each item goes to its rank in both
      constexpr int H = 8192;
      int r2 = 64;
      while (r2 < d - H) r2 <<= 1;
      for (int i = d + tid; i < H + r2; i += kAggThreads) items[i] = ~0ull;
      __syncthreads();
      bitonic(items, H, tid, kAggThreads, [] { __syncthreads(); });
      bitonic(items + H, r2, tid, kAggThreads, [] { __syncthreads(); });
    }
    if (tid == 0) {
      s_base = d ? atomicAdd(c.cursor, (unsigned long long)d) : 0ull;
      c.toff[a] = (int64_t)s_base;
      c.deg[a] = d;
    }
    __syncthreads();
    const bool two = n2 > ITEMS;
    const int fit = (int64_t)s_base + d <= c.room ? d : 0;
    for (int i = tid; i < fit; i += kAggThreads) {
      const uint64_t x = items[i];
      int pos = i;
      if (two) {  // rank in the other run
        constexpr int H = 8192;
        int lo = i < H ? H : 0, hi = i < H ? d : H;
        const int first = lo;
        while (lo < hi) {
          const int mid = (lo + hi) / 2;
          if (items[mid] < x) lo = mid + 1;
          else hi = mid;
        }
        pos = (i < H ? i : i - H) + lo - first;
      }
      const V wt = vals[(uint32_t)x];
      c.out_key[s_base + pos] = (int32_t)(x >> 32);
      out_val[s_base + pos] = wt;
      most = wt > most ? wt : most;
    }
    __syncthreads();  // the next coarse vertex reuses the shared memory
  }
  most = warp_max(most);
  if (lane == 0 && most) atomicMax(c.max_w, most);
}

// ---------------------------------------------------------------- coarse vertices beyond the tables
__global__ void k_mark_sorted(const int32_t *list, int64_t cnt, uint8_t *sorted) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
       i += (int64_t)gridDim.x * blockDim.x)
    sorted[list[i]] = 1;
}

// The rows of their members as items: longer rows in pieces of up to kChunkSize
// entries (compressed records below the chunking threshold whole), a warp each,
// from the front of items; rows of up to kLaneMaxDeg entries, a lane each, from
// its end (room entries; a warp each made the contraction of a mesh of 4.2 M
// vertices into 64 clusters 4.1 ms longer, compressed, and 1.1 as CSR).
// n_items: [0] long, [1] short.
template <bool COMP>
__global__ void k_row_items(GView g, const int32_t *map, const uint8_t *sorted, uint64_t *items,
                            int64_t room, unsigned long long *n_items) {
  for (int64_t u0 = (int64_t)blockIdx.x * blockDim.x; u0 < g.n;
       u0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = u0 + threadIdx.x;
    int64_t k = 0;
    bool lane_row = false;
    if (u < g.n && sorted[map[u]]) {
      int64_t deg;
      if (COMP) {
        const ZipNbr z = zip_nbr(g, u);
        deg = z.deg;
        k = z.nchunks;
      } else {
        deg = g.xadj[u + 1] - g.xadj[u];
        k = (deg + kChunkSize - 1) / kChunkSize;
      }
      lane_row = deg > 0 && deg <= kLaneMaxDeg;
      if (deg <= kLaneMaxDeg) k = 0;
    }
    const unsigned sh = __ballot_sync(kFull, lane_row);
    if (sh) {
      unsigned long long base = 0;
      if (lane_id() == 0) base = atomicAdd(&n_items[1], (unsigned long long)__popc(sh));
      base = __shfl_sync(kFull, base, 0);
      if (lane_row) items[room - 1 - (int64_t)base - __popc(sh & lanemask_lt())] = (uint64_t)u << 32;
    }
    const int64_t incl = warp_incl_scan(k);
    const int64_t total = __shfl_sync(kFull, incl, 31);
    if (total == 0) continue;  // uniform over the warp
    unsigned long long base = 0;
    if (lane_id() == 0) base = atomicAdd(&n_items[0], (unsigned long long)total);
    base = __shfl_sync(kFull, base, 0) + (unsigned long long)(incl - k);
    for (int64_t j = 0; j < k; ++j) items[base + j] = (uint64_t)u << 32 | (uint64_t)j;
  }
}

// Inter-cluster entries per item: the nl long ones, then the ns short ones.
struct RowItems {
  const uint64_t *items;
  int64_t room, nl, ns;
};
template <bool COMP>
__global__ void k_item_count(GView g, const int32_t *map, RowItems r, int64_t *cnt) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nt = (int64_t)gridDim.x * blockDim.x;
  for (int64_t it = t >> 5; it < r.nl; it += nt >> 5) {
    const int64_t u = (int64_t)(r.items[it] >> 32), j = (int64_t)(r.items[it] & 0xffffffffu);
    const int32_t a = map[u];
    int64_t c = 0;
    warp_neighbours<COMP>(g, u, j, [&](bool has, int32_t v, int64_t, int64_t) {
      c += has && map[v] != a;
    });
    c = warp_sum(c);
    if (lane_id() == 0) cnt[it] = c;
  }
  for (int64_t it = t; it < r.ns; it += nt) {
    const int64_t u = (int64_t)(r.items[r.room - 1 - it] >> 32);
    const int32_t a = map[u];
    int64_t c = 0;
    thread_neighbours<COMP>(g, u, [&](int32_t v, int64_t) { c += map[v] != a; });
    cnt[r.nl + it] = c;
  }
}

// Sort key of an inter-cluster entry: a * n' + b, with the fine edge weight
// in the low wbits bits (wbits = 0: weights apart, in vals, or unit).
__device__ __forceinline__ uint64_t entry_key(int32_t a, int32_t b, int64_t nc, int64_t w,
                                              int wbits) {
  const uint64_t k = (uint64_t)a * (uint64_t)nc + (uint64_t)b;
  return wbits ? (k << wbits) | (uint64_t)w : k;
}

template <bool COMP>
__global__ void k_item_emit(GView g, const int32_t *map, RowItems r, int64_t nc, int wbits,
                            const int64_t *off, uint64_t *keys, uint64_t *vals) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nt = (int64_t)gridDim.x * blockDim.x;
  for (int64_t it = t >> 5; it < r.nl; it += nt >> 5) {
    const int64_t u = (int64_t)(r.items[it] >> 32), j = (int64_t)(r.items[it] & 0xffffffffu);
    const int32_t a = map[u];
    int64_t pos = off[it];
    warp_neighbours<COMP>(g, u, j, [&](bool has, int32_t v, int64_t w, int64_t) {
      const int32_t b = has ? map[v] : a;
      const bool keep = has && b != a;
      const unsigned m = __ballot_sync(kFull, keep);
      if (keep) {
        const int64_t at = pos + __popc(m & lanemask_lt());
        keys[at] = entry_key(a, b, nc, w, wbits);
        if (vals) vals[at] = (uint64_t)w;
      }
      pos += __popc(m);
    });
  }
  for (int64_t it = t; it < r.ns; it += nt) {
    const int64_t u = (int64_t)(r.items[r.room - 1 - it] >> 32);
    const int32_t a = map[u];
    int64_t pos = off[r.nl + it];
    thread_neighbours<COMP>(g, u, [&](int32_t v, int64_t w) {
      const int32_t b = map[v];
      if (b == a) return;
      keys[pos] = entry_key(a, b, nc, w, wbits);
      if (vals) vals[pos] = (uint64_t)w;
      ++pos;
    });
  }
}

// Run-length reduction of the sorted entries, 4096 per tile. Pass 1: runs
// starting in every tile.
constexpr int kRleThreads = 256;
constexpr int64_t kRleTile = 4096;

__device__ __forceinline__ bool run_head(const uint64_t *keys, int64_t i, int wbits) {
  return i == 0 || (keys[i] >> wbits) != (keys[i - 1] >> wbits);
}

__global__ void __launch_bounds__(kRleThreads) k_rle_count(const uint64_t *keys, int64_t m,
                                                           int wbits, int64_t ntiles,
                                                           int64_t *tcnt) {
  __shared__ int32_t red[kRleThreads / 32];
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int64_t b = t * kRleTile, e = min(b + kRleTile, m);
    int32_t c = 0;
    for (int64_t i = b + threadIdx.x; i < e; i += kRleThreads) c += run_head(keys, i, wbits);
    c = warp_sum(c);
    if (lane_id() == 0) red[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
      int32_t tot = 0;
      for (int w = 0; w < kRleThreads / 32; ++w) tot += red[w];
      tcnt[t] = tot;
    }
    __syncthreads();
  }
}

// Pass 2: every entry adds its weight to its run's slot (the runs before it,
// from the tile's offset plus a block scan); a run's first entry also writes
// the neighbour and the coarse vertex, and counts its degree.
__global__ void __launch_bounds__(kRleThreads) k_rle_write(const uint64_t *keys,
                                                           const uint64_t *vals, int64_t m,
                                                           int64_t nc, int wbits, int64_t ntiles,
                                                           const int64_t *toff, int32_t *adj,
                                                           int64_t *ew, int32_t *row,
                                                           int64_t *deg) {
  __shared__ int32_t ws[kRleThreads / 32];
  const uint64_t wmask = wbits ? ((uint64_t)1 << wbits) - 1 : 0;
  const int lane = lane_id(), w = threadIdx.x >> 5;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    int64_t base = toff[t];  // runs started before this step
    const int64_t b = t * kRleTile, e = min(b + kRleTile, m);
    for (int64_t i0 = b; i0 < e; i0 += kRleThreads) {
      const int64_t i = i0 + threadIdx.x;
      const bool in = i < e;
      const int32_t h = in && run_head(keys, i, wbits);
      // block-wide inclusive scan of the head flags
      const unsigned bal = __ballot_sync(kFull, h);
      const int32_t winc = __popc(bal & (lanemask_lt() | (1u << lane)));
      if (lane == 31) ws[w] = winc;
      __syncthreads();
      int32_t before = 0, total = 0;
      for (int q = 0; q < kRleThreads / 32; ++q) {
        const int32_t c = ws[q];
        before += q < w ? c : 0;
        total += c;
      }
      if (in) {
        const int64_t slot = base + before + winc - 1;
        const uint64_t k = keys[i];
        const uint64_t key = k >> wbits;
        const uint64_t wt = wbits ? (k & wmask) : (vals ? vals[i] : 1ull);
        if (h) {
          adj[slot] = (int32_t)(key % (uint64_t)nc);
          row[slot] = (int32_t)(key / (uint64_t)nc);
          atomicAdd((unsigned long long *)&deg[key / (uint64_t)nc], 1ull);
        }
        atomicAdd((unsigned long long *)&ew[slot], (unsigned long long)wt);
      }
      base += total;
      __syncthreads();  // ws is rewritten by the next step
    }
  }
}

// The rows from the tables into the coarse CSR (sorted = those of hubs' coarse
// vertices, which come from the runs below).
template <class V>
__global__ void k_copy_rows(const int64_t *toff, const int64_t *xadj, const uint8_t *sorted,
                            int64_t nc, int lanes, const int32_t *key, const V *val, int32_t *adj,
                            int64_t *ew) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t ng = (int64_t)gridDim.x * blockDim.x / lanes;
  for (int64_t a = t / lanes; a < nc; a += ng) {
    if (sorted && sorted[a]) continue;
    const int64_t b = xadj[a], d = xadj[a + 1] - b, src = toff[a];
#pragma unroll 4
    for (int64_t i = t % lanes; i < d; i += lanes) {
      adj[b + i] = key[src + i];
      ew[b + i] = (int64_t)val[src + i];
    }
  }
}

// The runs of the sorted entries into the coarse CSR (start: first run of
// every coarse vertex), and the largest weight among them.
__global__ void k_copy_runs(const int64_t *start, const int64_t *xadj, int64_t runs,
                            const int32_t *row, const int32_t *key, const int64_t *val,
                            int32_t *adj, int64_t *ew) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < runs;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t a = row[i];
    const int64_t to = xadj[a] + i - start[a];
    adj[to] = key[i];
    ew[to] = val[i];
  }
}

__global__ void k_add_i64(const int64_t *a, int64_t n, int64_t *b) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    b[i] += a[i];
}

// How rows are summed: as it suits the graph, all sorted, or through the tables
// with no more room than a sample says.
enum RowMode { ROWS_ANY, ROWS_SORTED, ROWS_TIGHT };

// Graphs of at least this many vertices are sampled for the room of the rows.
constexpr int64_t kSampleFrom = (int64_t)1 << 20;

// Whether all rows are sorted at once instead of through the tables, which one
// after the other wait for their longest coarse vertices: skewed graphs of 2^18
// to 2^25 entries of which some coarse vertices are long (or of which few
// entries merge: long single rows overflow the table they start in), unless most
// entries are short rows' or merge strongly. R-MAT of 20 000, 64 752, 2e5, 4e5
// and 1e6 vertices, k = 2: 0.85, 1.13, 1.46, 1.85, 3.27 ms through the tables,
// 0.52, 0.63, 0.89, 1.32, 3.35 sorted; meshes of those sizes take twice as long
// sorted. cnt: coarse vertices by first size, low: entries of those of the
// smallest.
bool sort_pays(int64_t m2, int64_t nc, const int32_t (&cnt)[kAggSizes + 1], int64_t low) {
  if (m2 < ((int64_t)1 << 18) || m2 > ((int64_t)1 << 25) || (m2 > ((int64_t)1 << 21) && 5 * low > 4 * m2))
    return false;
  return (cnt[3] + cnt[4] > 0 && m2 <= 1300 * nc) || (cnt[2] > 0 && m2 <= 200 * nc);
}

// The block of k_agg_block / k_agg_warp grids: as many as fit the SMs, no more
// than the longest the list can become.
template <bool COMP, class V>
void launch_agg(const AggCtx &c, const int64_t (&most)[kAggSizes], cudaStream_t s) {
  const int sms = num_sms();
  auto run = [&](auto kern, int64_t blocks, int threads, size_t smem) {
    TP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int per_sm = std::max(1, std::min(2048 / threads, (int)((size_t)(228 * 1024) / (smem + 1024))));
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(blocks, (int64_t)sms * per_sm));
    launch(kern, grid, threads, smem, s, c);
    TP_LAUNCH_CHECK();
  };
  constexpr int W0 = agg_warps(0), W1 = agg_warps(1);
  if (most[0]) run(k_agg_warp<COMP, 0, V>, (most[0] + W0 - 1) / W0, 32 * W0, sizeof(AggWarp<COMP, 0, V>) * W0);
  if (most[1]) run(k_agg_warp<COMP, 1, V>, (most[1] + W1 - 1) / W1, 32 * W1, sizeof(AggWarp<COMP, 1, V>) * W1);
  if (most[2]) run(k_agg_block<COMP, 2, V>, most[2], kAggThreads, agg_block_smem<COMP, V>(2));
  if (most[3]) run(k_agg_block<COMP, 3, V>, most[3], kAggThreads, agg_block_smem<COMP, V>(3));
}

}  // namespace

// The contraction itself. own (nullable): holds g if g is a decoded copy, freed
// as soon as its rows are summed.
static tp_graph *contract_rows(const tp_graph *g, std::unique_ptr<tp_graph> *own, RowMode mode,
                               const int32_t *C, int32_t *d_map, cudaStream_t s,
                               const int64_t *seg_voff, int64_t nseg, int64_t *seg_coff) {
  const int64_t n = g->n;
  tp_graph *cg = new_graph();
  try {
    cg->err.alloc(1, s);
    TP_CUDA(cudaMemsetAsync(cg->err.get(), 0, sizeof(int32_t), s));
    cg->unit_vw = 0;
    cg->unit_ew = 0;
    if (n == 0) {
      cg->xadj.alloc(1, s);
      TP_CUDA(cudaMemsetAsync(cg->xadj.get(), 0, 8, s));
      TP_CUDA(cudaStreamSynchronize(s));
      return cg;
    }
    Buf<int64_t> rank(n + 1, s);
    {
      Buf<int32_t> flag(n, s);
      TP_CUDA(cudaMemsetAsync(flag.get(), 0, n * sizeof(int32_t), s));
      launch(k_mark, grid_for(n, 256), 256, 0, s, C, n, flag.get());
      TP_LAUNCH_CHECK();
      exclusive_scan_i32_to_i64(flag.get(), rank.get(), n, s);
    }
    if (seg_voff) {
      launch(k_seg_rank, grid_for(nseg + 1, 256), 256, 0, s, rank.get(), seg_voff, nseg, seg_coff);
      TP_LAUNCH_CHECK();
    }
    const int64_t nc = read_scalar(rank.get() + n, s);
    cg->n = nc;
    Buf<int32_t> own_map;
    int32_t *map = d_map;
    if (!map) {
      own_map.alloc(n, s);
      map = own_map.get();
    }
    cg->total_vw = g->total_vw;
    cg->sum_ew = ew_sum_bound(g);
    cg->vw.alloc(nc, s);
    if (!g->unit_vw) TP_CUDA(cudaMemsetAsync(cg->vw.get(), 0, nc * sizeof(int64_t), s));
    const GView v = view(g);
    const bool comp = g->compressed;
    // 32-bit sums in the tables: where all edge weights together fit, or weigh
    // one each: no coarse vertex of more than agg_start entries enters a table,
    // however many the graph has (compressed graphs of 2^31 entries and more
    // among them, whose kernels exist with this type only)
    const bool narrow = g->unit_ew || ew_sum_bound(g) < ((int64_t)1 << 31);

    // members by coarse vertex, and the first table size of each
    Buf<int32_t> members(n, s), lists((kAggSizes + 1) * nc, s);
    Buf<int64_t> mstart(nc + 1, s);
    // [0] cursor [1] largest weight [2], [3] items [4] rows' bound [5] entries of the
    // smallest table [6], [7] sample; then the lists' lengths (int32)
    constexpr int kAcc = 8;
    Buf<int64_t> acc(kAcc + (kAggSizes + 2) / 2, s);
    TP_CUDA(cudaMemsetAsync(acc.get(), 0, acc.n * sizeof(int64_t), s));
    int32_t *cnt = reinterpret_cast<int32_t *>(acc.get() + kAcc);
    Buf<int32_t> place(n, s), mcnt(nc, s);
    {
      Buf<unsigned long long> ent(nc, s);
      TP_CUDA(cudaMemsetAsync(mcnt.get(), 0, nc * sizeof(int32_t), s));
      TP_CUDA(cudaMemsetAsync(ent.get(), 0, nc * sizeof(unsigned long long), s));
      launch(k_map, grid_for(n, 256), 256, 0, s, v, C, rank.get(), map, cg->vw.get(), place.get(),
             mcnt.get(), ent.get());
      launch(k_agg_classes, grid_for(nc, 256), 256, 0, s, ent.get(), mcnt.get(), nc,
             g->unit_vw ? cg->vw.get() : nullptr, lists.get(), cnt,
             (unsigned long long *)(acc.get() + 4));
      if (n >= kSampleFrom || mode == ROWS_TIGHT)
        launch(comp ? k_row_sample<true> : k_row_sample<false>, (unsigned)(kRowSamples * 32 / 256), 256,
               0, s, v, map, (unsigned long long *)(acc.get() + 6));
      TP_LAUNCH_CHECK();
    }
    rank.release();
    int64_t ha[kAcc + (kAggSizes + 2) / 2];
    TP_CUDA(cudaMemcpyAsync(ha, acc.get(), sizeof(ha), cudaMemcpyDeviceToHost, s));
    TP_CUDA(cudaStreamSynchronize(s));
    int32_t hc[kAggSizes + 1];
    std::copy_n(reinterpret_cast<const int32_t *>(ha + kAcc), kAggSizes + 1, hc);
    // lists can grow by those that move up from the smaller sizes
    int64_t most[kAggSizes], sofar = 0;
    for (int i = 0; i < kAggSizes; ++i) most[i] = sofar += hc[i];

    // the tables' rows: no more entries than their coarse vertices' members have,
    // and in a large graph room for a quarter more than the sampled share of
    // inter-cluster ones (a third in a mesh, whose rows of all entries were the
    // peak of a partition); if that falls short the tables are filled again with
    // the room they turned out to need
    const bool keys_only =
        mode == ROWS_SORTED || (mode == ROWS_ANY && !seg_voff && sort_pays(g->m2, nc, hc, ha[5]));
    if (!keys_only) {
      exclusive_scan_i32_to_i64(mcnt.get(), mstart.get(), nc, s);
      launch(k_members, grid_for(n, 256), 256, 0, s, map, place.get(), mstart.get(), n, members.get());
      TP_LAUNCH_CHECK();
    }
    place.release();
    mcnt.release();
    int64_t room = keys_only ? 0 : std::min<int64_t>(ha[4], g->m2);
    if (!keys_only && ha[7] > 0)
      room = std::min<int64_t>(room, (int64_t)(1.25 * (double)g->m2 * (double)ha[6] / (double)ha[7]) + n / 16);
    Buf<int32_t> tkey;
    Buf<uint32_t> tval32;
    Buf<unsigned long long> tval64;
    Buf<int64_t> toff(nc, s);
    cg->xadj.alloc(nc + 1, s);
    TP_CUDA(cudaMemsetAsync(cg->xadj.get(), 0, (nc + 1) * sizeof(int64_t), s));
    AggCtx c{};
    c.g = v;
    c.map = map;
    c.members = members.get();
    c.mstart = mstart.get();
    c.nc = nc;
    c.lists = lists.get();
    c.cnt = cnt;
    c.cursor = (unsigned long long *)acc.get();
    c.max_w = (unsigned long long *)(acc.get() + 1);
    c.toff = toff.get();
    c.deg = cg->xadj.get();
    while (!keys_only) {
      tkey.alloc(std::max<int64_t>(room, 1), s);
      if (narrow) tval32.alloc(std::max<int64_t>(room, 1), s);
      else tval64.alloc(std::max<int64_t>(room, 1), s);
      c.room = room;
      c.out_key = tkey.get();
      c.out_val = narrow ? (void *)tval32.get() : (void *)tval64.get();
      if (comp) launch_agg<true, uint32_t>(c, most, s);
      else if (narrow) launch_agg<false, uint32_t>(c, most, s);
      else launch_agg<false, unsigned long long>(c, most, s);
      TP_CUDA(cudaMemcpyAsync(ha, acc.get(), sizeof(ha), cudaMemcpyDeviceToHost, s));
      TP_CUDA(cudaStreamSynchronize(s));
      if (ha[0] <= room) break;
      room = ha[0];
      tkey.release();
      tval32.release();
      tval64.release();
      TP_CUDA(cudaMemsetAsync(acc.get(), 0, 2 * sizeof(int64_t), s));
      TP_CUDA(cudaMemcpyAsync(cnt, hc, sizeof(hc), cudaMemcpyHostToDevice, s));
    }
    const int64_t n_sorted = keys_only ? nc : reinterpret_cast<const int32_t *>(ha + kAcc)[kAggSizes];
    int64_t max_w = ha[1], m2 = ha[0], runs = 0;

    // coarse vertices beyond the tables: keys, sort, run lengths
    Buf<uint8_t> sorted;
    Buf<int32_t> rkey, rrow;
    Buf<int64_t> rval, rstart;
    if (n_sorted) {
      sorted.alloc(nc, s);
      TP_CUDA(cudaMemsetAsync(sorted.get(), keys_only ? 1 : 0, nc, s));
      if (!keys_only)
        launch(k_mark_sorted, grid_for(n_sorted, 256), 256, 0, s, lists.get() + kAggSizes * nc, n_sorted,
               sorted.get());
      RowItems ri{};
      ri.room = n + g->m2 / kChunkSize + 1;
      Buf<uint64_t> items((size_t)ri.room, s);
      unsigned long long *n_items = (unsigned long long *)(acc.get() + 2);
      launch(comp ? k_row_items<true> : k_row_items<false>, grid_for(n, 256), 256, 0, s, v, map,
             sorted.get(), items.get(), ri.room, n_items);
      TP_LAUNCH_CHECK();
      int64_t hi[2];
      TP_CUDA(cudaMemcpyAsync(hi, n_items, sizeof(hi), cudaMemcpyDeviceToHost, s));
      TP_CUDA(cudaStreamSynchronize(s));
      ri.items = items.get();
      ri.nl = hi[0];
      ri.ns = hi[1];
      const int64_t ni = ri.nl + ri.ns;
      Buf<int64_t> off(ni + 1, s);
      const unsigned ib = grid_for(std::max(ri.nl * 32, ri.ns), 256);
      if (ni) {
        launch(comp ? k_item_count<true> : k_item_count<false>, ib, 256, 0, s, v, map, ri, off.get());
        TP_LAUNCH_CHECK();
      }
      exclusive_scan_i64(off.get(), off.get(), ni, s);
      const int64_t m = read_scalar(off.get() + ni, s);
      // weights ride in the keys' low bits when the pair fits 64 bits
      const bool weighted = !g->unit_ew;
      const int kbits = bits_for((uint64_t)nc * (uint64_t)nc - 1);
      const int wbits = weighted && kbits + bits_for((uint64_t)g->max_ew) <= 64
                            ? bits_for((uint64_t)g->max_ew)
                            : 0;
      Buf<uint64_t> keys(std::max<int64_t>(m, 1), s), vals;
      if (weighted && !wbits) vals.alloc(std::max<int64_t>(m, 1), s);
      if (ni) {
        launch(comp ? k_item_emit<true> : k_item_emit<false>, ib, 256, 0, s, v, map, ri, nc, wbits,
               off.get(), keys.get(), vals.get());
        TP_LAUNCH_CHECK();
      }
      items.release();
      off.release();
      radix_sort_pairs(keys.get(), vals.get(), m, kbits, s, wbits);
      const int64_t ntiles = (m + kRleTile - 1) / kRleTile;
      Buf<int64_t> rtile(ntiles + 1, s);
      const unsigned rb = (unsigned)std::max<int64_t>(1, std::min<int64_t>(ntiles, (int64_t)num_sms() * 16));
      if (ntiles) {
        launch(k_rle_count, rb, kRleThreads, 0, s, keys.get(), m, wbits, ntiles, rtile.get());
        TP_LAUNCH_CHECK();
      }
      exclusive_scan_i64(rtile.get(), rtile.get(), ntiles, s);
      runs = read_scalar(rtile.get() + ntiles, s);
      rkey.alloc(std::max<int64_t>(runs, 1), s);
      rrow.alloc(std::max<int64_t>(runs, 1), s);
      rval.alloc(std::max<int64_t>(runs, 1), s);
      rstart.alloc(nc + 1, s);
      TP_CUDA(cudaMemsetAsync(rval.get(), 0, rval.n * sizeof(int64_t), s));
      TP_CUDA(cudaMemsetAsync(rstart.get(), 0, (nc + 1) * sizeof(int64_t), s));
      if (ntiles) {
        launch(k_rle_write, rb, kRleThreads, 0, s, keys.get(), vals.get(), m, nc, wbits, ntiles,
               rtile.get(), rkey.get(), rval.get(), rrow.get(), rstart.get());
        TP_LAUNCH_CHECK();
      }
      keys.release();
      vals.release();
      launch(k_add_i64, grid_for(nc, 256), 256, 0, s, rstart.get(), nc, cg->xadj.get());
      TP_LAUNCH_CHECK();
      exclusive_scan_i64(rstart.get(), rstart.get(), nc, s);
      max_w = std::max(max_w, max_i64(rval.get(), runs, s));
      m2 += runs;
    }
    if (own) own->reset();
    exclusive_scan_i64(cg->xadj.get(), cg->xadj.get(), nc, s);
    cg->m2 = m2;
    cg->max_ew = max_w;
    cg->adj.alloc(m2 + kAdjPad, s);
    TP_CUDA(cudaMemsetAsync(cg->adj.get() + m2, 0, kAdjPad * sizeof(int32_t), s));
    cg->ew.alloc(m2, s);
    if (m2) {
      const int lanes = m2 / nc > 24 ? 32 : 8;
      const unsigned gr = grid_for(nc * lanes, 256);
      if (narrow)
        launch(k_copy_rows<uint32_t>, gr, 256, 0, s, toff.get(), cg->xadj.get(), sorted.get(), nc,
               lanes, tkey.get(), tval32.get(), cg->adj.get(), cg->ew.get());
      else
        launch(k_copy_rows<unsigned long long>, gr, 256, 0, s, toff.get(), cg->xadj.get(), sorted.get(),
               nc, lanes, tkey.get(), tval64.get(), cg->adj.get(), cg->ew.get());
      if (runs)
        launch(k_copy_runs, grid_for(runs, 256), 256, 0, s, rstart.get(), cg->xadj.get(), runs,
               rrow.get(), rkey.get(), rval.get(), cg->adj.get(), cg->ew.get());
      TP_LAUNCH_CHECK();
    }
    TP_CUDA(cudaStreamSynchronize(s));
  } catch (...) {
    delete cg;
    throw;
  }
  return cg;
}

tp_graph *contract(const tp_graph *g, const int32_t *C, int32_t *d_map, cudaStream_t s,
                   const int64_t *seg_voff, int64_t nseg, int64_t *seg_coff) {
  // a compressed graph with long records is decoded first (each chunk once, by
  // a warp): in the tables' kernels such a record is one warp's, and level 0
  // of R-MAT 2^22 spent 39 ms in them where decoding takes 2 and the CSR
  // kernels 13.5. Where there is no room for the decoded copy the records are
  // read as they are (a mesh with a hub needs half as much that way). Small ones
  // are sorted, which takes a record apart by chunks: R-MAT of 64 752 vertices,
  // k = 256: 0.97 -> 0.78 ms.
  RowMode mode = ROWS_ANY;
  if (g->compressed && g->max_deg > kAggDecodeDeg) {
    mode = ROWS_SORTED;
    if (g->m2 > kSortZip) {
      try {
        std::unique_ptr<tp_graph> csr(decompress(g, s));
        return contract_rows(csr.get(), &csr, ROWS_ANY, C, d_map, s, seg_voff, nseg, seg_coff);
      } catch (const Error &e) {
        if (e.code != TP_ERR_OOM && e.code != TP_ERR_BUDGET) throw;
      }
      mode = ROWS_TIGHT;
    }
  }
  return contract_rows(g, nullptr, mode, C, d_map, s, seg_voff, nseg, seg_coff);
}

}  // namespace tp
