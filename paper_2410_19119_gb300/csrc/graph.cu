// Graph handles: creation and validation, degrees and degree tiers, the
// compressed format (Section "Compression Scheme") and the small ABI calls.
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <unordered_map>
#include <mutex>
#include <new>

#include "decode.cuh"

namespace tp {

// ---------------------------------------------------------------- allocator
namespace {
// The current hook; hooks are immutable and never freed (buffers keep
// pointing at the one that made them). Null functions: cudaMallocAsync.
const AllocHook g_default_hook{nullptr, nullptr, nullptr};
std::atomic<const AllocHook *> g_hook{&g_default_hook};
std::atomic<int> g_sms{0};
}  // namespace

// Device bytes this host thread holds and its high-water mark (a call runs
// on one thread, so the peak of its working set is the mark's rise), and the
// most it may hold (mem_cap; an allocation beyond it fails with TP_ERR_BUDGET
// before anything is allocated).
thread_local int64_t t_live = 0, t_peak = 0, t_cap = INT64_MAX;

void mem_cap(int64_t bytes_above_now) {
  t_cap = bytes_above_now < 0 ? INT64_MAX : t_live + bytes_above_now;
}

int64_t mem_mark() {
  t_peak = t_live;
  return t_live;
}
int64_t mem_peak_since(int64_t mark) { return t_peak - mark; }

// Opt-in (environment TP_MEM_TRACE=1): the sizes of the buffers live at this
// thread's high-water mark, printed by mem_trace_dump (a diagnostic of what a
// call's peak consists of).
static bool mem_trace_on() {
  static const bool on = getenv("TP_MEM_TRACE") != nullptr;
  return on;
}
thread_local std::unordered_map<void *, int64_t> *t_live_bufs = nullptr;
thread_local std::vector<int64_t> *t_peak_bufs = nullptr;

static void mem_add(int64_t b) {
  t_live += b;
  if (t_live > t_peak) {
    t_peak = t_live;
    if (mem_trace_on() && t_live_bufs) {
      if (!t_peak_bufs) t_peak_bufs = new std::vector<int64_t>();
      t_peak_bufs->clear();
      for (const auto &kv : *t_live_bufs) t_peak_bufs->push_back(kv.second);
    }
  }
}

static void mem_track(void *p, int64_t b) {
  if (!mem_trace_on()) return;
  if (!t_live_bufs) t_live_bufs = new std::unordered_map<void *, int64_t>();
  if (b > 0) (*t_live_bufs)[p] = b;
  else t_live_bufs->erase(p);
}

void mem_trace_dump(const char *what) {
  if (!mem_trace_on() || !t_peak_bufs) return;
  std::vector<int64_t> v = *t_peak_bufs;
  std::sort(v.begin(), v.end(), std::greater<int64_t>());
  fprintf(stderr, "terapart mem: %s peak %.3f GB in %zu buffers; largest (GB):", what,
          (double)t_peak / 1e9, v.size());
  for (size_t i = 0; i < v.size() && i < 16; ++i) fprintf(stderr, " %.3f", (double)v[i] / 1e9);
  fprintf(stderr, "\n");
}

void *dev_alloc(size_t bytes, cudaStream_t s, const AllocHook **from) {
  if (bytes == 0) return nullptr;
  if (t_live + (int64_t)bytes > t_cap) throw Error{TP_ERR_BUDGET};
  void *p = nullptr;
  const AllocHook *h = g_hook.load();
  if (h->alloc) {
    p = h->alloc(bytes, (void *)s, h->ctx);
    if (!p) throw Error{TP_ERR_OOM};
  } else {
    cudaError_t e = cudaMallocAsync(&p, bytes, s);
    if (e != cudaSuccess) {
      (void)cudaGetLastError();
      throw Error{e == cudaErrorMemoryAllocation ? TP_ERR_OOM : TP_ERR_CUDA};
    }
  }
  mem_track(p, (int64_t)bytes);
  mem_add((int64_t)bytes);
  *from = h;
  return p;
}

void dev_free(void *p, size_t bytes, cudaStream_t s, const AllocHook *from) {
  if (!p) return;
  t_live -= (int64_t)bytes;
  mem_track(p, 0);
  if (from && from->free) {
    from->free(p, bytes, (void *)s, from->ctx);
    return;
  }
  cudaFreeAsync(p, s);
}

namespace {
std::atomic<uint64_t> g_launches{0};

struct ProfRecord {
  int family;
  cudaEvent_t a, b;
  double bytes;
};
// The profiler serves one host thread at a time (benchmarks); the scope flag
// is per thread so concurrent partitions (tp_partition_batch) never record.
thread_local bool t_prof_scope = false;
struct Profiler {
  bool enabled = false;
  std::vector<ProfRecord> recs;
  std::vector<cudaEvent_t> pool;
  cudaEvent_t open[PF_COUNT] = {};
  cudaEvent_t get() {
    if (!pool.empty()) {
      cudaEvent_t e = pool.back();
      pool.pop_back();
      return e;
    }
    cudaEvent_t e;
    TP_CUDA(cudaEventCreate(&e));
    return e;
  }
} g_prof;
}  // namespace

// Launches recorded into a CUDA graph are counted when the graph runs.
thread_local bool t_capturing = false;
thread_local uint64_t t_captured = 0;
void count_launch() {
  if (t_capturing) ++t_captured;
  else g_launches.fetch_add(1, std::memory_order_relaxed);
}
void count_launches(uint64_t k) { g_launches.fetch_add(k, std::memory_order_relaxed); }
uint64_t capture_counting(bool on) {
  t_capturing = on;
  if (on) t_captured = 0;
  return t_captured;
}
bool prof_active() { return t_prof_scope && g_prof.enabled; }
void prof_scope(bool on) { t_prof_scope = on; }
void prof_begin(int family, cudaStream_t s) {
  if (!prof_active()) return;
  cudaEvent_t e = g_prof.get();
  TP_CUDA(cudaEventRecord(e, s));
  g_prof.open[family] = e;
}
void prof_end(int family, cudaStream_t s, double alg_bytes) {
  if (!prof_active() || !g_prof.open[family]) return;
  cudaEvent_t e = g_prof.get();
  TP_CUDA(cudaEventRecord(e, s));
  g_prof.recs.push_back({family, g_prof.open[family], e, alg_bytes});
  g_prof.open[family] = nullptr;
}

int num_sms() {
  int v = g_sms.load(std::memory_order_relaxed);
  if (!v) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    if (v <= 0) v = 1;
    g_sms.store(v, std::memory_order_relaxed);  // every thread computes the same value
  }
  return v;
}

GView view(const tp_graph *g) {
  GView v;
  v.n = g->n;
  v.m2 = g->m2;
  v.xadj = g->xadj.get();
  v.adj = g->adj.get();
  v.vw = g->unit_vw ? nullptr : g->vw.get();
  v.ew = g->unit_ew ? nullptr : g->ew.get();
  v.bytes = g->bytes.get();
  v.off32 = g->off_is64 ? nullptr : g->off32.get();
  v.off64 = g->off_is64 ? g->off64.get() : nullptr;
  v.compressed = g->compressed;
  v.err = g->err.get();
  return v;
}

tp_graph *new_graph() { return new tp_graph(); }

// ---------------------------------------------------------------- reductions
namespace {

// out[0] += sum vw (or n if vw null); out[1] = max degree. One atomic pair
// per block: one per warp queued 2 x 39 000 atomics on two words (57 us for
// 3 M vertices, several times the 24 MB it reads).
__global__ void __launch_bounds__(256) k_sum_max(const int64_t *vw, const int64_t *xadj, int64_t n,
                                                 int64_t *out) {
  __shared__ int64_t ss[8], sm[8];
  int64_t s = 0, m = 0;
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    s += vw ? vw[u] : 1;
    if (xadj) {
      int64_t d = xadj[u + 1] - xadj[u];
      m = d > m ? d : m;
    }
  }
  s = warp_sum(s);
  m = warp_max(m);
  if (lane_id() == 0) ss[threadIdx.x >> 5] = s, sm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) s += ss[w], m = sm[w] > m ? sm[w] : m;
    atomicAdd((unsigned long long *)&out[0], (unsigned long long)s);
    atomicMax((long long *)&out[1], (long long)m);
  }
}

// ---- adjacency entries in tiles
// Work per adjacency entry (validation, encoding) is cut into tiles of kTile
// consecutive entries, one block each, so hubs and low-degree vertices load
// the GPU alike (a warp per vertex left most lanes idle at degree 16 and a
// hub of 1e5 neighbours to a single warp). tile_first[t] is the first vertex
// whose row starts at or behind entry t * kTile (tiles 0 .. m2 / kTile, one
// sentinel more: n + 1); vertex n stands for the end of the last row.
constexpr int kTileThreads = 256;
constexpr int kTileItems = 8;
constexpr int kTile = kTileThreads * kTileItems;

// Row-wise checks of a CSR graph (offsets, vertex weights) and the tiles'
// first vertices. bad[0] is set where a row is malformed; tile_first is
// complete only where it is not. empties (nullable): set if any row is empty.
__global__ void k_rows(const int64_t *xadj, const int64_t *vw, int64_t n, int64_t m2,
                       int32_t *tile_first, int32_t *bad, int32_t *empties) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u <= n;
       u += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = xadj[u], pb = u ? xadj[u - 1] : -1;
    const bool ok = b >= 0 && b <= m2 && b >= pb && (u != 0 || b == 0) && (u != n || b == m2) &&
                    (u == n || !vw || vw[u] > 0);
    if (!ok) {
      atomicCAS(bad, 0, 1);
      continue;
    }
    // (every writer writes the same; a store for each of 2^24 empty rows took 0.2 ms)
    if (empties && b == pb && *empties == 0) *empties = 1;
    // tiles t with pb < t * kTile <= b (for u = 0 that is tile 0)
    for (int64_t t = pb < 0 ? 0 : pb / kTile + 1; t * kTile <= b; ++t) tile_first[t] = (int32_t)u;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) tile_first[m2 / kTile + 1] = (int32_t)(n + 1);
}

__device__ __forceinline__ int tpad(int i) { return i + (i >> 5); }

// A tile behind a long run of empty rows has that many rows that start in it,
// and one block would walk them all. From this many on (512 KB of offsets)
// every entry of the tile searches its row instead, one after the other in a
// thread (eight side by side cost every tile registers: validation of a mesh of
// 4.2 M vertices 0.50 -> 0.53 ms). A graph with a gap of 2^27 rows took 71 ms to
// validate and 506 ms to compress, with the searches 1.1 and 1.3 ms.
constexpr int64_t kTileManyRows = 32 * (int64_t)kTile;

// The last of the rows lo .. hi that starts at or before entry e.
__device__ __forceinline__ int64_t row_of_entry(const int64_t *xadj, int64_t lo, int64_t hi,
                                                int64_t e) {
  for (int64_t left = hi - lo + 1; left > 1;) {
    const int64_t h = left >> 1;
    if (xadj[lo + h] <= e) lo += h;
    left -= h;
  }
  return lo;
}

__device__ __forceinline__ bool many_rows(const int32_t *tile_first, int64_t t) {
  return (int64_t)tile_first[t + 1] - tile_first[t] >= kTileManyRows;
}

// Row of every entry of tile t, relative to base = tile_first[t] - 1 (the row
// that contains the tile's first entry unless a row starts there): the rows
// that start inside the tile mark their first entry and a block-wide maximum
// scan carries the marks on (of several rows with one start, the last is the
// one with entries). row holds kTile + kTile / 32 words, indexed by tpad.
__device__ __forceinline__ void tile_rows(const int64_t *xadj, const int32_t *tile_first, int64_t t,
                                          int64_t n, int32_t *row) {
  __shared__ int32_t wmax[kTileThreads / 32];
  const int64_t e0 = t * kTile;
  const int32_t base = tile_first[t] - 1;
  for (int i = threadIdx.x; i < kTile; i += kTileThreads) row[tpad(i)] = 0;
  __syncthreads();
  const int64_t rend = min((int64_t)tile_first[t + 1], n);
  for (int64_t r = (int64_t)base + 1 + threadIdx.x; r < rend; r += kTileThreads)
    atomicMax(&row[tpad((int)(xadj[r] - e0))], (int32_t)(r - base));
  __syncthreads();
  const int i0 = threadIdx.x * kTileItems;
  int32_t v[kTileItems], m = 0;
#pragma unroll
  for (int j = 0; j < kTileItems; ++j) v[j] = m = max(m, row[tpad(i0 + j)]);
  int32_t x = m;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(kFull, x, o);
    if (lane_id() >= o) x = max(x, y);
  }
  if (lane_id() == 31) wmax[threadIdx.x >> 5] = x;
  __syncthreads();
  int32_t before = __shfl_up_sync(kFull, x, 1);
  if (lane_id() == 0) before = 0;
  for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) before = max(before, wmax[w]);
#pragma unroll
  for (int j = 0; j < kTileItems; ++j) row[tpad(i0 + j)] = max(before, v[j]);
  __syncthreads();
}

// Entry-wise checks of a CSR graph whose rows are well-formed: ids in range,
// no loops, strictly ascending rows, positive weights, and symmetry. A row is
// a set once it ascends, so symmetry needs one search per edge, not two: every
// entry (u, v) with v > u must have its mirror in row v, and as many entries
// lie above the diagonal as below (balance sums to zero), so the mirrors are
// all of the lower ones. The upper entries of a tile are listed first, so the
// searches run with full warps, kSearch of them in step per thread: bound by
// the searches' dependent loads.
constexpr int kSearch = 4;

// The same for a tile of very many rows, an entry at a time and apart from the
// others (as a branch among them it cost a mesh of 4.2 M vertices 0.50 -> 0.54
// ms). Returns this thread's upper minus lower entries.
__device__ __noinline__ int64_t validate_many(const GView &g, const int32_t *tile_first, int64_t t,
                                              int32_t *bad) {
  const int64_t lo = max(tile_first[t] - 1, 0), hi = min((int64_t)tile_first[t + 1], g.n) - 1;
  int64_t diff = 0;
  for (int64_t e = t * kTile + threadIdx.x; e < min((t + 1) * kTile, g.m2); e += kTileThreads) {
    const int64_t u = row_of_entry(g.xadj, lo, hi, e);
    const int32_t v = g.adj[e];
    int code = 0;
    if ((uint32_t)v >= (uint32_t)g.n || v == u) {
      code = 4;
    } else {
      if (g.xadj[u] < e && g.adj[e - 1] >= v) code = 6;
      if (g.ew && g.ew[e] <= 0) code = 7;
      diff += v > u ? 1 : -1;
      if (v > u) {  // the mirror: the last entry <= u of row v
        int64_t b = g.xadj[v], left = g.xadj[v + 1] - b;
        if (left == 0) {
          code = 8;
        } else {
          for (; left > 1; left -= left >> 1)
            if (g.adj[b + (left >> 1)] <= u) b += left >> 1;
          if (g.adj[b] != u || (g.ew && g.ew[b] != g.ew[e])) code = 8;
        }
      }
    }
    if (code) atomicCAS(bad, 0, code);
  }
  return diff;
}

__global__ void __launch_bounds__(kTileThreads) k_validate(GView g, const int32_t *tile_first,
                                                           int64_t ntiles,
                                                           const int32_t *bad_rows, int32_t *bad,
                                                           unsigned long long *balance) {
  __shared__ int32_t row[kTile + kTile / 32];
  __shared__ uint16_t upper[kTile];
  __shared__ int32_t n_upper;
  if (*bad_rows) return;  // set by k_rows: the rows cannot be followed
  int64_t diff = 0;  // (thread 0)
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    if (many_rows(tile_first, t)) {  // uniform over the block
      const int64_t d = validate_many(g, tile_first, t, bad);
      if (d) atomicAdd(balance, (unsigned long long)d);
      continue;
    }
    if (threadIdx.x == 0) n_upper = 0;
    tile_rows(g.xadj, tile_first, t, g.n, row);  // (with barriers)
    const int64_t e0 = t * kTile;
    const int32_t base = tile_first[t] - 1;
    const int len = (int)min((int64_t)kTile, g.m2 - e0);
    const int32_t *adj = g.adj + e0;
    int code = 0;
    int32_t vv[kTileItems], pv[kTileItems];
#pragma unroll
    for (int j = 0; j < kTileItems; ++j) {
      const int i = threadIdx.x + j * kTileThreads;
      vv[j] = i < len ? adj[i] : 0;
      pv[j] = i < len && e0 + i > 0 ? adj[i - 1] : 0;
    }
#pragma unroll
    for (int j = 0; j < kTileItems; ++j) {
      const int i = threadIdx.x + j * kTileThreads;
      bool up = false;
      if (i < len) {
        const int32_t r = row[tpad(i)], u = base + r, v = vv[j];
        if ((uint32_t)v >= (uint32_t)g.n || v == u) {
          code = 4;
        } else {
          const bool inside = i ? row[tpad(i - 1)] == r : g.xadj[u] < e0;
          if (inside && pv[j] >= v) code = 6;
          if (g.ew && g.ew[e0 + i] <= 0) code = 7;
          up = v > u;
        }
      }
      const unsigned m = __ballot_sync(kFull, up);
      if (m) {
        int32_t at = 0;
        if (lane_id() == 0) at = atomicAdd(&n_upper, __popc(m));
        at = __shfl_sync(kFull, at, 0);
        if (up) upper[at + __popc(m & lanemask_lt())] = (uint16_t)i;
      }
    }
    __syncthreads();
    const int nu = n_upper;
    if (threadIdx.x == 0) diff += 2 * nu - len;
    for (int q0 = threadIdx.x; q0 < nu; q0 += kSearch * kTileThreads) {
      int32_t u[kSearch], left[kSearch];
      const int32_t *p[kSearch];
      int most = 0;
#pragma unroll
      for (int k = 0; k < kSearch; ++k) {
        const int q = q0 + k * kTileThreads;
        const int i = q < nu ? upper[q] : -1;
        u[k] = i >= 0 ? base + row[tpad(i)] : 0;
        const int32_t v = i >= 0 ? adj[i] : 0;
        const int64_t b = i >= 0 ? g.xadj[v] : 0;
        left[k] = i >= 0 ? (int32_t)(g.xadj[v + 1] - b) : -1;
        p[k] = g.adj + b;
        most = max(most, left[k]);
      }
      // the last entry <= u of each row: halves until one entry is left
      while (most > 1) {
#pragma unroll
        for (int k = 0; k < kSearch; ++k) {
          const int32_t h = left[k] > 1 ? left[k] >> 1 : 0;
          if (h && p[k][h] <= u[k]) p[k] += h;
          left[k] -= h;
        }
        most -= most >> 1;
      }
#pragma unroll
      for (int k = 0; k < kSearch; ++k) {
        if (left[k] < 0) continue;
        if (left[k] == 0 || *p[k] != u[k]) code = 8;
        else if (g.ew && g.ew[p[k] - g.adj] != g.ew[e0 + upper[q0 + k * kTileThreads]]) code = 8;
      }
    }
    if (code) atomicCAS(bad, 0, code);
    __syncthreads();  // row, upper and n_upper are rebuilt by the next tile
  }
  if (threadIdx.x == 0 && diff) atomicAdd(balance, (unsigned long long)diff);
}

}  // namespace

// ---------------------------------------------------------------- tiers
namespace {

// Compressed lane-tier records longer than this take the decoder that loads
// beyond its 80-byte window; they join the lane tier only where they are
// common (skewed graphs: long gaps), else the warp tier rates them.
constexpr uint64_t kLaneShortRecord = 65;

// Degrees of a compressed graph from its headers (a lane reads its own, the
// next one's comes from the next lane), the number of lane-tier candidates
// (degree <= lane_max) and how many of them have long records.
__global__ void __launch_bounds__(256) k_zip_degrees(GView g, int32_t lane_max, int64_t *deg,
                                                     unsigned long long *cnt) {
  __shared__ uint32_t sa[8], sl[8];
  const int lane = lane_id();
  uint32_t a = 0, l = 0;
  for (int64_t u0 = (int64_t)blockIdx.x * blockDim.x; u0 < g.n;
       u0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = u0 + threadIdx.x;
    const bool in = u < g.n;
    uint64_t first = 0, rb = 0;
    if (u <= g.n) {
      rb = off_at(g, u);
      read_varint(g.bytes + rb, first);
    }
    uint64_t next = __shfl_down_sync(kFull, first, 1), re = __shfl_down_sync(kFull, rb, 1);
    if (!in) continue;  // (a whole warp, or lanes behind every shuffle source)
    if (lane == 31) {
      re = off_at(g, u + 1);
      read_varint(g.bytes + re, next);
    }
    const int64_t d = (int64_t)(next - first);
    deg[u] = d;
    if (d <= lane_max) ++a, l += re - rb > kLaneShortRecord;
  }
  a = __reduce_add_sync(kFull, a);
  l = __reduce_add_sync(kFull, l);
  if (lane == 0) sa[threadIdx.x >> 5] = a, sl[threadIdx.x >> 5] = l;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) a += sa[w], l += sl[w];
    if (a) atomicAdd(&cnt[0], (unsigned long long)a);
    if (l) atomicAdd(&cnt[1], (unsigned long long)l);
  }
}

// Tier lists: class 0 is the lane tier (no list), 1..8 the lists of TierCache
// in its order. Block b owns kTierSpan vertices and counts its vertices per
// class (cnt[class * nblocks + b]; an exclusive scan of the counts of classes
// 1..8 gives every block its place in one array of all lists) and adds up
// entries and vertices per tier. One pass and one scan for all lists; a flag
// array, a scan, a readback and a compaction per list took 30 launches and ten
// synchronisations.
constexpr int kTierSpan = 2048;
constexpr int kTierLists = 8;

__device__ __forceinline__ int64_t deg_of(const int64_t *xadj, const int64_t *deg, int64_t u) {
  return deg ? deg[u] : xadj[u + 1] - xadj[u];
}

__global__ void __launch_bounds__(256)
    k_classify(const int64_t *xadj, const int64_t *deg, int64_t n, int32_t lane_max,
               int32_t small_max, int32_t mid_max, const uint32_t *off32, const uint64_t *off64,
               bool long_records, uint8_t *tier, uint8_t *cls, int64_t *cnt,
               unsigned long long *stats) {
  __shared__ int32_t count[kTierLists + 1];
  __shared__ unsigned long long st[10];
  if (threadIdx.x <= kTierLists) count[threadIdx.x] = 0;
  if (threadIdx.x < 10) st[threadIdx.x] = 0;
  __syncthreads();
  int64_t e[5] = {0, 0, 0, 0, 0};
  int32_t c[5] = {0, 0, 0, 0, 0};
  const int64_t lo = (int64_t)blockIdx.x * kTierSpan;
  for (int64_t u = lo + threadIdx.x; u < min(lo + kTierSpan, n); u += 256) {
    const int64_t d = deg_of(xadj, deg, u);
    bool lane = lane_max > 0 && d <= lane_max;
    if (lane && !long_records && (off32 || off64)) {
      const uint64_t len = off32 ? (uint64_t)(off32[u + 1] - off32[u]) : off64[u + 1] - off64[u];
      lane = len <= kLaneShortRecord;
    }
    const uint8_t t = lane ? TIER_LANE
                      : d <= small_max ? TIER_SMALL
                      : d <= mid_max ? TIER_MID
                      : d <= kChunkThreshold ? TIER_BIG
                                     : TIER_HUGE;
    const uint8_t k = t == TIER_LANE    ? 0
                      : t == TIER_SMALL ? 1
                      : t == TIER_MID   ? (d <= kMidSplit ? 2 : 3)
                      : t == TIER_HUGE  ? 8
                      : d <= kBigTinySplit ? 4
                      : d <= kBigMidSplit  ? 5
                      : d <= kBigSplit     ? 6
                                           : 7;
    tier[u] = t;
    cls[u] = k;
    if (k) atomicAdd(&count[k], 1);
#pragma unroll
    for (int i = 0; i < 5; ++i)
      if (i == t) e[i] += d, ++c[i];
  }
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const int32_t w = warp_sum(c[i]);
    if (w == 0) continue;
    const int64_t v = warp_sum(e[i]);
    if (lane_id() == 0) atomicAdd(&st[i], (unsigned long long)v), atomicAdd(&st[5 + i], (unsigned long long)w);
  }
  __syncthreads();
  if (threadIdx.x < kTierLists)
    cnt[(int64_t)threadIdx.x * gridDim.x + blockIdx.x] = count[threadIdx.x + 1];
  if (threadIdx.x < 10 && st[threadIdx.x]) atomicAdd(&stats[threadIdx.x], st[threadIdx.x]);
}

// The lists' lengths behind the per-tier figures: off holds the scanned counts.
__global__ void k_tier_sizes(const int64_t *off, int64_t nblocks, unsigned long long *out) {
  const int k = threadIdx.x;
  if (k < kTierLists) out[k] = (unsigned long long)(off[(k + 1) * nblocks] - off[k * nblocks]);
}

__global__ void __launch_bounds__(256) k_tier_lists(const uint8_t *cls, int64_t n,
                                                    const int64_t *off, int32_t *lists) {
  __shared__ int64_t place[kTierLists];
  __shared__ int32_t used[kTierLists];
  if (threadIdx.x < kTierLists) {
    place[threadIdx.x] = off[(int64_t)threadIdx.x * gridDim.x + blockIdx.x];
    used[threadIdx.x] = 0;
  }
  __syncthreads();
  const int64_t lo = (int64_t)blockIdx.x * kTierSpan;
  for (int64_t u = lo + threadIdx.x; u < min(lo + kTierSpan, n); u += 256) {
    const int k = cls[u];
    if (k) lists[place[k - 1] + atomicAdd(&used[k - 1], 1)] = (int32_t)u;
  }
}

// Table capacity per listed vertex: the smallest power of two >= 2*deg.
__global__ void k_table_caps(const int32_t *list, int64_t cnt, const int64_t *xadj,
                             const int64_t *deg, int64_t *slots, int32_t *logcap, int64_t *chunks) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
       i += (int64_t)gridDim.x * blockDim.x) {
    int64_t d = deg_of(xadj, deg, list[i]);
    int lc = 1;
    while (((int64_t)1 << lc) < 2 * d) ++lc;
    logcap[i] = lc;
    slots[i] = (int64_t)1 << lc;
    chunks[i] = (d + kChunkSize - 1) / kChunkSize;
  }
}

// Segments per huge table (tables above kSegLog slots are cut into segments).
__global__ void k_table_segs(const int32_t *logcap, int64_t cnt, int64_t *segs) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
       i += (int64_t)gridDim.x * blockDim.x)
    segs[i] = logcap[i] - 1 > kSegLog ? (int64_t)1 << (logcap[i] - 1 - kSegLog) : 1;  // list = half
}

__global__ void k_fill_table(int32_t *keys, int64_t *vals, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    keys[i] = -1;
    vals[i] = 0;
  }
}

}  // namespace

void build_tiers(tp_graph *g, const tp_params &p, cudaStream_t s) {
  TierCache &T = g->tiers;
  // the lane tier rates with one lane per vertex and needs unit edge weights
  const bool lane_ok = g->unit_ew || g->max_ew < kLaneMaxEdgeWeight;
  int32_t lane_max = lane_ok ? std::max(0, std::min(p.tier_lane, kLaneMaxDeg)) : 0;
  int32_t small_max = std::max(lane_max, std::min(p.tier_small, 64));
  int32_t mid_max = std::max(small_max, std::min(p.tier_mid, 512));  // tables of 1024 slots
  if (T.built && T.small_max == small_max && T.mid_max == mid_max && T.lane_max == lane_max) return;
  // the old cache is freed on this call's stream: the stream it was built on
  // may be gone (calls on one graph are ordered by the caller)
  T.rehome(s);
  T = TierCache();
  T.lane_max = lane_max;
  T.small_max = small_max;
  T.mid_max = mid_max;
  int64_t n = g->n;
  T.tier.alloc(n, s);
  if (n == 0) {
    T.built = true;
    return;
  }
  Buf<int64_t> deg;
  const int64_t *xadj = g->compressed ? nullptr : g->xadj.get();
  Buf<unsigned long long> te(10 + kTierLists, s);
  TP_CUDA(cudaMemsetAsync(te.get(), 0, te.n * sizeof(unsigned long long), s));
  const uint32_t *o32 = g->compressed && !g->off_is64 ? g->off32.get() : nullptr;
  const uint64_t *o64 = g->compressed && g->off_is64 ? g->off64.get() : nullptr;
  bool long_records = false;
  if (g->compressed) {  // long lane records where more than 5% are long
    deg.alloc(n, s);
    launch(k_zip_degrees, grid_for(n, 256, (int64_t)num_sms() * 8), 256, 0, s, view(g), lane_max,
           deg.get(), te.get());
    TP_LAUNCH_CHECK();
    if (lane_max > 0) {
      unsigned long long lc[2];
      TP_CUDA(cudaMemcpyAsync(lc, te.get(), sizeof(lc), cudaMemcpyDeviceToHost, s));
      TP_CUDA(cudaStreamSynchronize(s));
      long_records = lc[1] * 20 > lc[0];
      T.lane_long = long_records;
    }
    TP_CUDA(cudaMemsetAsync(te.get(), 0, 2 * sizeof(unsigned long long), s));
  }
  const int64_t nblocks = (n + kTierSpan - 1) / kTierSpan;
  Buf<int64_t> off(kTierLists * nblocks + 1, s);
  Buf<uint8_t> cls(n, s);
  launch(k_classify, (unsigned)nblocks, 256, 0, s, xadj, deg.get(), n, lane_max, small_max, mid_max, o32,
         o64, long_records, T.tier.get(), cls.get(), off.get(), te.get());
  TP_LAUNCH_CHECK();
  exclusive_scan_i64(off.get(), off.get(), kTierLists * nblocks, s);
  launch(k_tier_sizes, 1, 32, 0, s, off.get(), nblocks, te.get() + 10);
  TP_LAUNCH_CHECK();
  unsigned long long hte[10 + kTierLists];
  TP_CUDA(cudaMemcpyAsync(hte, te.get(), sizeof(hte), cudaMemcpyDeviceToHost, s));
  TP_CUDA(cudaStreamSynchronize(s));
  for (int t = 0; t < 5; ++t) T.edges[t] = (int64_t)hte[t], T.count[t] = (int64_t)hte[5 + t];
  {
    int64_t *const len[kTierLists] = {&T.n_small, &T.n_mid, &T.n_mid2, &T.n_big0,
                                      &T.n_big1,  &T.n_big, &T.n_big2, &T.n_huge};
    TierList *const list[kTierLists] = {&T.small, &T.mid, &T.mid2, &T.big0,
                                        &T.big1,  &T.big, &T.big2, &T.huge};
    int64_t total = 0;
    for (int k = 0; k < kTierLists; ++k) total += *len[k] = (int64_t)hte[10 + k];
    T.lists.alloc(total, s);
    if (total) {
      launch(k_tier_lists, (unsigned)nblocks, 256, 0, s, cls.get(), n, off.get(), T.lists.get());
      TP_LAUNCH_CHECK();
    }
    int32_t *at = T.lists.get();
    for (int k = 0; k < kTierLists; ++k) list[k]->p = at, at += *len[k];
  }
  // global rating tables for the huge tier (the big tier rates in shared memory)
  T.huge_toff.alloc(T.n_huge + 1, s);
  T.huge_tcap.alloc(std::max<int64_t>(T.n_huge, 1), s);
  if (T.n_huge) {
    T.huge_chunk_start.alloc(T.n_huge + 1, s);
    Buf<int64_t> ch(T.n_huge, s);
    launch(k_table_caps, grid_for(T.n_huge, 256), 256, 0, s, T.huge.get(), T.n_huge, xadj, deg.get(),
           T.huge_toff.get(), T.huge_tcap.get(), ch.get());
    TP_LAUNCH_CHECK();
    exclusive_scan_i64(T.huge_toff.get(), T.huge_toff.get(), T.n_huge, s);
    exclusive_scan_i64(ch.get(), T.huge_chunk_start.get(), T.n_huge, s);
    TP_CUDA(cudaMemcpyAsync(&T.huge_slots, T.huge_toff.get() + T.n_huge, 8, cudaMemcpyDeviceToHost, s));
    TP_CUDA(cudaMemcpyAsync(&T.n_huge_chunks, T.huge_chunk_start.get() + T.n_huge, 8,
                            cudaMemcpyDeviceToHost, s));
    TP_CUDA(cudaStreamSynchronize(s));
  }
  if (T.n_huge) {
    T.huge_seg_start.alloc(T.n_huge + 1, s);
    launch(k_table_segs, grid_for(T.n_huge, 256), 256, 0, s, T.huge_tcap.get(), T.n_huge,
           T.huge_seg_start.get());
    TP_LAUNCH_CHECK();
    exclusive_scan_i64(T.huge_seg_start.get(), T.huge_seg_start.get(), T.n_huge, s);
    T.n_huge_segs = read_scalar(T.huge_seg_start.get() + T.n_huge, s);
    T.huge_seg_best.alloc((size_t)T.n_huge_segs * kSegBestBytes, s);
  }
  if (T.huge_slots) {
    T.tcount.alloc(std::max<int64_t>(T.n_huge, 1), s);
    TP_CUDA(cudaMemsetAsync(T.tcount.get(), 0, sizeof(int32_t) * std::max<int64_t>(T.n_huge, 1), s));
  }
  T.built = true;
}

// The hubs' global rating tables (2 to 4 slots of 14 bytes per hub
// neighbour) exist only while a rating call needs them: allocated empty on
// first use, left empty by every rating launch, freed when the call ends.
void ensure_hub_tables(tp_graph *g, cudaStream_t s) {
  TierCache &T = g->tiers;
  const int64_t total = T.huge_slots;
  if (!total || T.tkeys.get()) return;
  T.tkeys.alloc(total, s);
  T.tvals.alloc(total, s);
  T.tlist.alloc(total / 2 + 1, s);
  launch(k_fill_table, grid_for(total, 256), 256, 0, s, T.tkeys.get(), T.tvals.get(), total);
  TP_LAUNCH_CHECK();
}

void release_hub_tables(tp_graph *g, cudaStream_t s) {
  TierCache &T = g->tiers;
  T.tkeys.s = T.tvals.s = T.tlist.s = s;
  T.tkeys.release();
  T.tvals.release();
  T.tlist.release();
}

// ---------------------------------------------------------------- compression
namespace {

__device__ __forceinline__ int vlen(uint64_t x) {
  const int bits = 64 - __clzll((long long)(x | 1));
  return (bits + 6) / 7;
}
__device__ __forceinline__ int vlen32(uint32_t x) { return (38 - __clz(x | 1)) / 7; }

__device__ __forceinline__ uint32_t first_code(int32_t v, int32_t u) {
  return v >= u ? 2u * (uint32_t)(v - u) : 2u * (uint32_t)(u - v) + 1u;
}

// Stores the n-byte VarInt of x (n = vlen32(x)) at p.
__device__ __forceinline__ void put_varint(uint8_t *p, uint32_t x, int n) {
  p[0] = (uint8_t)(n > 1 ? x | 0x80u : x);
  if (n > 1) p[1] = (uint8_t)(n > 2 ? x >> 7 | 0x80u : x >> 7);
  if (n > 2) {
    p[2] = (uint8_t)(n > 3 ? x >> 14 | 0x80u : x >> 14);
    if (n > 3) p[3] = (uint8_t)(n > 4 ? x >> 21 | 0x80u : x >> 21);
    if (n > 4) p[4] = (uint8_t)(x >> 28);
  }
}
__device__ __forceinline__ void put_varint64(uint8_t *p, uint64_t x) {
  for (; x >= 128; x >>= 7) *p++ = (uint8_t)(0x80u | (x & 0x7fu));
  *p = (uint8_t)x;
}

// Encoding in tiles of adjacency entries. The bytes of a tile are those of its
// entries and of the headers (and chunk tables) of the rows that start in it,
// an unbroken piece of the stream, so their number per tile, summed over the
// tiles, gives every tile its place. A row's first edge id is the number of
// the entry it starts at, so headers need nothing but the mark of the start:
// start[i] is the row with entries that starts at entry i of the tile
// (relative to base, 0: none), empty[i] the number of empty rows just before
// it, whose headers hold the same number (k_zip_empty writes them). Pass 2
// puts a tile together in shared memory, eight entries a thread, and writes it
// in 16-byte pieces. Bound by instruction issue; the adjacency is read twice
// and the stream written once.
// Pass 1 (WRITE = false): bytes per tile. Pass 2: bytes, offsets, and the
// position of every chunk start (cpos[e / kChunkSize]: they lie at least
// kChunkSize apart). HUBS: some rows are chunked.
// First row of [0, hi] that starts at entry b (row hi does).
__device__ __forceinline__ int64_t first_row_at(const int64_t *xadj, int64_t hi, int64_t b) {
  int64_t lo = 0;
  while (lo < hi) {
    const int64_t mid = (lo + hi) / 2;
    if (xadj[mid] < b) lo = mid + 1;
    else hi = mid;
  }
  return hi;
}

constexpr int kZipStage = 12 * 1024;
template <bool WRITE, bool HUBS>
__global__ void __launch_bounds__(kTileThreads)
    k_zip_tiles(GView g, const int32_t *tile_first, int64_t ntiles, int64_t *tsize, uint8_t *out,
                uint32_t *o32, uint64_t *o64, int64_t *cpos) {
  __shared__ int32_t start[kTile + kTile / 32], empty[kTile];
  __shared__ int32_t val[kTile + kTile / 32];
  __shared__ int64_t wsum[kTileThreads / 32];
  __shared__ int32_t wrow[kTileThreads / 32];
  __shared__ int32_t s_empties;
  __shared__ __align__(16) uint8_t stage[WRITE ? kZipStage : 16];
  const int lane = lane_id(), w = threadIdx.x >> 5;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int64_t e0 = t * kTile;
    const int len = (int)min((int64_t)kTile, g.m2 - e0);
    for (int i = threadIdx.x; i < kTile; i += kTileThreads) {
      if (i < len) val[tpad(i)] = g.adj[e0 + i];
      start[tpad(i)] = 0;
    }
    if (threadIdx.x == 0) s_empties = 0;
    __syncthreads();
    const int32_t base = tile_first[t] - 1;
    const int64_t rend = min((int64_t)tile_first[t + 1], g.n);
    auto mark = [&](int64_t r, int64_t b) {  // row r with entries, from entry b on
      const int i = (int)(b - e0);
      start[tpad(i)] = (int32_t)(r - base);
      const bool after = r > 0 && g.xadj[r - 1] == b;
      empty[i] = after ? (int32_t)(r - first_row_at(g.xadj, r, b)) : 0;
      if (after) s_empties = 1;
    };
    if (many_rows(tile_first, t)) {  // uniform over the block
#pragma unroll 1
      for (int i = threadIdx.x; i < len; i += kTileThreads) {
        const int64_t r = row_of_entry(g.xadj, max(base, 0), rend - 1, e0 + i);
        if (g.xadj[r] == e0 + i) mark(r, e0 + i);
      }
    } else {
      for (int64_t r = (int64_t)base + 1 + threadIdx.x; r < rend; r += kTileThreads) {
        const int64_t b = g.xadj[r];
        if (g.xadj[r + 1] != b) mark(r, b);
      }
    }
    __syncthreads();
    const bool empties = s_empties != 0;
    // codes of eight consecutive entries, and the bytes before each
    const int i0 = threadIdx.x * kTileItems;
    uint32_t code[kTileItems];
    int64_t bytes = 0;
    int32_t chunks = 0;  // HUBS: bit j: entry j begins a later chunk of its row
    int32_t prev = i0 && i0 < len ? val[tpad(i0 - 1)] : (i0 == 0 && e0 ? g.adj[e0 - 1] : 0);
    int32_t u = base;  // HUBS: row of the current entry
    int64_t ub = 0, ud = 0;
    if constexpr (HUBS) {  // the last row that starts before this thread's entries
      int32_t m = 0;
#pragma unroll
      for (int j = 0; j < kTileItems; ++j) m = max(m, start[tpad(i0 + j)]);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(kFull, m, o);
        if (lane >= o) m = max(m, y);
      }
      if (lane == 31) wrow[w] = m;
      __syncthreads();
      m = __shfl_up_sync(kFull, m, 1);
      if (lane == 0) m = 0;
      for (int q = 0; q < w; ++q) m = max(m, wrow[q]);
      u = base + m;
      if (i0 < len && u >= 0) ub = g.xadj[u], ud = g.xadj[u + 1] - ub;
    }
#pragma unroll
    for (int j = 0; j < kTileItems; ++j) {
      const int i = i0 + j;
      code[j] = 0;
      if (i >= len) continue;
      const int32_t v = val[tpad(i)], st = start[tpad(i)];
      bool first = st != 0;
      if (first) bytes += (int64_t)(1 + (empties ? empty[i] : 0)) * vlen((uint64_t)(e0 + i));
      if constexpr (HUBS) {
        if (first) u = base + st, ub = e0 + i, ud = g.xadj[u + 1] - ub;
        if (ud > kChunkThreshold) {
          const int64_t rel = e0 + i - ub;
          if (rel == 0) bytes += 4 * ((ud + kChunkSize - 1) / kChunkSize - 1);
          else if (rel % kChunkSize == 0) first = true, chunks |= 1 << j;
        }
        code[j] = first ? first_code(v, u) : (uint32_t)(v - prev);
      } else {
        code[j] = first ? first_code(v, base + st) : (uint32_t)(v - prev);
      }
      prev = v;
      bytes += vlen32(code[j]);
    }
    const int64_t incl = warp_incl_scan(bytes);
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    int64_t before = 0, total = 0;
    for (int q = 0; q < kTileThreads / 32; ++q) {
      before += q < w ? wsum[q] : 0;
      total += wsum[q];
    }
    if (!WRITE) {
      if (threadIdx.x == 0) {
        // the last tile also holds the headers of the empty rows at the end
        const int64_t tail = t == ntiles - 1 ? g.n - first_row_at(g.xadj, g.n, g.m2) : 0;
        tsize[t] = total + tail * vlen((uint64_t)g.m2);
      }
      __syncthreads();
      continue;
    }
    const int64_t begin = tsize[t];
    const int shift = (int)(begin & 15);
    const bool staged = total + shift <= kZipStage;
    auto write = [&](uint8_t *buf) {  // buf: where the tile's first byte goes
      int64_t at = before + incl - bytes;
#pragma unroll
      for (int j = 0; j < kTileItems; ++j) {
        const int i = i0 + j;
        if (i >= len) continue;
        const int64_t e = e0 + i;
        const int32_t st = start[tpad(i)];
        if (st) {  // room for the empty rows' headers, then the row's own
          const int hl = vlen((uint64_t)e);
          if (empties) at += (int64_t)empty[i] * hl;
          if (o32) o32[base + st] = (uint32_t)(begin + at);
          else o64[base + st] = (uint64_t)(begin + at);
          put_varint64(buf + at, (uint64_t)e);
          at += hl;
          if constexpr (HUBS) {  // and for the chunk table (k_zip_tables)
            const int64_t d = g.xadj[base + st + 1] - e;
            if (d > kChunkThreshold) at += 4 * ((d + kChunkSize - 1) / kChunkSize - 1);
          }
        }
        const int n = vlen32(code[j]);
        if (HUBS && (chunks >> j & 1)) cpos[e / kChunkSize] = begin + at;
        put_varint(buf + at, code[j], n);
        at += n;
      }
    };
    if (staged) write(stage + shift);
    else write(out + begin);
    __syncthreads();
    if (staged) {  // whole 16-byte pieces, the ragged ends byte by byte
      uint8_t *dst = out + (begin - shift);
      const uint8_t *src = stage;
      const int n = (int)total + shift;
      for (int p = 16 * threadIdx.x; p < n; p += 16 * kTileThreads) {
        if (p >= shift && p + 16 <= n) {
          *reinterpret_cast<uint4 *>(dst + p) = *reinterpret_cast<const uint4 *>(src + p);
        } else {
          for (int q = max(p, shift); q < min(p + 16, n); ++q) dst[q] = src[q];
        }
      }
    }
    __syncthreads();
  }
}

// Headers and offsets of the empty rows, and the end: row n's offset, the
// terminal header (2m) and the zero bytes behind the stream. An
// empty row's header lies (w - u) headers before that of the next row w with
// entries, or before the end of the stream, and holds the same number.
__global__ void k_zip_empty(const int64_t *xadj, int64_t n, int64_t m2, int64_t body, bool empties,
                            uint8_t *out, uint32_t *o32, uint64_t *o64) {
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0) {
      if (o32) o32[n] = (uint32_t)body;
      else o64[n] = (uint64_t)body;
      put_varint64(out + body, (uint64_t)m2);
    }
    if (threadIdx.x < kBytePad) out[body + vlen((uint64_t)m2) + threadIdx.x] = 0;
  }
  if (!empties) return;
  const int lane = lane_id();
  constexpr int64_t kSpan = 256;  // consecutive rows of a warp, 32 at a time
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t s0 = gw * kSpan; s0 < n; s0 += nw * kSpan) {
    int64_t run = -1, run_end = 0;  // the last search: the run that starts at entry run ends in row run_end
    for (int64_t u0 = s0; u0 < min(s0 + kSpan, n); u0 += 32) {
      const int64_t u = min(u0 + lane, n - 1);
      const int64_t b = xadj[u], next = xadj[u + 1];
      // The last row that starts at entry b: where the starts go up among these
      // 32 rows, or, for empty rows whose run leaves them, found by the warp
      // together, 32 probes a step, once per run (a search of its own for every
      // row made 2^26 rows without entries take 0.25 s to compress, now 0.6 ms).
      const unsigned up = __ballot_sync(kFull, next != b) >> lane;
      int64_t lo = u0 + lane + __ffs(up) - 1;
      if (__any_sync(kFull, up == 0)) {
        const int64_t bl = __shfl_sync(kFull, b, 31);
        if (bl != run) {
          int64_t l = min(u0 + 32, n), h = n;
          while (l < h) {
            const int64_t step = (h - l + 31) / 32;
            const int64_t p = min(l + step * (lane + 1), h);
            const int in = __popc(__ballot_sync(kFull, xadj[p] <= bl));
            const int64_t nl = in ? min(l + step * in, h) : l;
            h = in == 32 ? nl : min(l + step * (in + 1), h) - 1;
            l = nl;
          }
          run = bl;
          run_end = l;
        }
        if (up == 0) lo = run_end;
      }
      if (u0 + lane >= n || next != b) continue;
      const int hl = vlen((uint64_t)b);
      const int64_t end = lo == n ? body : (o32 ? (int64_t)o32[lo] : (int64_t)o64[lo]);
      const int64_t off = end - (lo - u) * hl;
      if (o32) o32[u] = (uint32_t)off;
      else o64[u] = (uint64_t)off;
      put_varint64(out + off, (uint64_t)b);
    }
  }
}

// Chunk tables of the rows above kChunkThreshold: a warp per 32 rows, all of
// it on each chunked one.
__global__ void k_zip_tables(const int64_t *xadj, int64_t n, const uint32_t *o32,
                             const uint64_t *o64, const int64_t *cpos, uint8_t *out) {
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int lane = lane_id();
  for (int64_t base = gw * 32; base < n; base += nw * 32) {
    const int64_t u = base + lane;
    unsigned hubs = __ballot_sync(kFull, u < n && xadj[u + 1] - xadj[u] > kChunkThreshold);
    while (hubs) {
      const int64_t h = base + __ffs(hubs) - 1;
      hubs &= hubs - 1;
      const int64_t b = xadj[h], nch = (xadj[h + 1] - b + kChunkSize - 1) / kChunkSize;
      const int64_t off = o32 ? (int64_t)o32[h] : (int64_t)o64[h];
      for (int64_t k = 1 + lane; k < nch; k += 32) {
        const uint32_t rel = (uint32_t)(cpos[(b + k * kChunkSize) / kChunkSize] - off);
        uint8_t *t = out + off + vlen((uint64_t)b) + 4 * (k - 1);
        for (int q = 0; q < 4; ++q) t[q] = (uint8_t)(rel >> (8 * q));
      }
    }
  }
}

__global__ void k_off_narrow_u64(const uint64_t *off, int64_t cnt, uint32_t *o32) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
       i += (int64_t)gridDim.x * blockDim.x)
    o32[i] = (uint32_t)off[i];
}

// First edge ids of all rows: the headers (entry n: the terminal header).
__global__ void k_zip_first(GView g, int64_t *xadj) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u <= g.n;
       u += (int64_t)gridDim.x * blockDim.x) {
    uint64_t a;
    read_varint(g.bytes + off_at(g, u), a);
    xadj[u] = (int64_t)a;
  }
}

__global__ void k_zip_header_check(GView g, const int64_t *xadj, int32_t *bad) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < g.n;
       u += (int64_t)gridDim.x * blockDim.x)
    if (off_at(g, u + 1) < off_at(g, u) || (uint64_t)xadj[u + 1] < (uint64_t)xadj[u] ||
        (u == 0 && xadj[0] != 0))
      atomicCAS(bad, 0, 1);
}

// Decoding into CSR. A warp takes 32 consecutive records; every lane decodes
// its own, a word of the stream at a time, into a piece of shared memory where
// the warp's neighbours lie as they will in the adjacency, and the warp copies
// the piece out coalesced. (A warp per record used 30 of the 128 bytes of its
// window and left most lanes idle: 3.15 ms for a mesh of 3 M vertices, where
// this takes 0.20.) Records of more than kUnzipLane neighbours are listed, a
// chunk per item, for k_unzip_items. Every rule of the format is checked:
// VarInts of at most five bytes, gaps of at least one, ids inside the graph,
// the record's bytes used up exactly.
constexpr int kUnzipLane = 128;    // most neighbours of a lane's record
constexpr int kUnzipWarps = 8;
constexpr int kUnzipPiece = 1024;  // neighbours of a warp's piece

__global__ void __launch_bounds__(32 * kUnzipWarps)
    k_unzip_lane(GView g, const int64_t *xadj, int32_t *adj, uint64_t *items,
                 unsigned long long *n_items) {
  __shared__ int32_t piece_all[kUnzipWarps][kUnzipPiece];
  int32_t *piece = piece_all[threadIdx.x >> 5];
  const int lane = lane_id();
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t base = gw * 32; base < g.n; base += nw * 32) {
    const int64_t u = base + lane;
    const bool in = u < g.n;
    const int64_t pos = in ? xadj[u] : 0;
    const int64_t deg = in ? xadj[u + 1] - pos : 0;
    const bool mine = deg > 0 && deg <= kUnzipLane;
    if (deg > kUnzipLane) {
      const int64_t nch = deg > kChunkThreshold ? (deg + kChunkSize - 1) / kChunkSize : 1;
      const unsigned long long at = atomicAdd(n_items, (unsigned long long)nch);
      for (int64_t j = 0; j < nch; ++j) items[at + j] = (uint64_t)u << 32 | (uint64_t)j;
    }
    // the lanes' neighbours side by side in the piece; a warp whose records
    // do not fit writes straight to the adjacency
    const int32_t cnt = mine ? (int32_t)deg : 0;
    const int32_t incl = warp_incl_scan(cnt);
    const int32_t total = __shfl_sync(kFull, incl, 31);
    const bool staged = total <= kUnzipPiece;
    bool bad = false;
    if (mine) {
      int32_t *dst = staged ? piece + (incl - cnt) : adj + pos;
      const uint64_t b = off_at(g, u), e = off_at(g, u + 1);
      uint64_t skip;
      const int hl = read_varint(g.bytes + b, skip);
      int64_t left = (int64_t)(e - b) - hl;  // bytes of the codes
      const uint64_t p = b + (uint64_t)hl;
      const uint32_t *wp = reinterpret_cast<const uint32_t *>(g.bytes + (p & ~(uint64_t)3));
      uint32_t word = 0;
      int have = 0;     // bytes of word not yet taken
      bad = left < 0;   // the header runs over the record's end
      if (left > 0) {
        word = __ldg(wp) >> (8 * (p & 3));
        have = 4 - (int)(p & 3);
      }
      int64_t id = u;
      int32_t k = 0;
      while (k < cnt && !bad) {
        uint32_t v = 0;
        int n = 0;
        for (;;) {  // one VarInt
          if (left == 0 || n == 5) {
            bad = true;
            break;
          }
          if (have == 0) word = __ldg(++wp), have = 4;
          const uint32_t by = word & 255u;
          word >>= 8;
          --have, --left;
          v |= (by & 0x7fu) << (7 * n++);
          if (!(by & 0x80u)) break;
        }
        if (k == 0) id = (v & 1u) ? id - (int64_t)(v >> 1) : id + (int64_t)(v >> 1);
        else id += v, bad |= v == 0;
        bad |= id < 0 || id >= g.n;
        dst[k++] = (int32_t)id;
      }
      bad |= left != 0;
    }
    if (__any_sync(kFull, bad) && lane == 0) latch_error(g.err, TP_ERR_CORRUPT);
    __syncwarp();
    if (staged) {
      // rows of the piece are contiguous in the adjacency except across the
      // listed ones, so each entry finds its row by its lane's range
      const int64_t shift = pos - (incl - cnt);  // adjacency position minus piece position
      const unsigned gaps = __ballot_sync(kFull, deg > kUnzipLane);
      if (!gaps) {
        const int64_t s0 = __shfl_sync(kFull, shift, 0);
        for (int i = lane; i < total; i += 32) adj[s0 + i] = piece[i];
      } else {
        for (int l = 0; l < 32; ++l) {
          const int32_t c = __shfl_sync(kFull, cnt, l), x = __shfl_sync(kFull, incl, l) - c;
          const int64_t sl = __shfl_sync(kFull, shift, l);
          for (int i = x + lane; i < x + c; i += 32) adj[sl + i] = piece[i];
        }
      }
      __syncwarp();
    }
  }
}

// The listed records, a warp per chunk.
__global__ void k_unzip_items(GView g, const int64_t *xadj, int32_t *adj, const uint64_t *items,
                              const unsigned long long *n_items) {
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t n = (int64_t)*n_items;
  for (int64_t k = gw; k < n; k += nw) {
    const int64_t u = (int64_t)(items[k] >> 32), j = (int64_t)(items[k] & 0xffffffffu);
    const ZipNbr z = zip_nbr(g, u);
    uint64_t cb = 0, ce = 0;
    int64_t cnt = 0;
    bool ok = z.data <= z.end;  // the chunk table lies inside the record
    if (ok) {
      zip_chunk(g, z, j, cb, ce, cnt);
      ok = cb >= z.data && cb <= ce && ce <= z.end && (j > 0 || cb == z.data) &&
           (j + 1 < z.nchunks || ce == z.end);
    }
    if (!ok) {
      if (lane_id() == 0) latch_error(g.err, TP_ERR_CORRUPT);
      continue;
    }
    const int64_t at = xadj[u] + j * kChunkSize;
    warp_decode_chunk(g, u, cb, ce, cnt, [&](bool has, int32_t v, int64_t i) {
      if (has && i < cnt) adj[at + i] = v;
    });
  }
}

// Offsets inside the stream and in order; then the entries from the terminal
// header (-1 where the offsets are bad).
__global__ void k_off_check(const uint64_t *off, int64_t n, uint64_t nbytes, int32_t *bad) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u <= n;
       u += (int64_t)gridDim.x * blockDim.x)
    if (off[u] >= nbytes || (u && off[u] < off[u - 1])) atomicCAS(bad, 0, 1);
}

__global__ void k_widen(const uint32_t *a, uint64_t *b, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    b[i] = a[i];
}

__global__ void k_ones(int64_t *p, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    p[i] = 1;
}

}  // namespace

// Total vertex weight, largest degree and largest edge weight. acc holds two
// zeroed words.
static void launch_stats(const tp_graph *g, int64_t *acc, cudaStream_t s) {
  if (!g->n) return;
  launch(k_sum_max, grid_for(g->n, 256, (int64_t)num_sms() * 4), 256, 0, s,
         g->unit_vw ? nullptr : g->vw.get(), g->compressed ? nullptr : g->xadj.get(), g->n, acc);
  TP_LAUNCH_CHECK();
}

static void set_stats(tp_graph *g, const int64_t *h, cudaStream_t s) {
  g->total_vw = h[0];
  if (!g->compressed) g->max_deg = h[1];
  g->max_ew = g->unit_ew ? 1 : max_i64(g->ew.get(), g->m2, s);
}

// Validates CSR arrays on the device and fills the graph's statistics.
// Returns whether they make a valid graph. Synchronises.
static bool validate_csr(tp_graph *g, cudaStream_t s) {
  const int64_t ntiles = g->m2 / kTile + 1;
  Buf<int32_t> tile_first(ntiles + 1, s);
  // [0] weight [1] degree [2] upper minus lower entries [3] bad rows, bad entries (32 bits each)
  Buf<int64_t> acc(4, s);
  TP_CUDA(cudaMemsetAsync(acc.get(), 0, 4 * sizeof(int64_t), s));
  int32_t *bad = reinterpret_cast<int32_t *>(acc.get() + 3);
  launch(k_rows, grid_for(g->n + 1, 256), 256, 0, s, g->xadj.get(), g->unit_vw ? nullptr : g->vw.get(),
         g->n, g->m2, tile_first.get(), bad, nullptr);
  if (g->m2)
    launch(k_validate, grid_for(ntiles, 1, (int64_t)num_sms() * 16), kTileThreads, 0, s, view(g),
           tile_first.get(), ntiles, bad, bad + 1, (unsigned long long *)(acc.get() + 2));
  TP_LAUNCH_CHECK();
  launch_stats(g, acc.get(), s);
  int64_t h[4];
  TP_CUDA(cudaMemcpyAsync(h, acc.get(), sizeof(h), cudaMemcpyDeviceToHost, s));
  TP_CUDA(cudaStreamSynchronize(s));
  if (h[2] != 0 || h[3] != 0) return false;
  set_stats(g, h, s);
  return true;
}

// Offsets are u32 while the byte stream is below 4 GiB, else u64. Setting
// TP_OFFSETS_U64=1 in the environment selects u64 offsets for any stream, so
// that the wide-offset path can be checked on small graphs.
static bool wide_offsets(uint64_t nbytes) {
  if (nbytes >= (1ull << 32)) return true;
  const char *e = getenv("TP_OFFSETS_U64");
  return e && e[0] == '1' && e[1] == 0;
}

tp_graph *compress(const tp_graph *c, cudaStream_t s) {
  TP_REQUIRE(!c->compressed && c->unit_ew && c->unit_vw, TP_ERR_INVALID);
  tp_graph *z = new_graph();
  try {
    z->n = c->n;
    z->m2 = c->m2;
    z->compressed = 1;
    z->max_deg = c->max_deg;
    z->err.alloc(1, s);
    TP_CUDA(cudaMemsetAsync(z->err.get(), 0, sizeof(int32_t), s));
    GView v = view(c);
    int64_t n = c->n;
    const int64_t ntiles = c->m2 / kTile + 1;
    // the tiles' bytes (then their places and the stream's), a flag each of bad
    // rows and empty rows, and the tiles' first rows: one buffer, one copy back
    Buf<int64_t> work(ntiles + 2 + (ntiles + 2) / 2, s), cpos;
    int64_t *tsize = work.get();
    int32_t *flags = reinterpret_cast<int32_t *>(tsize + ntiles + 1), *tile_first = flags + 2;
    TP_CUDA(cudaMemsetAsync(flags, 0, 2 * sizeof(int32_t), s));
    const bool hubs = c->max_deg > kChunkThreshold;
    if (hubs) cpos.alloc(c->m2 / kChunkSize + 1, s);
    launch(k_rows, grid_for(n + 1, 256), 256, 0, s, c->xadj.get(), nullptr, n, c->m2, tile_first, flags,
           flags + 1);
    const unsigned tb = grid_for(ntiles, 1, (int64_t)num_sms() * 16);
    launch(hubs ? k_zip_tiles<false, true> : k_zip_tiles<false, false>, tb, kTileThreads, 0, s, v,
           tile_first, ntiles, tsize, nullptr, nullptr, nullptr, nullptr);
    TP_LAUNCH_CHECK();
    exclusive_scan_i64(tsize, tsize, ntiles, s);
    int64_t h[2];  // the body's bytes, the flags
    TP_CUDA(cudaMemcpyAsync(h, tsize + ntiles, sizeof(h), cudaMemcpyDeviceToHost, s));
    TP_CUDA(cudaStreamSynchronize(s));
    const int64_t body = h[0];
    const bool empties = h[1] >> 32 != 0;
    int tl = 1;
    for (uint64_t x = (uint64_t)c->m2; x >= 128; x >>= 7) ++tl;
    z->nbytes = (uint64_t)body + tl;
    z->bytes.alloc(z->nbytes + kBytePad, s);
    z->off_is64 = wide_offsets(z->nbytes);
    if (z->off_is64) z->off64.alloc(n + 1, s);
    else z->off32.alloc(n + 1, s);
    launch(hubs ? k_zip_tiles<true, true> : k_zip_tiles<true, false>, tb, kTileThreads, 0, s, v,
           tile_first, ntiles, tsize, z->bytes.get(), z->off32.get(), z->off64.get(), cpos.get());
    launch(k_zip_empty, empties ? grid_for((n + 7) / 8, 256) : 1, 256, 0, s, c->xadj.get(), n, c->m2,
           body, empties, z->bytes.get(), z->off32.get(), z->off64.get());
    if (hubs)
      launch(k_zip_tables, grid_for(n, 256), 256, 0, s, c->xadj.get(), n, z->off32.get(),
             z->off64.get(), cpos.get(), z->bytes.get());
    TP_LAUNCH_CHECK();
    z->total_vw = c->total_vw;
    TP_CUDA(cudaStreamSynchronize(s));
  } catch (...) {
    delete z;
    throw;
  }
  return z;
}

tp_graph *decompress(const tp_graph *z, cudaStream_t s) {
  TP_REQUIRE(z->compressed, TP_ERR_INVALID);
  tp_graph *c = new_graph();
  try {
    c->n = z->n;
    c->m2 = z->m2;
    c->err.alloc(1, s);
    TP_CUDA(cudaMemsetAsync(c->err.get(), 0, sizeof(int32_t), s));
    GView v = view(z);
    int64_t n = z->n;
    Buf<int32_t> bad(1, s);
    TP_CUDA(cudaMemsetAsync(bad.get(), 0, sizeof(int32_t), s));
    c->xadj.alloc(n + 1, s);
    launch(k_zip_first, grid_for(n + 1, 256), 256, 0, s, v, c->xadj.get());
    if (n) launch(k_zip_header_check, grid_for(n, 256), 256, 0, s, v, c->xadj.get(), bad.get());
    TP_LAUNCH_CHECK();
    int32_t hbad = 0;
    int64_t m2 = 0;
    TP_CUDA(cudaMemcpyAsync(&hbad, bad.get(), sizeof(hbad), cudaMemcpyDeviceToHost, s));
    TP_CUDA(cudaMemcpyAsync(&m2, c->xadj.get() + n, 8, cudaMemcpyDeviceToHost, s));
    TP_CUDA(cudaStreamSynchronize(s));
    // (without vertices nothing else looks at the terminal header)
    TP_REQUIRE(hbad == 0 && (n == 0 ? z->m2 == 0 : m2 == z->m2), TP_ERR_CORRUPT);
    if (n == 0) {
      m2 = 0;
      TP_CUDA(cudaMemsetAsync(c->xadj.get(), 0, 8, s));
    }
    c->adj.alloc(m2 + kAdjPad, s);
    TP_CUDA(cudaMemsetAsync(c->adj.get() + m2, 0, kAdjPad * sizeof(int32_t), s));
    Buf<int64_t> acc(3, s);  // [0] weight [1] degree [2] listed items
    TP_CUDA(cudaMemsetAsync(acc.get(), 0, 3 * sizeof(int64_t), s));
    // items: a chunk each of the rows above kUnzipLane neighbours
    Buf<uint64_t> items((size_t)(m2 / kUnzipLane + 1), s);
    unsigned long long *n_items = (unsigned long long *)(acc.get() + 2);
    if (n) {
      launch(k_unzip_lane, grid_for(n, 32 * kUnzipWarps), 32 * kUnzipWarps, 0, s, v, c->xadj.get(),
             c->adj.get(), items.get(), n_items);
      launch(k_unzip_items, grid_for((m2 / kUnzipLane + 1) * 32, 256), 256, 0, s, v, c->xadj.get(),
             c->adj.get(), items.get(), n_items);
      TP_LAUNCH_CHECK();
    }
    launch_stats(c, acc.get(), s);
    int32_t e = 0;
    int64_t h[2];
    TP_CUDA(cudaMemcpyAsync(&e, z->err.get(), sizeof(e), cudaMemcpyDeviceToHost, s));
    TP_CUDA(cudaMemcpyAsync(h, acc.get(), sizeof(h), cudaMemcpyDeviceToHost, s));
    TP_CUDA(cudaStreamSynchronize(s));
    if (e) {
      TP_CUDA(cudaMemsetAsync(z->err.get(), 0, sizeof(int32_t), s));
      throw Error{(tp_status)e};
    }
    set_stats(c, h, s);
  } catch (...) {
    delete c;
    throw;
  }
  return c;
}

__global__ void k_terminal_m2(const uint8_t *bytes, const uint64_t *off, int64_t n,
                              const int32_t *bad, int64_t *m2) {
  uint64_t x;
  *m2 = -1;
  if (*bad) return;
  read_varint(bytes + off[n], x);
  *m2 = (int64_t)x;
}

tp_graph *from_compressed(int64_t n, uint64_t nbytes, const uint8_t *bytes, const uint64_t *off,
                          int host, cudaStream_t s) {
  TP_REQUIRE(n >= 0 && n < (int64_t)INT32_MAX && bytes && off && nbytes > 0, TP_ERR_INVALID);
  cudaMemcpyKind kind = host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  tp_graph *z = new_graph();
  try {
    z->n = n;
    z->compressed = 1;
    z->nbytes = nbytes;
    z->err.alloc(1, s);
    TP_CUDA(cudaMemsetAsync(z->err.get(), 0, sizeof(int32_t), s));
    z->bytes.alloc(nbytes + kBytePad, s);
    TP_CUDA(cudaMemsetAsync(z->bytes.get() + nbytes, 0, kBytePad, s));
    TP_CUDA(cudaMemcpyAsync(z->bytes.get(), bytes, nbytes, kind, s));
    Buf<uint64_t> o(n + 1, s);
    TP_CUDA(cudaMemcpyAsync(o.get(), off, (n + 1) * sizeof(uint64_t), kind, s));
    // offsets must lie inside the stream before anything dereferences them
    Buf<int64_t> m2(1, s);
    Buf<int32_t> bad(1, s);
    TP_CUDA(cudaMemsetAsync(bad.get(), 0, sizeof(int32_t), s));
    launch(k_off_check, grid_for(n + 1, 256), 256, 0, s, o.get(), n, nbytes, bad.get());
    launch(k_terminal_m2, 1, 1, 0, s, z->bytes.get(), o.get(), n, bad.get(), m2.get());
    TP_LAUNCH_CHECK();
    z->m2 = read_scalar(m2.get(), s);
    TP_REQUIRE(z->m2 >= 0, TP_ERR_CORRUPT);
    z->off_is64 = wide_offsets(nbytes);
    if (z->off_is64) {
      z->off64 = std::move(o);
    } else {
      z->off32.alloc(n + 1, s);
      launch(k_off_narrow_u64, grid_for(n + 1, 256), 256, 0, s, o.get(), n + 1, z->off32.get());
      TP_LAUNCH_CHECK();
    }
    tp_graph *c = decompress(z, s);  // throws TP_ERR_CORRUPT on a malformed stream
    z->total_vw = n;
    z->max_deg = c->max_deg;
    bool valid = false;
    try {
      valid = validate_csr(c, s);
    } catch (...) {
      delete c;
      throw;
    }
    delete c;
    TP_REQUIRE(valid, TP_ERR_CORRUPT);
  } catch (...) {
    delete z;
    throw;
  }
  return z;
}

tp_graph *from_csr(int64_t n, const int64_t *xadj, const int32_t *adj, const int64_t *vwgt,
                   const int64_t *ewgt, int host, cudaStream_t s) {
  TP_REQUIRE(n >= 0 && n < (int64_t)INT32_MAX && xadj != nullptr, TP_ERR_INVALID);
  tp_graph *g = new_graph();
  try {
    cudaMemcpyKind kind = host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
    g->n = n;
    g->err.alloc(1, s);
    TP_CUDA(cudaMemsetAsync(g->err.get(), 0, sizeof(int32_t), s));
    g->xadj.alloc(n + 1, s);
    TP_CUDA(cudaMemcpyAsync(g->xadj.get(), xadj, (n + 1) * sizeof(int64_t), kind, s));
    int64_t m2 = host ? xadj[n] : read_scalar(g->xadj.get() + n, s);
    TP_REQUIRE(m2 >= 0, TP_ERR_INVALID);
    g->m2 = m2;
    TP_REQUIRE(m2 == 0 || adj != nullptr, TP_ERR_INVALID);
    g->adj.alloc(m2 + kAdjPad, s);  // padded: 16-byte loads may run past the last entry
    TP_CUDA(cudaMemsetAsync(g->adj.get() + m2, 0, kAdjPad * sizeof(int32_t), s));
    if (m2) TP_CUDA(cudaMemcpyAsync(g->adj.get(), adj, m2 * sizeof(int32_t), kind, s));
    g->unit_vw = vwgt == nullptr;
    g->unit_ew = ewgt == nullptr;
    if (vwgt) {
      g->vw.alloc(n, s);
      if (n) TP_CUDA(cudaMemcpyAsync(g->vw.get(), vwgt, n * sizeof(int64_t), kind, s));
    }
    if (ewgt) {
      g->ew.alloc(m2, s);
      if (m2) TP_CUDA(cudaMemcpyAsync(g->ew.get(), ewgt, m2 * sizeof(int64_t), kind, s));
    }
    TP_REQUIRE(validate_csr(g, s), TP_ERR_INVALID);
  } catch (...) {
    delete g;
    throw;
  }
  return g;
}

void export_csr(const tp_graph *g, int64_t *xadj, int32_t *adj, int64_t *vw, int64_t *ew,
                cudaStream_t s) {
  TP_REQUIRE(!g->compressed, TP_ERR_INVALID);
  if (xadj) TP_CUDA(cudaMemcpyAsync(xadj, g->xadj.get(), (g->n + 1) * 8, cudaMemcpyDeviceToDevice, s));
  if (adj && g->m2) TP_CUDA(cudaMemcpyAsync(adj, g->adj.get(), g->m2 * 4, cudaMemcpyDeviceToDevice, s));
  if (vw && g->n) {
    if (g->unit_vw) launch(k_ones, grid_for(g->n, 256), 256, 0, s, vw, g->n);
    else TP_CUDA(cudaMemcpyAsync(vw, g->vw.get(), g->n * 8, cudaMemcpyDeviceToDevice, s));
  }
  if (ew && g->m2) {
    if (g->unit_ew) launch(k_ones, grid_for(g->m2, 256), 256, 0, s, ew, g->m2);
    else TP_CUDA(cudaMemcpyAsync(ew, g->ew.get(), g->m2 * 8, cudaMemcpyDeviceToDevice, s));
  }
  TP_LAUNCH_CHECK();
}

void export_compressed(const tp_graph *g, uint8_t *bytes, uint64_t *off, cudaStream_t s) {
  TP_REQUIRE(g->compressed, TP_ERR_INVALID);
  if (bytes) TP_CUDA(cudaMemcpyAsync(bytes, g->bytes.get(), g->nbytes, cudaMemcpyDeviceToDevice, s));
  if (off) {
    if (g->off_is64) {
      TP_CUDA(cudaMemcpyAsync(off, g->off64.get(), (g->n + 1) * 8, cudaMemcpyDeviceToDevice, s));
    } else {
      launch(k_widen, grid_for(g->n + 1, 256), 256, 0, s, g->off32.get(), off, g->n + 1);
      TP_LAUNCH_CHECK();
    }
  }
}

}  // namespace tp

extern "C" uint64_t tp_launch_count(void) { return tp::g_launches.load(); }

extern "C" void tp_profile_enable(int on) {
  tp::g_prof.enabled = on != 0;
}

extern "C" int tp_profile_read(tp_profile_entry *out, int max, void *stream) {
  using namespace tp;
  for (int f = 0; f < max && f < PF_COUNT; ++f) out[f] = tp_profile_entry{f, 0, 0.0, 0.0};
  if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return -1;
  for (const ProfRecord &r : g_prof.recs) {
    float ms = 0;
    cudaEventElapsedTime(&ms, r.a, r.b);
    if (r.family < max) {
      out[r.family].launches += 1;
      out[r.family].ms += ms;
      out[r.family].bytes += r.bytes;
    }
    g_prof.pool.push_back(r.a);
    g_prof.pool.push_back(r.b);
  }
  g_prof.recs.clear();
  return PF_COUNT < max ? PF_COUNT : max;
}

extern "C" tp_status tp_set_allocator(void *(*alloc)(size_t, void *, void *),
                                      void (*free_fn)(void *, size_t, void *, void *), void *ctx) {
  if ((alloc == nullptr) != (free_fn == nullptr)) return TP_ERR_INVALID;
  if (!alloc) {
    tp::g_hook.store(&tp::g_default_hook);
    return TP_OK;
  }
  // kept for the process lifetime: buffers made through it free through it
  const tp::AllocHook *h = new (std::nothrow) tp::AllocHook{alloc, free_fn, ctx};
  if (!h) return TP_ERR_OOM;
  tp::g_hook.store(h);
  return TP_OK;
}
