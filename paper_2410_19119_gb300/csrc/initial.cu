// Initial partitioning of the coarsest graph by recursive bisection (the
// paper's KaMinPar uses a portfolio of greedy graph growing and 2-way FM,
// Section "KaMinPar"). Deterministic GPU form: every node of the bisection
// tree owns the blocks [offset, offset + kk); its vertices are bisected with
// kk0 = ceil(kk/2) and kk1 = floor(kk/2) blocks per side by T seeded attempts:
//   1. BFS from a hashed seed vertex (FIFO order, neighbours in ascending id,
//      unreached vertices appended in ascending id), computed level by level:
//      a vertex joins the next frontier behind the earliest frontier vertex
//      adjacent to it;
//   2. side 0 = the longest prefix of that order weighing at most
//      floor(W_sub * kk0 / kk);
//   3. refine_rounds rounds of 2-way label propagation with side caps
//      kk0 * L_max and kk1 * L_max and the same prefix approval as k-way LP;
//   4. the cut of the induced subgraph.
// The attempt with the smallest cut (lowest attempt on ties) wins; the tree
// is processed depth by depth, all nodes of a depth together. Batched
// graphs form a forest: every graph's root carries the hash key offset and
// L_max its graph would use alone, so each tree's result is that graph's.
//
// An attempt is run by one CTA whose state (BFS order, claims, connectivity,
// sides) lives in shared memory, or, where the node is too large for that or
// has so many edges that one SM would scan them for long, by a thread-block
// cluster of 2 to 16 CTAs with the state in global memory; the barriers are
// then the hardware's cluster barriers. The 2-way LP keeps every vertex's
// connectivity difference D = (weight to side 1) - (weight to side 0) and
// updates it along the edges of moved vertices only, so the 8 sub-rounds of a
// round cost the edges of the movers instead of all edges, and the cut is a
// sum over D.
#include <cooperative_groups.h>

#include <algorithm>
#include <vector>

#include "select.cuh"

namespace cg = cooperative_groups;

namespace tp {

namespace {

constexpr int kIPMaxThreads = 1024;

struct IPCtx {
  int64_t n;
  const int64_t *vw;       // null: unit
  const int32_t *vlist;    // vertices sorted by (node, id)
  const int64_t *nstart;   // node start in vlist
  // the subgraph induced by every node, in local positions: vertex vlist[p]
  // has neighbours ladj[lxadj[p] .. lxadj[p + 1]) (ascending, as in the graph)
  const int64_t *lxadj;
  const int32_t *ladj;
  const int64_t *lew;  // null: unit
  const int32_t *noff, *nkk;
  const int32_t *nkey;   // per node: the block offset its graph alone would give it (hash key)
  const int64_t *nlmax;  // per node: its graph's L_max
  const int32_t *nodes;  // nodes of this launch
  int32_t T;
  uint64_t seed;
  int32_t rounds, S;
  int32_t cap;      // vertices the shared-memory state has room for
  int32_t n_nodes;  // nodes of this depth
  // scratch of the cluster form, T * n entries each (cnt: T * (n + n_nodes),
  // a frontier's counts and their total)
  int32_t *ord, *claimer, *cnt, *list;
  void *dif;
  uint8_t *sub;
  uint8_t *side;  // T * n: the result of every attempt
  int64_t *cut;   // nodes * T
};

// What the CTAs of an attempt share (in the first CTA's shared memory). The
// movers' counters and weights rotate over three sub-rounds: the set two
// sub-rounds ahead is cleared while nobody can still read it.
struct IPCtl {
  unsigned long long W, wdeg, acc;
  unsigned long long inw[3][2], dlw[3];
  int32_t ncnt[3][2];
  int32_t nz, nnew;
  int32_t found[2], fb, fe;  // bfs_alone: vertices of a level and the next, the frontier
  unsigned long long w0;
  unsigned long long khi[2];
  uint32_t klo[2];
};

template <int NT>
__device__ __forceinline__ int64_t bscan_excl(int64_t v, int64_t &total) {
  constexpr int NW = NT / 32;
  __shared__ int64_t ws[NW];
  int l = lane_id(), w = threadIdx.x >> 5;
  int64_t incl = warp_incl_scan(v);
  if (l == 31) ws[w] = incl;
  __syncthreads();
  if (w == 0) {
    int64_t x = l < NW ? ws[l] : 0;
    x = warp_incl_scan(x);
    if (l < NW) ws[l] = x;
  }
  __syncthreads();
  int64_t off = w > 0 ? ws[w - 1] : 0;
  total = ws[NW - 1];
  __syncthreads();
  return off + incl - v;
}

// Exclusive scan of x[0..len) in place by one CTA, x[len] = total (int32: the
// sums are vertex counts). Four entries a thread and step: a quarter of the
// barriers of one entry a step.
template <int NT>
__device__ int32_t block_scan_array(int32_t *x, int32_t len) {
  int32_t carry = 0;
  for (int32_t q0 = 0; q0 < len; q0 += 4 * NT) {
    const int32_t q = q0 + 4 * (int32_t)threadIdx.x;
    int32_t v[4], sum = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) v[r] = q + r < len ? x[q + r] : 0, sum += v[r];
    int64_t tot;
    int32_t ex = carry + (int32_t)bscan_excl<NT>(sum, tot);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (q + r < len) x[q + r] = ex;
      ex += v[r];
    }
    carry += (int32_t)tot;
  }
  if (threadIdx.x == 0) x[len] = carry;
  __syncthreads();
  return carry;
}

// Neighbour counts of every listed vertex inside its node, then (after a
// scan into lxadj) the neighbours' positions, one warp per listed vertex.
__global__ void k_local_deg(const int64_t *xadj, const int32_t *adj, const int32_t *node_of,
                            const int32_t *vlist, int64_t m, int64_t *ldeg) {
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t p = gw; p < m; p += nw) {
    const int32_t u = vlist[p], j = node_of[u];
    int64_t k = 0;
    for (int64_t i = xadj[u] + lane_id(); i < xadj[u + 1]; i += 32) k += node_of[adj[i]] == j;
    k = warp_sum(k);
    if (lane_id() == 0) ldeg[p] = k;
  }
}

__global__ void k_local_fill(const int64_t *xadj, const int32_t *adj, const int64_t *ew,
                             const int32_t *node_of, const int32_t *loc, const int32_t *vlist,
                             int64_t m, const int64_t *lxadj, int32_t *ladj, int64_t *lew) {
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t p = gw; p < m; p += nw) {
    const int32_t u = vlist[p], j = node_of[u];
    int64_t pos = lxadj[p];
    const int64_t b = xadj[u], e = xadj[u + 1];
    for (int64_t i0 = b; i0 < e; i0 += 32) {
      const int64_t i = i0 + lane_id();
      int32_t v = 0;
      const bool in = i < e && node_of[v = adj[i]] == j;
      const unsigned msk = __ballot_sync(kFull, in);
      if (in) {
        const int64_t at = pos + __popc(msk & lanemask_lt());
        ladj[at] = loc[v];
        if (lew) lew[at] = ew[i];
      }
      pos += __popc(msk);
    }
  }
}

// Largest weighted degree (whether connectivity differences fit 32 bits).
__global__ void k_max_wdeg(const int64_t *xadj, const int64_t *ew, int64_t n,
                           unsigned long long *out) {
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int64_t best = 0;
  for (int64_t u = gw; u < n; u += nw) {
    int64_t w = 0;
    for (int64_t i = xadj[u] + lane_id(); i < xadj[u + 1]; i += 32) w += ew[i];
    w = warp_sum(w);
    best = w > best ? w : best;
  }
  if (lane_id() == 0) atomicMax(out, (unsigned long long)best);
}

// Shared-memory state of the one-CTA form for nodes of up to cap vertices:
// claimer / D (sizeof(V)), ord, cnt (cap + 1), list, side, sub.
template <class V>
__host__ __device__ constexpr size_t ip_smem_bytes(int64_t cap) {
  return (size_t)cap * (sizeof(V) + 12 + 2) + 16;
}

__device__ __forceinline__ void dif_add(int32_t *p, int64_t w) { atomicAdd(p, (int32_t)w); }
__device__ __forceinline__ void dif_add(int64_t *p, int64_t w) {
  atomicAdd((unsigned long long *)p, (unsigned long long)w);
}

// Cluster form: a BFS level of up to this many entries (the frontier times the
// average degree) is the first CTA's alone. A path has a vertex or two a level,
// and four cluster barriers for each: 20 000 vertices in one node took 116 ms,
// this way 23; a mesh of 53 953 vertices with 5.8 neighbours each 2.9 -> 2.6
// (with 8192 a mesh of degree 16 loses 40%). In a kernel of its own, for nodes of
// up to kIPNarrowDeg neighbours a vertex: denser ones have few levels, and the
// call alone costs their kernel 9% (36 030 vertices, 63 M entries: 7.3 -> 8.0 ms).
constexpr int64_t kIPAlone = 2048;
constexpr int64_t kIPNarrowDeg = 24;

// BFS levels by the first CTA of a cluster, from the frontier ord[fb .. fe) on
// (fe: the order's length), until one is too wide or nothing is left; the
// frontier is then in ctl. A level's steps as in k_bisect. Few vertices (a warp)
// are put in order by (claiming vertex, own number), which is the order of the
// adjacencies, without counting and emitting them.
template <int NT>
__device__ __noinline__ void bfs_alone(const int64_t *lx, const int32_t *ladj, int32_t *ord,
                                       int32_t *claimer, int32_t *cnt, int32_t *list, IPCtl *ctl,
                                       int gs, int32_t nz, int32_t width, int32_t fb, int32_t fe) {
  const int lane = lane_id(), gl = lane & (gs - 1);
  const unsigned gmask = gs == 32 ? kFull : ((1u << gs) - 1u) << (lane & ~(gs - 1));
  const int32_t gid = (int32_t)threadIdx.x / gs, ngr = NT / gs;
  if (threadIdx.x == 0) ctl->found[0] = ctl->found[1] = 0;
  __syncthreads();
  for (int32_t lev = 0; fb < fe && fe < nz && fe - fb <= width; ++lev) {
    int32_t *found = &ctl->found[lev & 1];
    if (threadIdx.x == 0) ctl->found[~lev & 1] = 0;  // (read before the last level's last barrier)
    for (int32_t i = fb + gid; i < fe; i += ngr) {
      const int32_t p = ord[i];
      if (gl == 0) cnt[i - fb] = 0;
      const int64_t e = lx[p + 1];
      for (int64_t q0 = lx[p]; q0 < e; q0 += gs) {
        const int32_t y = q0 + gl < e ? ladj[q0 + gl] : -1;
        const bool first = y >= 0 && claimer[y] > i && atomicMin(&claimer[y], i) == INT32_MAX;
        const unsigned m = __ballot_sync(gmask, first);
        if (m == 0) continue;
        int32_t base = 0;
        const int leader = __ffs(m) - 1;
        if (lane == leader) base = atomicAdd(found, __popc(m));
        base = __shfl_sync(gmask, base, leader);
        if (first) list[base + __popc(m & lanemask_lt())] = y;
      }
    }
    __syncthreads();
    const int32_t nn = *found;
    if (nn == 0) {
      fb = fe;
      break;
    }
    if (nn <= 32) {
      if (threadIdx.x < 32) {
        const int32_t y = lane < nn ? list[lane] : 0;
        const uint64_t k = lane < nn ? (uint64_t)(uint32_t)claimer[y] << 32 | (uint32_t)y : ~0ull;
        int32_t at = 0;
        for (int q = 0; q < nn; ++q) at += __shfl_sync(kFull, k, q) < k;
        if (lane < nn) {
          ord[fe + at] = y;
          claimer[y] = -1;
        }
      }
    } else {
      for (int32_t q = threadIdx.x; q < nn; q += NT) atomicAdd(&cnt[claimer[list[q]] - fb], 1);
      __syncthreads();
      block_scan_array<NT>(cnt, fe - fb);
      for (int32_t i = fb + gid; i < fe; i += ngr) {
        const int32_t c0 = cnt[i - fb], k = cnt[i - fb + 1] - c0;
        if (k == 0) continue;
        const int32_t p = ord[i];
        const int64_t e = lx[p + 1];
        int32_t done = 0;
        for (int64_t q0 = lx[p]; done < k && q0 < e; q0 += gs) {
          const int32_t y = q0 + gl < e ? ladj[q0 + gl] : -1;
          const bool mine = y >= 0 && claimer[y] == i;
          const unsigned m = __ballot_sync(gmask, mine);
          if (mine) {
            ord[fe + c0 + done + __popc(m & lanemask_lt())] = y;
            claimer[y] = -1;
          }
          done += __popc(m);
        }
      }
    }
    __syncthreads();
    fb = fe;
    fe += nn;
  }
  if (threadIdx.x == 0) ctl->fb = fb, ctl->fe = fe;
}

// One attempt of one node. SM: one CTA, state in shared memory; otherwise a
// cluster of any size, state in global memory (L1 lines are dropped by the
// barriers' acquire). V: type of the connectivity differences (int32_t where
// twice every weighted degree fits). Adjacencies are scanned by groups of gs
// lanes, gs picked from the node's average degree, so that a mesh's six
// neighbours do not occupy a warp each.
// Bound by latency: a mesh's BFS has about a hundred levels of four dependent
// steps with a barrier each, a dense node is read from HBM about four times
// (BFS claims and emission, D, the movers' rows).
// NARROW (clusters): narrow BFS levels are the first CTA's (bfs_alone).
template <int NT, bool SM, class V, bool NARROW = false>
__global__ void __launch_bounds__(NT, SM && NT <= 512 ? 1024 / NT : 1) k_bisect(IPCtx c) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ IPCtl s_ctl;
  cg::cluster_group cl = cg::this_cluster();
  const int cs = SM ? 1 : (int)cl.num_blocks(), rank = SM ? 0 : (int)cl.block_rank();
  IPCtl *ctl = SM ? &s_ctl : cl.map_shared_rank(&s_ctl, 0);
  auto sync_all = [&] {
    if (SM || cs == 1) __syncthreads();
    else cl.sync();
  };
  const int32_t at = (int32_t)(blockIdx.x / (unsigned)cs);
  const int32_t j = c.nodes[at / c.T], a = at % c.T;
  const int64_t nb = c.nstart[j];
  const int32_t ns = (int32_t)(c.nstart[j + 1] - nb);
  const int32_t kk = c.nkk[j], k0 = (kk + 1) / 2, k1 = kk / 2;
  if (ns == 0) {  // the whole cluster leaves
    if (rank == 0 && threadIdx.x == 0) c.cut[(int64_t)j * c.T + a] = 0;
    return;
  }
  const int64_t R = (int64_t)a * c.n + nb;  // scratch region of this attempt
  int32_t *claimer, *ord, *cnt, *list;
  uint8_t *sub, *side;
  V *dif;
  if constexpr (SM) {
    dif = reinterpret_cast<V *>(smem);  // claims are done with when D begins
    claimer = reinterpret_cast<int32_t *>(smem);
    ord = reinterpret_cast<int32_t *>(smem + sizeof(V) * c.cap);
    cnt = ord + c.cap;
    list = cnt + c.cap + 1;
    sub = reinterpret_cast<uint8_t *>(list + c.cap + 1);
    side = sub + c.cap;
  } else {
    claimer = c.claimer + R;
    ord = c.ord + R;
    cnt = c.cnt + (int64_t)a * (c.n + c.n_nodes) + nb + j;
    list = c.list + R;
    dif = static_cast<V *>(c.dif) + R;
    sub = c.sub + R;
    side = c.side + R;
  }
  const int64_t *lx = c.lxadj + nb;
  const int32_t *vs = c.vlist + nb;
  const uint64_t key = ((uint64_t)(uint32_t)c.nkey[j] << 32) | (uint32_t)kk;
  const int lane = lane_id();
  const int32_t tid = rank * NT + (int32_t)threadIdx.x, nthr = cs * NT;
  auto cw = [&](int32_t x) -> int64_t { return c.vw ? c.vw[vs[x]] : 1; };
  // lanes per adjacency
  const int64_t avg = (lx[ns] - lx[0]) / ns;
  const int gs = avg > 24 ? 32 : avg > 12 ? 16 : avg > 5 ? 8 : 4;
  const int gl = lane & (gs - 1);
  const unsigned gmask = gs == 32 ? kFull : ((1u << gs) - 1u) << (lane & ~(gs - 1));
  const int32_t gid = tid / gs, ngr = nthr / gs;

  if (threadIdx.x == 0 && rank == 0) s_ctl = IPCtl{};
  for (int32_t x = tid; x < ns; x += nthr) claimer[x] = INT32_MAX;
  sync_all();
  // ---------------- BFS order
  const int32_t seed_v =
      (int32_t)(round_key(c.seed, kTagIPSeed, key, (uint64_t)a) % (uint64_t)ns);
  {
    // vertices with neighbours (no BFS finds more) and the node's weight
    int32_t nz = 0;
    int64_t w = 0;
    for (int32_t x = tid; x < ns; x += nthr) nz += lx[x + 1] > lx[x], w += cw(x);
    nz = warp_sum(nz);
    w = warp_sum(w);
    if (lane == 0) {
      if (nz) atomicAdd(&ctl->nz, nz);
      atomicAdd(&ctl->W, (unsigned long long)w);
    }
    if (tid == 0) ord[0] = seed_v, claimer[seed_v] = -1;
  }
  sync_all();
  const int32_t nz = ctl->nz;
  const int64_t W = (int64_t)ctl->W;
  int32_t tail = 1;
  for (int32_t fb = 0, fe = 1; fb < fe && tail < nz;) {
    if constexpr (NARROW) {
      const int32_t width = (int32_t)(kIPAlone / max(avg, (int64_t)gs));
      if (cs > 1 && fe - fb <= width) {
        if (rank == 0)
          bfs_alone<NT>(lx, c.ladj, ord, claimer, cnt, list, &s_ctl, gs, nz, width, fb, fe);
        sync_all();
        fb = ctl->fb;
        fe = tail = ctl->fe;
        continue;
      }
    }
    // every undiscovered neighbour is claimed by its earliest frontier vertex
    // (claimer: INT32_MAX unclaimed, -1 already in the order); the first
    // claim of a vertex lists it
    for (int32_t i = fb + gid; i < fe; i += ngr) {
      const int32_t p = ord[i];
      if (gl == 0) cnt[i - fb] = 0;
      const int64_t e = lx[p + 1];
      for (int64_t q0 = lx[p]; q0 < e; q0 += 4 * gs) {
        int32_t y[4], cur[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) y[r] = q0 + r * gs + gl < e ? c.ladj[q0 + r * gs + gl] : -1;
#pragma unroll
        for (int r = 0; r < 4; ++r) cur[r] = y[r] >= 0 ? claimer[y[r]] : -1;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          bool first = false;
          if (cur[r] > i) first = atomicMin(&claimer[y[r]], i) == INT32_MAX;
          const unsigned m = __ballot_sync(gmask, first);
          if (m == 0) continue;
          int32_t base = 0;
          const int leader = __ffs(m) - 1;
          if (lane == leader) base = atomicAdd(&ctl->nnew, __popc(m));
          base = __shfl_sync(gmask, base, leader);
          if (first) list[base + __popc(m & lanemask_lt())] = y[r];
        }
      }
    }
    sync_all();
    const int32_t nn = ctl->nnew;
    if (nn == 0) break;
    for (int32_t q = tid; q < nn; q += nthr) atomicAdd(&cnt[claimer[list[q]] - fb], 1);
    sync_all();
    if (rank == 0) {
      block_scan_array<NT>(cnt, fe - fb);
      if (threadIdx.x == 0) ctl->nnew = 0;
    }
    if (cs > 1) sync_all();
    // claimed neighbours in frontier order, then adjacency order
    for (int32_t i = fb + gid; i < fe; i += ngr) {
      const int32_t c0 = cnt[i - fb], k = cnt[i - fb + 1] - c0;
      if (k == 0) continue;
      const int32_t p = ord[i];
      const int64_t e = lx[p + 1];
      int32_t done = 0;
      for (int64_t q0 = lx[p]; done < k && q0 < e; q0 += gs) {
        const int32_t y = q0 + gl < e ? c.ladj[q0 + gl] : -1;
        const bool mine = y >= 0 && claimer[y] == i;
        const unsigned m = __ballot_sync(gmask, mine);
        if (mine) {
          ord[tail + c0 + done + __popc(m & lanemask_lt())] = y;
          claimer[y] = -1;
        }
        done += __popc(m);
      }
    }
    sync_all();
    fb = fe;
    fe = tail = tail + nn;
  }
  // ---------------- the rest of the order, and greedy growing: the longest
  // prefix within target0 (first CTA)
  const int64_t target0 = (int64_t)(((__int128)W * k0) / kk);
  const int64_t caps[2] = {(int64_t)k0 * c.nlmax[j], (int64_t)k1 * c.nlmax[j]};
  if (rank == 0) {
    int32_t end = tail;  // append unreached vertices in ascending id
    if (tail < ns) {
      for (int32_t x0 = 0; x0 < ns; x0 += NT) {
        const int32_t x = x0 + (int32_t)threadIdx.x;
        const int64_t f = x < ns && claimer[x] != -1;
        int64_t tot;
        const int64_t ex = bscan_excl<NT>(f, tot);
        if (f) ord[end + ex] = x;
        end += (int32_t)tot;
      }
      __syncthreads();
    }
    int64_t carry = 0, w0 = 0;
    for (int32_t q0 = 0; q0 < ns; q0 += 4 * NT) {
      const int32_t q = q0 + 4 * (int32_t)threadIdx.x;
      int32_t x[4];
      int64_t w[4], sum = 0, tot;
#pragma unroll
      for (int r = 0; r < 4; ++r) x[r] = q + r < ns ? ord[q + r] : -1;
#pragma unroll
      for (int r = 0; r < 4; ++r) w[r] = x[r] >= 0 ? cw(x[r]) : 0, sum += w[r];
      int64_t incl = carry + bscan_excl<NT>(sum, tot);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        incl += w[r];
        if (x[r] < 0) continue;
        const bool in0 = incl <= target0;
        side[x[r]] = in0 ? 0 : 1;
        if (in0) w0 += w[r];
      }
      carry += tot;
    }
    w0 = warp_sum(w0);
    if (lane == 0) atomicAdd(&ctl->w0, (unsigned long long)w0);
  }
  sync_all();
  // ---------------- connectivity differences
  {
    int64_t wsum = 0;
    for (int32_t x = gid; x < ns; x += ngr) {
      int64_t d = 0;
      const int64_t b = lx[x], e = lx[x + 1];
#pragma unroll 4
      for (int64_t q = b + gl; q < e; q += gs) {
        const int64_t w = c.lew ? c.lew[q] : 1;
        wsum += w;
        d += side[c.ladj[q]] ? w : -w;
      }
      for (int o = gs >> 1; o > 0; o >>= 1) d += __shfl_xor_sync(gmask, d, o);
      if (gl == 0) dif[x] = (V)d;
    }
    __syncwarp();
    wsum = warp_sum(wsum);
    if (lane == 0 && wsum) atomicAdd(&ctl->wdeg, (unsigned long long)wsum);
  }
  sync_all();
  // ---------------- 2-way label propagation
  int64_t lw1 = W - (int64_t)ctl->w0, lw0 = (int64_t)ctl->w0;
  const int32_t nq = (ns + 3) / 4;
  int32_t step = 0;  // sub-rounds so far (selects the rotating counters)
  for (int32_t r = 0; r < c.rounds; ++r) {
    const uint64_t rk = round_key(c.seed, kTagIPLP, key, ((uint64_t)a << 8) + (uint64_t)r);
    for (int32_t t = tid; t < nq; t += nthr)  // each thread reads only its own entries below
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (4 * t + i < ns)
          sub[4 * t + i] = (uint8_t)sub_round_of(hstep(rk, (uint64_t)(4 * t + i)), c.S);
    bool moved = false;
    for (int32_t s = 0; s < c.S && s < 256; ++s, ++step) {
      const int cur = step % 3, nxt = (step + 1) % 3;
      if (tid == 0) {
        ctl->inw[nxt][0] = ctl->inw[nxt][1] = ctl->dlw[nxt] = 0;
        ctl->ncnt[nxt][0] = ctl->ncnt[nxt][1] = 0;
      }
      // movers into side 0 are listed from the front, into side 1 from the back
      for (int32_t t0 = tid - lane; t0 < nq; t0 += nthr) {
        const int32_t t = t0 + lane;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int32_t x = 4 * t + i;
          int to = -1;
          int64_t w = 0;
          if (t < nq && x < ns && sub[x] == s) {
            const int own = side[x];
            const int64_t d = own ? -(int64_t)dif[x] : (int64_t)dif[x];
            if (d > 0) {
              w = cw(x);
              if ((own ? lw0 : lw1) + w <= caps[1 - own]) to = 1 - own;
            }
          }
          const unsigned m0 = __ballot_sync(kFull, to == 0), m1 = __ballot_sync(kFull, to == 1);
          if (!(m0 | m1)) continue;
          const unsigned mine = to == 0 ? m0 : m1;
          int32_t base = 0;
          if (to >= 0) {
            atomicAdd(&ctl->inw[cur][to], (unsigned long long)w);
            if (lane == __ffs(mine) - 1) base = atomicAdd(&ctl->ncnt[cur][to], __popc(mine));
          }
          const int32_t b0 = m0 ? __shfl_sync(kFull, base, __ffs(m0) - 1) : 0;
          const int32_t b1 = m1 ? __shfl_sync(kFull, base, __ffs(m1) - 1) : 0;
          if (to >= 0) {
            const int32_t pos = (to ? b1 : b0) + __popc(mine & lanemask_lt());
            list[to ? ns - 1 - pos : pos] = x;
          }
        }
      }
      sync_all();
      const int32_t m0 = ctl->ncnt[cur][0], m1 = ctl->ncnt[cur][1];
      if (m0 + m1 == 0) continue;
      moved = true;
      // a side whose movers do not all fit takes the longest fitting prefix in
      // (gain desc, vertex asc) order
      const bool sel0 = m0 && lw0 + (int64_t)ctl->inw[cur][0] > caps[0];
      const bool sel1 = m1 && lw1 + (int64_t)ctl->inw[cur][1] > caps[1];
      uint64_t khi[2] = {~0ull, ~0ull};
      uint32_t klo[2] = {~0u, ~0u};
      if (sel0 || sel1) {
        for (int t = 0; t < 2; ++t) {
          if (!(t ? sel1 : sel0) || rank != (t && cs > 1 ? 1 : 0)) continue;
          auto item = [&](int64_t q, uint64_t &hi, uint32_t &lo, int64_t &w) {
            const int32_t x = list[t ? ns - 1 - q : q];
            const int64_t d = (int64_t)dif[x];
            hi = ~(uint64_t)(t ? d : -d);
            lo = (uint32_t)x;
            w = cw(x);
          };
          uint64_t h;
          uint32_t l;
          block_select(t ? m1 : m0, caps[t] - (t ? lw1 : lw0), W < (int64_t)1 << 31, item, h, l);
          if (threadIdx.x == 0) ctl->khi[t] = h, ctl->klo[t] = l;
        }
        sync_all();
        if (sel0) khi[0] = ctl->khi[0], klo[0] = ctl->klo[0];
        if (sel1) khi[1] = ctl->khi[1], klo[1] = ctl->klo[1];
      }
      // approved moves, and their neighbours' differences. A mover's own
      // difference may change under its neighbours' moves meanwhile, so with
      // a threshold the decisions are taken before any update.
      if (sel0 || sel1) {
        for (int32_t q = tid; q < m0 + m1; q += nthr) {
          const int t = q >= m0;
          const int32_t lq = t ? ns - 1 - (q - m0) : q;
          const int32_t x = list[lq];
          const int64_t d = (int64_t)dif[x];
          const uint64_t hi = ~(uint64_t)(t ? d : -d);
          if (hi > khi[t] || (hi == khi[t] && (uint32_t)x >= klo[t]))
            if (t ? sel1 : sel0) list[lq] = ~x;  // refused
        }
        sync_all();
      }
      for (int32_t q = gid; q < m0 + m1; q += ngr) {
        const int t = q >= m0;
        const int32_t x = list[t ? ns - 1 - (q - m0) : q];
        if (x < 0) continue;
        if (gl == 0) {
          side[x] = (uint8_t)t;
          const int64_t w = cw(x);
          atomicAdd(&ctl->dlw[cur], (unsigned long long)(t ? w : -w));
        }
        const int64_t b = lx[x], e = lx[x + 1];
#pragma unroll 4
        for (int64_t i = b + gl; i < e; i += gs) {
          const int64_t w = 2 * (c.lew ? c.lew[i] : (int64_t)1);
          dif_add(&dif[c.ladj[i]], t ? w : -w);
        }
      }
      sync_all();
      const int64_t dl = (int64_t)ctl->dlw[cur];
      lw1 += dl;
      lw0 -= dl;
    }
    // nothing moved in a whole round: every later round would find the same
    if (!moved) break;
  }
  // ---------------- cut of the induced subgraph: a vertex's outside weight
  // is (weighted degree +- D) / 2, the cut half of their sum
  {
    int64_t acc = 0;
    for (int32_t x = tid; x < ns; x += nthr) {
      const int64_t d = (int64_t)dif[x];
      acc += side[x] ? -d : d;
      if (SM) c.side[R + x] = side[x];
    }
    acc = warp_sum(acc);
    if (lane == 0 && acc) atomicAdd(&ctl->acc, (unsigned long long)acc);
  }
  sync_all();
  if (tid == 0)
    c.cut[(int64_t)j * c.T + a] = ((int64_t)ctl->wdeg + (int64_t)ctl->acc) / 4;
}

// The winning attempt of every node (smallest cut, lowest attempt on ties);
// blockIdx.y slices a node. flag[p] = 1 where position p lies on its side 0;
// vertices of finished children get their block.
__global__ void k_pick(IPCtx c, const int32_t *child0, const int32_t *child1, int32_t *flag,
                       int32_t *part) {
  const int32_t j = blockIdx.x;
  const int64_t nb = c.nstart[j], ns = c.nstart[j + 1] - nb;
  const int64_t x0 = (int64_t)blockIdx.y * blockDim.x + threadIdx.x;
  if (x0 - threadIdx.x >= ns) return;
  int32_t best = 0;
  for (int32_t a = 1; a < c.T; ++a)
    if (c.cut[(int64_t)j * c.T + a] < c.cut[(int64_t)j * c.T + best]) best = a;
  const int32_t k0 = (c.nkk[j] + 1) / 2;
  const int32_t c0 = child0[j], c1 = child1[j];
  for (int64_t x = x0; x < ns; x += (int64_t)gridDim.y * blockDim.x) {
    const int sd = c.side[(int64_t)best * c.n + nb + x];
    flag[nb + x] = sd == 0;
    if ((sd ? c1 : c0) < 0) part[c.vlist[nb + x]] = sd == 0 ? c.noff[j] : c.noff[j] + k0;
  }
}

// Side-0 vertices of every node: prefix of the flags at the node starts.
__global__ void k_side_prefix(const int64_t *pre, const int64_t *nstart, int32_t nodes,
                              int64_t *out) {
  for (int32_t j = blockIdx.x * blockDim.x + threadIdx.x; j <= nodes; j += gridDim.x * blockDim.x)
    out[j] = pre[nstart[j]];
}

// The next depth's vertex list: every node's list split stably into its
// children's (a stable partition replaces a sort by (node, id): the list is
// in that order already).
__global__ void k_split(const int64_t *nstart, const int32_t *child0, const int32_t *child1,
                        const int64_t *next_start, const int64_t *pre, const int32_t *flag,
                        const int32_t *vlist, int64_t m, int32_t *node_of, int32_t *loc,
                        int32_t *next_vlist) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < m;
       p += (int64_t)gridDim.x * blockDim.x) {
    const int32_t u = vlist[p], j = node_of[u];
    const int64_t r0 = pre[p] - pre[nstart[j]];
    const bool s0 = flag[p] != 0;
    const int32_t ch = s0 ? child0[j] : child1[j];
    if (ch >= 0) {
      const int64_t r = s0 ? r0 : p - nstart[j] - r0;
      next_vlist[next_start[ch] + r] = u;
      loc[u] = (int32_t)r;
    }
    node_of[u] = ch;
  }
}

__global__ void k_fill_i32(int32_t *p, int64_t n, int32_t v) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    p[i] = v;
}

// First depth: the vertices in order, each in its root (rs: the roots' starts).
__global__ void k_first_lists(const int64_t *rs, int32_t roots, int64_t n, int32_t *vlist,
                              int32_t *node_of, int32_t *loc) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    int32_t lo = 0, hi = roots - 1;
    while (lo < hi) {
      const int32_t mid = (lo + hi + 1) / 2;
      if (rs[mid] <= u) lo = mid;
      else hi = mid - 1;
    }
    vlist[u] = (int32_t)u;
    node_of[u] = lo;
    loc[u] = (int32_t)(u - rs[lo]);
  }
}

// Node table of one depth on the host.
struct Depth {
  std::vector<int32_t> off, kk, key, c0, c1;
  std::vector<int64_t> lmax, start, entries;  // entries: estimate of the adjacency entries
  int32_t nodes() const { return (int32_t)off.size(); }
  void add(int32_t o, int32_t k, int32_t h, int64_t l, int64_t ent) {
    off.push_back(o), kk.push_back(k), key.push_back(h), lmax.push_back(l), entries.push_back(ent);
  }
};

// Its device copy, one upload: start (nodes + 1) and lmax, then off, kk, key,
// c0, c1 and the launch classes' node lists.
struct DepthDev {
  Buf<int64_t> buf;
  const int64_t *start = nullptr, *lmax = nullptr;
  const int32_t *off = nullptr, *kk = nullptr, *key = nullptr, *c0 = nullptr, *c1 = nullptr,
                *order = nullptr;
  void upload(const Depth &d, const std::vector<int32_t> &ord, std::vector<int64_t> &host,
              cudaStream_t s) {
    const size_t N = (size_t)d.nodes();
    host.assign(2 * N + 1 + (6 * N + 1) / 2, 0);
    std::copy(d.start.begin(), d.start.end(), host.begin());
    std::copy(d.lmax.begin(), d.lmax.end(), host.begin() + N + 1);
    int32_t *h = reinterpret_cast<int32_t *>(host.data() + 2 * N + 1);
    std::copy(d.off.begin(), d.off.end(), h);
    std::copy(d.kk.begin(), d.kk.end(), h + N);
    std::copy(d.key.begin(), d.key.end(), h + 2 * N);
    std::copy(d.c0.begin(), d.c0.end(), h + 3 * N);
    std::copy(d.c1.begin(), d.c1.end(), h + 4 * N);
    std::copy(ord.begin(), ord.end(), h + 5 * N);
    buf.alloc(host.size(), s);
    TP_CUDA(cudaMemcpyAsync(buf.get(), host.data(), host.size() * 8, cudaMemcpyHostToDevice, s));
    start = buf.get();
    lmax = start + N + 1;
    off = reinterpret_cast<const int32_t *>(lmax + N);
    kk = off + N, key = kk + N, c0 = key + N, c1 = c0 + N, order = c1 + N;
  }
};

// How a node's attempts are run: one CTA of `threads` with its state in
// shared memory (cluster = 0), or a cluster of CTAs.
// (narrow: narrow BFS levels in the first one alone).
struct Shape {
  int threads, cluster;
  bool narrow;
  bool operator==(const Shape &o) const {
    return threads == o.threads && cluster == o.cluster && narrow == o.narrow;
  }
};

// Shared memory of the one-CTA form: what a block may have beside the static
// part (select and scan buffers).
constexpr size_t kIPSmem = 220 * 1024;
// A node of more adjacency entries than this is scanned by a cluster while
// SMs are idle: one SM reads about 0.1 TB/s, so a million 12-byte entries
// take it over 100 us a pass.
constexpr int64_t kIPClusterEntries = (int64_t)1 << 19;

// Most vertices whose state fits: a multiple of 16, as a launch rounds its
// largest node up to one (12 512 vertices, 10 224 with 64-bit differences).
template <class V>
constexpr int64_t ip_smem_cap() {
  return (int64_t)((kIPSmem - 16) / (sizeof(V) + 14)) & ~(int64_t)15;
}
static_assert(ip_smem_bytes<int32_t>(ip_smem_cap<int32_t>()) <= kIPSmem &&
                  ip_smem_bytes<int64_t>(ip_smem_cap<int64_t>()) <= kIPSmem,
              "the largest node's state fits");

template <class V>
bool ip_large(int64_t ns, int64_t entries) {
  return ns > ip_smem_cap<V>() || entries > kIPClusterEntries;
}

// attempts: of all nodes of the depth; large_attempts: of those that a
// cluster would run (they share the SMs among themselves).
template <class V>
Shape ip_shape(int64_t ns, int64_t entries, int64_t attempts, int64_t large_attempts) {
  if (ip_large<V>(ns, entries)) {
    const int64_t cl = std::max<int64_t>(1, std::min<int64_t>(16, num_sms() / large_attempts));
    if (cl > 1 || ns > ip_smem_cap<V>())
      return Shape{kIPMaxThreads, (int)cl, cl > 1 && entries <= kIPNarrowDeg * ns};
  }
  // smaller CTAs, several per SM, where many attempts are in flight: 100 graphs of
  // 200, 1000, 2000, 5000 and 12000 vertices in one batch took 3.1, 7.8, 12.3, 32
  // and 79 ms with 1024 threads everywhere, 2.6, 5.7, 5.5, 13 and 33 with these.
  // Few attempts are as fast as their own threads: a single random graph of 2000
  // vertices takes 0.42 ms with the smaller blocks, 0.37 with these; of 200 with
  // 1024 threads 0.19, with 256 0.17.
  const bool many = attempts >= 2LL * num_sms();
  const int threads = many ? (ns <= 512 ? 128 : ns <= 2048 ? 256 : ns <= 6144 ? 512 : 1024)
                           : (ns <= 256 ? 256 : ns <= 1024 ? 512 : 1024);
  return Shape{threads, 0, false};
}

template <int NT, bool SM, class V, bool NARROW = false>
void launch_bisect(const IPCtx &c, int64_t attempts, int cluster, cudaStream_t s) {
  const size_t smem = SM ? ip_smem_bytes<V>(c.cap) : 0;
  auto kern = k_bisect<NT, SM, V, NARROW>;
  if (SM)
    TP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kIPSmem));
  else
    TP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg{};
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // smaller clusters where the device cannot hold all attempts' at once
  for (; !SM && cluster > 1; --cluster) {
    attr[0].val.clusterDim.x = (unsigned)cluster;
    cfg.gridDim = dim3((unsigned)(attempts * cluster));
    int fit = 0;
    if (cudaOccupancyMaxActiveClusters(&fit, kern, &cfg) == cudaSuccess && fit >= attempts) break;
    (void)cudaGetLastError();
  }
  attr[0].val.clusterDim.x = (unsigned)(SM ? 1 : cluster);
  cfg.gridDim = dim3((unsigned)(attempts * (SM ? 1 : cluster)));
  TP_CUDA(cudaLaunchKernelEx(&cfg, kern, c));
  count_launch();
}

template <class V>
void bisect_forest(const tp_graph *g, const std::vector<IPRoot> &roots,
                   const std::vector<int64_t> &root_start, const tp_params &p, int32_t *d_part,
                   cudaStream_t s) {
  const int64_t n = g->n;
  const int32_t T = std::max(1, p.ip_attempts);
  const bool weighted = !g->unit_ew;
  Depth d;
  for (size_t r = 0; r < roots.size(); ++r) {
    TP_REQUIRE(roots[r].k >= 2, TP_ERR_INVALID);
    const int64_t nr = root_start[r + 1] - root_start[r];
    d.add(roots[r].off, roots[r].k, roots[r].key, roots[r].l_max,
          (int64_t)((double)g->m2 * (double)nr / (double)n));
  }
  d.start = root_start;
  Buf<int32_t> node_of(n, s), vlist(n, s), next_vlist(n, s), loc(n, s), flag(n, s);
  Buf<int64_t> pre(n + 1, s), lxadj;
  Buf<int32_t> ladj;
  Buf<int64_t> lew;
  Buf<uint8_t> side(T * n, s);
  Buf<int32_t> ord, claimer, cnt, list;  // cluster form only
  Buf<V> dif;
  Buf<uint8_t> sub;
  Buf<int64_t> cut;
  DepthDev dev, next_dev;
  // after every buffer that its kernels use: an error while the classes of a
  // depth run side by side waits for them before any of it is freed
  TierStreams streams;
  std::vector<int64_t> host, next_host;
  for (int depth = 0; d.nodes() > 0; ++depth) {
    const int32_t nodes = d.nodes();
    const int64_t m = d.start[nodes];
    // children of every node at the next depth (-1: leaf, assign the block)
    Depth nx;
    d.c0.assign(nodes, -1), d.c1.assign(nodes, -1);
    for (int32_t j = 0; j < nodes; ++j) {
      const int32_t k0 = (d.kk[j] + 1) / 2, k1 = d.kk[j] / 2;
      if (k0 >= 2) d.c0[j] = nx.nodes(), nx.add(d.off[j], k0, d.key[j], d.lmax[j], d.entries[j] / 2);
      if (k1 >= 2)
        d.c1[j] = nx.nodes(),
        nx.add(d.off[j] + k0, k1, d.key[j] + k0, d.lmax[j], d.entries[j] / 2);
    }
    // launch classes: nodes of the same shape, the largest first
    std::vector<int32_t> order(nodes);
    std::vector<Shape> shape(nodes);
    int64_t large = 0;
    for (int32_t j = 0; j < nodes; ++j)
      large += ip_large<V>(d.start[j + 1] - d.start[j], d.entries[j]);
    for (int32_t j = 0; j < nodes; ++j) {
      order[j] = j;
      shape[j] = ip_shape<V>(d.start[j + 1] - d.start[j], d.entries[j], (int64_t)nodes * T,
                             large * T);
    }
    std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) {
      if (shape[x].cluster != shape[y].cluster) return shape[x].cluster > shape[y].cluster;
      if (shape[x].narrow != shape[y].narrow) return shape[x].narrow < shape[y].narrow;
      return shape[x].threads > shape[y].threads;
    });
    DepthDev &cur = depth % 2 ? next_dev : dev;
    cur.upload(d, order, depth % 2 ? next_host : host, s);
    if (depth == 0) {
      launch(k_first_lists, grid_for(n, 256), 256, 0, s, cur.start, nodes, n, vlist.get(),
             node_of.get(), loc.get());
      TP_LAUNCH_CHECK();
    }
    IPCtx c{};
    // a single root's induced subgraph is the graph itself
    const bool whole = depth == 0 && nodes == 1;
    if (whole) {
      c.lxadj = g->xadj.get();
      c.ladj = g->adj.get();
      c.lew = weighted ? g->ew.get() : nullptr;
    } else if (m) {
      if (!ladj.get()) {
        lxadj.alloc(n + 1, s);
        ladj.alloc(std::max<int64_t>(g->m2, 1), s);
        if (weighted) lew.alloc(std::max<int64_t>(g->m2, 1), s);
      }
      const unsigned wg = grid_for(m * 32, 256);
      launch(k_local_deg, wg, 256, 0, s, g->xadj.get(), g->adj.get(), node_of.get(), vlist.get(), m,
             lxadj.get());
      TP_LAUNCH_CHECK();
      exclusive_scan_i64(lxadj.get(), lxadj.get(), m, s);
      launch(k_local_fill, wg, 256, 0, s, g->xadj.get(), g->adj.get(),
             weighted ? g->ew.get() : nullptr, node_of.get(), loc.get(), vlist.get(), m, lxadj.get(),
             ladj.get(), weighted ? lew.get() : nullptr);
      TP_LAUNCH_CHECK();
      c.lxadj = lxadj.get();
      c.ladj = ladj.get();
      c.lew = weighted ? lew.get() : nullptr;
    }
    if ((int64_t)cut.n < (int64_t)nodes * T) cut.alloc((int64_t)nodes * T, s);
    c.n = n;
    c.n_nodes = nodes;
    c.vw = g->unit_vw ? nullptr : g->vw.get();
    c.vlist = vlist.get();
    c.nstart = cur.start;
    c.noff = cur.off;
    c.nkk = cur.kk;
    c.nkey = cur.key;
    c.nlmax = cur.lmax;
    c.T = T;
    c.seed = p.seed;
    c.rounds = p.refine_rounds;
    c.S = p.sub_rounds;
    c.side = side.get();
    c.cut = cut.get();
    if (shape[order[0]].cluster) {
      const size_t counts = (size_t)T * (size_t)(n + nodes);
      if (!ord.get()) {
        ord.alloc(T * n, s), claimer.alloc(T * n, s), list.alloc(T * n, s);
        dif.alloc(T * n, s), sub.alloc(T * n, s);
      }
      if (cnt.n < counts) cnt.alloc(counts, s);
      c.ord = ord.get(), c.claimer = claimer.get(), c.cnt = cnt.get(), c.list = list.get();
      c.dif = dif.get(), c.sub = sub.get();
    }
    // classes side by side: each is as long as its longest attempt
    const bool fork = !(shape[order[0]] == shape[order[nodes - 1]]) && streams.make();
    if (fork) streams.begin(s);
    for (int32_t b = 0, number = 0; b < nodes; ++number) {
      const Shape sh = shape[order[b]];
      const cudaStream_t cls = fork && number ? streams.st[(number - 1) % TierStreams::kN] : s;
      int32_t e = b;
      int64_t largest = 1;
      for (; e < nodes && shape[order[e]] == sh; ++e)
        largest = std::max(largest, d.start[order[e] + 1] - d.start[order[e]]);
      c.nodes = cur.order + b;
      c.cap = (int32_t)((largest + 15) & ~(int64_t)15);
      const int64_t att = (int64_t)(e - b) * T;
      if (sh.narrow) launch_bisect<kIPMaxThreads, false, V, true>(c, att, sh.cluster, cls);
      else if (sh.cluster) launch_bisect<kIPMaxThreads, false, V>(c, att, sh.cluster, cls);
      else if (sh.threads == 128) launch_bisect<128, true, V>(c, att, 1, cls);
      else if (sh.threads == 256) launch_bisect<256, true, V>(c, att, 1, cls);
      else if (sh.threads == 512) launch_bisect<512, true, V>(c, att, 1, cls);
      else launch_bisect<1024, true, V>(c, att, 1, cls);
      b = e;
    }
    if (fork) streams.end(s);
    int64_t widest = 1;
    for (int32_t j = 0; j < nodes; ++j) widest = std::max(widest, d.start[j + 1] - d.start[j]);
    const dim3 pg((unsigned)nodes, (unsigned)std::min<int64_t>((widest + 255) / 256, 256));
    launch(k_pick, pg, 256, 0, s, c, cur.c0, cur.c1, flag.get(), d_part);
    TP_LAUNCH_CHECK();
    if (nx.nodes()) {
      // the children's sizes, from the prefix of the side flags
      exclusive_scan_i32_to_i64(flag.get(), pre.get(), m, s);
      Buf<int64_t> sp(nodes + 1, s);
      launch(k_side_prefix, grid_for(nodes + 1, 256), 256, 0, s, pre.get(), cur.start, nodes,
             sp.get());
      TP_LAUNCH_CHECK();
      std::vector<int64_t> hp((size_t)nodes + 1);
      TP_CUDA(cudaMemcpyAsync(hp.data(), sp.get(), (nodes + 1) * sizeof(int64_t),
                              cudaMemcpyDeviceToHost, s));
      TP_CUDA(cudaStreamSynchronize(s));
      nx.start.assign(1, 0);
      for (int32_t j = 0; j < nodes; ++j) {
        const int64_t n0 = hp[j + 1] - hp[j], n1 = d.start[j + 1] - d.start[j] - n0;
        if (d.c0[j] >= 0) nx.start.push_back(nx.start.back() + n0);
        if (d.c1[j] >= 0) nx.start.push_back(nx.start.back() + n1);
      }
      Buf<int64_t> ns(nx.start.size(), s);
      TP_CUDA(cudaMemcpyAsync(ns.get(), nx.start.data(), nx.start.size() * 8,
                              cudaMemcpyHostToDevice, s));
      if (m) {
        launch(k_split, grid_for(m, 256), 256, 0, s, cur.start, cur.c0, cur.c1, ns.get(), pre.get(),
               flag.get(), vlist.get(), m, node_of.get(), loc.get(), next_vlist.get());
        TP_LAUNCH_CHECK();
      }
      TP_CUDA(cudaStreamSynchronize(s));  // nx.start moves on below
      std::swap(vlist, next_vlist);
    }
    d = std::move(nx);
  }
  TP_CUDA(cudaStreamSynchronize(s));  // host tables outlive their copies
}

}  // namespace

void initial_partition(const tp_graph *g, int32_t k, int64_t l_max, const tp_params &p,
                       int32_t *d_part, cudaStream_t s) {
  TP_REQUIRE(!g->compressed, TP_ERR_INVALID);
  const int64_t n = g->n;
  if (n == 0) return;
  if (k <= 1) {
    launch(k_fill_i32, grid_for(n, 256), 256, 0, s, d_part, n, 0);
    TP_LAUNCH_CHECK();
    return;
  }
  initial_partition_roots(g, {IPRoot{0, 0, k, l_max}}, {0, n}, p, d_part, s);
}

void initial_partition_roots(const tp_graph *g, const std::vector<IPRoot> &roots,
                             const std::vector<int64_t> &root_start, const tp_params &p,
                             int32_t *d_part, cudaStream_t s) {
  TP_REQUIRE(!g->compressed, TP_ERR_INVALID);
  const int64_t n = g->n;
  if (n == 0 || roots.empty()) return;
  // connectivity differences in 32 bits where they and their steps (twice an
  // edge weight) fit; a bound from sizes first, the largest weighted degree
  // only where that does not settle it
  constexpr int64_t kFit = (int64_t)1 << 29;
  bool small = g->unit_ew ? n < kFit : ew_sum_bound(g) < kFit;
  if (!small && !g->unit_ew) {
    Buf<unsigned long long> mx(1, s);
    TP_CUDA(cudaMemsetAsync(mx.get(), 0, sizeof(unsigned long long), s));
    launch(k_max_wdeg, grid_for(n * 32, 256), 256, 0, s, g->xadj.get(), g->ew.get(), n, mx.get());
    TP_LAUNCH_CHECK();
    small = read_scalar(mx.get(), s) < (unsigned long long)kFit;
  }
  if (small) bisect_forest<int32_t>(g, roots, root_start, p, d_part, s);
  else bisect_forest<int64_t>(g, roots, root_start, p, d_part, s);
}

}  // namespace tp
