// All LP rounds of a small level in one launch. A sub-round of such a level is
// a few microseconds of work between the dependent steps rate, fit, apply;
// as seven or more kernels it cost 30 us and more, most of it launch latency,
// and a CUDA graph of them had to be captured and instantiated per level. Here
// one thread-block cluster (1 to 16 CTAs, by the level's size) runs every
// round and the steps are separated by the hardware's cluster barriers: three
// per sub-round, six where targets are contested. A CTA owns a range of
// vertices: their buckets by sub-round lie in its shared memory, their moves
// in its part of the mover arrays. Vertices of the lane tier are rated in
// batches of 32 as in k_rate_lane, the others (degree <= 512) by a warp each.
// Bound by the chain of dependent loads of one rating (entry, label, label
// weight) and the barriers.
#include <cooperative_groups.h>

#include <mutex>

#include "lp_rate.cuh"

namespace cg = cooperative_groups;

namespace tp {

namespace {

constexpr int kLpSmallWarps = 16;
constexpr int kLpSmallThreads = 32 * kLpSmallWarps;
constexpr int kLpSmallCluster = 16;
constexpr int kLpSmallItems = 4;
constexpr int64_t kLpSmallVertices = 16384;  // most vertices of a CTA (its bucket list)
constexpr int64_t kLpSmallEntries = (int64_t)1 << 17;  // most adjacency entries of a CTA's share

// A warp's part of the shared memory: the lane tier's columns or a hash table.
struct LpSmallWarp {
  uint32_t lab[kLaneMaxDeg][32];  // or 1024 keys
  uint32_t aux[kLaneMaxDeg][32];  // candidate ratings, or 1024 sums
  BatchMovers mv;
  int32_t mu[32], mt[32], mo[32];
  int64_t mg[32];
};
static_assert(sizeof(uint32_t) * kLaneMaxDeg * 32 == sizeof(int32_t) << kMidLog,
              "a column block holds the mid tier's largest table");

// What the CTAs share (in the first one's shared memory).
struct LpSmallCtl {
  int32_t targets;
  int32_t pool;
  int32_t big;  // targets of more than 32 movers
};

template <bool COMP, bool W>
__global__ void __launch_bounds__(kLpSmallThreads)
    k_lp_small(RateCtx c, ApproveCtx a, uint64_t seed, uint64_t tag, uint64_t ra, uint64_t rb,
               int32_t rounds) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ LpSmallCtl s_ctl;
  __shared__ unsigned long long s_cnt;  // this CTA's movers of the sub-round
  __shared__ uint64_t s_rk;
  // buckets: the lane tier's vertices of sub-round s, then the others'
  __shared__ int32_t boff[2 * 32 + 1], bcur[2 * 32];
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  LpSmallCtl *ctl = cl.map_shared_rank(&s_ctl, 0);
  auto sync_all = [&] {
    if (cs == 1) __syncthreads();
    else cl.sync();
  };
  const int lane = lane_id(), w = threadIdx.x >> 5;
  LpSmallWarp &ws = reinterpret_cast<LpSmallWarp *>(smem)[w];
  int32_t *list = reinterpret_cast<int32_t *>(smem + sizeof(LpSmallWarp) * kLpSmallWarps);
  const int64_t n = c.g.n;
  const int32_t v0 = (int32_t)(n * rank / cs), v1 = (int32_t)(n * (rank + 1) / cs);
  const int32_t S = c.S;
  // this CTA's part of the mover arrays
  c.mv_u += v0, c.mv_t += v0, c.mv_o += v0, c.mv_g += v0;
  c.counters = &s_cnt;
  c.rk_dev = &s_rk;
  uint32_t *col = &ws.lab[0][lane], *wcol = &ws.aux[0][lane];
  uint8_t *cnt8 = reinterpret_cast<uint8_t *>(&ws.aux[0][0]) + lane;
  MoverBuf mb{ws.mu, ws.mt, ws.mo, ws.mg, 0};
  if (threadIdx.x == 0) s_ctl = LpSmallCtl{0, 0, 0}, s_cnt = 0;
  for (int32_t r = 0; r < rounds; ++r) {
    // ---- buckets of this round
    const uint64_t rk = round_key(seed, tag, ra, rb + (uint64_t)r);
    if (threadIdx.x == 0) s_rk = rk;
    if (threadIdx.x < 2 * 32) bcur[threadIdx.x] = 0;
    __syncthreads();
    for (int32_t u = v0 + (int32_t)threadIdx.x; u < v1; u += kLpSmallThreads) {
      const int s = sub_round_of(hstep(rk, (uint64_t)u), S);
      atomicAdd(&bcur[2 * s + (c.tier[u] != TIER_LANE)], 1);
    }
    __syncthreads();
    if (w == 0) {
      const int32_t x0 = bcur[2 * lane], x1 = bcur[2 * lane + 1];
      const int32_t before = warp_incl_scan(x0 + x1) - x0 - x1;
      bcur[2 * lane] = boff[2 * lane] = before;
      bcur[2 * lane + 1] = boff[2 * lane + 1] = before + x0;
      if (lane == 31) boff[64] = before + x0 + x1;
    }
    __syncthreads();
    for (int32_t u = v0 + (int32_t)threadIdx.x; u < v1; u += kLpSmallThreads) {
      const int s = sub_round_of(hstep(rk, (uint64_t)u), S);
      list[atomicAdd(&bcur[2 * s + (c.tier[u] != TIER_LANE)], 1)] = u;
    }
    sync_all();
    for (int32_t s = 0; s < S; ++s) {
      // ---- ratings
      for (int32_t q = boff[2 * s] + 32 * w; q < boff[2 * s + 1]; q += 32 * kLpSmallWarps) {
        const bool has = q + lane < boff[2 * s + 1];
        const int32_t u = has ? list[q + lane] : 0;
        int deg = 0, nmv = 0;
        if (has) {
          if (COMP) deg = lane_decode<false>(c.g, off_at(c.g, u), off_at(c.g, u + 1), col);
          else deg = min((int)(c.g.xadj[u + 1] - c.g.xadj[u]), kLaneMaxDeg);
        }
        const unsigned maxdeg = __reduce_max_sync(kFull, (unsigned)deg);
        if (maxdeg <= 16)
          lane_batch<COMP, M_LP, W, 16, false, true>(c, has, u, deg, col, wcol, cnt8, ws.mv, nmv);
        else
          lane_batch<COMP, M_LP, W, kLaneMaxDeg, false, true>(c, has, u, deg, col, wcol, cnt8, ws.mv, nmv);
        __syncwarp();
        if (nmv) {
          int32_t base = 0;
          if (lane == 0) base = (int32_t)atomicAdd(&s_cnt, (unsigned long long)nmv);
          base = __shfl_sync(kFull, base, 0);
          if (lane < nmv) {
            c.mv_u[base + lane] = ws.mv.u[lane];
            c.mv_t[base + lane] = ws.mv.t[lane];
            c.mv_o[base + lane] = ws.mv.o[lane];
            c.mv_g[base + lane] = ws.mv.g[lane];
          }
          __syncwarp();
        }
      }
      for (int32_t q = boff[2 * s + 1] + w; q < boff[2 * s + 2]; q += kLpSmallWarps) {
        const int32_t u = list[q];
        ZipNbr z;
        const int64_t d = row_degree<COMP>(c.g, u, z);
        const int lc = table_log(c, d, kMidLog);
        int32_t *keys = reinterpret_cast<int32_t *>(&ws.lab[0][0]);
        uint32_t *vals = &ws.aux[0][0];
        __syncwarp();
        for (int i = lane; i < 1 << lc; i += 32) keys[i] = -1, vals[i] = 0;
        __syncwarp();
        rate_vertex_warp<COMP, M_LP, uint32_t>(c, u, keys, vals, lc, &mb, &z);
      }
      flush_movers(c, mb);
      sync_all();
      // ---- approval: targets that fit take every mover
      const int32_t nm = (int32_t)s_cnt;
      for (int32_t i = threadIdx.x; i < nm; i += kLpSmallThreads) {
        const int32_t t = c.mv_t[i];
        const bool fits = a.lw[t] + a.in_w[t] <= a.cap;
        a.mv_ok[v0 + i] = fits;
        if (!fits && atomicAdd(&a.ccnt[t], 1) == 0) a.ctarget[atomicAdd(&ctl->targets, 1)] = t;
      }
      sync_all();
      const int32_t nt = ctl->targets;
      if (nt) {
        // contested movers are grouped by target; every target approves the
        // longest fitting prefix in (gain desc, vertex asc) order
        for (int32_t j = rank * kLpSmallThreads + (int32_t)threadIdx.x; j < nt;
             j += cs * kLpSmallThreads) {
          const int32_t t = a.ctarget[j], cnt = a.ccnt[t];
          a.cbase[t] = atomicAdd(&ctl->pool, cnt);
          if (cnt > 32) a.cbig[atomicAdd(&ctl->big, 1)] = t;
        }
        sync_all();
        for (int32_t i = threadIdx.x; i < nm; i += kLpSmallThreads) {
          if (a.mv_ok[v0 + i]) continue;
          put_contested(a, v0 + i, c.mv_t[i]);
        }
        sync_all();
        approve_targets(a, nt, ctl->big, rank, cs);
        sync_all();
        if (rank == 0 && threadIdx.x == 0) s_ctl = LpSmallCtl{0, 0, 0};
      }
      // ---- approved moves
      for (int32_t i = threadIdx.x; i < nm; i += kLpSmallThreads) {
        const int32_t t = c.mv_t[i];
        if (a.mv_ok[v0 + i]) {
          const int32_t u = c.mv_u[i];
          const int64_t wt = vwt(a, u);
          a.label[u] = t;
          atomicAdd((unsigned long long *)&a.lw[t], (unsigned long long)wt);
          atomicAdd((unsigned long long *)&a.lw[c.mv_o[i]], (unsigned long long)(-wt));
        }
        a.in_w[t] = 0;
      }
      __syncthreads();  // every thread has read s_cnt
      if (threadIdx.x == 0) s_cnt = 0;
      sync_all();
    }
  }
}

// Whether one cluster rates a level's rounds in less time than the kernels of
// the sub-rounds take, most of it their launches. Both were measured on meshes
// and uniform random graphs of 2e3 to 2.6e5 vertices and degrees 4 to 450, with
// 2, 8 and 32 sub-rounds (16 CTAs, random graphs): a round costs a lane-tier
// vertex 0.4 ns and 0.17 an entry (a fifth more with edge weights, a seventh less
// compressed), one of the warp tiers 18 and 0.36. A sub-round saves 14 us and a
// call 0.4 ms, and where the warp tiers are most of the work 48 us a sub-round
// (they take that long on the other path too). With a limit of 2^21 entries
// alone, 2.6e5 vertices of degree 8 took 2.24 ms against 1.26, 2e4 of degree 100
// 5.4 against 2.3; at the line the two are within a tenth on random graphs, and
// on meshes the cluster is up to a third faster.
bool lp_small_pays(const tp_graph *g, int32_t rounds, int32_t S) {
  const TierCache &T = g->tiers;
  const double lanes = (g->compressed ? 0.85 : g->unit_ew ? 1.0 : 1.2) *
                       (0.4 * (double)T.count[TIER_LANE] + 0.17 * (double)T.edges[TIER_LANE]);
  const double warps = 18.0 * (double)(T.count[TIER_SMALL] + T.count[TIER_MID]) +
                       0.36 * (double)(T.edges[TIER_SMALL] + T.edges[TIER_MID]);
  return rounds * lanes / (400e3 + 14e3 * rounds * S) + warps / (48e3 * S) <= 1.0;
}

// Cluster size for a level that k_lp_small can take and that gains by it, 0 for
// the others: one graph, no vertex above the mid tier, 32-bit ratings, with edge
// weights labels that fit the lane tier's 32-bit sort keys (block numbers need
// not), at most 32 sub-rounds. The smallest cluster that gives a CTA at most
// kLpSmallItems batches or vertices per sub-round: the lanes of a batch read
// different rows and labels, and an SM's L1 looks up one line a cycle (a batch
// of degree 16 takes about 700), so 16 batches on one SM cost more than four on
// each of four and their barriers.
int lp_small_cluster(const tp_graph *g, const LpState &st, int32_t rounds, int32_t S) {
  const TierCache &T = g->tiers;
  if (st.seg.gid || S > 32 || T.lane_long ||
      T.count[TIER_BIG] + T.count[TIER_HUGE] > 0 ||
      (!g->unit_ew && (ew_sum_bound(g) >= ((int64_t)1 << 31) || st.nlabels > kLaneKeyLabels)))
    return 0;
  if (g->n > kLpSmallVertices * kLpSmallCluster || g->m2 > kLpSmallEntries * kLpSmallCluster ||
      !lp_small_pays(g, rounds, S))
    return 0;
  const int64_t items = (T.count[TIER_LANE] / 32 + T.count[TIER_SMALL] + T.count[TIER_MID]) / S;
  int cs = 1;
  while (cs < kLpSmallCluster && (cs * kLpSmallItems < items || g->n > kLpSmallVertices * cs)) cs <<= 1;
  return cs;
}

}  // namespace

bool lp_rounds_small(tp_graph *g, const LpState &st, LpWork &w, uint64_t seed, uint64_t tag,
                            uint64_t a, uint64_t b0, int32_t rounds, int32_t S, const tp_params &p,
                            cudaStream_t stream) {
  build_tiers(g, p, stream);
  int cs = lp_small_cluster(g, st, rounds, S);
  if (!cs) return false;
  auto kern = g->compressed ? k_lp_small<true, false>
              : g->unit_ew  ? k_lp_small<false, false>
                            : k_lp_small<false, true>;
  const size_t smem = sizeof(LpSmallWarp) * kLpSmallWarps + 4 * (size_t)kLpSmallVertices;
  static std::once_flag once;
  static int largest = 0;  // cluster the device can hold
  std::call_once(once, [&] {
    for (auto k : {k_lp_small<true, false>, k_lp_small<false, false>, k_lp_small<false, true>}) {
      TP_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      TP_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    }
    for (int c = kLpSmallCluster; c >= 1 && !largest; c >>= 1) {
      cudaLaunchConfig_t cfg{};
      cudaLaunchAttribute at[1];
      cfg.gridDim = dim3((unsigned)c), cfg.blockDim = dim3(kLpSmallThreads);
      cfg.dynamicSmemBytes = smem;
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = (unsigned)c, at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cfg.attrs = at, cfg.numAttrs = 1;
      int fit = 0;
      if (cudaOccupancyMaxActiveClusters(&fit, k_lp_small<false, true>, &cfg) == cudaSuccess && fit > 0)
        largest = c;
      else (void)cudaGetLastError();
    }
  });
  if (cs > largest && g->n > kLpSmallVertices * largest) return false;
  cs = std::min(cs, largest);
  if (cs < 1) return false;
  RateCtx c{};
  c.g = view(g);
  c.tier = g->tiers.tier.get();
  c.label = st.label;
  c.lw = st.lw;
  c.cap = st.cap;
  c.S = S;
  c.slack = 1;
  while (c.slack < std::max(1, std::min(8, p.table_slack))) c.slack <<= 1;
  c.mv_u = w.mv_u.get();
  c.mv_t = w.mv_t.get();
  c.mv_o = w.mv_o.get();
  c.mv_g = w.mv_g.get();
  c.in_w = w.in_w.get();
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[1];
  cfg.gridDim = dim3((unsigned)cs), cfg.blockDim = dim3(kLpSmallThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cs, at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at, cfg.numAttrs = 1;
  TP_CUDA(cudaLaunchKernelEx(&cfg, kern, c, approve_ctx(g, st, w), seed, tag, a, b0, rounds));
  count_launch();
  return true;
}

}  // namespace tp
