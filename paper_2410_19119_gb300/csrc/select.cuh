// Weighted radix select by one thread block, shared by the approval of
// contested moves and the bisection kernel.
#pragma once
#include "tp_internal.cuh"

namespace tp {

// Finds, among cnt items with 96-bit keys (hi, lo) in ascending order, the
// first whose inclusive weight prefix exceeds rem and returns its key in
// (khi, klo) to every thread. item(q, hi, lo, w) yields item q. Every thread
// of the block must call it (whole warps). Called only when the total weight
// exceeds rem, so every pass selects a byte that some remaining key carries;
// bytes on which all keys agree are taken without a pass or a barrier.
// Bound by its barriers and by the search through the 256 bins, which one
// warp does with a scan (eight bins a lane): a thread walking the bins took
// about 4 us a pass at 2 GHz, most of the select for the usual few hundred
// items. narrow: all weights together fit 31 bits, and the bins are summed with
// native 32-bit shared atomics (the 64-bit ones retry, and most items of a
// large segment share a few bins).
template <class Item>
__device__ void block_select(int64_t cnt, int64_t rem, bool narrow, Item item, uint64_t &khi,
                             uint32_t &klo) {
  __shared__ unsigned long long hist[256];
  __shared__ int64_t s_cum;
  __shared__ int s_bin;
  __shared__ unsigned long long and_hi, or_hi;
  __shared__ unsigned and_lo, or_lo;
  if (threadIdx.x == 0) and_hi = ~0ull, or_hi = 0, and_lo = ~0u, or_lo = 0;
  __syncthreads();
  {  // bytes on which every key agrees need no histogram pass
    unsigned long long ah = ~0ull, oh = 0;
    unsigned al = ~0u, ol = 0;
    for (int64_t q = threadIdx.x; q < cnt; q += blockDim.x) {
      uint64_t hi;
      uint32_t lo;
      int64_t w;
      item(q, hi, lo, w);
      ah &= hi, oh |= hi, al &= lo, ol |= lo;
    }
    if ((int64_t)threadIdx.x < cnt)
      atomicAnd(&and_hi, ah), atomicOr(&or_hi, oh), atomicAnd(&and_lo, al), atomicOr(&or_lo, ol);
    __syncthreads();
  }
  const uint64_t ahi = and_hi, xhi = and_hi ^ or_hi;
  const uint32_t alo = and_lo, xlo = and_lo ^ or_lo;
  uint64_t fhi = 0, mhi = 0;
  uint32_t flo = 0, mlo = 0;
  int64_t cum = 0;
  for (int pass = 0; pass < 12; ++pass) {
    const bool in_hi = pass < 8;
    const int shift = in_hi ? 56 - 8 * pass : 24 - 8 * (pass - 8);
    uint32_t byte;
    if ((in_hi ? (uint32_t)(xhi >> shift) & 255u : (xlo >> shift) & 255u) == 0) {
      byte = in_hi ? (uint32_t)(ahi >> shift) & 255u : (alo >> shift) & 255u;
    } else {
      for (int b = threadIdx.x; b < 256; b += blockDim.x) hist[b] = 0;
      __syncthreads();
      for (int64_t q = threadIdx.x; q < cnt; q += blockDim.x) {
        uint64_t hi;
        uint32_t lo;
        int64_t w;
        item(q, hi, lo, w);
        if ((hi & mhi) != fhi || (lo & mlo) != flo) continue;
        const uint32_t d = in_hi ? (uint32_t)(hi >> shift) & 255u : (lo >> shift) & 255u;
        if (narrow) atomicAdd(reinterpret_cast<unsigned *>(&hist[d]), (unsigned)w);  // (its low half)
        else atomicAdd(&hist[d], (unsigned long long)w);
      }
      __syncthreads();
      if (threadIdx.x < 32) {  // first bin whose inclusive prefix exceeds rem (else the last)
        const int lane = threadIdx.x;
        int64_t v[8], sum = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = (int64_t)hist[8 * lane + j], sum += v[j];
        int64_t run = cum + warp_incl_scan(sum) - sum;
        const unsigned over = __ballot_sync(kFull, run + sum > rem);
        const int owner = over ? __ffs(over) - 1 : 31;
        if (lane == owner) {
          int j = 0;
#pragma unroll
          for (int i = 0; i < 7; ++i) {
            if (j == i && run + v[i] <= rem) run += v[i], ++j;
          }
          s_bin = 8 * lane + j;
          s_cum = run;
        }
      }
      __syncthreads();
      byte = (uint32_t)s_bin;
      cum = s_cum;
    }
    if (in_hi) fhi |= (uint64_t)byte << shift, mhi |= 255ull << shift;
    else flo |= byte << shift, mlo |= 255u << shift;
  }
  khi = fhi;
  klo = flo;
  __syncthreads();  // the shared words are reused by the next call
}

}  // namespace tp
