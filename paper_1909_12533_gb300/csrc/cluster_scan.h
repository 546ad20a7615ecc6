// Exclusive prefix sums over an index range by one cluster of CTAS CTAs: the
// values are computed where they are used (no array of counts in memory), the
// CTAs' totals pass through distributed shared memory, and the cluster's
// hardware barrier replaces the launches between the phases of a scan.
#pragma once
#include <cooperative_groups.h>

#include <cstdint>

namespace sp2 {

constexpr int SCAN_CTAS = 8;
constexpr int SCAN_THREADS = 1024;
constexpr int SCAN_ITEMS = 4;      // consecutive indices of a thread in one round

__device__ __forceinline__ int scan_block_excl(int v, int* total) {
  __shared__ int wsum[33];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wsum[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    const int s = wsum[lane];
    int si = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, si, o);
      if (lane >= o) si += y;
    }
    wsum[lane] = si - s;
    if (lane == 31) wsum[32] = si;
  }
  __syncthreads();
  const int r = inc - v + wsum[wid];
  *total = wsum[32];
  __syncthreads();
  return r;
}

// count(i) -> int for 0 <= i < n (called twice, by the same thread, with a
// cluster barrier between the two); emit(i, value, exclusive prefix).  Returns
// the total in every thread.  Launch: __cluster_dims__(SCAN_CTAS), SCAN_THREADS
// threads, one cluster.
template <class Count, class Emit>
__device__ __forceinline__ int cluster_scan(int64_t n, Count count, Emit emit) {
  namespace cg = cooperative_groups;
  __shared__ int tot[SCAN_CTAS];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  cl.barrier_arrive();      // every CTA has started before the first remote write (waited for below)
  constexpr int ROUND = SCAN_THREADS * SCAN_ITEMS;
  const int64_t len = ((n + SCAN_CTAS - 1) / SCAN_CTAS + ROUND - 1) / ROUND * ROUND;
  const int64_t c0 = min(n, rank * len), c1 = min(n, c0 + len);
  const int lane_item = (int)threadIdx.x * SCAN_ITEMS;
  int s = 0;
  for (int64_t base = c0; base < c1; base += ROUND)
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
      const int64_t i = base + lane_item + k;
      if (i < c1) s += count(i);
    }
  int mine;
  scan_block_excl(s, &mine);
  cl.barrier_wait();
  if (threadIdx.x < SCAN_CTAS) cl.map_shared_rank(tot, threadIdx.x)[rank] = mine;
  cl.sync();
  int carry = 0, all = 0;
  for (int r = 0; r < SCAN_CTAS; ++r) {
    if (r < rank) carry += tot[r];
    all += tot[r];
  }
  for (int64_t base = c0; base < c1; base += ROUND) {
    int v[SCAN_ITEMS], t = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
      const int64_t i = base + lane_item + k;
      v[k] = i < c1 ? count(i) : 0;
      t += v[k];
    }
    int block;
    int ex = carry + scan_block_excl(t, &block);
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
      const int64_t i = base + lane_item + k;
      if (i < c1) emit(i, v[k], ex);
      ex += v[k];
    }
    carry += block;
  }
  return all;
}

}  // namespace sp2
