// Truncation X~_i = X_i + E_i with ||E_i|| <= tau_i (Section 2, Eqs. (6)-(8)).
//
// Selection rule (the paper states only the bound, so this is a reading):
//  - Frobenius mode: sort the tiles by (||X_IJ||_F^2, I * nb + J) ascending and drop
//    the longest prefix whose weighted squared norms fit into tau^2; weight 2 for
//    off-diagonal tiles (their mirror is dropped too), 1 for diagonal tiles.
//  - Frob-Inf mode (Section 3, Eq. (13), square partition of `part` rows): every
//    super-block (R, C) gets the budget tau / max(m_R, m_C), m_R = number of
//    nonzero super-blocks in super-row R; the Frobenius rule runs inside each
//    super-block (weight 2 only for off-diagonal tiles of diagonal super-blocks).
//    Then every super-row sum of ||E_RC||_F is <= tau, so ||E||_2 <= ||E||_M <= tau.
//  - Sums are taken in integer units of budget * 2^-36 with each tile's share
//    rounded up, so they are exact, independent of summation order, and never
//    understate ||E||_F^2.
//
// GPU form: a segmented most-significant-digit radix select over the 96-bit key
// (the squared norm's IEEE pattern -- non-negative doubles order like their bit
// patterns -- then the 32-bit linear tile index), one cluster of CL_CTAS CTAs
// per segment.  Each pass histograms the budget units of the remaining
// candidates in shared memory, the CTAs sum the bins through distributed shared
// memory and find the bucket in which the budget ends.  The cluster's hardware
// barrier orders the passes, so a selection is one launch; it ends as soon as
// one candidate is left, usually after three of the nine passes.  (A memset, a
// histogram and a one-thread-per-segment bucket walk for each of twelve 8-bit
// passes were 36 launches; one truncation of 180,300 device tiles, norms
// included, took 1.46 ms and takes 0.58 ms.)
// A single segment of at most 2048 tiles runs in one CTA.
#include <cmath>
#include <vector>

#include <cooperative_groups.h>

#include "sp2_internal.h"

namespace cg = cooperative_groups;

namespace sp2 {
namespace {

constexpr double Q_SCALE = 68719476736.0;          // 2^36
constexpr unsigned long long Q_BUDGET = 1ull << 36;
constexpr unsigned long long Q_CAP = 1ull << 37;
constexpr int MIXED_POWER_ITERS = 100;        // power steps of the mixed-norm bound

struct Work {
  unsigned long long* q;   // budget units of each tile
  double* scale;           // Frob-Inf: units per squared norm of each segment
  int32_t* nz;             // [nsb x nsb] pairs of super-rows with a tile, and one word behind them:
                           // set when the tiles are not sorted upper tiles
  int32_t* m;
  int64_t nseg;
  int32_t nsb;
};

inline size_t align_up(size_t x) { return (x + 255) & ~size_t(255); }

inline size_t nz_bytes(int nsb) { return ((size_t)nsb * nsb + 1) * 4; }

Work carve(void* base, int64_t nnzb, int64_t nseg, int nsb) {
  char* p = static_cast<char*>(base);
  Work w;
  w.q = reinterpret_cast<unsigned long long*>(p); p += align_up(nnzb * 8);
  w.scale = reinterpret_cast<double*>(p); p += align_up(nseg * 8);
  w.nz = reinterpret_cast<int32_t*>(p); p += align_up(nz_bytes(nsb));
  w.m = reinterpret_cast<int32_t*>(p); p += align_up((size_t)nsb * 4);
  w.nseg = nseg;
  w.nsb = nsb;
  return w;
}

// (segment indices R * nsb + C pass 2^31 from 46,341 super-blocks on: 64-bit)
__global__ void k_nz(const int32_t* __restrict__ brow, const int32_t* __restrict__ bcol, int64_t nnzb, int pt,
                     int nsb, int32_t* nz) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nnzb) return;
  const int R = brow[t] / pt, C = bcol[t] / pt;
  nz[(int64_t)R * nsb + C] = 1;
  nz[(int64_t)C * nsb + R] = 1;
  if (bcol[t] < brow[t] || (t > 0 && brow[t - 1] > brow[t])) nz[(int64_t)nsb * nsb] = 1;
}

__global__ void k_m(const int32_t* __restrict__ nz, int nsb, int32_t* m) {
  const int R = blockIdx.x * blockDim.x + threadIdx.x;
  if (R >= nsb) return;
  int c = 0;
  for (int C = 0; C < nsb; ++C) c += nz[(int64_t)R * nsb + C];
  m[R] = c;
}

// Frob-Inf: units per squared norm of segment R * nsb + C
__global__ void k_seg_scale(Work w, double tau) {
  const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (s >= w.nseg) return;
  const int R = (int)(s / w.nsb), C = (int)(s % w.nsb);
  const int mm = max(w.m[R], w.m[C]);
  const double beta = mm > 0 ? tau / (double)mm : 0.0;
  const double budget = beta * beta;
  w.scale[s] = budget > 0.0 ? Q_SCALE / budget : 0.0;
}

// budget units of a tile of squared norm v and weight wt (1: stored once, 2: mirrored),
// rounded up, at most Q_CAP, which no budget holds: also for a NaN (a tile with a
// NaN, a norm that was never computed), so that the sums of a selection stay
// below 2^64 (2^27 tiles are a terabyte) and exactly one bin holds its cut.  A NaN
// converted to an integer would be 2^63 units, a wrapped sum would let several
// CTAs of a cluster name a cut, and one could leave while another still reads
// its shared memory.  A zero tile has no units, whatever the scale (infinite
// for a tau whose square is subnormal).  The comparisons are made on the bit
// patterns (those of 2^37 and above, of NaN and of negative values are not below
// that of 2^37): the FP64 pipe compares two lanes a cycle.
__device__ __forceinline__ unsigned long long budget_units(double v, double wt, double sc) {
  const unsigned long long x = (unsigned long long)__double_as_longlong((wt * v) * sc);
  if (((unsigned long long)__double_as_longlong(v) << 1) == 0ull) return 0ull;
  if (((unsigned long long)__double_as_longlong(sc) << 1) == 0ull || x >= (1023ull + 37ull) << 52) return Q_CAP;
  return __double2ull_ru(__longlong_as_double((long long)x));
}

// mode 0: one segment, scale sc; mode 1: the segment's scale.  Its own launch
// over all SMs: the FP64 pipe (2 lanes per SM cycle) is too slow for it to sit
// in the few CTAs of the selection.
__global__ void k_q(const int32_t* __restrict__ brow, const int32_t* __restrict__ bcol,
                    const int32_t* __restrict__ slot, const double* __restrict__ n2, int64_t nnzb, int mode, int pt,
                    double sc, Work w) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nnzb) return;
  const int I = brow[t], J = bcol[t];
  double wt = (I == J) ? 1.0 : 2.0;
  if (mode == 1) {
    const int R = I / pt, C = J / pt;
    sc = w.scale[(int64_t)R * w.nsb + C];
    if (R != C) wt = 1.0;
  }
  w.q[t] = budget_units(n2[slot ? slot[t] : t], wt, sc);
}

__device__ __forceinline__ bool is_candidate(unsigned long long hi, uint32_t lo, int p, unsigned long long ph,
                                             uint32_t pl) {
  if (p == 0) return true;
  if (p <= 8) return (hi >> (64 - 8 * p)) == ph;
  return hi == ph && (lo >> (32 - 8 * (p - 8))) == pl;
}

__device__ __forceinline__ int digit_of(unsigned long long hi, uint32_t lo, int p) {
  if (p < 8) return (int)((hi >> (56 - 8 * p)) & 0xFFull);
  return (int)((lo >> (24 - 8 * (p - 8))) & 0xFFu);
}

// Radix select of one segment per cluster (mode 1: grid (nsb clusters, nsb),
// segment (R, C), R <= C, of the upper triangle of nsb x nsb super-blocks).
// The tiles are sorted by row, so the segment's tiles lie in the range of its
// super-row (all of them in mode 0); the CTAs of the cluster split that range.
// Tiles in another order, or below the diagonal, are no sp2_bsr, but a selection
// needs neither: with such a tile every segment reads the whole set, and
// those with R > C take part.
// Digits: the 12 bits of sign and exponent first (a tile set spans some 100
// octaves, so the shared-memory atomics of a warp rarely meet in one bin),
// 11 bits at a time after that.
// Two sizes: CL_CTAS x 1024 threads for segments of many tiles, one CTA of 256
// threads for small ones (Frob-Inf with a small partition has thousands, most
// of them without a tile, which leave at once, and most others with one tile or
// within their budget, or with few tiles, which need no histogram: one
// truncation of 178,230 tiles of a band in 3,000 x 3,000 segments takes 14.9 ms,
// in 750 x 750 1.4, of 131,328 tiles of a dense matrix in 256 x 256 0.8; with a
// histogram for every pair of super-rows 139.8, 9.9 and 2.5).
constexpr int CL_CTAS = 8;
constexpr int64_t CL_MANY = 4096;   // tiles of a segment (mean) from which the cluster is taken
// Tiles of a segment up to which the one-CTA select compares them with one
// another: 131,328 tiles in segments of 16 take 0.56 ms (1.06 with histograms),
// 8,256 tiles in segments of up to 256 128 us (111).
constexpr int DIRECT_MAX = 64;
// Mean tiles of a segment up to which that select sums its segment first; the sum
// reads the range once more (25,050 tiles in 55 segments: 152 us with it, 146).
constexpr int64_t SUM_FIRST_MAX = 256;
constexpr int CL_BINS = 4096;
constexpr int CL_PASSES = 9;      // 6 over the norm (52, 41, 30, 19, 8, 0), 3 over the index (21, 10, 0)
constexpr size_t CL_SMEM = (size_t)CL_BINS * 12;
constexpr int MLP = 4;            // norms of a thread loaded at once

__device__ __forceinline__ int cl_shift(int p) {
  return p < 5 ? 52 - 11 * p : p == 5 ? 0 : p == 6 ? 21 : p == 7 ? 10 : 0;
}

__device__ __forceinline__ int64_t first_row_ge(const int32_t* __restrict__ brow, int64_t n, int row) {
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (brow[mid] < row) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Adds a candidate's units q to its bin d.  Up to four bins that `share` or more of
// the candidates in the warp (the lanes that call this together) have take one
// addition each; the search ends at the first bin that fewer have.  The tiles of
// a periodic system have equal norms, and then all additions of a pass meet in a
// few bins.  One truncation without it, with it: 119,990 equal tiles 3.6 ms, 0.54;
// 888,825 equal tiles 27.7, 3.2; 178,230 tiles of random norms 0.537, 0.539.
__device__ __forceinline__ void hist_add(unsigned long long* hist, uint32_t* cnt, uint32_t d, unsigned long long q, int share) {
  const unsigned act = __activemask();
  const int lane = threadIdx.x & 31;
  unsigned left = act;
  bool alone = true;
  for (int r = 0; r < 4 && left != 0u; ++r) {
    const int lead = __ffs(left) - 1;
    const uint32_t d0 = __shfl_sync(act, d, lead);
    const unsigned peers = __ballot_sync(act, d == d0);
    if (__popc(peers) < share) break;
    left &= ~peers;
    if (d == d0) {
      const unsigned lo = __reduce_add_sync(peers, (unsigned)q & 0x7FFFFu);      // q <= 2^37: both sums fit
      const unsigned hi = __reduce_add_sync(peers, (unsigned)(q >> 19));
      if (lane == lead) {
        atomicAdd(&hist[d], ((unsigned long long)hi << 19) + lo);
        atomicAdd(&cnt[d], (uint32_t)__popc(peers));
      }
      alone = false;
    }
  }
  if (alone) {
    atomicAdd(&hist[d], q);
    atomicAdd(&cnt[d], 1u);
  }
}

template <int CTAS, int THREADS>
__global__ void __cluster_dims__(CTAS, 1, 1) __launch_bounds__(THREADS, 1024 / THREADS)
    k_trunc_cluster(const int32_t* __restrict__ brow, const int32_t* __restrict__ bcol,
                    const int32_t* __restrict__ slot, const double* __restrict__ n2,
                    const unsigned long long* __restrict__ q, const int32_t* __restrict__ nz, int64_t nnzb, int nb,
                    int mode, int pt, int nsb, int sum_first, int32_t* keep) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  unsigned long long* hist = reinterpret_cast<unsigned long long*>(cl_smem);   // [CL_BINS] units
  uint32_t* cnt = reinterpret_cast<uint32_t*>(hist + CL_BINS);                 // [CL_BINS] candidates
  __shared__ unsigned long long tot[CTAS];     // units in the bins of each CTA's share
  __shared__ unsigned long long wsum[32];
  __shared__ unsigned long long s_rem;            // budget left below the cut bucket
  __shared__ int s_cut, s_cnt;
  __shared__ int64_t range[2];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int C = 0, row0 = -1;      // the segment's super-column; its first row where the range does not say it
  auto inside = [&](int64_t t) {
    return bcol[t] / pt == C && (row0 < 0 || (unsigned)(brow[t] - row0) < (unsigned)pt);
  };
  if (mode == 1) {
    const int R = (int)blockIdx.y;
    C = (int)(blockIdx.x / CTAS);
    const bool has = nz[(int64_t)R * nsb + C] != 0, any_order = nz[(int64_t)nsb * nsb] != 0;
    if (!has || (C < R && !any_order)) return;     // the whole cluster
    if (any_order) row0 = R * pt;
    if (tid < 2) range[tid] = any_order ? tid * nnzb : first_row_ge(brow, nnzb, (R + tid) * pt);
  } else if (tid == 0) {
    range[0] = 0;
    range[1] = nnzb;
  }
  __syncthreads();
  const int64_t len = (range[1] - range[0] + CTAS - 1) / CTAS;
  const int64_t c0 = range[0] + rank * len, c1 = min(range[1], c0 + len);
  constexpr int SHARE = CL_BINS / CTAS;        // bins a CTA sums over the cluster
  constexpr int PER = SHARE > THREADS ? SHARE / THREADS : 1;
  unsigned long long ph = 0ull, rem = Q_BUDGET;
  uint32_t pl = 0u;
  int depth = 0;       // digits fixed in (ph, pl)
  bool all = false;    // every remaining candidate fits
  bool open = true;    // the cut is still to be found
  if (CTAS == 1 && sum_first) {
    // the segment's units and tiles: all fit, or the only one does not
    unsigned long long s = 0ull;
    uint32_t n = 0u;
    for (int64_t t = c0 + tid; t < c1; t += THREADS)
      if (inside(t)) {
        s += q[t];
        ++n;
      }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) {
      wsum[wid] = s;
      cnt[wid] = n;
    }
    __syncthreads();
    s = 0ull;
    n = 0u;
    for (int k = 0; k < THREADS / 32; ++k) {
      s += wsum[k];
      n += cnt[k];
    }
    all = s <= rem;
    open = !all && n > 1u;
    if (open && n <= (uint32_t)DIRECT_MAX) {
      // few tiles: each thread adds up the units of the tiles that are not behind
      // its own in the order of the keys
      unsigned long long* th = hist;                   // squared norms
      unsigned long long* tq = hist + DIRECT_MAX;      // units
      uint32_t* tl = cnt + DIRECT_MAX;                 // linear tile indices
      uint32_t* tt = cnt + 2 * DIRECT_MAX;             // tiles
      if (tid == 0) s_cnt = 0;
      __syncthreads();
      for (int64_t t = c0 + tid; t < c1; t += THREADS)
        if (inside(t)) {
          const int k = atomicAdd(&s_cnt, 1);
          th[k] = (unsigned long long)__double_as_longlong(n2[slot ? slot[t] : t]);
          tq[k] = q[t];
          tl[k] = (uint32_t)brow[t] * (uint32_t)nb + (uint32_t)bcol[t];
          tt[k] = (uint32_t)t;
        }
      __syncthreads();
      if (tid < (int)n) {
        const unsigned long long hi = th[tid];
        const uint32_t lo = tl[tid];
        unsigned long long sum = 0ull;
        for (uint32_t k = 0; k < n; ++k)
          if (th[k] < hi || (th[k] == hi && tl[k] <= lo)) sum += tq[k];
        keep[tt[tid]] = sum <= rem ? 0 : 1;
      }
      return;
    }
    __syncthreads();
  }
  for (int p = 0; open && p < CL_PASSES; ++p) {
    for (int k = tid; k < CL_BINS; k += THREADS) {
      hist[k] = 0ull;
      cnt[k] = 0u;
    }
    __syncthreads();
    const int sh = cl_shift(p), psh = p > 0 ? cl_shift(p - 1) : 0;
    const uint32_t dm = p == 0 ? 0xFFFu : p == 5 ? 0xFFu : p == 8 ? 0x3FFu : 0x7FFu;
    for (int64_t t0 = c0 + tid; t0 < c1; t0 += MLP * THREADS) {
      unsigned long long h[MLP];
#pragma unroll
      for (int u = 0; u < MLP; ++u) {
        const int64_t t = t0 + u * THREADS;
        h[u] = t < c1 ? (unsigned long long)__double_as_longlong(n2[slot ? slot[t] : t]) : 0ull;
      }
#pragma unroll
      for (int u = 0; u < MLP; ++u) {
        const int64_t t = t0 + u * THREADS;
        const unsigned long long hi = h[u];
        uint32_t lo = 0u;
        bool in = t < c1;
        if (p > 0 && p <= 6) in = in && (hi >> psh) == ph;
        if (p > 6) in = in && hi == ph;
        if (in && p >= 6) {
          lo = (uint32_t)brow[t] * (uint32_t)nb + (uint32_t)bcol[t];
          if (p > 6) in = (lo >> psh) == pl;
        }
        if (in && mode == 1) in = inside(t);
        if (in) hist_add(hist, cnt, (p < 6 ? (uint32_t)(hi >> sh) : lo >> sh) & dm, q[t], p == 0 ? 8 : 4);
      }
    }
    cl.sync();
    // this CTA's share of the bins, summed over the cluster (PER bins a thread),
    // and its prefix sums
    unsigned long long v = 0ull, bv[PER];
    uint32_t bc[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      bv[j] = 0ull;
      bc[j] = 0u;
      if (tid * PER < SHARE) {
        for (int r = 0; r < CTAS; ++r) {
          bv[j] += cl.map_shared_rank(hist, r)[rank * SHARE + tid * PER + j];
          bc[j] += cl.map_shared_rank(cnt, r)[rank * SHARE + tid * PER + j];
        }
      }
      v += bv[j];
    }
    unsigned long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    unsigned long long below = 0ull, mine = 0ull;
    for (int k = 0; k < THREADS / 32; ++k) {
      if (k < wid) below += wsum[k];
      mine += wsum[k];
    }
    if (tid < CTAS) cl.map_shared_rank(tot, tid)[rank] = mine;
    cl.sync();
    unsigned long long before = below + inc - v, grand = 0ull;
    for (int r = 0; r < CTAS; ++r) {
      if (r < rank) before += tot[r];
      grand += tot[r];
    }
    if (grand <= rem) {      // the same in every thread of the cluster
      all = true;
      break;
    }
    // the one bucket in which the budget ends
    if (before <= rem && before + v > rem) {
      bool here = true;
#pragma unroll
      for (int j = 0; j < PER; ++j) {
        if (here && before + bv[j] > rem) {
          for (int r = 0; r < CTAS; ++r) {
            *cl.map_shared_rank(&s_rem, r) = rem - before;
            *cl.map_shared_rank(&s_cut, r) = rank * SHARE + tid * PER + j;
            *cl.map_shared_rank(&s_cnt, r) = (int)bc[j];
          }
          here = false;
        }
        before += bv[j];
      }
    }
    cl.sync();
    rem = s_rem;
    if (p == 0) ph = (unsigned long long)s_cut;
    else if (p < 5) ph = (ph << 11) | (unsigned long long)s_cut;
    else if (p == 5) ph = (ph << 8) | (unsigned long long)s_cut;
    else if (p == 6) pl = (uint32_t)s_cut;
    else if (p == 7) pl = (pl << 11) | (uint32_t)s_cut;
    else pl = (pl << 10) | (uint32_t)s_cut;
    depth = p + 1;
    if (s_cnt == 1) break;   // the bucket's only candidate is the first tile that does not fit
  }
  // dropped: keys below the prefix; the prefix's own bucket only when everything fits
  const int dsh = depth > 0 ? cl_shift(depth - 1) : 0;
#pragma unroll 4
  for (int64_t t = c0 + tid; t < c1; t += THREADS) {
    if (mode == 1 && !inside(t)) continue;
    const unsigned long long hi = __double_as_longlong(n2[slot ? slot[t] : t]);
    bool less, equal;
    if (depth == 0) {
      less = false;
      equal = true;
    } else if (depth <= 6) {
      less = (hi >> dsh) < ph;
      equal = (hi >> dsh) == ph;
    } else {
      const uint32_t lo = ((uint32_t)brow[t] * (uint32_t)nb + (uint32_t)bcol[t]) >> dsh;
      less = hi < ph || (hi == ph && lo < pl);
      equal = hi == ph && lo == pl;
    }
    keep[t] = (less || (equal && all)) ? 0 : 1;
  }
}

// One CTA for a single segment of at most SMALL_MAX tiles: twelve 8-bit passes
// with keys and units held in shared memory, one launch.  All sums are the same
// exact integers, so the keep flags equal the cluster's.
constexpr int SMALL_MAX = 2048;
constexpr int SMALL_THREADS = 1024;

__global__ void __launch_bounds__(SMALL_THREADS)
    k_trunc_small(const int32_t* __restrict__ brow, const int32_t* __restrict__ bcol,
                  const int32_t* __restrict__ slot, const double* __restrict__ n2, int n, int nb, double budget,
                  int32_t* keep) {
  __shared__ unsigned long long s_hi[SMALL_MAX];
  __shared__ unsigned long long s_q[SMALL_MAX];
  __shared__ uint32_t s_lo[SMALL_MAX];
  __shared__ unsigned long long hist[256];
  __shared__ unsigned long long s_rem, s_ph;
  __shared__ uint32_t s_pl;
  __shared__ int s_state, s_depth;
  const double sc = budget > 0.0 ? Q_SCALE / budget : 0.0;
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const int I = brow[t], J = bcol[t];
    const double v = n2[slot ? slot[t] : t];
    s_hi[t] = __double_as_longlong(v);
    s_lo[t] = (uint32_t)I * (uint32_t)nb + (uint32_t)J;
    s_q[t] = budget_units(v, (I == J) ? 1.0 : 2.0, sc);
  }
  if (threadIdx.x == 0) {
    s_rem = Q_BUDGET;
    s_ph = 0ull;
    s_pl = 0u;
    s_state = 0;
    s_depth = 0;
  }
  for (int p = 0; p < 12; ++p) {
    for (int k = threadIdx.x; k < 256; k += blockDim.x) hist[k] = 0ull;
    __syncthreads();
    if (s_state != 0) break;
    const unsigned long long ph = s_ph;
    const uint32_t pl = s_pl;
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
      const unsigned long long hi = s_hi[t];
      const uint32_t lo = s_lo[t];
      if (is_candidate(hi, lo, p, ph, pl)) atomicAdd(&hist[digit_of(hi, lo, p)], s_q[t]);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      // bucket walk: lane l owns buckets 8l..8l+7, an inclusive
      // scan over the lanes finds the lane holding the cut
      const int lane = threadIdx.x;
      unsigned long long loc[8], sum = 0ull;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        loc[j] = hist[lane * 8 + j];
        sum += loc[j];
      }
      unsigned long long inc = sum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const unsigned long long v = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += v;
      }
      const unsigned long long rem = s_rem;
      const unsigned bal = __ballot_sync(0xffffffffu, inc > rem);
      if (bal == 0u) {
        if (lane == 0) {
          s_state = 1;      // every candidate fits
          s_depth = p;
        }
      } else if (lane == __ffs(bal) - 1) {
        unsigned long long r = rem - (inc - sum);
        int cut = 8 * lane + 7;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (loc[j] <= r) {
            r -= loc[j];
          } else {
            cut = 8 * lane + j;
            break;
          }
        }
        s_rem = r;
        if (p < 8) s_ph = (ph << 8) | (unsigned long long)cut;
        else s_pl = (pl << 8) | (uint32_t)cut;
      }
    }
    __syncthreads();
  }
  __syncthreads();
  const unsigned long long ph = s_ph;
  const uint32_t pl = s_pl;
  const int state = s_state, dep = s_depth;
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const unsigned long long hi = s_hi[t];
    const uint32_t lo = s_lo[t];
    bool drop;
    if (state == 1) {
      if (dep == 0) drop = true;
      else if (dep <= 8) drop = (hi >> (64 - 8 * dep)) <= ph;
      else drop = hi < ph || (hi == ph && (lo >> (32 - 8 * (dep - 8))) <= pl);
    } else {
      drop = hi < ph || (hi == ph && lo < pl);
    }
    keep[t] = drop ? 0 : 1;
  }
}

// ||tile||_F^2 of contiguous tiles, one warp per tile: lane l, j = 0..7, sums the
// elements l + 32 j + 256 k over k in order, then a fixed tree over j and the
// lanes.  All 32 loads of a lane are in flight at once; the FP64 pipe (1,408
// lane operations a tile at 2 per SM cycle, 0.42 ms for 180,300 tiles) bounds it, not
// HBM (0.22 ms).
constexpr int NORM_WARPS = 8;
__global__ void __launch_bounds__(32 * NORM_WARPS) k_tile_norms(const double* __restrict__ val, int64_t nnzb, double* n2) {
  const int64_t t = (int64_t)blockIdx.x * NORM_WARPS + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (t >= nnzb) return;
  const double* x = val + t * TE + lane;
  double v[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = x[32 * i];
  double a[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    a[j] = v[j] * v[j];
#pragma unroll
    for (int k = 1; k < 4; ++k) a[j] = fma(v[j + 8 * k], v[j + 8 * k], a[j]);
  }
#pragma unroll
  for (int h = 4; h > 0; h >>= 1)
#pragma unroll
    for (int j = 0; j < h; ++j) a[j] += a[j + h];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a[0] += __shfl_down_sync(0xffffffffu, a[0], o);
  if (lane == 0) n2[t] = a[0];
}

inline unsigned grid_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }


// ---------------------------------------------------------------- mixed norm
// Frobenius-spectral mixed norm of Section 3 on a partition of pt tiles:
// every tile gets its budget units q (weight 2 for an off-diagonal tile inside
// a diagonal block, units of tau^2 2^-36 rounded up, capped), the pattern of
// its squared norm (non-negative doubles order like their bit patterns) and
// its block index R * nsb + C.
__global__ void k_mixed_prep(const int32_t* __restrict__ brow, const int32_t* __restrict__ bcol,
                             const int32_t* __restrict__ slot, const double* __restrict__ n2, int64_t nnzb, int pt,
                             int nsb, double sc, unsigned long long* q, long long* bits, int32_t* blk) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nnzb) return;
  const int I = brow[t], J = bcol[t];
  const int R = I / pt, C = J / pt;
  const double wt = (R == C && I != J) ? 2.0 : 1.0;
  const double v = n2[slot ? slot[t] : t];
  const double x = (wt * v) * sc;
  q[t] = (x >= (double)Q_CAP) ? Q_CAP : (unsigned long long)ceil(x);
  bits[t] = __double_as_longlong(v);
  blk[t] = R * nsb + C;
}

// Block sums of the units of the tiles with bits <= theta (and the mirror block
// for R != C), exact integer atomics; cnt[0] counts the tiles with
// lo < bits <= hi (the bisection ends when none is left between its ends).
__global__ void k_mixed_probe(const unsigned long long* __restrict__ q, const long long* __restrict__ bits,
                              const int32_t* __restrict__ blk, int64_t nnzb, int nsb, long long theta, long long lo,
                              long long hi, unsigned long long* B2, unsigned long long* cnt) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  bool between = false;
  if (t < nnzb) {
    const long long b = bits[t];
    between = b > lo && b <= hi;
    if (b <= theta && q[t] != 0ull) {
      const int k = blk[t];
      const int R = k / nsb, C = k % nsb;
      atomicAdd(&B2[k], q[t]);
      if (R != C) atomicAdd(&B2[C * nsb + R], q[t]);
    }
  }
  const unsigned nb = __popc(__ballot_sync(0xffffffffu, between));
  if ((threadIdx.x & 31) == 0 && nb) atomicAdd(cnt, (unsigned long long)nb);
}

__global__ void k_mixed_keep(const long long* __restrict__ bits, int64_t nnzb, long long theta, int32_t* keep) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < nnzb) keep[t] = bits[t] <= theta ? 0 : 1;
}

}  // namespace

cudaError_t launch_tile_norms(const double* val, int64_t nnzb, double* n2, cudaStream_t st) {
  if (nnzb == 0) return cudaSuccess;
  { ++g_launches; k_tile_norms<<<grid_for(nnzb, NORM_WARPS), 32 * NORM_WARPS, 0, st>>>(val, nnzb, n2); }
  return cudaGetLastError();
}

size_t trunc_work_bytes(int64_t nnzb, int nb, int64_t part_tiles) {
  const int nsb = (int)((nb + part_tiles - 1) / part_tiles);
  const int64_t nseg = (int64_t)nsb * nsb;
  return align_up(nnzb * 8) + align_up(nseg * 8) + align_up(nz_bytes(nsb)) + align_up((size_t)nsb * 4) + 1024;
}

// x: the tiles of X_i (slot indexes n2); n2[slot] = ||X_i tile||_F^2; keep[t] out.
cudaError_t launch_truncate(const TileSet& x, const double* n2, int nb, double tau, int mode, int64_t part_tiles,
                            void* work, int32_t* keep, cudaStream_t st) {
  const int64_t nnzb = x.nnzb;
  if (nnzb == 0) return cudaSuccess;
  const int nsb = (int)((nb + part_tiles - 1) / part_tiles);
  const int64_t nseg = mode == 1 ? (int64_t)nsb * nsb : 1;
  if (nseg == 1 && nnzb <= SMALL_MAX) {
    // one segment: mode 1 with a single super-block has m = 1, so its budget is tau^2 too
    { ++g_launches; k_trunc_small<<<1, SMALL_THREADS, 0, st>>>(x.brow, x.bcol, x.slot, n2, (int)nnzb, nb, tau * tau, keep); }
    return cudaGetLastError();
  }
  Work w = carve(work, nnzb, nseg, nsb);
  const int md = nseg == 1 ? 0 : 1;   // mode 1 with a single super-block has m = 1: budget tau^2 as in mode 0
  double sc = 0.0;
  if (md == 1) {
    const cudaError_t e = cudaMemsetAsync(w.nz, 0, nz_bytes(nsb), st);
    if (e != cudaSuccess) return e;
    { ++g_launches; k_nz<<<grid_for(nnzb, 256), 256, 0, st>>>(x.brow, x.bcol, nnzb, (int)part_tiles, nsb, w.nz); }
    { ++g_launches; k_m<<<grid_for(nsb, 128), 128, 0, st>>>(w.nz, nsb, w.m); }
    { ++g_launches; k_seg_scale<<<grid_for(nseg, 256), 256, 0, st>>>(w, tau); }
  } else {
    const double budget = tau * tau;
    sc = budget > 0.0 ? Q_SCALE / budget : 0.0;
  }
  { ++g_launches; k_q<<<grid_for(nnzb, 256), 256, 0, st>>>(x.brow, x.bcol, x.slot, n2, nnzb, md, (int)part_tiles, sc, w); }
  const int64_t nclus = md == 1 ? (int64_t)nsb * (nsb + 1) / 2 : 1;
  const unsigned side = md == 1 ? (unsigned)nsb : 1u;
  auto launch = [&](auto kernel, int ctas, int threads) -> cudaError_t {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CL_SMEM);
    if (e != cudaSuccess) return e;
    ++g_launches;
    kernel<<<dim3(side * ctas, side), threads, CL_SMEM, st>>>(x.brow, x.bcol, x.slot, n2, w.q, w.nz, nnzb, nb, md,
                                                               (int)part_tiles, nsb,
                                                               nnzb <= SUM_FIRST_MAX * nclus ? 1 : 0, keep);
    return cudaGetLastError();
  };
  return nnzb >= CL_MANY * nclus || nclus == 1 ? launch(k_trunc_cluster<CL_CTAS, 1024>, CL_CTAS, 1024)
                                               : launch(k_trunc_cluster<1, 256>, 1, 256);
}

}  // namespace sp2

namespace sp2 {

// Collatz-Wielandt upper bound of rho(M), M = sqrt(B2) (nsb x nsb, symmetric,
// non-negative): rows that are all zero are skipped; x starts at all ones and
// MIXED_POWER_ITERS times takes u = max_i (M x)_i / x_i, then x = (M x + u x)
// / max(M x + u x); the smallest u is returned.  Sequential row sums without
// fused multiply-adds.
double mixed_norm_bound_host(const unsigned long long* B2, int nsb) {
  std::vector<int> live;
  for (int i = 0; i < nsb; ++i) {
    bool nz = false;
    for (int j = 0; j < nsb && !nz; ++j) nz = B2[(size_t)i * nsb + j] != 0ull;
    if (nz) live.push_back(i);
  }
  const int m = (int)live.size();
  if (m == 0) return 0.0;
  std::vector<double> M((size_t)m * m), x(m, 1.0), y(m);
  for (int a = 0; a < m; ++a)
    for (int b = 0; b < m; ++b) M[(size_t)a * m + b] = std::sqrt((double)B2[(size_t)live[a] * nsb + live[b]]);
  double best = INFINITY;
  for (int it = 0; it < MIXED_POWER_ITERS; ++it) {
    for (int a = 0; a < m; ++a) {
      double acc = 0.0;
      for (int b = 0; b < m; ++b) {
        const double prod = M[(size_t)a * m + b] * x[b];
        acc = acc + prod;
      }
      y[a] = acc;
    }
    double u = 0.0;
    for (int a = 0; a < m; ++a) u = std::max(u, y[a] / x[a]);
    best = std::min(best, u);
    double mx = 0.0;
    for (int a = 0; a < m; ++a) {
      const double ux = u * x[a];
      y[a] = y[a] + ux;
      mx = std::max(mx, y[a]);
    }
    for (int a = 0; a < m; ++a) x[a] = y[a] / mx;
  }
  return best;
}

size_t mixed_work_bytes(int64_t nnzb, int nsb) {
  return align_up((size_t)nnzb * 8) * 2 + align_up((size_t)nnzb * 4) + align_up((size_t)nsb * nsb * 8) + 256;
}

// keep[t] for the mixed-norm selection (see the oracle's reading): bisection
// over the 63-bit patterns of the squared norms for the largest theta whose
// dropped set has a bound of at most tau (in units: 2^18); each probe is one
// kernel and a host round trip; the bisection stops early once no tile lies
// between its ends.  Synchronises the stream.
cudaError_t mixed_select(const TileSet& x, const double* n2, int nb, double tau, int64_t part_tiles, void* work,
                         int32_t* keep, cudaStream_t st) {
  const int64_t nnzb = x.nnzb;
  if (nnzb == 0) return cudaSuccess;
  const int pt = (int)part_tiles;
  const int nsb = (int)((nb + pt - 1) / pt);
  char* p = static_cast<char*>(work);
  unsigned long long* q = reinterpret_cast<unsigned long long*>(p); p += align_up((size_t)nnzb * 8);
  long long* bits = reinterpret_cast<long long*>(p); p += align_up((size_t)nnzb * 8);
  int32_t* blk = reinterpret_cast<int32_t*>(p); p += align_up((size_t)nnzb * 4);
  unsigned long long* B2 = reinterpret_cast<unsigned long long*>(p); p += align_up((size_t)nsb * nsb * 8);
  unsigned long long* cnt = reinterpret_cast<unsigned long long*>(p);
  const unsigned g = grid_for(nnzb, 256);
  const double sc = tau > 0.0 ? Q_SCALE / (tau * tau) : 0.0;
  ++g_launches;
  k_mixed_prep<<<g, 256, 0, st>>>(x.brow, x.bcol, x.slot, n2, nnzb, pt, nsb, sc, q, bits, blk);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // tau = 0 keeps lo = 0: only tiles that are exactly zero are dropped
  long long lo = 0, hi = 0x7FFFFFFFFFFFFFFFll;
  if (tau > 0.0) {
    std::vector<unsigned long long> h((size_t)nsb * nsb + 1);
    const double limit = 262144.0;   // tau in units of tau 2^-18
    while (hi - lo > 1) {
      const long long mid = lo + (hi - lo) / 2;
      if ((e = cudaMemsetAsync(B2, 0, (size_t)nsb * nsb * 8, st)) != cudaSuccess) return e;
      if ((e = cudaMemsetAsync(cnt, 0, 8, st)) != cudaSuccess) return e;
      ++g_launches;
      k_mixed_probe<<<g, 256, 0, st>>>(q, bits, blk, nnzb, nsb, mid, lo, hi, B2, cnt);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      if ((e = cudaMemcpyAsync(h.data(), B2, (size_t)nsb * nsb * 8, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
        return e;
      if ((e = cudaMemcpyAsync(h.data() + (size_t)nsb * nsb, cnt, 8, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
        return e;
      if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
      if (h[(size_t)nsb * nsb] == 0) break;   // no tile between lo and hi: the result is lo
      if (mixed_norm_bound_host(h.data(), nsb) <= limit) lo = mid;
      else hi = mid;
    }
  }
  ++g_launches;
  k_mixed_keep<<<g, 256, 0, st>>>(bits, nnzb, lo, keep);
  return cudaGetLastError();
}

}  // namespace sp2
