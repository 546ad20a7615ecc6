// FP64 symmetric block-sparse square with the fused epilogue of Algorithm 2.
//
// For every output tile (I, J), I <= J, of the product pattern:
//   S_IJ = sum_{K in R(I) & R(J)} X~_IK X~_KJ            (X~_KJ = X~_JK^T, symmetry)
//   X_new = c0 I + c1 X~_IJ + c2 S_IJ                     (Algorithm 2: p=1 gives
//           c0=(1-a)^2, c1=2a(1-a), c2=a^2; p=0 gives c0=0, c1=2a, c2=-a^2)
// and per tile the partial sums of ||X~ - S||_F^2 (weight 2 off the diagonal:
// the mirrored tile is not stored), trace(S), trace(X~) on diagonal tiles and
// ||X_new tile||_F^2 for the truncation.  e_{i-1} = ||X~_{i-1} - X~_{i-1}^2||_F and
// t_{i-1} = trace(X~_{i-1} - X~_{i-1}^2) (Algorithm 2) come out of the same pass.
//
// Sym-sum mode (used by the adjoint): S_IJ = sum_K A_IK B_KJ + B_IK A_KJ.
//
// GB300's FP64 rate is the bound here (about 1.2 TFLOP/s for DFMA, the same
// for the FP64 MMA instruction), so the kernel is written for a busy FP64 pipe:
// one CTA of 256 threads per output tile, 4 outputs per thread, both operand
// tiles staged in shared memory (transposed on the fly when the stored tile is
// the mirror), several CTAs per SM hide the load latency.
#include <cooperative_groups.h>

#include "sp2_internal.h"

namespace cg = cooperative_groups;

namespace sp2 {
namespace {

struct PatDev {
  const uint32_t* bits;
  const int32_t* rowptr;
  const uint32_t* ref;
};

struct SqDev {
  PatDev A, B, Z;
  const double* apool;
  const double* bpool;
  const double* zpool;
  const int32_t* obrow;
  const int32_t* obcol;
  const int32_t* oslot;
  double* opool;
  double c0, c1, c2;
  int64_t n;
  int words;
  int general;   // both triangles stored: no mirror weight
  Partials part;
};

__device__ __forceinline__ void load_tile(double (*S)[TB + 1], const double* __restrict__ src, bool trans) {
#pragma unroll
  for (int q = 0; q < TE / 256; ++q) {
    const int idx = threadIdx.x + 256 * q;
    const int r = idx >> 5, c = idx & 31;
    const double v = src[idx];
    if (trans) S[c][r] = v; else S[r][c] = v;
  }
}

// acc += sum_K P_IK Q_KJ over K in R_P(I) & R_Q(J); Q_KJ = (Q_JK)^T.
__device__ __forceinline__ int accumulate(const PatDev& P, const double* __restrict__ ppool, const PatDev& Q,
                                          const double* __restrict__ qpool, int I, int J, int words,
                                          double (*As)[TB + 1], double (*Bs)[TB + 1], double acc[2][2]) {
  const uint32_t* bi = P.bits + (int64_t)I * words;
  const uint32_t* bj = Q.bits + (int64_t)J * words;
  int baseI = P.rowptr[I], baseJ = Q.rowptr[J];
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  int nk = 0;
  for (int w = 0; w < words; ++w) {
    const uint32_t mi = bi[w], mj = bj[w];
    uint32_t m = mi & mj;
    while (m) {
      const int b = __ffs(m) - 1;
      m &= m - 1;
      const uint32_t below = (1u << b) - 1u;
      const uint32_t ra = P.ref[baseI + __popc(mi & below)];
      const uint32_t rb = Q.ref[baseJ + __popc(mj & below)];
      // P_IK: stored tile, transposed when it is the mirror.
      load_tile(As, ppool + (int64_t)(ra & ~REF_T) * TE, (ra & REF_T) != 0);
      // Q_KJ = (Q_JK)^T: Q_JK is the stored tile (or its mirror), so transpose
      // exactly when Q_JK is not itself the mirror.
      load_tile(Bs, qpool + (int64_t)(rb & ~REF_T) * TE, (rb & REF_T) == 0);
      __syncthreads();
#pragma unroll 8
      for (int k = 0; k < TB; ++k) {
        const double a0 = As[ty][k], a1 = As[ty + 16][k];
        const double b0 = Bs[k][tx], b1 = Bs[k][tx + 16];
        acc[0][0] = fma(a0, b0, acc[0][0]);
        acc[0][1] = fma(a0, b1, acc[0][1]);
        acc[1][0] = fma(a1, b0, acc[1][0]);
        acc[1][1] = fma(a1, b1, acc[1][1]);
      }
      __syncthreads();
      ++nk;
    }
    baseI += __popc(mi);
    baseJ += __popc(mj);
  }
  return nk;
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int k = 0; k < 8; ++k) s += red[k];
  return s;
}

template <bool SYM>
__global__ void __launch_bounds__(256) k_square_f64(SqDev a) {
  __shared__ double As[TB][TB + 1];
  __shared__ double Bs[TB][TB + 1];
  __shared__ double red[8];
  const int64_t t = blockIdx.x;
  const int I = a.obrow[t], J = a.obcol[t];
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  int nk = accumulate(a.A, a.apool, a.B, a.bpool, I, J, a.words, As, Bs, acc);
  if (SYM) nk += accumulate(a.B, a.bpool, a.A, a.apool, I, J, a.words, As, Bs, acc);

  // Z_IJ (X~_IJ in the forward step): present iff bit J of Z's row I is set.
  const uint32_t* bz = a.Z.bits + (int64_t)I * a.words;
  const int wj = J >> 5;
  const uint32_t mz = bz[wj];
  const bool hasZ = (mz >> (J & 31)) & 1u;
  const double* Zt = nullptr;
  if (hasZ) {
    int pos = a.Z.rowptr[I];
    for (int w = 0; w < wj; ++w) pos += __popc(bz[w]);
    pos += __popc(mz & ((1u << (J & 31)) - 1u));
    Zt = a.zpool + (int64_t)(a.Z.ref[pos] & ~REF_T) * TE;  // I <= J: never a mirror
  }
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  double* O = a.opool + (int64_t)a.oslot[t] * TE;
  double e2 = 0.0, trS = 0.0, trX = 0.0, n2 = 0.0;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int r = ty + 16 * u, c = tx + 16 * v;
      const int64_t gi = (int64_t)I * TB + r, gj = (int64_t)J * TB + c;
      const bool inside = gi < a.n && gj < a.n;
      const double s = inside ? acc[u][v] : 0.0;
      const double z = (inside && hasZ) ? Zt[r * TB + c] : 0.0;
      const bool dg = inside && gi == gj;
      const double xn = inside ? ((dg ? a.c0 : 0.0) + a.c1 * z) + a.c2 * s : 0.0;
      O[r * TB + c] = xn;
      const double d = z - s;
      e2 += d * d;
      n2 += xn * xn;
      if (dg) { trS += s; trX += z; }
    }
  }
  const double w = (I == J || a.general) ? 1.0 : 2.0;
  e2 = block_sum(e2, red);
  if (threadIdx.x == 0) a.part.e2[t] = w * e2;
  n2 = block_sum(n2, red);
  if (threadIdx.x == 0) a.part.n2[t] = n2;
  if (I == J) {
    trS = block_sum(trS, red);
    if (threadIdx.x == 0) a.part.trS[t] = trS;
    trX = block_sum(trX, red);
    if (threadIdx.x == 0) a.part.trX[t] = trX;
  } else if (threadIdx.x == 0) {
    a.part.trS[t] = 0.0;
    a.part.trX[t] = 0.0;
  }
  if (threadIdx.x == 0) a.part.ktiles[t] = nk;
}

// The same for few output tiles: a cluster of four CTAs per tile, each with 8 of
// its 32 rows and one output element per thread.  With a CTA per tile the FP64
// pipe idles where a multiprocessor has one tile less than another, and between
// the tiles of a lone CTA's K loop; quarter tiles even the first out and the next
// K tile's operands are fetched into registers while the current ones are
// multiplied, so the second goes too.  The products of an element are added in
// the same order.  Strip s has rows 4 s .. 4 s + 3 and 16 + 4 s .. 16 + 4 s + 3: all
// elements that one thread of the kernel above sums, so the tile's partial sums
// are formed in its order too (the Step 3 estimates magnify their last bits) and
// meet in the cluster's first CTA.
constexpr int STRIPS = 4;
constexpr int SROWS = TB / STRIPS;

// Steps through the K of R_P(I) & R_Q(J) in ascending order.
struct KWalk {
  const uint32_t* bi;
  const uint32_t* bj;
  const uint32_t* pref;
  const uint32_t* qref;
  int words, w, baseI, baseJ;
  uint32_t mi, mj, m;
  __device__ KWalk(const PatDev& P, const PatDev& Q, int I, int J, int nw)
      : bi(P.bits + (int64_t)I * nw), bj(Q.bits + (int64_t)J * nw), pref(P.ref), qref(Q.ref), words(nw), w(0),
        baseI(P.rowptr[I]), baseJ(Q.rowptr[J]) {
    mi = bi[0];
    mj = bj[0];
    m = mi & mj;
  }
  __device__ bool next(uint32_t& ra, uint32_t& rb) {
    while (m == 0u) {
      baseI += __popc(mi);
      baseJ += __popc(mj);
      if (++w >= words) return false;
      mi = bi[w];
      mj = bj[w];
      m = mi & mj;
    }
    const uint32_t below = (m & (0u - m)) - 1u;
    m &= m - 1u;
    ra = pref[baseI + __popc(mi & below)];
    rb = qref[baseJ + __popc(mj & below)];
    return true;
  }
};

template <bool SYM>
__global__ void __cluster_dims__(STRIPS, 1, 1) __launch_bounds__(256) k_square_f64_strips(SqDev a) {
  __shared__ double As[2][SROWS][TB + 1];
  __shared__ double Bs[2][TB][TB + 1];
  __shared__ double val[3][SROWS][TB];     // S, X~ - S, X_new of the strip
  __shared__ double sums[4][8];            // e2, n2, trS, trX of the 8 warps of a whole-tile CTA (used in the first CTA)
  cg::cluster_group cl = cg::this_cluster();
  const int strip = (int)cl.block_rank();
  const int64_t t = blockIdx.x / STRIPS;
  const int I = a.obrow[t], J = a.obcol[t];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // tile row of strip row i
  auto row_of = [&](int i) { return 4 * strip + (i & 3) + 16 * (i >> 2); };
  double acc = 0.0;
  int nk = 0;
  for (int pass = 0; pass < (SYM ? 2 : 1); ++pass) {
    const PatDev& P = pass == 0 ? a.A : a.B;
    const PatDev& Q = pass == 0 ? a.B : a.A;
    const double* pp = pass == 0 ? a.apool : a.bpool;
    const double* qp = pass == 0 ? a.bpool : a.apool;
    KWalk walk(P, Q, I, J, a.words);
    double va, vb[4];
    uint32_t ra, rb;
    bool at = false, bt = false;
    auto fetch = [&]() -> bool {
      if (!walk.next(ra, rb)) return false;
      at = (ra & REF_T) != 0;
      bt = (rb & REF_T) == 0;      // Q_KJ = (Q_JK)^T
      const double* sa = pp + (int64_t)(ra & ~REF_T) * TE;
      const double* sb = qp + (int64_t)(rb & ~REF_T) * TE;
      // stored order for the strip's rows, or 8 columns of the 32 stored rows
      va = at ? sa[(threadIdx.x >> 3) * TB + row_of(threadIdx.x & 7)] : sa[row_of(warp) * TB + lane];
#pragma unroll
      for (int q = 0; q < 4; ++q) vb[q] = sb[threadIdx.x + 256 * q];
      return true;
    };
    bool more = fetch();
    int buf = 0;
    while (more) {
      if (at) As[buf][threadIdx.x & 7][threadIdx.x >> 3] = va;
      else As[buf][warp][lane] = va;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = warp + 8 * q;
        if (bt) Bs[buf][lane][r] = vb[q]; else Bs[buf][r][lane] = vb[q];
      }
      __syncthreads();
      more = fetch();
#pragma unroll 8
      for (int k = 0; k < TB; ++k) acc = fma(As[buf][warp][k], Bs[buf][k][lane], acc);
      buf ^= 1;      // the other buffer's last readers have passed the barrier above
      ++nk;
    }
    if (SYM) __syncthreads();
  }
  const uint32_t* bz = a.Z.bits + (int64_t)I * a.words;
  const int wj = J >> 5;
  const uint32_t mz = bz[wj];
  const bool hasZ = (mz >> (J & 31)) & 1u;
  const double* Zt = nullptr;
  if (hasZ) {
    int pos = a.Z.rowptr[I];
    for (int w = 0; w < wj; ++w) pos += __popc(bz[w]);
    pos += __popc(mz & ((1u << (J & 31)) - 1u));
    Zt = a.zpool + (int64_t)(a.Z.ref[pos] & ~REF_T) * TE;  // I <= J: never a mirror
  }
  const int r = row_of(warp);
  const int64_t gi = (int64_t)I * TB + r, gj = (int64_t)J * TB + lane;
  const bool inside = gi < a.n && gj < a.n;
  const double s = inside ? acc : 0.0;
  const double z = (inside && hasZ) ? Zt[r * TB + lane] : 0.0;
  const bool dg = inside && gi == gj;
  const double xn = inside ? ((dg ? a.c0 : 0.0) + a.c1 * z) + a.c2 * s : 0.0;
  a.opool[(int64_t)a.oslot[t] * TE + r * TB + lane] = xn;
  val[0][warp][lane] = s;
  val[1][warp][lane] = z - s;
  val[2][warp][lane] = xn;
  cl.sync();      // the values are written, and every CTA of the cluster has started
  if (threadIdx.x < 64) {
    // thread (ty, tx) of the whole-tile kernel: elements (ty + 16 u, tx + 16 v)
    const int i = threadIdx.x >> 4, tx = threadIdx.x & 15, ty = row_of(i);
    double e2 = 0.0, n2 = 0.0, trS = 0.0, trX = 0.0;
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const double d = val[1][i + 4 * u][tx + 16 * v], x = val[2][i + 4 * u][tx + 16 * v];
        e2 = fma(d, d, e2);
        n2 = fma(x, x, n2);
        if (I == J && ty == tx && u == v) {      // s and z of a padding element are zero
          const double sv = val[0][i + 4 * u][tx + 16 * v];
          trS += sv;
          trX += (int64_t)I * TB + ty + 16 * u < a.n && hasZ ? Zt[(ty + 16 * u) * (TB + 1)] : 0.0;
        }
      }
    for (int o = 16; o > 0; o >>= 1) {
      e2 += __shfl_xor_sync(0xffffffffu, e2, o);
      n2 += __shfl_xor_sync(0xffffffffu, n2, o);
      trS += __shfl_xor_sync(0xffffffffu, trS, o);
      trX += __shfl_xor_sync(0xffffffffu, trX, o);
    }
    if (lane == 0) {
      double (*dst)[8] = reinterpret_cast<double (*)[8]>(cl.map_shared_rank(&sums[0][0], 0));
      const int w = 2 * strip + warp;
      dst[0][w] = e2;
      dst[1][w] = n2;
      dst[2][w] = trS;
      dst[3][w] = trX;
    }
  }
  cl.sync();
  if (strip == 0 && threadIdx.x < 4) {
    const int q = threadIdx.x;
    double v = 0.0;
    for (int k = 0; k < 8; ++k) v += sums[q][k];
    if (q == 0) a.part.e2[t] = ((I == J || a.general) ? 1.0 : 2.0) * v;
    if (q == 1) a.part.n2[t] = v;
    if (q == 2) a.part.trS[t] = v;
    if (q == 3) a.part.trX[t] = v;
    if (q == 0) a.part.ktiles[t] = nk;
  }
}

// Fixed-order two-level reduction of the per-tile partials.  Block g sums the
// contiguous range [g c, (g+1) c), c = ceil(nt / RED_BLOCKS): thread k takes
// entries k, k + 256, ... of the range in order, then a fixed tree; one block
// (the last to finish) then sums the RED_BLOCKS results with the same tree.  The result depends on
// nt only, not on scheduling.
constexpr int RED_BLOCKS = 256;

struct RedPart {
  double e2, trS, trX;
  long long k;
};

__device__ RedPart block_tree(double a, double b, double c, long long k) {
  __shared__ double s0[256], s1[256], s2[256];
  __shared__ long long s3[256];
  __syncthreads();
  s0[threadIdx.x] = a; s1[threadIdx.x] = b; s2[threadIdx.x] = c; s3[threadIdx.x] = k;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) {
      s0[threadIdx.x] += s0[threadIdx.x + h];
      s1[threadIdx.x] += s1[threadIdx.x + h];
      s2[threadIdx.x] += s2[threadIdx.x + h];
      s3[threadIdx.x] += s3[threadIdx.x + h];
    }
    __syncthreads();
  }
  return RedPart{s0[0], s1[0], s2[0], s3[0]};
}

// The block that finishes last sums the results of all (ticket: zero before and
// after the launch).
__global__ void __launch_bounds__(256) k_reduce_step(Partials p, int64_t nt, RedPart* part, unsigned* ticket,
                                                     StepScalars* out) {
  const int64_t c = (nt + RED_BLOCKS - 1) / RED_BLOCKS;
  const int64_t lo = (int64_t)blockIdx.x * c, hi = min(nt, lo + c);
  double a = 0.0, b = 0.0, d = 0.0;
  long long k = 0;
  for (int64_t i = lo + threadIdx.x; i < hi; i += 256) {
    a += p.e2[i];
    b += p.trS[i];
    d += p.trX[i];
    k += p.ktiles[i];
  }
  const RedPart mine = block_tree(a, b, d, k);
  __shared__ bool last;
  if (threadIdx.x == 0) {
    part[blockIdx.x] = mine;
    __threadfence();
    last = atomicAdd(ticket, 1u) == RED_BLOCKS - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const volatile RedPart* vp = part;
  const RedPart q{vp[threadIdx.x].e2, vp[threadIdx.x].trS, vp[threadIdx.x].trX, vp[threadIdx.x].k};   // RED_BLOCKS == blockDim.x
  const RedPart r = block_tree(q.e2, q.trS, q.trX, q.k);
  if (threadIdx.x == 0) {
    out->e2 = r.e2;
    out->trS = r.trS;
    out->trX = r.trX;
    out->triplets = r.k;
    *ticket = 0u;
  }
}

// Output tiles up to which a tile is split over a cluster.  Dense matrices, one
// CTA per tile -> four: 10 tiles 45.9 -> 18.6 us a square, 36 tiles 79.6 -> 28.2,
// 91 tiles 122 -> 94, 136 tiles 147 -> 146, 210 tiles 336 -> 261 (two rounds of
// CTAs on 152 multiprocessors become 1.4); 300 tiles 400 -> 457, 435 tiles 719 ->
// 728 (clusters of four do not fill every multiprocessor), 528 tiles 1047 -> 995,
// 1176 tiles 3102 -> 3136.
constexpr int64_t STRIP_MAX_TILES = 240;

PatDev dev(const FullPattern* f) { return PatDev{f->bits, f->rowptr, f->ref}; }

}  // namespace

cudaError_t launch_square_f64(const SquareArgs& a, cudaStream_t st) {
  if (a.out->nnzb == 0) return cudaSuccess;
  SqDev d;
  d.A = dev(a.A); d.B = dev(a.B); d.Z = dev(a.Z);
  d.apool = a.apool; d.bpool = a.bpool; d.zpool = a.zpool;
  d.obrow = a.out->brow; d.obcol = a.out->bcol; d.oslot = a.out->slot; d.opool = a.outpool;
  d.c0 = a.c0; d.c1 = a.c1; d.c2 = a.c2;
  d.n = a.n; d.words = a.A->words;
  d.general = a.general ? 1 : 0;
  d.part = a.part;
  const unsigned nt = (unsigned)a.out->nnzb;
  ++g_launches;
  if (a.out->nnzb <= STRIP_MAX_TILES) {
    if (a.sym_sum) k_square_f64_strips<true><<<nt * STRIPS, 256, 0, st>>>(d);
    else k_square_f64_strips<false><<<nt * STRIPS, 256, 0, st>>>(d);
  } else {
    if (a.sym_sum) k_square_f64<true><<<nt, 256, 0, st>>>(d);
    else k_square_f64<false><<<nt, 256, 0, st>>>(d);
  }
  return cudaGetLastError();
}

size_t reduce_work_bytes() { return (RED_BLOCKS + 1) * sizeof(RedPart); }

cudaError_t launch_reduce_step(const Partials& p, int64_t ntiles, StepScalars* out, void* work, cudaStream_t st) {
  unsigned* ticket = static_cast<unsigned*>(work);
  RedPart* part = static_cast<RedPart*>(work) + 1;
  ++g_launches;
  k_reduce_step<<<RED_BLOCKS, 256, 0, st>>>(p, ntiles, part, ticket, out);
  return cudaGetLastError();
}

}  // namespace sp2
