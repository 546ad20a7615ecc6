// Tensor-core (tcgen05, sm_103a) symmetric block-sparse square with FP64-grade
// accuracy from FP16 slices, plus the fused epilogue of Algorithm 2.
//
// Slicing (a GB300-specific reading of "tile products in FP16 split precision"):
// every element x of X~ (|x| < 2 for an SP2 iterate, whose eigenvalues stay in
// about [0, 1]) is written on fixed absolute grids,
//     x ~= sum_{s=1..k} T_s * 2^-(11 s - 1),   T_s integers, |T_s| <= 2048,
// (11-bit slices; five slices use 10-bit ones, see slice_bits)
// so each slice T_s is exact in FP16.  The product of slices s and t has the
// unit 2^-(11 (s + t) - 2); all pairs with the same g = s + t share one FP32
// accumulator in tensor memory.  Their sums are integers: the g = 2 group
// (T_1 T_1) stays below 2^24 because rows of X~ have 2-norm <= ~1, so it is
// accumulated exactly; the smaller groups are exact in practice and their
// rounding error is scaled down by 2^-11 per group.  The epilogue combines the
// groups as an exact int64 fixed-point sum and converts once to FP64.  Pairs
// with s + t <= k + 1 are used (k = 4: 10 MMAs per K step, error ~2^-44 per
// element; k = 2 is the three-product hi+lo form).  Two places where the FP32
// sums would not stay exact are handled apart: the diagonal of S = X~^2, whose
// products of equal slices are all positive, is taken from FP64 squared row
// norms summed while the records are sliced; and long K loops (dense rows) are
// accumulated in segments whose exact sums the epilogue adds in int64.
//
// Operands are stored panel by panel: for a super-row R (tile rows 4R..4R+3)
// and a K tile present in any of its rows, one record holds slice s of the 4
// tiles as one contiguous 8 KB unit (the K-major layout the MMA reads, absent
// tiles zero), so one bulk copy moves a whole 128 x 32 operand slice.  The
// symmetric X~ needs one panel set for A and B alike.
//
// Most tiles of an SP2 iterate are small (density-matrix elements decay with
// distance): a tile with max |x| < 2^-11 has T_1 = 0, below 2^-22 also T_2 = 0.
// Each record notes its first slice that is not all zero.  For a K step the A
// record starts at slice fA, the B record at fB, and only the pairs s >= fA,
// t >= fB, s + t <= k + 1 are issued; only the slices they read are loaded.
// Pairs left out multiply zeros, so the result is the same bit for bit.
//
// Data path per CTA (one 128 x 128 output super-tile = 4 x 4 tiles of 32):
//   warp 0: planner -- for every K tile in the union of the super-rows'
//     patterns (32 at a time, found from the super-row bitmaps, their record
//     headers fetched one batch ahead), lists sub-steps of at most two A
//     slices x two B slices.
//   warps 18 and 19: issuers -- copy the A and the B units of every sub-step
//     into the stages (cp.async.bulk of 8 or 16 KB, completion tracked by an
//     mbarrier transaction count).
//   warp 1: issues tcgen05.mma kind::f16 (M = 128, N = 128, K = 16) for every
//     slice pair of the record into the TMEM accumulator of its group, then
//     tcgen05.commit frees the stage.
//   warps 2-17: epilogue -- tcgen05.ld of the accumulators that were written,
//     exact fixed-point combination, X_new = c0 I + c1 X~ + c2 S in FP64,
//     per-tile ||X~ - S||^2, traces and ||X_new||^2, FP64 stores of the
//     output tiles present.
// Every wait is bounded; on timeout the kernel records an error flag, stops
// issuing work and still frees its tensor memory.
#include "cluster_scan.h"
#include "sp2_internal.h"
#include <cuda_fp16.h>

namespace sp2 {
namespace {

constexpr int ST = 128;          // super-tile edge (4 tiles)

// Bits per slice: 11 (FP16 holds integers up to 2^11 exactly) for two to four
// slices; 10 for five, whose smaller digits keep the FP32 group sums of dense
// rows exact with room to spare (finest grid 2^-49, FP64 grade for |x| <= 1).
__host__ __device__ constexpr int slice_bits(int k) { return k == 5 ? 10 : 11; }
constexpr int SLICE_BYTES = 2048;  // one 32 x 32 FP16 slice

// ------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// How many of the four ring stages from s on have completed their phase (those
// past the wrap at `stages` the next one), without waiting: four tests in a row,
// whose latencies overlap; a stage counts if all before it have completed.
__device__ __forceinline__ int mbar_ready4(uint64_t* ring, int s, uint32_t parity, int stages) {
  const bool w1 = s + 1 >= stages, w2 = s + 2 >= stages, w3 = s + 3 >= stages;
  const uint32_t b = smem_u32(ring);
  int m;
  asm volatile(
      "{\n\t.reg .pred p, q, r, s;\n\t.reg .b32 x;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %5;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 q, [%2], %6;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 r, [%3], %7;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 s, [%4], %8;\n\t"
      "selp.b32 x, 4, 3, s;\n\t"
      "selp.b32 x, x, 2, r;\n\t"
      "selp.b32 x, x, 1, q;\n\t"
      "selp.b32 %0, x, 0, p;\n\t}"
      : "=r"(m)
      : "r"(b + 8u * (uint32_t)s), "r"(b + 8u * (uint32_t)(w1 ? s + 1 - stages : s + 1)),
        "r"(b + 8u * (uint32_t)(w2 ? s + 2 - stages : s + 2)), "r"(b + 8u * (uint32_t)(w3 ? s + 3 - stages : s + 3)),
        "r"(parity), "r"(parity ^ (w1 ? 1u : 0u)), "r"(parity ^ (w2 ? 1u : 0u)), "r"(parity ^ (w3 ? 1u : 0u))
      : "memory");
  return m;
}

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// try_wait that lets the hardware suspend the thread for up to hint_ns (it
// resumes when the phase completes): for waiters off the critical path, so
// they do not take issue slots from the warps sharing their sub-partition.
__device__ __forceinline__ bool mbar_try_wait_sleep(uint64_t* bar, uint32_t parity, uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}

// Timeout sites of a launch, for the error message (err[1], bit 0 self-test
// probe, 1 planner batch or tile slot, 2 issuer ring, 8 issuer batch, 9 copies
// still in flight at the exit, 3 MMA data, 4 MMA TMEM or segment slot, 5 MMA
// drain, 6 epilogue tile, 7 epilogue segment).
__device__ __forceinline__ void note_timeout(int32_t* err, int where) {
  if (err) atomicOr(err + 1, 1 << where);
}

// Limit of every bounded wait of a launch (ns), set from the launch arguments.
__device__ __forceinline__ unsigned long long& wait_limit_ns() {
  __shared__ unsigned long long lim;
  return lim;
}

// Bounded wait with suspension between polls: false on timeout.
__device__ __forceinline__ bool mbar_wait_sleep(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = now_ns(), lim = wait_limit_ns();
  while (!mbar_try_wait_sleep(bar, parity, 20000u))
    if (now_ns() - t0 > lim) return false;
  return true;
}

// Bounded wait: false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = now_ns(), lim = wait_limit_ns();
  while (!mbar_try_wait(bar, parity))
    if (now_ns() - t0 > lim) return false;
  return true;
}

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// The per-CTA fixed-point staging (128 KB per CTA, 19 MB in all) is written and
// read back by the same thread within one tile: an L2 evict_last policy keeps
// it out of DRAM while the operand records stream past.
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

__device__ __forceinline__ long long ld_staging(const long long* p, uint64_t pol) {
  long long v;
  asm volatile("ld.global.L2::cache_hint.s64 %0, [%1], %2;" : "=l"(v) : "l"(p), "l"(pol));
  return v;
}

__device__ __forceinline__ void st_staging(long long* p, long long v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.s64 [%0], %1, %2;" ::"l"(p), "l"(v), "l"(pol) : "memory");
}

// 0.0 - x, bit for bit (a zero gives +0), without an FP64 instruction
__device__ __forceinline__ double negated(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  return ((hi & 0x7FFFFFFF) | lo) == 0 ? 0.0 : __hiloint2double(hi ^ (int)0x80000000, lo);
}

// x * 2^k, exact, by exponent arithmetic on the high word; x an integer-valued
// double (0 or |x| >= 1) and a normal result.
__device__ __forceinline__ double int_times_pow2(double x, int k) {
  const int hi = __double2hiint(x);
  return (hi & 0x7FFFFFFF) == 0 ? x : __hiloint2double(hi + (k << 20), __double2loint(x));
}

// v * 2^k for |v| < 2^53 (exact; a normal result) with no FP64 instruction: the
// leading bit is shifted to bit 52 and the exponent added.
__device__ __forceinline__ double small_ll_times_pow2(long long v, int k) {
  const unsigned long long m = (unsigned long long)(v < 0 ? -v : v);
  const int c = __clzll((long long)m);                       // >= 11; 64 for zero
  const unsigned long long f = m << ((c - 11) & 63);         // bit 52 set
  const int hi = (int)(f >> 32) + ((1085 - c + k) << 20);    // 1085: bit 52 adds one
  const int sgn = (int)((unsigned long long)v >> 32) & (int)0x80000000;
  return m == 0ull ? 0.0 : __hiloint2double(hi | sgn, (int)(uint32_t)f);
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// 2 z exactly (an exponent increment for normal z; the FP64 add otherwise).
__device__ __forceinline__ double twice(double z) {
  const int hi = __double2hiint(z);
  const int e = (hi >> 20) & 0x7FF;
  return (e != 0 && e < 0x7FE) ? __hiloint2double(hi + (1 << 20), __double2loint(z)) : z + z;
}

// Shared-memory matrix descriptor, no swizzle, K-major canonical layout:
// core matrices of 8 rows x 16 bytes (128 contiguous bytes), LBO = byte stride
// between core matrices along K, SBO = byte stride between 8-row groups.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // fixed 0b001 field of tcgen05 descriptors
  return d;                // base offset 0, relative LBO, no swizzle
}

// Instruction descriptor, kind::f16: FP16 A and B, FP32 D, both K-major, M = 128, N = 128.
constexpr uint32_t IDESC = (1u << 4) | (0u << 7) | (0u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(IDESC), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// true in one lane of the (converged) warp, the same lane every time
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float* v) {
  uint32_t r[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}

// ------------------------------------------------------------------ slicing
constexpr int PANEL_BYTES = 4 * SLICE_BYTES;   // one slice of the 4 tiles of a record

// place in shared memory of the 16-byte core row cr = 32 (row / 8) + 8 (column / 8) + row % 8
__device__ __forceinline__ int panel_core_row(int cr) { return cr ^ (2 * ((cr >> 3) & 3)); }

// two integers |T| <= 2^11 as FP16, exact (the FP32 magic-number add, then one
// packed conversion: the integer-to-half instruction runs at a quarter of the rate)
__device__ __forceinline__ uint32_t pack_halves(int lo, int hi) {
  const float a = __int_as_float(0x4B400000 + lo) - 12582912.0f, b = __int_as_float(0x4B400000 + hi) - 12582912.0f;
  const __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// One CTA per panel record e: the 4 tiles of the record (index words from
// k_panel_fill: compact tile index, bit 31 = use the stored tile transposed;
// all ones = absent), sliced and written as k units of 8 KB,
//   byte offset = s * 8192 + q * 2048 + g * 512 + c * 128 + r * 16 + j * 2
// for the element in row 8g + r, column 8c + j of tile q, slice s.  The header
// byte holds the first slice that is not all zero in any of the 4 tiles (k if
// none) in bits 0-2 and the tiles present in bits 4-7; units below that slice
// are all zero, are never read, and are not written.
//
// rsq (optional): rsq[128 e + 32 q + r] = sum_c x_rc^2 of row r of tile q in
// FP64, unscaled (0 for an absent tile).  Summed over the records of a
// super-row (k_row_sq_sum) they give the squared row norms of the matrix, the
// diagonal of its square.
//
// Each thread takes four elements of a tile that are neighbours in a panel row
// (four of a stored row, or of a stored column of a tile used transposed), so a
// slice of them is one 8-byte shared-memory store.  16-byte core rows and, in odd
// row groups, their halves are permuted in shared memory so that neither
// orientation's stores collide; the copy to the record undoes it.  Absent tiles
// cost a zero fill.  With rsq the FP64 pipe is the floor: two to three lane
// operations an element at 2 per SM cycle, 0.5 ms for the 100,000 tiles of the
// water-like N = 24,000 case (as is HBM: 3.4 GB).  One element and 2-byte stores
// at a time, absent tiles worked through like the others, took 1.18 ms a launch;
// this takes 0.96 ms.
template <int K>
__global__ void __launch_bounds__(256, 4) k_panel_slices(const uint4* __restrict__ index, const int32_t* __restrict__ slot,
                                                       const double* __restrict__ pool, __half* data,
                                                       uint8_t* head, int32_t* err, double* rsq, int lscale,
                                                       int report_range) {
  __shared__ __align__(16) unsigned char sm[K * PANEL_BYTES];
  __shared__ uint32_t wnz[8];
  __shared__ int first_s;
  const int64_t e = blockIdx.x;
  if (report_range && e == 0 && threadIdx.x == 0 && err) atomicOr(err, 4);
  const uint4 iw = index[e];
  const uint32_t wd[4] = {iw.x, iw.y, iw.z, iw.w};
  constexpr int W = slice_bits(K);
  constexpr int FIN = W * K - 1;                   // finest grid 2^-FIN
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // all loads first (16 per thread), then the integer work
  long long xb[4][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (wd[q] == 0xFFFFFFFFu) continue;
    const double* src = pool + (int64_t)slot[wd[q] & ~REF_T] * TE;
    if (wd[q] & REF_T) {
#pragma unroll
      for (int k = 0; k < 4; ++k) xb[q][k] = __double_as_longlong(src[(4 * wid + k) * TB + lane]);
    } else {
      const longlong2* s2 = reinterpret_cast<const longlong2*>(src) + 2 * threadIdx.x;
      const longlong2 u = s2[0], v = s2[1];
      xb[q][0] = u.x; xb[q][1] = u.y; xb[q][2] = v.x; xb[q][3] = v.y;
    }
  }
  int any[K];                                      // bits set in any element of slice s
#pragma unroll
  for (int s = 0; s < K; ++s) any[s] = 0;
  // squared row sums (rsq): a row of a tile used as stored is complete in eight
  // lanes; of a tile used transposed each warp has a part of every row (lane =
  // row).  Fixed order throughout.
  double rs[4];
  uint32_t pres = 0;
  bool far = false;                                // |x / scale| >= 2, inf or NaN
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    unsigned char* st = sm + q * SLICE_BYTES;
    if (wd[q] == 0xFFFFFFFFu) {                    // absent: zero (the same for the whole CTA)
      for (int i = threadIdx.x; i < K * (SLICE_BYTES / 16); i += 256)
        *reinterpret_cast<uint4*>(st + (i >> 7) * PANEL_BYTES + (i & 127) * 16) = make_uint4(0u, 0u, 0u, 0u);
      rs[q] = 0.0;
      continue;
    }
    pres |= 1u << q;
    const bool tr = (wd[q] & REF_T) != 0;
    // panel row and first of four columns
    const int r = tr ? lane : (int)(threadIdx.x >> 3), c = tr ? 4 * wid : 4 * (int)(threadIdx.x & 7);
    if (rsq) {
      double x[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) x[k] = __longlong_as_double(xb[q][k]);
      rs[q] = fma(x[3], x[3], fma(x[2], x[2], fma(x[1], x[1], x[0] * x[0])));
      if (!tr) {
        rs[q] += __shfl_xor_sync(0xffffffffu, rs[q], 1);
        rs[q] += __shfl_xor_sync(0xffffffffu, rs[q], 2);
        rs[q] += __shfl_xor_sync(0xffffffffu, rs[q], 4);
      }
    }
    int T[4][K];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      // v = x / scale * 2^FIN rounded to the nearest integer (ties to even),
      // from the bits of x = m 2^(ex - 1075): v = m >> sh on the integer pipes
      const long long x = xb[q][k];
      const int ex = (int)((x >> 52) & 0x7FF);
      long long v = 0;
      if (ex - lscale >= 1024) {           // flagged below, clamped
        far = true;
        v = (1ll << (FIN + 1)) - 1;
        if (x < 0) v = -v;
      } else if (ex != 0) {
        const unsigned long long m = ((unsigned long long)x & 0x000FFFFFFFFFFFFFull) | (1ull << 52);
        // sh >= 3 for every slice count used (FIN <= 49); a left shift, exact
        // (|v| < 2^(FIN + 1)), covers sh <= 0
        const int sh = 1075 + lscale - FIN - ex;
        unsigned long long qv = 0;
        if (sh <= 0) {
          qv = m << (-sh);
        } else if (sh < 64) {
          qv = m >> sh;
          const unsigned long long rem = m & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
          if (rem > half || (rem == half && (qv & 1ull))) ++qv;
        }
        v = x < 0 ? -(long long)qv : (long long)qv;
      }
#pragma unroll
      for (int s = 0; s < K - 1; ++s) {
        const int sh = W * (K - 1 - s);
        const long long hi = (v + (1ll << (sh - 1))) >> sh;   // round to nearest (ties up)
        T[k][s] = (int)hi;
        v -= hi * (1ll << sh);
      }
      T[k][K - 1] = (int)v;
#pragma unroll
      for (int s = 0; s < K; ++s) any[s] |= T[k][s];
    }
    const int cr = (r >> 3) * 32 + (c >> 3) * 8 + (r & 7);
    unsigned char* dst = st + panel_core_row(cr) * 16 + ((((c >> 2) & 1) ^ ((cr >> 5) & 1)) * 8);
#pragma unroll
    for (int s = 0; s < K; ++s)
      *reinterpret_cast<uint2*>(dst + s * PANEL_BYTES) =
          make_uint2(pack_halves(T[0][s], T[1][s]), pack_halves(T[2][s], T[3][s]));
  }
  if (far && err) atomicOr(err, 4);
  uint32_t nz = 0;
#pragma unroll
  for (int s = 0; s < K; ++s) nz |= (any[s] != 0 ? 1u : 0u) << s;
  nz = __reduce_or_sync(0xffffffffu, nz);
  if (lane == 0) wnz[wid] = nz;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t m = 0;
    for (int w = 0; w < 8; ++w) m |= wnz[w];
    const int f = m ? __ffs(m) - 1 : K;
    first_s = f;
    head[e] = (uint8_t)(f | (pres << 4));
  }
  __syncthreads();
  // units below the first nonzero slice are all zero and never read: not written
  uint4* d4 = reinterpret_cast<uint4*>(data + e * (int64_t)(K * 4 * TE));
  for (int i = first_s * (PANEL_BYTES / 16) + threadIdx.x; i < K * (PANEL_BYTES / 16); i += 256) {
    const int cr = i & 127;
    uint4 v = *reinterpret_cast<const uint4*>(sm + ((i & ~127) | panel_core_row(cr)) * 16);
    if (cr & 32) v = make_uint4(v.z, v.w, v.x, v.y);
    d4[i] = v;
  }
  if (!rsq) return;
  __syncthreads();                                 // sm is free: reused for the parts of the row sums
  double* red = reinterpret_cast<double*>(sm);     // [8 warps][4 tiles][32 rows]
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (wd[q] == 0xFFFFFFFFu) continue;
    if (wd[q] & REF_T) red[wid * 128 + q * 32 + lane] = rs[q];
    else if ((lane & 7) == 0) red[q * 32 + (int)(threadIdx.x >> 3)] = rs[q];
  }
  __syncthreads();
  if (threadIdx.x < 128) {
    const uint32_t w = reinterpret_cast<const uint32_t*>(index + e)[threadIdx.x >> 5];
    double sum = 0.0;
    if (w != 0xFFFFFFFFu) {
      sum = red[threadIdx.x];
      if (w & REF_T)
#pragma unroll
        for (int u = 1; u < 8; ++u) sum += red[u * 128 + threadIdx.x];
    }
    rsq[e * 128 + threadIdx.x] = sum;
  }
}

// dsq[128 P + j] = sum of rsq[128 e + j] over the panel records e of
// super-row P (the squared row norms; see k_panel_slices).  One CTA per
// super-row, eight groups of 128 threads with an eighth of the records each (in
// record order), their sums added in order: a super-row has hundreds of records,
// and one group's chain of loads took 68 us at N = 24,000 (now 44; 12.5 -> 8.4 us at N = 2,424).
constexpr int SQ_GROUPS = 8;
__global__ void __launch_bounds__(128 * SQ_GROUPS) k_row_sq_sum(const int32_t* __restrict__ spos, int words,
                                                                const double* __restrict__ rsq, int64_t n,
                                                                double* dsq) {
  __shared__ double part[SQ_GROUPS][128];
  const int64_t P = blockIdx.x;
  const int j = threadIdx.x & 127, g = threadIdx.x >> 7;
  const int64_t lo = spos[P * words], hi = spos[(P + 1) * words];
  const int64_t len = (hi - lo + SQ_GROUPS - 1) / SQ_GROUPS;
  const int64_t e1 = min(hi, lo + (g + 1) * len);
  double acc = 0.0;
  int64_t e = lo + g * len;
  for (; e + 4 <= e1; e += 4) {
    const double v0 = rsq[e * 128 + j], v1 = rsq[(e + 1) * 128 + j], v2 = rsq[(e + 2) * 128 + j],
                 v3 = rsq[(e + 3) * 128 + j];
    acc += v0;
    acc += v1;
    acc += v2;
    acc += v3;
  }
  for (; e < e1; ++e) acc += rsq[e * 128 + j];
  part[g][j] = acc;
  __syncthreads();
  if (g != 0) return;
#pragma unroll
  for (int k = 1; k < SQ_GROUPS; ++k) acc += part[k][j];
  const int64_t gi = P * 128 + j;
  if (gi < n) dsq[gi] = acc;
}

// Super-row bitmaps (OR of the 4 tile rows) and the exclusive prefix sums of
// their words' set bits, one cluster launch.
__global__ void __cluster_dims__(SCAN_CTAS, 1, 1) __launch_bounds__(SCAN_THREADS)
    k_super_scan(const uint32_t* __restrict__ bits, int nb, int words, int nsr, uint32_t* sb, int32_t* spos,
                 int32_t* total) {
  const int64_t n = (int64_t)nsr * words;
  auto word = [&](int64_t i) {
    const int R = (int)(i / words), w = (int)(i % words);
    uint32_t m = 0;
    for (int a = 0; a < 4; ++a) {
      const int row = 4 * R + a;
      if (row < nb) m |= bits[(int64_t)row * words + w];
    }
    return m;
  };
  const int all = cluster_scan(
      n,
      [&](int64_t i) {
        const uint32_t m = word(i);
        sb[i] = m;
        return __popc(m);
      },
      [&](int64_t i, int, int ex) { spos[i] = ex; });
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    spos[n] = all;
    if (total) *total = all;
  }
}

// The same for more than SUPER_CLUSTER_MAX words: one warp per super-row over all
// multiprocessors writes its bitmap and, in its first offset, its set bits; one
// cluster scans those; the warps then write the offsets.
__global__ void __launch_bounds__(256) k_super_counts(const uint32_t* __restrict__ bits, int nb, int words, int nsr,
                                                      uint32_t* sb, int32_t* spos) {
  const int64_t R = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (R >= nsr) return;
  int c = 0;
  for (int w = lane; w < words; w += 32) {
    uint32_t m = 0;
#pragma unroll
    for (int a = 0; a < 4; ++a)
      if (4 * R + a < nb) m |= bits[(4 * R + a) * words + w];
    sb[R * words + w] = m;
    c += __popc(m);
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if (lane == 0) spos[R * words] = c;
}

__global__ void __cluster_dims__(SCAN_CTAS, 1, 1) __launch_bounds__(SCAN_THREADS)
    k_super_offsets(int words, int nsr, int32_t* spos, int32_t* total) {
  const int all = cluster_scan(
      nsr, [&](int64_t R) { return spos[R * words]; }, [&](int64_t R, int, int ex) { spos[R * words] = ex; });
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    spos[(int64_t)nsr * words] = all;
    if (total) *total = all;
  }
}

__global__ void __launch_bounds__(256) k_super_positions(const uint32_t* __restrict__ sb, int words, int nsr,
                                                         int32_t* spos) {
  const int64_t R = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (R >= nsr) return;
  int base = spos[R * words];
  __syncwarp();      // every lane has it before lane 0 writes that word again (the same value)
  for (int w0 = 0; w0 < words; w0 += 32) {
    const int w = w0 + lane;
    const int c = w < words ? __popc(sb[R * words + w]) : 0;
    int inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (w < words) spos[R * words + w] = base + inc - c;
    base += __shfl_sync(0xffffffffu, inc, 31);
  }
}

// Launch order of the super-tiles: blocks of RB super-rows x CB super-columns,
// row-major inside a block, blocks row-major.  CTAs that run at the same time
// then share A panels (same super-row) and B panels (same super-column), so the
// slices they stream are reused from L2 instead of each CTA pulling its own B
// panel from HBM.
constexpr int RB = 8, CB = 16;

__host__ __device__ inline int64_t blocked_size(int nsr) {
  const int64_t nbr = (nsr + RB - 1) / RB, nbc = (nsr + CB - 1) / CB;
  return nbr * nbc * RB * CB;
}

__device__ inline void blocked_decode(int64_t i, int nsr, int& R, int& C) {
  const int64_t nbc = (nsr + CB - 1) / CB;
  const int64_t b = i / (RB * CB), w = i % (RB * CB);
  R = (int)((b / nbc) * RB + w / CB);
  C = (int)((b % nbc) * CB + w % CB);
}

// 1 if the i-th super-tile (R, C) in launch order has an output tile (and R <= C
// unless the storage is general)
__device__ __forceinline__ int super_flag(const uint32_t* __restrict__ obits, int nb, int words, int nsr, int general,
                                          int64_t i, int& R, int& C) {
  blocked_decode(i, nsr, R, C);
  int f = 0;
  if (R < nsr && C < nsr && (general || R <= C)) {
    for (int a = 0; a < 4; ++a) {
      const int row = 4 * R + a;
      if (row >= nb) break;
      const int col0 = 4 * C;
      f |= ((obits[(int64_t)row * words + (col0 >> 5)] >> (col0 & 31)) & 0xFu) != 0;
    }
  }
  return f;
}

__global__ void k_super_flags(const uint32_t* __restrict__ obits, int nb, int words, int nsr, int general,
                              int32_t* flag) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int R, C;
  if (i < blocked_size(nsr)) flag[i] = super_flag(obits, nb, words, nsr, general, i, R, C);
}

// flags, scan and list in one cluster launch
__global__ void __cluster_dims__(SCAN_CTAS, 1, 1) __launch_bounds__(SCAN_THREADS)
    k_super_list(const uint32_t* __restrict__ obits, int nb, int words, int nsr, int general, int32_t* list,
                 int32_t* count) {
  int R, C;
  const int all = cluster_scan(
      blocked_size(nsr), [&](int64_t i) { return super_flag(obits, nb, words, nsr, general, i, R, C); },
      [&](int64_t i, int v, int ex) {
        if (!v) return;
        blocked_decode(i, nsr, R, C);
        list[ex] = R * nsr + C;
      });
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    count[0] = all;
    count[1] = 0;
  }
}

__global__ void k_super_fill(const int32_t* __restrict__ flag, const int32_t* __restrict__ pos, int64_t n, int nsr,
                             int32_t* list) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n || !flag[i]) return;
  int R, C;
  blocked_decode(i, nsr, R, C);
  list[pos[i]] = R * nsr + C;
}

// ------------------------------------------------------------------ main kernel
// One operand matrix of the product, as the kernel reads it: super-row
// bitmaps; the record of (super-row R, K tile) is number spos[R][word] +
// popcount of the lower bits of that word, with its header byte and k units
// of FP16 slices (see k_panel_slices).
struct TcOperand {
  const uint32_t* sbits;
  const int32_t* spos;
  const uint8_t* head;
  const __half* data;
};

struct TcArgs {
  TcOperand P, Q;           // S = sum_K P_IK Q_KJ  (+ Q_IK P_KJ when two_pass)
  int two_pass;
  const uint32_t* zbits;    // Z (the c1 term): pattern and FP64 values
  const int32_t* zwpre;
  const int32_t* zrowptr;
  const uint32_t* zref;
  const int32_t* zslot;     // value slot of Z's tile index (nullptr: identity)
  const double* zpool;
  const uint32_t* obits;    // output pattern bitmap, upper tiles only
  const int32_t* owpre;     // set bits of its row before each word
  const int32_t* orowptr;   // output tile row offsets
  const int32_t* list;      // active super-tiles, R * nsr + C
  const int32_t* count;     // number of active super-tiles (device)
  int32_t* work;            // work counter (zero at launch)
  double* opool;            // output tiles, slot = output index
  Partials part;
  double c0, c1, c2;
  double scale;             // product of the operands' slice scales
  int64_t n;
  int nb, words, nsr;
  int32_t* err;
  long long* scratch;       // per CTA: 128 x 128 fixed-point sums of the tile in its epilogue
  int seg_min;              // K loops of at least this many steps are cut into segments (0: never)
  int seg_ksteps;           // K steps per segment (8 or 16, divides the 32-step batch)
  unsigned long long wait_ns;   // limit of every bounded wait
  int selftest;             // 1: the planner first waits on a barrier nothing arrives at (timeout path test)
  int general;              // general storage: output tiles on both sides of the diagonal, weight 1 in e^2
  const double* dsq;        // S_ii = sum_k x_ik^2 in FP64 per global row (nullptr: from the tensor cores)
  int glo, ghi;             // slice-pair groups s + t of this launch (ghi - glo <= 3)
  int emode;                // 0: full epilogue; 1: write S (this launch's groups) into the output tiles only;
                            // 2: full epilogue on S + the S already in the output tiles
};

// A pipeline stage holds one sub-step: two A units and two B units, a unit being
// one slice of a 4-tile panel (128 rows x 32, 8 KB, 8-row groups 512 B apart):
// up to two adjacent slices of the A record and up to two of the B record, each
// side one bulk copy of 8 or 16 KB, or one unit of each of two K steps that have
// one product each.  A sub-step record (32 bits) tells the issuers what to copy
// and the MMA issuer what to multiply:
//   bits 0-2: 1 + the group (s + t - glo) of the first A x first B slice,
//   bit 3: a pair, two K steps of one product each (their slices add up to the
//   last group): products A0 x B0 and A1 x B1, both in that group,
//   bits 4-7: product mask, bit (2 i + j) for A slice a0 + i x B slice b0 + j,
//   bits 8-11: groups its products write,
//   bit 12: end of the super-tile, bit 13: no more super-tiles, bit 14: end of an
//   accumulation segment (these three have no data and no stage), bit 15: second
//   pass (A = Q, B = P), bits 16-19: groups that this segment writes first here,
//   bits 20-21, 22-24: A slices to copy and the first of them, bits 25-26, 27-29:
//   the same for B.  A super-tile whose K loop has at least
//   seg_min K steps closes a segment after every 16 K steps: the epilogue adds
//   the segment's exact fixed-point sums into the scratch and frees the TMEM,
//   so no FP32 accumulator sums more than 16 K steps (512 products per
//   element) and the groups stay exact for dense operands.
//
// What bounds the kernel is how fast its serial loops run (a warp by itself takes
// 5 to 8 cycles an instruction, and the loop of a sub-step costs the MMA issuer
// 200 to 300 cycles a product where the tensor pipe takes 128), not the copy path
// (a lone thread that issues 16 KB bulk copies fills 72 B per SM cycle out of L2;
// a K step needs 27 KB and has 210 cycles of MMAs), not shared memory (32 B per
// cycle of copies landing leave 128-wide MMAs at 66 cycles each) and not the
// tensor pipe (33%).  So all that can be done for 32 K steps side by side is done
// by the planner: it finds the K steps of a tile, reads their record headers and
// writes batches of finished sub-step records (at most 32 K steps each) into
// NPLAN buffers.  Two issuers copy the units, one the A side, one the B side, and
// the MMA issuer reads the same records; each of the three is one elected thread
// (elect.sync: in code that a comparison of the lane number guards, the operands
// of tcgen05.mma and cp.async.bulk cost twice as long to set up), with the next
// record loaded ahead.  Each tests four stages' barriers at once and then runs
// through as many sub-steps as are ready in an inner loop without a wait: a test
// or a wait in that loop, even one that never has to wait, makes every MMA dearer
// (a lone loop of four MMAs a sub-step: 445 cycles, 600 beside warps that do FP64
// work; four sub-steps at a time 335 and 375, the tensor pipe's time being 256).
// Cycles per super-tile, water-like N = 24,000 and 96,000, dense N = 4,096 with
// five slices (both launches): one producer warp 126,000, 96,000, 508,000;
// planner and one issuer 120,000, 81,000, 507,000; two issuers and 16 epilogue
// warps 103,000, 67,000, 455,000; pairs of one-product K steps, finished records,
// integer conversions in the epilogue 84,000, 58,000, 398,000; ready sub-steps
// without waits between them 80,000, 56,000, 341,000.  Two MMA issuers
// taking turns (one warp more, 80 registers instead of 96): 91,000, 64,000.  Two
// sub-steps for each barrier: 87,000, 59,000.
constexpr int UNIT_BYTES = PANEL_BYTES;
constexpr int STAGE_BYTES = 4 * UNIT_BYTES;
constexpr int STAGES = 6;                          // sub-steps in flight
constexpr int NPLAN = 4;                           // batches between the planner and the issuer
constexpr int PLAN = 104;                          // entries of a batch: 32 K steps x 3 + segment ends (+ 1 read ahead)
constexpr uint32_t REC_END = 1u << 12;
constexpr int EPI_WARPS = 16;                      // epilogue warps 2..17
constexpr int ISSUE_WARP = 2 + EPI_WARPS;          // issuer warps 18 (A units) and 19 (B units)
constexpr int TC_THREADS = 32 * (2 + EPI_WARPS + 2);   // + planner warp 0, MMA warp 1
constexpr uint32_t REC_LAST = 1u << 13;   // no more super-tiles (no data)
constexpr uint32_t REC_SEG = 1u << 14;    // end of an accumulation segment of the super-tile (no data)
constexpr uint32_t REC_PAIR = 1u << 3;
constexpr uint32_t REC_PASS1 = 1u << 15;
constexpr uint32_t REC_FRESH = 15u << 16;
constexpr uint32_t REC_CTL = REC_END | REC_LAST | REC_SEG;
constexpr uint32_t SEG_LAST = 1u << 31;   // segment record flag: last segment of its super-tile
constexpr int SEG_RING = 4;               // accumulation segments in flight between MMA and epilogue
constexpr int NSLOT = 3;                  // tiles in flight between the planner and the epilogue
constexpr int SEG_KSTEPS = 16;            // K steps per accumulation segment of a segmented tile (default)

// record header byte: first nonzero slice (bits 0-2), tiles present (bits 4-7)
constexpr uint32_t HEAD_NONE = 0x07u;   // header of a K index outside the step list

template <int K>
struct TcCfg {
  static constexpr int SMEM = STAGES * STAGE_BYTES + 2048 + NPLAN * PLAN * 16;
};

template <int K>
__global__ void __launch_bounds__(TC_THREADS, 1) k_square_tc(TcArgs a) {
  using Cfg = TcCfg<K>;
  constexpr unsigned FULLW = 0xffffffffu;
  // the group window and the epilogue mode vary only with five slices; fewer
  // slices take every group in one launch (compile-time constants)
  const int glo = K == 5 ? a.glo : 0, ghi = K == 5 ? a.ghi : K - 1, emode = K == 5 ? a.emode : 0;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* stages = smem_raw;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem_raw + STAGES * STAGE_BYTES);   // [STAGES] the sub-step's units are in
  uint64_t* empty = full + STAGES;         // [STAGES] its products are done
  uint64_t* acc_full = empty + STAGES;     // [SEG_RING] MMAs of a segment done (commit) + its record written
  uint64_t* tile_full = acc_full + SEG_RING;   // [NSLOT] tile slot written by the planner
  uint64_t* tile_empty = tile_full + NSLOT;    // [NSLOT] epilogue done with the tile slot (one arrive per warp)
  uint64_t* drain = tile_empty + NSLOT;    // MMAs issued before the exit are complete
  uint64_t* tmem_empty = drain + 1;        // [SEG_RING] every epilogue warp has read the segment's TMEM
  uint64_t* probe = tmem_empty + SEG_RING; // self-test: a barrier that nothing arrives at
  uint64_t* plan_full = probe + 1;         // [NPLAN] batch written by the planner
  uint64_t* plan_empty = plan_full + NPLAN;    // [NPLAN] batch read by the two issuers and the MMA issuer
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(plan_empty + NPLAN);
  int32_t* tslot = reinterpret_cast<int32_t*>(tmem_slot + 2);      // [NSLOT] super-tile list index, -1: none
  int32_t* kcount = tslot + NSLOT;                                  // [NSLOT][16] triplets per output tile
  uint32_t* gmap = reinterpret_cast<uint32_t*>(kcount + 16 * NSLOT);   // [SEG_RING] groups written, block of each, last flag
  int32_t* bcnt = reinterpret_cast<int32_t*>(gmap + SEG_RING);     // [NPLAN] entries of a batch
  int32_t* status = bcnt + NPLAN;                                   // [0] a wait timed out
  uint4* steps = reinterpret_cast<uint4*>(smem_raw + STAGES * STAGE_BYTES + 1024);   // [8][8] sub-steps of (first A, first B slice)
  uint4* plan = steps + 64;                                         // [NPLAN][PLAN] record, A unit, B unit, pair: steps to the second units

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 2);     // each issuer's arrival, with its bulk bytes
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < NPLAN; ++b) {
      mbar_init(&plan_full[b], 1);
      mbar_init(&plan_empty[b], 3);
    }
    for (int b = 0; b < SEG_RING; ++b) {
      mbar_init(&acc_full[b], 2);
      mbar_init(&tmem_empty[b], EPI_WARPS);
    }
    for (int b = 0; b < NSLOT; ++b) {
      mbar_init(&tile_full[b], 1);
      mbar_init(&tile_empty[b], EPI_WARPS);
    }
    mbar_init(drain, 1);
    mbar_init(probe, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    status[0] = 0;
    wait_limit_ns() = a.wait_ns;
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(FULLW, *tmem_slot, 0);
  const int total = *a.count;

  // Persistent and warp-specialised: the planner (warp 0) takes super-tiles from
  // the work counter, the issuers (warps 18, 19) stream their operand slices; the MMA issuer
  // (warp 1) accumulates each tile in TMEM blocks of 128 columns taken on
  // first use; the epilogue (warps 2-17) finishes tile i while tiles i + 1 and
  // i + 2 are being loaded and multiplied.  Tiles pass through NSLOT slots.
  if (warp == 0) {
    // ---------------- planner warp.  The record headers of 32 K steps are
    // fetched at a time (lane j: step j), one batch ahead of their use; the
    // lanes turn them into the batch's list of sub-steps.
    // steps[8 fa + fb]: the sub-steps of a K step whose A record starts at slice
    // fa and whose B record at fb -- the pairs s >= fa, t >= fb with
    // glo <= s + t <= ghi (the launch's group window), two A and two B slices
    // each; the B pair starts where A slice a0 + 1 meets glo.  At most three for
    // every window used (x, y, z: records; w: their number).
    for (int e = lane; e < 64; e += 32) {
      const int fa = e >> 3, fb = e & 7;
      uint32_t rv[3] = {0u, 0u, 0u};
      int ns = 0;
      for (int a0 = fa; a0 <= K - 1 && a0 + fb <= ghi; a0 += 2) {
        for (int b0 = max(fb, glo - a0 - 1); b0 <= K - 1 && a0 + b0 <= ghi; b0 += 2) {
          uint32_t mask = 0;
          for (int i = 0; i < 2; ++i)
            for (int j = 0; j < 2; ++j) {
              const int si = a0 + i, tj = b0 + j;
              if (si <= K - 1 && tj <= K - 1 && si + tj >= glo && si + tj <= ghi) mask |= 1u << (2 * i + j);
            }
          if (!mask) continue;
          const int base = a0 + b0 - glo;     // >= -1
          const uint32_t need = ((((mask & 1u) | ((mask & 6u) ? 2u : 0u) | ((mask & 8u) ? 4u : 0u)) << (base + 1)) >> 1) & 0xFu;
          const int uA0 = (mask & 3u) ? 1 : 0, uA1 = (mask & 12u) ? 1 : 0;
          const int uB0 = (mask & 5u) ? 1 : 0, uB1 = (mask & 10u) ? 1 : 0;
          const uint32_t v = (uint32_t)(base + 1) | (mask << 4) | (need << 8) | ((uint32_t)(uA0 + uA1) << 20) |
                             ((uint32_t)(a0 + 1 - uA0) << 22) | ((uint32_t)(uB0 + uB1) << 25) |
                             ((uint32_t)(b0 + 1 - uB0) << 27);
          if (ns == 0) rv[0] = v;
          else if (ns == 1) rv[1] = v;
          else rv[2] = v;
          ++ns;
        }
      }
      steps[e] = make_uint4(rv[0], rv[1], rv[2], (uint32_t)ns);
    }
    __syncwarp();
    bool ok = true;
    int nbat = 0;      // batches handed to the issuers and the MMA issuer
    unsigned long long nprod = 0;   // slice-pair products planned by this lane
    // all lanes: wait for the next batch buffer; false on timeout
    auto batch_open = [&]() -> bool {
      int good = 1;
      if (lane == 0) good = mbar_wait_sleep(&plan_empty[nbat % NPLAN], (((uint32_t)(nbat / NPLAN)) & 1u) ^ 1u) ? 1 : 0;
      good = __shfl_sync(FULLW, good, 0);
      if (!good && lane == 0) { status[0] = 1; note_timeout(a.err, 1); }
      return good != 0;
    };
    // all lanes: hand the batch's n entries to the issuer
    auto batch_close = [&](int n) {
      __syncwarp();
      if (lane == 0) {
        bcnt[nbat % NPLAN] = n;
        mbar_arrive(&plan_full[nbat % NPLAN]);   // release: the entries are visible
      }
      ++nbat;
    };
    // all lanes: a batch of one control entry
    auto batch_ctl = [&](uint32_t rv) -> bool {
      if (!batch_open()) return false;
      if (lane == 0) plan[(nbat % NPLAN) * PLAN] = make_uint4(rv, 0u, 0u, 0u);
      batch_close(1);
      return true;
    };
    // self-test of the timeout path: before any copy is issued, wait on a
    // barrier that nothing arrives at; the wait gives up after the wait limit,
    // the status is set, and the launch ends through the no-more-tiles path
    if (a.selftest) {
      int good = 1;
      if (lane == 0) good = mbar_wait(probe, 0) ? 1 : 0;
      good = __shfl_sync(FULLW, good, 0);
      if (!good && lane == 0) {
        status[0] = 1;
        note_timeout(a.err, 0);
      }
      __syncwarp();
    }
    int nidx = 0;      // next super-tile, taken from the work counter one tile ahead
    if (lane == 0) nidx = atomicAdd(a.work, 1);
    for (int it = 0; ok; ++it) {
      const int b = it % NSLOT;
      // the slot's previous tile (it - NSLOT) has left the epilogue
      int good = 1;
      if (lane == 0) good = mbar_wait_sleep(&tile_empty[b], (((uint32_t)(it / NSLOT)) & 1u) ^ 1u) ? 1 : 0;
      good = __shfl_sync(FULLW, good, 0);
      if (!good) {
        if (lane == 0) { status[0] = 1; note_timeout(a.err, 1); }
        break;
      }
      const int idx = __shfl_sync(FULLW, nidx, 0);
      if (idx >= total || *(volatile int32_t*)status != 0) {
        // no more tiles: tell the epilogue (slot) and the MMA issuer (record)
        if (lane == 0) {
          tslot[b] = -1;
          mbar_arrive(&tile_full[b]);
        }
        batch_ctl(REC_LAST);
        break;
      }
      if (lane == 0) nidx = atomicAdd(a.work, 1);
      const int stile = a.list[idx];
      const int R = stile / a.nsr, C = stile % a.nsr;
      // the epilogue learns the tile now (it drains segments while the tile is produced)
      if (lane == 0) {
        tslot[b] = idx;
        mbar_arrive(&tile_full[b]);
      }
      // K steps of the tile (both passes): long K loops are cut into segments
      int ktot = 0;
      if (a.seg_min > 0 && a.nb * (1 + a.two_pass) >= a.seg_min) {
        for (int pass = 0; pass < 1 + a.two_pass; ++pass) {
          const TcOperand& oa = pass == 0 ? a.P : a.Q;
          const TcOperand& ob = pass == 0 ? a.Q : a.P;
          for (int w = lane; w < a.words; w += 32)
            ktot += __popc(oa.sbits[(int64_t)R * a.words + w] & ob.sbits[(int64_t)C * a.words + w]);
        }
        ktot = __reduce_add_sync(FULLW, ktot);
      }
      const bool segmented = a.seg_min > 0 && ktot >= a.seg_min;
      int kdone = 0;
      uint32_t wmask = 0u;      // groups that the open segment has written
      // triplet counts: K steps with A tile q and B tile y both present, byte y of
      // acc[q] in every lane, moved to kc (lane 4 q + y) before a byte overflows
      int kc = 0, nacc = 0;
      uint32_t acc[4] = {0u, 0u, 0u, 0u};
      auto flush_counts = [&]() {
#pragma unroll
        for (int t = 0; t < 16; ++t) {
          const int s = __reduce_add_sync(FULLW, (int)((acc[t >> 2] >> (8 * (t & 3))) & 0xFFu));
          if (lane == t) kc += s;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = 0u;
        nacc = 0;
      };
      for (int pass = 0; pass < 1 + a.two_pass && ok; ++pass) {
        // pass 0: A = P (rows I), B = Q (rows J); pass 1: A = Q, B = P
        const TcOperand& opA = pass == 0 ? a.P : a.Q;
        const TcOperand& opB = pass == 0 ? a.Q : a.P;
        const int64_t offA = (int64_t)R * a.words, offB = (int64_t)C * a.words;
        for (int w0 = 0; w0 < a.words && ok; w0 += 32) {
          // lane L holds word w0 + L of both super-rows; the K steps are the set
          // bits of ma & mb, numbered through the inclusive prefix incl
          const int wl = w0 + lane;
          uint32_t ma = 0u, mb = 0u;
          int pa = 0, pb = 0;
          if (wl < a.words) {
            ma = opA.sbits[offA + wl];
            mb = opB.sbits[offB + wl];
            pa = opA.spos[offA + wl];
            pb = opB.spos[offB + wl];
          }
          const uint32_t mw = ma & mb;
          const int cnt = __popc(mw);
          int incl = cnt;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULLW, incl, o);
            if (lane >= o) incl += v;
          }
          const int total = __shfl_sync(FULLW, incl, 31);
          const int excl = incl - cnt;
          // records (A, B) of step j of this chunk and their header bytes
          auto fetch = [&](int j, int& ea, int& eb, uint32_t& ha, uint32_t& hb) {
            ea = eb = 0;
            ha = hb = HEAD_NONE;
            int L = 0;   // lanes whose prefix is <= j: the word lane of step j
#pragma unroll
            for (int h = 16; h > 0; h >>= 1)
              if (__shfl_sync(FULLW, incl, L + h - 1) <= j) L += h;
            const int Lc = min(L, 31);
            const uint32_t mL = __shfl_sync(FULLW, mw, Lc);
            const uint32_t maL = __shfl_sync(FULLW, ma, Lc);
            const uint32_t mbL = __shfl_sync(FULLW, mb, Lc);
            const int paL = __shfl_sync(FULLW, pa, Lc);
            const int pbL = __shfl_sync(FULLW, pb, Lc);
            const int exL = __shfl_sync(FULLW, excl, Lc);
            if (j < total) {
              // position of the set bit number j - exL
              uint32_t m = mL;
              int r = j - exL, pos = 0;
#pragma unroll
              for (int h = 16; h > 0; h >>= 1) {
                const int c = __popc(m & ((1u << h) - 1u));
                if (r >= c) {
                  r -= c;
                  m >>= h;
                  pos += h;
                }
              }
              const uint32_t below = (1u << pos) - 1u;
              ea = paL + __popc(maL & below);
              eb = pbL + __popc(mbL & below);
              ha = opA.head[ea];
              hb = opB.head[eb];
            }
          };
          int ea, eb;
          uint32_t ha, hb;
          fetch(lane, ea, eb, ha, hb);
          for (int jb = 0; jb < total && ok; jb += 32) {
            int ea_n, eb_n;
            uint32_t ha_n, hb_n;
            fetch(jb + 32 + lane, ea_n, eb_n, ha_n, hb_n);   // next batch, in flight during this one
            const uint32_t pa4 = (ha >> 4) & 0xFu;
            const uint32_t eb4 = (((hb >> 4) & 0xFu) * 0x00204081u) & 0x01010101u;   // one byte per B tile
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] += ((pa4 >> q) & 1u) ? eb4 : 0u;
            if (++nacc == 255) flush_counts();
            const uint4 sv = steps[(ha & 7u) * 8u + (hb & 7u)];   // HEAD_NONE: no sub-steps (and no products)
            nprod += (unsigned)(__popc((sv.x >> 4) & 15u) + __popc((sv.y >> 4) & 15u) + __popc((sv.z >> 4) & 15u));
            int ns = (int)sv.w;
            // a segmented tile also closes a segment before every seg_ksteps-th K
            // step inside the batch (the batch end closes one too)
            const int lead = (segmented && lane > 0 && (lane % a.seg_ksteps) == 0 && jb + lane < total) ? 1 : 0;
            const uint32_t ua = (uint32_t)ea * K + ((sv.x >> 22) & 7u), ub = (uint32_t)eb * K + ((sv.x >> 27) & 7u);
            // K steps of one product each are taken in pairs, in order: lane l of
            // an even number of single steps since the last other step (or segment
            // end) takes the next single step with it
            uint32_t rv0 = sv.x, second = 0u;
            const bool single = ns == 1 && ((sv.x >> 4) & 0xFu) == 1u;
            const uint32_t sm = __ballot_sync(FULLW, single), mm = __ballot_sync(FULLW, ns > 0 && !single);
            const uint32_t lt = (1u << lane) - 1u;
            int run0 = 32 - __clz(mm & lt);                     // first lane of the run
            if (segmented) run0 = max(run0, lane - lane % a.seg_ksteps);
            const int rank = __popc(sm & lt & ~((1u << run0) - 1u));
            const uint32_t later = sm & ~lt & ~(1u << lane);
            const int nxt = later ? __ffs(later) - 1 : lane;
            const uint32_t ua2 = __shfl_sync(FULLW, ua, nxt), ub2 = __shfl_sync(FULLW, ub, nxt);
            const bool fits = nxt > lane && (mm & ~lt & ((1u << nxt) - 1u)) == 0u &&
                              (!segmented || nxt / a.seg_ksteps == lane / a.seg_ksteps);
            if (single) {
              if (rank & 1) {
                ns = 0;      // taken by the step before
              } else if (fits) {
                rv0 = (rv0 & ~((3u << 20) | (3u << 25))) | REC_PAIR | (1u << 7) | (2u << 20) | (2u << 25);
                second = (ua2 - ua) | ((ub2 - ub) << 16);
              }
            }
            // groups that a sub-step writes first in its segment (seg0: the lane where
            // the segment begins)
            const uint32_t need0 = ns > 0 ? (sv.x >> 8) & 15u : 0u, need1 = ns > 1 ? (sv.y >> 8) & 15u : 0u;
            const uint32_t need2 = ns > 2 ? (sv.z >> 8) & 15u : 0u;
            const int seg0 = segmented ? lane - lane % a.seg_ksteps : 0;
            uint32_t before = seg0 == 0 ? wmask : 0u, all = 0u;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              const uint32_t bal = __ballot_sync(FULLW, ((need0 | need1 | need2) >> g) & 1u);
              if (bal & lt & ~((1u << seg0) - 1u)) before |= 1u << g;
              if (bal) all |= 1u << g;
            }
            wmask = segmented ? 0u : wmask | all;      // a segmented tile's batch ends its segment
            const uint32_t fr0 = (need0 & ~before) << 16, fr1 = (need1 & ~(before | need0)) << 16;
            const uint32_t fr2 = (need2 & ~(before | need0 | need1)) << 16;
            int soff = ns + lead;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const int v = __shfl_up_sync(FULLW, soff, o);
              if (lane >= o) soff += v;
            }
            int nsub = __shfl_sync(FULLW, soff, 31);
            soff -= ns;
            ok = batch_open();
            if (!ok) break;
            uint4* ul = plan + (nbat % NPLAN) * PLAN;
            const uint32_t pbit = pass ? REC_PASS1 : 0u;
            auto entry = [&](uint32_t rv) {
              return make_uint4(rv | pbit, (uint32_t)ea * K + ((rv >> 22) & 7u), (uint32_t)eb * K + ((rv >> 27) & 7u), 0u);
            };
            if (lead) ul[soff - 1] = make_uint4(REC_SEG, 0u, 0u, 0u);
            if (ns > 0) ul[soff] = make_uint4(rv0 | pbit | fr0, ua, ub, second);
            if (ns > 1) ul[soff + 1] = entry(sv.y | fr1);
            if (ns > 2) ul[soff + 2] = entry(sv.z | fr2);
            kdone += min(32, total - jb);
            if (segmented && kdone < ktot) {
              if (lane == 0) ul[nsub] = make_uint4(REC_SEG, 0u, 0u, 0u);
              ++nsub;
            }
            batch_close(nsub);
            ea = ea_n;
            eb = eb_n;
            ha = ha_n;
            hb = hb_n;
          }
        }
      }
      // counts before the end record: the barriers of its batch, its sub-step and
      // its segment order them before the epilogue's reads
      flush_counts();
      if (lane < 16) kcount[b * 16 + lane] = kc;
      __syncwarp();
      if (ok) ok = batch_ctl(REC_END);
    }
    // slice-pair products (each 2 MMAs of 128 x 128 x 16)
    if (a.err && nprod) atomicAdd(reinterpret_cast<unsigned long long*>(a.err + 2), nprod);
  } else if (warp >= ISSUE_WARP) {
    // ---------------- issuers: one thread of warp 18 copies the A units of every
    // planned sub-step into the next stage, one of warp 19 the B units.
    if (elect_one()) {
      const int side = warp - ISSUE_WARP;      // 0: A, 1: B
      const uint32_t first_used = side ? 0x50u : 0x30u;       // products that read the side's first slice
      const uint32_t mine = smem_u32(stages) + (uint32_t)side * (2 * UNIT_BYTES);
      int s = 0;                     // next stage
      uint32_t par = 1u;             // phase that frees it
      int ready = 0;                 // stages from s on known to be free
      int head = 0;                  // sub-steps issued
      bool done = false;
      for (int bat = 0; !done; ++bat) {
        if (!mbar_wait_sleep(&plan_full[bat % NPLAN], (uint32_t)(bat / NPLAN) & 1u)) {
          status[0] = 1;
          note_timeout(a.err, 8);
          break;
        }
        const uint4* ul = plan + (bat % NPLAN) * PLAN;
        const int n = bcnt[bat % NPLAN];
        int u = 0;
        uint4 nx = ul[0];              // record u
        while (u < n) {
          if (nx.x & REC_CTL) {
            if (nx.x & REC_LAST) done = true;
            nx = ul[++u];
            continue;
          }
          if (ready == 0) {
            ready = mbar_ready4(empty, s, par, STAGES);
            if (ready == 0) {
              if (!mbar_wait(&empty[s], par)) {
                status[0] = 1;
                note_timeout(a.err, 2);
                done = true;
                break;
              }
              ready = 1;
            }
          }
          // the free stages' copies, without a wait or a test among them
          uint4 en = nx;
#pragma unroll 1
          do {
            const uint32_t rv = en.x;
            const uint32_t unit = side ? en.z : en.y, second = side ? en.w >> 16 : en.w & 0xFFFFu;
            en = ul[++u];
            const __half* base = ((rv & REC_PASS1) != 0u) == (side != 0) ? a.P.data : a.Q.data;
            const unsigned char* src = reinterpret_cast<const unsigned char*>(base) + (uint64_t)unit * UNIT_BYTES;
            const uint32_t bytes = ((rv >> (side ? 25 : 20)) & 3u) * UNIT_BYTES;
            const uint32_t part = second != 0u ? UNIT_BYTES : bytes;       // a pair: two copies
            const uint32_t dst = mine + (uint32_t)s * STAGE_BYTES + ((rv & first_used) ? 0u : (uint32_t)UNIT_BYTES);
            mbar_expect_tx(&full[s], bytes);
            bulk_g2s(dst, src, part, &full[s]);
            if (second != 0u) bulk_g2s(dst + UNIT_BYTES, src + (uint64_t)second * UNIT_BYTES, UNIT_BYTES, &full[s]);
            ++head;
            if (++s == STAGES) { s = 0; par ^= 1u; }
            --ready;
          } while (ready > 0 && u < n && (en.x & REC_CTL) == 0u);
          nx = en;
        }
        mbar_arrive(&plan_empty[bat % NPLAN]);
      }
      // no bulk copy into this CTA's shared memory may be in flight when the CTA
      // exits: wait (bounded) for those of the last STAGES sub-steps
      for (int j = max(0, head - STAGES); j < head; ++j)
        if (!mbar_wait(&full[j % STAGES], (uint32_t)(j / STAGES) & 1u)) {
          status[0] = 1;
          note_timeout(a.err, 9);
        }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (elect_one()) {
    // ---------------- MMA issuer, one thread.  TMEM is four blocks of 128 columns; a group
    // accumulator of a segment (a whole super-tile, or seg_ksteps of its K steps) takes
    // a free block on its first product, and the blocks of a segment return to
    // the pool once every epilogue warp has read them (one arrival per warp on
    // the segment slot's tmem_empty barrier; segments are reclaimed in order).
    uint32_t free_mask = 0xFu;
    // blocks held by the segment in each ring slot (4 slots)
    uint32_t pend0 = 0u, pend1 = 0u, pend2 = 0u, pend3 = 0u;
    int released = 0;              // segments whose blocks are back in free_mask
    int seg = 0;                   // segments published
    bool ok = true, done = false;
    // the shared-memory descriptor of a unit is that of the first stage plus
    // a constant (the start-address field holds address / 16 in 14 bits; every
    // address here is below 2^18)
    const uint64_t dring = make_desc(smem_u32(stages), 128, 512);
    const uint32_t dlo = (uint32_t)dring & 0xFFFFu;              // start address / 16 (below 2^14 for every unit)
    const uint64_t dhi = dring & ~0xFFFFull;
    // take back the blocks of the oldest segment that still holds some; false on timeout
    auto reclaim = [&]() -> bool {
      if (!mbar_wait(&tmem_empty[released & (SEG_RING - 1)], ((uint32_t)released >> 2) & 1u)) {
        note_timeout(a.err, 4);
        return false;
      }
      tc_fence_after();
      switch (released & (SEG_RING - 1)) {
        case 0: free_mask |= pend0; pend0 = 0u; break;
        case 1: free_mask |= pend1; pend1 = 0u; break;
        case 2: free_mask |= pend2; pend2 = 0u; break;
        default: free_mask |= pend3; pend3 = 0u; break;
      }
      ++released;
      return true;
    };
    int s = 0;               // next stage and the phase that fills it
    uint32_t par = 0u;
    int ready = 0;           // stages from s on known to be full
    uint32_t gblk = 0u, used = 0u, written = 0u;   // open segment: block of each group, blocks, groups
    // the products of a sub-step, from the next stage; fr: groups (from the first
    // product's on) that it writes first, its first MMA into them overwrites
    auto sub_step = [&](uint32_t rv, uint32_t fr) {
      const uint32_t units = dlo + (uint32_t)s * (STAGE_BYTES >> 4);    // A0, A1, B0, B1 one unit apart
      const int base = (int)(rv & 7u) - 1;     // group of A0 x B0
      const uint32_t gb = base >= 0 ? gblk >> (2 * base) : gblk << 2;    // blocks of groups base, base + 1, base + 2
      // the unit of the super-column as the M operand, that of the super-row
      // as the N operand: TMEM holds the transposed super-tile
      auto product = [&](int i, int j, int k, uint32_t acc) {
        const uint32_t dcol = tmem + ((gb >> (2 * k)) & 3u) * ST;
        const uint32_t ua = units + (uint32_t)(i * (UNIT_BYTES >> 4)), ub = units + (uint32_t)((2 + j) * (UNIT_BYTES >> 4));
        mma_f16(dcol, dhi | ub, dhi | ua, acc);
        mma_f16(dcol, dhi | (ub + 16u), dhi | (ua + 16u), 1u);
      };
      if (rv & REC_PAIR) {
        product(0, 0, 0, (fr & 1u) ^ 1u);
        product(1, 1, 0, 1u);
      } else {
        if (rv & (1u << 4)) product(0, 0, 0, (fr & 1u) ^ 1u);
        if (rv & (1u << 5)) product(0, 1, 1, ((fr >> 1) & 1u) ^ 1u);
        if (rv & (1u << 6)) product(1, 0, 1, (((fr >> 1) & 1u) ^ 1u) | ((rv >> 5) & 1u));
        if (rv & (1u << 7)) product(1, 1, 2, ((fr >> 2) & 1u) ^ 1u);
      }
      mma_commit(&empty[s]);
      if (++s == STAGES) { s = 0; par ^= 1u; }
    };
    for (int bat = 0; ok && !done; ++bat) {
      if (!mbar_wait_sleep(&plan_full[bat % NPLAN], (uint32_t)(bat / NPLAN) & 1u)) {
        note_timeout(a.err, 8);
        ok = false;
        break;
      }
      const uint4* ul = plan + (bat % NPLAN) * PLAN;
      const int n = bcnt[bat % NPLAN];
      int u = 0;
      uint32_t nx = ul[0].x;   // record u
      while (u < n) {
        const uint32_t rv = nx;
        if (rv & REC_CTL) {
          if (rv & REC_LAST) { done = true; break; }
          // publish the segment in ring slot seg % SEG_RING once the segment that used
          // the slot before has been read and its blocks reclaimed
          while (released < seg - (SEG_RING - 1) && ok) ok = reclaim();
          if (!ok) break;
          const int q = seg & (SEG_RING - 1);
          switch (q) {
            case 0: pend0 = used; break;
            case 1: pend1 = used; break;
            case 2: pend2 = used; break;
            default: pend3 = used; break;
          }
          gmap[q] = written | (gblk << 8) | ((rv & REC_END) ? SEG_LAST : 0u);
          mma_commit(&acc_full[q]);    // arrives once every MMA of the segment has completed
          mbar_arrive(&acc_full[q]);   // release: segment record visible to the epilogue
          ++seg;
          gblk = used = written = 0u;
          nx = ul[++u].x;
          continue;
        }
        if (ready == 0) {
          ready = mbar_ready4(full, s, par, STAGES);
          if (ready == 0) {
            if (!mbar_wait(&full[s], par)) {
              ok = false;
              note_timeout(a.err, 3);
              break;
            }
            ready = 1;
          }
        }
        if (rv & REC_FRESH) {
          // groups (relative to the launch's window, at most four live) that the
          // segment writes first here take a TMEM block
          for (uint32_t f = (rv >> 16) & 15u; f != 0u; f &= f - 1u) {
            const int g = __ffs(f) - 1;
            while (free_mask == 0u && ok) ok = reclaim();
            if (!ok) break;
            const uint32_t blk = (uint32_t)(__ffs(free_mask) - 1);
            free_mask &= ~(1u << blk);
            used |= 1u << blk;
            gblk |= blk << (2 * g);
            written |= 1u << g;
          }
          if (!ok) break;
          const int base = (int)(rv & 7u) - 1;
          uint32_t fr = (rv >> 16) & 15u;
          fr = base >= 0 ? fr >> base : fr << 1;
          nx = ul[++u].x;
          sub_step(rv, fr);
          --ready;
          continue;
        }
        // the full stages' sub-steps, without a wait or a test among them
        uint32_t r = rv;
#pragma unroll 1
        do {
          const uint32_t cur = r;
          r = ul[++u].x;
          sub_step(cur, 0u);
          --ready;
        } while (ready > 0 && u < n && (r & (REC_CTL | REC_FRESH)) == 0u);
        nx = r;
      }
      mbar_arrive(&plan_empty[bat % NPLAN]);
    }
    if (!ok) status[0] = 1;
    mma_commit(drain);
    if (!mbar_wait(drain, 0)) {
      status[0] = 1;
      note_timeout(a.err, 5);
    }
    }
    __syncwarp();
  } else if (warp >= 2) {
    // ---------------- epilogue (warps 2-17, four per SM sub-partition).  TMEM holds
    // the super-tile transposed (lane = column, TMEM column = row): warp w reads
    // TMEM lanes 32 (w % 4)..+31 = tile column J0 + w % 4, lane = column inside
    // the tile; four warps share each tile column, one per row tile.  So the
    // 32 lanes of a warp hold 32 consecutive elements of a row of the row-major
    // tiles, and every access to the scratch, to X~ and to X_new is one
    // contiguous 256-byte piece.  With lane = row each 16-byte access touched 32
    // separate sectors, and the load/store unit cost as much as the FP64 pipe:
    // whole runs, before -> after: water-like N = 24,000 188.1 -> 172.3 ms, dense
    // N = 4,096 with five slices 95.7 -> 77.4 ms, same bits.
    // Phase 1 moves the exact fixed-point sums to the CTA's scratch and returns
    // the TMEM blocks, so the next tile's products run during phase 2, the FP64
    // arithmetic.  A thread reads back only what it wrote, so one scratch slot
    // per CTA serves all tiles.
    // Sixteen warps, one tile each, keep the FP64 pipe busier than eight with two
    // tiles each (phase 2 of a super-tile 63,000 -> 51,000 cycles at N = 24,000;
    // 1.7 to 2 FP64 lane operations per SM cycle are its floor).  The loops are
    // rolled over row chunks and groups, which keeps the code short (the
    // sub-partition's instruction cache is shared with the issuers) and the
    // registers below the 102 that 640 threads leave.
    constexpr int CH = 8;       // rows of a tile in one chunk of phase 2
    const int quarter = warp & 3;
    const int bt = (warp - 2) >> 2;
    // unit of the finest group of the window: with W bits per slice, slice s
    // lies on the grid 2^-(W s + W - 1), so group g = s + t has the unit
    // 2^-(W g + 2 W - 2)
    constexpr int W = slice_bits(K);
    const double su = ldexp(1.0, -(W * ghi + 2 * W - 2)) * a.scale;   // S = fx * su, su a power of two
    const int lsu = ilogb(su);
    // X_new = c0 I + c1 X~ + c2 S.  Without acceleration (alpha = 1) the two
    // polynomials need fewer FP64 operations, with the same results:
    //   x^2 (c0 = c1 = 0, c2 = 1): S itself;  2x - x^2 (c0 = 0, c1 = 2, c2 = -1): 2 z - S.
    const int form = (a.c0 == 0.0 && a.c1 == 0.0 && a.c2 == 1.0) ? 1
                   : (a.c0 == 0.0 && a.c1 == 2.0 && a.c2 == -1.0) ? 2 : 0;
    // index of tile (row, col) in a pattern given by row bitmaps, the bits before
    // each word and row offsets, -1 if absent
    auto find = [&](const uint32_t* bits, const int32_t* wpre, const int32_t* rowptr, int row, int col) -> int {
      const int64_t w = (int64_t)row * a.words + (col >> 5);
      const uint32_t m = bits[w];
      if (!((m >> (col & 31)) & 1u)) return -1;
      return rowptr[row] + wpre[w] + __popc(m & ((1u << (col & 31)) - 1u));
    };
    int seg = 0;   // segments consumed
    const uint64_t pol = policy_evict_last();
    for (int it = 0;; ++it) {
      const int b = it % NSLOT;
      const uint32_t par = ((uint32_t)(it / NSLOT)) & 1u;
      bool good = true;
      if (lane == 0) good = mbar_wait_sleep(&tile_full[b], par);
      good = __shfl_sync(FULLW, good ? 1 : 0, 0) != 0;
      if (!good) { if (lane == 0) { status[0] = 1; note_timeout(a.err, 6); } break; }
      __syncwarp();
      const int idx = tslot[b];
      if (idx < 0) break;
      const int stile = a.list[idx];
      const int R = stile / a.nsr, C = stile % a.nsr;
      const int I0 = 4 * R, J0 = 4 * C;
      const int Jb = J0 + quarter;           // tile column of this thread
      const int64_t gj = (int64_t)Jb * TB + lane;
      // scratch element of super-tile row i: scr[i * ST]
      long long* scr = a.scratch + (int64_t)blockIdx.x * (ST * ST) + quarter * 32 + lane;
      const int Ia = I0 + bt;                // tile row of this warp
      // output tile index
      const int oi = (Ia < a.nb && Jb < a.nb && (a.general || Ia <= Jb)) ? find(a.obits, a.owpre, a.orowptr, Ia, Jb) : -1;
      // Z_IJ of the output tile (X~_IJ in the forward step; absent -> null),
      // looked up and its rows requested into L2 before the accumulators are
      // waited for, so that the chain of dependent loads overlaps the wait
      const double* Z = nullptr;
      if (oi >= 0 && emode != 1) {
        const int zp = find(a.zbits, a.zwpre, a.zrowptr, Ia, Jb);
        if (zp >= 0) {
          const int64_t zi = (int64_t)(a.zref[zp] & ~REF_T);
          Z = a.zpool + (int64_t)(a.zslot ? a.zslot[zi] : zi) * TE;
          prefetch_l2(Z + lane * TB);
          prefetch_l2(Z + lane * TB + 16);
        }
      }
      // phase 1, once per accumulation segment: TMEM -> the exact fixed-point
      // sums of this thread's column in the scratch (the first segment stores, the
      // others add), then the segment's TMEM blocks go back to the MMA issuer
      for (bool first = true;; first = false) {
        const int q = seg & (SEG_RING - 1);
        const uint32_t spar = ((uint32_t)seg >> 2) & 1u;
        if (lane == 0) good = mbar_wait_sleep(&acc_full[q], spar);
        good = __shfl_sync(FULLW, good ? 1 : 0, 0) != 0;
        if (!good) {
          if (lane == 0) note_timeout(a.err, 7);
          break;
        }
        __syncwarp();
        tc_fence_after();
        const uint32_t gm = gmap[q];
        const uint32_t written = gm & 0xFu;
        // The group sums are integers, converted by the 32-bit instruction, which
        // saturates.  With two to four slices nothing bounds them by 2^31: second
        // slices reach 2^10, and a K loop without segments has thousands of products
        // of each of a group's pairs, all of one sign on a diagonal that does not come
        // from dsq or between alike rows.  A warp that met such a sum adds what the
        // conversion lost afterwards; the vote on that stands where the warp has to
        // meet anyway.  Squares of the water-like N = 192,000 case: 1,327 ms without a
        // test (and wrong sums), 1,331 so, 1,337 with a vote after each 16 rows, and a
        // vote before each group's conversion cost whole runs 0.4% to 0.9%.  Five
        // slices: 256 products a segment of at most 2^20 + 3 2^18, below 2^29.
        float top = 0.0f;
#pragma unroll 1
        for (int hc = 0; hc < 2 && oi >= 0; ++hc) {       // 16 rows at a time
          const int row0 = bt * 32 + hc * 16;
          long long fx[16];
          long long* sp = scr + row0 * ST;
#pragma unroll
          for (int i = 0; i < 16; ++i) fx[i] = 0;
          const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)row0;
#pragma unroll 1
          for (int gg = 0; gg <= ghi - glo; ++gg) {   // relative groups of the window, coarsest first
#pragma unroll
            for (int i = 0; i < 16; ++i) fx[i] *= 1ll << W;
            if ((written >> gg) & 1u) {        // warp-uniform: groups no product reached are zero
              float g[16];
              tmem_ld16(trow + ((gm >> (8 + 2 * gg)) & 3u) * ST, g);
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                if (K != 5) top = fmaxf(top, fabsf(g[i]));
                fx[i] += __float2int_rn(g[i]);
              }
            }
          }
          if (!first) {
#pragma unroll
            for (int i = 0; i < 16; ++i) fx[i] += ld_staging(sp + i * ST, pol);
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) st_staging(sp + i * ST, fx[i], pol);
        }
        // this warp's TMEM reads of the segment are complete (the vote is also the
        // warp's barrier)
        tc_fence_before();
        if (__any_sync(FULLW, K != 5 && top >= 2147483648.0f)) {
#pragma unroll 1
          for (int u = 0; u < 8 * (ghi - glo + 1); ++u) {       // 4 rows of a group at a time
            const int gg = u >> 3, row0 = bt * 32 + (u & 7) * 4;
            if (!((written >> gg) & 1u)) continue;
            float g[4];
            tmem_ld4(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)row0 + ((gm >> (8 + 2 * gg)) & 3u) * ST, g);
            long long* sp = scr + row0 * ST;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const long long lost = __float2ll_rn(g[i]) - __float2int_rn(g[i]);
              if (lost != 0)
                st_staging(sp + i * ST, ld_staging(sp + i * ST, pol) + lost * (1ll << (W * (ghi - glo - gg))), pol);
            }
          }
          tc_fence_before();
          __syncwarp();
        }
        if (lane == 0) mbar_arrive(&tmem_empty[q]);
        ++seg;
        if (gm & SEG_LAST) break;
      }
      if (!good) { if (lane == 0) status[0] = 1; break; }
      // phase 2: X_new, per-tile ||X~ - S||^2, ||X_new||^2 and traces
      if (oi >= 0) {
        double trS = 0.0, trX = 0.0, n2 = 0.0, e2 = 0.0;
        double* O = a.opool + (int64_t)oi * TE;
        // Everything that only some tiles need (the matrix edge, the diagonal) is
        // under a branch of its own, outside the loops over the chunk's rows: the
        // kernel is long for the instruction caches (99 KB; one instruction fetch in
        // nine missed the multiprocessor's cache), and the single-thread loops of the
        // issuers, which bound it, wait for their share of the misses.  With the
        // cases inside the row loops: water-like N = 24,000 115 ms a run, now 105,
        // N = 96,000 705 ms, now 610, dense N = 4,096 with five slices 47.0, now 45.7.
        const bool edge = (int64_t)(Ia + 1) * TB > a.n || (int64_t)(Jb + 1) * TB > a.n;
        const bool diag = Ia == Jb;
        const bool general = Z != nullptr || (form == 0 && diag);
#pragma unroll 1
        for (int ch = 0; ch < TB / CH; ++ch) {     // CH rows per chunk
          const long long* sp = scr + (bt * 32 + ch * CH) * ST;
          const int e0 = ch * CH * TB + lane;     // element of the chunk's first row in a tile
          double zv[CH];
          if (Z) {
#pragma unroll
            for (int i = 0; i < CH; ++i) zv[i] = Z[e0 + i * TB];
          } else {
#pragma unroll
            for (int i = 0; i < CH; ++i) zv[i] = 0.0;
          }
          long long fx[CH];
#pragma unroll
          for (int i = 0; i < CH; ++i) fx[i] = ld_staging(sp + i * ST, pol);
          // emode 2: the finer groups' S, left in the output tile by the launch before
          double prev[CH];
          if (emode == 2) {
#pragma unroll
            for (int i = 0; i < CH; ++i) prev[i] = O[e0 + i * TB];
          } else {
#pragma unroll
            for (int i = 0; i < CH; ++i) prev[i] = 0.0;
          }
          if (edge) {
            const int rows = gj < a.n ? (int)min((int64_t)CH, a.n - ((int64_t)Ia * TB + ch * CH)) : 0;
#pragma unroll
            for (int i = 0; i < CH; ++i)
              if (i >= rows) {
                fx[i] = 0;
                zv[i] = 0.0;
              }
          }
          // S = fx * su.  The sums of an iterate are below 2^53 units (|S_ij| <= 1),
          // and then the conversion is exact and done on the integer pipes, all
          // elements of the chunk side by side; the conversion instruction would
          // take a slot of the FP64 pipe (phase 2 of a super-tile at N = 24,000:
          // 51,000 -> 43,000 cycles; with a test for each element 84,000)
          double S[CH];
          bool large = false;
#pragma unroll
          for (int i = 0; i < CH; ++i) large |= ((unsigned long long)(fx[i] < 0 ? -fx[i] : fx[i]) >> 53) != 0ull;
          if (__any_sync(FULLW, large)) {
#pragma unroll
            for (int i = 0; i < CH; ++i) S[i] = int_times_pow2((double)fx[i], lsu);
          } else {
#pragma unroll
            for (int i = 0; i < CH; ++i) S[i] = small_ll_times_pow2(fx[i], lsu);
          }
          double out[CH];      // emode 1 (finer groups only): S
          if (emode == 2) {
#pragma unroll
            for (int i = 0; i < CH; ++i) S[i] += prev[i];
          }
          if (emode == 1) {
#pragma unroll
            for (int i = 0; i < CH; ++i) out[i] = S[i];
          } else {
            const int dr = diag && gj < a.n ? lane - ch * CH : -1;      // the chunk's row on the diagonal
            if (dr >= 0 && dr < CH) {
              // the diagonal of S = X~^2 is the squared row norm, taken in FP64
              // (its digit products are all positive and pass the exact range
              // of the FP32 group sums on dense rows)
              const double nrm = a.dsq ? a.dsq[gj] : 0.0;
#pragma unroll
              for (int i = 0; i < CH; ++i)
                if (i == dr) {
                  if (a.dsq) S[i] = nrm;
                  trS += S[i];
                  trX += zv[i];
                }
            }
            if (general) {
              if (form == 1) {
#pragma unroll
                for (int i = 0; i < CH; ++i) out[i] = S[i];
              } else if (form == 2) {
#pragma unroll
                for (int i = 0; i < CH; ++i) out[i] = twice(zv[i]) - S[i];
              } else {
                // c2 S = (c2 su) fx exactly (su is a power of two)
#pragma unroll
                for (int i = 0; i < CH; ++i) out[i] = fma(a.c2, S[i], fma(a.c1, zv[i], i == dr ? a.c0 : 0.0));
              }
#pragma unroll
              for (int i = 0; i < CH; ++i) {
                const double df = zv[i] - S[i];
                e2 = fma(df, df, e2);
                n2 = fma(out[i], out[i], n2);
              }
            } else {
              // no X~ tile here: z = 0.  X_new = S or 2 z - S = -S (forms 1 and 2):
              // every (z - S)^2 equals X_new^2, so one FMA per element gives both sums
              // (e2 is set from n2 below; the same values in the same order).  With
              // acceleration (form 0) ||X_new||^2 is c2^2 ||S||^2; a tile without
              // X~ tile on the diagonal, where c0 counts, takes the path above.
#pragma unroll
              for (int i = 0; i < CH; ++i) n2 = fma(S[i], S[i], n2);
              if (form == 0) {
#pragma unroll
                for (int i = 0; i < CH; ++i) out[i] = fma(a.c2, S[i], 0.0);
              } else {
#pragma unroll
                for (int i = 0; i < CH; ++i) out[i] = form == 1 ? S[i] : negated(S[i]);
              }
            }
          }
#pragma unroll
          for (int i = 0; i < CH; ++i) O[e0 + i * TB] = out[i];
        }
        if (!general) {
          e2 = n2;
          if (form == 0) n2 = (a.c2 * a.c2) * n2;
        }
        // warp reductions (the tile's 32 columns are this warp's 32 lanes)
        for (int o = 16; o > 0; o >>= 1) {
          e2 += __shfl_xor_sync(FULLW, e2, o);
          n2 += __shfl_xor_sync(FULLW, n2, o);
          trS += __shfl_xor_sync(FULLW, trS, o);
          trX += __shfl_xor_sync(FULLW, trX, o);
        }
        if (lane == 0 && emode != 1) {
          a.part.e2[oi] = (diag || a.general ? 1.0 : 2.0) * e2;
          a.part.n2[oi] = n2;
          a.part.trS[oi] = diag ? trS : 0.0;
          a.part.trX[oi] = diag ? trX : 0.0;
          a.part.ktiles[oi] = kcount[b * 16 + bt * 4 + quarter];
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&tile_empty[b]);
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
  if (threadIdx.x == 0 && status[0] != 0 && a.err) atomicOr(a.err, 1);
}

inline unsigned grid_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

size_t panel_record_bytes(int k) { return (size_t)k * UNIT_BYTES; }

cudaError_t launch_panel_slices(const uint32_t* index, int64_t nrec, const int32_t* slot, const double* pool,
                                void* data, uint8_t* head, int k, int32_t* err, double* rsq, double scale,
                                bool report_range, cudaStream_t st) {
  if (nrec == 0) return cudaSuccess;
  const uint4* ix = reinterpret_cast<const uint4*>(index);
  __half* d = static_cast<__half*>(data);
  const int ls = ilogb(scale);   // scale is a power of two
  const int rr = report_range ? 1 : 0;
  const unsigned g = (unsigned)nrec;
  ++g_launches;
  if (k == 2) k_panel_slices<2><<<g, 256, 0, st>>>(ix, slot, pool, d, head, err, rsq, ls, rr);
  else if (k == 3) k_panel_slices<3><<<g, 256, 0, st>>>(ix, slot, pool, d, head, err, rsq, ls, rr);
  else if (k == 5) k_panel_slices<5><<<g, 256, 0, st>>>(ix, slot, pool, d, head, err, rsq, ls, rr);
  else k_panel_slices<4><<<g, 256, 0, st>>>(ix, slot, pool, d, head, err, rsq, ls, rr);
  return cudaGetLastError();
}

// Record index words: one warp per tile row; every stored tile (row, K) of the
// both-triangle pattern writes its word (slot row % 4) of the record of
// (super-row row / 4, K): compact tile index, bit 31 when the stored tile is
// used transposed.  Words start all ones (absent).
__global__ void k_panel_fill(const int32_t* __restrict__ frowptr, const int32_t* __restrict__ fcol,
                             const uint32_t* __restrict__ fref, const uint32_t* __restrict__ sbits,
                             const int32_t* __restrict__ spos, int nb, int words, uint32_t* index) {
  const int row = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= nb) return;
  const int64_t o = (int64_t)(row >> 2) * words;
  for (int p = frowptr[row] + lane; p < frowptr[row + 1]; p += 32) {
    const int k = fcol[p];
    const int w = k >> 5;
    const int64_t e = spos[o + w] + __popc(sbits[o + w] & ((1u << (k & 31)) - 1u));
    index[e * 4 + (row & 3)] = fref[p];
  }
}

cudaError_t launch_row_sq_sum(const int32_t* spos, int nsr, int words, const double* rsq, int64_t n, double* dsq,
                              cudaStream_t st) {
  if (nsr == 0) return cudaSuccess;
  ++g_launches;
  k_row_sq_sum<<<(unsigned)nsr, 128 * SQ_GROUPS, 0, st>>>(spos, words, rsq, n, dsq);
  return cudaGetLastError();
}

cudaError_t launch_panel_fill(const FullPattern& fp, int nb, const uint32_t* sbits, const int32_t* spos,
                              uint32_t* index, cudaStream_t st) {
  if (nb == 0) return cudaSuccess;
  ++g_launches;
  k_panel_fill<<<grid_for((int64_t)nb * 32, 256), 256, 0, st>>>(fp.rowptr, fp.col, fp.ref, sbits, spos, nb, fp.words,
                                                                 index);
  return cudaGetLastError();
}

// max |x| over the tiles of a set (for the power-of-two slice scale of G)
__global__ void k_absmax(const int32_t* __restrict__ slot, const double* __restrict__ pool, int64_t nnzb,
                         unsigned long long* out) {
  double m = 0.0;
  for (int64_t t = blockIdx.x; t < nnzb; t += gridDim.x) {
    const double* x = pool + (int64_t)slot[t] * TE;
    for (int q = threadIdx.x; q < TE; q += blockDim.x) m = fmax(m, fabs(x[q]));
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

cudaError_t launch_absmax(const TileSet& x, const double* pool, unsigned long long* out, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned long long), st);
  if (e != cudaSuccess || x.nnzb == 0) return e;
  ++g_launches;
  k_absmax<<<(unsigned)std::min<int64_t>(x.nnzb, 152 * 8), 256, 0, st>>>(x.slot, pool, x.nnzb, out);
  return cudaGetLastError();
}

// upper-triangle bitmap of a tile set (bit J of row I for I <= J only)
__global__ void k_upper_bits(const int32_t* __restrict__ brow, const int32_t* __restrict__ bcol, int64_t nnzb,
                             uint32_t* bits, int words) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nnzb) return;
  const int i = brow[t], j = bcol[t];
  atomicOr(&bits[(int64_t)i * words + (j >> 5)], 1u << (j & 31));
}

cudaError_t launch_upper_bits(const TileSet& x, int nb, int words, uint32_t* bits, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(bits, 0, (size_t)nb * words * 4, st);
  if (e != cudaSuccess || x.nnzb == 0) return e;
  ++g_launches;
  k_upper_bits<<<grid_for(x.nnzb, 256), 256, 0, st>>>(x.brow, x.bcol, x.nnzb, bits, words);
  return cudaGetLastError();
}

// Words of the super-row bitmaps up to which one cluster makes them; above, three
// launches.  One cluster -> three launches: 31,500 words 10.3 -> 14.5 us, 49,375
// 16.5 -> 14.4, 282,000 (N = 192,000) 53 -> 17, 34 million (65,535 tile rows) 5,700 -> 173.
constexpr int64_t SUPER_CLUSTER_MAX = 1 << 15;

cudaError_t launch_super_scan(const FullPattern& fp, int nb, int nsr, uint32_t* sb, int32_t* spos, int32_t* total,
                              cudaStream_t st) {
  if ((int64_t)nsr * fp.words <= SUPER_CLUSTER_MAX) {
    ++g_launches;
    k_super_scan<<<SCAN_CTAS, SCAN_THREADS, 0, st>>>(fp.bits, nb, fp.words, nsr, sb, spos, total);
    return cudaGetLastError();
  }
  const unsigned g = grid_for((int64_t)nsr * 32, 256);
  ++g_launches;
  k_super_counts<<<g, 256, 0, st>>>(fp.bits, nb, fp.words, nsr, sb, spos);
  ++g_launches;
  k_super_offsets<<<SCAN_CTAS, SCAN_THREADS, 0, st>>>(fp.words, nsr, spos, total);
  ++g_launches;
  k_super_positions<<<g, 256, 0, st>>>(sb, fp.words, nsr, spos);
  return cudaGetLastError();
}

int64_t super_order_size(int nsr) { return blocked_size(nsr); }

// Launch positions up to which one cluster lists the super-tiles; above, one
// launch over all SMs for each phase.  The cluster takes 9 us for 512 positions and
// 19 us for 37,000, the five launches 17 us for 37,000 and the gaps between them.
constexpr int64_t LIST_CLUSTER_MAX = 1 << 15;

cudaError_t launch_super_list(const uint32_t* obits, int nb, int words, int nsr, int32_t* list, int32_t* count,
                              int32_t* flag, int32_t* pos, void* tmp, cudaStream_t st, bool general) {
  const int64_t n = blocked_size(nsr);
  if (n <= LIST_CLUSTER_MAX) {
    ++g_launches;
    k_super_list<<<SCAN_CTAS, SCAN_THREADS, 0, st>>>(obits, nb, words, nsr, general ? 1 : 0, list, count);
    return cudaGetLastError();
  }
  ++g_launches;
  k_super_flags<<<grid_for(n, 256), 256, 0, st>>>(obits, nb, words, nsr, general ? 1 : 0, flag);
  cudaError_t e = launch_scan_i32(flag, pos, n, count, tmp, st);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(count + 1, 0, 4, st);
  if (e != cudaSuccess) return e;
  ++g_launches;
  k_super_fill<<<grid_for(n, 256), 256, 0, st>>>(flag, pos, n, nsr, list);
  return cudaGetLastError();
}

cudaError_t launch_square_tc(const TcLaunch& L, cudaStream_t st) {
  if (L.nsuper == 0) return cudaSuccess;
  TcArgs a;
  a.P = TcOperand{L.P.sbits, L.P.spos, L.P.head, static_cast<const __half*>(L.P.data)};
  a.Q = TcOperand{L.Q.sbits, L.Q.spos, L.Q.head, static_cast<const __half*>(L.Q.data)};
  a.two_pass = L.two_pass ? 1 : 0;
  a.zbits = L.Z->bits; a.zwpre = L.Z->wpre; a.zrowptr = L.Z->rowptr; a.zref = L.Z->ref; a.zslot = L.zslot; a.zpool = L.zpool;
  a.obits = L.obits; a.owpre = L.owpre; a.orowptr = L.orowptr; a.list = L.list; a.count = L.count; a.work = L.work;
  a.opool = L.opool;
  a.part = L.part; a.c0 = L.c0; a.c1 = L.c1; a.c2 = L.c2; a.scale = L.scale; a.n = L.n; a.nb = L.nb;
  a.words = L.words; a.nsr = L.nsr; a.err = L.err; a.scratch = static_cast<long long*>(L.scratch);
  a.seg_min = L.seg_min;
  a.seg_ksteps = L.seg_ksteps > 0 ? L.seg_ksteps : SEG_KSTEPS;
  a.wait_ns = L.wait_ns;
  a.selftest = L.selftest ? 1 : 0;
  a.general = L.general ? 1 : 0;
  a.dsq = L.dsq;
  a.glo = L.glo;
  a.ghi = L.ghi < 0 ? L.k - 1 : L.ghi;
  a.emode = L.emode;
  cudaError_t e = cudaSuccess;
  switch (L.k) {
    case 2:
      e = cudaFuncSetAttribute(k_square_tc<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, TcCfg<2>::SMEM);
      if (e == cudaSuccess) { ++g_launches; k_square_tc<2><<<(unsigned)L.nsuper, TC_THREADS, TcCfg<2>::SMEM, st>>>(a); }
      break;
    case 3:
      e = cudaFuncSetAttribute(k_square_tc<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, TcCfg<3>::SMEM);
      if (e == cudaSuccess) { ++g_launches; k_square_tc<3><<<(unsigned)L.nsuper, TC_THREADS, TcCfg<3>::SMEM, st>>>(a); }
      break;
    case 5:
      e = cudaFuncSetAttribute(k_square_tc<5>, cudaFuncAttributeMaxDynamicSharedMemorySize, TcCfg<5>::SMEM);
      if (e == cudaSuccess) { ++g_launches; k_square_tc<5><<<(unsigned)L.nsuper, TC_THREADS, TcCfg<5>::SMEM, st>>>(a); }
      break;
    default:
      e = cudaFuncSetAttribute(k_square_tc<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, TcCfg<4>::SMEM);
      if (e == cudaSuccess) { ++g_launches; k_square_tc<4><<<(unsigned)L.nsuper, TC_THREADS, TcCfg<4>::SMEM, st>>>(a); }
      break;
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace sp2
