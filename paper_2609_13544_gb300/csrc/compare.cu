// Golden-vs-candidate error signature on sm_103a.
//
// Computes, per tensor or per segment of a packed tensor list, the error
// statistics of Section IV-B-3 ("FI Assessment Scores": the error is the
// absolute difference of golden and faulty values; max, mean and variance
// of it) plus the relative error, the ULP distance, a five-way class and two
// 64-bin histograms.  Every output is exact: integer outputs bit for bit,
// sums as the exact real sum rounded once to nearest-even binary64.
//
// One kernel (compare_stage1) per call: a persistent grid streams both
// tensors once through per-warp rings of bulk copies (cp.async.bulk +
// mbarrier).  CTA b owns the contiguous element range [lo_b, lo_{b+1}); per
// segment piece it touches it adds its integer totals (counts, histograms,
// sum digits) to the segment's accumulator with atomics and writes its maxima
// to slot s + b; the CTA that finishes a segment's last piece merges the
// slots in CTA order, rounds the exact sums once, writes the outputs and
// clears the accumulator.  All merged quantities are integers or exact
// values, so the result depends neither on the grid nor on the order of the
// atomics.  Per element pair:
//   - a "window" pair -- same sign, a small ULP distance (so c - g is exact,
//     Sterbenz), |d| inside the window of the piece -- increments shared
//     counters: one that names its log2-relative bin and ULP distance, and
//     (16-bit types) one that names the value of d, from which the exact sums
//     follow at the end of the piece; float32 differences are added as
//     integers instead.  The tolerance test is one float32 fma rounded down.
//     Every pair of a vector takes these steps without a branch; equal ones
//     land in counters that are left out;
//   - the maxima: a pair above the CTA's bounds so far (a few per piece) sends
//     its warp through a slow path that updates the exact records, lowest
//     index on ties;
//   - every other pair (non-finite, sign change, zeros, wide gaps, outside
//     the window) is found by the same checks, listed and evaluated exactly
//     after the piece, with float32 error-free transforms and integer digits
//     added to a CTA-wide carry-save fixed-point accumulator.
// What bounds it: instruction issue.  Per vector of 8 pairs and lane the dense
// 16-bit loop executes about 210 (bfloat16) to 255 (binary16) instructions, a
// vector of equal pairs about 80; all but the FP32 adds and fmas issue at half
// rate.  The kernel before it compacted unequal pairs into a queue and kept
// histogram rows per thread, about 60 instructions per unequal pair and 30 per
// pair.  Measured (back-to-back calls, one GB300): 67 M bfloat16 pairs of
// which half differ 182 -> 88 us, 355 M binary16 pairs in 292 segments 1007 ->
// 445 us, 268 M bfloat16 pairs of which 0.3 % differ 264 -> 202 us, 25.6 M
// float32 pairs in 161 segments 222 -> 110 us.  What a small call takes (20 to
// 40 us) is latency: the window sample, the piece end, the finalization.  The
// 16-bit window does not move within a piece: 67 M binary16 pairs whose rows lie
// over eight decades, most of them general then, take 882 us, with the kernel
// before 534; over two decades 124 and 409.
// Binary64 arithmetic is avoided per element (GB300 runs it at a small
// fraction of float32 rate); binary64 values appear only as containers and
// in the once-per-segment rounding.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstdint>

#include "exact.cuh"
#include "inject_models.cuh"
#include "meanvar.cuh"
#include <nvtx3/nvToolsExt.h>
#include "peat_internal.h"

namespace peat {
namespace {

// ---------------------------------------------------------------------------
// element types
// ---------------------------------------------------------------------------
// UBMAX: the largest ULP-distance bit length the window's position allows
// for (the window's floor sits 40 - UB binades below the largest golden seen).
// LBMIN and LBMAX bound the window's floor binade Lb so that 2^Lexp is at least
// 2^-100 (Lexp = Lb - BIAS - MB) and 1.5 * 2^(Lexp+44) is finite.
template <int DT>
struct Tr;
template <>
struct Tr<PEAT_F32> {
  static constexpr int BYTES = 4, VEC = 4, MB = 23, BIAS = 127, EMAX = 255;
  static constexpr int UBMAX = 20, LBMIN = 50, LBMAX = 221;
  static constexpr uint32_t SIGN = 0x80000000u, MAG = 0x7FFFFFFFu, INF = 0x7F800000u;
};
template <>
struct Tr<PEAT_F16> {
  static constexpr int BYTES = 2, VEC = 8, MB = 10, EMAX = 31;
  static constexpr uint32_t SIGN = 0x8000u, MAG = 0x7FFFu, INF = 0x7C00u;
};
template <>
struct Tr<PEAT_BF16> {
  static constexpr int BYTES = 2, VEC = 8, MB = 7, EMAX = 255;
  static constexpr uint32_t SIGN = 0x8000u, MAG = 0x7FFFu, INF = 0x7F80u;
};

// CTA geometry: the 16-bit kernel keeps its tables once per SM (one CTA of 16
// warps), the float32 kernel runs two CTAs of 8 warps.
template <int DT>
struct Geo {
  static constexpr int NT = DT == PEAT_F32 ? 256 : 512;
  static constexpr int NW = NT / 32;
  static constexpr int CTAS = DT == PEAT_F32 ? 2 : 1;
};

template <int DT>
__device__ __forceinline__ float to_f32(uint32_t b) {
  if constexpr (DT == PEAT_F32) return __uint_as_float(b);
  else if constexpr (DT == PEAT_BF16) return __uint_as_float(b << 16);
  else return __half2float(__ushort_as_half((unsigned short)b));
}

template <int DT>
__device__ __forceinline__ uint32_t lane_bits(const uint4& v, int j) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  if constexpr (Tr<DT>::BYTES == 4) return w[j];
  else return (w[j >> 1] >> (16 * (j & 1))) & 0xFFFFu;
}

template <int DT>
__device__ __forceinline__ uint32_t load_scalar(const void* base, int64_t i) {
  if constexpr (Tr<DT>::BYTES == 4) return __ldg(reinterpret_cast<const uint32_t*>(base) + i);
  else return (uint32_t)__ldg(reinterpret_cast<const unsigned short*>(base) + i);
}

// The candidate of a fused call: the golden after the call's element-wise
// models, in order (the same arithmetic as the injector's passes).
// (out of line: the scalar paths that call it are rare, and one copy keeps
// the generation code out of their inlined bodies)
template <int DT>
__device__ __noinline__ uint32_t inj_chain(const CompareParams& p, uint32_t b, int64_t i) {
  for (int m = 0; m < p.inj_n; m++) {
    bool fired;
    b = inj::apply_model<DT>(b, i, p.inj[m].kind, p.inj[m].model, p.inj[m].threshold, p.inj[m].x, p.inj_k0,
                             p.inj_k1, fired);
  }
  return b;
}
// candidate element i (golden bits G): generated (fused) or read
template <int DT, bool INJ>
__device__ __forceinline__ uint32_t cand_at(const CompareParams& p, int64_t i, uint32_t G) {
  if constexpr (INJ) return inj_chain<DT>(p, G, i);
  else return load_scalar<DT>(p.c, i);
}
template <int DT>
__device__ __forceinline__ void unpack_vec(const uint4& v, uint32_t (&e)[16 / Tr<DT>::BYTES]) {
#pragma unroll
  for (int j = 0; j < 16 / Tr<DT>::BYTES; j++) e[j] = lane_bits<DT>(v, j);
}
template <int DT>
__device__ __forceinline__ uint4 pack_vec(const uint32_t (&e)[16 / Tr<DT>::BYTES]) {
  if constexpr (Tr<DT>::BYTES == 4) return make_uint4(e[0], e[1], e[2], e[3]);
  else
    return make_uint4(e[0] | (e[1] << 16), e[2] | (e[3] << 16), e[4] | (e[5] << 16), e[6] | (e[7] << 16));
}

// the candidate vector of golden vector gv whose first element is i0: whole
// blocks of four (one draw each) when i0 is on the block grid, else element
// by element
template <int DT>
__device__ __forceinline__ uint4 inj_vec(const CompareParams& p, const uint4& gv, int64_t i0) {
  constexpr int VEC = 16 / Tr<DT>::BYTES, NB = VEC / 4;
  uint32_t e[VEC];
  unpack_vec<DT>(gv, e);
  if ((i0 & 3) == 0) {
    for (int m = 0; m < p.inj_n; m++) {
      const InjStep st = p.inj[m];
      inj::with_kind(st.kind, [&](auto k) {
        inj::apply_blocks<DT, decltype(k)::value, NB>(e, i0, st.model, st.threshold, st.x, p.inj_k0, p.inj_k1);
      });
    }
  } else {
#pragma unroll
    for (int j = 0; j < VEC; j++) e[j] = inj_chain<DT>(p, e[j], i0 + j);
  }
  return pack_vec<DT>(e);
}

// The candidate chunk of a fused call, ct[v] for golden gt[v], v = lane,
// lane + 32, ... < nvalid, vector v starting at element i0 + v VEC: model by
// model over the chunk (one branch on the kind per model, then code without
// branches), each lane rewriting its own vectors in place.  Out of line,
// called once per chunk.
template <int DT>
__device__ __noinline__ void inj_chunk(const CompareParams& p, const uint4* gt, uint4* ct, int nvalid, int64_t i0) {
  constexpr int VEC = 16 / Tr<DT>::BYTES, NB = VEC / 4;
  const int lane = threadIdx.x & 31;
  if ((i0 & 3) != 0) {  // off the block grid
    for (int v = lane; v < nvalid; v += 32) ct[v] = inj_vec<DT>(p, gt[v], i0 + (int64_t)v * VEC);
    return;
  }
  for (int m = 0; m < p.inj_n; m++) {
    const InjStep st = p.inj[m];
    const uint4* src = m == 0 ? gt : ct;
    inj::with_kind(st.kind, [&](auto k) {
      for (int v = lane; v < nvalid; v += 32) {
        uint32_t e[VEC];
        unpack_vec<DT>(src[v], e);
        inj::apply_blocks<DT, decltype(k)::value, NB>(e, i0 + (int64_t)v * VEC, st.model, st.threshold, st.x,
                                                       p.inj_k0, p.inj_k1);
        ct[v] = pack_vec<DT>(e);
      }
    });
  }
}

// one candidate vector, out of line (the window sample of a piece)
template <int DT>
__device__ __noinline__ uint4 inj_one(const CompareParams& p, uint4 gv, int64_t i0) {
  return inj_vec<DT>(p, gv, i0);
}

__device__ __forceinline__ uint4 load_vec(const void* base, int64_t byte_off) {
  const uint4* p = reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(base) + byte_off);
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// ---- bulk-copy (TMA) staging: mbarrier + cp.async.bulk, waits bounded -----
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
// true in one lane of the (converged) warp
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xFFFFFFFF;\n selp.u32 %0, 1, 0, q;\n}" : "=r"(p));
  return p != 0;
}
// global -> shared bulk copy of `bytes` (16-byte aligned, multiple of 16), completing on bar
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// wait for phase `parity` of bar to complete, giving up after `limit` polls
// (limit 0: give up without polling)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t limit) {
  for (uint32_t it = 0; it < limit; it++)
    if (mbar_test(bar, parity)) return true;
  return false;
}
// order earlier generic-proxy accesses of the stage before the next bulk write into it
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
constexpr uint32_t DRAIN_LIMIT = 1u << 26;  // polls before a drain wait gives up (far beyond any copy)

// ---------------------------------------------------------------------------
// exact integer digits
// ---------------------------------------------------------------------------
// A local exact accumulator: integer digits only (off the hot path).
struct XAcc {
  int64_t d[NLIMB];
  __device__ void zero() {
#pragma unroll
    for (int j = 0; j < NLIMB; j++) d[j] = 0;
  }
  __device__ void add_m(unsigned __int128 m, int e, bool neg) {
    for_digits(m, e, neg, [&](int j, int64_t v) { d[j] += v; });
  }
  // +-x * 2^sc
  __device__ void add_f(float x, bool neg = false, int sc = 0) {
    if (x == 0.0f) return;
    int e;
    uint32_t m = split_float(x, e);
    add_m(m, e + sc, neg ^ (x < 0));
  }
  __device__ void add_prod_f(float x, float y, bool neg = false, int sc = 0) {
    if (x == 0.0f || y == 0.0f) return;
    int ex, ey;
    uint32_t mx = split_float(x, ex), my = split_float(y, ey);
    add_m((unsigned __int128)((uint64_t)mx * my), ex + ey + sc, neg ^ (x < 0) ^ (y < 0));
  }
  __device__ void add_prod(double x, double y, bool neg = false) {
    if (x == 0.0 || y == 0.0) return;
    int ex, ey;
    uint64_t mx = split_double(x, ex), my = split_double(y, ey);
    add_m((unsigned __int128)mx * my, ex + ey, neg ^ (x < 0) ^ (y < 0));
  }
  // carry-propagate: digits 0..NLIMB-2 into [0, 2^32), top digit signed
  __device__ void normalize() {
    int64_t carry = 0;
    for (int j = 0; j < NLIMB - 1; j++) {
      int64_t v = d[j] + carry;
      carry = v >> 32;  // arithmetic shift: floor division
      d[j] = v & 0xFFFFFFFFll;
    }
    d[NLIMB - 1] += carry;
  }
  __device__ int sign() {  // after normalize
    if (d[NLIMB - 1] < 0) return -1;
    for (int j = 0; j < NLIMB; j++)
      if (d[j]) return 1;
    return 0;
  }
  __device__ void negate() {
    for (int j = 0; j < NLIMB; j++) d[j] = -d[j];
    normalize();
  }
};

// ---------------------------------------------------------------------------
// exact magnitudes as float32 pairs
// ---------------------------------------------------------------------------
// |d| is carried as (hi + lo) * 2^sc with hi = RN32(|d| 2^-sc), |lo| <= half a
// step of hi, sc in {0, 1} (sc = 1 only when |d| exceeds the float32 range).

__device__ __forceinline__ void two_sum_f(float x, float y, float& s, float& t) {
  s = __fadd_rn(x, y);
  float yv = __fsub_rn(s, x);
  float xv = __fsub_rn(s, yv);
  t = __fadd_rn(__fsub_rn(x, xv), __fsub_rn(y, yv));
}

// sign(x - y) for two exact pair magnitudes
__device__ __forceinline__ int cmp_mag(float h1, float l1, int s1, float h2, float l2, int s2) {
  if (s1 != s2) return s1 > s2 ? 1 : -1;  // scaled values exceed every unscaled float32
  if (h1 != h2) return h1 > h2 ? 1 : -1;
  return l1 > l2 ? 1 : (l1 < l2 ? -1 : 0);
}

// sign(a1/g1 - a2/g2), a = (hi + lo) 2^sc >= 0, g >= 0; g = 0 < a means +inf
__device__ __noinline__ int cmp_rel_exact(float h1, float l1, int s1, float g1, float h2, float l2, int s2, float g2) {
  int k1 = h1 == 0.0f ? 0 : (g1 == 0.0f ? 2 : 1);
  int k2 = h2 == 0.0f ? 0 : (g2 == 0.0f ? 2 : 1);
  if (k1 != k2) return k1 > k2 ? 1 : -1;
  if (k1 != 1) return 0;
  XAcc x;
  x.zero();
  x.add_prod_f(h1, g2, false, s1);
  x.add_prod_f(l1, g2, false, s1);
  x.add_prod_f(h2, g1, true, s2);
  x.add_prod_f(l2, g1, true, s2);
  x.normalize();
  return x.sign();
}

// sign(a1/g1 - a2/g2) for positive normal float32 values (a2 may be 0):
// compares the 48-bit products of the significands.
__device__ __forceinline__ int cmp_ratio_f(float a1, float g1, float a2, float g2) {
  if (a2 == 0.0f) return 1;
  uint32_t b1 = __float_as_uint(a1), c1 = __float_as_uint(g1), b2 = __float_as_uint(a2), c2 = __float_as_uint(g2);
  uint64_t P1 = (uint64_t)((b1 & 0x7FFFFFu) | 0x800000u) * ((c2 & 0x7FFFFFu) | 0x800000u);
  uint64_t P2 = (uint64_t)((b2 & 0x7FFFFFu) | 0x800000u) * ((c1 & 0x7FFFFFu) | 0x800000u);
  int x1 = (int)(b1 >> 23) + (int)(c2 >> 23), x2 = (int)(b2 >> 23) + (int)(c1 >> 23);
  if (x1 > x2 + 1) return 1;
  if (x2 > x1 + 1) return -1;
  if (x1 > x2) P1 <<= 1;
  else if (x2 > x1) P2 <<= 1;
  return P1 > P2 ? 1 : (P1 < P2 ? -1 : 0);
}

// log2-like key of the ratio (hi + lo) 2^sc / g, within 8 of an increasing
// function of its exact value (2^22 units per binade): the quotient of the
// significands, rounded, under the difference of the exponents.
__device__ __forceinline__ int ratio_key(float h, int sc, float g) {
  if (h == 0.0f) return -0x7FFFFFFF;
  if (g == 0.0f) return 0x7FFFFFFF;
  int e = sc;
  if (h < 1.17549435e-38f) h = __fmul_rn(h, 1.8446744e19f), e -= 64;  // subnormals scaled by 2^64
  if (g < 1.17549435e-38f) g = __fmul_rn(g, 1.8446744e19f), e += 64;
  const uint32_t bh = __float_as_uint(h), bg = __float_as_uint(g);
  e += (int)(bh >> 23) - (int)(bg >> 23);
  const float q = __fdividef(__uint_as_float((bh & 0x7FFFFFu) | 0x3F800000u), __uint_as_float((bg & 0x7FFFFFu) | 0x3F800000u));
  return ((int)(__float_as_uint(q) - 0x3F800000u) >> 1) + e * (1 << 22);
}
constexpr int RATIO_MARGIN = 32;  // keys further apart decide (the key's error, and lo against hi, below 8 each)

// sign((h1 + l1) 2^s1 / g1 - (h2 + l2) 2^s2 / g2): by the keys when they
// differ clearly, by the exact products otherwise
__device__ __forceinline__ int cmp_rel_close(float h1, float l1, int s1, float g1, float h2, float l2, int s2, float g2) {
  const float tiny = 1.17549435e-38f;
  if (h1 == h2 && l1 == l2 && s1 == s2 && g1 == g2) return 0;
  if (l1 == 0.0f && l2 == 0.0f && s1 == 0 && s2 == 0 && h1 >= tiny && h2 >= tiny && g1 >= tiny && g2 >= tiny)
    return cmp_ratio_f(h1, g1, h2, g2);
  return cmp_rel_exact(h1, l1, s1, g1, h2, l2, s2, g2);
}
__device__ __forceinline__ int cmp_rel_rec(float h1, float l1, int s1, float g1, float h2, float l2, int s2, float g2) {
  const int k1 = ratio_key(h1, s1, g1), k2 = ratio_key(h2, s2, g2);
  const long long d = (long long)k1 - k2;
  if (d > RATIO_MARGIN) return 1;
  if (d < -RATIO_MARGIN) return -1;
  return cmp_rel_close(h1, l1, s1, g1, h2, l2, s2, g2);
}

// float32 filter for a rel best: a value <= rel with a margin for the
// approximate per-lane ratio a * rcp(|g|)
__device__ __forceinline__ float rel_filter(float hi, int sc, float g) {
  if (g == 0.0f) return __int_as_float(0x7F800000);
  float q = __fdiv_rd(hi, g);
  if (sc) q = __fmul_rd(q, 2.0f);
  return __fmul_rd(q, 0.99999809265136719f);  // 1 - 2^-19
}

// ---------------------------------------------------------------------------
// shared memory
// ---------------------------------------------------------------------------
// Exact maxima records and class counters of the general path (|d| as
// (hi + lo) 2^sc, see Partial); registers of run_general.
struct GenRec {
  float abs_hi, abs_lo;
  float rel_hi, rel_lo, rel_g;
  float rel_f;  // filter of the rel best
  uint32_t ulp;
  uint32_t n_gw, n_gm, n_ga, n_gf, n_nf, n_geq;
  int abs_sc, rel_sc;
  long long abs_idx, rel_idx, ulp_idx;
};

// The exact relative-error record of one warp's window pairs: |d| = a and |g|
// of the best ratio so far (a = 0: none) at offset li from the CTA's first
// element.  q: the ratio rounded to float32 (16-bit types: distinct ratios
// round apart, see rel_key).
struct RelRec {
  float a, g, q;
  uint32_t li;
};

// Per-warp staging ring for the bulk copies: NSTAGE stages, each one warp
// tile of CHV 16-byte vectors of each tensor (two vectors per lane).

// scratch of the mean and variance of |d|: S1 = sum |d| and S2 = sum d^2,
// both NLIMB digits weighing 2^(32 j + LIMB_LSB) (two more after carrying)
using MV = MeanVarScratch<NLIMB + 2, NLIMB + 2, -LIMB_LSB / 32>;
static_assert(LIMB_LSB % 32 == 0, "the S2 shift is a whole number of digits");

// scratch of a segment's finalization
struct FinScratch {
  unsigned long long cnt[8];
  long long limbs[NSUM * NLIMB];
  Partial wbest[16], best;
  double sums[NSUM], max_abs, max_rel;
};
constexpr int NSTAGE = 2;  // a power of two: stage and phase are bit fields of the use count
constexpr int RWMAX = 6;   // window moves per warp and piece (float32)
constexpr int CHV = 64;

// The window tables: shared counters that every window pair increments by
// one.  An increment by the constant one costs a cycle per distinct address
// of a bank (lanes with the same address are merged; measured: 32 lanes on
// one address 1.2 cycles, on random addresses 2.6, while adding a variable
// serialises equal addresses), so the counters need no private copies.
//
// Every pair of a vector increments them, equal ones too (a predicated
// increment compiles to a branch, five instructions): equal pairs (d = 0) land
// in cells of their own that are left out.
//
// T1 (16-bit types) counts pairs by the value of d.  |d| has at most 8
// significant bits, so 1 + 6 + 7 bits (bfloat16: the sign, the exponent modulo
// 64, the significand field; the window holds 64 exponents) or 1 + 5 + 7
// (binary16 scaled by 2^s, see Win) name it.  The low five bits of the index
// are exclusive-ored with those of the exponent, or powers of two would share
// a bank.  The three exact sums are formed from the counters at the end of a
// piece.  d = 0 shares bfloat16's cell of exponent 0 mod 64, significand 0;
// its number is known from T2 and taken off.
//
// T2 gives the bins.  bfloat16: by (ULP steps + 64, the golden's significand
// field), which fixes the ratio |d| / |g| and so the log2-relative bin, and
// (with atol = 0) the class.  binary16 and float32: by (floor(log2(|d| / |g|))
// modulo 32, ULP steps + 128 or min(ULP steps, 63)), the two bins themselves.
template <int DT>
struct Tab;
template <>
struct Tab<PEAT_F32> {
  static constexpr int N1 = 0, N2 = 32 * 64, UMAX = (1 << 23) - 1;
};
template <>
struct Tab<PEAT_F16> {
  static constexpr int N1 = 2 * 32 * 128, N2 = 32 * 256, ROWS = 32, UMAX = 127;
};
template <>
struct Tab<PEAT_BF16> {
  static constexpr int N1 = 2 * 64 * 128, N2 = 128 * 128, ROWS = 64, UMAX = 63;
};

template <int NW>
struct Ring {
  uint4 g[NW][NSTAGE][CHV];
  uint4 c[NW][NSTAGE][CHV];
};

// totals and scratch, the same for both geometries
template <int NW>
struct Common {
  unsigned long long bar[NW][NSTAGE];
  unsigned long long hist[HBINS];
  unsigned long long sacc[NSUM][NLIMB];
  unsigned long long cnt[8];
  Partial wbest[NW];
  long long lo;                    // the CTA's first element
  long long ff, fu;                // first finite pair, first pair without NaN (search result)
  uint32_t* glist;                 // this CTA's list of general pairs, gcap entries
  uint32_t gcap;
  uint32_t gn;                     // entries appended in this piece (may exceed gcap)
  uint32_t nfe;                    // bitwise-equal pairs holding NaN or Inf
  int last;                        // this CTA finished the last piece of a one-segment call
  int first, final;                // a one-segment call's pieces: the CTAs first .. final
  int lb, ub;
  // the CTA's window maxima of the piece: value in the high word, the
  // complement of the pair's offset in the low one (the larger key is the
  // larger value, then the lower index; low word 0: a starting bound taken
  // from the window sample, no pair yet).  kabs: float32 bits of |d|; kulp:
  // the ULP distance; krel: float32 bits of the ratio (float32 operands: a
  // lower bound of it, the pairs are in wrel).
  unsigned long long kabs, kulp, krel;
  RelRec wrel[NW];
  uint4 edge_g[CHV], edge_c[CHV];  // the staged head or tail of a piece
  uint32_t wem[NW], wum[NW];       // float32: largest golden exponent and ULP distance of the vectors slow_vec saw in a tile
  // float32: each warp's windows in the current piece: window r applies from
  // the warp's chunk wstart[w][r] on (r = 0: the piece's initial window)
  uint32_t nwin[NW];
  uint32_t wstart[NW][RWMAX + 1];
  int wlb[NW][RWMAX + 1];
  FinScratch fin;
  // the general path's totals, one copy per warp (fewer threads contend for an
  // address), folded into hist and sacc at the end of a piece that used them
  uint32_t ghist[NW][HBINS];  // (a piece has below 2^31 pairs)
  int gsacc[NW][NSUM * NLIMB][2];  // sums of the low and the high 16 bits of each digit (gen_flush)
};

template <int DT>
struct __align__(128) Smem {
  static constexpr int NW = Geo<DT>::NW;
  uint32_t t1[Tab<DT>::N1 ? Tab<DT>::N1 : 32];
  uint32_t t2[Tab<DT>::N2];
  union {  // the mean/variance scratch of a finalizing CTA reuses the (by then idle) staging ring
    Ring<NW> ring;
    MV mv;
  };
  Common<NW> k;
};
static_assert(sizeof(Smem<PEAT_F32>) <= 113 * 1024, "two float32 CTAs per SM");
static_assert(sizeof(Smem<PEAT_BF16>) <= 227 * 1024 && sizeof(Smem<PEAT_F16>) <= 227 * 1024, "one 16-bit CTA per SM");
static_assert(sizeof(MV) <= sizeof(Ring<8>), "the scratch fits the ring");
static_assert(offsetof(Smem<PEAT_BF16>, ring) % 128 == 0 && offsetof(Smem<PEAT_F16>, ring) % 128 == 0 &&
                  offsetof(Smem<PEAT_F32>, ring) % 128 == 0,
              "bulk copies into the ring");


template <int DT>
__device__ __forceinline__ void sacc_add(Smem<DT>& sm, int which, unsigned __int128 m, int e, bool neg) {
  for_digits(m, e, neg, [&](int j, int64_t v) { atomicAdd(&sm.k.sacc[which][j], (unsigned long long)v); });
}
// A general-path term +-m 2^e into the warp's copy of a sum's digits.  A copy
// holds each digit's 32-bit contributions as two sums of 16-bit halves in
// signed 32-bit words, which shared memory adds natively (64-bit adds there
// are compare-and-swap loops, and grouping the lanes by digit first, match
// and reductions, took 6 us for the terms of one round; this takes 1.3).
// gen_flush empties the words before they can overflow.
__device__ __forceinline__ void wsacc_add(int* d, uint64_t m, int e, bool neg) {
  const int p = e - LIMB_LSB, j = p >> 5, r = p & 31;
  const uint32_t m0 = (uint32_t)m, m1 = (uint32_t)(m >> 32);
  const uint32_t out[3] = {m0 << r, (m1 << r) | (r ? m0 >> (32 - r) : 0u), r ? m1 >> (32 - r) : 0u};
#pragma unroll
  for (int k = 0; k < 3; k++) {
    if (out[k] == 0u) continue;
    if ((unsigned)(j + k) >= (unsigned)NLIMB) {  // (excluded by the bounds on the terms, see for_digits)
      digit_dropped();
      continue;
    }
    const int lo = (int)(out[k] & 0xFFFFu), hi = (int)(out[k] >> 16);
    atomicAdd(d + 2 * (j + k), neg ? -lo : lo);
    atomicAdd(d + 2 * (j + k) + 1, neg ? -hi : hi);
  }
}
// Three terms of a round go to one sum: 256 rounds of 32 lanes stay below 2^31.
constexpr int GEN_FLUSH = 256;
template <int DT>
__device__ __noinline__ void gen_flush(Smem<DT>& sm) {
  __syncwarp();
  int(*d)[2] = sm.k.gsacc[threadIdx.x >> 5];
  for (int j = threadIdx.x & 31; j < NSUM * NLIMB; j += 32) {
    const int64_t v = (int64_t)d[j][1] * 65536 + d[j][0];
    d[j][0] = d[j][1] = 0;
    if (v) atomicAdd(&sm.k.sacc[0][0] + j, (unsigned long long)v);
  }
  __syncwarp();
}
// one histogram bin per lane (bin < 0: none), an increment by the constant one
// (see the tables)
template <int DT>
__device__ __forceinline__ void whist_add(Smem<DT>& sm, int bin) {
  if (bin >= 0 && PEAT_CHECK(bin < HBINS))
    asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(smem_addr(&sm.k.ghist[threadIdx.x >> 5][bin])) : "memory");
}

// floor(log2(a / g)) for a = (hi + lo) 2^sc > 0 and g > 0 (float32 pair, any range)
__device__ int log2_ratio(float hi, float lo, int sc, float g) {
  float hs = hi, gs = g;
  if (hs < 1.17549435e-38f || gs < 1.17549435e-38f) {  // scale subnormals by 2^64
    if (hs >= 1.8446744e19f) return 200;              // ratio far above the clamp
    if (gs >= 1.8446744e19f) return -200;
    hs = __fmul_rn(hs, 1.8446744e19f);
    gs = __fmul_rn(gs, 1.8446744e19f);
  }
  uint32_t bh = __float_as_uint(hs), bg = __float_as_uint(gs);
  int k = ((int)(bh - bg)) >> 23;
  if (lo < 0.0f && (bh & 0x7FFFFFu) == (bg & 0x7FFFFFu)) k--;  // a just below 2^k g
  return k + sc;
}

// The general path: the definitions evaluated exactly, for any pair.  The
// per-lane part: class counters and maxima into cd; the histogram bins and
// the sum terms it returns are added by the whole warp (general_lane).
struct GenOut {
  int hb0, hb1;      // log2-relative bin and 64 + ULP bin, or -1
  float s, t;        // d = (s + t) 2^sc, both zero when the pair adds no terms
  int sc;
};
template <int DT>
__device__ __forceinline__ void general_pair(GenRec& cd, GenOut& o, uint32_t G, uint32_t C, int64_t idx, float rtol,
                                             float atol) {
  using T = Tr<DT>;
  uint32_t ag_m = G & T::MAG, ac_m = C & T::MAG;
  bool gnan = ag_m > T::INF, cnan = ac_m > T::INF, ginf = ag_m == T::INF, cinf = ac_m == T::INF;
  bool gs = (G & T::SIGN) != 0, cs = (C & T::SIGN) != 0;
  int64_t kg = gs ? -(int64_t)ag_m : (int64_t)ag_m, kc = cs ? -(int64_t)ac_m : (int64_t)ac_m;
  uint64_t u = (uint64_t)(kc > kg ? kc - kg : kg - kc);
  bool ulpdef = !gnan && !cnan;
  if (ulpdef && u > 0 && (u > cd.ulp || (u == cd.ulp && idx < cd.ulp_idx))) {
    cd.ulp = (uint32_t)u;
    cd.ulp_idx = idx;
  }
  if (gnan || cnan || ginf || cinf) {
    cd.n_nf++;
    bool equal = (gnan && cnan) || (ginf && cinf && gs == cs);
    if (equal) {
      cd.n_geq++;
      return;
    }
    cd.n_ga++;
    o.hb0 = 63;
    o.hb1 = 64 + (ulpdef ? (u < 63 ? (int)u : 63) : 63);
    return;
  }
  float gf = to_f32<DT>(G), cf = to_f32<DT>(C);
  if (gf == cf) {  // +0 and -0
    cd.n_geq++;
    return;
  }
  float s, t;
  int sc = 0;
  two_sum_f(cf, -gf, s, t);
  if (!(fabsf(s) < __int_as_float(0x7F800000))) {  // |d| above the float32 range: halve exactly
    two_sum_f(__fmul_rn(cf, 0.5f), __fmul_rn(-gf, 0.5f), s, t);
    sc = 1;
  }
  float hi = fabsf(s), lo = s < 0.0f ? -t : t;
  float ag = fabsf(gf);
  // WITHIN_TOL: a <= atol + rtol |g|, decided in float32 when clear, exactly otherwise
  bool within;
  float thr = __fmaf_rn(rtol, ag, atol);
  if (sc == 0 && hi >= 1e-30f && thr >= 1e-30f && __fmul_rn(hi, 1.0000005f) < __fmul_rn(thr, 0.9999995f)) {
    within = true;
  } else if (sc == 0 && hi >= 1e-30f && __fmul_rn(hi, 0.9999995f) > __fmul_rn(thr, 1.0000005f)) {
    within = false;
  } else {
    XAcc x;
    x.zero();
    x.add_f(hi, false, sc);
    x.add_f(lo, false, sc);
    x.add_f(atol, true);
    x.add_prod_f(rtol, ag, true);
    x.normalize();
    within = x.sign() <= 0;
  }
  if (within) cd.n_gw++;
  else if (gf != 0.0f && cf != 0.0f && gs != cs) cd.n_gf++;
  else cd.n_gm++;
  // log2-relative bin and ULP bin
  int rb;
  if (ag == 0.0f) {
    rb = 63;
  } else {
    int k = log2_ratio(hi, lo, sc, ag) + 48;
    rb = k < 1 ? 1 : (k > 62 ? 62 : k);
  }
  o.hb0 = rb;
  o.hb1 = 64 + (u < 63 ? (int)u : 63);
  // maxima, full (value, index) order
  {
    int c = cd.abs_idx < 0 ? 1 : cmp_mag(hi, lo, sc, cd.abs_hi, cd.abs_lo, cd.abs_sc);
    if (c > 0 || (c == 0 && idx < cd.abs_idx)) {
      cd.abs_hi = hi;
      cd.abs_lo = lo;
      cd.abs_sc = sc;
      cd.abs_idx = idx;
    }
  }
  {
    bool maybe = cd.rel_idx < 0 || ag == 0.0f || sc ||
                 __fmul_rn(__fmul_rn(hi, rcp_approx(ag)), 1.00001f) >= cd.rel_f;
    if (maybe) {
      int c = cd.rel_idx < 0 ? 1 : cmp_rel_rec(hi, lo, sc, ag, cd.rel_hi, cd.rel_lo, cd.rel_sc, cd.rel_g);
      if (c > 0 || (c == 0 && idx < cd.rel_idx)) {
        cd.rel_hi = hi;
        cd.rel_lo = lo;
        cd.rel_sc = sc;
        cd.rel_g = ag;
        cd.rel_idx = idx;
        cd.rel_f = rel_filter(hi, sc, ag);
      }
    }
  }
  o.s = s;
  o.t = t;
  o.sc = sc;
}
// binary16: every finite difference is D 2^-24 for an integer D below 2^41 in
// size, so where a piece has many general pairs their sums are integers in
// registers: of |D|, of |D| over the negative ones, and of D^2 (at most 2^22
// pairs per thread and piece).  Through the digits in shared memory a round of
// 32 pairs took 1700 instructions, 14 of them conflicting increments, now 600;
// but the integers' own reduction at the end takes 2 to 3 us, hence GEN_MANY.
struct GenSum {
  uint64_t a = 0, n = 0;
  unsigned __int128 q = 0;
};
constexpr uint32_t GEN_MANY = 4096;
__device__ __forceinline__ int64_t f16_units(uint32_t b) {
  const uint32_t e = (b >> 10) & 31u, m = b & 0x3FFu;
  const int64_t k = e ? (int64_t)(m | 0x400u) << (e - 1) : (int64_t)m;
  return (b & 0x8000u) ? -k : k;
}
// One general pair per lane of a converged warp (valid: the lane has one):
// the per-lane part, then the histogram bins and the exact sums, d = (s + t)
// 2^sc, |d| = (hi + lo) 2^sc with (hi, lo) = +-(s, t), d^2 = (s^2 + 2st +
// t^2) 4^sc, added by the whole warp.
template <int DT>
__device__ __forceinline__ void general_lane(Smem<DT>& sm, GenRec& cd, GenSum& gs, bool many, uint32_t G, uint32_t C,
                                             int64_t idx, float rtol, float atol, bool valid) {
  GenOut o{-1, -1, 0.0f, 0.0f, 0};
  if (valid) general_pair<DT>(cd, o, G, C, idx, rtol, atol);
  whist_add(sm, o.hb0);
  whist_add(sm, o.hb1);
  const bool on = o.s != 0.0f;
  if (DT == PEAT_F16 && many) {
    if (on) {
      const int64_t d = f16_units(C) - f16_units(G);
      const uint64_t a = (uint64_t)(d < 0 ? -d : d);
      gs.a += a;
      gs.n += d < 0 ? a : 0ull;
      gs.q += (unsigned __int128)a * a;
    }
    return;
  }
  // the seven terms through one copy of the code: a piece with few general
  // pairs spends most of this path's time on fetching it
  int* d = &sm.k.gsacc[threadIdx.x >> 5][0][0];
#pragma unroll 1
  for (int k = 0; k < 7; k++) {
    // s, t | |d|'s parts, s and t with the sign of s | s^2, 2 s t, t^2
    float x = k == 1 || k == 3 || k == 6 ? o.t : o.s;
    const float y = k < 4 ? 1.0f : (k == 4 ? o.s : o.t);
    if ((k == 2 || k == 3) && o.s < 0.0f) x = -x;
    const bool use = on && x != 0.0f && y != 0.0f;
    if (many && !__any_sync(0xFFFFFFFFu, use)) continue;  // (t is zero where c - g is a float32 value, most often)
    if (use) {
      int ex = 0, ey = 0;
      const uint32_t mx = split_float(x, ex), my = split_float(y, ey);
      wsacc_add(d + min(k >> 1, 2) * (2 * NLIMB), (uint64_t)mx * my, ex + ey + (k < 4 ? o.sc : 2 * o.sc + (k == 5)),
                (x < 0.0f) != (y < 0.0f));
    }
  }
}

// ---------------------------------------------------------------------------
// per-thread window state and per-piece window constants (registers)
// ---------------------------------------------------------------------------
// mism: window pairs above the tolerance (a float32 count, exact below 2^24).
// float32 only, since the last flush, with |d| = (V1 2^21 + V2) 2^Lexp: A the
// sum of |d| and S of d in units of 2^Lexp, Q11, Q12, Q22 the sums of V1 V1,
// V1 V2, V2 V2.
struct Lane {
  float mism;
  int64_t A, S, Q12;
  uint64_t Q11, Q22;
};

// float32: the window (warp-uniform; a warp moves it when too many of a
// tile's pairs fall outside): Lb is the floor binade, Lexp = Lb - BIAS - MB,
// |d| a multiple of 2^Lexp below 2^(Lexp + 42).  bfloat16: fe, the float32 exponent field of the
// smallest |d|; T1 holds 64 exponents from there.  binary16: fe = s, the
// values are scaled by 2^s (exactly), so that their differences are normal.
struct Win {
  float rtol, atol;  // binary16: atol scaled by 2^s
  float lim;         // 2^(Lexp + 42)
  // 1.5 * 2^(23 + e): bits(x + M) - bits(M) is x / 2^e rounded to an integer,
  // for |x| < 2^(e + 22); e = Lexp + 21 for M1, Lexp for M2
  float M1, M2;
  int lb;            // Lb
  int fe;
};

// the window with floor binade lb
template <int DT>
__device__ __forceinline__ void set_window_lb(Win& W, int lb) {
  using Ty = Tr<DT>;
  const int lexp = lb - Ty::BIAS - Ty::MB;
  W.lb = lb;
  W.lim = __uint_as_float((uint32_t)(lexp + 42 + 127) << 23);
  W.M1 = __uint_as_float(((uint32_t)(lexp + 44 + 127) << 23) | 0x400000u);
  W.M2 = __uint_as_float(((uint32_t)(lexp + 23 + 127) << 23) | 0x400000u);
}
// The window placed for data whose largest finite golden exponent is emax and
// whose ULP distances have ubits bits: |d| < 2^(Lexp + 42) for such pairs with
// goldens up to 2 binades above emax (one bit to spare on u).
template <int DT>
__device__ __forceinline__ int window_floor(int emax, int ubits) {
  using Ty = Tr<DT>;
  const int UB = min(ubits + 1, Ty::UBMAX);
  const int lb = emax + UB - 40;
  return lb < Ty::LBMIN ? Ty::LBMIN : (lb > Ty::LBMAX ? Ty::LBMAX : lb);
}
template <int DT>
__device__ __forceinline__ int win_lexp(const Win& W) {
  return W.lb - Tr<DT>::BIAS - Tr<DT>::MB;
}
// The window of 16-bit data whose largest finite golden exponent field is
// emax.  bfloat16: a difference of at most 63 steps lies below 2^1 times the
// golden's binade, so T1 ends 4 binades above the largest golden seen and
// covers 59 below it; |d| stays at or above 2^-100 (tolerance differences
// are then normal numbers, see count_mismatch).  binary16: the scale takes
// the largest golden seen to 2^13, two binades below overflow; s >= 0 loses no
// bits, and from s = 10 on even the smallest subnormal becomes normal.
template <int DT>
__device__ __forceinline__ int window16(int emax) {
  if constexpr (DT == PEAT_F16) return min(max(28 - emax, 0), 15);
  else return min(max(emax + 4 - 63, 27), 254 - 63);
}

__device__ __forceinline__ void lane_init(Lane& L) {
  L.mism = 0.0f;
  L.A = L.S = L.Q12 = 0;
  L.Q11 = L.Q22 = 0;
}
__device__ __forceinline__ void gen_init(GenRec& c) {
  c.abs_hi = c.abs_lo = 0.0f;
  c.rel_hi = c.rel_lo = 0.0f;
  c.rel_g = 1.0f;
  c.rel_f = 0.0f;
  c.ulp = 0;
  c.n_gw = c.n_gm = c.n_ga = c.n_gf = c.n_nf = c.n_geq = 0;
  c.abs_sc = c.rel_sc = 0;
  c.abs_idx = c.rel_idx = c.ulp_idx = -1;
}

// a1 / g1 > a2 / g2 for window pairs (positive normal a, g): the ratios
// normalised to g in [1, 2), then exact products
__device__ __forceinline__ void norm_ratio(float a, float g, float& an, float& mg) {
  const uint32_t gb = __float_as_uint(g);
  an = __uint_as_float(__float_as_uint(a) - (gb & 0x7F800000u) + 0x3F800000u);
  mg = __uint_as_float((gb & 0x007FFFFFu) | 0x3F800000u);
}
__device__ __forceinline__ bool rel_greater(float a1, float g1, float a2, float g2) {
  if (a2 == 0.0f) return a1 > 0.0f;
  if (a1 == 0.0f) return false;
  float an1, m1, an2, m2;
  norm_ratio(a1, g1, an1, m1);
  norm_ratio(a2, g2, an2, m2);
  const float p = __fmul_rn(an1, m2), q = __fmul_rn(an2, m1);
  // error terms of the products, exact (no underflow: both products exceed 2^-26)
  const float ep = __fmaf_rn(an1, m2, -p), eq = __fmaf_rn(an2, m1, -q);
  return p > q || (p == q && ep > eq);
}

// ---------------------------------------------------------------------------
// window pairs
// ---------------------------------------------------------------------------
// Whether a pair of unequal patterns is a window pair: a pure function of the
// bits and the window, so that a rescan of the piece decides as the tiles did.
// G, C: raw bits.
//
// 16-bit types: both finite, C - G at most UMAX steps of the pattern either way
// (the signs then agree), the golden not zero.  c - g is then exact in the type
// itself (Sterbenz; a subnormal pair's difference is a multiple of the
// smallest step) with at most 8 significant bits.  bfloat16: |d| also inside
// T1 (so that both operands are normal).  binary16: the golden scaled by 2^fe
// finite, and the scaled golden and difference normal.
//
// float32: ULP distance below 2^23 (so the signs agree and c is within a
// factor 2 of g: c - g is exact, Sterbenz), |d| < lim and |d| a multiple of
// 2^Lexp: |d| rounded to a multiple of 2^(Lexp + 21) and the (exact) remainder
// are then read as integers V1, V2 from the bits of sums with M1 and M2; with
// the remainder of the first, 42 bits hold the distances of goldens 20 binades
// apart and more, so few pairs are left out.  2^Lexp is a normal number, so a golden that is zero or
// subnormal never passes (its |d| is below 2^23 2^-149).
template <int DT>
__device__ __forceinline__ bool pair_window(uint32_t G, uint32_t C, const Win& W, uint32_t& u, float& gf, float& a) {
  using Ty = Tr<DT>;
  gf = to_f32<DT>(G);
  const float cf = to_f32<DT>(C);
  const float d = __fsub_rn(cf, gf);
  a = fabsf(d);
  u = C > G ? C - G : G - C;
  if constexpr (DT == PEAT_F32) {
    const float l = __fsub_rn(a, __fsub_rn(__fadd_rn(a, W.M1), W.M1));
    return u < (1u << 23) && a < W.lim && __fsub_rn(__fadd_rn(l, W.M2), W.M2) == l;
  } else {
    const uint32_t mg = G & Ty::MAG, mc = C & Ty::MAG;
    const bool ok = mg < Ty::INF && mc < Ty::INF && mg != 0u && u <= (uint32_t)Tab<DT>::UMAX && ((G ^ C) & Ty::SIGN) == 0u;
    if constexpr (DT == PEAT_BF16) {
      return ok && ((__float_as_uint(a) >> 23) - (uint32_t)W.fe) < 64u;
    } else {
      const float lo = __uint_as_float((uint32_t)(127 - 14 - W.fe) << 23);  // 2^-14 before scaling
      return ok && (int)(mg >> 10) + W.fe <= 30 && a >= lo && fabsf(gf) >= lo;
    }
  }
}

// a pair outside the window: append it to the CTA's general list (evaluated
// at the end of the piece; past gcap entries the piece is rescanned)
template <int DT>
__device__ __forceinline__ void defer_pair(uint32_t li, Smem<DT>& sm) {
  const uint32_t slot = atomicAdd(&sm.k.gn, 1u);
  if (slot < sm.k.gcap) sm.k.glist[slot] = li;
}

// lanes of one vector whose golden value is NaN or Inf, as a bitmask
template <int DT>
__device__ __forceinline__ uint32_t nonfinite_lanes(const uint4& v) {
  using T = Tr<DT>;
  uint32_t m = 0;
#pragma unroll
  for (int j = 0; j < T::VEC; j++) m |= ((lane_bits<DT>(v, j) & T::MAG) >= T::INF ? 1u : 0u) << j;
  return m;
}
// any NaN/Inf among the lanes of one vector (cheap test)
template <int DT>
__device__ __forceinline__ bool any_nonfinite(const uint4& v) {
  using T = Tr<DT>;
  if constexpr (T::BYTES == 2) {  // x * 0 is NaN for NaN and infinity, else a zero
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t z = 0;
#pragma unroll
    for (int i = 0; i < 4; i++) {
      if constexpr (DT == PEAT_BF16) {
        const __nv_bfloat162 r = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&w[i]), __floats2bfloat162_rn(0.0f, 0.0f),
                                         *reinterpret_cast<const __nv_bfloat162*>(&z));
        z = *reinterpret_cast<const uint32_t*>(&r);
      } else {
        const __half2 r = __hfma2(*reinterpret_cast<const __half2*>(&w[i]), __floats2half2_rn(0.0f, 0.0f),
                                  *reinterpret_cast<const __half2*>(&z));
        z = *reinterpret_cast<const uint32_t*>(&r);
      }
    }
    return (z & 0x7FFF7FFFu) != 0u;
  } else {
    uint32_t m = max(max(v.x & T::MAG, v.y & T::MAG), max(v.z & T::MAG, v.w & T::MAG));
    return m >= T::INF;
  }
}

// A vector of equal pairs: every one is EXACT; the ones holding NaN/Inf also
// count as non-finite pairs.
template <int DT>
__device__ __forceinline__ void count_equal(const uint4& g, Smem<DT>& sm) {
  if (any_nonfinite<DT>(g)) atomicAdd(&sm.k.nfe, (uint32_t)__popc(nonfinite_lanes<DT>(g)));
}

__device__ __forceinline__ uint64_t wsum64(uint64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// float32: this warp's window sums (in units of 2^lexp) into the CTA's exact
// accumulator: |A|, |S| < 2^59, Q11, Q22 and |Q12| < 2^58 per thread between
// flushes; combined in 128 bits.
__device__ __forceinline__ void flush_sums(Lane& L, Smem<PEAT_F32>& sm, int lexp) {
  const uint64_t A = wsum64((uint64_t)L.A), S = wsum64((uint64_t)L.S);
  const uint64_t q11 = wsum64(L.Q11), q12 = wsum64((uint64_t)L.Q12), q22 = wsum64(L.Q22);
  const int lane = threadIdx.x & 31;
  if (lane < NSUM) {  // a lane per sum
    const bool neg = lane == 0 && (int64_t)S < 0;
    const unsigned __int128 q = ((unsigned __int128)q11 << 42) + (unsigned __int128)((__int128)(int64_t)q12 << 22) + q22;
    const unsigned __int128 m = lane == 0 ? (unsigned __int128)(neg ? 0ull - S : S) : (lane == 1 ? (unsigned __int128)A : q);
    sacc_add<PEAT_F32>(sm, lane, m, lane == 2 ? 2 * lexp : lexp, neg);
  }
  L.A = L.S = L.Q12 = 0;
  L.Q11 = L.Q22 = 0;
}

// binary16: the warp's general sums into the CTA's digits, word by word
__device__ __forceinline__ void gen_sums(const GenSum& gs, Smem<PEAT_F16>& sm) {
#pragma unroll 1
  for (int w = 0; w < 4; w++) {
    const uint64_t a = w < 2 ? wsum64((uint32_t)(gs.a >> (32 * w))) : 0;
    const uint64_t n = w < 2 ? wsum64((uint32_t)(gs.n >> (32 * w))) : 0;
    const uint64_t q = wsum64((uint32_t)(gs.q >> (32 * w)));
    if ((threadIdx.x & 31) == 0) {
      if (a) sacc_add<PEAT_F16>(sm, 1, a, 32 * w - 24, false), sacc_add<PEAT_F16>(sm, 0, a, 32 * w - 24, false);
      if (n) sacc_add<PEAT_F16>(sm, 0, n, 32 * w - 23, true);  // sum d = sum |d| - 2 sum of the negative ones
      if (q) sacc_add<PEAT_F16>(sm, 2, q, 32 * w - 48, false);
    }
  }
}

// float32: when the slow path sent many pairs of a tile (at least 32, and a
// quarter of the unequal ones it saw) to the general path, the warp moves its
// window to the data it saw there -- largest finite golden exponent, largest
// same-sign ULP distance (wem, wum) -- after flushing the sums kept in the old window's
// units, and logs the move so that a rescan of the piece applies to every pair
// the window it saw.  At most RWMAX moves per warp and piece.
// (This part: the new floor binade, logged; -1: the window stays.)
__device__ __noinline__ int next_window(int lb0, uint32_t ichunk, Smem<PEAT_F32>& sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t r = sm.k.nwin[warp];
  const int lb = window_floor<PEAT_F32>((int)sm.k.wem[warp], 32 - __clz(sm.k.wum[warp]));
  if (r >= (uint32_t)RWMAX || lb == lb0) return -1;
  __syncwarp();
  if (lane == 0) {
    sm.k.wstart[warp][r + 1] = ichunk + 1;
    sm.k.wlb[warp][r + 1] = lb;
    sm.k.nwin[warp] = r + 1;
  }
  __syncwarp();
  return lb;
}

// The bounds a tile's pairs are tested against, from the CTA's records.  A
// pair above one of them takes the slow path; pairs at or below all of them
// cannot be a maximum of the piece.  A record at or after the tile's first
// element (another warp is ahead, or a starting bound) is lowered one step,
// so that an equal value at a lower index is seen.  A starting bound may come
// from a pair outside the window, so each is capped at the window's own.
struct Bounds {
  uint32_t ab;  // |d|: float32 bits, or the (scaled) 16-bit pattern in both halves
  uint32_t ub;  // ULP distance
  float r;      // ratio: a pair is above when |d| - |g| r > 0
  bool low;     // one of them was lowered: read again before the next tile
};
template <int DT>
__device__ __forceinline__ Bounds read_bounds(const Smem<DT>& sm, uint32_t tli, const Win& W) {
  const unsigned long long ka = *(volatile const unsigned long long*)&sm.k.kabs;
  const unsigned long long ku = *(volatile const unsigned long long*)&sm.k.kulp;
  const unsigned long long kr = *(volatile const unsigned long long*)&sm.k.krel;
  Bounds b;
  // (a record above what the window can hold, a general pair's in the sample,
  // bounds every window pair as it is; the general path has that pair)
  const uint32_t av = (uint32_t)(ka >> 32), uv = (uint32_t)(ku >> 32);
  uint32_t cap;
  if constexpr (DT == PEAT_BF16) {
    cap = (((uint32_t)(W.fe + 64) << 23) - 0x10000u) >> 16;
    b.ab = av >> 16;
  } else if constexpr (DT == PEAT_F16) {
    cap = 0x7BFFu;
    const float sc = __fmul_rn(__uint_as_float(av), __uint_as_float((uint32_t)(127 + W.fe) << 23));
    b.ab = sc < 65536.0f ? (uint32_t)__half_as_ushort(__float2half_rn(sc)) : 0x7C00u;
  } else {
    cap = __float_as_uint(W.lim) - 1u;
    b.ab = av;
  }
  b.low = ~(uint32_t)ka >= tli && b.ab != 0u && b.ab <= cap;
  b.ab = min(b.ab, cap);
  if (b.low) b.ab--;
  if constexpr (DT != PEAT_F32) b.ab |= b.ab << 16;
  b.ub = min(uv, (uint32_t)Tab<DT>::UMAX);
  const bool lu = ~(uint32_t)ku >= tli && b.ub != 0u && uv <= (uint32_t)Tab<DT>::UMAX, lr = ~(uint32_t)kr >= tli;
  if (lu) b.ub--;
  b.low = b.low || lu || (DT != PEAT_F32 && lr && kr != 0ull);
  const float q = __uint_as_float((uint32_t)(kr >> 32));
  // 16-bit types: q is the record's ratio rounded to nearest, and two distinct
  // ratios of window pairs (|d| and |g| of at most 8 and 11 significant bits)
  // differ by more than 2^-20 of their value, so a factor 1 +- 2^-22 separates
  // them exactly.  float32: always lowered (q is a lower bound already).
  b.r = __fmul_rn(q, DT == PEAT_F32 || lr ? 0.99999976158142090f : 1.0000002384185791f);
  return b;
}

// atomicMax of a 64-bit shared key (a compare-and-swap loop that every warp of
// a CTA would run for every vector here) only where it raises the key
__device__ __forceinline__ void raise_key(unsigned long long* k, unsigned long long v) {
  if (v > *reinterpret_cast<volatile unsigned long long*>(k)) atomicMax(k, v);
}

// One vector position of a staged tile, all lanes of the warp, when some pair
// of it is out of the window or above a bound: pairs out of the window go to
// the general list, the window maxima into the CTA's records, and the tile's
// pairs that the table phase must not see (general pairs, equal pairs holding
// NaN, Inf or a golden above the window) are zeroed in the stage.  Returns the
// lane's general pairs and (high half) unequal pairs.  Out of line: it runs a
// few times per warp on ordinary data.
template <int DT>
__device__ __noinline__ uint32_t slow_vec(Smem<DT>& sm, uint4* gt, uint4* ct, uint32_t li0, int lb, int fe) {
  using Ty = Tr<DT>;
  using E = typename std::conditional<Ty::BYTES == 4, uint32_t, unsigned short>::type;
  Win W;
  if constexpr (DT == PEAT_F32) set_window_lb<DT>(W, lb);
  else W.lim = W.M1 = W.M2 = 0.0f, W.lb = 0;
  W.rtol = W.atol = 0.0f;
  W.fe = fe;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  E* g = reinterpret_cast<E*>(gt);
  E* c = reinterpret_cast<E*>(ct);
  float ba = 0.0f, rq = 0.0f, ra = 0.0f, rg = 1.0f;
  const float qlow = __uint_as_float((uint32_t)(*reinterpret_cast<volatile unsigned long long*>(&sm.k.krel) >> 32));
  uint32_t ai = 0, bu = 0, ui = 0, ri = 0, nd = 0, ne = 0, nf = 0, em = 0, um0 = 0;
  {
#pragma unroll 1
    for (int j = 0; j < Ty::VEC; j++) {
      const uint32_t G = g[j], C = c[j];
      if constexpr (DT == PEAT_F32) {  // what places the next window
        const uint32_t mg = G & Ty::MAG;
        if (mg < Ty::INF) em = max(em, mg >> Ty::MB);
        if (((G ^ C) & Ty::SIGN) == 0u && mg < Ty::INF && (C & Ty::MAG) < Ty::INF) um0 = max(um0, G > C ? G - C : C - G);
      }
      if (G == C) {
        // binary16: an equal pair whose scaled golden overflows would count
        // d = -inf in T1
        const uint32_t over = DT == PEAT_F16 ? min((uint32_t)(31 - fe) << 10, Ty::INF) : Ty::INF;
        if ((G & Ty::MAG) >= over) {
          if ((G & Ty::MAG) >= Ty::INF) nf++;
          g[j] = 0;
          c[j] = 0;
        }
        continue;
      }
      ne++;
      uint32_t u;
      float gf, a;
      if (!pair_window<DT>(G, C, W, u, gf, a)) {
        defer_pair<DT>(li0 + j, sm);
        nd++;
        g[j] = 0;
        c[j] = 0;
        continue;
      }
      const float ag = fabsf(gf);
      if (a > ba) ba = a, ai = li0 + j;
      if (u > bu) bu = u, ui = li0 + j;
      // the ratio only where it can reach the CTA's best (the margin covers the reciprocal's error)
      if (__fmul_rn(__fmul_rn(a, rcp_approx(ag)), 1.00001f) < qlow) continue;
      if constexpr (DT == PEAT_F32) {
        if (rel_greater(a, ag, ra, rg)) ra = a, rg = ag, ri = li0 + j;
      } else {
        const float q = __fdiv_rn(a, ag);
        if (q > rq) rq = q, ra = a, rg = ag, ri = li0 + j;
      }
    }
  }
  if (nf) atomicAdd(&sm.k.nfe, nf);
  if constexpr (DT == PEAT_F32) {
    em = __reduce_max_sync(0xFFFFFFFFu, em);
    um0 = __reduce_max_sync(0xFFFFFFFFu, um0);
    if (lane == 0) {
      sm.k.wem[warp] = max(sm.k.wem[warp], em);
      sm.k.wum[warp] = max(sm.k.wum[warp], um0);
    }
  }
  // lanes hold consecutive elements, so the lowest lane has the lowest index
  const uint32_t am = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(ba));
  if (am) {
    const unsigned who = __ballot_sync(0xFFFFFFFFu, __float_as_uint(ba) == am);
    if (lane == __ffs(who) - 1) raise_key(&sm.k.kabs, ((unsigned long long)am << 32) | (uint32_t)~ai);
  }
  const uint32_t um = __reduce_max_sync(0xFFFFFFFFu, bu);
  if (um) {
    const unsigned who = __ballot_sync(0xFFFFFFFFu, bu == um);
    if (lane == __ffs(who) - 1) raise_key(&sm.k.kulp, ((unsigned long long)um << 32) | (uint32_t)~ui);
  }
  if (__any_sync(0xFFFFFFFFu, ra > 0.0f)) {
    RelRec& R = sm.k.wrel[warp];
    if constexpr (DT == PEAT_F32) {
      // the lanes near the best approximate ratio, in order, compared exactly
      const float qa = ra > 0.0f ? __fdiv_rn(ra, rg) : 0.0f;
      const float qm = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(qa)));
      unsigned cand = __ballot_sync(0xFFFFFFFFu, ra > 0.0f && qa >= __fmul_rn(qm, 0.999999f));
      float xa = R.a, xg = R.g;
      uint32_t xi = R.li;
      bool up = false;
      while (cand) {
        const int s = __ffs(cand) - 1;
        cand &= cand - 1u;
        const float ya = __shfl_sync(0xFFFFFFFFu, ra, s), yg = __shfl_sync(0xFFFFFFFFu, rg, s);
        const uint32_t yi = __shfl_sync(0xFFFFFFFFu, ri, s);
        if (rel_greater(ya, yg, xa, xg)) xa = ya, xg = yg, xi = yi, up = true;
      }
      __syncwarp();
      if (up && lane == 0) {
        R.a = xa;
        R.g = xg;
        R.li = xi;
        atomicMax(&sm.k.krel, (unsigned long long)__float_as_uint(__fdiv_rd(xa, xg)) << 32);
      }
    } else {
      const uint32_t qm = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(rq));
      const unsigned who = __ballot_sync(0xFFFFFFFFu, __float_as_uint(rq) == qm);
      if (lane == __ffs(who) - 1 && rq > R.q) {
        R.a = ra;
        R.g = rg;
        R.q = rq;
        R.li = ri;
        atomicMax(&sm.k.krel, ((unsigned long long)qm << 32) | (uint32_t)~ri);
      }
    }
  }
  fence_proxy_async();  // the zeroed pairs before the next bulk copy into the stage
  __syncwarp();
  return nd | (ne << 16);
}

// ---- the tile loops ---------------------------------------------------------
// Per vector and lane: the checks of every pair (no branches), one vote, then
// the table increments.  The checks flag a pair that is not a window pair or
// lies above one of the bounds; a warp with a flagged pair runs slow_vec and
// then the table phase on what is left.  Everything the signature needs comes
// from the tables, except the tolerance count and (float32) the sums.
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ __half2 h2(uint32_t v) { return *reinterpret_cast<const __half2*>(&v); }
__device__ __forceinline__ __nv_bfloat162 b2(uint32_t v) { return *reinterpret_cast<const __nv_bfloat162*>(&v); }
template <class T>
__device__ __forceinline__ uint32_t bits2(const T& v) {
  return *reinterpret_cast<const uint32_t*>(&v);
}
// add one to the shared word at byte offset off of the dynamic shared memory
// (constant plus a register: one instruction)
extern __shared__ __align__(128) unsigned char smem_raw[];
__device__ __forceinline__ void inc_shared(uint32_t base, uint32_t off) {
  asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(base + off));
}
// mism += |d| > atol + rtol |g|, exactly: |d| is a float32, so it exceeds the
// bound when it exceeds the bound rounded down, and the difference (a normal
// number, |d| >= 2^-100) times 2^127 saturates to 0 or 1.  All on the FP32
// pipe, which has twice the rate of compares and integer adds.
__device__ __forceinline__ void count_mismatch(float& mism, float d, float g, const Win& W) {
  const float over = __fsub_rn(fabsf(d), __fmaf_rd(W.rtol, fabsf(g), W.atol));
  mism += __saturatef(__fmul_rn(over, 0x1p127f));
}

// the two halves of a packed pair as float32
__device__ __forceinline__ float lo_b(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float hi_b(uint32_t v) { return __uint_as_float(v & 0xFFFF0000u); }

// NP packed pairs of pairs: what both phases use
template <int NP>
struct Vec16 {
  uint32_t t[NP];  // packed ULP steps + UMAX + 1
  uint32_t d[NP];  // packed (scaled) differences c - g
  uint32_t g[NP];  // packed (scaled) goldens
};
// Packed pattern differences plus the bias: each half in (0, 2 bias) for a
// window pair.  A borrow or a carry out of the low half means that the low pair
// is flagged as well (out of range, or holding NaN or Inf).
template <int DT, int NP>
__device__ __forceinline__ void prep16(Vec16<NP>& v, const uint32_t (&g)[NP], const uint32_t (&c)[NP], uint32_t scale2) {
  constexpr uint32_t BIAS = (uint32_t)(Tab<DT>::UMAX + 1) * 0x10001u;
#pragma unroll
  for (int i = 0; i < NP; i++) {
    v.t[i] = c[i] - g[i] + BIAS;
    if constexpr (DT == PEAT_BF16) {
      v.g[i] = g[i];
      v.d[i] = bits2(__hsub2(b2(c[i]), b2(g[i])));
    } else {
      const __half2 gs = __hmul2(h2(g[i]), h2(scale2));
      v.g[i] = bits2(gs);
      v.d[i] = bits2(__hfma2(h2(c[i]), h2(scale2), __hneg2(gs)));
    }
  }
}
// true when a pair of the vector is flagged; um: the largest step count of each
// half, above UMAX or NaN when a pair is too far apart
template <int DT, int NP>
__device__ __forceinline__ bool check16(const Vec16<NP>& v, const Win& W, const Bounds& B, __half2& um) {
  // the biased step counts are binary16 subnormals: exact sums in units of 2^-24
  constexpr uint32_t NBIAS = (uint32_t)(Tab<DT>::UMAX + 1) * 0x10001u | 0x80008000u;
  um = h2(0u);
  float xm = 0.0f;
  bool bad;
#pragma unroll
  for (int i = 0; i < NP; i++) um = __hmax2_nan(um, __habs2(__hadd2(h2(v.t[i]), h2(NBIAS))));
  bad = !__hble2(um, h2(B.ub * 0x10001u));
  if constexpr (DT == PEAT_BF16) {
    const __nv_bfloat162 fl = b2((uint32_t)W.fe * 0x00800080u);
    __nv_bfloat162 am = b2(0u), tiny = b2(0u);
#pragma unroll
    for (int i = 0; i < NP; i++) {
      const __nv_bfloat162 ad = __habs2(b2(v.d[i]));
      am = __hmax2_nan(am, ad);
      tiny = __hfma2(__hlt2(ad, fl), ad, tiny);  // a difference below T1 (but not zero)
      xm = max3(xm, __fmaf_rn(-fabsf(lo_b(v.g[i])), B.r, fabsf(lo_b(v.d[i]))),
                __fmaf_rn(-fabsf(hi_b(v.g[i])), B.r, fabsf(hi_b(v.d[i]))));
    }
    bad = bad || !__hble2(am, b2(B.ab)) || (bits2(tiny) & 0x7FFF7FFFu) != 0u;
  } else {
    __half2 am = h2(0u);
#pragma unroll
    for (int i = 0; i < NP; i++) {
      am = __hmax2_nan(am, __habs2(h2(v.d[i])));
      xm = max3(xm, __fmaf_rn(-fabsf(__low2float(h2(v.g[i]))), B.r, fabsf(__low2float(h2(v.d[i])))),
                __fmaf_rn(-fabsf(__high2float(h2(v.g[i]))), B.r, fabsf(__high2float(h2(v.d[i])))));
    }
    bad = bad || !__hble2(am, h2(B.ab));
    if (W.fe < 10) {  // a subnormal golden or difference (but not zero)
      const __half2 fl = h2(0x04000400u);
      __half2 tiny = h2(0u);
#pragma unroll
      for (int i = 0; i < NP; i++) {
        const __half2 ad = __habs2(h2(v.d[i]));
        tiny = __hmax2(tiny, __hmul2(__hlt2(__hmin2(ad, __habs2(h2(v.g[i]))), fl), ad));
      }
      bad = bad || (bits2(tiny) & 0x7FFF7FFFu) != 0u;
    }
  }
  return bad || xm > 0.0f;
}
// the table phase
template <int DT, int NP>
__device__ __forceinline__ void count16(const Vec16<NP>& v, const Win& W, uint32_t t1, uint32_t t2, float& mism) {
#pragma unroll
  for (int i = 0; i < NP; i++) {
    const uint32_t d = v.d[i];
    uint32_t o1, o2;  // packed byte offsets
    if constexpr (DT == PEAT_BF16) {
      o1 = ((d & 0x1FFF1FFFu) * 4u) | (d & 0x80008000u);
      o1 ^= (d >> 5) & 0x007C007Cu;
      o2 = v.t[i] * 512u + (v.g[i] & 0x007F007Fu) * 4u;
      if (W.atol != 0.0f) {
        count_mismatch(mism, lo_b(d), lo_b(v.g[i]), W);
        count_mismatch(mism, hi_b(d), hi_b(v.g[i]), W);
      }
    } else {
      o1 = (d >> 1) & 0x7FFC7FFCu;
      o1 ^= (d >> 8) & 0x007C007Cu;
      // |d| - |g| as patterns: 1024 (floor(log2(|d| / |g|)) + 32) + a remainder
      const uint32_t y = (d | 0x80008000u) - (v.g[i] & 0x7FFF7FFFu);
      o2 = (y & 0x7C007C00u) | (v.t[i] * 4u);
      count_mismatch(mism, __low2float(h2(d)), __low2float(h2(v.g[i])), W);
      count_mismatch(mism, __high2float(h2(d)), __high2float(h2(v.g[i])), W);
    }
    inc_shared(t1, o1 & 0xFFFFu);
    inc_shared(t1, o1 >> 16);
    inc_shared(t2, o2 & 0xFFFFu);
    inc_shared(t2, o2 >> 16);
  }
}

// The pairs of a vector that are more than UMAX steps apart, each lane's in m
// (general ones, as pair_window has it): to the list, the lanes' entries taken
// together, and zeroed in the stage.
template <int DT>
__device__ __forceinline__ void drop_far(Smem<DT>& sm, uint4* gt, uint4* ct, uint32_t li, uint32_t m) {
  constexpr uint32_t ALL = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31;
  // the lanes' first places from a running count over the warp
  const uint32_t k = __popc(m);
  uint32_t at = k;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(ALL, at, o);
    if (lane >= o) at += y;
  }
  uint32_t base = 0;
  if (lane == 31) base = atomicAdd(&sm.k.gn, at);
  at += __shfl_sync(ALL, base, 31) - k;
  unsigned short *g = reinterpret_cast<unsigned short*>(gt), *c = reinterpret_cast<unsigned short*>(ct);
#pragma unroll 1
  for (; m; m &= m - 1u, at++) {
    const int j = __ffs(m) - 1;
    if (at < sm.k.gcap) sm.k.glist[at] = li + j;
    g[j] = c[j] = 0;
  }
  fence_proxy_async();  // the zeroed pairs before the next bulk copy into the stage
  __syncwarp();
}
// A dense vector with a pair too far apart.  Additive noise leaves such pairs in
// nearly every vector, so they are taken out first, without slow_vec's look at the
// maxima, and slow_vec runs only if a pair is still flagged.  Measured, 67 M pairs,
// slow_vec alone and now: noise of 1 % of the scale, bfloat16 428 -> 268 us,
// binary16 765 -> 352; of 0.1 %, 234 -> 162 and 381 -> 230.
template <int DT>
__device__ __noinline__ void slow16(Smem<DT>& sm, uint4* gt, uint4* ct, uint32_t li, int fe) {
  constexpr uint32_t UM = (uint32_t)Tab<DT>::UMAX, ALL = 0xFFFFFFFFu;
  uint32_t m = 0;
  const uint32_t *gw = reinterpret_cast<const uint32_t*>(gt), *cw = reinterpret_cast<const uint32_t*>(ct);
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const uint32_t x = gw[i], y = cw[i];
    const uint32_t lo = (y & 0xFFFFu) - (x & 0xFFFFu) + UM, hi = (y >> 16) - (x >> 16) + UM;
    m |= (lo > 2u * UM ? 1u : 0u) << (2 * i) | (hi > 2u * UM ? 2u : 0u) << (2 * i);
  }
  if (__any_sync(ALL, m != 0u)) {
    drop_far<DT>(sm, gt, ct, li, m);
    Win W;
    W.rtol = W.atol = W.lim = W.M1 = W.M2 = 0.0f, W.lb = 0;
    W.fe = fe;
    const Bounds B = read_bounds<DT>(sm, li - (threadIdx.x & 31u) * 8u, W);
    const uint32_t g[4] = {gw[0], gw[1], gw[2], gw[3]}, c[4] = {cw[0], cw[1], cw[2], cw[3]};
    Vec16<4> v;
    prep16<DT, 4>(v, g, c, (uint32_t)(15 + fe) * 0x04000400u);
    __half2 um;
    if (!__any_sync(ALL, check16<DT, 4>(v, W, B, um))) return;
  }
  slow_vec<DT>(sm, gt, ct, li, 0, fe);
}

// A vector of which few lanes hold an unequal pair: each lane visits its own
// unequal words (two pairs at a time), the rest of the warp an equal one.
// (Out of line of the dense path: late steps of a sweep and fault injections
// leave most vectors with one or two unequal pairs.)
template <int DT>
__device__ __forceinline__ void sparse16(Smem<DT>& sm, uint4* gt, uint4* ct, uint32_t m, uint32_t li,
                                         uint32_t next, const Win& W, Bounds& B, uint32_t t1, uint32_t t2, uint32_t scale2, float& mism) {
  const uint32_t* g = reinterpret_cast<const uint32_t*>(gt);
  const uint32_t* c = reinterpret_cast<const uint32_t*>(ct);
  bool checked = false;
  while (__any_sync(0xFFFFFFFFu, m != 0u)) {
    const int i = __ffs(m | 8u) - 1;  // a lane without unequal words left takes word 3, as a pair of equal ones
    uint32_t gw[1] = {g[i]}, cw[1] = {c[i]};
    if (m == 0u) cw[0] = gw[0] = 0u;
    Vec16<1> v;
    prep16<DT, 1>(v, gw, cw, scale2);
    __half2 um;
    if (!checked && __any_sync(0xFFFFFFFFu, check16<DT, 1>(v, W, B, um))) {
      slow_vec<DT>(sm, gt, ct, li, 0, W.fe);
      B = read_bounds<DT>(sm, next, W);
      checked = true;  // the whole vector
      continue;        // general pairs are zero now
    }
    m &= m - 1u;
    count16<DT, 1>(v, W, t1, t2, mism);
  }
}

// vectors with at most this many lanes holding unequal pairs take sparse16
// (a word costs about half of a whole vector)
constexpr int SPARSE_LANES = 10;

// A tile of CHV vectors (two per lane)
template <int DT>
__device__ __forceinline__ void tile16(Lane& L, Smem<DT>& sm, uint4* gt, uint4* ct, uint32_t tli, const Win& W,
                                       Bounds& B) {
  const int lane = threadIdx.x & 31;
  const uint32_t t1 = smem_addr(smem_raw) + (uint32_t)offsetof(Smem<DT>, t1);
  const uint32_t t2 = smem_addr(smem_raw) + (uint32_t)offsetof(Smem<DT>, t2);
  const uint32_t scale2 = (uint32_t)(15 + W.fe) * 0x04000400u;  // binary16: 2^s in both halves
  gt += lane;
  ct += lane;
  uint32_t li = tli + (uint32_t)lane * 8u;
#pragma unroll 1
  for (int i = 0; i < CHV / 32; i++, gt += 32, ct += 32, li += 256u) {
    uint4 gv = *gt, cv = *ct;
    const uint32_t x0 = gv.x ^ cv.x, x1 = gv.y ^ cv.y, x2 = gv.z ^ cv.z, x3 = gv.w ^ cv.w;
    const unsigned lanes = __ballot_sync(0xFFFFFFFFu, (x0 | x1 | x2 | x3) != 0u);
    if (__popc(lanes) <= SPARSE_LANES) {
      // equal lanes: EXACT pairs; the ones holding NaN or Inf also count as non-finite
      // (slow_vec when some lane has unequal words: it counts the equal pairs and zeroes them)
      if (__any_sync(0xFFFFFFFFu, any_nonfinite<DT>(gv))) {
        if (lanes == 0u) count_equal<DT>(gv, sm);
        else slow_vec<DT>(sm, gt, ct, li, 0, W.fe);
      }
      if (lanes) {
        const uint32_t m = (x0 ? 1u : 0u) | (x1 ? 2u : 0u) | (x2 ? 4u : 0u) | (x3 ? 8u : 0u);
        sparse16<DT>(sm, gt, ct, m, li, tli + (uint32_t)(i + 1) * 256u, W, B, t1, t2, scale2, L.mism);
      }
      continue;
    }
    Vec16<4> v;
    uint32_t g[4] = {gv.x, gv.y, gv.z, gv.w}, c[4] = {cv.x, cv.y, cv.z, cv.w};
    prep16<DT, 4>(v, g, c, scale2);
    __half2 um;
    if (__any_sync(0xFFFFFFFFu, check16<DT, 4>(v, W, B, um))) {
      // (a vector flagged for its maxima alone goes straight to slow_vec: the few
      // of them at the start of a piece are a chain, 1.5 us more each through slow16)
      if (__any_sync(0xFFFFFFFFu, !__hble2(um, h2((uint32_t)Tab<DT>::UMAX * 0x10001u)))) slow16<DT>(sm, gt, ct, li, W.fe);
      else slow_vec<DT>(sm, gt, ct, li, 0, W.fe);
      gv = *gt;
      cv = *ct;
      const uint32_t gn[4] = {gv.x, gv.y, gv.z, gv.w}, cn[4] = {cv.x, cv.y, cv.z, cv.w};
      prep16<DT, 4>(v, gn, cn, scale2);
      B = read_bounds<DT>(sm, tli + (uint32_t)(i + 1) * 256u, W);
    }
    count16<DT, 4>(v, W, t1, t2, L.mism);
  }
}

__device__ __forceinline__ void tile32(Lane& L, Smem<PEAT_F32>& sm, uint4* gt, uint4* ct, uint32_t tli, Win& W,
                                       Bounds& B, uint32_t ichunk) {
  const int lane = threadIdx.x & 31;
  const uint32_t t2 = smem_addr(smem_raw) + (uint32_t)offsetof(Smem<PEAT_F32>, t2);
  uint32_t nd = 0, total = 0;
  const uint32_t M1b = __float_as_uint(W.M1), M2b = __float_as_uint(W.M2);
  // sums of the bits of |d| + M1, its remainder + M2, and the same of d: per
  // tile 8 times the bits of M1 and M2 too many
  uint32_t a1 = 0, a2 = 0, s1 = 0, s2 = 0;
  gt += lane;
  ct += lane;
  uint32_t li = tli + (uint32_t)lane * 4u;
#pragma unroll 1
  for (int v = 0; v < CHV / 32; v++, gt += 32, ct += 32, li += 128u) {
    uint4 gv = *gt, cv = *ct;
    const bool diff = ((gv.x ^ cv.x) | (gv.y ^ cv.y) | (gv.z ^ cv.z) | (gv.w ^ cv.w)) != 0u;
    if (!__any_sync(0xFFFFFFFFu, diff)) {
      count_equal<PEAT_F32>(gv, sm);
      a1 += 4u * M1b;
      s1 += 4u * M1b;
      a2 += 4u * M2b;
      s2 += 4u * M2b;
      continue;
    }
    float d[4];
    int t[4];
    auto prep = [&] {
      const uint32_t g[4] = {gv.x, gv.y, gv.z, gv.w}, c[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
      for (int j = 0; j < 4; j++) {
        d[j] = __fsub_rn(__uint_as_float(c[j]), __uint_as_float(g[j]));
        t[j] = (int)(c[j] - g[j]);
      }
    };
    prep();
    {
      const float g[4] = {__uint_as_float(gv.x), __uint_as_float(gv.y), __uint_as_float(gv.z), __uint_as_float(gv.w)};
      float am = 0.0f, em = 0.0f, xm = 0.0f;
      int tmx = 0, tmn = 0;
      auto err = [&](float x) {  // d not a multiple of 2^Lexp
        const float l = __fsub_rn(x, __fsub_rn(__fadd_rn(x, W.M1), W.M1));
        return fabsf(__fsub_rn(__fsub_rn(__fadd_rn(l, W.M2), W.M2), l));
      };
#pragma unroll
      for (int j = 0; j < 4; j += 2) {
        tmx = max(tmx, max(t[j], t[j + 1]));
        tmn = min(tmn, min(t[j], t[j + 1]));
        am = max3_nan(am, fabsf(d[j]), fabsf(d[j + 1]));
        em = max3(em, err(d[j]), err(d[j + 1]));
        xm = max3(xm, __fmaf_rn(-fabsf(g[j]), B.r, fabsf(d[j])), __fmaf_rn(-fabsf(g[j + 1]), B.r, fabsf(d[j + 1])));
      }
      const bool bad = !(am <= __uint_as_float(B.ab)) || em != 0.0f || xm > 0.0f || tmx > (int)B.ub || tmn < -(int)B.ub;
      if (__any_sync(0xFFFFFFFFu, bad)) {
        if (total == 0 && lane == 0) sm.k.wem[threadIdx.x >> 5] = sm.k.wum[threadIdx.x >> 5] = 0;
        const uint32_t r = slow_vec<PEAT_F32>(sm, gt, ct, li, W.lb, 0);
        nd += __reduce_add_sync(0xFFFFFFFFu, r & 0xFFFFu);
        total += __reduce_add_sync(0xFFFFFFFFu, r >> 16);
        gv = *gt;
        cv = *ct;
        prep();
        B = read_bounds<PEAT_F32>(sm, tli + (uint32_t)(v + 1) * 128u, W);
      }
    }
    const uint32_t g[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
    for (int j = 0; j < 4; j++) {
      count_mismatch(L.mism, d[j], __uint_as_float(g[j]), W);
      const float a = fabsf(d[j]);
      const float x1 = __fadd_rn(d[j], W.M1), y1 = __fadd_rn(a, W.M1);
      const float x2 = __fadd_rn(__fsub_rn(d[j], __fsub_rn(x1, W.M1)), W.M2);
      const float y2 = __fadd_rn(__fsub_rn(a, __fsub_rn(y1, W.M1)), W.M2);
      s1 += __float_as_uint(x1);
      s2 += __float_as_uint(x2);
      a1 += __float_as_uint(y1);
      a2 += __float_as_uint(y2);
      const int v1 = (int)(__float_as_uint(y1) - M1b), v2 = (int)(__float_as_uint(y2) - M2b);
      L.Q11 += (uint64_t)((int64_t)v1 * v1);
      L.Q12 += (int64_t)v1 * v2;
      L.Q22 += (uint64_t)((int64_t)v2 * v2);
      // row floor(log2(|d| / |g|)) mod 32: bits 23 .. 27 of the difference of
      // the patterns (the signs only reach bit 31)
      const uint32_t y = __float_as_uint(d[j]) - g[j];
      inc_shared(t2, ((y >> 15) & 0x1F00u) | (uint32_t)(min(abs(t[j]), 63) * 4));
    }
  }
  L.A += ((int64_t)(int32_t)(a1 - 8u * M1b) << 21) + (int32_t)(a2 - 8u * M2b);
  L.S += ((int64_t)(int32_t)(s1 - 8u * M1b) << 21) + (int32_t)(s2 - 8u * M2b);
  if (nd >= 32u && nd * 4u >= total) {
    const int lb = next_window(W.lb, ichunk, sm);
    if (lb >= 0) {
      flush_sums(L, sm, win_lexp<PEAT_F32>(W));
      set_window_lb<PEAT_F32>(W, lb);
      B.low = true;  // the bound on |d| depends on the window
    }
  }
}

// The tile loop out of line: tiles staged by the warp's lanes and partial ones
// (a second inlined copy would only cost registers and instruction cache; by
// value, so that the caller's state stays in registers).
struct ColdOut {
  Lane L;
  int lb;
};
template <int DT>
__device__ __noinline__ ColdOut tile_cold(Lane L, Smem<DT>& sm, uint4* gt, uint4* ct, uint32_t tli, Win W, int ichunk) {
  fence_proxy_async();  // the lanes' stores to the stage, before a later bulk copy into it
  __syncwarp();
  Bounds B = read_bounds<DT>(sm, tli, W);
  if constexpr (DT == PEAT_F32) tile32(L, sm, gt, ct, tli, W, B, (uint32_t)ichunk);
  else tile16<DT>(L, sm, gt, ct, tli, W, B);
  __syncwarp();
  return ColdOut{L, W.lb};
}

// Elements [e0, e1) (at most a tile) staged by the warp's lanes; the rest of the
// tile: pairs of zeros (EXACT, not counted).
template <int DT, bool INJ>
__device__ __noinline__ void stage_scalar(const CompareParams& p, uint4* gt, uint4* ct, int64_t e0, int64_t e1) {
  using Ty = Tr<DT>;
  using E = typename std::conditional<Ty::BYTES == 4, uint32_t, unsigned short>::type;
  for (int e = threadIdx.x & 31; e < CHV * Ty::VEC; e += 32) {
    uint32_t G = 0, C = 0;
    if (e0 + e < e1) {
      G = load_scalar<DT>(p.g, e0 + e);
      C = cand_at<DT, INJ>(p, e0 + e, G);
    }
    reinterpret_cast<E*>(gt)[e] = (E)G;
    reinterpret_cast<E*>(ct)[e] = (E)C;
  }
}


// ---------------------------------------------------------------------------
// CTA ranges: boundaries precomputed on the host
// ---------------------------------------------------------------------------
// The last CTA b with bounds[b] <= i (0 <= i), searched by a whole warp:
// each round the lanes probe 32 evenly spaced bounds of the bracket and a
// ballot keeps the last one at or below i, so 32^r CTAs take r rounds of
// parallel loads instead of a chain of log2(nctas) dependent ones.
__device__ __forceinline__ int cta_of_warp(int64_t i, const CompareParams& p) {
  const int lane = threadIdx.x & 31;
  int lo = 0, hi = p.nctas - 1;  // bounds[lo] = 0 <= i: the answer lies in [lo, hi]
  while (lo < hi) {
    const int step = (hi - lo + 32) / 32;
    const int q = lo + lane * step;
    const bool ok = lane == 0 || (q <= hi && __ldg(p.bounds + q) <= i);  // a prefix of the lanes (bounds ascend)
    const int t = 31 - __clz(__ballot_sync(0xFFFFFFFFu, ok));
    lo += t * step;
    hi = min(hi, lo + step - 1);
  }
  return lo;
}

// first segment s with offsets[s+1] > i
__device__ int64_t seg_of(int64_t i, const int64_t* off, int64_t nseg) {
  int64_t lo = 0, hi = nseg - 1;
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (off[mid + 1] > i) hi = mid;
    else lo = mid + 1;
  }
  return lo;
}

// ---------------------------------------------------------------------------
// merging maxima records
// ---------------------------------------------------------------------------
__device__ __forceinline__ void part_none(Partial& r) {
  r.abs_hi = r.abs_lo = 0.0f;
  r.abs_sc = r.pad0 = 0;
  r.abs_idx = -1;
  r.rel_hi = r.rel_lo = 0.0f;
  r.rel_g = 1.0f;
  r.rel_sc = 0;
  r.rel_idx = -1;
  r.ulp = 0;
  r.ulp_idx = -1;
  r.first_fin = r.first_ulp = -1;
}

__device__ __forceinline__ int64_t min_idx(int64_t a, int64_t b) {
  if (a < 0) return b;
  if (b < 0) return a;
  return a < b ? a : b;
}

// x <- the better of x and y, field by field; ties to the lower index
__device__ __forceinline__ void part_merge(Partial& x, const Partial& y) {
  if (y.abs_idx >= 0) {
    int c = x.abs_idx < 0 ? 1 : cmp_mag(y.abs_hi, y.abs_lo, y.abs_sc, x.abs_hi, x.abs_lo, x.abs_sc);
    if (c > 0 || (c == 0 && y.abs_idx < x.abs_idx)) {
      x.abs_hi = y.abs_hi;
      x.abs_lo = y.abs_lo;
      x.abs_sc = y.abs_sc;
      x.abs_idx = y.abs_idx;
    }
  }
  if (y.rel_idx >= 0) {
    int c = x.rel_idx < 0 ? 1 : cmp_rel_rec(y.rel_hi, y.rel_lo, y.rel_sc, y.rel_g, x.rel_hi, x.rel_lo, x.rel_sc, x.rel_g);
    if (c > 0 || (c == 0 && y.rel_idx < x.rel_idx)) {
      x.rel_hi = y.rel_hi;
      x.rel_lo = y.rel_lo;
      x.rel_sc = y.rel_sc;
      x.rel_g = y.rel_g;
      x.rel_idx = y.rel_idx;
    }
  }
  if (y.ulp_idx >= 0 && (x.ulp_idx < 0 || y.ulp > x.ulp || (y.ulp == x.ulp && y.ulp_idx < x.ulp_idx))) {
    x.ulp = y.ulp;
    x.ulp_idx = y.ulp_idx;
  }
  x.first_fin = min_idx(x.first_fin, y.first_fin);
  x.first_ulp = min_idx(x.first_ulp, y.first_ulp);
}

__device__ __forceinline__ uint64_t warp_min64(uint64_t v) {
  const uint32_t h = __reduce_min_sync(0xFFFFFFFFu, (uint32_t)(v >> 32));
  const uint32_t l = __reduce_min_sync(0xFFFFFFFFu, (uint32_t)(v >> 32) == h ? (uint32_t)v : 0xFFFFFFFFu);
  return ((uint64_t)h << 32) | l;
}

// The best of the warp's 32 records, field by field, into *out (shared or
// global; the warp synchronises afterwards).  Each maximum goes by 32-bit
// warp reductions over keys (value, then rounding error, then index), and the
// lane that holds it stores it: no record travels between lanes.  A ratio's
// key is approximate; the lanes within its margin of the best are compared
// exactly with one of them, all at once, until none is greater.  Out of line
// and by value: its four callers run once each, so the fetch of the code is
// most of its time and they share it (a tournament of whole records over
// shuffles took 2 to 10 us at each place, this 0.7 to 2).
__device__ __noinline__ void warp_best(float ah, float al, int as, int64_t ai, float rh, float rl, float rg, int rs,
                                       int64_t ri, uint64_t u, int64_t ui, int64_t ff, int64_t fu, Partial* out) {
  const uint32_t all = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31;
  {
    // (scaled values exceed every unscaled float32)
    const uint32_t k = ai < 0 ? 0u : __float_as_uint(ah) + ((uint32_t)as << 23) + 1u;
    const uint32_t m = __reduce_max_sync(all, k);
    const uint32_t b = __float_as_uint(al);
    const uint32_t kl = k != m ? 0u : (al == 0.0f ? 0x80000000u : ((b & 0x80000000u) ? ~b : (b | 0x80000000u)));
    const uint32_t ml = __reduce_max_sync(all, kl);
    const bool c = k == m && kl == ml;
    const uint64_t i = warp_min64(c ? (uint64_t)ai : ~0ull);
    if (m ? (c && (uint64_t)ai == i) : lane == 0) {
      out->abs_hi = ah;
      out->abs_lo = al;
      out->abs_sc = as;
      out->pad0 = 0;
      out->abs_idx = ai;
    }
  }
  {
    constexpr int NONE = (int)0x80000000;
    const int k = ri < 0 ? NONE : ratio_key(rh, rs, rg);
    const int m = __reduce_max_sync(all, k);
    uint32_t cand = __ballot_sync(all, ri >= 0 && (long long)k >= (long long)m - RATIO_MARGIN);
    while (cand & (cand - 1)) {
      const int w = __ffs(cand) - 1;
      const float wh = __shfl_sync(all, rh, w), wl = __shfl_sync(all, rl, w), wg = __shfl_sync(all, rg, w);
      const int ws = __shfl_sync(all, rs, w);
      const int c = lane == w ? 0 : ((cand >> lane) & 1u) ? cmp_rel_close(rh, rl, rs, rg, wh, wl, ws, wg) : -1;
      const uint32_t gt = __ballot_sync(all, c > 0), eq = __ballot_sync(all, c == 0);
      cand = gt ? gt : eq;
      if (!gt) break;
    }
    const bool c = ((cand >> lane) & 1u) != 0;
    const uint64_t i = warp_min64(c ? (uint64_t)ri : ~0ull);
    if (cand ? (c && (uint64_t)ri == i) : lane == 0) {
      out->rel_hi = rh;
      out->rel_lo = rl;
      out->rel_g = rg;
      out->rel_sc = rs;
      out->rel_idx = ri;
    }
  }
  {
    const uint64_t v = ui < 0 ? 0ull : u;  // a recorded distance is positive
    const uint64_t m = ~warp_min64(~v);
    const uint64_t i = warp_min64(m && v == m ? (uint64_t)ui : ~0ull);
    if (m ? (v == m && (uint64_t)ui == i) : lane == 0) {
      out->ulp = u;
      out->ulp_idx = ui;
    }
  }
  // -1 (none) is the largest unsigned value
  const uint64_t f = warp_min64((uint64_t)ff), g = warp_min64((uint64_t)fu);
  if (lane == 0) {
    out->first_fin = (int64_t)f;
    out->first_ulp = (int64_t)g;
  }
  __syncwarp();
}
__device__ __forceinline__ void warp_best(const Partial& x, Partial* out) {
  warp_best(x.abs_hi, x.abs_lo, x.abs_sc, x.abs_idx, x.rel_hi, x.rel_lo, x.rel_g, x.rel_sc, x.rel_idx, x.ulp, x.ulp_idx,
            x.first_fin, x.first_ulp, out);
}

// warp sums of the general path's class counters into the CTA counters
template <int DT>
__device__ __forceinline__ void gen_counts(const GenRec& g, Smem<DT>& sm) {
  const int lane = threadIdx.x & 31;
  const uint32_t gen = g.n_gw + g.n_gm + g.n_ga + g.n_gf + g.n_geq;
  const uint32_t c[7] = {g.n_geq, gen, g.n_nf, g.n_gw, g.n_gm, g.n_ga, g.n_gf};
  uint32_t v[7];
#pragma unroll
  for (int k = 0; k < 7; k++) v[k] = __reduce_add_sync(0xFFFFFFFFu, c[k]);
  if (lane == 0) {
    // EXACT: the piece length less the window pairs, less the general pairs that differ
    if (v[1] != v[0]) atomicAdd(&sm.k.cnt[0], 0ull - (unsigned long long)(v[1] - v[0]));
    if (v[2]) atomicAdd(&sm.k.cnt[3], (unsigned long long)v[2]);
    if (v[3]) atomicAdd(&sm.k.cnt[4], (unsigned long long)v[3]);
    if (v[4]) atomicAdd(&sm.k.cnt[5], (unsigned long long)v[4]);
    if (v[5]) atomicAdd(&sm.k.cnt[6], (unsigned long long)v[5]);
    if (v[6]) atomicAdd(&sm.k.cnt[7], (unsigned long long)v[6]);
  }
}

// The rescan of a piece whose general pairs overflowed its list: slot k of the
// warp's, its general pairs added to the cnt entries of the warp's queue (in its
// part of the staging ring, idle now), so that general_lane runs on full warps.
// Slot 0 is the head, then 32 x VEC elements of the body each, the last one the
// tail.  With one round of general_lane per 32 elements, whatever they held: 67 M
// binary16 pairs of which 5 % are general 2520 us, float32 pairs of which a third
// are 3250; now 765 and 1085.
template <int DT>
struct Queue {
  static constexpr uint32_t SLOT = 32 * Tr<DT>::VEC;
  uint32_t *i, *g, *c;  // offsets from the CTA's first element; goldens (16-bit types: with the candidate); candidates
  __device__ __forceinline__ Queue(Smem<DT>& sm) {
    i = reinterpret_cast<uint32_t*>(sm.ring.g[threadIdx.x >> 5]);
    c = reinterpret_cast<uint32_t*>(sm.ring.c[threadIdx.x >> 5]);
    g = DT == PEAT_F32 ? i + CHV * 4 * NSTAGE / 2 : c;
  }
};
static_assert(Queue<PEAT_F16>::SLOT + 31 <= CHV * 4 * NSTAGE && Queue<PEAT_F32>::SLOT + 31 <= CHV * 4 * NSTAGE / 2,
              "the queue fits the ring");
template <int DT, bool INJ>
__device__ __noinline__ uint32_t scan_slot(Win W, Smem<DT>& sm, const CompareParams& p, int64_t pb, int64_t pe, int64_t vb,
                                           int64_t ve, int64_t k, uint32_t cnt) {
  constexpr int VEC = Tr<DT>::VEC, B = Tr<DT>::BYTES, NW = Geo<DT>::NW;
  constexpr uint32_t SLOT = Queue<DT>::SLOT;
  const uint32_t lane = threadIdx.x & 31u;
  const Queue<DT> q(sm);
  const int64_t b = k == 0 ? pb : vb + (k - 1) * (int64_t)SLOT;
  const int64_t e = k == 0 ? vb : b < ve ? min(b + SLOT, ve) : pe, b1 = k == 0 || b < ve ? b : ve;
  if constexpr (DT == PEAT_F32) {
    // the window this slot was tested with: the head ran with the initial
    // window, a body chunk with its warp's window of that time, the tail with
    // warp 0's last window
    int w = 0;
    uint32_t ik = 0;
    if (vb < ve && k > 0) {
      if (b >= ve) {
        ik = 0xFFFFFFFFu;
      } else {
        const int64_t t = (b - vb) / (CHV * VEC);
        w = (int)(t % NW);
        ik = (uint32_t)(t / NW);
      }
    }
    int r = (int)sm.k.nwin[w];
    while (r > 0 && sm.k.wstart[w][r] > ik) r--;
    set_window_lb<DT>(W, sm.k.wlb[w][r]);
  }
  uint32_t G[VEC], C[VEC];
  // whole vectors where the slot holds them on their grid, else elements lane + 32 j
  const uintptr_t ob = (uintptr_t)b1 * B;
  const bool vec = e - b1 == SLOT && ((((uintptr_t)p.g + ob) | (INJ ? 0 : (uintptr_t)p.c + ob)) & 15u) == 0;
  if (vec) {
    const int64_t i0 = b1 + (int64_t)lane * VEC;
    const uint4 gv = load_vec(p.g, i0 * B);
    const uint4 cv = INJ ? inj_one<DT>(p, gv, i0) : load_vec(p.c, i0 * B);
    unpack_vec<DT>(gv, G);
    unpack_vec<DT>(cv, C);
  } else {
#pragma unroll
    for (int j = 0; j < VEC; j++) {
      const int64_t i = b1 + lane + 32 * j;
      G[j] = C[j] = 0;
      if (i < e) {
        G[j] = load_scalar<DT>(p.g, i);
        C[j] = cand_at<DT, INJ>(p, i, G[j]);
      }
    }
  }
  const uint32_t li = (uint32_t)(b1 - sm.k.lo);
#pragma unroll
  for (int j = 0; j < VEC; j++) {
    uint32_t u;
    float gf, a;
    const bool want = G[j] != C[j] && !pair_window<DT>(G[j], C[j], W, u, gf, a);
    const unsigned m = __ballot_sync(0xFFFFFFFFu, want);
    if (want) {
      const uint32_t at = cnt + __popc(m & ((1u << lane) - 1u));
      q.i[at] = li + (vec ? lane * VEC + j : lane + 32 * j);
      q.g[at] = DT == PEAT_F32 ? G[j] : G[j] | (C[j] << 16);
      if constexpr (DT == PEAT_F32) q.c[at] = C[j];
    }
    cnt += __popc(m);
  }
  __syncwarp();
  return cnt;
}

// The general pairs of a piece [pb, pe), evaluated exactly by every thread of
// the CTA: from the list when it held them all, else found again by a rescan
// of the piece with the same window test.  ALL: every pair of the piece.  Out of line, so that the hot loop
// carries no call.  Leaves each warp's general maxima in sm.k.wbest[warp].
template <int DT, bool INJ, bool ALL>
__device__ __noinline__ void run_general(Win W, Smem<DT>& sm, const CompareParams& p, int64_t pb, int64_t pe,
                                         int64_t vb, int64_t ve) {
  constexpr int NT = Geo<DT>::NT, NW = Geo<DT>::NW;
  // entered only after a barrier and with at least one general pair (finish_piece)
  const uint32_t n = ALL ? (uint32_t)(pe - pb) : sm.k.gn;
  const int64_t lo = sm.k.lo;
  GenRec cd;
  gen_init(cd);
  GenSum gs;
  // whole warps in every round (general_lane counts with the whole warp)
  const uint32_t lane = threadIdx.x & 31u;
  const bool listed = ALL || n <= sm.k.gcap, many = !ALL && n > GEN_MANY;
  uint32_t b = threadIdx.x & ~31u, cnt = 0;  // the warp's place in the list; its queue
  int64_t k = threadIdx.x >> 5;
  const int64_t slots = (ve - vb + Queue<DT>::SLOT - 1) / Queue<DT>::SLOT + 2;
  for (int rounds = 0;; rounds++) {
    int64_t i = 0;
    uint32_t G = 0, C = 0;
    bool valid;
    if (listed) {
      if (b >= n) break;
      valid = b + lane < n;
      if (valid) {
        i = ALL ? pb + b + lane : lo + sm.k.glist[b + lane];
        if (!PEAT_CHECK(i >= 0 && i < p.n_total)) i = lo;  // a listed offset outside the tensor
        G = load_scalar<DT>(p.g, i);
        C = cand_at<DT, INJ>(p, i, G);
      }
      b += NT;
    } else {
      for (; cnt < 32u && k < slots; k += NW) cnt = scan_slot<DT, INJ>(W, sm, p, pb, pe, vb, ve, k, cnt);
      if (cnt == 0u) break;
      const uint32_t take = min(cnt, 32u);
      const Queue<DT> q(sm);
      cnt -= take;
      valid = lane < take;
      if (valid) {
        i = lo + q.i[cnt + lane];
        G = q.g[cnt + lane];
        if constexpr (DT == PEAT_F32) C = q.c[cnt + lane];
        else C = G >> 16, G &= 0xFFFFu;
      }
      __syncwarp();
    }
    if (rounds == GEN_FLUSH) gen_flush<DT>(sm), rounds = 0;
    general_lane<DT>(sm, cd, gs, many, G, C, i, p.rtol, p.atol, valid);
  }
  if constexpr (DT == PEAT_F16)
    if (many) gen_sums(gs, sm);
  fence_proxy_async();  // the queue, before the next piece's bulk copies into the ring
  gen_counts<DT>(cd, sm);
  warp_best(cd.abs_hi, cd.abs_lo, cd.abs_sc, cd.abs_idx, cd.rel_hi, cd.rel_lo, cd.rel_g, cd.rel_sc, cd.rel_idx, cd.ulp,
            cd.ulp_idx, -1, -1, &sm.k.wbest[threadIdx.x >> 5]);
  __syncthreads();
  // the per-warp totals into the CTA's
  for (int b = threadIdx.x; b < HBINS; b += NT) {
    unsigned long long v = 0;
#pragma unroll
    for (int w = 0; w < NW; w++) {
      v += sm.k.ghist[w][b];
      sm.k.ghist[w][b] = 0;
    }
    if (v) atomicAdd(&sm.k.hist[b], v);
  }
  for (int j = threadIdx.x; j < NSUM * NLIMB; j += NT) {
    int64_t v = 0;
#pragma unroll
    for (int w = 0; w < NW; w++) {
      v += (int64_t)sm.k.gsacc[w][j][1] * 65536 + sm.k.gsacc[w][j][0];
      sm.k.gsacc[w][j][0] = sm.k.gsacc[w][j][1] = 0;
    }
    if (v) atomicAdd(&sm.k.sacc[0][0] + j, (unsigned long long)v);
  }
}

// [pb, pe): the lowest index of a finite pair and of a pair without NaN
// (the argmax when every error is zero), searched NT elements at a time
// (the piece's first pair, which settles both unless it holds NaN or Inf, is
// tested when the piece starts; this search runs only when it did not)
template <int DT, bool INJ>
__device__ __noinline__ void first_pairs(Smem<DT>& sm, const CompareParams& p, int64_t pb, int64_t pe) {
  using Ty = Tr<DT>;
  constexpr long long NONE = 0x7FFFFFFFFFFFFFFFll;
  for (int64_t base = pb;; base += Geo<DT>::NT) {
    // read between two barriers, where no warp lowers them: every thread leaves
    // after the same round
    __syncthreads();
    const bool found = sm.k.ff != NONE && sm.k.fu != NONE;
    __syncthreads();
    if (base >= pe || found) break;
    const int64_t i = base + threadIdx.x;
    if (i < pe) {
      const uint32_t Gi = load_scalar<DT>(p.g, i);
      const uint32_t ag = Gi & Ty::MAG, ac = cand_at<DT, INJ>(p, i, Gi) & Ty::MAG;
      if (ag < Ty::INF && ac < Ty::INF) atomicMin(&sm.k.ff, (long long)i);
      if (ag <= Ty::INF && ac <= Ty::INF) atomicMin(&sm.k.fu, (long long)i);
    }
  }
}

// Add n pairs of log2-relative exponent k, each lane its own (n = 0: none; the
// whole warp calls it): one shared atomic per distinct k of the warp.
template <int DT>
__device__ __forceinline__ void add_rel(Smem<DT>& sm, int k, uint32_t n) {
  unsigned todo = __ballot_sync(0xFFFFFFFFu, n != 0u);
  while (todo) {
    const int k0 = __shfl_sync(0xFFFFFFFFu, k, __ffs(todo) - 1);
    const bool mine = n != 0u && k == k0;
    const uint32_t s = __reduce_add_sync(0xFFFFFFFFu, mine ? n : 0u);
    if ((threadIdx.x & 31) == 0) atomicAdd(&sm.k.hist[min(max(48 + k0, 1), 62)], (unsigned long long)s);
    todo &= ~__ballot_sync(0xFFFFFFFFu, mine);
  }
}

// The window tables into the CTA's totals, leaving them zero (called by every
// thread, between barriers).
template <int DT>
__device__ __forceinline__ void fold_tables(Smem<DT>& sm, const Win& W) {
  constexpr int NT = Geo<DT>::NT, NW = Geo<DT>::NW;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t zeros = 0;  // bfloat16, warp 0: the pairs with d = 0 in T1
  uint32_t nwin = 0, nover = 0;
  if constexpr (DT == PEAT_BF16) {
    // a warp per ULP distance row, cells by the golden's significand field
    for (int t = warp; t < 128; t += NW) {
      uint32_t n[4], any = 0;
#pragma unroll
      for (int j = 0; j < 4; j++) {
        n[j] = sm.t2[t * 128 + lane + 32 * j];
        any |= n[j];
      }
      if (!__any_sync(0xFFFFFFFFu, any != 0u)) continue;
#pragma unroll
      for (int j = 0; j < 4; j++) sm.t2[t * 128 + lane + 32 * j] = 0;
      const uint32_t row = __reduce_add_sync(0xFFFFFFFFu, n[0] + n[1] + n[2] + n[3]);
      if (t == 64) {
        zeros = row;
        continue;
      }
      const int u = t - 64;
      if (lane == 0) atomicAdd(&sm.k.hist[64 + abs(u)], (unsigned long long)row);
#pragma unroll
      for (int j = 0; j < 4; j++) {
        // golden and candidate in half steps of the golden's binade [256, 512)
        const int x = 128 + lane + 32 * j + u;
        const int g2 = 2 * (128 + lane + 32 * j), c2 = x >= 256 ? 4 * x - 512 : (x < 128 ? 128 + x : 2 * x);
        const int a2 = abs(c2 - g2);
        const float fa = (float)a2, fg = (float)g2;
        const int k = (int)(__float_as_uint(fa) - __float_as_uint(fg)) >> 23;
        add_rel<DT>(sm, k, n[j]);
        // atol = 0: |d| <= rtol |g| does not depend on the binade
        if (W.atol == 0.0f && fa > __fmul_rd(W.rtol, fg)) nover += n[j];
      }
      nwin += lane == 0 ? row : 0u;
    }
  } else {
    // T2: a thread holds every (NT / COLS)-th row of one column
    constexpr int COLS = DT == PEAT_F32 ? 64 : 256, R = NT / COLS;
    constexpr int ZERO = DT == PEAT_F32 ? 0 : 128;  // the column of d = 0
    const int col = tid % COLS, r0 = tid / COLS;
#pragma unroll 4
    for (int i = 0; i < 32 / R; i++) {
      const int row = r0 + i * R;
      uint32_t* q = sm.t2 + row * COLS + col;
      const uint32_t v = col == ZERO ? 0u : *q;
      *q = 0;
      if (!__any_sync(0xFFFFFFFFu, v != 0u)) continue;
      nwin += v;
      // (a warp covers 32 columns of one row; a piece has below 2^31 pairs)
      const uint32_t s = __reduce_add_sync(0xFFFFFFFFu, v);
      const int k = row < 16 && DT == PEAT_F16 ? row : (row == 0 ? 0 : row - 32);
      if (lane == 0) atomicAdd(&sm.k.hist[min(max(48 + k, 1), 62)], (unsigned long long)s);
    }
    if (nwin) atomicAdd(&sm.k.hist[64 + (DT == PEAT_F32 ? col : min(abs(col - 128), 63))], (unsigned long long)nwin);
  }
  nwin = __reduce_add_sync(0xFFFFFFFFu, nwin);
  nover = __reduce_add_sync(0xFFFFFFFFu, nover);
  if (lane == 0 && nwin) {
    atomicAdd(&sm.k.cnt[1], (unsigned long long)nwin);            // window pairs
    atomicAdd(&sm.k.cnt[2], (unsigned long long)nwin - nover);    // of them within tolerance (mismatches taken off)
    atomicAdd(&sm.k.cnt[0], 0ull - (unsigned long long)nwin);     // are not EXACT
  }
  // T1: a warp per exponent; each counter adds count * v to sum |d| and sum d
  // and count * v^2 to sum d^2, v = 128 + M in units of the exponent's step
  if constexpr (DT != PEAT_F32) {
    constexpr int ROWS = Tab<DT>::ROWS;
    for (int r = warp; r < ROWS; r += NW) {
      uint32_t* tp = sm.t1 + r * 128;
      uint32_t* tn = tp + ROWS * 128;
      uint32_t cp[4], cn[4];
      uint32_t any = 0;
#pragma unroll
      for (int j = 0; j < 4; j++) {
        cp[j] = tp[lane + 32 * j];
        cn[j] = tn[lane + 32 * j];
      }
      if (r == 0) {  // d = 0 (warp 0, lane 0, j = 0)
        if (lane == 0) cp[0] -= DT == PEAT_BF16 ? zeros : cp[0];
        tp[lane] = 0;
      }
#pragma unroll
      for (int j = 0; j < 4; j++) any |= cp[j] | cn[j];
      if (!__any_sync(0xFFFFFFFFu, any != 0u)) continue;
      uint64_t sp = 0, sn = 0, q = 0;
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const uint32_t m = 128u + (uint32_t)((lane ^ (r & 31)) + 32 * j);
        sp += (uint64_t)cp[j] * m;
        sn += (uint64_t)cn[j] * m;
        q += (uint64_t)cp[j] * (m * m) + (uint64_t)cn[j] * (m * m);
        tp[lane + 32 * j] = 0;
        tn[lane + 32 * j] = 0;
      }
      sp = wsum64(sp);
      sn = wsum64(sn);
      q = wsum64(q);
      if (lane < NSUM) {  // a lane per sum
        const int u = DT == PEAT_BF16 ? W.fe + ((r - W.fe) & 63) - 134 : r - 22 - W.fe;
        const uint64_t m = lane == 0 ? (sp >= sn ? sp - sn : sn - sp) : (lane == 1 ? sp + sn : q);
        sacc_add<DT>(sm, lane, (unsigned __int128)m, lane == 2 ? 2 * u : u, lane == 0 && sp < sn);
      }
    }
  }
}

// The window maxima of the CTA's piece, for lane 0 of warp 0 (the whole warp
// calls it).
template <int DT>
__device__ __forceinline__ void window_best(Smem<DT>& sm, Partial& x) {
  constexpr int NW = Geo<DT>::NW;
  const int lane = threadIdx.x & 31;
  part_none(x);
  const int64_t lo = sm.k.lo;
  if ((uint32_t)sm.k.kabs) {
    x.abs_hi = __uint_as_float((uint32_t)(sm.k.kabs >> 32));
    x.abs_idx = lo + (uint32_t)~(uint32_t)sm.k.kabs;
  }
  if ((uint32_t)sm.k.kulp) {
    x.ulp = sm.k.kulp >> 32;
    x.ulp_idx = lo + (uint32_t)~(uint32_t)sm.k.kulp;
  }
  RelRec r{0.0f, 1.0f, 0.0f, 0u};
  if (lane < NW) r = sm.k.wrel[lane];
  if constexpr (DT == PEAT_F32) {
#pragma unroll
    for (int o = NW / 2; o > 0; o >>= 1) {
      const float ya = __shfl_down_sync(0xFFFFFFFFu, r.a, o), yg = __shfl_down_sync(0xFFFFFFFFu, r.g, o);
      const uint32_t yi = __shfl_down_sync(0xFFFFFFFFu, r.li, o);
      if (ya > 0.0f && (rel_greater(ya, yg, r.a, r.g) || (yi < r.li && !rel_greater(r.a, r.g, ya, yg))))
        r.a = ya, r.g = yg, r.li = yi;
    }
  } else {
    // the CTA's key names the winning pair: its warp holds it
    const uint32_t kl = (uint32_t)sm.k.krel;
    const unsigned who = __ballot_sync(0xFFFFFFFFu, kl != 0u && r.a > 0.0f && r.li == ~kl);
    const int s = who ? __ffs(who) - 1 : 0;
    r.a = __shfl_sync(0xFFFFFFFFu, who ? r.a : 0.0f, s);
    r.g = __shfl_sync(0xFFFFFFFFu, r.g, s);
    r.li = __shfl_sync(0xFFFFFFFFu, r.li, s);
  }
  if (r.a > 0.0f) {
    x.rel_hi = r.a;
    x.rel_g = r.g;
    x.rel_idx = lo + r.li;
  }
}

template <int NT>
__device__ __noinline__ void finalize_segment(const CompareParams& p, int64_t s, int b0, int b1, FinScratch& f, MV& mv);
__device__ void write_empty_segments(const CompareParams& p);

// the window maxima, class counters and list of a new piece
template <int DT>
__device__ __forceinline__ void piece_init(Smem<DT>& sm) {
  const int tid = threadIdx.x;
  if (tid < Geo<DT>::NW) sm.k.wrel[tid] = RelRec{0.0f, 1.0f, 0.0f, 0xFFFFFFFFu};
  if (tid == 32) sm.k.kabs = sm.k.kulp = sm.k.krel = 0ull;
  if (tid == 33) {
    sm.k.gn = 0;
    sm.k.nfe = 0;
    sm.k.lb = sm.k.ub = 0;
  }
  if (tid >= 64 && tid < 72) sm.k.cnt[tid - 64] = 0;
}

// End of one segment piece [pb, pe) (ALL: of which nothing has been done yet, see
// compare_short): the integer totals go to the segment's
// accumulator (global atomics), the maxima to the CTA's partial slot.  The
// CTA that finishes the segment's last piece then finalizes the segment.
template <int DT, bool INJ, bool ALL>
__device__ __forceinline__ void finish_piece(Lane& L, const Win& W, Smem<DT>& sm, const CompareParams& p,
                                             int64_t seg, int64_t pb, int64_t pe, int64_t vb, int64_t ve) {
  constexpr int NT = Geo<DT>::NT, NW = Geo<DT>::NW;
  Partial* out = p.partials + seg + blockIdx.x;
  SegAcc* acc = p.acc + seg;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if constexpr (DT == PEAT_F32 && !ALL) flush_sums(L, sm, win_lexp<DT>(W));
  if constexpr (!ALL) {
    const uint32_t over = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)L.mism);
    if (lane == 0 && over) atomicAdd(&sm.k.cnt[2], 0ull - (unsigned long long)over);
  }
  lane_init(L);
  __syncthreads();  // every tile is in the tables, the list and the records
  // the piece's general pairs, if any: the out-of-line call (and its register
  // traffic) only when there is one
  const bool gen = ALL || sm.k.gn != 0;
  if (gen) run_general<DT, INJ, ALL>(W, sm, p, pb, pe, vb, ve);
  if (sm.k.ff == 0x7FFFFFFFFFFFFFFFll || sm.k.fu == 0x7FFFFFFFFFFFFFFFll) first_pairs<DT, INJ>(sm, p, pb, pe);
  if (warp == 0) {
    Partial x;
    window_best<DT>(sm, x);
    const bool ok = PEAT_CHECK(seg >= 0 && seg < p.nseg && seg + (int64_t)blockIdx.x < p.nseg + p.nctas && pb <= pe &&
                               pe <= p.n_total);
    if (lane == 0) {
      constexpr long long NONE = 0x7FFFFFFFFFFFFFFFll;
      x.first_fin = sm.k.ff == NONE ? -1 : sm.k.ff;
      x.first_ulp = sm.k.fu == NONE ? -1 : sm.k.fu;
      if (!gen && ok) *out = x;
      atomicAdd(&sm.k.cnt[0], (unsigned long long)(pe - pb));
      atomicAdd(&sm.k.cnt[3], (unsigned long long)sm.k.nfe);
    }
    if (gen) {  // the window's records and each warp's general ones
      if (lane >= 1 && lane <= NW) x = sm.k.wbest[lane - 1];
      else if (lane > NW) part_none(x);
      if (ok) warp_best(x, out);
    }
  }
  if constexpr (!ALL) fold_tables<DT>(sm, W);
  __syncthreads();  // the totals are complete
  for (int b = tid; b < HBINS; b += NT) {
    if (sm.k.hist[b]) atomicAdd(&acc->hist[b], sm.k.hist[b]);
    sm.k.hist[b] = 0;
  }
  if (tid >= 128 && tid < 136 && sm.k.cnt[tid - 128]) atomicAdd(&acc->cnt[tid - 128], sm.k.cnt[tid - 128]);
  for (int j = tid - 160; j >= 0 && j < NSUM * NLIMB; j += NT) {
    const unsigned long long v = (&sm.k.sacc[0][0])[j];
    if (v) atomicAdd(reinterpret_cast<unsigned long long*>(&acc->limbs[0][0]) + j, v);
    (&sm.k.sacc[0][0])[j] = 0;
  }
  // publish, then count this piece: the segment's pieces are the CTAs whose
  // ranges meet it (a multi-segment call finalizes in a second launch, after
  // this one)
  if (p.nseg == 1) {
    __threadfence();
    __syncthreads();
    if (tid == 0) sm.k.last = atomicAdd(&acc->done, 1u) == (unsigned)(sm.k.final - sm.k.first);
    __syncthreads();
    if (sm.k.last) {
      __threadfence();
      finalize_segment<NT>(p, seg, sm.k.first, sm.k.final, sm.k.fin, sm.mv);
    }
  } else {
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// stage 1
// ---------------------------------------------------------------------------
// The window sample: VEC (or one) pairs per thread, from the start of the
// piece (float32) or from places all over it, give the largest finite golden
// exponent (16-bit types: of the unequal pairs that a window can take, if there
// are any, plus 256) and the largest ULP distance of a pair of one sign (they
// place the window), and starting bounds for the three maxima.  A starting bound
// is the value of some pair of the piece, so no maximum lies below it.
template <int DT, int NV>
__device__ __forceinline__ void sample_pairs(const uint32_t (&g)[NV], const uint32_t (&c)[NV], uint32_t& emax,
                                             uint32_t& umax, uint32_t& ab, uint32_t& qb) {
  using Ty = Tr<DT>;
  float am = 0.0f, qm = 0.0f;
#pragma unroll
  for (int j = 0; j < NV; j++) {
    const uint32_t G = g[j], C = c[j], mg = G & Ty::MAG, mc = C & Ty::MAG;
    const uint32_t e = mg >> Ty::MB;
    if (e < (uint32_t)Ty::EMAX && e > emax) emax = e;
    if (((G ^ C) & Ty::SIGN) == 0u && mg < Ty::INF && mc < Ty::INF && G != C) {
      const uint32_t u = G > C ? G - C : C - G;
      umax = max(umax, u);
      if (u <= (uint32_t)Tab<DT>::UMAX && mg != 0u) {
        if constexpr (DT != PEAT_F32) emax = max(emax, 256u + e);
        const float gf = fabsf(to_f32<DT>(G)), a = fabsf(__fsub_rn(to_f32<DT>(C), to_f32<DT>(G)));
        am = fmaxf(am, a);
        qm = fmaxf(qm, DT == PEAT_F32 ? __fdiv_rd(a, gf) : __fdiv_rn(a, gf));
      }
    }
  }
  ab = __float_as_uint(am);
  qb = __float_as_uint(qm);
}

// Which of a piece's n vectors (or elements) thread tid samples.  The 16-bit
// window stays where the sample puts it, so every two warps look at neighbours in
// an eighth of the piece, at a place that differs from one eighth to the next
// (rows that begin with padding would hide their data from places a multiple
// of their length apart).  Measured with the piece's first vectors sampled
// instead: 67 M bfloat16 pairs of a batch with zero padding 2246 us, now 94; an
// embedding with a zero first row 1805, now 102.  Sixteen places cost 1 to 3 us
// more (address translation), a place per thread 4.
template <int DT>
__device__ __forceinline__ uint32_t sample_at(uint32_t n, int tid) {
  constexpr uint32_t NT = Geo<DT>::NT, PLACES = 8, PER = NT / PLACES;
  if (DT == PEAT_F32 || n < 2 * NT) return (uint32_t)tid;
  const uint32_t w = (uint32_t)tid / PER, part = n / PLACES;  // (fractional parts of w times the golden ratio)
  return part * w + __umulhi(part - PER, w * 0x9E3779B9u) + (uint32_t)tid % PER;
}

template <int DT, bool INJ>
__global__ void __launch_bounds__(Geo<DT>::NT, Geo<DT>::CTAS) compare_stage1(CompareParams p) {
  using Ty = Tr<DT>;
  constexpr int VEC = Ty::VEC, NT = Geo<DT>::NT, NW = Geo<DT>::NW;
  constexpr int64_t TILE = (int64_t)CHV * VEC;
  Smem<DT>& sm = *reinterpret_cast<Smem<DT>*>(smem_raw);
  pdl_trigger();  // a multi-segment call's finalize kernel may start launching (it waits for this grid)
  // (the shuffle tells the compiler that the warp's number is the same in all
  // its lanes: addresses derived from it stay in uniform registers, as the
  // bulk copies want them)
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
  for (int b = tid; b < HBINS; b += NT) sm.k.hist[b] = 0;
  for (int j = tid; j < NSUM * NLIMB; j += NT) (&sm.k.sacc[0][0])[j] = 0;
  {  // the tables, 16 bytes per store
    uint4* tz = reinterpret_cast<uint4*>(sm.t2);
    for (int j = tid; j < Tab<DT>::N2 / 4; j += NT) tz[j] = make_uint4(0, 0, 0, 0);
    tz = reinterpret_cast<uint4*>(sm.t1);
    for (int j = tid; j < Tab<DT>::N1 / 4; j += NT) tz[j] = make_uint4(0, 0, 0, 0);
  }
  for (int j = tid; j < NW * HBINS; j += NT) (&sm.k.ghist[0][0])[j] = 0;
  for (int j = tid; j < NW * NSUM * NLIMB * 2; j += NT) (&sm.k.gsacc[0][0][0])[j] = 0;
  const int64_t lo = p.bounds[blockIdx.x], hi = p.bounds[blockIdx.x + 1];
  if (tid == 0) {
    sm.k.lo = lo;
    sm.k.glist = p.glist + (size_t)blockIdx.x * p.gcap;
    sm.k.gcap = p.gcap;
  }
  if (lane == 0) {
    for (int st = 0; st < NSTAGE; st++) mbar_init(smem_addr(&sm.k.bar[warp][st]), 1);
    mbar_init_fence();
  }
  Win W;
  W.rtol = p.rtol;
  W.atol = p.atol;
  W.lim = W.M1 = W.M2 = 0.0f;
  W.lb = W.fe = 0;
  Lane L;
  lane_init(L);
  if (p.nseg == 1 && p.n_total > 0 && warp == 0) {  // (counted here, off the tail of the last piece)
    const int b1 = cta_of_warp(p.n_total - 1, p), b0 = cta_of_warp(0, p);
    if (lane == 0) sm.k.first = b0, sm.k.final = b1;
  }
  __syncthreads();
  if (blockIdx.x == 0 && p.has_empty) write_empty_segments(p);
  uint32_t seq = 0;      // this warp's bulk-copy stage uses so far (stage = seq % NSTAGE)
  bool failed = false;   // a pipeline wait expired: skip the data, keep the barriers
  int64_t s = seg_of(lo, p.offsets, p.nseg);
  int64_t pb = lo;
  const char* gbase = reinterpret_cast<const char*>(p.g);
  const char* cbase = reinterpret_cast<const char*>(p.c);
  while (pb < hi) {
    while (p.offsets[s + 1] <= pb) s++;  // skip empty segments
    const int64_t pe = min(hi, p.offsets[s + 1]);
    // the body [vb, ve): on the aligned vector grid, with a head and a tail of
    // fewer than VEC elements; without a common grid (p0 < 0) the whole piece,
    // staged element by element
    const bool scalar = !(p.p0 >= 0 && p.p0 < p.n_total);
    int64_t vb = pe, ve = pe;
    if (!scalar) {
      int64_t a0 = pb <= p.p0 ? p.p0 : p.p0 + ((pb - p.p0 + VEC - 1) / VEC) * VEC;
      int64_t a1 = pe <= p.p0 ? p.p0 : p.p0 + ((pe - p.p0) / VEC) * VEC;
      if (a0 < a1) vb = a0, ve = a1;
    }
    const bool body_scalar = scalar || vb >= ve;  // also a piece inside one vector
    if (body_scalar) vb = pb, ve = pe;
    const int64_t nvec = (ve - vb + VEC - 1) / VEC;
    const int64_t nchunk = (nvec + CHV - 1) / CHV;
    // this warp's chunks: warp + NW i, i < nmy; only the piece's last chunk is partial
    const int nmy = nchunk > warp ? (int)((nchunk - warp + NW - 1) / NW) : 0;
    const uint32_t lastv = (uint32_t)(nvec - (nchunk - 1) * CHV);  // its vectors
    const int ilast = (int)((nchunk - 1) % NW) == warp ? nmy - 1 : -2;
    // start this warp's copies before anything else
    const char* gnext = gbase + (vb + warp * TILE) * Ty::BYTES;
    const char* cnext = cbase + (vb + warp * TILE) * Ty::BYTES;
    const uint32_t bar0 = smem_addr(&sm.k.bar[warp][0]);
    const uint32_t rg0 = smem_addr(&sm.ring.g[warp][0][0]), rc0 = smem_addr(&sm.ring.c[warp][0][0]);
    constexpr uint32_t STAGEB = CHV * 16u;
    auto issue = [&](uint32_t sq, int i) {  // chunk i, at gnext, into stage sq % NSTAGE, by one lane
      const uint32_t st = sq % NSTAGE;
      const uint32_t bytes = i == ilast ? lastv * 16u : STAGEB;
      if (elect_one()) {  // (the stage was only read since the last copy, or its writers fenced)
        mbar_expect_tx(bar0 + 8u * st, INJ ? bytes : 2 * bytes);
        bulk_load(rg0 + STAGEB * st, gnext, bytes, bar0 + 8u * st);
        if (!INJ) bulk_load(rc0 + STAGEB * st, cnext, bytes, bar0 + 8u * st);
      }
    };
    constexpr uint32_t STEP = (uint32_t)NW * STAGEB;  // bytes between a warp's chunks
    if (!failed && !body_scalar)
      for (int i = 0; i < NSTAGE && i < nmy; i++, gnext += STEP, cnext += STEP) issue(seq + (uint32_t)i, i);
    piece_init<DT>(sm);
    // the sample's loads and the piece's first pair
    uint32_t emax = 0, umax = 0, ab = 0, qb = 0;
    uint32_t G0 = 0, C0 = 0;
    if (tid == 0) {
      G0 = load_scalar<DT>(p.g, pb);
      C0 = cand_at<DT, INJ>(p, pb, G0);
    }
    if (!body_scalar) {
      const uint32_t sv = sample_at<DT>((uint32_t)nvec, tid);
      if (sv < (uint32_t)nvec) {
        const int64_t si = vb + (int64_t)sv * VEC;
        const uint4 gv = load_vec(p.g, si * Ty::BYTES);
        const uint4 cv = INJ ? inj_one<DT>(p, gv, si) : load_vec(p.c, si * Ty::BYTES);
        uint32_t ge[VEC], ce[VEC];
        unpack_vec<DT>(gv, ge);
        unpack_vec<DT>(cv, ce);
        sample_pairs<DT, VEC>(ge, ce, emax, umax, ab, qb);
      }
    } else if (const int64_t si = vb + sample_at<DT>((uint32_t)(ve - vb), tid); si < ve) {
      uint32_t ge[1], ce[1];
      ge[0] = load_scalar<DT>(p.g, si);
      ce[0] = cand_at<DT, INJ>(p, si, ge[0]);
      sample_pairs<DT, 1>(ge, ce, emax, umax, ab, qb);
    }
    emax = __reduce_max_sync(0xFFFFFFFFu, emax);
    umax = __reduce_max_sync(0xFFFFFFFFu, umax);
    ab = __reduce_max_sync(0xFFFFFFFFu, ab);
    qb = __reduce_max_sync(0xFFFFFFFFu, qb);
    __syncthreads();  // piece_init is visible
    if (lane == 0) {
      if (emax) atomicMax(&sm.k.lb, (int)emax);
      if (umax) atomicMax(&sm.k.ub, (int)(32 - __clz(umax)));
      if (ab) atomicMax(&sm.k.kabs, (unsigned long long)ab << 32);
      if (umax) atomicMax(&sm.k.kulp, (unsigned long long)umax << 32);
      if (qb) atomicMax(&sm.k.krel, (unsigned long long)qb << 32);
    }
    if (tid == 0) {
      constexpr long long NONE = 0x7FFFFFFFFFFFFFFFll;
      const bool fin = (G0 & Ty::MAG) < Ty::INF && (C0 & Ty::MAG) < Ty::INF;
      sm.k.ff = fin ? pb : NONE;
      sm.k.fu = fin ? pb : NONE;
    }
    __syncthreads();
    if constexpr (DT == PEAT_F32) {
      // the piece's initial window, the first entry of every warp's window log
      const int lb0 = window_floor<DT>(sm.k.lb, sm.k.ub);
      set_window_lb<DT>(W, lb0);
      if (lane == 0) {
        sm.k.nwin[warp] = 0;
        sm.k.wstart[warp][0] = 0;
        sm.k.wlb[warp][0] = lb0;
      }
      __syncwarp();
    } else {
      W.fe = window16<DT>(sm.k.lb & 255);
      if constexpr (DT == PEAT_F16) W.atol = __fmul_rn(p.atol, __uint_as_float((uint32_t)(127 + W.fe) << 23));
    }
    // Tiles: warp w takes chunks w, w + NW, ... of CHV vectors from its
    // staging ring (NSTAGE chunks in flight ahead of the one processed);
    // warp 0 also the head (i = -1, before its chunks) and the tail (after).
    uint32_t tli = (uint32_t)(vb - lo) + (uint32_t)warp * (uint32_t)TILE;
    Bounds B;
    auto run_cold = [&](uint4* gt, uint4* ct, uint32_t li, int i) {
      const ColdOut o = tile_cold<DT>(L, sm, gt, ct, li, W, i);
      L = o.L;
      if constexpr (DT == PEAT_F32) {
        if (o.lb != W.lb) set_window_lb<DT>(W, o.lb);
      }
      B.low = true;
    };
    if (warp == 0 && pb < vb) {
      stage_scalar<DT, INJ>(p, sm.k.edge_g, sm.k.edge_c, pb, vb);
      run_cold(sm.k.edge_g, sm.k.edge_c, (uint32_t)(pb - lo), -1);
    }
    B = read_bounds<DT>(sm, tli, W);
    int fail_i = -1;
    uint32_t fail_seq = 0;
    if (body_scalar) {
#pragma unroll 1
      for (int i = 0; i < nmy; i++, tli += (uint32_t)(NW * TILE)) {
        const int64_t e0 = vb + (warp + (int64_t)NW * i) * TILE;
        __syncwarp();
        stage_scalar<DT, INJ>(p, sm.ring.g[warp][0], sm.ring.c[warp][0], e0, min(ve, e0 + TILE));
        run_cold(sm.ring.g[warp][0], sm.ring.c[warp][0], tli, i);
        if constexpr (DT == PEAT_F32)
          if ((i & 8191) == 8191) flush_sums(L, sm, win_lexp<DT>(W));
      }
    } else if (!failed) {
#pragma unroll 1
      for (int i = 0; i < nmy; i++) {
        const uint32_t st = seq % NSTAGE;
        if (!mbar_test(bar0 + 8u * st, (seq / NSTAGE) & 1u) || p.wait_limit == 0) {
          if (!mbar_wait(bar0 + 8u * st, (seq / NSTAGE) & 1u, p.wait_limit)) {
            failed = true;  // chunks i .. i + NSTAGE - 1 may still be in flight
            fail_i = i;
            fail_seq = seq;
            if (lane == 0) atomicOr(p.status, 1u);
            break;
          }
        }
        uint4 *gt = sm.ring.g[warp][st], *ct = sm.ring.c[warp][st];
        if (!PEAT_CHECK((warp + (int64_t)NW * i) * CHV < nvec && vb - lo + (warp + (int64_t)NW * i) * TILE < ((int64_t)1 << 32)))
          break;
        if constexpr (INJ) {
          // the candidate tile, generated from the golden tile into the candidate ring
          inj_chunk<DT>(p, gt, ct, i == ilast ? (int)lastv : CHV, vb + (warp + (int64_t)NW * i) * TILE);
          __syncwarp();
        }
        if (i == ilast && lastv < (uint32_t)CHV) {  // a partial tile
          for (int v = lane; v < CHV; v += 32)
            if (v >= (int)lastv) gt[v] = ct[v] = make_uint4(0, 0, 0, 0);
          run_cold(gt, ct, tli, i);
        } else {
          if (B.low || (i & 3) == 0) B = read_bounds<DT>(sm, tli, W);
          if constexpr (DT == PEAT_F32) tile32(L, sm, gt, ct, tli, W, B, (uint32_t)i);
          else tile16<DT>(L, sm, gt, ct, tli, W, B);
        }
        __syncwarp();
        if (i + NSTAGE < nmy) {
          issue(seq + NSTAGE, i + NSTAGE);
          gnext += STEP;
          cnext += STEP;
        }
        seq++;
        tli += (uint32_t)(NW * TILE);
        // V1, V2 < 2^21 and 8 pairs per lane and chunk: the products stay below 2^59 between flushes
        if constexpr (DT == PEAT_F32)
          if ((i & 8191) == 8191) flush_sums(L, sm, win_lexp<DT>(W));
      }
    }
    if (warp == 0 && ve < pe) {
      stage_scalar<DT, INJ>(p, sm.k.edge_g, sm.k.edge_c, ve, pe);
      run_cold(sm.k.edge_g, sm.k.edge_c, (uint32_t)(ve - lo), nmy);
    }
    if (fail_i >= 0) {
      // copies this warp issued but never consumed: wait for them before the
      // staging memory is reused or the CTA exits
      for (int j = fail_i; j < nmy && j < fail_i + NSTAGE; j++) {
        const uint32_t sq = fail_seq + (uint32_t)(j - fail_i);
        mbar_wait(bar0 + 8u * (sq % NSTAGE), (sq / NSTAGE) & 1u, DRAIN_LIMIT);
      }
    }
    finish_piece<DT, INJ, false>(L, W, sm, p, s, pb, pe, vb, ve);
    pb = pe;
  }
}

// Stage 1 of a list of short segments, at most a pair per thread each: every pair
// on the general path, all warps of the CTA at a segment, without the window,
// copies and tables, which take 13 us a piece whatever it holds.  Measured (16 000
// segments of 100 and 4000 of 500 bfloat16 pairs): 1370 -> 831 us and 399 -> 255;
// with two pairs per thread there is no gain, with four it is a third slower.  A
// kernel of its own: the same choice inside compare_stage1 cost every 16-bit call
// 1.5 to 2 us.
template <int DT>
__global__ void __launch_bounds__(Geo<DT>::NT, Geo<DT>::CTAS) compare_short(CompareParams p) {
  constexpr int NT = Geo<DT>::NT, NW = Geo<DT>::NW;
  Smem<DT>& sm = *reinterpret_cast<Smem<DT>*>(smem_raw);
  pdl_trigger();
  const int tid = threadIdx.x;
  for (int b = tid; b < HBINS; b += NT) sm.k.hist[b] = 0;
  for (int j = tid; j < NSUM * NLIMB; j += NT) (&sm.k.sacc[0][0])[j] = 0;
  for (int j = tid; j < NW * HBINS; j += NT) (&sm.k.ghist[0][0])[j] = 0;
  for (int j = tid; j < NW * NSUM * NLIMB * 2; j += NT) (&sm.k.gsacc[0][0][0])[j] = 0;
  const int64_t lo = p.bounds[blockIdx.x], hi = p.bounds[blockIdx.x + 1];
  if (tid == 0) sm.k.lo = lo;
  Win W;
  W.rtol = p.rtol;
  W.atol = p.atol;
  W.lim = W.M1 = W.M2 = 0.0f;
  W.lb = W.fe = 0;
  Lane L;
  lane_init(L);
  __syncthreads();
  if (blockIdx.x == 0 && p.has_empty) write_empty_segments(p);
  int64_t s = seg_of(lo, p.offsets, p.nseg);
  for (int64_t pb = lo; pb < hi;) {
    while (p.offsets[s + 1] <= pb) s++;  // skip empty segments
    const int64_t pe = min(hi, p.offsets[s + 1]);
    piece_init<DT>(sm);
    if (tid == 0) {
      const uint32_t G = load_scalar<DT>(p.g, pb), C = load_scalar<DT>(p.c, pb);
      const bool fin = (G & Tr<DT>::MAG) < Tr<DT>::INF && (C & Tr<DT>::MAG) < Tr<DT>::INF;
      sm.k.ff = sm.k.fu = fin ? pb : 0x7FFFFFFFFFFFFFFFll;
    }
    finish_piece<DT, false, true>(L, W, sm, p, s, pb, pe, pe, pe);
    pb = pe;
  }
}

// ---------------------------------------------------------------------------
// stage 2: one CTA per segment: merge the maxima of the segment's pieces,
// round the exact sums once, write the outputs, clear the accumulator
// ---------------------------------------------------------------------------
// RN64 of the quotient (hi + lo) 2^sc / g > 0.  When hi + lo is a binary64
// number (always, unless lo is more than 29 binades below hi) the numerator
// is exact and one correctly rounded division gives the answer; otherwise the
// candidate with the smallest exact residual wins, ties to the even significand.
__device__ double rel_value(float hi, float lo, int sc, float g) {
  if (hi == 0.0f) return 0.0;
  if (g == 0.0f) return __longlong_as_double(0x7FF0000000000000ll);
  const double dh = hi, dl = lo;
  const double num = __dadd_rn(dh, dl);
  if (__dsub_rn(num, dh) == dl) return __ddiv_rn(sc ? num * 2.0 : num, (double)g);
  double q = __ddiv_rn(sc ? num * 2.0 : num, (double)g);  // within a few units of the exact quotient
  for (int i = 0; i < 3; i++) q = nextafter(q, 0.0);
  double best = q;
  XAcc bres;
  bool have = false;
  for (int step = 0; step < 7; step++, q = nextafter(q, __longlong_as_double(0x7FF0000000000000ll))) {
    XAcc r;
    r.zero();
    r.add_f(hi, false, sc);
    r.add_f(lo, false, sc);
    r.add_prod(q, (double)g, true);
    r.normalize();
    if (r.sign() < 0) r.negate();
    if (!have) {
      best = q, bres = r, have = true;
      continue;
    }
    int c = 0;
    for (int j = NLIMB - 1; j >= 0 && c == 0; j--)
      if (r.d[j] != bres.d[j]) c = r.d[j] > bres.d[j] ? 1 : -1;
    const bool qeven = (__double_as_longlong(q) & 1) == 0, beven = (__double_as_longlong(best) & 1) == 0;
    if (c < 0 || (c == 0 && qeven && !beven)) best = q, bres = r;
  }
  return best;
}


// Copy of a partial written by another CTA (read from L2, past this SM's L1).
__device__ __forceinline__ Partial load_partial(const Partial* src) {
  Partial x;
  const unsigned long long* w = reinterpret_cast<const unsigned long long*>(src);
  unsigned long long* d = reinterpret_cast<unsigned long long*>(&x);
#pragma unroll
  for (int k = 0; k < (int)(sizeof(Partial) / 8); k++) d[k] = __ldcg(w + k);
  return x;
}

// The whole CTA, once every piece of segment s (those of CTAs b0 .. b1) is in:
// merge the pieces' maxima, round the exact sums once, write the outputs and clear the
// accumulator for the next call.  Latency is all that matters here (one CTA,
// at the end of the call): the last step of the maxima and the rounding of
// the three sums run on warps of their own beside the mean and the variance.
template <int NT>
__device__ __noinline__ void finalize_segment(const CompareParams& p, int64_t s, int b0, int b1, FinScratch& f, MV& mv) {
  static_assert(NT >= HBINS && NT >= 128, "one bin per thread, four warps");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t s0 = p.offsets[s], s1 = p.offsets[s + 1];
  SegAcc* acc = p.acc + s;
  unsigned long long hv = 0;
  if (tid < HBINS) {
    hv = __ldcg(&acc->hist[tid]);
    acc->hist[tid] = 0;
  }
  const int j = NT > HBINS ? tid - HBINS : tid;  // with more threads than bins the others take the rest
  if (j >= 0 && j < NSUM * NLIMB) {
    f.limbs[j] = __ldcg(&acc->limbs[0][0] + j);
    (&acc->limbs[0][0])[j] = 0;
  } else if (j >= NSUM * NLIMB && j < NSUM * NLIMB + 8) {
    f.cnt[j - NSUM * NLIMB] = __ldcg(&acc->cnt[j - NSUM * NLIMB]);
    acc->cnt[j - NSUM * NLIMB] = 0;
  } else if (j == NSUM * NLIMB + 8) {
    acc->done = 0;
  }
  {
    Partial x;
    part_none(x);
#pragma unroll 1
    for (int b = b0 + tid; b <= b1; b += NT) part_merge(x, load_partial(p.partials + s + b));
    warp_best(x, &f.wbest[warp]);
  }
  __syncthreads();
  if (tid == 0) carry_to_digits(f.limbs + 1 * NLIMB, NLIMB, mv.A);   // S1 = sum |d|
  if (tid == 32) carry_to_digits(f.limbs + 2 * NLIMB, NLIMB, mv.B);  // S2 = sum d^2
  // the mean and variance of |d| over the finite pairs
  mean_var_block(mv, (uint64_t)(s1 - s0) - f.cnt[3], LIMB_LSB, [&] {
    if (warp == 2) {
      Partial x;
      if (lane < NT / 32) x = f.wbest[lane];
      else part_none(x);
      warp_best(x, &f.best);
      if (lane == 0) {
        const Partial& y = f.best;
        f.max_abs = y.abs_idx >= 0 ? __dadd_rn((double)y.abs_hi, (double)y.abs_lo) * (y.abs_sc ? 2.0 : 1.0) : 0.0;
        f.max_rel = y.rel_idx >= 0 ? rel_value(y.rel_hi, y.rel_lo, y.rel_sc, y.rel_g) : 0.0;
      }
    } else if (warp == 3 && lane < NSUM) {
      f.sums[lane] = limbs_to_double(f.limbs + lane * NLIMB);
    }
  });
  if (tid == 0) {
    const unsigned long long* cnt = f.cnt;
    const Partial& x = f.best;
    peat_stats_t r;
    const uint64_t n = (uint64_t)(s1 - s0);
    r.n = n;
    r.count[PEAT_EXACT] = cnt[0];
    r.count[PEAT_WITHIN_TOL] = cnt[2] + cnt[4];
    r.count[PEAT_MISMATCH] = (cnt[1] - cnt[2]) + cnt[5];
    r.count[PEAT_NAN_INF_ASYM] = cnt[6];
    r.count[PEAT_SIGN_FLIP] = cnt[7];
    r.n_finite = n - cnt[3];
    const int64_t first = x.first_fin >= 0 ? x.first_fin - s0 : -1;
    r.max_abs = f.max_abs;
    r.argmax_abs = x.abs_idx >= 0 ? x.abs_idx - s0 : first;
    r.max_rel = f.max_rel;
    r.argmax_rel = x.rel_idx >= 0 ? x.rel_idx - s0 : first;
    if (x.ulp_idx >= 0) {
      r.max_ulp = x.ulp;
      r.argmax_ulp = x.ulp_idx - s0;
    } else {
      r.max_ulp = 0;
      r.argmax_ulp = x.first_ulp >= 0 ? x.first_ulp - s0 : -1;
    }
    r.sum_signed = f.sums[0];
    r.sum_abs = f.sums[1];
    r.sum_sq = f.sums[2];
    r.rtol_eff = p.rtol;
    r.atol_eff = p.atol;
    r.mean_abs = mv.mean;
    r.var_abs = mv.var;
    if (p.status && (*reinterpret_cast<volatile unsigned int*>(p.status) & 1u))
      r.argmax_abs = r.argmax_rel = r.argmax_ulp = -2;  // a bounded wait expired: the outputs are invalid
    p.stats[s] = r;
  }
  if (p.hist && tid < HBINS) p.hist[s * HBINS + tid] = hv + ((tid == 0 || tid == 64) ? f.cnt[0] : 0ull);
  __syncthreads();
}

// Segments of a multi-segment call, one CTA each, after stage 1.  Four small
// CTAs per SM: a segment takes 7 us of latency whatever its threads (4000
// segments of 500 bfloat16 pairs: 436 us with 256 threads, 393 with 128).
constexpr int FIN_NT = 128;
__global__ void __launch_bounds__(FIN_NT) compare_finalize(CompareParams p) {
  __shared__ FinScratch f;
  __shared__ MV mv;
  pdl_wait();  // stage 1 complete
  const int64_t s0 = p.offsets[blockIdx.x], s1 = p.offsets[blockIdx.x + 1];
  if (s0 < s1) finalize_segment<FIN_NT>(p, blockIdx.x, cta_of_warp(s0, p), cta_of_warp(s1 - 1, p), f, mv);
}

// The outputs of every empty segment (no pairs): zero counts and sums, argmax -1.
__device__ __noinline__ void write_empty_segments(const CompareParams& p) {
  for (int64_t s = threadIdx.x; s < p.nseg; s += blockDim.x) {
    if (p.offsets[s] != p.offsets[s + 1]) continue;
    peat_stats_t r;
    memset(&r, 0, sizeof(r));
    r.argmax_abs = r.argmax_rel = r.argmax_ulp = -1;
    r.rtol_eff = p.rtol;
    r.atol_eff = p.atol;
    p.stats[s] = r;
    if (p.hist)
      for (int b = 0; b < HBINS; b++) p.hist[s * HBINS + b] = 0;
  }
}

template <int DT>
cudaError_t launch_t(const CompareParams& p, cudaStream_t st) {
  // NVTX ranges (host-side enqueue of each stage) for profilers; no cost without one attached
  nvtxRangePushA(p.inj_n > 0 ? "peat inject+compare stage 1" : "peat compare stage 1");
  if (p.shorts) compare_short<DT><<<p.nctas, Geo<DT>::NT, sizeof(Smem<DT>), st>>>(p);
  else if (p.inj_n > 0) compare_stage1<DT, true><<<p.nctas, Geo<DT>::NT, sizeof(Smem<DT>), st>>>(p);
  else compare_stage1<DT, false><<<p.nctas, Geo<DT>::NT, sizeof(Smem<DT>), st>>>(p);
  cudaError_t e = cudaGetLastError();
  nvtxRangePop();
  if (e == cudaSuccess && p.stage1_event) e = cudaEventRecord(static_cast<cudaEvent_t>(p.stage1_event), st);
  if (e != cudaSuccess || p.nseg <= 1) return e;
  nvtxRangePushA("peat compare stage 2 (per-segment finalize)");
  // a programmatic dependent of stage 1 (its launch overlaps the end of stage
  // 1), unless an event was recorded between the two
  if (p.stage1_event) {
    compare_finalize<<<(unsigned)p.nseg, FIN_NT, 0, st>>>(p);
    e = cudaGetLastError();
  } else {
    e = launch_dependent(compare_finalize, (unsigned)p.nseg, FIN_NT, 0, st, p);
  }
  nvtxRangePop();
  return e;
}

template <int DT>
__host__ __device__ int64_t bound_t(int64_t b, int nctas, int64_t n, int64_t p0) {
  if (b <= 0) return 0;
  if (b >= nctas) return n;
  constexpr int VEC = Tr<DT>::VEC;
  if (p0 < 0 || p0 >= n) return (n / nctas) * b + (n % nctas) * b / nctas;
  int64_t nv = (n - p0) / VEC;
  int64_t lo = p0 + ((nv / nctas) * b + (nv % nctas) * b / nctas) * VEC;
  return lo < n ? lo : n;
}

// offsets {0, n} and the CTA bounds of a one-tensor call, written on the
// device; a non-null status word is cleared for the compare that follows
template <int DT>
__global__ void compare_bounds(int64_t* offsets, int64_t* bounds, int nctas, int64_t n, int64_t p0,
                               unsigned int* status) {
  for (int b = threadIdx.x; b <= nctas; b += blockDim.x) bounds[b] = bound_t<DT>(b, nctas, n, p0);
  if (threadIdx.x == 0) {
    offsets[0] = 0;
    offsets[1] = n;
    if (status) *status = 0u;
  }
}

}  // namespace

cudaError_t launch_bounds_on_device(int dtype, int64_t* offsets, int64_t* bounds, int nctas, int64_t n, int64_t p0,
                                    unsigned int* status, cudaStream_t s) {
  switch (dtype) {
    case PEAT_F32: compare_bounds<PEAT_F32><<<1, BLOCK, 0, s>>>(offsets, bounds, nctas, n, p0, status); break;
    case PEAT_F16: compare_bounds<PEAT_F16><<<1, BLOCK, 0, s>>>(offsets, bounds, nctas, n, p0, status); break;
    case PEAT_BF16: compare_bounds<PEAT_BF16><<<1, BLOCK, 0, s>>>(offsets, bounds, nctas, n, p0, status); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_compare(int dtype, const CompareParams& p, cudaStream_t s) {
  switch (dtype) {
    case PEAT_F32: return launch_t<PEAT_F32>(p, s);
    case PEAT_F16: return launch_t<PEAT_F16>(p, s);
    case PEAT_BF16: return launch_t<PEAT_BF16>(p, s);
  }
  return cudaErrorInvalidValue;
}

int64_t compare_cta_bound(int dtype, int64_t b, int nctas, int64_t n, int64_t p0) {
  switch (dtype) {
    case PEAT_F32: return bound_t<PEAT_F32>(b, nctas, n, p0);
    case PEAT_F16: return bound_t<PEAT_F16>(b, nctas, n, p0);
    default: return bound_t<PEAT_BF16>(b, nctas, n, p0);
  }
}

// once per device, before the first launch
cudaError_t prepare_one(void (*kernel)(CompareParams), size_t smem) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)  // as much shared memory as the SM offers: Geo<DT>::CTAS CTAs of sizeof(Smem<DT>) each
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  return e;
}
template <int DT>
cudaError_t prepare_t() {
  cudaError_t e = prepare_one(compare_stage1<DT, false>, sizeof(Smem<DT>));
  if (e == cudaSuccess) e = prepare_one(compare_stage1<DT, true>, sizeof(Smem<DT>));
  return e == cudaSuccess ? prepare_one(compare_short<DT>, sizeof(Smem<DT>)) : e;
}

cudaError_t compare_prepare() {
  cudaError_t e = prepare_t<PEAT_F32>();
  if (e == cudaSuccess) e = prepare_t<PEAT_F16>();
  if (e == cudaSuccess) e = prepare_t<PEAT_BF16>();
  return e;
}

int compare_short_pairs(int dtype) { return dtype == PEAT_F32 ? Geo<PEAT_F32>::NT : Geo<PEAT_BF16>::NT; }
int compare_ctas_per_sm(int dtype) { return dtype == PEAT_F32 ? Geo<PEAT_F32>::CTAS : Geo<PEAT_BF16>::CTAS; }
size_t compare_partial_bytes() { return sizeof(Partial); }
size_t compare_segacc_bytes() { return sizeof(SegAcc); }

cudaError_t register_digit_status_compare(unsigned int* word) { return set_digit_status_here(word); }

// The index arithmetic of for_digits run on the host (a test of the digit
// split and of its range check; no GPU involved).
int test_for_digits(uint64_t m_lo, uint64_t m_hi, int e, int neg, int64_t* out) {
  for (int j = 0; j < NLIMB; j++) out[j] = 0;
  t_host_digit_dropped = false;
  for_digits(((unsigned __int128)m_hi << 64) | m_lo, e, neg != 0, [&](int j, int64_t v) { out[j] += v; });
  return t_host_digit_dropped ? 1 : 0;
}

// The binary64 rounding of the exact quotients behind the mean and the
// variance, run on the host (a test of quot_rn; no GPU involved).
double test_quot_rn(uint64_t w_hi, uint64_t w_lo, int sticky, int e, uint64_t d) {
  return quot_rn(((unsigned __int128)w_hi << 64) | w_lo, sticky != 0, e, d);
}

}  // namespace peat
