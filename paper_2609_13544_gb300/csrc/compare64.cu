// The error signature (Section IV-B-3, with the classes, ULP distances and
// histograms of the compare) for binary64 operands: the FP32-FP64 pairs of
// Fig. 5 once the float32 side is widened (exactly) to binary64.
//
// Most pairs (one sign, patterns less than 2^51 apart, zero atol) are finished
// in integer arithmetic on the patterns (fast64).  For the others d = c - g is
// an exact double-double (hi, lo) from Fast2Sum on the operands ordered by
// magnitude, held halved with a scale of one when the difference
// overflows binary64 (both operands are then large, so halving is exact).  Decisions that rounding could
// flip (the tolerance, the relative maximum) take a binary64 or float32 test
// with a margin first and otherwise the sign of an exact sum of integer
// terms; the relative bin comes from exponents and significands exactly; the
// three sums are added as 32-bit digits to a shared-memory superaccumulator
// per work item, merged per segment and rounded once.
#include <cstdint>

#include "exact64.cuh"
#include "meanvar.cuh"
#include "peat_internal.h"

namespace peat {
namespace {

constexpr int TB = 256;
using namespace x64;

// significand in [1, 2) as 52 fraction bits, and exponent, of a finite nonzero double
__device__ __forceinline__ void norm_d(double x, uint64_t& f, int& e) {
  uint64_t m;
  int ex;
  split_d(x, m, ex);
  const int lz = __clzll((long long)m) - 11;  // shift the leading one to bit 52
  f = (m << lz) & 0xFFFFFFFFFFFFFull;
  e = ex + 52 - lz;
}

// floor(log2(a / ag)) for a > 0, ag > 0, exactly
__device__ __forceinline__ int rel_log2_floor64(const Mag& a, double ag) {
  uint64_t fa, fg;
  int ea, eg;
  norm_d(a.hi, fa, ea);
  norm_d(ag, fg, eg);
  const int k0 = ea + a.sc - eg;
  if (fa != fg) return fa > fg ? k0 : k0 - 1;
  return neg64(a.lo) ? k0 - 1 : k0;  // hi = ag 2^k0 exactly: lo decides
}

// relative error records: a / g with kind 0 (a = 0), 1 (finite), 2 (g = 0 < a)
struct Rel {
  Mag a;
  double g;
  int kind;
  int le;    // log2 of the ratio, approximately (kind 1): le + lf, le exact,
  float lf;  // lf = log2 of the significands' ratio within 2^-20
};

__device__ __forceinline__ void approx_log2(const Mag& a, double g, int& le, float& lf) {
  uint64_t fa, fg;
  int ea, eg;
  norm_d(a.hi, fa, ea);
  norm_d(g, fg, eg);
  const float ra = __uint_as_float(0x3F800000u | (uint32_t)(fa >> 29));
  const float rg = __uint_as_float(0x3F800000u | (uint32_t)(fg >> 29));
  le = ea + a.sc - eg;
  lf = __log2f(__fdividef(ra, rg));
}

// log2(x) - log2(y) of two finite ratios, within 2^-18 (clamped far from zero)
__device__ __forceinline__ float lg_diff(int xe, float xf, int ye, float yf) {
  const int de = xe - ye;
  if (de > 4) return 8.0f;
  if (de < -4) return -8.0f;
  return (float)de + (xf - yf);
}

// x > y exactly
__device__ bool rel_gt(const Rel& x, const Rel& y) {
  if (x.kind != y.kind) return x.kind > y.kind;
  if (x.kind != 1) return false;
  if (x.a.lo == 0.0 && y.a.lo == 0.0 && x.a.sc == 0 && y.a.sc == 0) {
    // single binary64 magnitudes: the cross products of the 53-bit
    // significands (106 bits, leading bit 104 or 105), aligned
    uint64_t xa, xg, ya, yg;
    int exa, exg, eya, eyg;
    norm_d(x.a.hi, xa, exa);
    norm_d(x.g, xg, exg);
    norm_d(y.a.hi, ya, eya);
    norm_d(y.g, yg, eyg);
    const uint64_t ONE = 1ull << 52;
    const u128 l = (u128)(xa | ONE) * (yg | ONE), r = (u128)(ya | ONE) * (xg | ONE);
    const int dl = (exa + eyg) - (eya + exg);
    if (dl > 2 || dl < -2) return dl > 0;
    return dl >= 0 ? (l << dl) > r : l > (r << -dl);
  }
  XTerm t[4] = {prod_term(x.a.hi, y.g, x.a.sc, false), prod_term(fabs(x.a.lo), y.g, x.a.sc, x.a.lo < 0.0),
                prod_term(y.a.hi, x.g, y.a.sc, true), prod_term(fabs(y.a.lo), x.g, y.a.sc, y.a.lo >= 0.0)};
  return xsign(t, 4) > 0;
}

// ---------------------------------------------------------------------------
// the per-item superaccumulator: 32-bit digits in signed 64-bit limbs

constexpr int SLSB = XLSB, SL = XL;
static_assert(SL == P64_LIMBS, "record limbs");

__device__ __forceinline__ void sacc_add(long long* acc, u128 m, int e, bool neg) {
  if (m == 0) return;
  const int p = e - SLSB;
  const int limb = p >> 5, sh = p & 31;
  const u128 lo = m << sh;
  const unsigned long long hi = sh ? (unsigned long long)(m >> (128 - sh)) : 0ull;
#pragma unroll
  for (int q = 0; q < 5; q++) {
    const unsigned long long dig = q < 4 ? (unsigned long long)(lo >> (32 * q)) & 0xFFFFFFFFull : hi & 0xFFFFFFFFull;
    if (dig) atomicAdd(reinterpret_cast<unsigned long long*>(acc + limb + q),
                       neg ? (unsigned long long)(-(long long)dig) : dig);
  }
}

// Per-thread windows in front of the superaccumulator: a term whose exponent
// lies within a fixed distance of the thread's first one is added to a
// register integer (signed 128 bits for sum d and sum |d|, 53-bit terms
// shifted by at most 56; unsigned 192 bits for sum d^2, 106-bit terms shifted
// by at most 70; at most 2^14 terms per thread and item, so neither
// overflows), any other term goes to the shared digits.  Flushed at the end
// of each item.
using i128 = __int128;

__device__ __forceinline__ void win_add(i128& acc, int& base, uint64_t m, int e, bool neg, long long* S) {
  if (m == 0) return;
  if (base == INT32_MIN) base = e - 28;
  const int sh = e - base;
  if (sh >= 0 && sh <= 56) {
    const i128 v = (i128)((u128)m << sh);
    acc += neg ? -v : v;
  } else {
    sacc_add(S, (u128)m, e, neg);
  }
}
__device__ __forceinline__ void win_flush(i128 acc, int base, long long* S) {
  if (acc == 0) return;
  const bool neg = acc < 0;
  sacc_add(S, neg ? (u128)(-acc) : (u128)acc, base, neg);
}

struct W192 {
  unsigned long long w0, w1, w2;
  int base;
};
__device__ __forceinline__ void win3_add(W192& a, u128 m, int e, long long* S) {
  if (m == 0) return;
  if (a.base == INT32_MIN) a.base = e - 35;
  const int sh = e - a.base;
  if (sh < 0 || sh > 70) {
    sacc_add(S, m, e, false);
    return;
  }
  const unsigned long long m0 = (unsigned long long)m, m1 = (unsigned long long)(m >> 64);
  unsigned long long v0, v1, v2;
  if (sh == 0) {
    v0 = m0, v1 = m1, v2 = 0;
  } else if (sh < 64) {
    v0 = m0 << sh, v1 = (m1 << sh) | (m0 >> (64 - sh)), v2 = m1 >> (64 - sh);
  } else {
    const int t = sh - 64;
    v0 = 0, v1 = m0 << t, v2 = (m1 << t) | (t ? m0 >> (64 - t) : 0ull);
  }
  a.w0 += v0;
  const unsigned long long c0 = a.w0 < v0 ? 1ull : 0ull;
  const unsigned long long s1 = a.w1 + v1;
  const unsigned long long c1 = (s1 < v1 ? 1ull : 0ull);
  a.w1 = s1 + c0;
  a.w2 += v2 + c1 + (a.w1 < c0 ? 1ull : 0ull);
}
__device__ __forceinline__ void win3_flush(const W192& a, long long* S) {
  // as two parts of at most 96 + 96 bits
  const u128 lo = ((u128)(a.w1 & 0xFFFFFFFFull) << 64) | a.w0;
  const u128 hi = ((u128)a.w2 << 32) | (a.w1 >> 32);
  if (lo) sacc_add(S, lo, a.base, false);
  if (hi) sacc_add(S, hi, a.base + 96, false);
}

// ---------------------------------------------------------------------------
// per-thread totals within one work item (offsets: position in the item + 1, 0 = none)

struct Acc64 {
  uint32_t cnt[PEAT_NCLASS], nfin;
  i128 sd, sa;   // windows of sum d and sum |d|
  int bd, ba;
  W192 sq;       // window of sum d^2
  Mag ma;
  uint32_t ia;
  Rel mr;
  uint32_t ir;
  unsigned long long mu;
  uint32_t iu;
};

__device__ __forceinline__ void acc64_init(Acc64& t) {
#pragma unroll
  for (int k = 0; k < PEAT_NCLASS; k++) t.cnt[k] = 0;
  t.nfin = 0;
  t.sd = t.sa = 0;
  t.bd = t.ba = INT32_MIN;
  t.sq = W192{0ull, 0ull, 0ull, INT32_MIN};
  t.ma = Mag{0.0, 0.0, 0};
  t.ia = 0;
  t.mr = Rel{Mag{0.0, 0.0, 0}, 1.0, 0, 0, 0.0f};
  t.ir = 0;
  t.mu = 0;
  t.iu = 0;
}

__device__ __forceinline__ void hist_add(unsigned* H, int bin) {
  const unsigned grp = __match_any_sync(0xFFFFFFFFu, bin);
  if (bin >= 0 && (int)(threadIdx.x & 31) == __ffs(grp) - 1) atomicAdd(H + bin, (unsigned)__popc(grp));
}

// one pair slot of the warp (every lane calls it; ok: this lane holds the pair at item offset off)
__device__ __forceinline__ void pair64(const Cmp64Params& p, Acc64& t, unsigned* H, long long* S, uint64_t G,
                                       uint64_t C, bool ok, uint32_t off) {
  int relbin = -1, ulpbin = -1, cls = -1;
  if (ok) {
    const uint64_t mg = G & 0x7FFFFFFFFFFFFFFFull, mc = C & 0x7FFFFFFFFFFFFFFFull;
    const bool sg = (G >> 63) != 0, sc = (C >> 63) != 0;
    const uint64_t INF = 0x7FF0000000000000ull;
    const bool gnan = mg > INF, cnan = mc > INF, gfin = mg < INF, cfin = mc < INF;
    const long long kg = sg ? -(long long)mg : (long long)mg, kc = sc ? -(long long)mc : (long long)mc;
    const unsigned long long u = kc >= kg ? (unsigned long long)kc - (unsigned long long)kg
                                          : (unsigned long long)kg - (unsigned long long)kc;
    if (!gfin || !cfin) {
      const bool eq = (gnan && cnan) || (mg == INF && mc == INF && sg == sc);
      cls = eq ? PEAT_EXACT : PEAT_NAN_INF_ASYM;
      relbin = eq ? 0 : 63;
    } else {
      const double gd = from_bits64(G), cd = from_bits64(C);
      bool dneg;
      const Mag a = diff64(gd, cd, dneg);
      const double ag = from_bits64(mg);  // |g|
      const bool azero = bits64(a.hi) == 0;
      t.nfin++;
      // sums: d = +-(hi + lo) 2^sc, |d|, d^2 = (hi^2 + 2 hi lo + lo^2) 4^sc
      {
        uint64_t mh, ml;
        int eh, el;
        split_d(a.hi, mh, eh);
        split_d(a.lo, ml, el);  // split_d takes the magnitude
        const bool lneg = (bits64(a.lo) >> 63) != 0;
        win_add(t.sd, t.bd, mh, eh + a.sc, dneg, S);
        win_add(t.sa, t.ba, mh, eh + a.sc, false, S + SL);
        win3_add(t.sq, (u128)mh * mh, 2 * (eh + a.sc), S + 2 * SL);
        if (ml) {
          win_add(t.sd, t.bd, ml, el + a.sc, dneg != lneg, S);
          win_add(t.sa, t.ba, ml, el + a.sc, lneg, S + SL);
          if (lneg) sacc_add(S + 2 * SL, (u128)mh * ml, eh + el + 2 * a.sc + 1, true);  // rare: straight to digits
          else win3_add(t.sq, (u128)mh * ml, eh + el + 2 * a.sc + 1, S + 2 * SL);
          win3_add(t.sq, (u128)ml * ml, 2 * (el + a.sc), S + 2 * SL);
        }
      }
      if (t.ia == 0 || mag_gt(a, t.ma)) t.ma = a, t.ia = off + 1;
      // relative maximum: an approximate log2 rules out all but the candidates
      Rel r;
      r.a = a;
      r.g = ag;
      r.kind = azero ? 0 : (mg == 0 ? 2 : 1);
      r.le = 0;
      r.lf = 0.0f;
      if (r.kind == 1) approx_log2(a, ag, r.le, r.lf);
      const bool maybe = t.ir == 0 || r.kind > t.mr.kind ||
                         (r.kind == 1 && t.mr.kind == 1 && lg_diff(r.le, r.lf, t.mr.le, t.mr.lf) >= -0x1p-16f);
      if (maybe && (t.ir == 0 || rel_gt(r, t.mr))) t.mr = r, t.ir = off + 1;
      if (azero) {
        cls = PEAT_EXACT;
        relbin = 0;
      } else {
        if (within64(a, ag, p.rtol, p.atol)) cls = PEAT_WITHIN_TOL;
        else if (mg != 0 && mc != 0 && sg != sc) cls = PEAT_SIGN_FLIP;
        else cls = PEAT_MISMATCH;
        if (mg == 0) {
          relbin = 63;
        } else {
          const int k = rel_log2_floor64(a, ag) + 48;
          relbin = k < 1 ? 1 : (k > 62 ? 62 : k);
        }
      }
    }
    if (gnan || cnan) {
      ulpbin = (gnan && cnan) ? 0 : 63;
    } else {
      ulpbin = (int)(u < 63 ? u : 63);
      if (t.iu == 0 || u > t.mu) t.mu = u, t.iu = off + 1;
    }
  }
#pragma unroll
  for (int k = 0; k < PEAT_NCLASS; k++) t.cnt[k] += cls == k;
  hist_add(H, relbin);
  hist_add(H, ulpbin < 0 ? -1 : 64 + ulpbin);
}

// (out of line: the pairs that the integer path leaves)
__device__ __noinline__ void pair64_slow(const Cmp64Params& p, Acc64& t, unsigned* H, long long* S, uint64_t G, uint64_t C,
                                         bool ok, uint32_t off) {
  pair64(p, t, H, S, G, C, ok, off);
}

// x better than y: larger, or equal at a lower index (-1: absent, worst)
__device__ __forceinline__ bool better_mag(const Mag& x, long long ix, const Mag& y, long long iy) {
  if (ix < 0) return false;
  if (iy < 0) return true;
  return mag_gt(x, y) || (!mag_gt(y, x) && ix < iy);
}
__device__ __forceinline__ bool better_rel(const Rel& x, long long ix, const Rel& y, long long iy) {
  if (ix < 0) return false;
  if (iy < 0) return true;
  if (x.kind == 1 && y.kind == 1) {  // far apart: the approximations decide
    const float dl = lg_diff(x.le, x.lf, y.le, y.lf);
    if (fabsf(dl) > 0x1p-16f) return dl > 0.0f;
  }
  return rel_gt(x, y) || (!rel_gt(y, x) && ix < iy);
}
__device__ __forceinline__ bool better_u(unsigned long long x, long long ix, unsigned long long y, long long iy) {
  if (ix < 0) return false;
  if (iy < 0) return true;
  return x > y || (x == y && ix < iy);
}

// merge record o into r (both within one segment)
__device__ void rec_merge(Part64Rec& r, const Part64Rec& o) {
  for (int k = 0; k < PEAT_NCLASS; k++) r.cnt[k] += o.cnt[k];
  r.nfin += o.nfin;
  const Mag ra{r.ahi, r.alo, r.asc}, oa{o.ahi, o.alo, o.asc};
  if (better_mag(oa, o.ia, ra, r.ia)) r.ahi = o.ahi, r.alo = o.alo, r.asc = o.asc, r.ia = o.ia;
  const Rel rr{Mag{r.rhi, r.rlo, r.rsc}, r.rg, r.rkind, r.rle, r.rlf};
  const Rel orr{Mag{o.rhi, o.rlo, o.rsc}, o.rg, o.rkind, o.rle, o.rlf};
  if (better_rel(orr, o.ir, rr, r.ir))
    r.rhi = o.rhi, r.rlo = o.rlo, r.rsc = o.rsc, r.rg = o.rg, r.rkind = o.rkind, r.rle = o.rle, r.rlf = o.rlf,
    r.ir = o.ir;
  if (better_u(o.mu, o.iu, r.mu, r.iu)) r.mu = o.mu, r.iu = o.iu;
}

__device__ __forceinline__ void rec_from_acc(Part64Rec& r, const Acc64& a, long long ib) {
  for (int k = 0; k < PEAT_NCLASS; k++) r.cnt[k] = a.cnt[k];
  r.nfin = a.nfin;
  r.ahi = a.ma.hi, r.alo = a.ma.lo, r.asc = a.ma.sc, r.ia = a.ia ? ib + a.ia - 1 : -1;
  r.rhi = a.mr.a.hi, r.rlo = a.mr.a.lo, r.rsc = a.mr.a.sc, r.rg = a.mr.g, r.rkind = a.mr.kind, r.rle = a.mr.le, r.rlf = a.mr.lf;
  r.ir = a.ir ? ib + a.ir - 1 : -1;
  r.mu = a.mu, r.iu = a.iu ? ib + a.iu - 1 : -1;
}

// the CTA's records merged into thread 0's (every thread calls it; buf holds
// half of them)
__device__ void block_merge(Part64Rec& r, Part64Rec* buf) {
  for (int w = TB / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x >= w && (int)threadIdx.x < 2 * w) buf[threadIdx.x - w] = r;
    __syncthreads();
    if ((int)threadIdx.x < w) rec_merge(r, buf[threadIdx.x]);
    __syncthreads();
  }
}

__device__ __forceinline__ uint64_t wsum_u64(uint64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// The integer path.  A window pair has patterns less than 2^51 apart (so one
// sign, exponents at most one apart, c - g exact): with el the smaller
// exponent field, |d| = a 2^(el - 1075) for the integer a = |C - G|, plus the
// larger operand's fraction field when the exponents differ (its steps are
// two units).  With s = el - base in [0, WS]:
//   - sum |d| and the sum of the negative ones: a << s in 128-bit registers;
//   - sum d^2: a * a shifted by 2 s, added as 32-bit digits to the thread's own
//     64-bit counters in shared memory;
//   - the two bins from shared counters by (floor(log2(|d| / |g|)) mod 64,
//     min(ULP distance, 63)) (increments by one merge equal addresses; column
//     0 takes the lanes without an unequal pair and is left out);
//   - the tolerance (atol = 0; with another atol every unequal pair goes to
//     pair64) and the relative maximum from the ratio in float32, within 2^-21:
//     closer calls take the slow path.
// A pair outside the window, non-finite, or above one of the warp's maxima so
// far goes to pair64.  The warp's iterations visit its pairs in index order, so a
// pair equal to a maximum of an earlier round cannot win.
//
// What bounds it: integer instruction issue (no FP64 instruction, whose pipe
// takes 64 cycles per warp here, and no local memory): about 250 instructions
// per pair slot of a warp.  12.3 M pairs (a float32 rounding widened, rtol
// 1e-7), one call: 2200 -> 207 us, of which the finalization 32 (atol 1e-8: 2210 -> 870);
// before, every
// term went through binary64 Fast2Sum and local-memory windows (1070
// instructions and 1.9 GB of local-memory traffic).
constexpr int WS = 56, QD = 8;

struct CtaBounds {  // the largest of the warps' bounds
  unsigned long long kabs, ku;
  unsigned rb;
};
struct Fast64 {
  u128 s1, n1;         // sum |d|, sum of |d| over negative d, in units of 2^(base - 1075)
  uint32_t mism;       // pairs above the tolerance
  int base;            // -1: not placed yet (no unequal finite pair seen)
  uint32_t miss;       // pairs of small distance outside the window since it was placed
  // the warp's bounds: a pair above one of them takes the slow path.  Its own
  // maxima, and the CTA's less one step (a pair of another warp may have the
  // same value at a higher index).
  uint64_t kabs, ku;   // |d| as a key (exponent, significand), ULP distance
  float rb;            // ratio, lowered by 2^-19
  // maxima seen in this round, bounds from the next one on (a lane's second
  // pair precedes the next lane's first)
  uint64_t pk, pu;
  uint32_t nslow;      // pairs given to pair64 (the whole warp's)
};

// The integer path's sums into the item's digits (the whole warp calls it):
// words summed over the warp, then added by one lane.
// By value, so that the caller's state stays in registers.
__device__ __noinline__ void fast_flush(int base, u128 s1, u128 n1, long long* S, unsigned long long* Q) {
  const int lane = threadIdx.x & 31;
  const int u = base - 1075;
#pragma unroll 1
  for (int w = 0; w < 4; w++) {
    const uint64_t a1 = wsum_u64((uint32_t)(s1 >> (32 * w))), an = wsum_u64((uint32_t)(n1 >> (32 * w)));
    if (lane == 0) {
      sacc_add(S + SL, a1, u + 32 * w, false);
      sacc_add(S, a1, u + 32 * w, false);  // sum d = sum |d| - 2 sum of the negative ones
      sacc_add(S, (u128)an << 1, u + 32 * w, true);
    }
  }
#pragma unroll 1
  for (int w = 0; w < QD; w++) {
    const uint64_t qs = wsum_u64(Q[w * TB]);
    Q[w * TB] = 0ull;
    if (lane == 0) sacc_add(S + 2 * SL, qs, 2 * u + 32 * w, false);
  }
}

// one pair slot of the warp (every lane calls it; a lane without a pair passes equal zeros and ok = false)
__device__ __forceinline__ void fast64(const Cmp64Params& p, Fast64& f, Acc64& acc, unsigned* H, long long* S,
                                       uint32_t t2, unsigned long long* Q, CtaBounds* cb, uint64_t G, uint64_t C,
                                       bool ok, uint32_t off, float rlo, float rhi) {
  constexpr uint64_t FRAC = 0xFFFFFFFFFFFFFull;
  const int64_t U = (int64_t)(C - G);
  const uint64_t au = U < 0 ? (uint64_t)-U : (uint64_t)U;
  const bool nz = au != 0;
  const uint64_t mx = (U > 0 ? C : G) & MAG64, mn = (U > 0 ? G : C) & MAG64;
  const uint32_t eu = (uint32_t)(mx >> 52), el = (uint32_t)(mn >> 52);
  const uint64_t a0 = au + (eu != el ? mx & FRAC : 0ull);
  if (f.base < 0) {  // (warp-uniform) place the window by the first unequal pairs
    const uint32_t em = __reduce_max_sync(0xFFFFFFFFu, nz && el < 0x7FFu ? el : 0u);
    if (em) f.base = max((int)em - 40, 64);
  }
  const int s0 = (int)el - f.base;
  const bool win = nz && au < (1ull << 51) && (unsigned)s0 <= (unsigned)WS && el < 0x7FFu && eu < 0x7FFu && f.base >= 0 && p.atol == 0.0;
  bool exc = nz ? !win : (ok && el == 0x7FFu);
  // |d| normalised: a << lz has its leading one at bit 63
  const int lz = __clzll((long long)(a0 | 1ull));
  const uint64_t am = a0 << lz;
  const int ea = (int)el + 63 - lz;  // |d| = (am / 2^63) 2^(ea - 1075)
  const int eg = (int)((uint32_t)(G >> 52) & 0x7FFu);
  const uint64_t gn = (((G & FRAC) | (1ull << 52)) << 11);
  const int dk = ea - eg - 52;
  const int k = dk - (am < gn ? 1 : 0);
  const uint64_t key = ((uint64_t)(uint32_t)ea << 52) + ((am << 1) >> 12);
  const float fa = __uint_as_float(0x3F800000u | ((uint32_t)(am >> 40) & 0x7FFFFFu));
  const float fg = __uint_as_float(0x3F800000u | ((uint32_t)(G >> 29) & 0x7FFFFFu));
  float rc;
  asm("rcp.approx.f32 %0, %1;" : "=f"(rc) : "f"(fg));
  const float rf = __uint_as_float(__float_as_uint(fa * rc) + ((uint32_t)dk << 23));
  exc = exc || (win && (key > f.kabs || au > f.ku || rf >= f.rb || (rf > rlo && rf < rhi)));
  const bool use = win && !exc;
  const uint64_t a = use ? a0 : 0ull;
  const int s = use ? s0 : 0;
  f.mism += use && rf >= rhi ? 1u : 0u;
  const uint32_t uc = use ? (uint32_t)(au < 63 ? au : 63) : 0u;
  asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(t2 + ((((uint32_t)k & 63u) << 6) | uc) * 4u));
  const uint64_t vlo = a << s, vhi = (a >> 1) >> (63 - s);
  const u128 v = ((u128)vhi << 64) | vlo;
  f.s1 += v;
  const bool neg = (U < 0) != ((int64_t)G < 0);
  f.n1 += neg ? v : (u128)0;
  {
    const uint32_t alo = (uint32_t)a, ahi = (uint32_t)(a >> 32);
    const uint32_t w = (uint32_t)(2 * s) >> 5, b = (uint32_t)(2 * s) & 31u;
    unsigned long long* q = Q + w * TB;
    if (!__any_sync(0xFFFFFFFFu, ahi != 0u)) {  // a < 2^32: three digits
      const uint64_t pp = (uint64_t)alo * alo;
      const uint32_t p0 = (uint32_t)pp, p1 = (uint32_t)(pp >> 32);
      q[0] += p0 << b;
      q[TB] += __funnelshift_l(p0, p1, b);
      q[2 * TB] += __funnelshift_l(p1, 0u, b);
    } else {
      const u128 pp = (u128)a * a;
      const uint32_t p0 = (uint32_t)pp, p1 = (uint32_t)(pp >> 32), p2 = (uint32_t)(pp >> 64), p3 = (uint32_t)(pp >> 96);
      q[0] += p0 << b;
      q[TB] += __funnelshift_l(p0, p1, b);
      q[2 * TB] += __funnelshift_l(p1, p2, b);
      q[3 * TB] += __funnelshift_l(p2, p3, b);
      q[4 * TB] += __funnelshift_l(p3, 0u, b);
    }
  }
  const unsigned who = __ballot_sync(0xFFFFFFFFu, exc);
  if (who) {
    pair64_slow(p, acc, H, S, G, C, exc, off);
    f.nslow += (uint32_t)__popc(who);
    // too many pairs outside the window: place it again by the next unequal ones
    f.miss += (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, exc && !win && au < (1ull << 51) && f.base >= 0 && p.atol == 0.0));
    if (f.miss >= 256u) {
      fast_flush(f.base, f.s1, f.n1, S, Q);
      f.s1 = f.n1 = 0;
      f.base = -1;
      f.miss = 0;
    }
    // the warp's bounds (only window pairs raise them)
    const bool up = exc && win;
    const uint32_t kh = __reduce_max_sync(0xFFFFFFFFu, up ? (uint32_t)(key >> 32) : 0u);
    const uint32_t kl = __reduce_max_sync(0xFFFFFFFFu, up && (uint32_t)(key >> 32) == kh ? (uint32_t)key : 0u);
    const uint32_t uh = __reduce_max_sync(0xFFFFFFFFu, up ? (uint32_t)(au >> 32) : 0u);
    const uint32_t ul = __reduce_max_sync(0xFFFFFFFFu, up && (uint32_t)(au >> 32) == uh ? (uint32_t)au : 0u);
    const float rm = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, up ? __float_as_uint(rf) : 0u));
    f.pk = max(f.pk, ((uint64_t)kh << 32) | kl);
    f.pu = max(f.pu, ((uint64_t)uh << 32) | ul);
    f.rb = fmaxf(f.rb, rm * 0.999998f);
    if ((threadIdx.x & 31) == 0) {
      atomicMax(&cb->kabs, (unsigned long long)f.pk);
      atomicMax(&cb->ku, (unsigned long long)f.pu);
      atomicMax(&cb->rb, __float_as_uint(f.rb));
    }
  }
}

__global__ void __launch_bounds__(TB, 2) compare64_stage1(Cmp64Params p) {
  __shared__ unsigned H[PEAT_HIST_BINS];
  __shared__ long long S[3 * SL];
  __shared__ unsigned long long tot[2];  // window pairs, of them above the tolerance; pairs given to pair64
  __shared__ unsigned long long nsl;
  __shared__ unsigned first;  // offset of the item's first equal finite pair (searched when it matters)
  __shared__ int need;
  __shared__ CtaBounds cb;
  union Scratch {
    struct {
      uint32_t t2[64 * 64];
      unsigned long long q[QD][TB];
    } w;
    Part64Rec buf[TB / 2];
  };
  __shared__ Scratch sc;
  pdl_trigger();  // the finalize kernel may start launching (it waits for this grid)
  const int lane = threadIdx.x & 31;
  const uint32_t t2 = (uint32_t)__cvta_generic_to_shared(sc.w.t2);
  // the tolerance on the float32 ratio: closer than 2^-18 to rtol takes the exact test
  const float rt = (float)p.rtol, rlo = rt * 0.999996f, rhi = rt * 1.000004f;
  Fast64 f;
  long long prev = -1;
  for (long long item = blockIdx.x; item < p.nitems; item += gridDim.x) {
    const long long b = p.item_b[item], e = p.item_e[item], seg = p.item_seg[item];
    const long long base = p.offsets[seg];
    for (int k = threadIdx.x; k < PEAT_HIST_BINS; k += TB) H[k] = 0u;
    for (int k = threadIdx.x; k < 3 * SL; k += TB) S[k] = 0;
    for (int k = threadIdx.x; k < 64 * 64; k += TB) sc.w.t2[k] = 0u;
#pragma unroll
    for (int k = 0; k < QD; k++) sc.w.q[k][threadIdx.x] = 0ull;
    if (threadIdx.x < 2) tot[threadIdx.x] = 0ull;
    if (threadIdx.x == 2) nsl = 0ull;
    if (threadIdx.x == 3 && seg != prev) cb.kabs = cb.ku = 0ull, cb.rb = 0u;
    __syncthreads();
    Acc64 acc;
    acc64_init(acc);
    f.s1 = f.n1 = 0;
    f.mism = f.nslow = f.miss = 0;
    f.base = -1;
    // bounds carry over within a segment: its items come in index order
    if (seg != prev) {
      f.kabs = f.ku = f.pk = f.pu = 0ull;
      f.rb = 0.0f;
      prev = seg;
    }
    // pairs of elements (one 16-byte vector of each tensor) on the absolute
    // index grid, the next ones loaded while these are processed
    // (offsets in the item are 32-bit: it has at most 2^22 elements)
    const int len = (int)(e - b), o0 = -(int)(b & 1);  // vector v holds the item's offsets o0 + 2 v, o0 + 2 v + 1
    const int nq = (len - o0 + 1) >> 1;
    const char* gp = reinterpret_cast<const char*>(p.g) + (b + o0) * 8;
    const char* cp = reinterpret_cast<const char*>(p.c) + (b + o0) * 8;
    auto load = [&](int v, ulonglong2& gv, ulonglong2& cv) {
      gv = cv = make_ulonglong2(0ull, 0ull);
      const int o = o0 + 2 * v;
      if (p.vec && o >= 0 && o + 2 <= len) {
        gv = __ldg(reinterpret_cast<const ulonglong2*>(gp) + v);
        cv = __ldg(reinterpret_cast<const ulonglong2*>(cp) + v);
      } else {
        const unsigned long long* gq = reinterpret_cast<const unsigned long long*>(gp) + 2 * v;
        const unsigned long long* cq = reinterpret_cast<const unsigned long long*>(cp) + 2 * v;
        if (o >= 0 && o < len) gv.x = __ldg(gq), cv.x = __ldg(cq);
        if (o + 1 < len) gv.y = __ldg(gq + 1), cv.y = __ldg(cq + 1);
      }
    };
    ulonglong2 gn, cn;
    int v = threadIdx.x;
    load(v, gn, cn);
    // whole warps in every round
    for (int r = threadIdx.x & ~31; r < nq; r += TB, v += TB) {
      const ulonglong2 gc = gn, cc = cn;
      load(v + TB, gn, cn);
      const int o = o0 + 2 * v;
      {
        const volatile CtaBounds* vb = &cb;
        const uint64_t ka = (uint64_t)vb->kabs, ku = (uint64_t)vb->ku;
        f.kabs = max(max(f.kabs, f.pk), ka - (ka ? 1 : 0));
        f.ku = max(max(f.ku, f.pu), ku - (ku ? 1 : 0));
        f.rb = fmaxf(f.rb, __uint_as_float(vb->rb));
      }
      fast64(p, f, acc, H, S, t2, &sc.w.q[0][threadIdx.x], &cb, gc.x, cc.x, o >= 0 && o < len, (uint32_t)o, rlo, rhi);
      fast64(p, f, acc, H, S, t2, &sc.w.q[0][threadIdx.x], &cb, gc.y, cc.y, o + 1 < len, (uint32_t)(o + 1), rlo, rhi);
    }
    win_flush(acc.sd, acc.bd, S);
    win_flush(acc.sa, acc.ba, S + SL);
    win3_flush(acc.sq, S + 2 * SL);
    if (f.base >= 0) fast_flush(f.base, f.s1, f.n1, S, &sc.w.q[0][threadIdx.x]);
    const uint32_t mism = __reduce_add_sync(0xFFFFFFFFu, f.mism);
    if (lane == 0) {
      if (mism) atomicAdd(&tot[1], (unsigned long long)mism);
      if (f.nslow) atomicAdd(&nsl, (unsigned long long)f.nslow);
    }
    __syncthreads();
    // the bins: a thread holds every fourth row of one column
    {
      const int col = threadIdx.x & 63;
      uint32_t cs = 0;
      for (int i = 0; i < 16; i++) {
        const int row = (threadIdx.x >> 6) + 4 * i;
        const uint32_t v = col == 0 ? 0u : sc.w.t2[row * 64 + col];
        if (!__any_sync(0xFFFFFFFFu, v != 0u)) continue;
        cs += v;
        const uint32_t rs = __reduce_add_sync(0xFFFFFFFFu, v);
        const int k = row == 0 ? 0 : row - 64;
        if (lane == 0) atomicAdd(H + max(k + 48, 1), rs);
      }
      if (cs) atomicAdd(H + 64 + col, cs);
      cs = __reduce_add_sync(0xFFFFFFFFu, cs);
      if (lane == 0 && cs) atomicAdd(&tot[0], (unsigned long long)cs);
    }
    __syncthreads();
    Part64Rec r;
    rec_from_acc(r, acc, b - base);
    block_merge(r, sc.buf);
    Part64* out = p.parts + item;
    const unsigned long long fast = (unsigned long long)(e - b) - nsl, same = fast - tot[0];
    if (threadIdx.x == 0) {
      // the integer path's pairs: finite, unequal ones within or above the
      // tolerance (one sign: no flips), the rest bitwise equal
      r.cnt[PEAT_EXACT] += same;
      r.cnt[PEAT_WITHIN_TOL] += tot[0] - tot[1];
      r.cnt[PEAT_MISMATCH] += tot[1];
      r.nfin += fast;
      H[0] += (unsigned)same;
      H[64] += (unsigned)same;
      // an equal pair has |d| = 0 and u = 0: it matters when nothing larger was recorded
      need = same != 0ull && (r.ia < 0 || r.ahi == 0.0 || r.iu < 0 || r.mu == 0ull);
      first = nsl == 0ull ? 0u : 0xFFFFFFFFu;
    }
    __syncthreads();
    if (need && nsl != 0ull) {
      for (long long x = b; x < e && first == 0xFFFFFFFFu; x += TB) {
        __syncthreads();
        const long long i = x + threadIdx.x;
        if (i < e) {
          const uint64_t G = __ldg(reinterpret_cast<const unsigned long long*>(p.g) + i);
          const uint64_t C = __ldg(reinterpret_cast<const unsigned long long*>(p.c) + i);
          if (G == C && (G & MAG64) < INF64) atomicMin(&first, (unsigned)(i - b));
        }
        __syncthreads();
      }
    }
    if (threadIdx.x == 0) {
      if (need) {
        const long long z = b - base + first;
        if (r.ia < 0 || (r.ahi == 0.0 && z < r.ia)) r.ahi = r.alo = 0.0, r.asc = 0, r.ia = z;
        if (r.ir < 0 || (r.rkind == 0 && z < r.ir)) r.rkind = 0, r.ir = z;
        if (r.iu < 0 || (r.mu == 0ull && z < r.iu)) r.mu = 0ull, r.iu = z;
      }
      out->rec = r;
    }
    __syncthreads();
    // one carry step (limbs below 2^33 in magnitude afterwards, the top one as it is)
    for (int k = threadIdx.x; k < P64_MASK * 32; k += TB) {
      const int j = k % SL;
      const long long v = k < 3 * SL ? (j == SL - 1 ? S[k] : (S[k] & 0xFFFFFFFFll)) + (j > 0 ? S[k - 1] >> 32 : 0ll) : 0ll;
      if (k < 3 * SL) out->limbs[k] = v;
      const unsigned m = __ballot_sync(0xFFFFFFFFu, v != 0);
      if (lane == 0) out->mask[k >> 5] = m;
    }
    if (p.hist)
      for (int k = threadIdx.x; k < PEAT_HIST_BINS; k += TB)
        if (H[k]) atomicAdd(p.hist + seg * PEAT_HIST_BINS + k, (unsigned long long)H[k]);
    __syncthreads();
  }
}

// RN64 of the carry-save digits d[0..n) (digit j weighs 2^(32 (lo + j) + SLSB);
// all others are zero), with the subnormal grid below 2^-1022 and +-inf past the
// largest double.  d has room for two more digits, which take the carry; it
// is rewritten as the magnitude.
__device__ double digits_rn64(long long* d, int n, int lo) {
  auto carry_up = [&](int m) {
    long long carry = 0;
    for (int j = 0; j < m; j++) {
      const long long v = d[j] + carry;
      carry = v >> 32;
      d[j] = v & 0xFFFFFFFFll;
    }
    return carry;
  };
  d[n] = d[n + 1] = 0;
  const bool neg = carry_up(n + 2) < 0;  // (a sum is below 2^64 of its top digit's weight)
  if (neg) {
    long long borrow = 0;
    for (int j = 0; j < n + 2; j++) {
      long long v = -d[j] - borrow;
      borrow = v < 0 ? 1 : 0;
      d[j] = v + (borrow ? (1ll << 32) : 0);
    }
  }
  int t = n + 1;
  while (t >= 0 && d[t] == 0) t--;
  if (t < 0) return 0.0;
  // the leading four digits as W, whose bit 0 weighs 2^(32 (lo + t - 3) + SLSB)
  auto dig = [&](int j) -> u128 { return j >= 0 ? (u128)(uint32_t)d[j] : (u128)0; };
  const u128 W = (dig(t) << 96) | (dig(t - 1) << 64) | (dig(t - 2) << 32) | dig(t - 3);
  const int b0 = 32 * (lo + t - 3) + SLSB, top = b0 + 127 - __clz((int)(uint32_t)d[t]);
  int low = top - 52;
  if (low < -1074) low = -1074;
  const int sh = low - b0;  // at least 96 - 52
  unsigned long long mant = sh < 128 ? (unsigned long long)(W >> sh) : 0ull;
  const bool round = sh <= 128 && ((W >> (sh - 1)) & 1) != 0;
  bool sticky = sh > 128 ? W != 0 : (W << (129 - sh)) != 0;
  for (int j = t - 4; j >= 0 && !sticky; j--) sticky = d[j] != 0;
  if (round && (sticky || (mant & 1ull))) mant++;
  const double r = ldexp((double)mant, low);  // +inf past the largest double
  return neg ? -r : r;
}

// RN64 of (hi + lo) 2^sc / g (finite positive): the candidate around the
// binary64 quotient whose neighbouring midpoints bracket the exact value
__device__ double rel_value64(const Mag& a, double g) {
  if (a.lo == 0.0 && a.sc == 0) return __ddiv_rn(a.hi, g);  // one binary64 number over another: correctly rounded
  // at or past (2^54 - 1) 2^970 (the rounding threshold of the largest double): +inf
  {
    uint64_t mg;
    int eg;
    split_d(g, mg, eg);
    XTerm t[3] = {dbl_term(a.hi, a.sc, false), dbl_term(fabs(a.lo), a.sc, a.lo < 0.0),
                  XTerm{(u128)mg * ((1ull << 54) - 1), eg + 970, true}};
    if (xsign(t, 3) >= 0) return __longlong_as_double(0x7FF0000000000000ll);
  }
  double q = ldexp(__ddiv_rn(a.hi, g), a.sc);
  if (!(q <= 1.7976931348623157e308)) q = 1.7976931348623157e308;
  // sign of x - m g for x = (hi + lo) 2^sc and a midpoint m = (q1 + q2) / 2
  auto above_mid = [&](double q1, double q2) -> int {
    XTerm t[4] = {dbl_term(a.hi, a.sc + 1, false), dbl_term(fabs(a.lo), a.sc + 1, a.lo < 0.0),
                  prod_term(q1, g, 0, true), prod_term(q2, g, 0, true)};
    return xsign(t, 4);
  };
  for (int it = 0; it < 8; it++) {
    const double up = nextafter(q, 1.0 / 0.0), dn = nextafter(q, 0.0);
    if (q < 1.7976931348623157e308) {  // below the threshold checked above, the result is finite
      const int su = above_mid(q, up);
      if (su > 0 || (su == 0 && (__double_as_longlong(q) & 1))) {
        q = up;
        continue;
      }
    }
    if (q > 0.0) {
      const int sd = above_mid(dn, q);
      if (sd < 0 || (sd == 0 && (__double_as_longlong(q) & 1))) {
        q = dn;
        continue;
      }
    }
    break;
  }
  return q;
}

__global__ void __launch_bounds__(TB) compare64_finalize(Cmp64Params p) {
  __shared__ Part64Rec buf[TB / 2];
  __shared__ long long S[3 * SL];
  pdl_wait();  // stage 1 complete
  const long long seg = blockIdx.x;
  const long long f0 = p.seg_first[seg], f1 = p.seg_first[seg + 1];
  Part64Rec r;
  for (int k = 0; k < PEAT_NCLASS; k++) r.cnt[k] = 0;
  r.nfin = 0;
  r.ahi = r.alo = 0.0, r.asc = 0, r.ia = -1;
  r.rhi = r.rlo = 0.0, r.rsc = 0, r.rg = 1.0, r.rkind = 0, r.rle = 0, r.rlf = 0.0f, r.ir = -1;
  r.mu = 0, r.iu = -1;
  for (long long it = f0 + threadIdx.x; it < f1; it += TB) rec_merge(r, p.parts[it].rec);
  block_merge(r, buf);
  // the items' digits: only the columns that some item has (a dozen of 408 on
  // ordinary data), a warp per column; the range of each sum
  __shared__ unsigned cols[P64_MASK];
  __shared__ unsigned short list[3 * SL];
  __shared__ int nlist, lo[3], hi[3];
  __shared__ long long D[3 * (SL + 2)];
  __shared__ double sums[3];
  __shared__ unsigned long long nfin;
  // the mean and variance of |d| from S1 = sum |d| and S2 = sum d^2, both SL
  // digits weighing 2^(32 j + SLSB) (two more after carrying)
  __shared__ MeanVarScratch<SL + 2, SL + 2, -SLSB / 32> mv;
  static_assert(SLSB % 32 == 0, "the S2 shift is a whole number of digits");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = threadIdx.x; k < 3 * SL; k += TB) S[k] = 0;
  for (int k = threadIdx.x; k < SL + 2; k += TB) mv.A[k] = mv.B[k] = 0u;
  if (threadIdx.x < P64_MASK) cols[threadIdx.x] = 0u;
  if (threadIdx.x < 3) lo[threadIdx.x] = SL, hi[threadIdx.x] = -1;
  if (threadIdx.x == 0) nlist = 0, nfin = r.nfin;
  __syncthreads();
  for (long long it = f0 * P64_MASK + threadIdx.x; it < f1 * P64_MASK; it += TB) {
    const unsigned m = p.parts[it / P64_MASK].mask[it % P64_MASK];
    if (m) atomicOr(&cols[it % P64_MASK], m);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 3 * SL; k += TB)
    if ((cols[k >> 5] >> (k & 31)) & 1u) {
      list[atomicAdd(&nlist, 1)] = (unsigned short)k;
      atomicMin(&lo[k / SL], k % SL);
      atomicMax(&hi[k / SL], k % SL);
    }
  __syncthreads();
  for (int x = warp; x < nlist; x += TB / 32) {
    const int k = list[x];
    long long v = 0;
#pragma unroll 8
    for (long long it = f0 + lane; it < f1; it += 32) v += p.parts[it].limbs[k];
    v = (long long)wsum_u64((uint64_t)v);
    if (lane == 0) S[k] = v;
  }
  __syncthreads();
  // the digits of S1 and S2 carried (non-negative: two more take the carry), and
  // the three sums rounded, a warp each
  if (lane == 0 && warp < 2) {
    const int q = warp + 1, n = hi[q] - lo[q] + 1;
    if (n > 0) {
      uint32_t* out = warp ? mv.B : mv.A;
      // (at most SL + 2 digits: the carry of the top ones stays inside)
      carry_to_digits(S + q * SL + lo[q], n, out + lo[q]);
    }
  }
  if (lane == 0 && warp >= 2 && warp < 5) {
    const int q = warp - 2, n = hi[q] - lo[q] + 1;
    long long* d = D + q * (SL + 2);
    for (int j = 0; j < n; j++) d[j] = S[q * SL + lo[q] + j];
    sums[q] = n > 0 ? digits_rn64(d, n, lo[q]) : 0.0;
  }
  mean_var_block(mv, nfin, SLSB);
  if (threadIdx.x != 0) return;
  peat_stats_t o;
  o.n = (uint64_t)(p.offsets[seg + 1] - p.offsets[seg]);
  for (int k = 0; k < PEAT_NCLASS; k++) o.count[k] = r.cnt[k];
  o.n_finite = r.nfin;
  o.max_abs = r.ia >= 0 ? (r.asc ? __dmul_rn(r.ahi, 2.0) : r.ahi) : 0.0;  // RN(2 x) = 2 RN(x), +inf on overflow
  o.argmax_abs = r.ia;
  if (r.ir < 0 || r.rkind == 0) o.max_rel = 0.0;
  else if (r.rkind == 2) o.max_rel = __longlong_as_double(0x7FF0000000000000ll);
  else o.max_rel = rel_value64(Mag{r.rhi, r.rlo, r.rsc}, r.rg);
  o.argmax_rel = r.ir;
  o.max_ulp = r.iu >= 0 ? r.mu : 0;
  o.argmax_ulp = r.iu;
  o.sum_signed = sums[0];
  o.sum_abs = sums[1];
  o.sum_sq = sums[2];
  o.rtol_eff = p.rtol;
  o.atol_eff = p.atol;
  o.mean_abs = mv.mean;
  o.var_abs = mv.var;
  p.stats[seg] = o;
}

}  // namespace

cudaError_t launch_compare64(const Cmp64Params& p, int nctas, cudaStream_t s) {
  if (p.nitems == 0) {
    compare64_finalize<<<(unsigned)p.nseg, TB, 0, s>>>(p);
    return cudaGetLastError();
  }
  compare64_stage1<<<nctas, TB, 0, s>>>(p);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_dependent(compare64_finalize, (unsigned)p.nseg, TB, 0, s, p);  // overlaps stage 1's end
}

}  // namespace peat
