// The error signature (Section IV-B-3: maximum, mean and variance of
// |c - g|, with the classes, ULP distances and histograms of the compare) for
// the two 8-bit formats of the OCP FP8 specification, E4M3 and E5M2 (the
// paper lists 8-bit precisions among those a kernel may run in).
//
// Every finite value of these formats is an integer multiple of 2^-S (S = 9
// for E4M3, 16 for E5M2) below 2^32 in units of 2^-S, so d = c - g is an exact
// 64-bit integer D in those units and |d|, d and d^2 accumulate exactly as
// integers (d^2 in 128 bits), and the tolerance test is one integer
// comparison against a bound per golden magnitude computed exactly on the host.  Work items are contiguous runs of one segment; each
// item's totals go to a record of its own, and one CTA per segment merges
// its items (integer sums, maxima by exact comparison with the lowest index
// on ties: the order of the merge does not matter).
#include <cstdint>
#include <type_traits>

#include "meanvar.cuh"
#include "peat_internal.h"

namespace peat {
namespace {

constexpr int TB = 1024;      // threads of a stage-1 CTA (one per SM)
constexpr int FB = 512;       // threads of a finalize CTA

template <int DT>
struct F8;
template <>
struct F8<PEAT_F8E4M3> {
  static constexpr int S = 9, MB = 3;  // value = K 2^-9; 3 fraction bits, bias 7
};
template <>
struct F8<PEAT_F8E5M2> {
  static constexpr int S = 16, MB = 2;  // value = K 2^-16; 2 fraction bits, bias 15
};

// magnitude (7 bits): 0 finite, 1 infinite, 2 NaN
template <int DT>
__device__ __forceinline__ int f8_kind(uint32_t mag) {
  if constexpr (DT == PEAT_F8E4M3) return mag == 0x7Fu ? 2 : 0;
  else return mag < 0x7Cu ? 0 : (mag == 0x7Cu ? 1 : 2);
}
// |value| 2^S of a finite magnitude: subnormal m, normal (2^MB + m) 2^(e - 1)
template <int DT>
__device__ __forceinline__ uint32_t f8_units(uint32_t mag) {
  constexpr int MB = F8<DT>::MB;
  const uint32_t e = mag >> MB, m = mag & ((1u << MB) - 1u);
  return e == 0 ? m : ((m | (1u << MB)) << (e - 1));
}

// the magnitude whose value is K units (none: there is no such finite value)
template <int DT>
__device__ __forceinline__ uint32_t f8_encode(unsigned long long K, uint32_t none) {
  constexpr int MB = F8<DT>::MB;
  if (K < (1ull << MB)) return (uint32_t)K;
  const int msb = 63 - __clzll((long long)K);
  const uint32_t mag = (uint32_t)((msb - MB + 1) << MB) | ((uint32_t)(K >> (msb - MB)) & ((1u << MB) - 1u));
  return mag < 128u && f8_kind<DT>(mag) == 0 && f8_units<DT>(mag) == K ? mag : none;
}

using u128 = unsigned __int128;
using i128 = __int128;

// totals of a run of pairs
struct Tot {
  unsigned long long cnt[PEAT_NCLASS], nfin;
  u128 s1, s2;  // sum |D|, sum D^2
  i128 sd;      // sum D
  unsigned long long ma;  // max |D|, at index ia (-1: no finite pair)
  long long ia;
  unsigned long long ra, rb;  // max |D| / |G| as the fraction ra / rb (rb = 0: +inf), at ir
  long long ir;
  unsigned long long mu;  // max ULP distance, at iu (-1: none)
  long long iu;
};

__device__ __forceinline__ void tot_init(Tot& t) {
  for (int k = 0; k < PEAT_NCLASS; k++) t.cnt[k] = 0;
  t.nfin = 0;
  t.s1 = 0;
  t.s2 = 0;
  t.sd = 0;
  t.ma = 0, t.ia = -1;
  t.ra = 0, t.rb = 1, t.ir = -1;
  t.mu = 0, t.iu = -1;
}

// x better than y: larger, or equal at a lower index; an absent record (index -1) is worst
__device__ __forceinline__ bool better_u(unsigned long long x, long long ix, unsigned long long y, long long iy) {
  if (ix < 0) return false;
  if (iy < 0) return true;
  return x > y || (x == y && ix < iy);
}
// compare xa/xb with ya/yb (b = 0: +inf; a = 0 always carries b = 1)
__device__ __forceinline__ int cmp_frac(unsigned long long xa, unsigned long long xb, unsigned long long ya,
                                        unsigned long long yb) {
  if (xb == 0 || yb == 0) return (xb == 0) - (yb == 0);
  const u128 l = (u128)xa * yb, r = (u128)ya * xb;
  return (l > r) - (l < r);
}
__device__ __forceinline__ bool better_rel(unsigned long long xa, unsigned long long xb, long long ix,
                                           unsigned long long ya, unsigned long long yb, long long iy) {
  if (ix < 0) return false;
  if (iy < 0) return true;
  const int c = cmp_frac(xa, xb, ya, yb);
  return c > 0 || (c == 0 && ix < iy);
}

__device__ __forceinline__ void tot_merge(Tot& t, const Tot& o) {
  for (int k = 0; k < PEAT_NCLASS; k++) t.cnt[k] += o.cnt[k];
  t.nfin += o.nfin;
  t.s1 += o.s1;
  t.s2 += o.s2;
  t.sd += o.sd;
  if (better_u(o.ma, o.ia, t.ma, t.ia)) t.ma = o.ma, t.ia = o.ia;
  if (better_rel(o.ra, o.rb, o.ir, t.ra, t.rb, t.ir)) t.ra = o.ra, t.rb = o.rb, t.ir = o.ir;
  if (better_u(o.mu, o.iu, t.mu, t.iu)) t.mu = o.mu, t.iu = o.iu;
}

// sums over the warp, modulo 2^64 and 2^128 (so signs wrap): 27-bit pieces
// through the 32-bit reduction instruction
__device__ __forceinline__ uint64_t wsum(uint64_t v) {
  uint64_t r = 0;
#pragma unroll
  for (int k = 0; k < 3; k++) r += (uint64_t)__reduce_add_sync(0xFFFFFFFFu, (uint32_t)(v >> (27 * k)) & 0x7FFFFFFu) << (27 * k);
  return r;
}
__device__ __forceinline__ uint64_t wmax(uint64_t v) {
  const uint32_t h = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(v >> 32));
  const uint32_t l = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(v >> 32) == h ? (uint32_t)v : 0u);
  return ((uint64_t)h << 32) | l;
}
// the lowest index among the lanes with ok (-1: none)
__device__ __forceinline__ long long wfirst(bool ok, long long i) {
  const uint64_t m = wmax(ok ? ~(uint64_t)i : 0ull);
  return m ? (long long)~m : -1;
}
__device__ __forceinline__ u128 wsum128(u128 v) {
  u128 r = 0;
#pragma unroll
  for (int k = 0; k < 5; k++) r += (u128)__reduce_add_sync(0xFFFFFFFFu, (uint32_t)(v >> (27 * k)) & 0x7FFFFFFu) << (27 * k);
  return r;
}
// every lane ends with the warp's totals (reductions by value, then by index:
// a tournament of the whole record took 26 us for the 32 warps of a CTA)
__device__ __forceinline__ void warp_total(Tot& t) {
#pragma unroll
  for (int k = 0; k < PEAT_NCLASS; k++) t.cnt[k] = wsum(t.cnt[k]);
  t.nfin = wsum(t.nfin);
  t.s1 = wsum128(t.s1);
  t.s2 = wsum128(t.s2);
  t.sd = (i128)wsum128((u128)t.sd);
  const uint64_t ma = wmax(t.ia >= 0 ? t.ma : 0ull);
  t.ia = wfirst(t.ia >= 0 && t.ma == ma, t.ia);
  t.ma = ma;
  const uint64_t mu = wmax(t.iu >= 0 ? t.mu : 0ull);
  t.iu = wfirst(t.iu >= 0 && t.mu == mu, t.iu);
  t.mu = mu;
  unsigned long long ba = t.ir >= 0 ? t.ra : 0ull, bb = t.ir >= 0 ? t.rb : 1ull;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long ya = __shfl_xor_sync(0xFFFFFFFFu, ba, o), yb = __shfl_xor_sync(0xFFFFFFFFu, bb, o);
    if (cmp_frac(ya, yb, ba, bb) > 0) ba = ya, bb = yb;
  }
  t.ir = wfirst(t.ir >= 0 && cmp_frac(t.ra, t.rb, ba, bb) == 0, t.ir);
  t.ra = ba, t.rb = bb;
}
// the CTA's totals, complete in every lane of warp 0 (every thread calls it; at most 32 warps)
__device__ __noinline__ void block_total(Tot& x, Tot* warp_tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Tot t = x;
  warp_total(t);
  if (lane == 0) warp_tot[warp] = t;
  __syncthreads();
  if (warp == 0) {
    if (lane < (int)(blockDim.x >> 5)) t = warp_tot[lane];
    else tot_init(t);
    warp_total(t);
    x = t;
  }
  __syncthreads();
}

// floor(log2(a / b)) for a, b >= 1
__device__ __forceinline__ int floor_log2_ratio(unsigned long long a, unsigned long long b) {
  const int ea = 63 - __clzll((long long)a), eb = 63 - __clzll((long long)b);
  return (ea - eb) - ((a << (63 - ea)) < (b << (63 - eb)) ? 1 : 0);
}

// add one to shared bin `bin` for every lane that has one (bin < 0: none), one atomic per distinct bin
__device__ __forceinline__ void hist_add(unsigned* H, int bin) {
  const unsigned grp = __match_any_sync(0xFFFFFFFFu, bin);
  if (bin >= 0 && (int)(threadIdx.x & 31) == __ffs(grp) - 1) atomicAdd(H + bin, (unsigned)__popc(grp));
}

// A thread's totals within one work item, in the narrowest exact types:
// |D| < 2^19 (E4M3) or 2^33 (E5M2), at most 2^14 pairs per thread and item.
// Offsets are positions in the item plus one (0: none); they only grow along a
// thread's pairs, so a strict comparison keeps the earliest on ties.
template <int DT>
struct Acc8 {
  using A = typename std::conditional<DT == PEAT_F8E4M3, uint32_t, unsigned long long>::type;
  uint32_t cnt[PEAT_NCLASS], nfin;
  unsigned long long s1, s2lo, s2hi;
  long long sd;
  A ma;
  uint32_t ia;
  A ra;
  uint32_t rb, ir;
  float rt;  // ra / rb in float32 lowered by 1e-5 (more than its error): a pair below it cannot win
  uint32_t mu, iu;
};

template <int DT>
__device__ __forceinline__ void acc_init(Acc8<DT>& t) {
#pragma unroll
  for (int k = 0; k < PEAT_NCLASS; k++) t.cnt[k] = 0;
  t.nfin = 0;
  t.s1 = t.s2lo = t.s2hi = 0;
  t.sd = 0;
  t.ma = 0, t.ia = 0;
  t.ra = 0, t.rb = 1, t.ir = 0, t.rt = 0.0f;
  t.mu = 0, t.iu = 0;
}

template <int DT>
__device__ __forceinline__ float to_f(typename Acc8<DT>::A a) {
  if constexpr (DT == PEAT_F8E4M3) return __uint2float_rn(a);
  else return __fmaf_rn(__uint2float_rn((uint32_t)(a >> 32)), 4294967296.0f, __uint2float_rn((uint32_t)a));
}

// xa / xb > ya / yb exactly (xb, yb: |g| in units, 0 = the ratio is +inf; xa = 0 carries xb = 1)
template <int DT>
__device__ __forceinline__ bool frac_gt(typename Acc8<DT>::A xa, uint32_t xb, typename Acc8<DT>::A ya, uint32_t yb) {
  if (xb == 0 || yb == 0) return xb == 0 && yb != 0;
  if constexpr (DT == PEAT_F8E4M3) {
    return (unsigned long long)xa * yb > (unsigned long long)ya * xb;  // below 2^37
  } else {
    const u128 l = (u128)xa * yb, r = (u128)ya * xb;
    return l > r;
  }
}

// one pair slot of the warp (every lane calls it; ok: this lane holds the pair at item offset off;
// amax: the tolerance bound per golden magnitude)
template <int DT>
__device__ __forceinline__ void pair8(const unsigned long long* amax, Acc8<DT>& t, unsigned* H, uint32_t G,
                                      uint32_t C, bool ok, uint32_t off) {
  using A = typename Acc8<DT>::A;
  int relbin = -1, ulpbin = -1, cls = -1;
  if (ok) {
    const uint32_t mg = G & 0x7Fu, mc = C & 0x7Fu, sg = G >> 7, sc = C >> 7;
    const int kg = f8_kind<DT>(mg), kc = f8_kind<DT>(mc);
    const int keyg = sg ? -(int)mg : (int)mg, keyc = sc ? -(int)mc : (int)mc;
    const uint32_t u = (uint32_t)(keyc > keyg ? keyc - keyg : keyg - keyc);
    const bool nan = kg == 2 || kc == 2;
    if (kg | kc) {
      const bool eq = (kg == 2 && kc == 2) || (kg == 1 && kc == 1 && sg == sc);
      cls = eq ? PEAT_EXACT : PEAT_NAN_INF_ASYM;
      relbin = eq ? 0 : 63;
    } else {
      const uint32_t Kg = f8_units<DT>(mg), Kc = f8_units<DT>(mc);
      A a;
      long long D;
      if constexpr (DT == PEAT_F8E4M3) {
        const int d = (sc ? -(int)Kc : (int)Kc) - (sg ? -(int)Kg : (int)Kg);
        D = d;
        a = (uint32_t)(d < 0 ? -d : d);
        t.s2lo += (unsigned long long)a * a;
      } else {
        D = (sc ? -(long long)Kc : (long long)Kc) - (sg ? -(long long)Kg : (long long)Kg);
        a = (unsigned long long)(D < 0 ? -D : D);
        const unsigned long long lo = a * a, hi = __umul64hi(a, a);
        t.s2lo += lo;
        t.s2hi += hi + (t.s2lo < lo ? 1ull : 0ull);
      }
      t.nfin++;
      t.s1 += a;
      t.sd += D;
      if (a > t.ma || t.ia == 0) t.ma = a, t.ia = off + 1;
      // the relative maximum: one float32 multiply rules out all but the candidates
      const uint32_t rb = a == 0 ? 1u : Kg;
      if (t.ir == 0 || to_f<DT>(a) >= __fmul_rn(t.rt, __uint2float_rn(rb))) {
        if (t.ir == 0 || frac_gt<DT>(a, rb, t.ra, t.rb)) {
          t.ra = a, t.rb = rb, t.ir = off + 1;
          t.rt = rb == 0 ? __int_as_float(0x7F800000)
                         : __fmul_rn(__fdiv_rn(to_f<DT>(a), __uint2float_rn(rb)), 0.99999f);
        }
      }
      if (a == 0) {
        cls = PEAT_EXACT;
        relbin = 0;
      } else {
        if ((unsigned long long)a <= amax[mg]) cls = PEAT_WITHIN_TOL;
        else if (Kg != 0 && Kc != 0 && sg != sc) cls = PEAT_SIGN_FLIP;
        else cls = PEAT_MISMATCH;
        if (Kg == 0) {
          relbin = 63;
        } else {
          const int k = floor_log2_ratio((unsigned long long)a, Kg) + 48;
          relbin = k < 1 ? 1 : (k > 62 ? 62 : k);
        }
      }
    }
    if (nan) {
      ulpbin = (kg == 2 && kc == 2) ? 0 : 63;  // no ULP distance with a NaN
    } else {
      ulpbin = (int)(u < 63 ? u : 63);
      if (u > t.mu || t.iu == 0) t.mu = u, t.iu = off + 1;
    }
  }
#pragma unroll
  for (int k = 0; k < PEAT_NCLASS; k++) t.cnt[k] += cls == k;
  hist_add(H, relbin);
  hist_add(H, ulpbin < 0 ? -1 : 64 + ulpbin);
}

// (out of line: the pairs that the table does not take)
template <int DT>
__device__ __noinline__ void pair8_slow(const unsigned long long* amax, Acc8<DT>& t, unsigned* H, uint32_t G, uint32_t C,
                                        bool ok, uint32_t off) {
  pair8<DT>(amax, t, H, G, C, ok, off);
}

// a thread's item totals as segment totals (item starts at segment position ib)
template <int DT>
__device__ __forceinline__ void acc_to_tot(Tot& t, const Acc8<DT>& a, long long ib) {
#pragma unroll
  for (int k = 0; k < PEAT_NCLASS; k++) t.cnt[k] = a.cnt[k];
  t.nfin = a.nfin;
  t.s1 = a.s1;
  t.s2 = ((u128)a.s2hi << 64) | a.s2lo;
  t.sd = a.sd;
  t.ma = a.ma, t.ia = a.ia ? ib + a.ia - 1 : -1;
  t.ra = a.ra, t.rb = a.rb, t.ir = a.ir ? ib + a.ir - 1 : -1;
  t.mu = a.mu, t.iu = a.iu ? ib + a.iu - 1 : -1;
}

__device__ __forceinline__ void store_tot(Part8* d, const Tot& t) {
  for (int k = 0; k < PEAT_NCLASS; k++) d->cnt[k] = t.cnt[k];
  d->nfin = t.nfin;
  d->s1lo = (unsigned long long)t.s1, d->s1hi = (unsigned long long)(t.s1 >> 64);
  d->s2lo = (unsigned long long)t.s2, d->s2hi = (unsigned long long)(t.s2 >> 64);
  d->sdlo = (unsigned long long)(u128)t.sd, d->sdhi = (unsigned long long)((u128)t.sd >> 64);
  d->ma = t.ma, d->ia = t.ia;
  d->ra = t.ra, d->rb = t.rb, d->ir = t.ir;
  d->mu = t.mu, d->iu = t.iu;
}
__device__ __forceinline__ void load_tot(Tot& t, const Part8* d) {
  for (int k = 0; k < PEAT_NCLASS; k++) t.cnt[k] = d->cnt[k];
  t.nfin = d->nfin;
  t.s1 = ((u128)d->s1hi << 64) | d->s1lo;
  t.s2 = ((u128)d->s2hi << 64) | d->s2lo;
  t.sd = (i128)(((u128)d->sdhi << 64) | d->sdlo);
  t.ma = d->ma, t.ia = d->ia;
  t.ra = d->ra, t.rb = d->rb, t.ir = d->ir;
  t.mu = d->mu, t.iu = d->iu;
}

// The table.  A pair of one sign is one of 2^15 (golden byte, candidate
// magnitude) combinations: stage 1 only counts them, in one shared word each (an
// increment by the constant one costs a cycle per distinct address of a bank),
// about six instructions per pair, and evaluates the definitions once per
// combination that occurred, at the end of an item.  Pairs of opposite signs go
// through pair8, a warp's together (opposite8).  The counts hold no indices: the finalization searches the
// first item that holds a maximum for the first pair that attains it.
//
// What bounds it: the shared-memory increments (about three cycles per 32
// pairs and SM), then instruction issue.  Measured (33.5 M E4M3 pairs with
// noise, back-to-back calls): 328 us with every pair evaluated (about 220
// instructions per 32 pairs), 83 us now, of which the counting takes 16, the
// rest of this kernel 18 and the finalization 35 (latency).
constexpr int CELLS = 1 << 15;
constexpr int SMEM8 = CELLS * 4 + CELLS * 2;  // the counters and the list of those that are not zero
static_assert(CELLS * 2 >= (TB / 32) * 512 * 4, "the pairs of opposite signs of a round fit the list");

// two 15-bit cell numbers from the low bytes of both halves: golden << 7 | candidate's magnitude
__device__ __forceinline__ uint32_t cells2(uint32_t g, uint32_t c) {
  return (g & 0x00FF00FFu) * 128u + (c & 0x007F007Fu);
}
__device__ __forceinline__ void inc_cell(uint32_t table, uint32_t cell) {
  asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(table + cell * 4u));
}

// n pairs (G, C) of the table into the totals and the bins (the definitions of pair8)
template <int DT>
__device__ __forceinline__ void eval_cell(const unsigned long long* amax, Tot& t, unsigned* H, uint32_t G, uint32_t C,
                                          uint32_t n) {
  const uint32_t mg = G & 0x7Fu, mc = C & 0x7Fu;
  const int kg = f8_kind<DT>(mg), kc = f8_kind<DT>(mc);
  const uint32_t u = mc > mg ? mc - mg : mg - mc;  // one sign
  int relbin, cls;
  if (kg | kc) {
    const bool eq = (kg == 2 && kc == 2) || (kg == 1 && kc == 1);
    cls = eq ? PEAT_EXACT : PEAT_NAN_INF_ASYM;
    relbin = eq ? 0 : 63;
  } else {
    const uint32_t Kg = f8_units<DT>(mg), Kc = f8_units<DT>(mc);
    const unsigned long long a = Kc > Kg ? Kc - Kg : Kg - Kc;
    const bool neg = (Kc < Kg) != ((G >> 7) != 0);
    t.nfin += n;
    t.s1 += (u128)a * n;
    t.s2 += (u128)a * a * n;
    t.sd += neg ? -(i128)((u128)a * n) : (i128)((u128)a * n);
    const unsigned long long rb = a == 0 ? 1ull : Kg;
    if (better_u(a, 0, t.ma, t.ia)) t.ma = a, t.ia = 0;
    if (better_rel(a, rb, 0, t.ra, t.rb, t.ir)) t.ra = a, t.rb = rb, t.ir = 0;
    if (a == 0) {
      cls = PEAT_EXACT;
      relbin = 0;
    } else {
      cls = a <= amax[mg] ? PEAT_WITHIN_TOL : PEAT_MISMATCH;
      relbin = 63;
      if (Kg != 0) relbin = min(max(floor_log2_ratio(a, Kg) + 48, 1), 62);
    }
  }
  int ulpbin = kg == 2 ? 0 : 63;  // with a NaN: 0 when both are
  if (kg == 2 || kc == 2) {
    if (kg != kc) ulpbin = 63;
  } else {
    ulpbin = (int)min(u, 63u);
    if (better_u(u, 0, t.mu, t.iu)) t.mu = u, t.iu = 0;
  }
#pragma unroll
  for (int k = 0; k < PEAT_NCLASS; k++) t.cnt[k] += cls == k ? n : 0u;
  atomicAdd(H + relbin, n);
  atomicAdd(H + 64 + ulpbin, n);
}

// Every pair evaluated by itself: the whole of a call with fewer than
// C8_TABLE_MIN pairs, where the passes over the table and the search for the
// maxima's first pairs would cost more than they save.
constexpr int DTB = 256;
template <int DT>
__global__ void __launch_bounds__(DTB) compare8_direct(Cmp8Params p) {
  __shared__ unsigned H[PEAT_HIST_BINS];
  __shared__ Tot warp_tot[DTB / 32];
  __shared__ unsigned long long AM[128];
  pdl_trigger();  // the finalize kernel may start launching (it waits for this grid)
  const int lane = threadIdx.x & 31;
  for (int k = threadIdx.x; k < 128; k += DTB) AM[k] = p.amax[k];
  for (long long item = blockIdx.x; item < p.nitems; item += gridDim.x) {
    const long long b = p.item_b[item], e = p.item_e[item], seg = p.item_seg[item];
    const long long base = p.offsets[seg];  // indices are reported within the segment
    for (int k = threadIdx.x; k < PEAT_HIST_BINS; k += DTB) H[k] = 0u;
    __syncthreads();
    Acc8<DT> acc;
    acc_init(acc);
    uint32_t nsame = 0;  // pairs of the equal-group fast path (rel and ULP bin 0)
    // groups of 16 elements on the absolute index grid, whole warps in every round
    const long long q0 = b >> 4, q1 = (e + 15) >> 4;
    for (long long q = q0 + threadIdx.x; __any_sync(0xFFFFFFFFu, q < q1); q += DTB) {
      const bool okq = q < q1;
      const long long i0 = q << 4;
      uint32_t w[4] = {0u, 0u, 0u, 0u}, x[4] = {0u, 0u, 0u, 0u};
      if (okq && p.vec && i0 >= b && i0 + 16 <= e) {
        const uint4 gv = __ldg(reinterpret_cast<const uint4*>(p.g) + q);
        const uint4 cv = __ldg(reinterpret_cast<const uint4*>(p.c) + q);
        w[0] = gv.x, w[1] = gv.y, w[2] = gv.z, w[3] = gv.w;
        x[0] = cv.x, x[1] = cv.y, x[2] = cv.z, x[3] = cv.w;
      } else if (okq) {
#pragma unroll
        for (int j = 0; j < 16; j++) {
          const long long i = i0 + j;
          if (i >= b && i < e) {
            w[j >> 2] |= (uint32_t)__ldg(reinterpret_cast<const unsigned char*>(p.g) + i) << (8 * (j & 3));
            x[j >> 2] |= (uint32_t)__ldg(reinterpret_cast<const unsigned char*>(p.c) + i) << (8 * (j & 3));
          }
        }
      }
      // a warp slot of bitwise-equal, finite whole groups (decided for the whole warp):
      // 16 EXACT pairs per lane with |d| = 0 and u = 0
      bool fast = !okq;
      if (okq && p.vec && i0 >= b && i0 + 16 <= e && w[0] == x[0] && w[1] == x[1] && w[2] == x[2] && w[3] == x[3]) {
        bool fin = true;
#pragma unroll
        for (int j = 0; j < 16; j++) fin &= f8_kind<DT>((w[j >> 2] >> (8 * (j & 3))) & 0x7Fu) == 0;
        fast = fin;
      }
      if (__all_sync(0xFFFFFFFFu, fast)) {
        if (okq) {
          const uint32_t off = (uint32_t)(i0 - b);
          acc.cnt[PEAT_EXACT] += 16;
          acc.nfin += 16;
          if (acc.ia == 0) acc.ma = 0, acc.ia = off + 1;
          if (acc.ir == 0) acc.ra = 0, acc.rb = 1, acc.ir = off + 1, acc.rt = 0.0f;
          if (acc.iu == 0) acc.mu = 0, acc.iu = off + 1;
          nsame += 16;
        }
        continue;
      }
      // one copy of the pair code: the loop stays rolled (the body is long)
#pragma unroll 1
      for (int j = 0; j < 16; j++) {
        const long long i = i0 + j;
        const bool ok = okq && i >= b && i < e;
        const uint32_t gw = j < 8 ? (j < 4 ? w[0] : w[1]) : (j < 12 ? w[2] : w[3]);
        const uint32_t cw = j < 8 ? (j < 4 ? x[0] : x[1]) : (j < 12 ? x[2] : x[3]);
        pair8<DT>(AM, acc, H, (gw >> (8 * (j & 3))) & 0xFFu, (cw >> (8 * (j & 3))) & 0xFFu, ok, (uint32_t)(i - b));
      }
    }
    {
      const uint32_t ns = __reduce_add_sync(0xFFFFFFFFu, nsame);
      if (lane == 0 && ns) {
        atomicAdd(&H[0], ns);
        atomicAdd(&H[64], ns);
      }
    }
    Tot t;
    acc_to_tot<DT>(t, acc, b - base);
    block_total(t, warp_tot);
    if (threadIdx.x == 0) store_tot(p.parts + item, t);
    if (p.hist)
      for (int k = threadIdx.x; k < PEAT_HIST_BINS; k += DTB)
        if (H[k]) atomicAdd(p.hist + seg * PEAT_HIST_BINS + k, (unsigned long long)H[k]);
    __syncthreads();
  }
}

// The pairs of opposite signs (bits todo) among the lanes' groups (16 pairs from
// offset o of the item; the whole warp calls it): taken back from the table, gathered in order
// in the warp's part of the list (idle while pairs are counted) and evaluated
// by full warps.  Measured, E5M2 with 16 % of such pairs, 4.3 M and 9 M: each lane
// its own in turn, which takes as many rounds as the fullest lane has, 121 and
// 170 us, now 103 and 132.  Where no lane has two, the caller takes them at once
// (E4M3 with 0.04 % of such pairs, 10 M: 74 us gathered, 72 at once).
template <int DT>
__device__ __noinline__ void opposite8(const unsigned long long* amax, Acc8<DT>& acc, unsigned* H, uint32_t* T, uint4 g,
                                       uint4 c, int o, uint32_t todo) {
  const int lane = threadIdx.x & 31;
  const uint32_t w[4] = {g.x, g.y, g.z, g.w}, x[4] = {c.x, c.y, c.z, c.w};
  uint32_t* q = T + CELLS + (threadIdx.x >> 5) * 512;
  const uint32_t k = __popc(todo);
  uint32_t at = k;
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, at, s);
    if (lane >= s) at += y;
  }
  const uint32_t n = __shfl_sync(0xFFFFFFFFu, at, 31);
  at -= k;
#pragma unroll 1
  for (; todo; todo &= todo - 1u) {
    const int j = __ffs(todo) - 1;
    const uint32_t gw = j < 8 ? (j < 4 ? w[0] : w[1]) : (j < 12 ? w[2] : w[3]);
    const uint32_t cw = j < 8 ? (j < 4 ? x[0] : x[1]) : (j < 12 ? x[2] : x[3]);
    const uint32_t G = (gw >> (8 * (j & 3))) & 0xFFu, C = (cw >> (8 * (j & 3))) & 0xFFu;
    atomicSub(T + (G * 128u + (C & 0x7Fu)), 1u);
    q[at++] = G | (C << 8) | (uint32_t)(16 * lane + j) << 16;
  }
  __syncwarp();
#pragma unroll 1
  for (uint32_t b = 0; b < n; b += 32) {
    const bool ok = b + lane < n;
    const uint32_t e = ok ? q[b + lane] : 0u;
    pair8<DT>(amax, acc, H, e & 0xFFu, (e >> 8) & 0xFFu, ok, (uint32_t)(o - 16 * lane) + (e >> 16));
  }
  __syncwarp();
}

template <int DT>
__global__ void __launch_bounds__(TB, 1) compare8_stage1(Cmp8Params p) {
  extern __shared__ __align__(16) uint32_t T[];  // CELLS counters, then the list
  __shared__ unsigned H[PEAT_HIST_BINS];
  __shared__ Tot warp_tot[TB / 32];
  __shared__ unsigned long long AM[128];
  __shared__ int any_slow, nlist;
  unsigned short* list = reinterpret_cast<unsigned short*>(T + CELLS);  // CELLS entries
  pdl_trigger();  // the finalize kernel may start launching (it waits for this grid)
  const uint32_t table = (uint32_t)__cvta_generic_to_shared(T);
  for (int k = threadIdx.x; k < 128; k += TB) AM[k] = p.amax[k];
  for (int k = threadIdx.x; k < CELLS / 4; k += TB) reinterpret_cast<uint4*>(T)[k] = make_uint4(0, 0, 0, 0);
  for (long long item = blockIdx.x; item < p.nitems; item += gridDim.x) {
    const long long b = p.item_b[item], e = p.item_e[item], seg = p.item_seg[item];
    const long long base = p.offsets[seg];  // indices are reported within the segment
    for (int k = threadIdx.x; k < PEAT_HIST_BINS; k += TB) H[k] = 0u;
    if (threadIdx.x == 0) any_slow = nlist = 0;
    __syncthreads();
    Acc8<DT> acc;
    acc_init(acc);
    // groups of 16 elements on the absolute index grid, whole warps in every
    // round, the next group loaded while this one is counted
    const int len = (int)(e - b), o0 = -(int)(b & 15), nq = (len - o0 + 15) >> 4;
    const unsigned char* gp = reinterpret_cast<const unsigned char*>(p.g) + b + o0;
    const unsigned char* cp = reinterpret_cast<const unsigned char*>(p.c) + b + o0;
    auto load = [&](int v, uint4& gv, uint4& cv) {
      gv = cv = make_uint4(0, 0, 0, 0);
      const int o = o0 + 16 * v;
      if (p.vec && o >= 0 && o + 16 <= len) {
        gv = __ldg(reinterpret_cast<const uint4*>(gp) + v);
        cv = __ldg(reinterpret_cast<const uint4*>(cp) + v);
      } else if (o < len) {
        uint32_t w[4] = {0u, 0u, 0u, 0u}, x[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int j = 0; j < 16; j++)
          if (o + j >= 0 && o + j < len) {
            w[j >> 2] |= (uint32_t)__ldg(gp + 16 * v + j) << (8 * (j & 3));
            x[j >> 2] |= (uint32_t)__ldg(cp + 16 * v + j) << (8 * (j & 3));
          }
        gv = make_uint4(w[0], w[1], w[2], w[3]);
        cv = make_uint4(x[0], x[1], x[2], x[3]);
      }
    };
    uint4 gn, cn;
    int v = threadIdx.x;
    load(v, gn, cn);
    for (int r = threadIdx.x & ~31; r < nq; r += TB, v += TB) {
      const uint4 gc = gn, cc = cn;
      load(v + TB, gn, cn);
      const int o = o0 + 16 * v;
      const uint32_t w[4] = {gc.x, gc.y, gc.z, gc.w}, x[4] = {cc.x, cc.y, cc.z, cc.w};
      const bool edge = o < 0 || o + 16 > len;
      const bool odd = (((w[0] ^ x[0]) | (w[1] ^ x[1]) | (w[2] ^ x[2]) | (w[3] ^ x[3])) & 0x80808080u) != 0u || edge;
      const bool odd_w = __any_sync(0xFFFFFFFFu, odd);
      if (!odd_w || !__any_sync(0xFFFFFFFFu, edge)) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const uint32_t c0 = cells2(w[i], x[i]), c1 = cells2(w[i] >> 8, x[i] >> 8);
          inc_cell(table, c0 & 0xFFFFu);
          inc_cell(table, c0 >> 16);
          inc_cell(table, c1 & 0xFFFFu);
          inc_cell(table, c1 >> 16);
        }
        if (!odd_w) continue;
        // pairs of opposite signs, taken back from the table
        any_slow = 1;
        uint32_t todo = 0;
#pragma unroll
        for (int i = 0; i < 4; i++) todo |= ((((w[i] ^ x[i]) >> 7 & 0x01010101u) * 0x01020408u) >> 24 & 0xFu) << (4 * i);
        if (__any_sync(0xFFFFFFFFu, (todo & (todo - 1u)) != 0u)) {
          opposite8<DT>(AM, acc, H, T, gc, cc, o, todo);
          continue;
        }
        const int j = todo ? __ffs(todo) - 1 : 0;
        const uint32_t gw = j < 8 ? (j < 4 ? w[0] : w[1]) : (j < 12 ? w[2] : w[3]);
        const uint32_t cw = j < 8 ? (j < 4 ? x[0] : x[1]) : (j < 12 ? x[2] : x[3]);
        const uint32_t G = (gw >> (8 * (j & 3))) & 0xFFu, C = (cw >> (8 * (j & 3))) & 0xFFu;
        if (todo) atomicSub(T + (G * 128u + (C & 0x7Fu)), 1u);
        pair8_slow<DT>(AM, acc, H, G, C, todo != 0u, (uint32_t)(o + j));
        continue;
      }
      // groups at an item's edge
#pragma unroll 1
      for (int j = 0; j < 16; j++) {
        const uint32_t gw = j < 8 ? (j < 4 ? w[0] : w[1]) : (j < 12 ? w[2] : w[3]);
        const uint32_t cw = j < 8 ? (j < 4 ? x[0] : x[1]) : (j < 12 ? x[2] : x[3]);
        const uint32_t G = (gw >> (8 * (j & 3))) & 0xFFu, C = (cw >> (8 * (j & 3))) & 0xFFu;
        const bool ok = o + j >= 0 && o + j < len, slow = ok && ((G ^ C) & 0x80u) != 0u;
        if (ok && !slow) atomicAdd(T + (G * 128u + (C & 0x7Fu)), 1u);
        if (__any_sync(0xFFFFFFFFu, slow)) {
          any_slow = 1;
          pair8_slow<DT>(AM, acc, H, G, C, slow, (uint32_t)(o + j));
        }
      }
    }
    __syncthreads();
    // the combinations that occurred, listed first: a few thousand of 32768,
    // so that every lane evaluates one
    for (int k0 = 0; k0 < CELLS; k0 += 4 * TB) {
      const int k = k0 + 4 * (int)threadIdx.x;
      const uint4 n = *reinterpret_cast<const uint4*>(T + k);
      const uint32_t m = (n.x ? 1u : 0u) | (n.y ? 2u : 0u) | (n.z ? 4u : 0u) | (n.w ? 8u : 0u);
      if (m == 0u) continue;
      int at = atomicAdd(&nlist, __popc(m));
#pragma unroll
      for (int j = 0; j < 4; j++)
        if ((m >> j) & 1u) list[at++] = (unsigned short)(k + j);
    }
    __syncthreads();
    Tot t;
    tot_init(t);
    const int nl = nlist;
#pragma unroll 1
    for (int x = threadIdx.x; x < nl; x += TB) {
      const uint32_t k = list[x], n = T[k], G = k >> 7;
      T[k] = 0u;
      eval_cell<DT>(AM, t, H, G, (G & 0x80u) | (k & 0x7Fu), n);
    }
    block_total(t, warp_tot);
    if (threadIdx.x == 0) store_tot(p.parts + 2 * item, t);  // indices: 0 for a value that occurred
    tot_init(t);
    if (any_slow) {  // (the same for the whole CTA after block_total's barriers)
      acc_to_tot<DT>(t, acc, b - base);
      block_total(t, warp_tot);
    }
    if (threadIdx.x == 0) store_tot(p.parts + 2 * item + 1, t);
    if (p.hist)
      for (int k = threadIdx.x; k < PEAT_HIST_BINS; k += TB)
        if (H[k]) atomicAdd(p.hist + seg * PEAT_HIST_BINS + k, (unsigned long long)H[k]);
    __syncthreads();
  }
}

// thread-block clusters: barrier, a CTA's shared address, minimum into it
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(const void* smem, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(smem)), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_min(uint32_t addr, uint32_t v) {
  asm volatile("red.relaxed.cluster.shared::cluster.min.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// RN64 of a 128-bit magnitude
__device__ double u128_to_double(u128 x) {
  const unsigned long long hi = (unsigned long long)(x >> 64);
  if (hi == 0) return __ull2double_rn((unsigned long long)x);
  const int sh = __clzll((long long)hi);
  const u128 y = x << sh;
  // the top 64 bits, with every lower bit folded into a sticky bit below the rounding position
  const unsigned long long top = (unsigned long long)(y >> 64) | ((unsigned long long)y != 0 ? 1ull : 0ull);
  return ldexp(__ull2double_rn(top), 64 - sh);
}

// The segment's totals (thread 0's t) rounded and written (every thread calls it).
template <int DT>
__device__ void write_stats(const Cmp8Params& p, long long seg, const Tot& t, MeanVarScratch<4, 4, 0>& mv,
                            unsigned long long& nfin) {
  constexpr int S = F8<DT>::S;
  if (threadIdx.x == 0) {
    for (int j = 0; j < 4; j++) {
      mv.A[j] = (uint32_t)(t.s1 >> (32 * j));
      mv.B[j] = (uint32_t)(t.s2 >> (32 * j));
    }
    nfin = t.nfin;
  }
  __syncthreads();
  mean_var_block(mv, nfin, -S);
  if (threadIdx.x != 0) return;
  peat_stats_t r;
  r.n = (uint64_t)(p.offsets[seg + 1] - p.offsets[seg]);
  for (int k = 0; k < PEAT_NCLASS; k++) r.count[k] = t.cnt[k];
  r.n_finite = t.nfin;
  r.max_abs = t.ia >= 0 ? ldexp((double)t.ma, -S) : 0.0;
  r.argmax_abs = t.ia;
  if (t.ir < 0 || t.ra == 0) r.max_rel = 0.0;
  else if (t.rb == 0) r.max_rel = __longlong_as_double(0x7FF0000000000000ll);
  else r.max_rel = __ddiv_rn((double)t.ra, (double)t.rb);  // both exact in binary64: one rounding
  r.argmax_rel = t.ir;
  r.max_ulp = t.iu >= 0 ? t.mu : 0;
  r.argmax_ulp = t.iu;
  r.sum_abs = ldexp(u128_to_double(t.s1), -S);
  r.sum_sq = ldexp(u128_to_double(t.s2), -2 * S);
  const double sdm = ldexp(u128_to_double(t.sd < 0 ? (u128)(-t.sd) : (u128)t.sd), -S);
  r.sum_signed = t.sd < 0 ? -sdm : sdm;
  r.rtol_eff = (double)p.rtol;
  r.atol_eff = (double)p.atol;
  r.mean_abs = mv.mean;
  r.var_abs = mv.var;
  p.stats[seg] = r;
}

// One cluster of CL CTAs per segment: every CTA merges the items (a few KB), and
// the search for the first pair of a maximum is split over them.
constexpr int CL = 8;
template <int DT>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(FB) compare8_finalize(Cmp8Params p) {
  __shared__ Tot warp_tot[FB / 32];
  __shared__ Tot tab, slow;
  __shared__ uint32_t cand[3][256];  // two candidate bytes per golden byte and maximum
  __shared__ unsigned found[3];  // of the cluster's first CTA: offsets in the items
  // S1 = s1 2^-S and S2 = s2 2^-2S: four digits each, no shift between them
  __shared__ MeanVarScratch<4, 4, 0> mv;
  __shared__ unsigned long long nfin;
  pdl_wait();  // stage 1 complete
  const long long seg = blockIdx.x / CL;
  const unsigned rank = blockIdx.x % CL;
  // the items' table values (their index: the item, so that the first one wins
  // a tie) and the records of the pairs of opposite signs
  Tot t;
  tot_init(t);
  for (long long it = p.seg_first[seg] + threadIdx.x; it < p.seg_first[seg + 1]; it += FB) {
    Tot o;
    load_tot(o, p.parts + 2 * it);
    o.ia = o.ia < 0 ? -1 : it;
    o.ir = o.ir < 0 ? -1 : it;
    o.iu = o.iu < 0 ? -1 : it;
    tot_merge(t, o);
  }
  block_total(t, warp_tot);
  if (threadIdx.x == 0) tab = t;
  tot_init(t);
  bool have = false;
  for (long long it = p.seg_first[seg] + threadIdx.x; it < p.seg_first[seg + 1]; it += FB) {
    Tot o;
    load_tot(o, p.parts + 2 * it + 1);
    for (int k = 0; k < PEAT_NCLASS; k++) have = have || o.cnt[k] != 0ull;
    tot_merge(t, o);
  }
  if (__syncthreads_or(have)) block_total(t, warp_tot);
  else tot_init(t);
  if (threadIdx.x == 0) slow = t;
  if (threadIdx.x < 3) found[threadIdx.x] = 0xFFFFFFFFu;
  cluster_sync();
  const uint32_t found0 = cluster_addr(found, 0);
  // The first pair that attains each of the table's maxima, in its item.  Per
  // golden byte at most two candidate bytes attain a given |d|, ratio or
  // ULP distance: a table of them, then one lookup per pair; the three items'
  // loads go out together.
  const long long base0 = p.offsets[seg];
  long long where[3];
  const unsigned char *gp[3], *cp[3];
  unsigned len[3], head[3], mine[3];
#pragma unroll
  for (int m = 0; m < 3; m++) {
    const long long it = m == 0 ? tab.ia : (m == 1 ? tab.ir : tab.iu);
    const bool use = it >= 0 && !(m == 0   ? slow.ia >= 0 && slow.ma > tab.ma
                                  : m == 1 ? slow.ir >= 0 && cmp_frac(slow.ra, slow.rb, tab.ra, tab.rb) > 0
                                           : slow.iu >= 0 && slow.mu > tab.mu);
    const long long b = use ? p.item_b[it] : 0;
    where[m] = use ? b - base0 : -1;
    len[m] = use ? (unsigned)(p.item_e[it] - b) : 0u;
    gp[m] = reinterpret_cast<const unsigned char*>(p.g) + b;
    cp[m] = reinterpret_cast<const unsigned char*>(p.c) + b;
    head[m] = p.vec ? min(len[m], (unsigned)((16 - (b & 15)) & 15)) : len[m];
    mine[m] = 0xFFFFFFFFu;
  }
  for (int x = threadIdx.x; x < 3 * 256; x += FB) {
    const uint32_t m = (uint32_t)x >> 8, G = (uint32_t)x & 0xFFu, mg = G & 0x7Fu;
    const int kg = f8_kind<DT>(mg);
    constexpr uint32_t none = 0xFFFFu;  // no byte
    uint32_t c1 = none, c2 = none;
    if (m == 2) {
      const uint32_t u = (uint32_t)tab.mu;
      if (kg != 2 && mg + u < 128u && f8_kind<DT>(mg + u) != 2) c1 = mg + u;
      if (kg != 2 && mg >= u) c2 = mg - u;
    } else if (kg == 0) {
      const uint32_t Kg = f8_units<DT>(mg);
      unsigned long long a = tab.ma;
      bool ok = true;
      if (m == 1) {
        if (tab.rb == 0) {  // +inf: golden zero, any other value (searched below as a special case)
          ok = false;
        } else {
          const u128 q = (u128)tab.ra * Kg;
          ok = q % tab.rb == 0 && (q / tab.rb != 0 || tab.ra == 0);
          a = (unsigned long long)(q / tab.rb);
        }
      }
      if (ok) {
        c1 = f8_encode<DT>(Kg + a, none);
        c2 = a <= Kg ? f8_encode<DT>(Kg - a, none) : none;
        if (m == 1 && Kg == 0 && tab.ra != 0) c1 = c2 = none;
        if (m == 1 && Kg == 0 && tab.ra == 0) c1 = c2 = 0u;
      }
    }
    const uint32_t sg = G & 0x80u;
    cand[m][G] = (c1 | (c1 == none ? 0u : sg)) | ((c2 | (c2 == none ? 0u : sg)) << 16);
  }
  __syncthreads();
  const bool zero_golden = tab.ir >= 0 && tab.rb == 0;
  auto hit = [&](int m, uint32_t G, uint32_t C) {
    if (m == 1 && zero_golden)
      return (G & 0x7Fu) == 0u && ((G ^ C) & 0x80u) == 0u && (C & 0x7Fu) != 0u && f8_kind<DT>(C & 0x7Fu) == 0;
    const uint32_t w = cand[m][G];
    return C == (w & 0xFFFFu) || C == (w >> 16);
  };
  const unsigned t0 = rank * FB + threadIdx.x;
  unsigned nv[3], most = 0;
#pragma unroll
  for (int m = 0; m < 3; m++) {
    for (unsigned i = t0; i < head[m] && mine[m] == 0xFFFFFFFFu; i += CL * FB)
      if (hit(m, gp[m][i], cp[m][i])) mine[m] = i;
    nv[m] = (len[m] - head[m]) >> 4;
    most = max(most, nv[m]);
  }
  for (unsigned q = t0; q < most; q += CL * FB) {
    uint4 gv[3], cv[3];
    bool on[3];
#pragma unroll
    for (int m = 0; m < 3; m++) {
      on[m] = q < nv[m] && mine[m] == 0xFFFFFFFFu;
      gv[m] = cv[m] = make_uint4(0, 0, 0, 0);
      if (on[m]) {
        gv[m] = __ldg(reinterpret_cast<const uint4*>(gp[m] + head[m]) + q);
        cv[m] = __ldg(reinterpret_cast<const uint4*>(cp[m] + head[m]) + q);
      }
    }
#pragma unroll
    for (int m = 0; m < 3; m++) {
      if (!on[m]) continue;
      const uint32_t w[4] = {gv[m].x, gv[m].y, gv[m].z, gv[m].w}, x[4] = {cv[m].x, cv[m].y, cv[m].z, cv[m].w};
#pragma unroll
      for (int j = 15; j >= 0; j--)
        if (hit(m, (w[j >> 2] >> (8 * (j & 3))) & 0xFFu, (x[j >> 2] >> (8 * (j & 3))) & 0xFFu)) mine[m] = head[m] + 16 * q + j;
    }
  }
#pragma unroll
  for (int m = 0; m < 3; m++) {
    for (unsigned i = head[m] + 16 * nv[m] + t0; i < len[m] && mine[m] == 0xFFFFFFFFu; i += CL * FB)
      if (hit(m, gp[m][i], cp[m][i])) mine[m] = i;
    mine[m] = __reduce_min_sync(0xFFFFFFFFu, mine[m]);
    if ((threadIdx.x & 31) == 0 && mine[m] != 0xFFFFFFFFu) cluster_min(found0 + 4u * m, mine[m]);
  }
  cluster_sync();
  if (rank != 0) return;
  for (int m = 0; m < 3; m++)
    if (where[m] >= 0) where[m] += found[m];
  if (threadIdx.x == 0) {
    // both kinds together; a table value equal to a record's takes the lower index
    t = slow;
    Tot o = tab;
    o.ia = where[0], o.ir = where[1], o.iu = where[2];
    tot_merge(t, o);
  }
  write_stats<DT>(p, seg, t, mv, nfin);
}

// the same for items of compare8_direct, one record each
template <int DT>
__global__ void __launch_bounds__(DTB) compare8_finalize_direct(Cmp8Params p) {
  __shared__ Tot warp_tot[DTB / 32];
  __shared__ MeanVarScratch<4, 4, 0> mv;
  __shared__ unsigned long long nfin;
  pdl_wait();
  const long long seg = blockIdx.x;
  Tot t;
  tot_init(t);
  for (long long it = p.seg_first[seg] + threadIdx.x; it < p.seg_first[seg + 1]; it += DTB) {
    Tot o;
    load_tot(o, p.parts + it);
    tot_merge(t, o);
  }
  block_total(t, warp_tot);
  write_stats<DT>(p, seg, t, mv, nfin);
}

template <int DT>
cudaError_t launch_t(const Cmp8Params& p, int nctas, cudaStream_t s) {
  if (p.nitems == 0) {
    compare8_finalize_direct<DT><<<(unsigned)p.nseg, DTB, 0, s>>>(p);
    return cudaGetLastError();
  }
  if (p.direct) {
    compare8_direct<DT><<<nctas, DTB, 0, s>>>(p);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_dependent(compare8_finalize_direct<DT>, (unsigned)p.nseg, DTB, 0, s, p);
  }
  compare8_stage1<DT><<<nctas, TB, SMEM8, s>>>(p);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_dependent(compare8_finalize<DT>, (unsigned)p.nseg * CL, FB, 0, s, p);  // overlaps stage 1's end
}

}  // namespace

// once per device, before the first launch
cudaError_t compare8_prepare() {
  cudaError_t e = cudaFuncSetAttribute(compare8_stage1<PEAT_F8E4M3>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM8);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(compare8_stage1<PEAT_F8E5M2>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM8);
  return e;
}

cudaError_t launch_compare8(int dtype, const Cmp8Params& p, int nctas, cudaStream_t s) {
  switch (dtype) {
    case PEAT_F8E4M3: return launch_t<PEAT_F8E4M3>(p, nctas, s);
    case PEAT_F8E5M2: return launch_t<PEAT_F8E5M2>(p, nctas, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace peat
