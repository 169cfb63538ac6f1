// Shared parts of the ungrouped scans (plain, host-fed, allocation-free and
// bit-packed columns): the per-thread accumulators (the fold of Fig. 4), the
// block partials with their error bound, the fixed-order warp and block
// reduction and the merge of block partials into one result.
#pragma once

#include <cfloat>
#include <climits>
#include <cmath>

#include "common.cuh"

namespace agg {

// One block's partial aggregate (48 bytes). Integer columns use w0 (the sum mod
// 2^64); float columns hold their sum as the 128-bit fixed-point number w1:w0
// of Fix128 at the scale of exponent E, so that warps, blocks and the grid
// merge with integer additions: GB300 issues few float64 operations, and a
// float64 TwoSum in every shuffle step made a 2^20-row int32 scan 17 us long
// and put 40 us on every float64 scan. What a merge shifts below the unit goes
// to rest, in float64: nothing in a column whose rows lie within some 30
// binades of each other, and in any other what keeps a sum right whose largest
// rows cancel.
struct Partial {
  uint64_t w0, w1;
  uint64_t mn, mx;   // order-preserving images of min / max
  double rest;       // float: the sum's part below the unit of w1:w0
  int16_t E;         // exponent field the fixed-point sum is scaled to (0: no value yet)
  uint16_t special;  // float: kPosInf | kNegInf | kNan seen
  float eb;          // float32: bound on the roundings of the threads' compensation words
};
static_assert(sizeof(Partial) == 48, "partials of the static scratch");
constexpr uint32_t kPosInf = 1, kNegInf = 2, kNan = 4;

template <int DT> struct Traits;
template <> struct Traits<AGG_I32> { using T = int32_t; static constexpr bool FP = false; };
template <> struct Traits<AGG_I64> { using T = int64_t; static constexpr bool FP = false; };
template <> struct Traits<AGG_U32> { using T = uint32_t; static constexpr bool FP = false; };
template <> struct Traits<AGG_F32> { using T = float; static constexpr bool FP = true; };
template <> struct Traits<AGG_F64> { using T = double; static constexpr bool FP = true; };

// ---------------------------------------------------------------------------
// Per-thread accumulators. fold() is the aggregate() of Fig. 4.
// ---------------------------------------------------------------------------
template <int DT, bool SUM, bool MM, bool FP = Traits<DT>::FP>
struct Acc;

template <int DT, bool SUM, bool MM>
struct Acc<DT, SUM, MM, false> {
  using T = typename Traits<DT>::T;
  int64_t s;
  T mn, mx;
  __device__ void init() {
    s = 0;
    if (DT == AGG_I32) { mn = (T)INT_MAX; mx = (T)INT_MIN; }
    if (DT == AGG_U32) { mn = (T)UINT_MAX; mx = (T)0; }
    if (DT == AGG_I64) { mn = (T)LLONG_MAX; mx = (T)LLONG_MIN; }
  }
  __device__ __forceinline__ void fold(T v) {
    if (SUM) s += (int64_t)v;
    if (MM) { mn = min(mn, v); mx = max(mx, v); }
  }
  __device__ __forceinline__ void fold_vec(const uint4& r) {
    if (sizeof(T) == 4) {
      fold((T)r.x); fold((T)r.y); fold((T)r.z); fold((T)r.w);
    } else {
      fold((T)(((uint64_t)r.y << 32) | r.x));
      fold((T)(((uint64_t)r.w << 32) | r.z));
    }
  }
  __device__ void to_partial(Partial& p, uint32_t) const {
    p = Partial{};
    p.w0 = (uint64_t)s;
    p.mn = img_i64((int64_t)mn);
    p.mx = img_i64((int64_t)mx);
  }
};

template <class F> struct FpImg;
template <> struct FpImg<float> {
  using U = uint32_t;
  __device__ static U img(float x) { return img_f32(x); }
  __device__ static double value(uint64_t m) { return (double)f32_of_img((uint32_t)m); }
};
template <> struct FpImg<double> {
  using U = uint64_t;
  __device__ static U img(double x) { return img_f64(x); }
  __device__ static double value(uint64_t m) { return f64_of_img(m); }
};

// float64 SUM on the integer pipes: a 128-bit two's-complement fixed-point
// number (hi:lo) scaled to the largest exponent field E seen so far, worth
// (hi:lo) x 2^(E - 1075 - kFixGuard). A row with significand m (53 bits,
// implicit bit included) and exponent field e >= 1 is worth m x 2^(e - 1075),
// i.e. m shifted left by kFixGuard - (E - e) units. Rows more than kFixGuard
// binades below E reach into a further word ext, whose unit is 2^-64 of that of
// lo (a row loses less than that, 2^-147 of the largest row); a row with a larger
// exponent shifts the sum right (again less than a unit of ext lost). Sums of up to
// 2^43 rows per thread cannot overflow (|m x 2^kFixGuard| < 2^84). A guard of
// 31 bits keeps the fast path's shift below one word. Infinities and NaNs are noted
// on the side, so that a column holding one sums to a non-finite value.
// GB300 issues few float64 operations per clock (a TwoSum per row held the
// float64 scan to 0.6 TB/s); this takes only integer operations per row.
// E starts at kFixFirst, where the unit is the smallest subnormal: nothing is
// lost there, and the exponent field of a subnormal (0) lies below every base,
// so that one test on the high word selects the fast path.
constexpr int kFixGuard = 31;
constexpr int kFixFirst = kFixGuard + 1;

// x 2^k for -1140 <= k <= 1022, rounded at most once (two normal factors).
__device__ __forceinline__ double scaled(double x, int k) {
  const int h = k / 2;
  return x * __hiloint2double((h + 1023) << 20, 0) * __hiloint2double((k - h + 1023) << 20, 0);
}

struct Fix128 {
  uint64_t lo, hi;
  uint64_t ext;   // the bits below lo's unit (slow path only)
  uint32_t nneg;  // negative rows added on the fast path as ~v, each still owing +1
  int E;
  uint32_t base;  // (E - kFixGuard) << 20: a row's high word minus this holds the row's shift
  uint32_t special;  // kPosInf | kNegInf | kNan
  __device__ void init() {
    lo = 0;
    hi = 0;
    ext = 0;
    nneg = 0;
    E = kFixFirst;
    base = 1u << 20;
    special = 0;
  }
  // Scale for rows of exponent fields up to ef + 1, where the thread's own first
  // rows reach up to own: at most 64 binades above those, so that ext still holds
  // every bit that a scale of the thread's own rows would (the sum so far is zero
  // or exact).
  __device__ __forceinline__ void start(uint32_t ef, uint32_t own) {
    if (ef == 0x7FFu) return;
    ef = min(min(ef, own + 63u), 0x7FDu);
    if (ef > 0 && (int)ef >= E) rescale((int)ef + 1);
  }
  // -v = ~v + 1: the fast path adds ~v and counts the +1s, added here.
  __device__ __forceinline__ void fold_neg() {
    lo += nneg;
    hi += lo < nneg ? 1ull : 0ull;
    nneg = 0;
  }
  // (vhi:vlo) >> k for 1 <= k < 127, rounding toward minus infinity (less than one unit).
  __device__ static __forceinline__ void shift_right(uint64_t& vlo, uint64_t& vhi, int k) {
    if (k >= 64) {
      vlo = (uint64_t)((int64_t)vhi >> (k - 64));
      vhi = (uint64_t)((int64_t)vhi >> 63);
    } else {
      vlo = (vlo >> k) | (vhi << (64 - k));
      vhi = (uint64_t)((int64_t)vhi >> k);
    }
  }
  __device__ __forceinline__ void rescale(int e) {  // e > E
    fold_neg();
    int k = e - E;
    if (k >= 191) {  // nothing of the sum reaches ext's unit
      ext = lo = hi = 0;
      k = 0;
    }
    for (; k >= 64; k -= 64) {
      ext = lo;
      lo = hi;
      hi = (uint64_t)((int64_t)hi >> 63);
    }
    if (k > 0) {
      ext = (ext >> k) | (lo << (64 - k));
      shift_right(lo, hi, k);
    }
    E = e;
    base = (uint32_t)(e - kFixGuard) << 20;
  }
  // A row's high word relative to base. Bits 20 to 30 hold ef - (E - kFixGuard)
  // mod 2^11 (1 <= E - kFixGuard <= 2015): the shift, 0 to 31, of a normal value
  // within kFixGuard binades of E, and 32 or more (a bit of kFixOut is set) for
  // every other row.
  static constexpr uint32_t kFixOut = 0x7E000000u;
  __device__ __forceinline__ uint32_t rel(uint32_t uh) const { return uh - base; }
  // A row on the fast path (x = rel(uh)): its 53-bit significand m, in one's
  // complement when negative (the +1 counted in nneg), shifted left by less
  // than 32 on 32-bit words (three funnel shifts, which use the low five bits of
  // the amount), added with one carry chain.
  __device__ __forceinline__ void add_fast(uint32_t uh, uint32_t ul, uint32_t x) {
    static_assert(kFixGuard == 31, "the fast path shifts by less than one word");
    const unsigned sh = x >> 20;
    const uint32_t s = (uint32_t)((int32_t)uh >> 31);            // all ones for a negative row
    const uint32_t mh = ((uh & 0x000FFFFFu) | 0x00100000u) ^ s;  // m's high 21 bits (implicit bit included)
    const uint32_t ml = ul ^ s;
    const uint32_t x0 = __funnelshift_l(s, ml, sh);
    const uint32_t x1 = __funnelshift_l(ml, mh, sh);
    const uint32_t x2 = __funnelshift_l(mh, s, sh);  // m >> (32 - sh), 0 when sh = 0
    const uint32_t x3 = s;
    asm("{\n\t.reg .u32 a0, a1, a2, a3;\n\t"
        "mov.b64 {a0, a1}, %0;\n\t"
        "mov.b64 {a2, a3}, %1;\n\t"
        "add.cc.u32 a0, a0, %2;\n\t"
        "addc.cc.u32 a1, a1, %3;\n\t"
        "addc.cc.u32 a2, a2, %4;\n\t"
        "addc.u32 a3, a3, %5;\n\t"
        "mov.b64 %0, {a0, a1};\n\t"
        "mov.b64 %1, {a2, a3};\n\t}"
        : "+l"(lo), "+l"(hi)
        : "r"(x0), "r"(x1), "r"(x2), "r"(x3));
    nneg -= s;
  }
  // Any row. (Not through add_fast where that would do: a warp with a row outside
  // the window would take both paths one after the other.)
  __device__ __forceinline__ void add(uint64_t u) {
    const uint32_t uh = (uint32_t)(u >> 32);
    uint32_t ml = (uint32_t)u;
    if (((uh << 1) | ml) == 0u) return;
    const int ef = (int)((uh >> 20) & 0x7FFu);
    if (ef > E) {
      if (ef == 0x7FF) {  // infinity or NaN
        special |= (u & 0x000FFFFFFFFFFFFFull) ? kNan : (int64_t)u < 0 ? kNegInf : kPosInf;
        return;
      }
      rescale(ef);
    }
    // The significand m (subnormals: exponent 1, no implicit bit) in units of ext
    // is m shifted left by kFixGuard + 64 - (E - e): three words x0, x1, x2 at
    // word q of the six words hi:lo:ext.
    uint32_t mh = (uh & 0x000FFFFFu) | (ef > 0 ? 0x00100000u : 0u);
    int sh = kFixGuard + 64 - E + max(ef, 1);
    if (sh < 0) {
      const uint64_t m = sh > -64 ? (((uint64_t)mh << 32) | ml) >> -sh : 0ull;
      ml = (uint32_t)m;
      mh = (uint32_t)(m >> 32);
      sh = 0;
    }
    const int q = sh >> 5;  // 0 to 2
    const uint32_t s = (uint32_t)((int32_t)uh >> 31);  // a negative row: the complement, plus one
    const uint32_t x0 = __funnelshift_l(0u, ml, sh) ^ s;
    const uint32_t x1 = __funnelshift_l(ml, mh, sh) ^ s;
    const uint32_t x2 = __funnelshift_l(mh, 0u, sh) ^ s;
    asm("{\n\t.reg .u32 t, a0, a1, a2, a3, a4, a5;\n\t"
        "mov.b64 {a0, a1}, %0;\n\t"
        "mov.b64 {a2, a3}, %1;\n\t"
        "mov.b64 {a4, a5}, %2;\n\t"
        "add.cc.u32 t, %8, %8;\n\t"  // carry: the sign
        "addc.cc.u32 a0, a0, %3;\n\t"
        "addc.cc.u32 a1, a1, %4;\n\t"
        "addc.cc.u32 a2, a2, %5;\n\t"
        "addc.cc.u32 a3, a3, %6;\n\t"
        "addc.cc.u32 a4, a4, %7;\n\t"
        "addc.u32 a5, a5, %8;\n\t"
        "mov.b64 %0, {a0, a1};\n\t"
        "mov.b64 %1, {a2, a3};\n\t"
        "mov.b64 %2, {a4, a5};\n\t}"
        : "+l"(ext), "+l"(lo), "+l"(hi)
        : "r"(q == 0 ? x0 : s), "r"(q == 0 ? x1 : q == 1 ? x0 : s), "r"(q == 0 ? x2 : q == 1 ? x1 : x0),
          "r"(q == 1 ? x2 : q == 2 ? x1 : s), "r"(q == 2 ? x2 : s), "r"(s));
  }
};

// The sum of a partial without its rest, as an unevaluated float64 pair (rel.
// error about 2^-106 before scaling): the 128-bit integer in three chunks that
// float64 holds exactly, added with TwoSum, then scaled by 2^(E - 1075 - kFixGuard).
__device__ inline void fix_to_pair(const Partial& p, double& h, double& l) {
  const uint64_t lo = p.w0, hi = p.w1;
  const uint64_t m43 = (1ull << 43) - 1ull;
  const double q0 = (double)(lo & m43);
  const double q1 = (double)(((lo >> 43) | (hi << 21)) & m43);
  const double q2 = (double)((int64_t)hi >> 22);
  double s1, e1, s2, e2;
  two_sum(q2 * 0x1p86, q1 * 0x1p43, s1, e1);
  two_sum(s1, q0, s2, e2);
  double t, f;
  two_sum(s2, e1 + e2, t, f);
  const int sc = p.E - 1075 - kFixGuard;
  h = ldexp(t, sc);
  l = ldexp(f, sc);
  if (p.special) {  // both infinities, or a NaN: NaN
    l = 0.0;
    h = __longlong_as_double(p.special == kPosInf   ? 0x7ff0000000000000ll
                             : p.special == kNegInf ? (long long)0xfff0000000000000ull
                                                    : 0x7ff8000000000000ll);
  }
}

template <int DT, bool SUM, bool MM>
struct Acc<DT, SUM, MM, true> {
  using T = typename Traits<DT>::T;
  using U = typename FpImg<T>::U;
  static constexpr bool F64 = sizeof(T) == 8;
  T s, c;       // float32: TwoSum-compensated pair
  T cmax;       // float32: largest |c| so far (bounds the roundings of c)
  Fix128 fx;    // float64
  U mn, mx;
  __device__ void init() {
    s = 0; c = 0; cmax = 0;
    if (F64) fx.init();
    mn = (U)~(U)0; mx = 0;
  }
  __device__ __forceinline__ void fold(T v) {
    if (SUM) {
      if (F64) {
        fx.add((uint64_t)__double_as_longlong((double)v));
      } else {
        T t, e;
        two_sum(s, v, t, e);
        s = t;
        c += e;
        cmax = fmaxf(cmax, fabsf(c));
      }
    }
    if (MM) {
      if (F64) {
        // the image's high word decides unless it ties with an extreme's:
        // the 64-bit compares run only for a row that may move min or max
        const uint64_t b = (uint64_t)__double_as_longlong((double)v);
        const uint32_t s = (uint32_t)((int32_t)(b >> 32) >> 31);
        const uint32_t ih = (uint32_t)(b >> 32) ^ (s | 0x80000000u);
        if (ih <= (uint32_t)((uint64_t)mn >> 32) || ih >= (uint32_t)((uint64_t)mx >> 32)) {
          const U m = (U)(((uint64_t)ih << 32) | ((uint32_t)b ^ s));
          mn = min(mn, m);
          mx = max(mx, m);
        }
      } else {
        U m = FpImg<T>::img(v);
        mn = min(mn, m);
        mx = max(mx, m);
      }
    }
  }
  __device__ __forceinline__ void fold_vec(const uint4& r) {
    if (sizeof(T) == 4) {
      fold(__uint_as_float(r.x)); fold(__uint_as_float(r.y));
      fold(__uint_as_float(r.z)); fold(__uint_as_float(r.w));
    } else {
      // two rows share the tests for the fixed-point sum's fast path and for a
      // high word that may move an extreme
      if (SUM) {
        const uint32_t x0 = fx.rel(r.y), x1 = fx.rel(r.w);
        if (((x0 | x1) & Fix128::kFixOut) == 0u) {
          fx.add_fast(r.y, r.x, x0);
          fx.add_fast(r.w, r.z, x1);
        } else {
          fx.add(((uint64_t)r.y << 32) | r.x);
          fx.add(((uint64_t)r.w << 32) | r.z);
        }
      }
      if (MM) {
        const uint32_t s0 = (uint32_t)((int32_t)r.y >> 31), s1 = (uint32_t)((int32_t)r.w >> 31);
        const uint32_t h0 = r.y ^ (s0 | 0x80000000u), h1 = r.w ^ (s1 | 0x80000000u);
        if (min(h0, h1) <= (uint32_t)((uint64_t)mn >> 32) || max(h0, h1) >= (uint32_t)((uint64_t)mx >> 32)) {
          const U m0 = (U)(((uint64_t)h0 << 32) | (r.x ^ s0)), m1 = (U)(((uint64_t)h1 << 32) | (r.z ^ s1));
          mn = min(mn, min(m0, m1));
          mx = max(mx, max(m0, m1));
        }
      }
    }
  }
  // float64 MIN/MAX, all lanes of the warp: every lane's extremes take the
  // warp's high words, with low words that no value of theirs lies beyond (the
  // lane that holds the warp's extreme keeps it). Only rows that may move the
  // warp's extremes then pass the filter, not all that move one lane's.
  __device__ __forceinline__ void share_extremes() {
    const uint32_t lo = __reduce_min_sync(0xffffffffu, (uint32_t)((uint64_t)mn >> 32));
    const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)((uint64_t)mx >> 32));
    mn = min(mn, (U)(((uint64_t)lo << 32) | 0xFFFFFFFFull));
    mx = max(mx, (U)((uint64_t)hi << 32));
  }
  // rows: the number of values this thread folded.
  __device__ void to_partial(Partial& p, uint32_t rows) const {
    p = Partial{};
    if (SUM) {
      Fix128 f = fx;
      if (!F64) {
        // the float32 pair as two rows of a fixed-point sum (s's exponent and
        // 31 binades below it: all of c's bits but a guard's worth)
        f.init();
        f.add((uint64_t)__double_as_longlong((double)s));
        f.add((uint64_t)__double_as_longlong((double)c));
        // TwoSum leaves s + c short only by the roundings of c: each at most
        // 2^-24 of |c| after the add (2^-150 when c is subnormal)
        p.eb = __fmul_ru(__uint2float_ru(rows), __fadd_ru(__fmul_ru((float)cmax, 0x1.000002p-24f), 0x1p-149f));
      }
      f.fold_neg();
      p.w0 = f.lo;
      p.w1 = f.hi;
      if (f.ext != 0) {  // to the nearest unit (see lower_scale)
        if ((int64_t)f.ext < 0 && ++p.w0 == 0) ++p.w1;
        p.rest = scaled((double)(int64_t)f.ext, f.E - 1075 - kFixGuard - 64);
      }
      p.E = (int16_t)f.E;
      p.special = (uint16_t)f.special;
    }
    p.mn = mn == (U)~(U)0 ? ~0ull : (uint64_t)mn;
    p.mx = mx;
  }
};

// ---------------------------------------------------------------------------
// Warp / block reduction of Partial values (fixed shuffle tree).
// ---------------------------------------------------------------------------
// w1:w0 at the scale of E moved to that of E + k (1 <= k), to the nearest unit: what
// that leaves, half a unit at most, is returned, rounded to float64. (Rounded down,
// what a small negative sum leaves would be nearly a unit, and its own bits lost.)
__device__ __forceinline__ double lower_scale(uint64_t& w0, uint64_t& w1, int E, int k) {
  uint64_t l0, l1;  // what is left, two's complement
  if (k < 127) {
    const uint64_t h0 = k <= 64 ? 1ull << (k - 1) : 0ull, h1 = k > 64 ? 1ull << (k - 65) : 0ull;  // half a unit
    w0 += h0;
    w1 += h1 + (w0 < h0 ? 1ull : 0ull);
    l0 = k < 64 ? w0 & ((1ull << k) - 1ull) : w0;
    l1 = k > 64 ? w1 & ((1ull << (k - 64)) - 1ull) : 0ull;
    Fix128::shift_right(w0, w1, k);
    l1 -= h1 + (l0 < h0 ? 1ull : 0ull);
    l0 -= h0;
  } else {  // below half a unit
    l0 = w0;
    l1 = w1;
    w0 = w1 = 0;
  }
  if ((l0 | l1) == 0) return 0.0;
  const bool neg = (int64_t)l1 < 0;
  if (neg) {
    l0 = 0ull - l0;
    l1 = ~l1 + (l0 == 0 ? 1ull : 0ull);
  }
  const double d = scaled(fma((double)l1, 18446744073709551616.0, (double)l0), E - 1075 - kFixGuard);
  return neg ? -d : d;
}

// The sum of a partial moved to the scale of exponent E >= its own.
__device__ __forceinline__ void raise_scale(Partial& p, int E) {
  if (p.E == E) return;
  const double d = lower_scale(p.w0, p.w1, p.E, E - p.E);
  if (d != 0.0) p.rest += d;
  p.E = (int16_t)E;
}

template <bool FP>
__device__ __forceinline__ void combine(Partial& a, Partial b) {
  if (FP) {
    const int E = max(a.E, b.E);
    raise_scale(a, E);
    raise_scale(b, E);
    a.w0 += b.w0;
    a.w1 += b.w1 + (a.w0 < b.w0 ? 1ull : 0ull);
    if (b.rest != 0.0) a.rest += b.rest;
    a.special |= b.special;
    a.eb = __fadd_ru(a.eb, b.eb);
  } else {
    a.w0 += b.w0;
  }
  a.mn = min(a.mn, b.mn);
  a.mx = max(a.mx, b.mx);
}

__device__ __forceinline__ Partial empty_partial() {
  Partial p{};
  p.mn = ~0ull;
  return p;
}

__device__ __forceinline__ uint64_t warp_min64(uint64_t v) {  // the high words' minimum, then the low words of the lanes holding it
  const uint32_t h = __reduce_min_sync(0xffffffffu, (uint32_t)(v >> 32));
  return ((uint64_t)h << 32) | __reduce_min_sync(0xffffffffu, (uint32_t)(v >> 32) == h ? (uint32_t)v : 0xFFFFFFFFu);
}

// The lanes' partials (the first LANES of them hold one), in lane 0. Floats: all
// lanes take the largest exponent's scale first, so that the sums are plain
// integer additions (with a shift in every step, the end of a float scan was 7 us
// longer); the float64 parts below the unit are added only when a lane has one.
template <bool FP, int LANES>
__device__ __forceinline__ void warp_combine(Partial& p) {
  constexpr unsigned kAll = 0xffffffffu;
  if (FP) {
    raise_scale(p, (int)__reduce_max_sync(kAll, (uint32_t)p.E));
    p.special = (uint16_t)__reduce_or_sync(kAll, p.special);
    if (__any_sync(kAll, p.rest != 0.0)) {
#pragma unroll 1
      for (int m = LANES / 2; m >= 1; m >>= 1) p.rest += __shfl_xor_sync(kAll, p.rest, m);
    }
  }
#pragma unroll
  for (int m = LANES / 2; m >= 1; m >>= 1) {
    const uint64_t b0 = __shfl_xor_sync(kAll, p.w0, m);
    p.w0 += b0;
    if (FP) {
      p.w1 += __shfl_xor_sync(kAll, p.w1, m) + (p.w0 < b0 ? 1ull : 0ull);
      p.eb = __fadd_ru(p.eb, __shfl_xor_sync(kAll, p.eb, m));
    }
  }
  p.mn = warp_min64(p.mn);
  p.mx = ~warp_min64(~p.mx);
}

// Block-wide reduction; the result is valid in thread 0.
template <bool FP, int BLOCK>
__device__ Partial block_reduce(Partial p) {
  __shared__ Partial sm[BLOCK / 32];
  warp_combine<FP, 32>(p);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sm[w] = p;
  __syncthreads();
  if (w == 0) {
    p = l < BLOCK / 32 ? sm[l] : empty_partial();
    warp_combine<FP, BLOCK / 32>(p);
  }
  return p;
}

// Merge np partials (written by other blocks or launches) into *out.
// Called by one whole block; thread 0 writes.
template <int DT, int BLOCK>
__device__ void merge_partials(const Partial* parts, int np, agg_scalar* out, uint32_t ops,
                               int64_t count) {
  constexpr bool FP = Traits<DT>::FP;
  Partial acc = empty_partial();
  for (int i = threadIdx.x; i < np; i += BLOCK) {
    const uint4* q4 = reinterpret_cast<const uint4*>(&parts[i]);
    union {
      uint4 v[3];
      Partial p;
    } q;
#pragma unroll
    for (int k = 0; k < 3; ++k) q.v[k] = __ldcg(q4 + k);
    combine<FP>(acc, q.p);
  }
  __syncthreads();
  acc = block_reduce<FP, BLOCK>(acc);
  if (threadIdx.x != 0) return;
  agg_scalar r;
  r.count = count;
  r.dtype = DT;
  r.ops = ops;
  r.err_bound = 0.0;
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  if constexpr (FP) {
    const double inf = __longlong_as_double(0x7ff0000000000000ll);
    double hi, lo;
    fix_to_pair(acc, hi, lo);
    double s = hi + lo;
    const double parts = fabs(hi) + fabs(acc.rest);
    if (acc.rest != 0.0 && isfinite(s)) {
      double e;
      two_sum(hi, acc.rest, s, e);
      s += e + lo;
    }
    r.sum_i = 0;
    r.sum_f = s;
    // Bound on |s - exact sum|: the threads' compensation words (float32); the
    // rounding of what is below the unit, a thread's ext word and the part that
    // a merge shifts out (each less than a unit, 2^-52 of it lost), and of the
    // additions to rest (2^-53 of at most a unit per row merged, at a depth of
    // less than 2^20): 2^-30 of a unit a row holds all of it, and the rows'
    // 2^-64; fix_to_pair and the addition of rest (under 2^-100 of the parts,
    // and the subnormal range); the rounding of the result and the oracle's own
    // rounding of the exact sum (each at most 2^-53 of the value); and a margin
    // for the roundings of the bound's own sums.
    if (ops & (AGG_SUM | AGG_AVG)) {
      const double units = acc.E > kFixFirst ? ldexp((double)count, acc.E - 1075 - kFixGuard - 30) : 0.0;
      r.err_bound = ((double)acc.eb + units + fabs(s) * 0x1p-52 + parts * 0x1p-99 + 0x1p-1072) * (1.0 + 0x1p-40);
      // a column holding an infinity or a NaN has no finite bound
      if (acc.special || !isfinite(s) || !isfinite(r.err_bound)) r.err_bound = inf;
    }
    r.avg = count ? s / (double)count : nan;
    r.min_f = count ? FpImg<typename Traits<DT>::T>::value(acc.mn) : inf;
    r.max_f = count ? FpImg<typename Traits<DT>::T>::value(acc.mx) : -inf;
    r.min_i = 0;
    r.max_i = 0;
  } else {
    r.sum_i = (int64_t)acc.w0;
    r.sum_f = (double)r.sum_i;
    r.avg = count ? r.sum_f / (double)count : nan;
    r.min_i = count ? i64_of_img(acc.mn) : LLONG_MAX;
    r.max_i = count ? i64_of_img(acc.mx) : LLONG_MIN;
    r.min_f = 0.0;
    r.max_f = 0.0;
  }
  *out = r;
}

constexpr int kBlock = 256;
constexpr int kUnroll = 4;

}  // namespace agg
