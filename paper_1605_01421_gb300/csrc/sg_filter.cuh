// sg_filter.cuh -- decisions of the direct method from FP32 intervals.
//
// A draw of the direct method (Appendix A) decides two things: whether the
// next event falls before the next unit time (t + tau < Tn, tau = E / lambda,
// E = -log r1) and which transition fires (the first running sum of the rates
// that reaches lambda r2).  Both sides are defined in FP64, and GB300 issues
// one FP64 warp instruction per sub-partition every ~76 cycles (an FP32 one
// every cycle), so here every FP64 quantity x is enclosed in an interval
// [lo, hi] of FP32 numbers, lo <= x <= hi, and a decision is taken from the
// intervals only where they settle it; where they overlap it is taken in
// FP64 (the transition: on the spot; the event time: the unit's day is run
// again with exact times).  The trajectory is therefore the FP64 one, bit for
// bit.
//
// Why the enclosures hold.  FP32 numbers are FP64 numbers, and rounding is
// monotone: from lo <= y <= hi with lo and hi in FP64 follows lo <= RN64(y)
// <= hi.  So an operation on intervals with its ends rounded outward (the
// _rd / _ru intrinsics) encloses the FP64 operation, rounding included, and
// an FP64 expression is enclosed by the same expression on intervals.
// Overflow in FP32 gives an infinite or NaN end, which settles nothing.
#pragma once

#include "sg_device.cuh"

namespace sg {

struct Itv {
  float lo, hi;
};

constexpr float kItvMax = 0x1.0p100f, kItvMin = 0x1.0p-100f;

__device__ __forceinline__ Itv itv_nan() {
  const float q = __int_as_float(0x7fffffff);
  return Itv{q, q};
}

// Hardware reciprocal and base-2 logarithm.  PTX bounds them: rcp.approx
// within 1 ulp (relative 2^-23) of 1 / x for normal x whose reciprocal is
// normal; lg2.approx within 2^-22 absolutely for x in (0.5, 2), within 2^-22
// relatively elsewhere.
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Ends of 1 / b for b in [kItvMin, kItvMax] (the factor covers the 1 ulp of
// the hardware reciprocal twice).
__device__ __forceinline__ float rcp_lo(float b_hi) {
  return __fmul_rd(rcp_approx(b_hi), 1.0f - 0x1.0p-22f);
}
__device__ __forceinline__ float rcp_hi(float b_lo) {
  return __fmul_ru(rcp_approx(b_lo), 1.0f + 0x1.0p-22f);
}

// A double x >= 0: truncated bits and their successor, by integer
// instructions.  Values below the FP32 normal range give [0, 2^-126];
// anything else (negative, too large, NaN) gives NaN.
__device__ __forceinline__ Itv itv_nonneg(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  if (b == 0ull) return Itv{0.0f, 0.0f};
  const int e = (int)(b >> 52) - 1023;  // sign bit set: e > 1023
  if (e >= 127) return itv_nan();
  if (e < -126) return Itv{0.0f, 0x1.0p-126f};
  const uint32_t lo =
      ((uint32_t)(e + 127) << 23) | (uint32_t)((b & 0x000fffffffffffffull) >> 29);
  return Itv{__uint_as_float(lo), __uint_as_float(lo + 1u)};
}

__device__ __forceinline__ Itv itv_neg(Itv a) { return Itv{-a.hi, -a.lo}; }
__device__ __forceinline__ Itv itv_add(Itv a, Itv b) {
  return Itv{__fadd_rd(a.lo, b.lo), __fadd_ru(a.hi, b.hi)};
}
__device__ __forceinline__ Itv itv_sub(Itv a, Itv b) {
  return Itv{__fsub_rd(a.lo, b.hi), __fsub_ru(a.hi, b.lo)};
}
// a * b, both >= 0
__device__ __forceinline__ Itv itv_mul_pos(Itv a, Itv b) {
  return Itv{__fmul_rd(a.lo, b.lo), __fmul_ru(a.hi, b.hi)};
}
// a * b for an exact b >= 0
__device__ __forceinline__ Itv itv_scale(Itv a, float b) {
  return Itv{__fmul_rd(a.lo, b), __fmul_ru(a.hi, b)};
}
// a * b for an interval b >= 0
__device__ __forceinline__ Itv itv_scale(Itv a, Itv b) {
  return Itv{__fmul_rd(a.lo, a.lo >= 0.0f ? b.lo : b.hi),
             __fmul_ru(a.hi, a.hi >= 0.0f ? b.hi : b.lo)};
}
// a count: any int32 >= 0, else NaN
__device__ __forceinline__ Itv itv_count(int n) {
  return n >= 0 ? Itv{__int2float_rd(n), __int2float_ru(n)} : itv_nan();
}
__device__ __forceinline__ Itv itv_of(float x) { return Itv{x, x}; }
__device__ __forceinline__ Itv itv_of(Itv x) { return x; }
__device__ __forceinline__ Itv itv_mul(Itv a, Itv b) {
  if (!(fabsf(a.lo) < kItvMax && fabsf(a.hi) < kItvMax && fabsf(b.lo) < kItvMax &&
        fabsf(b.hi) < kItvMax))
    return itv_nan();  // fminf / fmaxf would drop a NaN product
  const float lo = fminf(fminf(__fmul_rd(a.lo, b.lo), __fmul_rd(a.lo, b.hi)),
                         fminf(__fmul_rd(a.hi, b.lo), __fmul_rd(a.hi, b.hi)));
  const float hi = fmaxf(fmaxf(__fmul_ru(a.lo, b.lo), __fmul_ru(a.lo, b.hi)),
                         fmaxf(__fmul_ru(a.hi, b.lo), __fmul_ru(a.hi, b.hi)));
  return Itv{lo, hi};
}
// 1 / b for b in [kItvMin, kItvMax] or its negative, else NaN
__device__ __forceinline__ Itv itv_rcp_pos(Itv b) {
  const Itv r{rcp_lo(b.hi), rcp_hi(b.lo)};
  return b.lo >= kItvMin && b.hi <= kItvMax ? r : itv_nan();
}
__device__ __forceinline__ Itv itv_div_pos(Itv a, Itv b) { return itv_mul_pos(a, itv_rcp_pos(b)); }
__device__ __forceinline__ Itv itv_div(Itv a, Itv b) {
  if (b.hi < 0.0f) return itv_mul(itv_neg(a), itv_rcp_pos(itv_neg(b)));
  return itv_mul(a, itv_rcp_pos(b));
}

// The waiting-time numerator E = -log r1 of the draw with Philox words (w0,
// w1), r1 = (w1 2^21 + 2 (w0 >> 12) + 1) 2^-53.  The FP32 argument is within
// 2^-23 of r1 relatively (two roundings), which moves the logarithm by at
// most 1.2e-7; lg2.approx adds 2^-22 ln 2 = 1.7e-7 near 1 and 2^-22
// relatively elsewhere, the factor ln 2 and the product 2^-23 relatively.
// The enclosure takes 3.2e-7 absolutely and 2^-21 relatively (FP64's own
// ulp is far inside).
constexpr float kLogAbs = 3.2e-7f, kLogRel = 0x1.0p-21f;
__device__ __forceinline__ Itv itv_neglog(uint32_t w0, uint32_t w1) {
  const float low = __uint2float_rn(((w0 >> 12) << 1) | 1u) * 0x1.0p-53f;  // exact
  const float x = __fmaf_rn(__uint2float_rn(w1), 0x1.0p-32f, low);
  const float e = lg2_approx(x) * -0.69314718f;
  return Itv{fmaxf(0.0f, __fmaf_rd(e, 1.0f - kLogRel, -kLogAbs)),
             __fmaf_ru(e, 1.0f + kLogRel, kLogAbs)};
}

// r2 = (w3 + f) 2^-32 with f in (0, 1): truncation of w3 loses less than
// 2^-23 of it.
__device__ __forceinline__ Itv itv_r2(uint32_t w3) {
  const float lo = __uint2float_rd(w3) * 0x1.0p-32f;
  return Itv{lo, __fmaf_ru(lo, 1.0f + 0x1.0p-22f, 0x1.0p-32f)};
}

// The kind's rates as intervals.  load() takes the counts and the day's rate
// factors (ModelTraits::prepare) and tells whether the intervals apply;
// sums() gives the running sums of the rates in index order; fire(n) moves
// the counts x by transition n of the kind's own S (used only where
// DayArgs::fast says that the model's S is the kind's).  Counts of the
// built-in kinds are kept as FP32: their transitions keep every node's total,
// so with each count below 2^20 at the start they stay exact.
//
// The general form is that of models from transition strings: sums and
// moves are generated (ModelTraits::sums_itv, move), the parameters' values
// in them; counts outside 0 .. 2^23 settle nothing.
template <int KIND> struct Filter {
  using M = ModelTraits<KIND>;
  float x[M::C];
  __device__ __forceinline__ bool load(const int *u, const double *, const SgTables &) {
    bool in = true;
#pragma unroll
    for (int p = 0; p < M::C; ++p) {
      x[p] = (float)u[p];
      in = in && (uint32_t)u[p] < (1u << 23);
    }
    return in;
  }
  __device__ __forceinline__ bool sums(Itv *P, const SgTables &) const {
    bool good = M::sums_itv(x, P);
#pragma unroll
    for (int p = 0; p < M::C; ++p) good = good && x[p] >= 0.0f && x[p] <= 0x1.0p23f;
    return good;
  }
  __device__ __forceinline__ void fire(int n, const SgTables &) { M::move(n, x); }
};

__device__ __forceinline__ bool small_counts(const int *u, int n) {
  int all = 0;
#pragma unroll
  for (int p = 0; p < n; ++p) all |= u[p];
  return (uint32_t)all < (1u << 20);
}

template <> struct Filter<SG_SIR> {
  float x[3];
  Itv inv, g0, g1;
  __device__ __forceinline__ bool load(const int *u, const double *, const SgTables &tb) {
#pragma unroll
    for (int p = 0; p < 3; ++p) x[p] = (float)u[p];
    const float n = fmaxf(x[0] + x[1] + x[2], 1.0f);  // exact; rates are 0 in an empty node
    inv = Itv{rcp_lo(n), rcp_hi(n)};
    g0 = Itv{tb.g_lo[0], tb.g_hi[0]};
    g1 = Itv{tb.g_lo[1], tb.g_hi[1]};
    return small_counts(u, 3);
  }
  __device__ __forceinline__ bool sums(Itv *P, const SgTables &) const {
    const Itv w = itv_scale(itv_scale(g0, x[0]), x[1]);
    P[0] = Itv{__fmul_rd(w.lo, inv.lo), __fmul_ru(w.hi, inv.hi)};
    P[1] = itv_add(P[0], itv_scale(g1, x[1]));
    return true;
  }
  __device__ __forceinline__ void fire(int n, const SgTables &) {
    x[0] -= n == 0 ? 1.0f : 0.0f;
    x[1] += n == 0 ? 1.0f : -1.0f;
    x[2] += n == 0 ? 0.0f : 1.0f;
  }
};

// SIS, SISe: S -> I and back.
struct FilterSI {
  float x[2];
  Itv g0, g1;
  __device__ __forceinline__ void fire(int n, const SgTables &) {
    const float d = n == 0 ? 1.0f : -1.0f;
    x[0] -= d;
    x[1] += d;
  }
};

template <> struct Filter<SG_SIS> : FilterSI {
  __device__ __forceinline__ bool load(const int *u, const double *, const SgTables &tb) {
    x[0] = (float)u[0];
    x[1] = (float)u[1];
    g0 = Itv{tb.g_lo[0], tb.g_hi[0]};
    g1 = Itv{tb.g_lo[1], tb.g_hi[1]};
    return small_counts(u, 2);
  }
  __device__ __forceinline__ bool sums(Itv *P, const SgTables &) const {
    P[0] = itv_scale(itv_scale(g0, x[0]), x[1]);
    P[1] = itv_add(P[0], itv_scale(g1, x[1]));
    return true;
  }
};

template <> struct Filter<SG_SISE> : FilterSI {
  // g0: upsilon phi of the day
  __device__ __forceinline__ bool load(const int *u, const double *kf, const SgTables &tb) {
    x[0] = (float)u[0];
    x[1] = (float)u[1];
    g0 = itv_nonneg(kf[0]);
    g1 = Itv{tb.g_lo[1], tb.g_hi[1]};
    return small_counts(u, 2);
  }
  __device__ __forceinline__ bool sums(Itv *P, const SgTables &) const {
    P[0] = itv_scale(g0, x[0]);
    P[1] = itv_add(P[0], itv_scale(g1, x[1]));
    return true;
  }
};

template <> struct Filter<SG_SISE_SP> : Filter<SG_SISE> {};

template <> struct Filter<SG_SISE3> {
  float x[6];
  Itv k[3], g[3];
  __device__ __forceinline__ bool load(const int *u, const double *kf, const SgTables &tb) {
#pragma unroll
    for (int p = 0; p < 6; ++p) x[p] = (float)u[p];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      k[a] = itv_nonneg(kf[a]);
      g[a] = Itv{tb.g_lo[3 + a], tb.g_hi[3 + a]};
    }
    return small_counts(u, 6);
  }
  __device__ __forceinline__ bool sums(Itv *P, const SgTables &) const {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const Itv w = itv_scale(k[a], x[2 * a]);
      P[2 * a] = a == 0 ? w : itv_add(P[2 * a - 1], w);
      P[2 * a + 1] = itv_add(P[2 * a], itv_scale(g[a], x[2 * a + 1]));
    }
    return true;
  }
  __device__ __forceinline__ void fire(int n, const SgTables &) {
    const float d = (n & 1) ? -1.0f : 1.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float y = (n >> 1) == a ? d : 0.0f;
      x[2 * a] -= y;
      x[2 * a + 1] += y;
    }
  }
};

// The rates as intervals for any counts, kept as int32 (a count above 2^24 is
// an interval itself), moved by the model's S.  Used for a caller's own S, for
// counts beyond Filter's, and where a day may take the counts out of the
// range in which FP32 holds them exactly (a model from transition strings can
// grow by 127 a transition).
template <int KIND> struct FilterWide {
  using M = ModelTraits<KIND>;
  static constexpr bool kPhi = KIND == SG_SISE || KIND == SG_SISE_SP || KIND == SG_SISE3;
  int x[M::C];
  Itv k[M::NK];
  __device__ __forceinline__ bool load(const int *u, const double *kf, const SgTables &) {
#pragma unroll
    for (int p = 0; p < M::C; ++p) x[p] = u[p];
#pragma unroll
    for (int i = 0; i < M::NK; ++i) k[i] = kPhi ? itv_nonneg(kf[i]) : Itv{0.0f, 0.0f};
    return true;
  }
  __device__ __forceinline__ bool sums(Itv *P, const SgTables &tb) const {
    Itv c[M::C];
#pragma unroll
    for (int p = 0; p < M::C; ++p) c[p] = itv_count(x[p]);
    if constexpr (KIND == SG_GENERIC) {
      return M::sums_itv(c, P);
    } else {
      auto g = [&](int i) { return Itv{tb.g_lo[i], tb.g_hi[i]}; };
      if constexpr (KIND == SG_SISE3) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const Itv w = itv_mul_pos(k[a], c[2 * a]);
          P[2 * a] = a == 0 ? w : itv_add(P[2 * a - 1], w);
          P[2 * a + 1] = itv_add(P[2 * a], itv_mul_pos(g(3 + a), c[2 * a + 1]));
        }
      } else {
        if constexpr (KIND == SG_SIR) {
          // the rate is 0 in an empty node
          const long long n = (long long)x[0] + x[1] + x[2];
          const float lo = fmaxf(__ll2float_rd(n), 1.0f), hi = fmaxf(__ll2float_ru(n), 1.0f);
          P[0] = itv_div_pos(itv_mul_pos(itv_mul_pos(g(0), c[0]), c[1]), Itv{lo, hi});
          P[0] = x[2] >= 0 ? P[0] : itv_nan();
        } else if constexpr (KIND == SG_SIS) {
          P[0] = itv_mul_pos(itv_mul_pos(g(0), c[0]), c[1]);
        } else {
          P[0] = itv_mul_pos(k[0], c[0]);
        }
        P[1] = itv_add(P[0], itv_mul_pos(g(1), c[1]));
      }
      return true;
    }
  }
  __device__ __forceinline__ void fire(int n, const SgTables &tb) {
#pragma unroll
    for (int p = 0; p < M::C; ++p) x[p] += tb.S[n][p];
  }
};

// The transition that lambda r2 selects, from the running sums' intervals;
// -1 where they do not settle it.  With lambda r2 > 0 the first running sum
// that reaches it belongs to a positive rate (adding a zero rate leaves the
// sum unchanged), so counting the sums below it is the inversion.
template <int T>
__device__ __forceinline__ int itv_select(const Itv *P, Itv r2) {
  const float tl = __fmul_rd(P[T - 1].lo, r2.lo), th = __fmul_ru(P[T - 1].hi, r2.hi);
  int sure = 0, maybe = 0;  // sums certainly, possibly below the target
#pragma unroll
  for (int j = 0; j < T; ++j) {
    sure += P[j].hi < tl ? 1 : 0;
    maybe += P[j].lo < th ? 1 : 0;
  }
  return sure == maybe ? sure : -1;  // maybe < T: the last sum reaches it
}

}  // namespace sg
