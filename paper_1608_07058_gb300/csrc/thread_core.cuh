// One trajectory per thread: the adaptive explicit-implicit tau-leaping loop for small
// networks (N <= 8 species, M <= 16 reactions), templated on the table capacities
// (NM, MM) and on the arithmetic (P = PrecRef: FP64, fixed operation order, bitwise
// reproducible; P = PrecFast: FP32 propensities, step sizes, Poisson means and G
// increments, FP64 time and G totals, and an FP64 implicit Newton solve -- or, on
// request, an FP32 solve for the increment).  All per-trajectory arrays are indexed with
// compile-time indices only so that they live in registers.
//
// Steps (paper Section 2, with the published methods it names):
//   propensities a_j = theta_j g_j(x), a0                       (Section 1)
//   critical reactions: a_j > 0 and min_s floor(x_s/|nu_js|) < n_c
//   tau_ex: Cao 2006 bound on mean and variance of each reactant's change
//   partial-equilibrium pairs, tau_im without them, implicit iff tau_im >> tau_ex
//   tau2 ~ Exp(a0c); SSA burst if min(tau1, tau2) < ssa_factor / a0
//   explicit Poisson leap or implicit Newton leap (Rathinam 2003); one critical firing
//   negativity check (halve tau1 and retry); commit x, r, G (trapezoid) and t.
#pragma once
#ifndef __CUDACC_RTC__
#include <cstdint>
#endif

#include "dev_common.cuh"
#include "ml_internal.h"
#include "matleap.h"

namespace mlk {

// Canonical sum over reactions for a0 and a0c: element j on lane j (j < 32); lanes
// combined pairwise at xor distances 16, 8, 4, 2, 1; lane 0's value.  Written for one
// thread holding all elements (MM <= 32), with empty lanes holding 0.
template <int MM, class R>
__device__ __forceinline__ R lane_tree_sum(const R (&v)[MM]) {
  static_assert(MM <= 32, "thread variant holds at most 32 reactions");
  // the additions of empty lanes' zeros are left out (the elements are not negative, so
  // v + 0 is v): MM - 1 additions instead of 31
  R lane[MM];
#pragma unroll
  for (int l = 0; l < MM; ++l) lane[l] = v[l];
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
#pragma unroll
    for (int l = 0; l < d; ++l)
      if (l + d < MM) lane[l] = lane[l] + lane[l + d];
  }
  return lane[0];
}

// Sum over reactions: the canonical lane tree in reference precision (bitwise parity with
// the CPU reference); fast precision may add in any order and adds sequentially.
template <int MM, class R, bool kRef>
__device__ __forceinline__ R reaction_sum(const R (&v)[MM]) {
  if (kRef) return lane_tree_sum<MM, R>(v);
  R s = v[0];
#pragma unroll
  for (int j = 1; j < MM; ++j) s = s + v[j];
  return s;
}

// A count as the working precision (x >= 0), without the FP64 unit.
template <class R>
__device__ __forceinline__ R of_count(long long x);
template <>
__device__ __forceinline__ float of_count<float>(long long x) { return f32_of_count(x); }
template <>
__device__ __forceinline__ double of_count<double>(long long x) { return f64_of_count(x); }

// C(v, m) for m = 1, 2, 3 on a real argument, in this operation order.
// The third order, with its division, is out of line: the precompiled kernels have a site per
// reactant, and their code size is what slows them down (instruction fetch).
template <class R>
__device__ __noinline__ R comb_three(R v) {
  return ((v * (v - R(1))) * (v - R(2))) / R(6);
}
template <class R>
__device__ __forceinline__ R comb_factor(R v, int m) {
  if (m == 1) return v;
  if (m == 2) return (v * (v - R(1))) * R(0.5);
  return comb_three<R>(v);
}

// C(x, m) of a count: as comb_factor on the converted count.  In FP64 C(x, 2) is an integer
// operation while x (x - 1) stays below 2^53, where every step of comb_factor is exact.
template <class R>
__device__ __forceinline__ R comb_count(long long x, int m) {
  if (sizeof(R) == 8 && m == 2 && x < 94906265LL)
    return of_count<R>((long long)(((unsigned long long)x * (unsigned long long)(x - 1)) >> 1));
  return comb_factor<R>(of_count<R>(x), m);
}

// d/dv C(v, m): 1, v - 1/2, (3 v^2 - 6 v + 2) / 6, in this operation order.
template <class T>
__device__ __noinline__ T comb_three_deriv(T v) {
  return ((T(3) * (v * v) - T(6) * v) + T(2)) / T(6);
}
template <class T>
__device__ __forceinline__ T comb_factor_deriv(T v, int m) {
  if (m == 1) return T(1);
  if (m == 2) return v - T(0.5);
  return comb_three_deriv<T>(v);
}

// C(x + z, m) - C(x, m) written as z times a polynomial, so that no two large nearby
// values are subtracted: m = 2: z (2x + z - 1) / 2; m = 3 with u = x + z:
// z (u^2 + u x + x^2 - 3 (u + x) + 2) / 6.
template <class R>
__device__ __forceinline__ R comb_diff(R xv, R z, int m) {
  if (m == 1) return z;
  if (m == 2) return (z * ((R(2) * xv + z) - R(1))) * R(0.5);
  const R u = xv + z;
  return (z * (((u * u + u * xv) + xv * xv) - R(3) * (u + xv) + R(2))) / R(6);
}

// Double-float (hi + lo FP32 pair) arithmetic for the fast-precision reaction pick: sums
// by TwoSum (Knuth) renormalized with Fast2Sum, about 46 significant bits, all on the
// FP32 pipe.
struct DF {
  float hi, lo;
};
__device__ __forceinline__ DF df_norm(float s, float e) {
  const float hi = s + e;
  return DF{hi, e - (hi - s)};
}
__device__ __forceinline__ DF df_add(DF a, float b) {
  const float s = a.hi + b;
  const float bb = s - a.hi;
  const float err = (a.hi - (s - bb)) + (b - bb);
  return df_norm(s, err + a.lo);
}
__device__ __forceinline__ DF df_add(DF a, DF b) {
  const float s = a.hi + b.hi;
  const float bb = s - a.hi;
  const float err = (a.hi - (s - bb)) + (b.hi - bb);
  return df_norm(s, err + (a.lo + b.lo));
}
__device__ __forceinline__ DF df_sub(DF a, DF b) { return df_add(a, DF{-b.hi, -b.lo}); }
__device__ __forceinline__ bool df_lt(DF a, DF b) {
  return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
}
// u * t for a 48-bit uniform u = (w_hi>>8) 2^-24 + ((w_lo>>8) + 1/2) 2^-48 in (0, 1).
__device__ __forceinline__ DF df_uniform_times(DF t, uint32_t w_hi, uint32_t w_lo) {
  const float uh = (float)(w_hi >> 8) * 0x1p-24f;
  const float ul = ((float)(w_lo >> 8) + 0.5f) * 0x1p-48f;
  const float p = uh * t.hi;
  const float e = fmaf(uh, t.hi, -p);
  return df_norm(p, e + (uh * t.lo + ul * t.hi));
}

// Compensated (Kahan) FP32 accumulation: the sum is s - c.
__device__ __forceinline__ void kahan_add(float& s, float& c, float v) {
  const float y = v - c;
  const float t = s + y;
  c = (t - s) - y;
  s = t;
}

// a < b for values in [0, +inf] (not -0) or NaN
__device__ __forceinline__ bool lt_pos(double a, double b) { return f64_lt_pos(a, b); }
__device__ __forceinline__ bool lt_pos(float a, float b) { return a < b; }

// ... of the product a b, fused into the correction.
__device__ __forceinline__ void kahan_fma(float& s, float& c, float a, float b) {
  const float y = __fmaf_rn(a, b, -c);
  const float t = s + y;
  c = (t - s) - y;
  s = t;
}

// Highest-order-reaction factor h_s (Cao 2006) from the species' flags and count.
template <class R>
__device__ __forceinline__ R hor_factor_at(uint8_t f, long long x) {
  const R xd = of_count<R>(x);
  R h = R(0);
  if (f & kHorO1) h = lt_pos(h, R(1)) ? R(1) : h;
  if (f & kHorO2M1) h = lt_pos(h, R(2)) ? R(2) : h;
  if (f & kHorO2M2) {
    const R v = x >= 2 ? R(2) + R(1) / (xd - R(1)) : R(2);
    h = lt_pos(h, v) ? v : h;
  }
  if (f & kHorO3M1) h = lt_pos(h, R(3)) ? R(3) : h;
  if (f & kHorO3M2) {
    const R v = x >= 2 ? R(1.5) * (R(2) + R(1) / (xd - R(1))) : R(3);
    h = lt_pos(h, v) ? v : h;
  }
  if (f & kHorO3M3) {
    const R v = x >= 3 ? (R(3) + R(1) / (xd - R(1))) + R(2) / (xd - R(2)) : R(3);
    h = lt_pos(h, v) ? v : h;
  }
  return h;
}

template <class R>
__device__ __noinline__ R hor_factor_call(uint8_t f, long long x) {
  return hor_factor_at<R>(f, x);
}
// Out of line where the flags are read at run time (four divisions), inline where they are
// compiled in.
template <class R, bool kInline = false>
__device__ __forceinline__ R hor_factor(uint8_t f, long long x) {
  return kInline ? hor_factor_at<R>(f, x) : hor_factor_call<R>(f, x);
}

struct PrecRef {
  using R = double;
  static constexpr bool kRef = true;
  // a b rounded, and a b + c with the product rounded, whatever the compiler would contract
  __device__ static __forceinline__ R mul(R a, R b) { return __dmul_rn(a, b); }
  __device__ static __forceinline__ R mad(R a, R b, R c) { return __dadd_rn(__dmul_rn(a, b), c); }
  __device__ static __forceinline__ R u(const Words4& w, int k) {
    return k == 0 ? u01_f64(w.w0, w.w1) : u01_f64(w.w2, w.w3);
  }
  // comparisons of values in [0, +inf] (not -0) or NaN, on the integer pipe
  __device__ static __forceinline__ bool lt(R a, R b) { return f64_lt_pos(a, b); }
  __device__ static __forceinline__ bool le(R a, R b) { return f64_le_pos(a, b); }
  __device__ static __forceinline__ bool positive(R a) { return f64_lt_pos(0.0, a); }
  __device__ static __forceinline__ bool zero(R a) {
    return (__double_as_longlong(a) << 1) == 0;
  }
  __device__ static __forceinline__ bool negative(R a) {  // below zero (-0 is not)
    return __double_as_longlong(a) < 0 && !zero(a);
  }
  __device__ static __forceinline__ R of_f64(double v) { return v; }
  __device__ static __forceinline__ double to_f64(R v) { return v; }
  __device__ static __forceinline__ R eps(const SimArgs& A) { return A.eps; }
  __device__ static __forceinline__ R ssa_factor(const SimArgs& A) { return A.ssa_factor; }
  __device__ static __forceinline__ R pe_delta(const SimArgs& A) { return A.pe_delta; }
  __device__ static __forceinline__ R stiff_ratio(const SimArgs& A) { return A.stiff_ratio; }
  __device__ static __forceinline__ R log(R x) { return refmath::log_ref(x); }
  __device__ static __forceinline__ R exp(R x) { return refmath::exp_ref(x); }
  __device__ static __forceinline__ R lfact(long long k) {
    return refmath::log_factorial_ref(k);
  }
  __device__ static __forceinline__ R sqrt(R x) { return ::sqrt(x); }
  __device__ static __forceinline__ R inf() {
    return __longlong_as_double(0x7ff0000000000000LL);
  }
};

struct PrecFast {
  using R = float;
  static constexpr bool kRef = false;
  // a b rounded, and a b + c fused, whatever the compiler would contract
  __device__ static __forceinline__ R mul(R a, R b) { return __fmul_rn(a, b); }
  __device__ static __forceinline__ R mad(R a, R b, R c) { return __fmaf_rn(a, b, c); }
  __device__ static __forceinline__ R u(const Words4& w, int k) {
    return k == 0 ? u01_f32(w.w0) : u01_f32(w.w2);
  }
  __device__ static __forceinline__ bool lt(R a, R b) { return a < b; }
  __device__ static __forceinline__ bool le(R a, R b) { return a <= b; }
  __device__ static __forceinline__ bool positive(R a) { return a > 0.f; }
  __device__ static __forceinline__ bool zero(R a) { return a == 0.f; }
  __device__ static __forceinline__ bool negative(R a) { return a < 0.f; }
  __device__ static __forceinline__ R of_f64(double v) { return f32_of_f64(v); }
  __device__ static __forceinline__ double to_f64(R v) { return f64_of_f32(v); }
  __device__ static __forceinline__ R eps(const SimArgs& A) { return A.eps_f; }
  __device__ static __forceinline__ R ssa_factor(const SimArgs& A) { return A.ssa_factor_f; }
  __device__ static __forceinline__ R pe_delta(const SimArgs& A) { return A.pe_delta_f; }
  __device__ static __forceinline__ R stiff_ratio(const SimArgs& A) { return A.stiff_ratio_f; }
  // accurate logf: the waiting times -log(u)/a0 need relative accuracy for u near 1,
  // where the hardware approximation's absolute error would bias the clock
  __device__ static __forceinline__ R log(R x) { return logf(x); }
  __device__ static __forceinline__ R exp(R x) { return __expf(x); }
  __device__ static __forceinline__ R lfact(long long k) {
    return lgammaf((float)k + 1.0f);
  }
  __device__ static __forceinline__ R sqrt(R x) { return sqrtf(x); }
  __device__ static __forceinline__ R log1p(R x) { return log1pf(x); }
  __device__ static __forceinline__ R inf() { return __int_as_float(0x7f800000); }
};

// FP64 PTRS with library functions, used by the fast path for very large means where
// FP32 cannot hold the integer count exactly.
struct PrecWide {
  using R = double;
  static constexpr bool kRef = false;
  // a b rounded, and a b + c fused, whatever the compiler would contract
  __device__ static __forceinline__ R mul(R a, R b) { return __dmul_rn(a, b); }
  __device__ static __forceinline__ R mad(R a, R b, R c) { return __fma_rn(a, b, c); }
  __device__ static __forceinline__ bool negative(R a) { return PrecRef::negative(a); }
  __device__ static __forceinline__ R u(const Words4& w, int k) {
    return k == 0 ? u01_f64(w.w0, w.w1) : u01_f64(w.w2, w.w3);
  }
  __device__ static __forceinline__ R log(R x) { return ::log(x); }
  __device__ static __forceinline__ R exp(R x) { return ::exp(x); }
  __device__ static __forceinline__ R lfact(long long k) { return ::lgamma((double)k + 1.0); }
  __device__ static __forceinline__ R sqrt(R x) { return ::sqrt(x); }
  __device__ static __forceinline__ R log1p(R x) { return ::log1p(x); }
  __device__ static __forceinline__ R inf() {
    return __longlong_as_double(0x7ff0000000000000LL);
  }
};

constexpr int kPtrsMaxTrials = 256;

struct PoissonDraw {
  long long k;
  uint32_t flags;  // ML_ST_PTRS_CAP when the trial cap was hit
};

// The integer of a non-negative integral value.
__device__ __forceinline__ long long count_of(float v) {
  if (v < 2147483648.f) return (long long)(int)v;
  long long k;
  asm volatile("cvt.rzi.s64.f32 %0, %1;" : "=l"(k) : "f"(v));
  return k;
}
__device__ __forceinline__ long long count_of(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int e = (int)(b >> 52) - 1023;  // sign 0
  if (e < 0) return 0;
  const unsigned long long m = (b & 0x000fffffffffffffULL) | 0x0010000000000000ULL;
  if (e <= 52) return (long long)(m >> (52 - e));
  long long k;
  asm volatile("cvt.rzi.s64.f64 %0, %1;" : "=l"(k) : "d"(v));
  return k;
}

// PTRS: Hoermann (1993), transformed rejection with squeeze, for mean mu >= 10.  Trial b
// uses block b of the stream: U from the first uniform, V from the second.

// The acceptance test beyond the squeeze, in the precision's own arithmetic.
template <class P>
__device__ __noinline__ bool ptrs_accept(typename P::R mu, typename P::R a, typename P::R b,
                                         typename P::R us, typename P::R V, typename P::R kd) {
  using R = typename P::R;
  const R inv_alpha = R(1.1239) + R(1.1328) / (b - R(3.4));
  const R lhs = (P::log(V) + P::log(inv_alpha)) - P::log(a / (us * us) + b);
  if constexpr (!P::kRef) {
    if (!lt_pos(kd, R(10))) {
      // log of the Poisson pmf without cancellation: with z = k + 1 and Stirling's series
      // for log Gamma(z), -mu + k log mu - log k! =
      //   (z - mu) + (z - 1) log1p((mu - z)/z) - log(z)/2 - log(2 pi)/2 - 1/(12 z) + 1/(360 z^3)
      const R z = kd + R(1);
      const R iz = R(1) / z;
      const R rhs = ((z - mu) + (z - R(1)) * P::log1p((mu - z) * iz)) - R(0.5) * P::log(z) -
                    R(0.91893853320467274178) -
                    iz * (R(1) / R(12) - (iz * iz) * (R(1) / R(360)));
      return lhs <= rhs;
    }
  }
  const R loglam = P::log(mu);
  return lhs <= (-mu + kd * loglam) - P::lfact(count_of(kd));
}

// The same test estimated in FP32: 1 accept, -1 reject, 0 too close to tell (then the caller
// evaluates it in its own arithmetic, so the outcome is that of ptrs_accept).  The four
// logarithms of the exact test cost about 250 instructions on the FP64 unit (16,000 cycles
// of it) or 150 in FP32; some lane of a warp nearly always needs the test.
//   lhs = log(V inv_alpha us^2 / (a + b us^2)) by one hardware logarithm;
//   rhs = z (L - x) - L - log(z)/2 - log(2 pi)/2 - 1/(12 z) + 1/(360 z^3), x = d/z, d = mu - z,
//   L = log1p(x): since z - mu = -z x, the large terms cancel before they are formed, and for
//   |x| < 1/4 L - x is its series to x^8 (relative error below 2e-5).
// Errors: Stirling's series 8e-4 at z = 1; the estimate 1e-4 of |z (L - x)| with room; the
// FP32 form of ptrs_accept, which does form z - mu, up to 4e-7 |d|.  us >= 1e-4 here.
__device__ __forceinline__ int ptrs_estimate(float inv_alpha, float a, float b, float us,
                                             float V, float z, float d) {
  const float u2 = us * us;
  const float lhs = 0.69314718f * __log2f(__fdividef(V * inv_alpha * u2, a + b * u2));
  const float iz = __fdividef(1.f, z), x = d * iz;
  float L, t;
  if (fabsf(x) < 0.25f) {
    float q = -0.125f;
    q = q * x + (1.f / 7.f);
    q = q * x - (1.f / 6.f);
    q = q * x + 0.2f;
    q = q * x - 0.25f;
    q = q * x + (1.f / 3.f);
    q = q * x - 0.5f;
    const float s = q * x * x;
    L = x + s;
    t = z * s;
  } else {
    L = 0.69314718f * __log2f(1.f + x);
    t = z * (L - x);
  }
  const float rhs = t - L - 0.34657359f * __log2f(z) - 0.91893853f -
                    iz * (0.083333333f - iz * iz * 0.0027777778f);
  const float gap = rhs - lhs;
  const float margin = 4.0e-3f + 1.0e-4f * fabsf(t) + 2.0e-6f * fabsf(d);
  return gap > margin ? 1 : gap < -margin ? -1 : 0;
}

// One trial in the precision's own arithmetic (FP32: the estimate before the exact test).
template <class P>
__device__ __forceinline__ bool ptrs_trial_own(typename P::R mu, const Words4& w, long long& k) {
  using R = typename P::R;
  const R slam = P::sqrt(mu);
  const R b = P::mad(R(2.53), slam, R(0.931));
  const R a = P::mad(R(0.02483), b, R(-0.059));
  const R v_r = R(0.9277) - R(3.6224) / (b - R(2));
  const R U = P::u(w, 0) - R(0.5);
  const R V = P::u(w, 1);
  const R us = R(0.5) - fabs(U);  // positive: |U| < 1/2
  const R kd = floor(P::mad((R(2) * a) / us + b, U, mu) + R(0.43));
  bool ok = false;
  if (!lt_pos(us, R(0.07)) && !lt_pos(v_r, V)) {
    ok = true;
  } else if (!(P::negative(kd) || (lt_pos(us, R(0.013)) && lt_pos(us, V)))) {
    int est = 0;
    if constexpr (sizeof(R) == 4) {
      const float z = kd + 1.f;
      if (us > 1.0e-4f)
        est = ptrs_estimate(1.1239f + __fdividef(1.1328f, b - 3.4f), a, b, us, V, z, mu - z);
    }
    ok = est != 0 ? est > 0 : ptrs_accept<P>(mu, a, b, us, V, kd);
  }
  if (ok) k = count_of(kd);
  return ok;
}
template <class P>
__device__ __noinline__ bool ptrs_trial_exact(typename P::R mu, const Words4& w, long long& k) {
  return ptrs_trial_own<P>(mu, w, k);
}

// Reference precision: the trial with FP32 setup and FP32 estimates, the proposal
// k = floor(x) kept to FP64 by adding its FP32 part (relative error below 3e-6) to mu + 0.43;
// where a floor, a comparison or the test could go either way, the exact trial decides
// (about 1e-2 of the trials at mu = 1e4).  Four FP64 additions instead of about 60 operations
// with a square root and three divisions, and 250 more with the test.
__device__ __forceinline__ bool ptrs_trial_near(double mu, const Words4& w, long long& k) {
  const long long n1 = ((long long)(w.w0 >> 6) << 26) | (long long)(w.w1 >> 6);
  const long long n2 = ((long long)(w.w2 >> 6) << 26) | (long long)(w.w3 >> 6);
  // U = m 2^-53, us = (2^52 - |m|) 2^-53, exact integers
  const long long m = 2 * n1 + 1 - (1LL << 52);
  const long long am = m < 0 ? -m : m;
  const float Ua = f32_of_count(am) * 0x1p-53f, us = f32_of_count((1LL << 52) - am) * 0x1p-53f;
  const float V = f32_of_count(2 * n2 + 1) * 0x1p-53f;
  const float b = 0.931f + 2.53f * sqrtf(f32_of_f64(mu));
  const float a = -0.059f + 0.02483f * b;
  const float prod = (__fdividef(2.f * a, us) + b) * (m < 0 ? -Ua : Ua);
  const double kx = (mu + 0.43) + f64_of_f32(prod);
  const float err = 1.0e-6f + 3.0e-6f * fabsf(prod);
  if (us > 1.0e-4f && f64_lt_pos(mu, 1.0e9)) {
    if (__double2hiint(kx) < 0) {  // k < 0: rejected (us < 0.07 there)
      if (f32_of_f64(-kx) > 1.f + err) return false;
    } else {
      k = count_of(kx);
      const float frac = f32_of_f64(kx - f64_of_count(k));
      const float v_r = 0.9277f - __fdividef(3.6224f, b - 2.f);
      if (frac > err && frac < 1.f - err && fabsf(us - 0.07f) > 1.0e-6f &&
          fabsf(us - 0.013f) > 1.0e-6f) {
        if (us > 0.07f && V < v_r - 4.0e-6f) return true;
        if (us < 0.07f || V > v_r + 4.0e-6f) {
          if (us < 0.013f && V > us + 1.0e-6f) return false;
          if (us > 0.013f || V < us - 1.0e-6f) {
            const double z = f64_of_count(k + 1);
            const int est =
                ptrs_estimate(1.1239f + __fdividef(1.1328f, b - 3.4f), a, b, us, V,
                              f32_of_count(k + 1), f32_of_f64(mu - z));
            if (est != 0) return est > 0;
          }
        }
      }
    }
  }
  return ptrs_trial_exact<PrecRef>(mu, w, k);
}

template <class P>
__device__ __forceinline__ bool ptrs_trial(typename P::R mu, const Words4& w, long long& k) {
  if constexpr (P::kRef) return ptrs_trial_near(mu, w, k);
  else return ptrs_trial_own<P>(mu, w, k);
}

template <class P>
__device__ __noinline__ PoissonDraw poisson_ptrs(typename P::R mu, uint32_t k0, uint32_t k1,
                                                 uint32_t id, uint32_t step, uint32_t stream) {
  using R = typename P::R;
  long long k = 0;
  for (uint32_t trial = 0; trial < (uint32_t)kPtrsMaxTrials; ++trial)
    if (ptrs_trial<P>(mu, philox_block(k0, k1, id, step, stream, trial), k))
      return PoissonDraw{k, 0u};
  return PoissonDraw{(long long)floor(mu + R(0.5)), ML_ST_PTRS_CAP};
}

// mu / k rounded to nearest, for mu in (2^-60, 10) and an integer k >= 1: with z near 1/k
// (relative error below 2^-20 in FP32, 2^-50 in FP64), q = mu z and the remainder
// r = mu - k q (exact: one FMA), q + r z misses mu / k by far less than the smallest
// distance of mu / k from a midpoint of two numbers: mu / k = c/k ulps with an integer c, so
// it is no midpoint (k times an odd half-integer of the quotient's precision does not fit
// the significand of mu) and at least 1/(2k) ulp away from one.  So the result is that
// of the IEEE division, in 4 instructions (FP32), or in 3 on the FP64 unit (192 of its
// cycles; a division occupies it for 564) and a conversion of k on the integer pipe.
__device__ __forceinline__ float div_by_int(float mu, int k) {
  const float kf = (float)k;
  const float z = __fdividef(1.f, kf);
  const float q = __fmul_rn(mu, z);
  return __fmaf_rn(__fmaf_rn(-kf, q, mu), z, q);
}
constexpr int kRecips = 48;
struct Recips {
  double v[kRecips];
};
constexpr Recips make_recips() {
  Recips t{};
  t.v[0] = 0.0;
  for (int k = 1; k < kRecips; ++k) t.v[k] = 1.0 / (double)k;
  return t;
}
__constant__ constexpr Recips kRecip = make_recips();
__device__ __forceinline__ double div_by_int(double mu, int k) {
  const double kd = f64_of_i32(k);
  if (k >= kRecips) return mu / kd;
  const double z = kRecip.v[k];
  const double q = __dmul_rn(mu, z);
  return __fma_rn(__fma_rn(-kd, q, mu), z, q);
}

// Means below 10: inversion by sequential search (mu > 0).
template <class P>
__device__ __forceinline__ int poisson_invert(typename P::R mu, typename P::R u) {
  using R = typename P::R;
  R p = P::exp(-mu);
  R F = p;
  int k = 0;
  while (P::lt(F, u)) {
    k = k + 1;
    p = p * div_by_int(mu, k);
    if (P::zero(p)) break;
    F = F + p;
  }
  return k;
}
__device__ __noinline__ inline int poisson_invert_exact(double mu, double u) {
  return poisson_invert<PrecRef>(mu, u);
}
// Reference precision: the search in FP32 first.  The FP32 cumulative sums are within 2e-6 of
// the FP64 ones (an exponential, at most 60 products and sums), so while u stays farther
// than 1e-5 from each of them the FP64 search makes the same steps; otherwise (a few 1e-4 of
// the draws) it runs: an exponential of about 30 FP64 operations and five more per step.
__device__ __forceinline__ int poisson_invert_near(double mu, double u) {
  const float m = f32_of_f64(mu), uf = f32_of_f64(u);
  float p = __expf(-m), F = p;
  int k = 0;
  bool clear = fabsf(uf - F) > 1.0e-5f;
  while (F < uf && clear && k < 60) {
    ++k;
    p = p * __fdividef(m, (float)k);
    F = F + p;
    clear = fabsf(uf - F) > 1.0e-5f;
  }
  return clear && k < 60 ? k : poisson_invert_exact(mu, u);
}

template <class P>
__device__ __forceinline__ int poisson_invert_at(typename P::R mu, typename P::R u) {
  if constexpr (P::kRef) return poisson_invert_near(mu, u);
  else return poisson_invert<P>(mu, u);
}

template <class P>
__device__ __noinline__ int poisson_invert_call(typename P::R mu, typename P::R u) {
  return poisson_invert_at<P>(mu, u);
}

// Poisson(mu) for mu < 10: 0 for mu <= 0 (no draw).
template <class P>
__device__ __noinline__ int poisson_small(typename P::R mu, uint32_t k0, uint32_t k1,
                                          uint32_t id, uint32_t step, uint32_t stream) {
  if (!P::positive(mu)) return 0;
  const Words4 w = philox_block(k0, k1, id, step, stream, 0);
  return poisson_invert_at<P>(mu, P::u(w, 0));
}

// Poisson(mu): inversion by sequential search below 10; PTRS.
template <class P>
__device__ __forceinline__ PoissonDraw poisson_sample(typename P::R mu, uint32_t k0, uint32_t k1,
                                                   uint32_t id, uint32_t step, uint32_t stream) {
  using R = typename P::R;
  if (!P::positive(mu) || P::lt(mu, R(10)))
    return PoissonDraw{(long long)poisson_small<P>(mu, k0, k1, id, step, stream), 0u};
  return (!P::kRef && mu > R(4.0e6)) ? poisson_ptrs<PrecWide>((double)mu, k0, k1, id, step, stream)
                                     : poisson_ptrs<P>(mu, k0, k1, id, step, stream);
}

template <class P>
__device__ __forceinline__ long long poisson_draw(typename P::R mu, uint32_t k0, uint32_t k1,
                                                  uint32_t id, uint32_t step, uint32_t stream,
                                                  uint32_t& status) {
  const PoissonDraw d = poisson_sample<P>(mu, k0, k1, id, step, stream);
  status |= d.flags;
  return d.k;
}

// v t for a net change v: the common changes by one are exact without a product.
__device__ __noinline__ inline double nu_times_call(int v, double t) { return f64_of_i32(v) * t; }
__device__ __forceinline__ double nu_times(int v, double t) {
  return v == 1 ? t : v == -1 ? -t : v == 2 ? 2.0 * t : v == -2 ? -2.0 * t
                                                                : nu_times_call(v, t);
}

// MDL: the model tables' type -- the shared-memory ThreadModel staged at kernel start, or
// a type with the same members known at compile time.
template <int NM, int MM, class P, class MDL = ThreadModel<NM, MM>>
struct ThreadTraj {
  using R = typename P::R;
  using Model = MDL;

  // g_j of a state by the table's reactant word: comb(x_s, m) of the k-th reactant, the
  // product in increasing s, 0 when some x_s < m_js.  The code is a tenth of a loop over
  // all (reaction, species) pairs with a branch per order, on which the precompiled kernels
  // stall in instruction fetch.
  // Orders above two are out of line (bit 31 of the word).
  template <class V>
  __device__ static __forceinline__ V sel(const V (&x)[NM], int sp) {
    V v = x[0];
#pragma unroll
    for (int s = 1; s < NM; ++s) v = s == sp ? x[s] : v;
    return v;
  }
  template <class V, class F>
  __device__ static __forceinline__ auto g_slots(uint32_t rx, const V (&x)[NM], F comb) {
    using O = decltype(comb(x[0], 1));
    O v = O(1);
    bool zero = false;
    const int nr = (int)(rx >> 24) & 3;
    for (int k = 0; k < nr; ++k) {
      const int m = (int)(rx >> (8 * k + 4)) & 15;
      const V xs = sel(x, (int)(rx >> (8 * k)) & 15);
      zero = zero || xs < (V)m;
      const O f = comb(xs, m);
      v = k == 0 ? f : v * f;
    }
    return zero ? O(0) : v;
  }
  __device__ static __noinline__ R g_int_slots(uint32_t rx, const long long (&x)[NM]) {
    return g_slots(rx, x, [](long long xs, int m) { return comb_count<R>(xs, m); });
  }
  __device__ static __noinline__ float g_flt_slots(uint32_t rx, const float (&x)[NM]) {
    return g_slots(rx, x, [](float xs, int m) { return comb_factor<float>(xs, m); });
  }
  // Order two at most: 1, x, C(x, 2) or x y.
  __device__ static __forceinline__ float g_flt_word(uint32_t rx, const float (&x)[NM]) {
    const float u = sel(x, (int)rx & 15), v = sel(x, (int)(rx >> 8) & 15);
    const uint32_t nr = rx >> 24;
    const float pair = u < 2.f ? 0.f : (u * (u - 1.f)) * 0.5f;
    const float one = (rx & 0x20u) ? pair : u;
    return nr == 0u ? 1.f : nr == 1u ? one : u * v;
  }
  __device__ static __forceinline__ R g_int_word(uint32_t rx, const long long (&x)[NM]) {
    const uint32_t nr = rx >> 24;
    if constexpr (sizeof(R) == 4) {
      float xf[NM];
#pragma unroll
      for (int s = 0; s < NM; ++s) xf[s] = f32_of_count(x[s]);
      return g_flt_word(rx, xf);
    } else {
      if (nr == 0u) return R(1);
      const long long u = sel(x, (int)rx & 15);
      if (nr == 1u) {
        if (rx & 0x20u) return u < 2 ? R(0) : comb_count<R>(u, 2);
        return of_count<R>(u);
      }
      return of_count<R>(u) * of_count<R>(sel(x, (int)(rx >> 8) & 15));
    }
  }

  // g_j at an integer state (0 when some x_s < m_js), product in increasing s.
  __device__ static __forceinline__ R g_int(const Model& md, int j, const long long (&x)[NM]) {
    if constexpr (!Model::kCompiled) {
      const uint32_t rx = md.rx[j];
      return (int)rx < 0 ? g_int_slots(rx, x) : g_int_word(rx, x);
    } else {
      R v = R(1);
      bool zero = false;
#pragma unroll
      for (int s = 0; s < NM; ++s) {
        const int m = md.ord[j][s];
        if (m != 0) {
          if (x[s] < m) zero = true;
          else v = v * comb_count<R>(x[s], m);
        }
      }
      return zero ? R(0) : v;
    }
  }

  // Fast precision: g_j from an FP32 copy of the state (exact while counts stay below
  // 2^24, where it equals g_int; above, FP32 rounds the count as g_int's conversion does).
  __device__ static __forceinline__ float g_flt(const Model& md, int j, const float (&xf)[NM]) {
    if constexpr (!Model::kCompiled) {
      const uint32_t rx = md.rx[j];
      return (int)rx < 0 ? g_flt_slots(rx, xf) : g_flt_word(rx, xf);
    } else {
      float v = 1.f;
      bool zero = false;
#pragma unroll
      for (int s = 0; s < NM; ++s) {
        const int m = md.ord[j][s];
        if (m != 0) {
          if (xf[s] < (float)m) zero = true;
          else v = v * comb_factor<float>(xf[s], m);
        }
      }
      return zero ? 0.f : v;
    }
  }

  // g_j at a real state (implicit solve), FP64 always.
  __device__ static __forceinline__ double g_real(const Model& md, int j,
                                                  const double (&y)[NM]) {
    double v = 1.0;
    if constexpr (!Model::kCompiled) {
      const uint32_t rx = md.rx[j];
      const int nr = (int)(rx >> 24) & 3;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (k < nr) {
          const int m = (int)(rx >> (8 * k + 4)) & 15;
          const double f = comb_factor<double>(sel(y, (int)(rx >> (8 * k)) & 15), m);
          v = k == 0 ? f : v * f;
        }
      }
    } else {
#pragma unroll
      for (int s = 0; s < NM; ++s) {
        const int m = md.ord[j][s];
        if (m != 0) v = v * comb_factor<double>(y[s], m);
      }
    }
    return v;
  }

  // exact d g_j / d y_q: the product with species q's factor replaced by its derivative
  template <class T>
  __device__ static __forceinline__ T g_real_deriv(const Model& md, int j, const T (&y)[NM],
                                                   int q) {
    T v = T(1);
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const int m = md.ord[j][s];
      if (m != 0) v = v * (s == q ? comb_factor_deriv<T>(y[s], m) : comb_factor<T>(y[s], m));
    }
    return v;
  }

  // The reaction that holds the integral G of reaction j: the lowest one with the same
  // reactants, whose g, and so whose G, is the same number.  Known only where the tables are
  // compiled in (gene expression: 4 integrals for 6 reactions); padded reactions have none.
  __device__ static __forceinline__ constexpr int g_owner(int j) {
    if constexpr (Model::kCompiled) return Model{}.gown[j];
    else return j;
  }

  __device__ static __forceinline__ void eval_props(const Model& md, const long long (&x)[NM],
                                                    const R (&th)[MM], R (&g)[MM], R (&a)[MM]) {
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      g[j] = g_int(md, j, x);
      a[j] = P::mul(th[j], g[j]);
    }
  }

  // Cao 2006 step size over reactions in `use`: per reactant species,
  // mu = sum nu a, var = sum nu^2 a (increasing j, nonzero nu), bound = max(eps x/h, 1),
  // tau_s = min(bound/|mu|, bound^2/var); the minimum over species.
  __device__ static __forceinline__ R tau_select(const Model& md, const R (&a)[MM],
                                                 const long long (&x)[NM], uint32_t use, R eps) {
    if constexpr (Model::kCompiled) return tau_select_at(md, a, x, use, eps);
    else return tau_select_call(md, a, x, use, eps);
  }
  __device__ static __noinline__ R tau_select_call(const Model& md, const R (&a)[MM],
                                                   const long long (&x)[NM], uint32_t use,
                                                   R eps) {
    return tau_select_at(md, a, x, use, eps);
  }
  __device__ static __forceinline__ R tau_select_at(const Model& md, const R (&a)[MM],
                                                    const long long (&x)[NM], uint32_t use,
                                                    R eps) {
    R tau = P::inf();
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      if (md.isreact[s]) {
        R mu = R(0), var = R(0);
#pragma unroll
        for (int j = 0; j < MM; ++j) {
          const int v = md.nu[j][s];
          if (((use >> j) & 1u) && v != 0) {
            if (P::kRef && (v == 1 || v == -1)) {  // the products are exact
              mu = v > 0 ? mu + a[j] : mu - a[j];
              var = var + a[j];
            } else {
              mu = P::mad((R)v, a[j], mu);
              var = P::mad((R)(v * v), a[j], var);
            }
          }
        }
        R bound = eps * of_count<R>(x[s]);
        if (md.hor[s] != kHorO1)  // h = 1 for a first-order reactant
          bound = bound / hor_factor<R, Model::kCompiled>(md.hor[s], x[s]);
        if (P::lt(bound, R(1))) bound = R(1);
        const R t1 = bound / fabs(mu);
        const R t2 = (bound * bound) / var;
        const R ts = P::lt(t1, t2) ? t1 : t2;
        if (P::lt(ts, tau)) tau = ts;
      }
    }
    return tau;
  }

  // Implicit leap (Rathinam 2003): solve y = c + tau sum_j nu_j a_j(y) over the
  // non-critical reactions by Newton's method: residual, iterate and stopping test in
  // FP64; the Jacobian (forward differences or exact) assembled and factorized by Gaussian
  // elimination with partial pivoting and column-oriented back substitution in the
  // working precision R (FP64 in reference precision; FP32 in fast precision, where an
  // approximate Jacobian changes only the rate of convergence, not the FP64 root).
  // Returns 0 converged, 1 not converged, 2 singular.
  __device__ static __forceinline__ int implicit_solve(const Model& md, const R (&th)[MM],
                                       const long long (&x)[NM], uint32_t nc,
                                       const long long (&Pk)[MM], const R (&a)[MM],
                                       double tau, double tol, int maxit, double fd_h,
                                       bool analytic, double (&y)[NM]) {
    double c[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const double xs = f64_of_count(x[s]);
      double acc = xs;
#pragma unroll
      for (int j = 0; j < MM; ++j) {
        const int v = md.nu[j][s];
        if (((nc >> j) & 1u) && v != 0)
          acc = acc + nu_times(v, f64_of_count(Pk[j]) - (double)a[j] * tau);
      }
      c[s] = acc;
      y[s] = xs;
    }
    const R taur = (R)tau;
    for (int it = 0; it < maxit; ++it) {
      double ay[MM];
#pragma unroll
      for (int j = 0; j < MM; ++j) ay[j] = (double)th[j] * g_real(md, j, y);
      R A[NM][NM], b[NM];
#pragma unroll
      for (int s = 0; s < NM; ++s) {
        double acc = 0.0;
#pragma unroll
        for (int j = 0; j < MM; ++j) {
          const int v = md.nu[j][s];
          if (((nc >> j) & 1u) && v != 0) acc = acc + nu_times(v, ay[j]);
        }
        b[s] = (R)(-((y[s] - c[s]) - tau * acc));
      }
      R yr[NM];
#pragma unroll
      for (int s = 0; s < NM; ++s) yr[s] = (R)y[s];
#pragma unroll
      for (int q = 0; q < NM; ++q) {
        R Dq[MM];
        if (analytic) {
#pragma unroll
          for (int j = 0; j < MM; ++j)
            Dq[j] = (((nc >> j) & 1u) && md.ord[j][q] != 0)
                        ? th[j] * g_real_deriv<R>(md, j, yr, q)
                        : R(0);
        } else {
          const double aq = fabs(y[q]);
          const double h = fd_h * (aq > 1.0 ? aq : 1.0);
          double yq[NM];
#pragma unroll
          for (int s = 0; s < NM; ++s) yq[s] = y[s];
          yq[q] = y[q] + h;
          const double he = yq[q] - y[q];
#pragma unroll
          for (int j = 0; j < MM; ++j)
            Dq[j] = (((nc >> j) & 1u) && md.ord[j][q] != 0)
                        ? (R)(((double)th[j] * g_real(md, j, yq) - ay[j]) / he)
                        : R(0);
        }
#pragma unroll
        for (int s = 0; s < NM; ++s) {
          R acc = R(0);
#pragma unroll
          for (int j = 0; j < MM; ++j) {
            const int v = md.nu[j][s];
            if (((nc >> j) & 1u) && v != 0 && md.ord[j][q] != 0)
              acc = acc + nu_times(v, Dq[j]);
          }
          A[s][q] = (s == q ? R(1) : R(0)) - taur * acc;
        }
      }
      // elimination with partial pivoting (row swaps by compile-time selects)
#pragma unroll
      for (int k = 0; k < NM; ++k) {
        int piv = k;
        R best = fabs(A[k][k]);
#pragma unroll
        for (int i = k + 1; i < NM; ++i) {
          if (f64_abs_gt(A[i][k], best)) {
            best = fabs(A[i][k]);
            piv = i;
          }
        }
        if (P::zero(best)) return 2;
#pragma unroll
        for (int i = k + 1; i < NM; ++i) {
          if (i == piv) {
#pragma unroll
            for (int cc = 0; cc < NM; ++cc) {
              const R tmp = A[k][cc];
              A[k][cc] = A[i][cc];
              A[i][cc] = tmp;
            }
            const R tb = b[k];
            b[k] = b[i];
            b[i] = tb;
          }
        }
#pragma unroll
        for (int i = k + 1; i < NM; ++i) {
          const R l = A[i][k] / A[k][k];
#pragma unroll
          for (int cc = k + 1; cc < NM; ++cc) A[i][cc] = A[i][cc] - l * A[k][cc];
          b[i] = b[i] - l * b[k];
        }
      }
      R d[NM];
#pragma unroll
      for (int i = NM - 1; i >= 0; --i) {
        d[i] = b[i] / A[i][i];
#pragma unroll
        for (int rr = 0; rr < i; ++rr) b[rr] = b[rr] - A[rr][i] * d[i];
      }
      double dmax = 0.0, ymax = 0.0;
#pragma unroll
      for (int s = 0; s < NM; ++s) {
        const double ds = (double)d[s];
        y[s] = y[s] + ds;
        if (fabs(ds) > dmax) dmax = fabs(ds);
        if (fabs(y[s]) > ymax) ymax = fabs(y[s]);
      }
      if (dmax <= tol * (ymax > 1.0 ? ymax : 1.0)) return 0;
    }
    return 1;
  }

  // g_j(x + z) - g_j(x) over the reactant species in increasing s, by the recursion
  // D <- f(u) D + (f(u) - f(x)) B, B <- f(x) B with f = C(., m_js), u = x + z.
  __device__ static __forceinline__ R g_diff(const Model& md, int j, const R (&xf)[NM],
                                             const R (&z)[NM]) {
    R D = R(0), B = R(1);
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const int m = md.ord[j][s];
      if (m != 0) {
        D = comb_factor<R>(xf[s] + z[s], m) * D + comb_diff<R>(xf[s], z[s], m) * B;
        B = comb_factor<R>(xf[s], m) * B;
      }
    }
    return D;
  }

  // Fast precision: the implicit leap for the increment z = y - x, entirely in FP32.  The
  // equation z = c + tau sum_j nu_j theta_j (g_j(x + z) - g_j(x)), c_s = sum_j nu_js P_j
  // (an exact integer sum), has no cancellation between propensities of size a tau: the
  // differences of the binomial factors are polynomials in z.  So FP32 keeps the firing
  // counts K_j = P_j + round(tau theta_j (g_j(x + z) - g_j(x))) within rounding of the
  // FP64 solution (on dimerisation states one leap in about 200 differs by one firing,
  // with no preferred sign).  The stopping test uses max(tol, 1e-6) (FP32 cannot resolve
  // 1e-10).  On success K holds the counts.  The Jacobian is always the exact one (the paper's symbolic Jacobian): in
  // this FP32 solve it only sets the rate of convergence, the exact derivative is the
  // cheaper to evaluate, and leaving out the forward-difference variant keeps the
  // generic 8 x 16 build compact.  Returns 0 converged, 1 not converged, 2 singular.
  __device__ static __forceinline__ int implicit_solve_fast(const Model& md, const R (&th)[MM],
                                            const long long (&x)[NM], uint32_t nc,
                                            long long (&K)[MM], R tau,
                                            double tol, int maxit) {
    R xf[NM], z[NM], c[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      xf[s] = (R)x[s];
      z[s] = R(0);
      long long cs = 0;
#pragma unroll
      for (int j = 0; j < MM; ++j)
        if ((nc >> j) & 1u) cs += (long long)md.nu[j][s] * K[j];
      c[s] = (R)cs;
    }
    const R tolr = tol > 1e-6 ? (R)tol : R(1e-6);
    for (int it = 0; it < maxit; ++it) {
      R dg[MM];
#pragma unroll
      for (int j = 0; j < MM; ++j) dg[j] = ((nc >> j) & 1u) ? g_diff(md, j, xf, z) : R(0);
      R A[NM][NM], b[NM], yr[NM];
#pragma unroll
      for (int s = 0; s < NM; ++s) {
        R acc = R(0);
#pragma unroll
        for (int j = 0; j < MM; ++j) {
          const int v = md.nu[j][s];
          if (((nc >> j) & 1u) && v != 0) acc = acc + (R)v * (th[j] * dg[j]);
        }
        b[s] = -((z[s] - c[s]) - tau * acc);
        yr[s] = xf[s] + z[s];
      }
#pragma unroll
      for (int q = 0; q < NM; ++q) {
        R Dq[MM];
#pragma unroll
        for (int j = 0; j < MM; ++j)
          Dq[j] = (((nc >> j) & 1u) && md.ord[j][q] != 0)
                      ? th[j] * g_real_deriv<R>(md, j, yr, q)
                      : R(0);
#pragma unroll
        for (int s = 0; s < NM; ++s) {
          R acc = R(0);
#pragma unroll
          for (int j = 0; j < MM; ++j) {
            const int v = md.nu[j][s];
            if (((nc >> j) & 1u) && v != 0 && md.ord[j][q] != 0) acc = acc + (R)v * Dq[j];
          }
          A[s][q] = (s == q ? R(1) : R(0)) - tau * acc;
        }
      }
#pragma unroll
      for (int k = 0; k < NM; ++k) {
        int piv = k;
        R best = fabs(A[k][k]);
#pragma unroll
        for (int i = k + 1; i < NM; ++i) {
          if (fabs(A[i][k]) > best) {
            best = fabs(A[i][k]);
            piv = i;
          }
        }
        if (!(best > R(0))) return 2;
#pragma unroll
        for (int i = k + 1; i < NM; ++i) {
          if (i == piv) {
#pragma unroll
            for (int cc = 0; cc < NM; ++cc) {
              const R tmp = A[k][cc];
              A[k][cc] = A[i][cc];
              A[i][cc] = tmp;
            }
            const R tb = b[k];
            b[k] = b[i];
            b[i] = tb;
          }
        }
#pragma unroll
        for (int i = k + 1; i < NM; ++i) {
          const R l = A[i][k] / A[k][k];
#pragma unroll
          for (int cc = k + 1; cc < NM; ++cc) A[i][cc] = A[i][cc] - l * A[k][cc];
          b[i] = b[i] - l * b[k];
        }
      }
      R d[NM];
#pragma unroll
      for (int i = NM - 1; i >= 0; --i) {
        d[i] = b[i] / A[i][i];
#pragma unroll
        for (int rr = 0; rr < i; ++rr) b[rr] = b[rr] - A[rr][i] * d[i];
      }
      R dmax = R(0), ymax = R(0);
#pragma unroll
      for (int s = 0; s < NM; ++s) {
        z[s] = z[s] + d[s];
        if (fabs(d[s]) > dmax) dmax = fabs(d[s]);
        const R ys = fabs(xf[s] + z[s]);
        if (ys > ymax) ymax = ys;
      }
      if (!(dmax == dmax)) return 1;
      if (dmax <= tolr * (ymax > R(1) ? ymax : R(1))) {
#pragma unroll
        for (int j = 0; j < MM; ++j) {
          if ((nc >> j) & 1u) {
            const R d = tau * (th[j] * g_diff(md, j, xf, z));
            if (!(d < R(kLeapLimit))) {  // beyond the leap limit (or NaN): saturate
              K[j] = kCountLimit;
            } else {
              const long long kj = K[j] + llroundf(d);
              K[j] = kj > 0 ? kj : 0;
            }
          }
        }
        return 0;
      }
    }
    return 1;
  }

  // Inverse-CDF pick of a reaction with probability v_j / sum v, from the second uniform
  // of block w (words 2, 3).  Reference: sequential prefix sums in index order (the
  // canonical order), target u * sum with the lane-tree sum.  Fast: see pick_fast.
  // Rounding that leaves no hit picks the last positive entry.
  // tot: the lane-tree sum of v (reference precision).
  __device__ static __forceinline__ int pick_reaction(const R (&v)[MM], const Words4& w,
                                                      R tot) {
    if constexpr (!P::kRef) {
      return pick_fast(v, w);
    } else {
      bool clear;
      const int pk = pick_near(v, w, clear);
      return clear ? pk : pick_ref(v, w, tot);
    }
  }

  // Reference precision's pick, first in FP32 on truncated values: they are off by 2^-23
  // relative, each of the M sums by 2^-24, so prefixes and total lie within (M + 2) 2^-24
  // tot of the FP64 ones (themselves within M 2^-53 tot of exact) and the target, with the
  // uniform's upper 24 bits, within (M + 5) 2^-24 tot; when the target is farther than
  // (M + 4) 2^-23 tot from every prefix the FP64 search gives the same reaction.  Otherwise
  // (about 1e-5 of the picks), and when the total is outside FP32's middle range, the FP64
  // search has to run: M additions, a product and comparisons on the FP64 unit.
  __device__ static __forceinline__ int pick_near(const R (&v)[MM], const Words4& w,
                                                  bool& clear) {
    float pre[MM];
    float acc = 0.f;
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      acc = acc + f32_near((double)v[j]);
      pre[j] = acc;
    }
    const int pk = search_prefix(pre, w.w2, MM + 4, clear);
    clear = clear && acc > 0x1p-60f && acc < 0x1p60f;
    return pk;
  }

  // An FP64 value in [0, 2^127) as FP32 within 2^-23 relative (truncated; below the FP32
  // normal range 0; beyond it infinity, which the caller's range test catches).
  __device__ static __forceinline__ float f32_near(double d) {
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    if (hi < 0x38100000u) return 0.f;
    if (hi >= 0x47e00000u) return inf32();
    return __uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29));
  }
  __device__ static __forceinline__ float inf32() { return __int_as_float(0x7f800000); }

  __device__ static __noinline__ int pick_ref(const R (&v)[MM], const Words4& w, R tot) {
    int pk = -1, last = -1;
    const R target = P::u(w, 1) * tot;
    R acc = R(0);
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      if (P::positive(v[j])) last = j;
      acc = acc + v[j];
      if (pk < 0 && P::lt(target, acc)) pk = j;
    }
    return pk < 0 ? last : pk;
  }

  // The reaction whose prefix interval holds the target, by FP32 prefix sums `pre` (the
  // last one the total) and the upper 24 bits of the uniform; clear = the target is farther
  // than `ulps` 2^-23 of the total from every prefix.
  __device__ static __forceinline__ int search_prefix(const float (&pre)[MM], uint32_t w2,
                                                      int ulps, bool& clear) {
    const float target = (float)(w2 >> 8) * 0x1p-24f * pre[MM - 1];
    const float margin = (float)ulps * 0x1p-23f * pre[MM - 1];
    int pk = 0;
    float near = inf32();
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      pk += pre[j] <= target ? 1 : 0;
      near = fminf(near, fabsf(pre[j] - target));
    }
    clear = near > margin && pk < MM;
    return pk;
  }

  // Fast precision pick with a 48-bit uniform u = (w2>>8) 2^-24 + ((w3>>8) + 1/2) 2^-48.
  // First in FP32: prefix sums P_j and the target (w2>>8) 2^-24 P_{M-1}.  Against exact
  // arithmetic each P_j is off by less than M 2^-24 P_{M-1} and the target by less than
  // (M + 1) 2^-24 P_{M-1}, so when the target is farther than (M + 2) 2^-23 P_{M-1} from
  // every P_j the FP32 search selects the reaction the exact one does.  Otherwise (about
  // 2 M (M + 2) 2^-23 of the picks, ~1e-5) the double-float search decides, which keeps
  // reactions many decades below the total at their exact share.
  __device__ static __forceinline__ int pick_fast(const R (&v)[MM], const Words4& w) {
    float pre[MM];
    float acc = 0.f;
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      acc = acc + (float)v[j];
      pre[j] = acc;
    }
    bool clear;
    const int pk = search_prefix(pre, w.w2, MM + 2, clear);
    return clear ? pk : pick_df(v, w);
  }

  // The same search over double-float (TwoSum) prefix sums of the FP32 values with the
  // full 48-bit uniform; rarely taken, so kept out of line.
  __device__ static __noinline__ int pick_df(const R (&v)[MM], const Words4& w) {
    int pk = -1, last = -1;
    DF pre[MM];
    DF acc{0.f, 0.f};
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      if (v[j] > R(0)) last = j;
      acc = df_add(acc, (float)v[j]);
      pre[j] = acc;
    }
    const DF target = df_uniform_times(acc, w.w2, w.w3);
#pragma unroll
    for (int j = 0; j < MM; ++j)
      if (pk < 0 && df_lt(target, pre[j])) pk = j;
    return pk < 0 ? last : pk;
  }

};


// Inputs and outputs of one implicit leap of the fast kernels, passed to the non-inlined
// solve through local memory so that the leap loop's arrays stay in registers.
template <int NM, int MM>
struct ImplicitIo {
  long long x[NM];
  long long K[MM];  // in: Poisson draws P_j (and the critical firing); out: firing counts
  float th[MM];
};

// 1 / b within 0.501 ulp: with FP32's reciprocal y (within 2^-21) and e = 1 - b y, the sum
// y + y (e + e^2) misses 1 / b by e^3 before its rounding, so it is the rounded quotient but
// for at most one b in a thousand (then its neighbour).  Three FP64 instructions; used where
// fast precision's Newton system divides by a difference step or a pivot.
__device__ __forceinline__ double near_recip(double b) {
  const uint32_t ex = ((uint32_t)__double2hiint(b) >> 20) & 0x7ffu;
  if (ex - 923u > 200u) return 1.0 / b;
  const double y = f64_of_f32(__fdividef(1.f, f32_of_f64(b)));
  const double e = __fma_rn(-b, y, 1.0);
  return __fma_rn(y, __fma_rn(e, e, e), y);
}

// The implicit leap on tables read at run time: the operations of implicit_solve (kRecip
// false: the canonical order, a division per Jacobian entry, eliminated row and unknown) or of
// implicit_leap_wide (true: reciprocals), with loops over the real sizes and arrays in local
// memory.  The unrolled form carries a branch per (reaction, species, order) and a division
// sequence per Jacobian entry: the precompiled reference kernel waited 20 cycles for an
// instruction (20,000 dimerisation trajectories), while a local load is short beside the 64
// cycles of an FP64 instruction.  Entries that are zero need no elimination.  On success K
// holds the firing counts.  Returns 0 converged, 1 not converged, 2 singular.
template <int NM, int MM, class MDL, bool kRecip>
__device__ __noinline__ int implicit_leap_rolled(const MDL& md, const long long (&x)[NM],
                                                 long long (&K)[MM], const double (&th)[MM],
                                                 const double (&ax)[MM], uint32_t nc, double tau,
                                                 double tol, int maxit, double fd_h,
                                                 bool analytic) {
  const int N = md.N, M = md.M;
  double y[NM], c[NM], ay[MM], yp[NM], he[NM], A[NM][NM], b[NM], inv[NM];
  auto g_at = [&](uint32_t rx) {
    double v = 1.0;
    const int nr = (int)(rx >> 24) & 3;
#pragma unroll 1
    for (int k = 0; k < nr; ++k) {
      const double f = comb_factor<double>(y[(rx >> (8 * k)) & 15], (int)(rx >> (8 * k + 4)) & 15);
      v = k == 0 ? f : v * f;
    }
    return v;
  };
#pragma unroll 1
  for (int s = 0; s < N; ++s) {
    y[s] = f64_of_count(x[s]);
    double acc = y[s];
#pragma unroll 1
    for (int j = 0; j < M; ++j) {
      const int v = md.nu[j][s];
      if (((nc >> j) & 1u) && v != 0) acc = acc + nu_times(v, f64_of_count(K[j]) - ax[j] * tau);
    }
    c[s] = acc;
  }
  int rc = 1;
#pragma unroll 1
  for (int it = 0; it < maxit; ++it) {
#pragma unroll 1
    for (int j = 0; j < M; ++j) ay[j] = th[j] * g_at(md.rx[j]);
#pragma unroll 1
    for (int s = 0; s < N; ++s) {
      double acc = 0.0;
#pragma unroll 1
      for (int j = 0; j < M; ++j) {
        const int v = md.nu[j][s];
        if (((nc >> j) & 1u) && v != 0) acc = acc + nu_times(v, ay[j]);
      }
      b[s] = -((y[s] - c[s]) - tau * acc);
#pragma unroll 1
      for (int q = 0; q < N; ++q) A[s][q] = 0.0;
      if (!analytic) {
        const double h = fd_h * (f64_abs_gt(y[s], 1.0) ? fabs(y[s]) : 1.0);
        yp[s] = y[s] + h;
        he[s] = yp[s] - y[s];
        if (kRecip) he[s] = near_recip(he[s]);
      }
    }
#pragma unroll 1
    for (int j = 0; j < M; ++j) {
      const uint32_t rx = md.rx[j];
      const int nr = ((nc >> j) & 1u) ? (int)(rx >> 24) & 3 : 0;
#pragma unroll 1
      for (int k = 0; k < nr; ++k) {
        const int q = (int)(rx >> (8 * k)) & 15;
        double D;
        if (analytic) {
          double v = 1.0;
#pragma unroll 1
          for (int kk = 0; kk < nr; ++kk) {
            const double yv = y[(rx >> (8 * kk)) & 15];
            const int m = (int)(rx >> (8 * kk + 4)) & 15;
            v = v * (kk == k ? comb_factor_deriv<double>(yv, m) : comb_factor<double>(yv, m));
          }
          D = th[j] * v;
        } else {
          const double keep = y[q];
          y[q] = yp[q];
          const double diff = th[j] * g_at(rx) - ay[j];
          y[q] = keep;
          D = kRecip ? diff * he[q] : diff / he[q];
        }
#pragma unroll 1
        for (int s = 0; s < N; ++s) {
          const int v = md.nu[j][s];
          if (v != 0) A[s][q] = A[s][q] + nu_times(v, D);
        }
      }
    }
#pragma unroll 1
    for (int s = 0; s < N; ++s) {
#pragma unroll 1
      for (int q = 0; q < N; ++q) {
        const double e = s == q ? 1.0 : 0.0;
        A[s][q] = (__double_as_longlong(A[s][q]) << 1) == 0 ? e : e - tau * A[s][q];
      }
    }
#pragma unroll 1
    for (int k = 0; k < N; ++k) {
      int piv = k;
      double best = fabs(A[k][k]);
#pragma unroll 1
      for (int i = k + 1; i < N; ++i) {
        if (f64_abs_gt(A[i][k], best)) {
          best = fabs(A[i][k]);
          piv = i;
        }
      }
      if (kRecip ? !f64_abs_gt(best, 0.0) : best == 0.0) return 2;
      if (piv != k) {
#pragma unroll 1
        for (int cc = 0; cc < N; ++cc) {
          const double t = A[k][cc];
          A[k][cc] = A[piv][cc];
          A[piv][cc] = t;
        }
        const double t = b[k];
        b[k] = b[piv];
        b[piv] = t;
      }
      if (kRecip) inv[k] = near_recip(A[k][k]);
#pragma unroll 1
      for (int i = k + 1; i < N; ++i) {
        if ((__double_as_longlong(A[i][k]) << 1) == 0) continue;
        const double l = kRecip ? A[i][k] * inv[k] : A[i][k] / A[k][k];
#pragma unroll 1
        for (int cc = k + 1; cc < N; ++cc) A[i][cc] = A[i][cc] - l * A[k][cc];
        b[i] = b[i] - l * b[k];
      }
    }
    double dmax = 0.0, ymax = 0.0;
#pragma unroll 1
    for (int i = N - 1; i >= 0; --i) {
      const double d = kRecip ? b[i] * inv[i] : b[i] / A[i][i];
#pragma unroll 1
      for (int rr = 0; rr < i; ++rr) b[rr] = b[rr] - A[rr][i] * d;
      y[i] = y[i] + d;
      if (f64_abs_gt(d, dmax)) dmax = fabs(d);
      if (f64_abs_gt(y[i], ymax)) ymax = fabs(y[i]);
    }
    if (dmax <= tol * (ymax > 1.0 ? ymax : 1.0)) {
      rc = 0;
      break;
    }
  }
  if (rc == 0) {
#pragma unroll 1
    for (int j = 0; j < M; ++j) {
      if ((nc >> j) & 1u) {
        const double v = (th[j] * g_at(md.rx[j]) * tau + f64_of_count(K[j])) - ax[j] * tau;
        const double rv = round(v);
        K[j] = !(rv < 0x1p62) ? kCountLimit : (rv > 0.0 ? (long long)rv : 0);
      }
    }
  }
  return rc;
}

// Fast precision, FP64 implicit leap (Rathinam 2003): FP64 propensities a_j(x) =
// theta_j g_j(x) from the FP32 rate constants, Newton's method from y = x with the FP64
// residual F(y) = y - c - tau sum_j nu_j a_j(y), Jacobian (forward differences or exact),
// partial pivoting and stopping test max |dy| <= tol max(1, max |y|), then
// K_j = max(0, round((a_j(y) tau + P_j) - a_j(x) tau)) for the non-critical reactions.
// Unlike the reference solve it need not reproduce a fixed operation order, so it divides
// once per species and pivot (reciprocals of the difference steps and pivots) instead of
// once per Jacobian entry and eliminated element: FP64 division is a long instruction
// sequence on this GPU.  Not inlined: its FP64 working set stays out of the register
// allocation of the leap loop.  Returns 0 converged, 1 not converged, 2 singular.
template <int NM, int MM, class MDL>
__device__ __noinline__ int implicit_leap_wide(const MDL& md,
                                               ImplicitIo<NM, MM>& io, uint32_t nc,
                                               double tau, double tol, int maxit, double fd_h,
                                               bool analytic) {
  using TR = ThreadTraj<NM, MM, PrecRef, MDL>;
  double th[MM], ax[MM], y[NM], c[NM];
#pragma unroll
  for (int j = 0; j < MM; ++j) {
    th[j] = f64_of_f32(io.th[j]);
    ax[j] = th[j] * TR::g_int(md, j, io.x);
  }
  if constexpr (!MDL::kCompiled)
    return implicit_leap_rolled<NM, MM, MDL, true>(md, io.x, io.K, th, ax, nc, tau, tol, maxit,
                                                   fd_h, analytic);
#pragma unroll
  for (int s = 0; s < NM; ++s) {
    const double xs = f64_of_count(io.x[s]);
    double acc = xs;
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      const int v = md.nu[j][s];
      if (((nc >> j) & 1u) && v != 0) acc += nu_times(v, f64_of_count(io.K[j]) - ax[j] * tau);
    }
    c[s] = acc;
    y[s] = xs;
  }
  int rc = 1;
  for (int it = 0; it < maxit && rc == 1; ++it) {
    double ay[MM];
#pragma unroll
    for (int j = 0; j < MM; ++j) ay[j] = ((nc >> j) & 1u) ? th[j] * TR::g_real(md, j, y) : 0.0;
    double A[NM][NM], b[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      double acc = 0.0;
#pragma unroll
      for (int j = 0; j < MM; ++j) {
        const int v = md.nu[j][s];
        if (v != 0) acc += nu_times(v, ay[j]);
      }
      b[s] = -((y[s] - c[s]) - tau * acc);
    }
#pragma unroll
    for (int q = 0; q < NM; ++q) {
      double Dq[MM];
      if (analytic) {
#pragma unroll
        for (int j = 0; j < MM; ++j)
          Dq[j] = (((nc >> j) & 1u) && md.ord[j][q] != 0)
                      ? th[j] * TR::template g_real_deriv<double>(md, j, y, q)
                      : 0.0;
      } else {
        double yq[NM];
#pragma unroll
        for (int s = 0; s < NM; ++s) yq[s] = y[s];
        yq[q] = y[q] + fd_h * (f64_abs_gt(y[q], 1.0) ? fabs(y[q]) : 1.0);
        const double inv_h = near_recip(yq[q] - y[q]);
#pragma unroll
        for (int j = 0; j < MM; ++j)
          Dq[j] = (((nc >> j) & 1u) && md.ord[j][q] != 0)
                      ? (th[j] * TR::g_real(md, j, yq) - ay[j]) * inv_h
                      : 0.0;
      }
#pragma unroll
      for (int s = 0; s < NM; ++s) {
        double acc = 0.0;
#pragma unroll
        for (int j = 0; j < MM; ++j) {
          const int v = md.nu[j][s];
          if (v != 0 && md.ord[j][q] != 0) acc += nu_times(v, Dq[j]);
        }
        A[s][q] = (s == q ? 1.0 : 0.0) - tau * acc;
      }
    }
    double inv_piv[NM];
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      int piv = k;
      double best = fabs(A[k][k]);
#pragma unroll
      for (int i = k + 1; i < NM; ++i) {
        if (f64_abs_gt(A[i][k], best)) {
          best = fabs(A[i][k]);
          piv = i;
        }
      }
      if (!f64_abs_gt(best, 0.0)) {
        rc = 2;
        break;
      }
#pragma unroll
      for (int i = k + 1; i < NM; ++i) {
        if (i == piv) {
#pragma unroll
          for (int cc = 0; cc < NM; ++cc) {
            const double tmp = A[k][cc];
            A[k][cc] = A[i][cc];
            A[i][cc] = tmp;
          }
          const double tb = b[k];
          b[k] = b[i];
          b[i] = tb;
        }
      }
      inv_piv[k] = near_recip(A[k][k]);
#pragma unroll
      for (int i = k + 1; i < NM; ++i) {
        const double l = A[i][k] * inv_piv[k];
#pragma unroll
        for (int cc = k + 1; cc < NM; ++cc) A[i][cc] -= l * A[k][cc];
        b[i] -= l * b[k];
      }
    }
    if (rc == 2) break;
    double dmax = 0.0, ymax = 0.0;
#pragma unroll
    for (int i = NM - 1; i >= 0; --i) {
      const double d = b[i] * inv_piv[i];
#pragma unroll
      for (int rr = 0; rr < i; ++rr) b[rr] -= A[rr][i] * d;
      y[i] += d;
      dmax = f64_abs_gt(d, dmax) ? fabs(d) : dmax;
    }
#pragma unroll
    for (int s = 0; s < NM; ++s) ymax = f64_abs_gt(y[s], ymax) ? fabs(y[s]) : ymax;
    if (dmax <= tol * (ymax > 1.0 ? ymax : 1.0)) rc = 0;
  }
  if (rc == 0) {
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      if ((nc >> j) & 1u) {
        const double v = (th[j] * TR::g_real(md, j, y) * tau + (double)io.K[j]) - ax[j] * tau;
        const double rv = round(v);
        io.K[j] = !(rv < 0x1p62) ? kCountLimit : (rv > 0.0 ? (long long)rv : 0);
      }
    }
  }
  return rc;
}

// Fast precision, FP32 implicit leap for the increment z = y - x (ThreadTraj::
// implicit_solve_fast), also not inlined.
template <int NM, int MM, class MDL>
__device__ __noinline__ int implicit_leap_fp32(const MDL& md,
                                               ImplicitIo<NM, MM>& io, uint32_t nc, float tau,
                                               double tol, int maxit) {
  using TF = ThreadTraj<NM, MM, PrecFast, MDL>;
  float th[MM];
  long long x[NM], K[MM];
#pragma unroll
  for (int j = 0; j < MM; ++j) {
    th[j] = io.th[j];
    K[j] = io.K[j];
  }
#pragma unroll
  for (int s = 0; s < NM; ++s) x[s] = io.x[s];
  const int rc = TF::implicit_solve_fast(md, th, x, nc, K, tau, tol, maxit);
#pragma unroll
  for (int j = 0; j < MM; ++j) io.K[j] = K[j];
  return rc;
}

// One trajectory per thread, driven as a per-lane state machine so that a warp does not
// hold lanes in one phase while others run a long phase: a step of the machine is either
// one leap evaluation (propensities, critical set, step sizes, leap or burst decision) or
// a bounded slice of the SSA burst.  The drivers below (round-based, pool, sequential)
// only decide which lane runs which step when; each lane performs exactly the arithmetic
// of the sequential algorithm, so results do not depend on the schedule.  MDL: the model
// tables read at run time (ThreadModel in shared memory) or compiled in (specialized
// kernels).
// kGrid: time-grid output compiled in.  Without it the grid code is absent, so the
// kernels that serve calls without a grid are exactly the plain simulation.
constexpr int kSsaPerRound = 8;  // firings of a slice
constexpr int kUnit = 4;         // firings done together without a branch

template <int NM, int MM, class P, bool kGrid = false, class MDL = ThreadModel<NM, MM>>
struct ThreadLane {
  static_assert(kSsaPerRound < 16 && MM <= 16, "a slice's firings are 4 bits per reaction");
  using R = typename P::R;
  using TT = ThreadTraj<NM, MM, P, MDL>;
  using Model = MDL;
  enum : int { kIdle = 0, kEval = 1, kSsa = 2, kDone = 3 };

  long long i;
  uint32_t id, status, step;
  int reject_run, mode;
  int kobs;  // next unrecorded grid point
  double t, T;
  R th[MM];
  long long x[NM];
  long long r[MM];
  double G[MM];
  long long cnt[4];
  R g[MM], a[MM];
  // SSA burst
  int b, n_max;
  R a0;

  __device__ __forceinline__ void start(const Model& md, const SimArgs& A, long long idx) {
    i = idx;
    id = (uint32_t)(A.id_base + (unsigned long long)idx);
    status = 0;
    bool bad = false;
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      double v = 0.0;
      if (j < A.M) v = A.theta ? A.theta[idx * A.M + j] : md.rates[j];
      if (!(v >= 0.0)) bad = true;
      th[j] = (R)v;
    }
    const int64_t* x0 = A.x0_per ? A.x0 + idx * A.N : A.x0;
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      x[s] = s < A.N ? x0[s] : 0;
      if (x[s] < 0) bad = true;
    }
    T = A.T_per ? A.T[idx] : A.T[0];
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      r[j] = 0;
      G[j] = 0.0;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) cnt[c] = 0;
    t = 0.0;
    step = 0;
    reject_run = 0;
    if (kGrid) kobs = 0;
    if (kGrid && A.K_obs > 0 && !grid_ok(A)) bad = true;
    if (bad) {
      status |= ML_ST_BAD_INPUT;
      t = T;
    }
    if (T != T) {  // NaN horizon: finishes at once
      t = 0.0;
      T = -1.0;
    }
    mode = kEval;
    if (kGrid && A.K_obs > 0) record(A, t, true);  // grid points at t = 0 see x0
  }

  // Time-grid output.  The path is right-continuous and piecewise constant (it changes
  // at SSA firings and at the ends of leaps), so X(t_k) is the state after every change
  // at a time <= t_k.  Writes the current state to each pending point with t_k < tcut
  // (strict) or t_k <= tcut (inclusive).
  __device__ __forceinline__ void record(const SimArgs& A, double tcut, bool inclusive) {
    while (kobs < A.K_obs) {
      const double tk = __ldg(A.t_obs + kobs);
      if (inclusive ? !(tk <= tcut) : !(tk < tcut)) break;
      int64_t* o = A.X_obs + ((long long)i * A.K_obs + kobs) * A.N;
#pragma unroll
      for (int s = 0; s < NM; ++s)
        if (s < A.N) o[s] = x[s];
      ++kobs;
    }
  }

  // A leap ends exactly at the next grid point, as it does at T.
  __device__ __forceinline__ double stop_time(const SimArgs& A) const {
    if (kobs < A.K_obs) {
      const double tk = __ldg(A.t_obs + kobs);
      if (tk < T) return tk;
    }
    return T;
  }

  __device__ static bool grid_ok(const SimArgs& A) {
    double prev = 0.0;
    for (int k = 0; k < A.K_obs; ++k) {
      const double tk = __ldg(A.t_obs + k);
      if (!(tk >= prev) || !(tk <= 1.0e300)) return false;
      prev = tk;
    }
    return true;
  }

  __device__ __forceinline__ void finish(const SimArgs& A, bool staged) {
    // grid points past the end (beyond T, after a step-limit stop, or all of a rejected
    // grid) see the final state
    if (kGrid) {
      for (; kobs < A.K_obs; ++kobs) {
        int64_t* o = A.X_obs + ((long long)i * A.K_obs + kobs) * A.N;
#pragma unroll
        for (int s = 0; s < NM; ++s)
          if (s < A.N) o[s] = x[s];
      }
    }
#pragma unroll
    for (int s = 0; s < NM; ++s)
      if (s < A.N) A.X[i * A.N + s] = x[s];
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      if (j < A.M) {
        A.r[i * A.M + j] = r[j];
        A.G[i * A.M + j] = G[TT::g_owner(j)];
      }
    }
    A.status[i] = status | (staged ? 0u : ML_ST_STAGE_TIMEOUT);
    if (A.counters) {
#pragma unroll
      for (int c = 0; c < 4; ++c) A.counters[i * 4 + c] = cnt[c];
    }
    mode = kIdle;
  }

  // The lane state as 32-bit words of a shared-memory record (pool driver): word k of
  // slot q at rec[k * kPoolSlots + q], the mode first.  g, a and a0 are not kept: a
  // loaded lane recomputes them from x and theta before use.
  template <class MD>
  __device__ static constexpr int g_owner_count() {
    if constexpr (MD::kCompiled) return MD::n_gown;
    else return MM;
  }
  static constexpr int kRWords = (int)(sizeof(R) / 4);
  static constexpr int kWords =
      lane_record_words(NM, MM, kRWords == 2) - 2 * (MM - g_owner_count<Model>());
  template <int S>
  __device__ __forceinline__ void save(uint32_t* rec, int q) const {
    int k = 0;
    auto put = [&](uint32_t v) { rec[(k++) * S + q] = v; };
    auto put64 = [&](unsigned long long v) {
      put((uint32_t)v);
      put((uint32_t)(v >> 32));
    };
    put((uint32_t)mode);
    put(id);
    put(status);
    put(step);
    put((uint32_t)reject_run);
    put((uint32_t)b);
    put((uint32_t)n_max);
    put64((unsigned long long)i);
    put64((unsigned long long)__double_as_longlong(t));
    put64((unsigned long long)__double_as_longlong(T));
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      if constexpr (kRWords == 2) put64((unsigned long long)__double_as_longlong((double)th[j]));
      else put(__float_as_uint((float)th[j]));
    }
#pragma unroll
    for (int s2 = 0; s2 < NM; ++s2) put64((unsigned long long)x[s2]);
#pragma unroll
    for (int j = 0; j < MM; ++j) put64((unsigned long long)r[j]);
#pragma unroll
    for (int j = 0; j < MM; ++j)
      if (TT::g_owner(j) == j) put64((unsigned long long)__double_as_longlong(G[j]));
#pragma unroll
    for (int c = 0; c < 4; ++c) put64((unsigned long long)cnt[c]);
  }
  template <int S>
  __device__ __forceinline__ void load(const uint32_t* rec, int q) {
    int k = 0;
    auto get = [&]() { return rec[(k++) * S + q]; };
    auto get64 = [&]() {
      const unsigned long long lo = get();
      return lo | ((unsigned long long)get() << 32);
    };
    mode = (int)get();
    id = get();
    status = get();
    step = get();
    reject_run = (int)get();
    b = (int)get();
    n_max = (int)get();
    i = (long long)get64();
    t = __longlong_as_double((long long)get64());
    T = __longlong_as_double((long long)get64());
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      if constexpr (kRWords == 2) th[j] = (R)__longlong_as_double((long long)get64());
      else th[j] = (R)__uint_as_float(get());
    }
#pragma unroll
    for (int s2 = 0; s2 < NM; ++s2) x[s2] = (long long)get64();
#pragma unroll
    for (int j = 0; j < MM; ++j) r[j] = (long long)get64();
#pragma unroll
    for (int j = 0; j < MM; ++j)
      if (TT::g_owner(j) == j) G[j] = __longlong_as_double((long long)get64());
#pragma unroll
    for (int c = 0; c < 4; ++c) cnt[c] = (long long)get64();
  }

  __device__ __forceinline__ void begin_burst(int n) {
    mode = kSsa;
    b = 0;
    n_max = n;
  }

  __device__ __forceinline__ void end_burst() {
    step++;
    reject_run = 0;
    mode = kEval;
  }

  // Adds v to the integral of every reaction that holds one.
  template <class F>
  __device__ __forceinline__ void add_G(F v) {
#pragma unroll
    for (int j = 0; j < MM; ++j)
      if (TT::g_owner(j) == j) G[j] = G[j] + v(j);
  }

  // The net changes of reaction `pick` on the FP32 state copy / on the counts.
  __device__ __forceinline__ static void fire_f(const Model& md, int pick, float (&xf)[NM]) {
    if constexpr (Model::kCompiled) {  // one predicated update per nonzero entry
#pragma unroll
      for (int j = 0; j < MM; ++j) {
#pragma unroll
        for (int s = 0; s < NM; ++s)
          if (md.nu[j][s] != 0 && j == pick) xf[s] += md.nuf[j][s];
      }
    } else {
#pragma unroll
      for (int s = 0; s < NM; ++s) xf[s] += md.nuf[pick][s];
    }
  }
  __device__ __forceinline__ static void fire_x(const Model& md, int pick, long long (&x)[NM]) {
    if constexpr (Model::kCompiled) {
#pragma unroll
      for (int j = 0; j < MM; ++j) {
#pragma unroll
        for (int s = 0; s < NM; ++s)
          if (md.nu[j][s] != 0 && j == pick) x[s] += md.nu[j][s];
      }
    } else {
#pragma unroll
      for (int s = 0; s < NM; ++s) x[s] += md.nu[pick][s];
    }
  }
  // ... and of the firings counted in the nibbles of `fired`.
  __device__ __forceinline__ void fold_x(const Model& md, unsigned long long fired) {
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      const int c = (int)(fired >> (4 * j)) & 15;
#pragma unroll
      for (int s = 0; s < NM; ++s) x[s] += (long long)((int)md.nu[j][s] * c);
    }
  }

  // A slice's running sums: elapsed time (compensated FP32), G increments, the FP32 copy
  // of the state, and the firings, 4 bits per reaction.
  struct Slice {
    float el, elc;
    float Gs[MM], xf[NM];
    unsigned long long fired;
  };

  // kUnit firings without a branch: their random blocks, waiting times' logarithms and
  // uniforms first (independent of each other and of the state, so their chains overlap),
  // then the firings, each with its choices as selects.  Nothing is committed (false) when
  // one of them needs more: no reaction possible, the horizon or (kGrid) an observation
  // point reached, or a pick too near a prefix for FP32; the careful loop of ssa_slices
  // then does them one by one.  A lane spends most of its time here, and with few warps per
  // scheduler the chains' latency decides: one firing at a time, with its four branches,
  // took about 1,300 cycles on the immigration-death batch of 10,000 (one warp per
  // scheduler), most of it waiting for the ten rounds of Philox and the logarithm.
  __device__ __forceinline__ bool unit(const Model& md, const SimArgs& A, Slice& sl,
                                       float remf) {
    const uint32_t k0 = (uint32_t)A.seed, k1 = (uint32_t)(A.seed >> 32);
    R wait[kUnit];
    Words4 w[kUnit];
#pragma unroll
    for (int i = 0; i < kUnit; ++i) {
      w[i] = philox_block(k0, k1, id, step, (uint32_t)A.M + 2u, (uint32_t)b + (uint32_t)i);
      wait[i] = -P::log(P::u(w[i], 0));
    }
    bool ok = true;
    if constexpr (P::kRef) {
      double tn = t, Gn[MM];
      long long xn[NM];
#pragma unroll
      for (int j = 0; j < MM; ++j) Gn[j] = G[j];
#pragma unroll
      for (int s = 0; s < NM; ++s) xn[s] = x[s];
      unsigned long long fired = sl.fired;
#pragma unroll
      for (int i = 0; i < kUnit; ++i) {
        TT::eval_props(md, xn, th, g, a);
        a0 = reaction_sum<MM, R, P::kRef>(a);
        const double dt = wait[i] / a0;
        tn = tn + dt;
        ok = ok && P::positive(a0) && !past_horizon(tn, T);
#pragma unroll
        for (int j = 0; j < MM; ++j)
          if (TT::g_owner(j) == j) Gn[j] = Gn[j] + (double)g[j] * dt;
        bool clear;
        const int pick = TT::pick_near(a, w[i], clear);
        ok = ok && clear;
        if (!ok) return false;
        fire_x(md, pick, xn);
        fired += 1ULL << (4 * pick);
      }
      if (kGrid && kobs < A.K_obs && !(__ldg(A.t_obs + kobs) > tn)) return false;
      t = tn;
#pragma unroll
      for (int j = 0; j < MM; ++j) G[j] = Gn[j];
#pragma unroll
      for (int s = 0; s < NM; ++s) x[s] = xn[s];
      sl.fired = fired;
    } else {
      Slice n = sl;
      if (kGrid) n.fired = 0;
#pragma unroll
      for (int i = 0; i < kUnit; ++i) {
        float pre[MM];
        props_f(md, n.xf, pre);
        const float dt = __fdividef(wait[i], pre[MM - 1]);  // about 2 ulp
        ok = ok && pre[MM - 1] > 0.f && !((n.el - n.elc) + dt > remf);
#pragma unroll
        for (int j = 0; j < MM; ++j)
          if (TT::g_owner(j) == j) n.Gs[j] = fmaf((float)g[j], dt, n.Gs[j]);
        kahan_add(n.el, n.elc, dt);
        bool clear;
        int pick = TT::search_prefix(pre, w[i].w2, MM + 2, clear);
        ok = ok && clear;
        pick = pick < MM ? pick : 0;
        fire_f(md, pick, n.xf);
        n.fired += 1ULL << (4 * pick);
      }
      if (kGrid && kobs < A.K_obs &&
          !(__ldg(A.t_obs + kobs) > t + ((double)n.el - (double)n.elc)))
        return false;
      if (!ok) return false;
      if (kGrid) {
        fold_x(md, n.fired);
        n.fired += sl.fired;
      }
      sl = n;
    }
    b += kUnit;
    return true;
  }

  // Fast precision: g and a from the FP32 state copy, and the prefix sums of a, whose last
  // is the sequential total.
  __device__ __forceinline__ void props_f(const Model& md, const float (&xf)[NM],
                                          float (&pre)[MM]) {
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      g[j] = (R)TT::g_flt(md, j, xf);
      a[j] = P::mul(th[j], g[j]);
      pre[j] = j == 0 ? (float)a[0] : __fadd_rn(pre[j - 1], (float)a[j]);
    }
  }

  // Up to n_slices slices of kSsaPerRound firings of the SSA burst (Gillespie 1977 direct
  // method) at outer step `step`, firing index b.
  // Fast precision accumulates a slice's G increments in FP32 and its elapsed time in
  // compensated FP32 and folds them into the FP64 totals at the end of the slice: one FP64
  // addition per integral, its operand widened on the integer pipe (every driver folds at
  // the same firings).  The propensities read an FP32 copy of the state that the firings
  // update; x and r take the slice's firings at its end.
  // kUnits: firings in units, for the drivers whose few warps wait on the latency of a
  // firing; the pool driver, bound by instruction fetch and issue, is slower with the larger
  // loop (1,000,000 gene-expression trajectories: 375 ms against 300).
  template <bool kUnits>
  __device__ __forceinline__ void ssa_slices(const Model& md, const SimArgs& A, int n_slices) {
    const uint32_t k0 = (uint32_t)A.seed, k1 = (uint32_t)(A.seed >> 32);
    const int b_first = b;
    bool burst_over = false;
    for (;;) {
      const double rem = P::kRef ? 0.0 : T - t;
      const float remf = P::kRef ? 0.f : f32_of_f64(rem);
      Slice sl;
      sl.el = sl.elc = 0.f;
      sl.fired = 0;
#pragma unroll
      for (int j = 0; j < MM; ++j) sl.Gs[j] = 0.f;
      // an FP32 copy of the state, synchronized at every slice start
#pragma unroll
      for (int s = 0; s < NM; ++s) sl.xf[s] = P::kRef ? 0.f : f32_of_count(x[s]);
      bool to_horizon = false;
      const int b_end = b + kSsaPerRound < n_max ? b + kSsaPerRound : n_max;
#pragma unroll 1
      while (b < b_end && !burst_over) {
        if constexpr (kUnits && (Model::kCompiled || MM <= 2))
          if (b + kUnit <= b_end && unit(md, A, sl, remf)) continue;
        // one by one
        const int b_stop = b + kUnit < b_end ? b + kUnit : b_end;
#pragma unroll 1
        for (; b < b_stop; ++b) {
          if constexpr (P::kRef) {
            TT::eval_props(md, x, th, g, a);
            a0 = reaction_sum<MM, R, P::kRef>(a);
          } else {
            float pre[MM];
            props_f(md, sl.xf, pre);
            a0 = (R)pre[MM - 1];
          }
          if (P::zero(a0)) {
            to_horizon = burst_over = true;
            break;
          }
          const Words4 w = philox_block(k0, k1, id, step, (uint32_t)A.M + 2u, (uint32_t)b);
          if constexpr (P::kRef) {
            const R dt = -P::log(P::u(w, 0)) / a0;
            const double tn = t + (double)dt;
            if (past_horizon(tn, T)) {
              to_horizon = burst_over = true;
              break;
            }
            add_G([&](int j) { return (double)g[j] * (double)dt; });
            if (kGrid && A.K_obs > 0) record(A, tn, false);  // points before the firing: old state
            t = tn;
          } else {
            const float dt = __fdividef(-P::log(P::u(w, 0)), a0);
            if ((sl.el - sl.elc) + dt > remf) {
              to_horizon = burst_over = true;
              break;
            }
            // a slice holds at most kSsaPerRound firings: its G sums of that many positive
            // terms are within 8 FP32 roundings; the elapsed time is summed compensated
#pragma unroll
            for (int j = 0; j < MM; ++j)
              if (TT::g_owner(j) == j) sl.Gs[j] = fmaf((float)g[j], dt, sl.Gs[j]);
            kahan_add(sl.el, sl.elc, dt);
            if (kGrid && A.K_obs > 0) record(A, t + ((double)sl.el - (double)sl.elc), false);
          }
          const int pick = TT::pick_reaction(a, w, a0);
          if (P::kRef || kGrid) fire_x(md, pick, x);
          if (!P::kRef) fire_f(md, pick, sl.xf);
          sl.fired += 1ULL << (4 * pick);
          if (kGrid && A.K_obs > 0)  // a point at the firing time: new state
            record(A, P::kRef ? t : t + ((double)sl.el - (double)sl.elc), true);
        }
      }
      if (b >= n_max) burst_over = true;
#pragma unroll
      for (int j = 0; j < MM; ++j) r[j] += (int)(sl.fired >> (4 * j)) & 15;
      if (!P::kRef && !kGrid) fold_x(md, sl.fired);
      if constexpr (P::kRef) {
        if (to_horizon) {
          const double rm = T - t;
          add_G([&](int j) { return (double)g[j] * rm; });
          t = T;
        }
      } else {
        const double elapsed = f64_of_f32(sl.el) - f64_of_f32(sl.elc);
        add_G([&](int j) { return f64_of_f32(sl.Gs[j]); });
        if (to_horizon) {
          const double left = rem - elapsed > 0.0 ? rem - elapsed : 0.0;
          add_G([&](int j) { return (double)g[j] * left; });
          t = T;
        } else {
          t = t + elapsed;
        }
      }
      if (burst_over || --n_slices <= 0) break;
    }
    cnt[2] += b - b_first;
    if (burst_over) end_burst();
  }

  // One outer step: either a committed leap (stays in kEval), the start of an SSA burst,
  // or the end of the trajectory.
  __device__ __forceinline__ void eval_phase(const Model& md, const SimArgs& A) {
    const uint32_t k0 = (uint32_t)A.seed, k1 = (uint32_t)(A.seed >> 32);
    const uint32_t Mr = (uint32_t)A.M;  // stream numbering uses the real M
    if (!before_horizon(t, T)) {
      mode = kDone;
      return;
    }
    if ((long long)step >= A.max_steps) {
      status |= ML_ST_STEP_LIMIT;
      mode = kDone;
      return;
    }
    {
      bool big = false;
#pragma unroll
      for (int s = 0; s < NM; ++s) big = big || x[s] > kCountLimit;
#pragma unroll
      for (int j = 0; j < MM; ++j) big = big || r[j] > kCountLimit;
      if (big) {
        status |= ML_ST_OVERFLOW;
        mode = kDone;
        return;
      }
    }
    TT::eval_props(md, x, th, g, a);
    a0 = reaction_sum<MM, R, P::kRef>(a);
    if (P::zero(a0)) {
      const double rm = T - t;
      add_G([&](int j) { return (double)g[j] * rm; });
      t = T;
      mode = kDone;
      return;
    }
    int burst = 0;
    const R eps = P::eps(A);
    if (A.mode == ML_MODE_SSA_ONLY) {
      burst = A.n_ssa_ex;
    } else {
      // critical reactions: a_j > 0 and min over consumed species of floor(x_s/|nu_js|)
      // below n_c, i.e. some consumed species has x_s < n_c |nu_js| (no division needed)
      uint32_t nc = 0;
      R ac[MM];
#pragma unroll
      for (int j = 0; j < MM; ++j) {
        bool crit = false;
        if (P::positive(a[j])) {
#pragma unroll
          for (int s = 0; s < NM; ++s) {
            const int v = md.nu[j][s];
            if (v < 0 && x[s] < (long long)A.n_c * (long long)(-v)) crit = true;
          }
        }
        if (!crit) nc |= 1u << j;
        ac[j] = crit ? a[j] : R(0);
      }
      const R a0c = reaction_sum<MM, R, P::kRef>(ac);
      const R tau_ex = TT::tau_select(md, a, x, nc, eps);
      // partial equilibrium and the implicit step size
      bool implicit = false;
      R tau1 = tau_ex;
      if (A.mode == ML_MODE_ADAPTIVE && md.n_pairs > 0) {
        uint32_t pe = 0;
#pragma unroll
        for (int j = 0; j < MM; ++j) {
          const int k = md.partner[j];
          if (k >= 0 && ((nc >> j) & 1u) && ((nc >> k) & 1u)) {
            R ak = R(0);
#pragma unroll
            for (int kk = 0; kk < MM; ++kk)
              if (kk == k) ak = a[kk];
            const R lo = P::lt(a[j], ak) ? a[j] : ak;
            if (P::le(fabs(a[j] - ak), P::pe_delta(A) * lo)) pe |= (1u << j) | (1u << k);
          }
        }
        if (pe != 0) {
          const R tau_im = TT::tau_select(md, a, x, nc & ~pe, eps);
          if (P::lt(P::stiff_ratio(A) * tau_ex, tau_im)) {
            implicit = true;
            tau1 = tau_im;
          }
        }
      }
      // attempt loop: tau2, SSA switch, leap, negativity check
      for (;;) {
        if (reject_run >= A.max_reject) {
          status |= ML_ST_REJECT_LIMIT;
          burst = A.n_ssa_ex;
          break;
        }
        R tau2 = P::inf();
        if (P::positive(a0c)) {
          const Words4 w = philox_block(k0, k1, id, step, Mr, 0u);
          tau2 = -P::log(P::u(w, 0)) / a0c;
        }
        const R tmin = P::lt(tau1, tau2) ? tau1 : tau2;
        if (P::lt(tmin, P::ssa_factor(A) / a0)) {
          burst = implicit ? A.n_ssa_im : A.n_ssa_ex;
          break;
        }
        const double stop = kGrid ? stop_time(A) : T;
        const double rm = stop - t;
        R tau = tau1;
        if (P::lt(tau2, tau)) tau = tau2;
        bool at_horizon = false;
        const R rmr = P::of_f64(rm);
        if (P::le(rmr, tau)) {
          tau = rmr;
          at_horizon = true;
        }
        const bool crit_fire = P::le(tau2, tau1) && P::le(tau2, rmr);
        {
          bool over = false;
#pragma unroll
          for (int j = 0; j < MM; ++j)
            over = over || (((nc >> j) & 1u) && P::lt((R)kLeapLimit, P::mul(a[j], tau)));
          if (over) {
            status |= ML_ST_OVERFLOW;
            mode = kDone;
            return;
          }
        }
        long long K[MM];
#pragma unroll
        for (int j = 0; j < MM; ++j) K[j] = 0;
        if (crit_fire) {
          const Words4 w = philox_block(k0, k1, id, step, Mr + 1u, 0u);
          const int pick = TT::pick_reaction(ac, Words4{0u, 0u, w.w0, w.w1}, a0c);
#pragma unroll
          for (int j = 0; j < MM; ++j) K[j] = (j == pick) ? 1 : 0;
        }
        const bool implicit_step = implicit && P::lt(tau_ex, tau);
        // Poisson firings of the non-critical reactions (explicit counts, or the noise
        // term P_j of the implicit equation)
        // The small means by inversion, reaction by reaction; the large ones by a loop over
        // (reaction, PTRS trial) in which every lane is at a reaction of its own, so that the
        // trial's code runs as often as the busiest lane needs it, not once per reaction that
        // some lane of the warp draws by it.
        // The first random block of every reaction is generated before any is used: their
        // chains of ten dependent rounds (150 cycles each) overlap.
        uint32_t big = 0;
        R mus[MM];
        long long drawn[MM];
        Words4 first[MM];
#pragma unroll
        for (int j = 0; j < MM; ++j)
          if (Model::kCompiled || j < A.M)
            first[j] = philox_block(k0, k1, id, step, (uint32_t)j, 0u);
#pragma unroll
        for (int j = 0; j < MM; ++j) {
          mus[j] = P::mul(a[j], tau);
          if (((nc >> j) & 1u) && P::positive(mus[j])) {
            if (P::lt(mus[j], R(10)))
              K[j] = Model::kCompiled ? poisson_invert_at<P>(mus[j], P::u(first[j], 0))
                                      : poisson_invert_call<P>(mus[j], P::u(first[j], 0));
            else big |= 1u << j;
          }
        }
        const uint32_t by_trials = big;
        uint32_t trial = 0;
        while (big != 0) {
          const int j = __ffs((int)big) - 1;
          const R mu = mus[j];
          long long k = 0;
          bool done;
          if (!P::kRef && mu > R(4.0e6)) {
            const PoissonDraw d =
                poisson_ptrs<PrecWide>((double)mu, k0, k1, id, step, (uint32_t)j);
            k = d.k;
            status |= d.flags;
            done = true;
          } else {
            const Words4 w = trial == 0u ? first[j]
                                         : philox_block(k0, k1, id, step, (uint32_t)j, trial);
            done = ptrs_trial<P>(mu, w, k);
            if (++trial == (uint32_t)kPtrsMaxTrials && !done) {
              k = (long long)floor(mu + R(0.5));
              status |= ML_ST_PTRS_CAP;
              done = true;
            }
          }
          if (done) {
            drawn[j] = k;
            big &= big - 1u;
            trial = 0;
          }
        }
#pragma unroll
        for (int j = 0; j < MM; ++j)
          if ((by_trials >> j) & 1u) K[j] = drawn[j];
        if (implicit_step) {
          int rc;
          if constexpr (P::kRef && !Model::kCompiled) {
            rc = implicit_leap_rolled<NM, MM, Model, false>(
                md, x, K, th, a, nc, tau, A.newton_tol, A.newton_maxit, A.fd_h,
                A.jacobian == ML_JAC_ANALYTIC);
          } else if constexpr (P::kRef) {
            double y[NM];
            const double taud = (double)tau;
            rc = TT::implicit_solve(md, th, x, nc, K, a, taud, A.newton_tol, A.newton_maxit,
                                    A.fd_h, A.jacobian == ML_JAC_ANALYTIC, y);
            if (rc == 0) {
#pragma unroll
              for (int j = 0; j < MM; ++j) {
                if ((nc >> j) & 1u) {
                  const double ayj = (double)th[j] * TT::g_real(md, j, y);
                  const double v = (ayj * taud + f64_of_count(K[j])) - (double)a[j] * taud;
                  const double rv = round(v);
                  K[j] = !(rv < 0x1p62) ? kCountLimit : (rv > 0.0 ? (long long)rv : 0);
                }
              }
            }
          } else {
            ImplicitIo<NM, MM> io;
#pragma unroll
            for (int s = 0; s < NM; ++s) io.x[s] = x[s];
#pragma unroll
            for (int j = 0; j < MM; ++j) {
              io.K[j] = K[j];
              io.th[j] = (float)th[j];
            }
            rc = A.newton_fp32
                     ? implicit_leap_fp32<NM, MM>(md, io, nc, (float)tau, A.newton_tol,
                                                  A.newton_maxit)
                     : implicit_leap_wide<NM, MM>(md, io, nc, P::to_f64(tau), A.newton_tol,
                                                  A.newton_maxit, A.fd_h,
                                                  A.jacobian == ML_JAC_ANALYTIC);
#pragma unroll
            for (int j = 0; j < MM; ++j) K[j] = io.K[j];
          }
          if (rc != 0) {
            status |= ML_ST_NEWTON_FAIL;
            implicit = false;
            tau1 = tau_ex;
            step++;
            continue;
          }
        }
        if (implicit_step) {
          bool over = false;
#pragma unroll
          for (int j = 0; j < MM; ++j) over = over || (((nc >> j) & 1u) && K[j] > kLeapLimitInt);
          if (over) {
            status |= ML_ST_OVERFLOW;
            mode = kDone;
            return;
          }
        }
        long long xn[NM];
        bool negative = false;
#pragma unroll
        for (int s = 0; s < NM; ++s) {
          long long v = x[s];
#pragma unroll
          for (int j = 0; j < MM; ++j) v += (long long)md.nu[j][s] * K[j];
          xn[s] = v;
          if (v < 0) negative = true;
        }
        if (negative) {
          tau1 = tau1 * R(0.5);
          step++;
          reject_run++;
          cnt[3] += 1;
          continue;
        }
        const R half_r = tau * R(0.5);
#pragma unroll
        for (int j = 0; j < MM; ++j) {
          r[j] += K[j];
          if (TT::g_owner(j) == j) {  // fast precision: an FP32 increment
            const R gn = TT::g_int(md, j, xn);
            G[j] = G[j] + P::to_f64(half_r * (g[j] + gn));
          }
        }
#pragma unroll
        for (int s = 0; s < NM; ++s) x[s] = xn[s];
        t = at_horizon ? stop : t + P::to_f64(tau);
        if (kGrid && A.K_obs > 0) record(A, t, true);
        cnt[implicit_step ? 1 : 0] += 1;
        step++;
        reject_run = 0;
        break;
      }
    }
    if (burst > 0) begin_burst(burst);
  }
};

#ifndef ML_THREAD_MIN_BLOCKS
#define ML_THREAD_MIN_BLOCKS 1
#endif
#if ML_THREAD_MIN_BLOCKS == 2
// the occupancy build: at most 128 threads per CTA, about 168 registers, 3 CTAs per SM
#define ML_THREAD_BOUNDS __launch_bounds__(128, 3)
#else
#define ML_THREAD_BOUNDS __launch_bounds__(256, 1)
#endif

// Warp schedule: in every round a lane that needs a leap evaluation performs one, and a
// lane inside an SSA burst performs up to kSsaPerRound firings (about the cost of one
// evaluation), so lanes in different phases progress together instead of a whole burst
// holding the warp.  (Running only one phase per round, the evaluations once at least 4
// or 8 lanes need one, measured 2.6 and 1.8 times slower on the gene-expression batch.)
// The first trajectory of a lane (n_traj: none): from the queue, or in the plain form by
// position, per_warp of them to each warp.
__device__ __forceinline__ long long first_index(const SimArgs& args, bool on) {
  if (!on) return args.n_traj;
  if (args.queue) return queue_claim(args.queue, args.order, args.n_traj);
  const long long warp = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  return warp * args.per_warp + (threadIdx.x & 31);
}

// Round-based driver: plain form (queue null): thread i runs trajectory i.  Persistent
// form: lanes claim trajectory indices from the device queue (in the caller's order, if
// any) and refill as soon as their trajectory ends.
template <int NM, int MM, class P, class MDL>
__device__ __forceinline__ void run_rounds(const MDL& md, bool staged, const SimArgs& args) {
  using Lane = ThreadLane<NM, MM, P, false, MDL>;
  Lane L;
  L.mode = Lane::kIdle;
  const bool on = (int)(threadIdx.x & 31) < args.per_warp;
  const long long first = first_index(args, on);
  if (first < args.n_traj) L.start(md, args, first);
  for (;;) {
    if (L.mode == Lane::kDone) {
      L.finish(args, staged);
      if (args.queue) {
        const long long nxt = queue_claim(args.queue, args.order, args.n_traj);
        if (nxt < args.n_traj) L.start(md, args, nxt);
      }
    }
    if (!__any_sync(0xffffffffu, L.mode != Lane::kIdle)) break;
    if (L.mode == Lane::kEval) {
      L.eval_phase(md, args);
    } else if (L.mode == Lane::kSsa) {
      L.template ssa_slices<true>(md, args, 1);
    }
  }
}

// Pool driver: every warp keeps kPoolSlots trajectories (two per lane) in shared memory
// and in each round runs one phase for 32 of them: SSA slices while at least 32 (or more
// than the evaluations waiting) are inside a burst, else leap evaluations.  A lane loads
// the chosen trajectory's state, runs the phase and stores it back, so the lanes of a
// warp execute the same phase instead of taking turns between the evaluation and the SSA
// code (the round-based driver's lanes diverge there).  A finished trajectory is written
// out and its slot refilled from the work queue at once.  Persistent form only.

constexpr int kPoolSlices = 13;  // slices of a visit: a burst of 100 firings to its end

// Position of the (n+1)-th set bit of m (n < popcount(m)).
__device__ __forceinline__ int nth_set_bit(unsigned long long m, int n) {
  const uint32_t lo = (uint32_t)m, hi = (uint32_t)(m >> 32);
  const int clo = __popc(lo);
  uint32_t v = n < clo ? lo : hi;
  int k = n < clo ? n : n - clo;
  for (; k > 0; --k) v &= v - 1u;
  return (n < clo ? 0 : 32) + __ffs((int)v) - 1;
}

template <int NM, int MM, class P, class MDL>
__device__ __forceinline__ void run_pool(const MDL& md, bool staged, const SimArgs& args,
                                         uint32_t* pool_words) {
  using Lane = ThreadLane<NM, MM, P, false, MDL>;
  const int lane = threadIdx.x & 31;
  uint32_t* rec = pool_words + (size_t)(threadIdx.x >> 5) * Lane::kWords * kPoolSlots;
#pragma unroll 1
  for (int h = lane; h < kPoolSlots; h += 32) {
    Lane L;
    L.mode = Lane::kIdle;
    const long long idx =
        h < args.per_warp ? queue_claim(args.queue, args.order, args.n_traj) : args.n_traj;
    if (idx < args.n_traj) L.start(md, args, idx);
    L.template save<kPoolSlots>(rec, h);
  }
  __syncwarp();
  // the search for ready slots starts at a rotating position, so that no slot waits
  // while others are served round after round
  int rot = 0;
  for (;;) {
    const uint32_t m_lo = rec[lane], m_hi = rec[32 + lane];  // mode words
    const unsigned long long ms =
        (unsigned long long)__ballot_sync(0xffffffffu, m_lo == (uint32_t)Lane::kSsa) |
        ((unsigned long long)__ballot_sync(0xffffffffu, m_hi == (uint32_t)Lane::kSsa) << 32);
    const unsigned long long me =
        (unsigned long long)__ballot_sync(0xffffffffu, m_lo == (uint32_t)Lane::kEval) |
        ((unsigned long long)__ballot_sync(0xffffffffu, m_hi == (uint32_t)Lane::kEval) << 32);
    const int ns = __popcll(ms), ne = __popcll(me);
    if (ns + ne == 0) break;
    const bool ssa = ns >= 32 || (ne < 32 && ns >= ne);
    const int n_run = ssa ? ns : ne;
    const unsigned long long m = ssa ? ms : me;
    const int r0 = rot;
    rot = (rot + 29) & (kPoolSlots - 1);
    const unsigned long long mr = r0 ? (m >> r0) | (m << (kPoolSlots - r0)) : m;
    if (lane < n_run) {
      const int q = (nth_set_bit(mr, lane) + r0) & (kPoolSlots - 1);
      Lane L;
      L.template load<kPoolSlots>(rec, q);
      if (ssa) L.template ssa_slices<false>(md, args, kPoolSlices);
      else L.eval_phase(md, args);
      if (L.mode == Lane::kDone) {
        L.finish(args, staged);
        const long long nxt = queue_claim(args.queue, args.order, args.n_traj);
        if (nxt < args.n_traj) L.start(md, args, nxt);
      }
      L.template save<kPoolSlots>(rec, q);
    }
    __syncwarp();
  }
}

// Sequential per-lane driver over the same lane state machine: each thread runs its
// trajectory to the end before claiming the next one.  It has less scheduling overhead
// and suits leap-dominated workloads; the autotuner picks between the drivers.  Its kGrid
// build serves every thread-shape call with time-grid output (the drivers give identical
// results).
template <int NM, int MM, class P, bool kGrid, class MDL>
__device__ __forceinline__ void run_sequential(const MDL& md, bool staged, const SimArgs& args) {
  using Lane = ThreadLane<NM, MM, P, kGrid, MDL>;
  Lane L;
  const bool on = (int)(threadIdx.x & 31) < args.per_warp;
  long long i = first_index(args, on);
  while (i < args.n_traj) {
    L.start(md, args, i);
    while (L.mode != Lane::kDone) {
      if (L.mode == Lane::kEval) L.eval_phase(md, args);
      else L.template ssa_slices<true>(md, args, 1);
    }
    L.finish(args, staged);
    if (!args.queue) break;
    i = queue_claim(args.queue, args.order, args.n_traj);
  }
}

// Kernels over the run-time tables: stage the model once per CTA into shared memory (one
// bulk copy), then run a driver.
template <int NM, int MM, class P>
__global__ void ML_THREAD_BOUNDS k_thread(const ThreadModel<NM, MM>* __restrict__ gmd,
                                          const SimArgs args) {
  __shared__ ThreadModel<NM, MM> smd;
  __shared__ uint64_t mbar;
  const bool staged = stage_model_bulk(&smd, gmd, (uint32_t)thread_model_bytes<NM, MM>(), &mbar,
                                       args.stage_polls);
  run_rounds<NM, MM, P>(smd, staged, args);
}

template <int NM, int MM, class P>
__global__ void ML_THREAD_BOUNDS k_thread_pool(const ThreadModel<NM, MM>* __restrict__ gmd,
                                               const SimArgs args) {
  __shared__ ThreadModel<NM, MM> smd;
  __shared__ uint64_t mbar;
  extern __shared__ uint32_t pool_words[];
  const bool staged = stage_model_bulk(&smd, gmd, (uint32_t)thread_model_bytes<NM, MM>(), &mbar,
                                       args.stage_polls);
  run_pool<NM, MM, P>(smd, staged, args, pool_words);
}

template <int NM, int MM, class P, bool kGrid = false>
__global__ void ML_THREAD_BOUNDS k_thread_seq(const ThreadModel<NM, MM>* __restrict__ gmd,
                                              const SimArgs args) {
  __shared__ ThreadModel<NM, MM> smd;
  __shared__ uint64_t mbar;
  const bool staged = stage_model_bulk(&smd, gmd, (uint32_t)thread_model_bytes<NM, MM>(), &mbar,
                                       args.stage_polls);
  run_sequential<NM, MM, P, kGrid>(smd, staged, args);
}

}  // namespace mlk
