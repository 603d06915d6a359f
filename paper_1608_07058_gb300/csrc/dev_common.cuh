// Device building blocks: counter-based random numbers, the FP64 elementary functions
// of the reference-precision path, and bulk staging of model tables into shared memory.
#pragma once
#ifndef __CUDACC_RTC__  // runtime compilation (model-specialized kernels) brings its own types
#include <cstdint>

#include <cuda_runtime.h>
#endif

namespace mlk {

// ---------------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC11): ten rounds, each two 32x32->64
// products of counter words 0 and 2 with fixed multipliers, xored into the other words
// with the key, the key bumped by two Weyl constants between rounds.
// Counter = (trajectory id, step, stream, block), key = (seed lo, seed hi).
// ---------------------------------------------------------------------------------
struct Words4 {
  uint32_t w0, w1, w2, w3;
};

__device__ __forceinline__ Words4 philox_block(uint32_t k0, uint32_t k1, uint32_t id,
                                               uint32_t step, uint32_t stream,
                                               uint32_t block) {
  uint32_t c0 = id, c1 = step, c2 = stream, c3 = block;
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    if (round > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    // one wide multiplication each (both halves of the product in one instruction)
    const unsigned long long a = (unsigned long long)0xD2511F53u * c0;
    const unsigned long long b = (unsigned long long)0xCD9E8D57u * c2;
    c0 = (uint32_t)(b >> 32) ^ c1 ^ k0;
    c1 = (uint32_t)b;
    c2 = (uint32_t)(a >> 32) ^ c3 ^ k1;
    c3 = (uint32_t)a;
  }
  return Words4{c0, c1, c2, c3};
}

// ---------------------------------------------------------------------------------
// Exact conversions and comparisons on the integer pipe.  The FP64 unit serves one warp
// instruction per scheduler in 64 cycles, whatever its active lanes and however many
// independent ones a warp has, and every conversion to or from a 64-bit type runs on it
// too (int64 -> float: 64 cycles, 100 of latency; int32 -> float: 4 and 15).  The same
// values by integer operations take 3 to 12 issue slots.  Results are those of the
// conversion instructions (round to nearest even); what is out of a fast form's range takes
// the instruction, as volatile assembly so that it is not executed speculatively.
// ---------------------------------------------------------------------------------

// float(v), v >= 0: below 2^32 by the 32-bit conversion; above, the top 32 bits with the
// rest folded into the last one (sticky) round the same way, and the scaling is exact.
__device__ __forceinline__ float f32_of_count(long long v) {
  const uint32_t hi = (uint32_t)((unsigned long long)v >> 32), lo = (uint32_t)v;
  if (hi == 0u) return (float)lo;
  const int s = __clz((int)hi);  // >= 1: v >= 0
  const uint32_t top = __funnelshift_l(lo, hi, s) | ((lo << s) != 0u ? 1u : 0u);
  return (float)top * __int_as_float((159 - s) << 23);
}

// double(v), v >= 0: below 2^53 by shifting the leading one to bit 52.
__device__ __forceinline__ double f64_of_count(long long v) {
  const uint32_t hi = (uint32_t)((unsigned long long)v >> 32), lo = (uint32_t)v;
  if (hi != 0u) {
    if (hi < 0x00200000u) {
      const int s = __clz((int)hi) - 11;
      return __longlong_as_double((v << s) + ((long long)(1074 - s) << 52));
    }
    double d;
    asm volatile("cvt.rn.f64.s64 %0, %1;" : "=d"(d) : "l"(v));
    return d;
  }
  const int s = __clz((int)lo);
  const uint32_t m = lo << (s & 31);
  const uint32_t h = lo ? (m >> 11) + ((uint32_t)(1053 - s) << 20) : 0u;
  return __hiloint2double((int)h, (int)(lo ? m << 21 : 0u));
}

// double(f): normal numbers and zero.
__device__ __forceinline__ double f64_of_f32(float f) {
  const uint32_t u = __float_as_uint(f), a = u & 0x7fffffffu;
  if (a - 0x00800000u < 0x7f000000u)
    return __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(u << 29));
  if (a == 0u) return __hiloint2double((int)u, 0);
  double d;
  asm volatile("cvt.f64.f32 %0, %1;" : "=d"(d) : "f"(f));
  return d;
}

// float(d), round to nearest even: results in the normal range and zero.
__device__ __forceinline__ float f32_of_f64(double d) {
  const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
  const uint32_t a = hi & 0x7fffffffu;
  if (a - 0x38100000u < 0x0fd00000u) {  // exponents -126 .. 126: rounding cannot overflow
    const uint32_t m = ((a - 0x38000000u) << 3) | (lo >> 29), rest = lo & 0x1fffffffu;
    const uint32_t up = (rest + (m & 1u)) > 0x10000000u ? 1u : 0u;
    return __uint_as_float((hi & 0x80000000u) | (m + up));
  }
  if ((a | lo) == 0u) return __uint_as_float(hi);
  float f;
  asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(f) : "d"(d));
  return f;
}

// double(k), 32-bit, exact.
__device__ __forceinline__ double f64_of_i32(int k) {
  const uint32_t a = (uint32_t)(k < 0 ? -k : k);
  const int s = __clz((int)a);
  const uint32_t m = a << (s & 31);
  const uint32_t h = ((uint32_t)k & 0x80000000u) | ((m >> 11) + ((uint32_t)(1053 - s) << 20));
  return __hiloint2double((int)(a ? h : 0u), (int)(m << 21));
}

// t < T for a time t in [0, +inf] (not -0) or NaN and a horizon T that is not NaN (it may be
// negative): as integers, false for a NaN of either sign (0 inf gives one whose sign is set,
// which lies below every number; the other lies above).
__device__ __forceinline__ bool before_horizon(double t, double T) {
  const long long bt = __double_as_longlong(t);
  return bt >= 0 && bt < __double_as_longlong(T);
}

// tn > T for a time tn in [0, +inf] (not -0) or NaN of either sign and a horizon T > 0: false
// for a NaN (a set sign makes it negative).
__device__ __forceinline__ bool past_horizon(double tn, double T) {
  const long long bt = __double_as_longlong(tn);
  return bt > __double_as_longlong(T) && bt <= 0x7ff0000000000000LL;
}

// a < b for operands that are each in [0, +inf] (not -0) or NaN of either sign.  Unsigned: the
// mask may be compiled to an FP64 absolute value, which leaves a NaN's sign.
__device__ __forceinline__ bool f64_lt_pos(double a, double b) {
  const unsigned long long m = 0x7fffffffffffffffULL, inf = 0x7ff0000000000000ULL;
  const unsigned long long ub = (unsigned long long)__double_as_longlong(b) & m;
  return ((unsigned long long)__double_as_longlong(a) & m) < ub && ub <= inf;
}

// a <= b for operands that are each in [0, +inf] (not -0) or NaN.
__device__ __forceinline__ bool f64_le_pos(double a, double b) {
  const unsigned long long m = 0x7fffffffffffffffULL, inf = 0x7ff0000000000000ULL;
  const unsigned long long ub = (unsigned long long)__double_as_longlong(b) & m;
  return ((unsigned long long)__double_as_longlong(a) & m) <= ub && ub <= inf;
}

// abs(a) > abs(b) (false when a is NaN; b is not NaN).
__device__ __forceinline__ bool f64_abs_gt(double a, double b) {
  const unsigned long long m = 0x7fffffffffffffffULL, inf = 0x7ff0000000000000ULL;
  const unsigned long long ua = (unsigned long long)__double_as_longlong(a) & m;
  const unsigned long long ub = (unsigned long long)__double_as_longlong(b) & m;
  return ua > ub && ua <= inf;
}

// FP64 uniform in (0,1) from two words: 52 bits n, u = (n + 1/2) 2^-52 (exact): the odd
// integer 2n + 1 shifted so that its leading one is the implicit bit.
__device__ __forceinline__ double u01_f64(uint32_t hi, uint32_t lo) {
  const unsigned long long v =
      ((((unsigned long long)(hi >> 6) << 26) | (unsigned long long)(lo >> 6)) << 1) | 1ULL;
  const int s = __clzll((long long)v);  // >= 11
  return __longlong_as_double(
      (long long)((v << (s - 11)) + ((unsigned long long)(1032 - s) << 52)));
}

// FP32 uniform in (0,1) from one word: 23 bits n, u = (n + 1/2) 2^-23 (exact).
__device__ __forceinline__ float u01_f32(uint32_t w) {
  return ((float)(w >> 9) + 0.5f) * 0x1p-23f;
}

// ---------------------------------------------------------------------------------
// FP64 elementary functions of the reference path (Cody & Waite 1980 style): additive
// reduction by k ln2 with ln2 split in a 32-bit head and a tail, then a polynomial.
// Only +,-,*,/ (the reference translation unit is compiled without FMA contraction),
// so the results are fixed by the operation order below.
// ---------------------------------------------------------------------------------
namespace refmath {
constexpr double kLn2Head = 0x1.62e42fee00000p-1;   // 32 leading bits of ln 2
constexpr double kLn2Tail = 0x1.a39ef35793c76p-33;  // ln 2 - kLn2Head
constexpr double kInvLn2 = 0x1.71547652b82fep+0;
constexpr unsigned long long kSqrt2Frac = 0x6a09e667f3bcdULL;  // fraction bits of sqrt 2
constexpr double kHalfLog2Pi = 0x1.d67f1c864beb5p-1;

// exp(x) on [-708, 709]: x = k ln2 + r, Taylor series of e^r to r^13 by Horner.
__device__ __forceinline__ double exp_ref(double x) {
  // the range by the high word: |x| below 708 needs no further test
  if ((uint32_t)(__double2hiint(x) & 0x7fffffff) >= 0x40862000u) {
    if (x != x) return x;
    if (x < -708.0) return 0.0;
    if (x > 709.0) return __longlong_as_double(0x7ff0000000000000LL);
  }
  const double kx = x * kInvLn2 + 0.5;
  // floor and its integer, by integer operations (|kx| < 1024)
  const uint32_t kh = (uint32_t)__double2hiint(kx), kl = (uint32_t)__double2loint(kx);
  const int ke = (int)((kh >> 20) & 0x7ffu) - 1023;
  const uint32_t km = (kh & 0xfffffu) | 0x100000u;
  int k = ke < 0 ? 0 : (int)(km >> (20 - ke));
  const bool frac = ke < 0 ? ((kh & 0x7fffffffu) | kl) != 0u
                           : ((km & ((1u << (20 - ke)) - 1u)) | kl) != 0u;
  if (kh >> 31) k = -k - (frac ? 1 : 0);
  const double kd = f64_of_i32(k);
  const double r = (x - kd * kLn2Head) - kd * kLn2Tail;
  double p = 1.0 / 6227020800.0;
  p = p * r + 1.0 / 479001600.0;
  p = p * r + 1.0 / 39916800.0;
  p = p * r + 1.0 / 3628800.0;
  p = p * r + 1.0 / 362880.0;
  p = p * r + 1.0 / 40320.0;
  p = p * r + 1.0 / 5040.0;
  p = p * r + 1.0 / 720.0;
  p = p * r + 1.0 / 120.0;
  p = p * r + 1.0 / 24.0;
  p = p * r + 1.0 / 6.0;
  p = p * r + 0.5;
  p = p * r + 1.0;
  p = p * r + 1.0;
  return p * __hiloint2double((k + 1023) << 20, 0);
}

// log(x) for positive normal x: x = 2^e m, m in [sqrt(1/2), sqrt(2)); with f = m - 1 and
// s = f/(2+f), log m = 2 atanh s = 2s (1 + z/3 + ... + z^11/23), z = s^2.
__device__ __forceinline__ double log_ref(double x) {
  const long long sb = __double_as_longlong(x);
  if (sb <= 0LL || sb >= 0x7ff0000000000000LL) {  // zero, negative, infinity, NaN
    if (x != x || x < 0.0) return __longlong_as_double(0x7ff8000000000000LL);
    if (x == 0.0) return __longlong_as_double((long long)0xfff0000000000000ULL);
    return x;
  }
  // mantissa in [1, 2) above sqrt 2 is halved: the comparison and the halving on its bits
  const unsigned long long bits = (unsigned long long)sb, frac = bits & 0x000fffffffffffffULL;
  const bool above = frac > kSqrt2Frac;
  const int e = (int)(bits >> 52) - (above ? 1022 : 1023);
  const double m = __longlong_as_double(
      (long long)(frac | (above ? 0x3fe0000000000000ULL : 0x3ff0000000000000ULL)));
  const double f = m - 1.0;
  const double s = f / (2.0 + f);
  const double z = s * s;
  double q = 1.0 / 23.0;
  q = q * z + 1.0 / 21.0;
  q = q * z + 1.0 / 19.0;
  q = q * z + 1.0 / 17.0;
  q = q * z + 1.0 / 15.0;
  q = q * z + 1.0 / 13.0;
  q = q * z + 1.0 / 11.0;
  q = q * z + 1.0 / 9.0;
  q = q * z + 1.0 / 7.0;
  q = q * z + 1.0 / 5.0;
  q = q * z + 1.0 / 3.0;
  const double two_s = s + s;
  const double logm = two_s + (two_s * z) * q;
  const double ed = f64_of_i32(e);
  return ed * kLn2Head + (ed * kLn2Tail + logm);
}

// log k!: exact product then log below 16; Stirling series of log Gamma(k+1) from 16.
__device__ __forceinline__ double log_factorial_ref(long long k) {
  if (k < 2) return 0.0;
  if (k < 16) {
    double f = 1.0;
    for (long long i = 2; i <= k; ++i) f = f * (double)i;
    return log_ref(f);
  }
  const double z = (double)k + 1.0;
  const double w = 1.0 / z;
  const double w2 = w * w;
  double ser = 1.0 / 1188.0;
  ser = ser * w2 - 1.0 / 1680.0;
  ser = ser * w2 + 1.0 / 1260.0;
  ser = ser * w2 - 1.0 / 360.0;
  ser = ser * w2 + 1.0 / 12.0;
  ser = ser * w;
  return (((z - 0.5) * log_ref(z) - z) + kHalfLog2Pi) + ser;
}
}  // namespace refmath

// ---------------------------------------------------------------------------------
// Persistent form: the next trajectory to run.  The k-th claim on the work queue is
// trajectory order[k] when the caller gave an order (meant to be a permutation of
// 0..n-1, longest first), else trajectory k.  Entries outside [0, n) are passed over, so a
// malformed order cannot index out of bounds (trajectories it leaves out are not run).
// Returns n_traj when the queue is exhausted.
// ---------------------------------------------------------------------------------
__device__ __forceinline__ long long queue_claim(unsigned long long* queue, const int64_t* order,
                                                 long long n_traj) {
  for (;;) {
    const long long k = (long long)atomicAdd(queue, 1ULL);
    if (k >= n_traj) return n_traj;
    if (!order) return k;
    const long long i = __ldg(order + k);
    if (i >= 0 && i < n_traj) return i;
  }
}

// ---------------------------------------------------------------------------------
// Model staging: one bulk asynchronous copy (TMA engine, cp.async.bulk) of the model
// tables from global to shared memory, completed on an mbarrier.  The wait is bounded
// (poll_limit polls per thread); if it runs out the CTA waits again, bounded, for its copy
// in flight, then copies the tables with plain loads and reports it.
// bytes must be a multiple of 16 and both addresses 16-byte aligned.
// ---------------------------------------------------------------------------------
__device__ __forceinline__ bool stage_model_bulk(void* smem_dst, const void* gmem_src,
                                                 uint32_t bytes, uint64_t* mbar,
                                                 int poll_limit) {
  const uint32_t bar = (uint32_t)__cvta_generic_to_shared(mbar);
  const uint32_t dst = (uint32_t)__cvta_generic_to_shared(smem_dst);
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile(
        "mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
        : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
        "[%3];" ::"r"(dst),
        "l"(gmem_src), "r"(bytes), "r"(bar)
        : "memory");
  }
  // every thread waits on phase 0, at most poll_limit polls
  uint32_t done = 0;
  for (int it = 0; it < poll_limit && !done; ++it) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar)
        : "memory");
  }
  const int ok = __syncthreads_and((int)done);
  if (!ok) {
    // The copy may still be in flight: wait again (bounded) before overwriting.
    for (int it = 0; it < (1 << 22) && !done; ++it) {
      asm volatile(
          "{\n\t.reg .pred p;\n\t"
          "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(done)
          : "r"(bar)
          : "memory");
    }
    __syncthreads();
    const uint4* src = reinterpret_cast<const uint4*>(gmem_src);
    uint4* d = reinterpret_cast<uint4*>(smem_dst);
    for (uint32_t k = threadIdx.x; k < bytes / 16; k += blockDim.x) d[k] = src[k];
    __syncthreads();
  }
  return ok != 0;
}

}  // namespace mlk
