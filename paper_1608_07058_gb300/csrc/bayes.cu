// The Bayesian step after a simulation (paper Section 1): per-trajectory draws from the
// conjugate posterior Gamma(alpha_j + r_j, beta_j + G_j) of every rate constant, and
// systematic resampling of particles from log-weights.  Compiled without FMA contraction:
// the FP64 arithmetic follows a fixed operation order and reproduces an independent
// implementation of the same definitions bit for bit.
#include <cstdint>

#include <cuda_runtime.h>

#include "dev_common.cuh"
#include "matleap.h"
#include "ml_internal.h"

namespace mlk {
namespace {

constexpr int kGammaMaxTrials = 64;

// Gamma(shape, rate) by Marsaglia & Tsang (2000): d = a - 1/3, c = 1/sqrt(9d); normal z by
// the Marsaglia polar method; v = (1 + c z)^3; accept iff log u < z^2/2 + d - d v + d log v;
// shape < 1 draws Gamma(shape + 1) and multiplies by U^(1/shape).  Counter (id, 0x80000000 +
// stream, 0, block): block 2t the polar pair of trial t, block 2t+1 the acceptance uniform
// (words 0, 1) and the boost uniform (words 2, 3).
//
// The draw is bound by the FP64 unit (64 cycles per warp instruction, whatever its active
// lanes), so what does not set a bit of the result stays off it: the polar pairs are exact
// integers, s < 1 and the acceptance are decided in FP32 with a margin and in FP64 only when
// FP32 cannot tell, and a lane looks for its next polar pair before the warp enters the FP64
// part (about a fifth of the pairs fall outside the unit circle).  6,000,000 draws: 7.0 ms
// with three FP64 logarithms in every trial of every lane.

// v = 2u - 1 for the uniform of two words, exact: an odd integer times 2^-52.
struct Signed52 {
  long long m;  // v = m 2^-52
  __device__ float f32() const {
    const float a = f32_of_count(m < 0 ? -m : m) * 0x1p-52f;
    return m < 0 ? -a : a;
  }
  __device__ double f64() const {
    const long long a = m < 0 ? -m : m;  // below 2^52, odd
    const int s = __clzll(a) - 11;
    const long long b = (a << s) + ((long long)(1022 - s) << 52);
    return __longlong_as_double(m < 0 ? (long long)(b | (1LL << 63)) : b);
  }
};
__device__ __forceinline__ Signed52 signed52(uint32_t hi, uint32_t lo) {
  return Signed52{((((long long)(hi >> 6) << 26) | (long long)(lo >> 6)) << 1) + 1 - (1LL << 52)};
}

// log u < z^2/2 + d - d v + d log v with v = (1 + y)^3, y = c z, d c^2 = 1/9, estimated in FP32:
// 1 accept, -1 reject, 0 too close.  The right side is 3 d (log1p(y) - y + y^2/2 - y^3/3) =
// 3 d (-y^4/4 + y^5/5 - ...): the large terms cancel before they are formed.  For |y| < 1/4
// the series to y^11 (relative error below 1e-5); else the logarithm, where d <= 16 z^2 / 9 <
// 140 (|z| < 8.7 from 52-bit uniforms) keeps its FP32 error 3 d 4e-7 below 2e-4; next to
// y = -1, where the rounding of y counts for more, it does not tell.  The FP64 test adds terms
// of size d, so it is itself off by up to about 4 d 2^-53: below the margin by a factor of 30
// up to d = 2^36; from there on (and for NaN) it does not tell either.
__device__ __forceinline__ int gamma_estimate(float u, float y, float d) {
  const float y2 = y * y;
  float t;
  if (y < -0.999f || !(d < 0x1p36f)) return 0;
  if (fabsf(y) < 0.25f) {
    float q = 1.f / 11.f;
    q = q * y - 0.1f;
    q = q * y + (1.f / 9.f);
    q = q * y - 0.125f;
    q = q * y + (1.f / 7.f);
    q = q * y - (1.f / 6.f);
    q = q * y + 0.2f;
    q = q * y - 0.25f;
    t = 3.f * d * (q * y2 * y2);
  } else {
    t = 3.f * d * (log1pf(y) - y + 0.5f * y2 - y2 * y * (1.f / 3.f));
  }
  const float gap = t - __logf(u);
  const float margin = 1.0e-3f + 1.0e-4f * fabsf(t);
  return gap > margin ? 1 : gap < -margin ? -1 : 0;
}

__device__ double gamma_draw(double shape, double rate, uint32_t k0, uint32_t k1, uint32_t id,
                             uint32_t stream, uint32_t& flags) {
  if (!(shape > 0.0) || !(rate > 0.0)) return __longlong_as_double(0x7ff8000000000000LL);
  const bool boost = shape < 1.0;
  const double a = boost ? shape + 1.0 : shape;
  const double d = a - 1.0 / 3.0;
  const double c = 1.0 / sqrt(9.0 * d);
  const uint32_t cstep = 0x80000000u + stream;
  uint32_t t = 0;
  for (;;) {
    // the next polar pair inside the unit circle
    Signed52 m1{0}, m2{0};
    double v1 = 0.0, s = 0.0;
    bool found = false;
    for (; t < (uint32_t)kGammaMaxTrials && !found; ++t) {
      const Words4 w = philox_block(k0, k1, id, cstep, 0u, 2u * t);
      m1 = signed52(w.w0, w.w1);
      m2 = signed52(w.w2, w.w3);
      const float f1 = m1.f32(), f2 = m2.f32();
      const float sf = f1 * f1 + f2 * f2;
      if (fabsf(sf - 1.f) < 1.0e-5f) {
        const double e1 = m1.f64(), e2 = m2.f64();
        found = e1 * e1 + e2 * e2 < 1.0;
      } else {
        found = sf < 1.f;
      }
    }
    if (!found) break;
    // trial t - 1
    v1 = m1.f64();
    const double v2 = m2.f64();
    s = v1 * v1 + v2 * v2;
    const double z = v1 * sqrt((-2.0 * refmath::log_ref(s)) / s);
    const double y = c * z;
    const double base = 1.0 + y;
    if (__double2hiint(base) < 0 || base == 0.0) continue;
    const double v = (base * base) * base;
    const Words4 w2 = philox_block(k0, k1, id, cstep, 0u, 2u * (t - 1u) + 1u);
    const double u = u01_f64(w2.w0, w2.w1);
    const int est = gamma_estimate(f32_of_f64(u), f32_of_f64(y), f32_of_f64(d));
    const bool ok = est != 0 ? est > 0
                             : refmath::log_ref(u) < ((0.5 * (z * z) + d) - d * v) +
                                                         d * refmath::log_ref(v);
    if (ok) {
      double x = d * v;
      if (boost) {
        const double ub = u01_f64(w2.w2, w2.w3);
        x = x * refmath::exp_ref(refmath::log_ref(ub) / shape);
      }
      return x / rate;
    }
  }
  flags |= 1u;
  return shape / rate;
}

// One thread per (trajectory, reaction).
__global__ void k_posterior(int64_t n, int32_t M, const double* __restrict__ alpha,
                            int32_t alpha_per, const double* __restrict__ beta, int32_t beta_per,
                            const int64_t* __restrict__ r, const double* __restrict__ G,
                            uint64_t seed, uint64_t id_base, double* __restrict__ theta,
                            uint32_t* __restrict__ status) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * (long long)M) return;
  const long long i = e / M;
  const int j = (int)(e - i * M);
  const double al = alpha_per ? alpha[e] : alpha[j];
  const double be = beta_per ? beta[e] : beta[j];
  uint32_t flags = 0;
  const long long re = r[e];
  const double rd = re >= 0 ? f64_of_count(re) : (double)re;
  theta[e] = gamma_draw(al + rd, be + G[e], (uint32_t)seed, (uint32_t)(seed >> 32),
                        (uint32_t)(id_base + (unsigned long long)i), (uint32_t)j, flags);
  if (status && flags) atomicOr(status + i, flags);
}

// ---- systematic resampling ----------------------------------------------------------
constexpr int kScanBlock = 1024;

__device__ __forceinline__ double neg_inf() {
  return __longlong_as_double((long long)0xfff0000000000000ULL);
}
__device__ __forceinline__ double warp_max_f64(double m) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    const double o = __shfl_xor_sync(0xffffffffu, m, d);
    m = o > m ? o : m;
  }
  return m;
}

// Maximum of f(i) over i < n by the CTA (NaN never compares greater); all threads return it.
template <class F>
__device__ __forceinline__ double block_max(int64_t first, int64_t n, int64_t step, F f,
                                            double* sm) {
  double m = neg_inf();
#pragma unroll 8
  for (long long i = first; i < n; i += step) {
    const double v = f(i);
    if (v > m) m = v;
  }
  m = warp_max_f64(m);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  m = warp_max_f64((threadIdx.x & 31) < (blockDim.x >> 5) ? sm[threadIdx.x & 31] : neg_inf());
  __syncthreads();
  return m;
}

// Per-block maxima of the log-weights.
__global__ void k_block_max(int64_t n, const double* __restrict__ logw, double* __restrict__ out) {
  __shared__ double sm[32];
  const double m = block_max((long long)blockIdx.x * blockDim.x + threadIdx.x, n,
                             (long long)gridDim.x * blockDim.x,
                             [&](long long i) { return logw[i]; }, sm);
  if (threadIdx.x == 0) out[blockIdx.x] = m;
}

// Inclusive prefix over the CTA of kScanBlock threads (exact integers), by warp shuffles.
__device__ __forceinline__ uint64_t block_scan(uint64_t v, uint64_t* sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += o;
  }
  if (lane == 31) sm[warp] = v;
  __syncthreads();
  uint64_t t = sm[lane];  // kScanBlock / 32 = 32 warps
  uint64_t e = t;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t o = __shfl_up_sync(0xffffffffu, e, d);
    if (lane >= d) e += o;
  }
  const uint64_t before = __shfl_sync(0xffffffffu, e - t, warp);
  __syncthreads();
  return v + before;
}

// Quantized weights q_i = floor(exp(logw_i - max) 2^40) (0 for NaN) and their inclusive
// prefix within each block of kScanBlock; block totals to bsum.  The maximum is that of the
// nmax block maxima, taken again by every CTA.
__global__ void k_quantize_scan(int64_t n, const double* __restrict__ logw,
                                const double* __restrict__ maxima, int nmax,
                                uint64_t* __restrict__ incl, uint64_t* __restrict__ bsum) {
  __shared__ double smx[32];
  __shared__ uint64_t sm[32];
  const double mx = block_max(threadIdx.x, nmax, kScanBlock,
                              [&](long long i) { return maxima[i]; }, smx);
  const long long i = (long long)blockIdx.x * kScanBlock + threadIdx.x;
  uint64_t q = 0;
  if (i < n) {
    const double l = logw[i];
    const double wgt = l == l ? refmath::exp_ref(l - mx) : 0.0;
    q = (uint64_t)floor(wgt * 1099511627776.0);  // 2^40
  }
  const uint64_t in = block_scan(q, sm);
  if (i < n) incl[i] = in;
  if (threadIdx.x == kScanBlock - 1) bsum[blockIdx.x] = in;
}

// Inclusive prefix of the block totals, one CTA walking them in chunks; then the quotients
// and remainders by n of the total Q and of floor(u Q), and whether resampling is possible
// (a positive weight, a maximum that is neither -inf nor +inf).
struct ResampleTotals {
  uint64_t q_div, q_rem, u_div, u_rem;
  int32_t valid;
};
__global__ void k_scan_blocks(int nb, uint64_t* __restrict__ bsum, int64_t n,
                              const double* __restrict__ maxima, int nmax, uint64_t seed,
                              uint64_t id_base, ResampleTotals* __restrict__ tot) {
  __shared__ uint64_t sm[32];
  __shared__ uint64_t carry;
  __shared__ double smx[32];
  const double mx = block_max(threadIdx.x, nmax, kScanBlock,
                              [&](long long i) { return maxima[i]; }, smx);
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < nb; base += kScanBlock) {
    const int i = base + threadIdx.x;
    const uint64_t v = i < nb ? bsum[i] : 0;
    const uint64_t in = block_scan(v, sm) + carry;
    if (i < nb) bsum[i] = in;
    __syncthreads();
    if (threadIdx.x == kScanBlock - 1) carry = in;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const uint64_t Q = carry;
    const Words4 w = philox_block((uint32_t)seed, (uint32_t)(seed >> 32), (uint32_t)id_base,
                                  0xC0000000u, 0u, 0u);
    const uint64_t uQ = (uint64_t)floor(u01_f64(w.w0, w.w1) * (double)Q);
    tot->q_div = Q / (uint64_t)n;
    tot->q_rem = Q % (uint64_t)n;
    tot->u_div = uQ / (uint64_t)n;
    tot->u_rem = uQ % (uint64_t)n;
    tot->valid = mx > neg_inf() && mx != __longlong_as_double(0x7ff0000000000000LL) && Q != 0;
  }
}

// Ancestor k: the first i whose inclusive prefix exceeds (k Q + floor(u Q)) / n, by quotients
// and remainders (k < n < 2^24, so the remainders' sum fits 64 bits); first the block, by
// the blocks' inclusive totals, then within its kScanBlock prefixes, whose lines the
// neighbouring ancestors share.
__global__ void k_ancestors(int64_t n, int nb, const uint64_t* __restrict__ incl,
                            const uint64_t* __restrict__ bsum,
                            const ResampleTotals* __restrict__ tot, int64_t* __restrict__ anc) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const ResampleTotals t = *tot;
  if (!t.valid) {
    anc[k] = -1;
    return;
  }
  const uint64_t target = (uint64_t)k * t.q_div + t.u_div +
                          ((uint64_t)k * t.q_rem + t.u_rem) / (uint64_t)n;
  int lo = 0, hi = nb - 1;  // first block with total > target (exists: target < Q)
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (bsum[mid] > target) hi = mid;
    else lo = mid + 1;
  }
  const uint64_t rest = target - (lo > 0 ? bsum[lo - 1] : 0);
  long long a = (long long)lo * kScanBlock, b = a + kScanBlock - 1;
  if (b > n - 1) b = n - 1;
  while (a < b) {
    const long long mid = (a + b) >> 1;
    if (incl[mid] > rest) b = mid;
    else a = mid + 1;
  }
  anc[k] = a;
}

// Workspace: n prefixes, nb block totals, then (16-byte aligned) the totals and the maxima.
// Its size is what callers hold already: 512 bytes beyond the prefixes and block totals, so
// the maxima are at most 48.
constexpr int kMaxima = 48;
size_t resample_tail(int64_t n) {
  const int64_t nb = (n + kScanBlock - 1) / kScanBlock;
  return ((size_t)n * 8 + (size_t)nb * 8 + 15) / 16 * 16;
}
size_t resample_ws(int64_t n) {
  const int64_t nb = (n + kScanBlock - 1) / kScanBlock;
  return 256 + (size_t)n * 8 + (size_t)nb * 8 + 256;
}

}  // namespace
}  // namespace mlk

extern "C" {

int ml_posterior_sample(int64_t n, int32_t M, const double* alpha, int32_t alpha_per_traj,
                        const double* beta, int32_t beta_per_traj, const int64_t* r,
                        const double* G, uint64_t seed, uint64_t traj_id_base, double* theta_out,
                        uint32_t* status_out, void* stream) {
  using namespace mlk;
  if (n < 0 || M < 1 || M > 4096) return set_error(ML_ERR_ARG, "need n >= 0 and 1 <= M <= 4096");
  if (traj_id_base > 0xffffffffULL || (uint64_t)n > 0x100000000ULL - traj_id_base)
    return set_error(ML_ERR_ARG, "trajectory ids must stay below 2^32");
  if (n == 0) return ML_OK;
  const void* req[] = {alpha, beta, r, G, theta_out};
  for (const void* p : req)
    if (!is_device_pointer(p)) return set_error(ML_ERR_ARG, "alpha, beta, r, G and theta_out must be device memory");
  if (status_out && !is_device_pointer(status_out)) return set_error(ML_ERR_ARG, "status_out must be device memory");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (status_out) {
    cudaError_t e = cudaMemsetAsync(status_out, 0, (size_t)n * 4, s);
    if (e != cudaSuccess) return set_error(ML_ERR_CUDA, cudaGetErrorString(e));
  }
  const long long total = n * (long long)M;
  const int block = 256;
  const long long grid = (total + block - 1) / block;
  if (grid > 0x7fffffffLL) return set_error(ML_ERR_ARG, "n * M too large for one launch");
  k_posterior<<<(unsigned)grid, block, 0, s>>>(n, M, alpha, alpha_per_traj, beta, beta_per_traj,
                                                r, G, seed, traj_id_base, theta_out, status_out);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ML_OK : set_error(ML_ERR_CUDA, cudaGetErrorString(e));
}

size_t ml_resample_workspace_bytes(int64_t n) { return n < 1 ? 0 : mlk::resample_ws(n); }

int ml_resample_systematic(int64_t n, const double* logw, uint64_t seed, uint64_t id_base,
                           int64_t* ancestors, void* workspace, size_t workspace_bytes,
                           void* stream) {
  using namespace mlk;
  // q_i <= 2^40, so the 64-bit prefix sums stay exact for n < 2^24.
  if (n < 1 || n >= (1LL << 24)) return set_error(ML_ERR_ARG, "need 1 <= n < 2^24");
  if (!is_device_pointer(logw) || !is_device_pointer(ancestors) || !is_device_pointer(workspace))
    return set_error(ML_ERR_ARG, "logw, ancestors and workspace must be device memory");
  if (workspace_bytes < resample_ws(n))
    return set_error(ML_ERR_ARG, "workspace smaller than ml_resample_workspace_bytes(n)");
  if (reinterpret_cast<uintptr_t>(workspace) % 16)
    return set_error(ML_ERR_ARG, "workspace must be 16-byte aligned");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char* ws = static_cast<char*>(workspace);
  // Four launches: block maxima, quantization with block scans, the scan of the block totals,
  // the ancestors.  1,000,000 particles: 155 us with six launches, a maximum over 32 CTAs
  // and a 128-bit division per ancestor; the quantization's exponentials on the FP64 unit
  // take about 50 us.
  const int64_t nb = (n + kScanBlock - 1) / kScanBlock;
  const int nmax = (int)(nb < kMaxima ? nb : kMaxima);
  uint64_t* incl = reinterpret_cast<uint64_t*>(ws);           // n prefixes within blocks
  uint64_t* bsum = incl + n;                                  // nb block totals
  char* tail = ws + resample_tail(n);
  ResampleTotals* tot = reinterpret_cast<ResampleTotals*>(tail);
  double* mx = reinterpret_cast<double*>(tail + 64);          // nmax maxima
  k_block_max<<<nmax, 1024, 0, s>>>(n, logw, mx);
  k_quantize_scan<<<(unsigned)nb, kScanBlock, 0, s>>>(n, logw, mx, nmax, incl, bsum);
  k_scan_blocks<<<1, kScanBlock, 0, s>>>((int)nb, bsum, n, mx, nmax, seed, id_base, tot);
  k_ancestors<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, (int)nb, incl, bsum, tot, ancestors);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ML_OK : set_error(ML_ERR_CUDA, cudaGetErrorString(e));
}

}  // extern "C"
