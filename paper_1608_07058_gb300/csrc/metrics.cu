// Accuracy metric of the paper's Section 3 (Table 1): the Kullback-Leibler divergence of
// a method's marginal distributions from those of exact SSA, per time point and species,
// averaged over all of them.  Binned, half-count-smoothed empirical distributions (the
// paper does not say how it forms them): bins of integer width w = ceil((hi - lo + 1) /
// max_bins) on the pooled range of both samples, 1/2 added to every bin.  Compiled without
// FMA contraction; the counts are exact integers and the FP64 sums take a fixed lane
// order, so the results are bit-reproducible.
#include <cstdint>

#include <cuda_runtime.h>

#include "dev_common.cuh"
#include "matleap.h"
#include "ml_internal.h"

namespace mlk {
namespace {

constexpr int kKlThreads = 1024;  // 32 warps: one per lane of the final reductions
constexpr int kKlMaxBins = 4096;
constexpr int kKlTable = 320;  // counts with a tabulated logarithm

__device__ __forceinline__ long long warp_min(long long v) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    const long long o = __shfl_xor_sync(0xffffffffu, v, d);
    v = o < v ? o : v;
  }
  return v;
}

__device__ __forceinline__ long long warp_max(long long v) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    const long long o = __shfl_xor_sync(0xffffffffu, v, d);
    v = o > v ? o : v;
  }
  return v;
}

// Sum in the canonical order: lane l adds elements l, l + 32, ... in increasing index
// (an empty lane holds 0), then lanes combine pairwise at xor distances 16, 8, 4, 2, 1.
// Called by one full warp; every lane returns the sum.
template <class F>
__device__ __forceinline__ double lane_tree(int n, int lane, F elem) {
  double v = 0.0;
  for (int j = lane; j < n; j += 32) v = (j < 32) ? elem(j) : v + elem(j);
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) v = v + __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

// A bin's term p (log p - log q) in the order of the definition: p = (c + 1/2) / d.
struct Prob {
  double p, lp;
};
__device__ __forceinline__ Prob prob_of(unsigned c, double d) {
  const double p = (f64_of_count((long long)c) + 0.5) / d;
  return Prob{p, refmath::log_ref(p)};
}

// Values of a sample, kKlBatch loads in flight per thread: one CTA reads a column of the
// sample array (stride K N), so the loads' latency, not their bytes, is what it waits for.
constexpr int kKlBatch = 8;
template <class F>
__device__ __forceinline__ void for_samples(const int64_t* __restrict__ x, long long n,
                                            long long stride, F f) {
  long long i = threadIdx.x;
  for (; i + (kKlBatch - 1) * kKlThreads < n; i += kKlBatch * kKlThreads) {
    long long v[kKlBatch];
#pragma unroll
    for (int q = 0; q < kKlBatch; ++q) v[q] = x[(i + q * kKlThreads) * stride];
#pragma unroll
    for (int q = 0; q < kKlBatch; ++q) f(v[q]);
  }
  for (; i < n; i += kKlThreads) f(x[i * stride]);
}

// One CTA per (time point k, species s).  X layout [n][K][N].  The probabilities and
// logarithms are computed once per distinct count (a bin holds at most a few dozen of the
// samples, and the tails' bins hold the same few counts) by all warps, and the terms by all
// warps; one warp only adds them in the canonical order.  10,000 trajectories of 20 points and
// 3 species (60 CTAs, 9.6 MB): 40 us, bound by the latency of the strided loads; 124 us with
// 256 threads, one load in flight each and one warp taking two logarithms and two divisions
// per bin (about 120 instructions of 64 cycles on the FP64 unit for each 32 of some 700 bins).
__global__ void __launch_bounds__(kKlThreads) k_kl(int64_t n_ref, const int64_t* __restrict__ Xr,
                                                  int64_t n_test, const int64_t* __restrict__ Xt,
                                                  int K, int N, int max_bins,
                                                  double* __restrict__ kl) {
  __shared__ uint2 bin[kKlMaxBins];          // counts of both samples, then the bin's term
  __shared__ Prob ta[kKlTable], tb[kKlTable];  // by count
  __shared__ long long red_lo[kKlThreads / 32], red_hi[kKlThreads / 32];
  __shared__ unsigned max_a, max_b;
  const int ks = blockIdx.x;  // k * N + s
  const long long stride = (long long)K * N;
  const int64_t* a = Xr + ks;
  const int64_t* b = Xt + ks;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  // pooled range (exact integer reductions)
  long long lo = a[0], hi = lo;
  auto widen = [&](long long v) {
    lo = v < lo ? v : lo;
    hi = v > hi ? v : hi;
  };
  for_samples(a, n_ref, stride, widen);
  for_samples(b, n_test, stride, widen);
  lo = warp_min(lo);
  hi = warp_max(hi);
  if (lane == 0) {
    red_lo[warp] = lo;
    red_hi[warp] = hi;
  }
  for (int j = threadIdx.x; j < max_bins; j += kKlThreads) bin[j] = make_uint2(0u, 0u);
  if (threadIdx.x == 0) max_a = max_b = 0u;
  __syncthreads();
  lo = warp_min(red_lo[lane]);
  hi = warp_max(red_hi[lane]);
  // bin width w = ceil((d + 1) / max_bins) = floor(d / max_bins) + 1 with d = hi - lo, in
  // unsigned arithmetic so that any pair of int64 values gives a bin index < max_bins
  const unsigned long long d = (unsigned long long)hi - (unsigned long long)lo;
  const unsigned long long w = d / (unsigned long long)max_bins + 1ull;
  const int nbins = (int)(d / w + 1ull);
  // the division in 32 bits where range and width both fit (one bin over a range of 2^32 - 1
  // has a width of 2^32)
  const bool narrow = ((d | w) >> 32) == 0ull;
  auto bin_of = [&](long long v) {
    const unsigned long long o = (unsigned long long)v - (unsigned long long)lo;
    return w == 1ull ? (int)o : narrow ? (int)((unsigned)o / (unsigned)w) : (int)(o / w);
  };

  for_samples(a, n_ref, stride, [&](long long v) { atomicAdd(&bin[bin_of(v)].x, 1u); });
  for_samples(b, n_test, stride, [&](long long v) { atomicAdd(&bin[bin_of(v)].y, 1u); });
  __syncthreads();

  unsigned ma = 0u, mb = 0u;
  for (int j = threadIdx.x; j < nbins; j += kKlThreads) {
    ma = max(ma, bin[j].x);
    mb = max(mb, bin[j].y);
  }
  ma = __reduce_max_sync(0xffffffffu, ma);
  mb = __reduce_max_sync(0xffffffffu, mb);
  if (lane == 0) {
    atomicMax(&max_a, ma);
    atomicMax(&max_b, mb);
  }
  __syncthreads();
  const double da = f64_of_count(n_ref) + 0.5 * f64_of_count(nbins);
  const double db = f64_of_count(n_test) + 0.5 * f64_of_count(nbins);
  // tables of the counts that occur, where they are fewer than the bins; larger counts
  // directly
  const unsigned na = min(max_a + 1u, (unsigned)kKlTable), nb = min(max_b + 1u, (unsigned)kKlTable);
  const bool table = na + nb < 2u * (unsigned)nbins;
  if (table) {
    for (unsigned c = threadIdx.x; c < na + nb; c += kKlThreads) {
      if (c < na) ta[c] = prob_of(c, da);
      else tb[c - na] = prob_of(c - na, db);
    }
    __syncthreads();
  }
  double* term = reinterpret_cast<double*>(bin);
  for (int j = threadIdx.x; j < nbins; j += kKlThreads) {
    const uint2 c = bin[j];
    const Prob p = table && c.x < na ? ta[c.x] : prob_of(c.x, da);
    const Prob q = table && c.y < nb ? tb[c.y] : prob_of(c.y, db);
    term[j] = p.p * (p.lp - q.lp);
  }
  __syncthreads();
  if (warp == 0) {
    const double sum = lane_tree(nbins, lane, [&](int j) { return term[j]; });
    if (lane == 0) kl[ks] = sum;
  }
}

// Mean over the K x N divergences in the canonical lane order (one warp).
__global__ void k_kl_mean(int n, const double* __restrict__ kl, double* __restrict__ mean) {
  const double s = lane_tree(n, threadIdx.x & 31, [&](int j) { return kl[j]; });
  if (threadIdx.x == 0) *mean = s / (double)n;
}

}  // namespace
}  // namespace mlk

extern "C" int ml_kl_divergence(int64_t n_ref, const int64_t* X_ref, int64_t n_test,
                                const int64_t* X_test, int32_t K, int32_t N, int32_t max_bins,
                                double* kl_out, double* kl_mean_out, void* stream) {
  using namespace mlk;
  if (n_ref < 1 || n_test < 1 || n_ref >= (1LL << 31) || n_test >= (1LL << 31))
    return set_error(ML_ERR_ARG, "need 1 <= n_ref, n_test < 2^31");
  if (K < 1 || N < 1 || (int64_t)K * N > 0x7fffffffLL)
    return set_error(ML_ERR_ARG, "need K >= 1, N >= 1 and K * N < 2^31");
  if (max_bins < 1 || max_bins > kKlMaxBins)
    return set_error(ML_ERR_ARG, "need 1 <= max_bins <= 4096");
  if (!is_device_pointer(X_ref) || !is_device_pointer(X_test) || !is_device_pointer(kl_out))
    return set_error(ML_ERR_ARG, "X_ref, X_test and kl_out must be device memory");
  if (kl_mean_out && !is_device_pointer(kl_mean_out))
    return set_error(ML_ERR_ARG, "kl_mean_out must be device memory");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  k_kl<<<(unsigned)(K * N), kKlThreads, 0, s>>>(n_ref, X_ref, n_test, X_test, K, N, max_bins,
                                                 kl_out);
  if (kl_mean_out) k_kl_mean<<<1, 32, 0, s>>>(K * N, kl_out, kl_mean_out);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ML_OK : set_error(ML_ERR_CUDA, cudaGetErrorString(e));
}
