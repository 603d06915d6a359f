// Compares near_recip with the division on 2^24 values over its range of exponents and both
// signs, and on values outside the range (built and run by tests/test_gpu_edges.py).
// Output: values compared, those that differ, largest difference in units in the last place.
#include <cstdio>

#include "thread_core.cuh"

__global__ void k_compare(unsigned long long* out) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  const mlk::Words4 w = mlk::philox_block(1u, 2u, i, 0u, 0u, 0u);
  // exponents 2^-110 .. 2^110: the fast range is 2^-100 .. 2^100
  const unsigned e = 1023u - 110u + w.w2 % 221u;
  const double b = __hiloint2double((int)((w.w3 << 31) | (e << 20) | (w.w0 & 0xfffffu)), (int)w.w1);
  const long long d = __double_as_longlong(mlk::near_recip(b)) - __double_as_longlong(1.0 / b);
  if (d != 0) atomicAdd(out, 1ULL);
  atomicMax(out + 1, (unsigned long long)(d < 0 ? -d : d));
}

int main() {
  unsigned long long* out = nullptr;
  if (cudaMallocManaged(&out, 16) != cudaSuccess) return 1;
  out[0] = out[1] = 0;
  k_compare<<<1 << 16, 256>>>(out);
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  std::printf("%d %llu %llu\n", 1 << 24, out[0], out[1]);
  return 0;
}
