// The library's FP64 square root (sqrt_nr, swe_kernels.cuh) against CUDA's
// IEEE square root, bit for bit: 2^26 arguments whose roots lie next to half
// way between two doubles (squares of such numbers, rounded, and their
// neighbours, in both halves of the range of even and odd exponents), as many
// random ones, exponents over the whole range. Prints how many differ. Test
// code: built and run by tests/test_gpu_fp64_range.py.
#include <cstdio>

#include "../paper_1807_00672_gb300/csrc/swe_kernels.cuh"

__global__ void k_check(int per, unsigned long long* differ) {
  unsigned long long s = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * per;
  unsigned long long bad = 0;
  for (int j = 0; j < per; ++j) {
    unsigned long long z = ++s * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    // v in [1, 2)
    const double v = __longlong_as_double((long long)((z >> 12) | 0x3ff0000000000000ull));
    double x = v;
    if (j & 1) {  // next to (v + 2^-53)^2
      const double p = v * v, e = fma(v, v, -p);
      x = p + (e + 2.0 * v * 1.1102230246251565e-16);
      x = __longlong_as_double(__double_as_longlong(x) + (long long)(z & 3u) - 1);
    } else if (j & 2) {
      x *= 2.0;
    }
    x = scalbn(x, 2 * ((int)((z >> 2) & 1023u) - 511));
    if (!(x == x) || isinf(x)) continue;
    if (__double_as_longlong(swe::sqrt_nr(x)) != __double_as_longlong(__dsqrt_rn(x))) ++bad;
  }
  if (bad) atomicAdd(differ, bad);
}

int main() {
  unsigned long long *d, h = 1;
  if (cudaMalloc(&d, 8) != cudaSuccess || cudaMemset(d, 0, 8) != cudaSuccess) return 2;
  k_check<<<4096, 256>>>(128, d);
  if (cudaDeviceSynchronize() != cudaSuccess) return 3;
  cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost);
  std::printf("differ %llu\n", h);
  return 0;
}
