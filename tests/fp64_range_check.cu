// Accuracy of the library's FP64 reciprocal, square root and inverse cube
// root (swe_kernels.cuh) against CUDA's IEEE functions over the whole range of
// exponents: 2^20 seeded arguments log-uniform in [2^-1020, 2^1020], every
// power of two and its neighbours there, and the special values. Prints the
// largest error of each in units of the last place of the IEEE result, and
// the number of special values that differ. Test code: built and run by
// tests/test_gpu_fp64_range.py.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <vector>

#include "../paper_1807_00672_gb300/csrc/swe_kernels.cuh"

__device__ double ulps(double got, double want) {
  if (got == want) return 0.0;
  const long long g = __double_as_longlong(got), w = __double_as_longlong(want);
  return fabs((double)(g - w));
}
__device__ bool same(double a, double b) { return a == b || (isnan(a) && isnan(b)); }

__global__ void k_check(const double* x, int n, double* out, const double* sp, int nsp, int* bad) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    const double a = x[i];
    out[3 * i + 0] = ulps(swe::rcp_nr(a), 1.0 / a);
    out[3 * i + 1] = ulps(swe::sqrt_nr(a), sqrt(a));
    out[3 * i + 2] = ulps(swe::icbrt_nr(a), 1.0 / cbrt(a));
  }
  if (i < nsp && !same(swe::sqrt_nr(sp[i]), sqrt(sp[i]))) atomicAdd(bad, 1);
}

int main() {
  std::vector<double> x;
  uint64_t s = 0x9E3779B97F4A7C15ull;
  auto next = [&]() {
    s ^= s << 13; s ^= s >> 7; s ^= s << 17;
    return (double)(s >> 11) / 9007199254740992.0;
  };
  for (int i = 0; i < 1 << 20; ++i) x.push_back(std::exp2(-1020.0 + 2040.0 * next()));
  for (int e = -1020; e <= 1020; ++e) {
    const double p = std::ldexp(1.0, e);
    x.push_back(p);
    x.push_back(std::nextafter(p, 0.0));
    x.push_back(std::nextafter(p, INFINITY));
    x.push_back(p * (1.0 + std::ldexp(1.0, -23)));
    x.push_back(p * (1.0 + std::ldexp(1.0, -24) + std::ldexp(1.0, -52)));
  }
  const std::vector<double> sp = {0.0, -0.0, INFINITY, -INFINITY, NAN, -1.0, 4.9e-324, 1e-310, 2.3e-308, 1.7e308};
  const int n = (int)x.size(), nsp = (int)sp.size();
  double *dx, *dsp, *dout;
  int* dbad;
  if (cudaMalloc(&dx, n * 8) != cudaSuccess || cudaMalloc(&dsp, nsp * 8) != cudaSuccess ||
      cudaMalloc(&dout, 3 * (size_t)n * 8) != cudaSuccess || cudaMalloc(&dbad, 4) != cudaSuccess) {
    printf("alloc failed\n");
    return 2;
  }
  cudaMemcpy(dx, x.data(), n * 8, cudaMemcpyHostToDevice);
  cudaMemcpy(dsp, sp.data(), nsp * 8, cudaMemcpyHostToDevice);
  cudaMemset(dbad, 0, 4);
  k_check<<<(n + 255) / 256, 256>>>(dx, n, dout, dsp, nsp, dbad);
  if (cudaDeviceSynchronize() != cudaSuccess) {
    printf("kernel failed\n");
    return 3;
  }
  std::vector<double> ho(3 * (size_t)n);
  int bad = 0;
  cudaMemcpy(ho.data(), dout, ho.size() * 8, cudaMemcpyDeviceToHost);
  cudaMemcpy(&bad, dbad, 4, cudaMemcpyDeviceToHost);
  double mx[3] = {0, 0, 0};
  for (int i = 0; i < n; ++i)
    for (int c = 0; c < 3; ++c) mx[c] = std::fmax(mx[c], ho[3 * (size_t)i + c]);
  printf("rcp %.3f\nsqrt %.3f\nicbrt %.3f\nspecial %d\n", mx[0], mx[1], mx[2], bad);
  return 0;
}
