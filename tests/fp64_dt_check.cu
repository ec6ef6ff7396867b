// The CFL time step (cfl_dt, swe_kernels.cuh) against CUDA's IEEE division, bit
// for bit: 2^26 random rates for Courant numbers 0.7 and random ones, quotients
// next to half way between two doubles among them, exponents of rate, Courant
// number and quotient up to 2^+-440, and rates of 0 and infinity; beyond, up to
// the ends of the range, within an ulp. Prints how many differ. Test code: built and run by tests/test_gpu_fp64_range.py.
#include <cstdio>

#include "../paper_1807_00672_gb300/csrc/swe_kernels.cuh"

__device__ bool differs(double c, double r) {
  const double got = swe::cfl_dt(c, r), want = __ddiv_rn(c, r);
  return __double_as_longlong(got) != __double_as_longlong(want) && !(got != got && want != want);
}

__global__ void k_check(int per, unsigned long long* differ) {
  unsigned long long s = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * per, bad = 0;
  for (int j = 0; j < per; ++j) {
    unsigned long long z = ++s * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    const double r = __longlong_as_double((long long)((z >> 12) | 0x3ff0000000000000ull));  // [1, 2)
    const double f = __longlong_as_double((long long)(((z * 0xD6E8FEB86659FD93ull) >> 12) | 0x3ff0000000000000ull));
    double c = 0.7, x = r;
    if (j & 1) {  // next to (f + 2^-53) r
      const double p = f * r, e = fma(f, r, -p);
      c = p + (e + r * 1.1102230246251565e-16);
      c = __longlong_as_double(__double_as_longlong(c) + (long long)(z & 3u) - 1);
    }
    if (j & 2) x = scalbn(x, (int)(z % 440u) - 220);
    if (j & 4) c = scalbn(c, (int)((z >> 20) % 440u) - 220);
    bad += differs(c, x);
    const double far = scalbn(r, (int)(z % 2040u) - 1018), want = __ddiv_rn(0.7, far);
    if (want > 2.3e-308 && want < INFINITY && !(fabs(swe::cfl_dt(0.7, far) - want) <= want * 2.3e-16)) ++bad;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    for (double c : {0.7, 1.0, 1e-3, 1e3, 1e-300, 1e300})
      for (double r : {0.0, (double)INFINITY}) bad += differs(c, r);
  }
  if (bad) atomicAdd(differ, bad);
}

int main() {
  unsigned long long *d, h = 1;
  if (cudaMalloc(&d, 8) != cudaSuccess || cudaMemset(d, 0, 8) != cudaSuccess) return 2;
  k_check<<<2048, 256>>>(128, d);
  if (cudaDeviceSynchronize() != cudaSuccess) return 3;
  cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost);
  std::printf("differ %llu\n", h);
  return 0;
}
