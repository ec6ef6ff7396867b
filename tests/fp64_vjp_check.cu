// The transposed friction of one cell in FP64 (cell_vjp, swe_adjoint.cuh): its
// depth part against the same expression with an IEEE 1 / h, over 2^20 seeded
// wet cells (depths log-uniform in [2^-12, 2^6]). 1 / h enters once, by a
// reciprocal within an ulp of IEEE's: at most two units in the last place.
// Prints the largest difference in those units. Test code: built and run by
// tests/test_gpu_fp64_range.py.
#include <cstdio>

#include "../paper_1807_00672_gb300/csrc/swe_adjoint.cuh"

__global__ void k_check(int n, int* most) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  unsigned long long s = (i + 1) * 0x9E3779B97F4A7C15ull;
  auto next = [&]() {
    s ^= s << 13; s ^= s >> 7; s ^= s << 17;
    return (double)(s >> 11) / 9007199254740992.0;
  };
  for (int k = 0; k < 8; ++k) next();
  const double h = exp2(-12.0 + 18.0 * next()), qx = 4.0 * next() - 2.0, qy = 4.0 * next() - 2.0;
  const double lx = 2.0 * next() - 1.0, ly = 2.0 * next() - 1.0, gn2 = 0.02 * next() + 1e-4, dt = next();
  const swe::Num num{9.81, 0.7, 1e-6, 1e-6f, 1u};
  double mh, mx, my, b;
  swe::cell_vjp(h, qx, qy, swe::Ops<double>::rcp(h), 0.0, lx, ly, gn2, dt, num, mh, mx, my, b);
  const double c = __dmul_rn(__dmul_rn(dt, swe::Ops<double>::pow_m73(h)), gn2);
  const double cq = __dmul_rn(c, __dsqrt_rn(__fma_rn(qx, qx, __dmul_rn(qy, qy))));
  const double ql = __fma_rn(qx, lx, __dmul_rn(qy, ly));
  const double want = __dmul_rn(__dmul_rn(7.0 / 3.0, __dmul_rn(cq, __ddiv_rn(1.0, h))), ql);
  const long long d = llabs(__double_as_longlong(mh) - __double_as_longlong(want));
  atomicMax(most, (int)min(d, 1000000ll));
}

int main() {
  int *d, h = -1;
  if (cudaMalloc(&d, 4) != cudaSuccess || cudaMemset(d, 0, 4) != cudaSuccess) return 2;
  k_check<<<4096, 256>>>(1 << 20, d);
  if (cudaDeviceSynchronize() != cudaSuccess) return 3;
  cudaMemcpy(&h, d, 4, cudaMemcpyDeviceToHost);
  std::printf("ulps %d\n", h);
  return 0;
}
