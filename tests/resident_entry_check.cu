// How blocks enter a resident launch (swe_resident.cuh, pass_entry): over
// launches of several scenarios, whose blocks pass the entry in any order and
// each with the epoch it read before, every block of a launch reads the same
// epoch, the scenario's last block advances it past the launch's (also over
// the wrap of 32 bits), and the ticket is 0 again. Prints "ok" or the first
// difference. Test code: built and run by tests/test_gpu_resident.py.
#include <cstdio>

#include "../paper_1807_00672_gb300/csrc/swe_resident.cuh"

constexpr int kScen = 5, kMost = 152;

__global__ void k_enter(swe::Ctl* ctls, uint32_t* epoch, uint32_t n_steps, const int* nblocks,
                        uint32_t* read) {
  const int scen = blockIdx.x / kMost, b = blockIdx.x % kMost;
  if (threadIdx.x != 0 || b >= nblocks[scen]) return;
  const uint32_t e0 = *(volatile uint32_t*)(epoch + scen) + 1u;
  read[blockIdx.x] = e0;
  swe::pass_entry(ctls + scen, epoch + scen, e0 + n_steps + 1u, nblocks[scen]);
}

int main() {
  swe::Ctl h[kScen] = {};
  uint32_t e[kScen] = {0, 7, 0xfffffff0u, 3, 1}, want[kScen], read[kScen * kMost];
  const int nblocks[kScen] = {1, 2, 31, 151, 152};
  for (int i = 0; i < kScen; ++i) want[i] = e[i];
  swe::Ctl* dc;
  uint32_t *de, *dr;
  int* dn;
  if (cudaMalloc(&dc, sizeof h) != cudaSuccess || cudaMalloc(&de, sizeof e) != cudaSuccess ||
      cudaMalloc(&dn, sizeof nblocks) != cudaSuccess || cudaMalloc(&dr, sizeof read) != cudaSuccess)
    return 2;
  cudaMemcpy(dc, h, sizeof h, cudaMemcpyHostToDevice);
  cudaMemcpy(de, e, sizeof e, cudaMemcpyHostToDevice);
  cudaMemcpy(dn, nblocks, sizeof nblocks, cudaMemcpyHostToDevice);
  for (uint32_t l = 0; l < 200; ++l) {
    const uint32_t n = 1u + 5u * (l % 7u);
    k_enter<<<kScen * kMost, 32>>>(dc, de, n, dn, dr);
    if (cudaDeviceSynchronize() != cudaSuccess) return 3;
    cudaMemcpy(h, dc, sizeof h, cudaMemcpyDeviceToHost);
    cudaMemcpy(e, de, sizeof e, cudaMemcpyDeviceToHost);
    cudaMemcpy(read, dr, sizeof read, cudaMemcpyDeviceToHost);
    for (int i = 0; i < kScen; ++i) {
      bool bad = false;
      for (int b = 0; b < nblocks[i]; ++b) bad = bad || read[i * kMost + b] != want[i] + 1u;
      want[i] += n + 2u;
      if (bad || e[i] != want[i] || h[i].ticket != 0u) {
        std::printf("launch %u scenario %d: epoch %u (%u) ticket %u\n", l, i, e[i], want[i], h[i].ticket);
        return 1;
      }
    }
  }
  std::printf("ok\n");
  return 0;
}
