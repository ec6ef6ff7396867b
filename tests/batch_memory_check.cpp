// swe_mesh_create_batch with operator new (this program's own, which the
// library takes too) failing from the k-th allocation on, for many k up to the
// number it needs before it asks for a device: SWE_ENOMEM each time, and
// SWE_ECUDA (no device is visible) with enough. Prints "ok <failures seen>" or
// the first other status. Test code: built and run by tests/test_host_memory.py.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include <vector>

#include "../include/swe.h"

static std::atomic<long long> g_left{-1}, g_count{0};
void* operator new(std::size_t n) {
  g_count += 1;
  if (g_left.load() >= 0 && g_left.fetch_sub(1) <= 0) {
    g_left = 0;
    throw std::bad_alloc();
  }
  if (void* p = std::malloc(n ? n : 1)) return p;
  throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

int main() {
  constexpr int kScen = 12;
  const int32_t nx = 60, ny = 40;
  std::vector<double> xy;
  std::vector<int32_t> tri;
  for (int32_t j = 0; j <= ny; ++j)
    for (int32_t i = 0; i <= nx; ++i) {
      xy.push_back(i);
      xy.push_back(j);
    }
  for (int32_t j = 0; j < ny; ++j)
    for (int32_t i = 0; i < nx; ++i) {
      const int32_t a = j * (nx + 1) + i, b = a + 1, c = a + nx + 2, d = a + nx + 1;
      for (int32_t v : {a, b, c, a, c, d}) tri.push_back(v);
    }
  const double* xys[kScen];
  const int32_t* tris[kScen];
  int64_t nodes[kScen], cells[kScen];
  for (int i = 0; i < kScen; ++i) {
    xys[i] = xy.data();
    tris[i] = tri.data();
    nodes[i] = (int64_t)xy.size() / 2;
    cells[i] = (int64_t)tri.size() / 3;
  }
  swe_params p;
  swe_params_default(&p);
  p.precision = SWE_F32;
  auto create = [&]() {
    swe_mesh* m = nullptr;
    return swe_mesh_create_batch(kScen, xys, nodes, tris, cells, &p, nullptr, &m);
  };
  g_count = 0;
  if (create() != SWE_ECUDA) {
    std::printf("with memory: not SWE_ECUDA\n");
    return 1;
  }
  const long long need = g_count;
  int seen = 0;
  for (int f = 0; f < 40; ++f) {
    g_left = need * f / 40;
    const swe_status st = create();
    g_left = -1;
    if (st != SWE_ENOMEM && st != SWE_ECUDA) {
      std::printf("allocation %lld: status %d\n", need * f / 40, (int)st);
      return 1;
    }
    seen += st == SWE_ENOMEM;
  }
  if (create() != SWE_ECUDA) return 1;
  std::printf("ok %d\n", seen);
  return 0;
}
