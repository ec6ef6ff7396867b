// Host memory that runs out inside the mesh builder (mesh_build.cpp): with
// operator new failing from the k-th allocation on, on whichever host thread
// that falls, for many k up to the number a build needs, each stage returns
// (or throws std::bad_alloc on the calling thread) with every thread joined,
// and works again afterwards. argv[1]: "parts" (build_resident_parts: false),
// "banks" (order_records_for_banks: each tile reordered or left alone) or
// "guard" (OnThrow, which gives up handles under construction). Prints "ok <failures seen>" or the first difference. Test code: built and
// run by tests/test_host_memory.py.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "../paper_1807_00672_gb300/csrc/mesh_build.h"

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

// OnThrow: runs on the way of an exception out of its scope, also one thrown
// while another is under way, and not on a return.
static int g_ran = 0;
static void scope(bool throws) {
  swe::OnThrow on_throw([] { ++g_ran; });
  if (throws) throw std::bad_alloc();
}
struct Unwinding {
  ~Unwinding() { scope(false); }
};
static int guard_check() {
  scope(false);
  if (g_ran != 0) return 1;
  try {
    Unwinding u;
    scope(true);
  } catch (const std::bad_alloc&) {
  }
  std::printf("ok %d\n", g_ran);
  return g_ran == 1 ? 0 : 1;
}

int main(int, char** argv) {
  if (!std::strcmp(argv[1], "guard")) return guard_check();
  const bool banks = !std::strcmp(argv[1], "banks");
  const int32_t nx = banks ? 420 : 120, ny = banks ? 250 : 100;  // threads from 200,000 and 4,000 cells
  std::vector<double> xy;
  std::vector<int32_t> tri;
  for (int32_t j = 0; j <= ny; ++j)
    for (int32_t i = 0; i <= nx; ++i) {
      xy.push_back(i + 0.2 * ((7 * i + 3 * j) % 5) / 5.0);
      xy.push_back(j);
    }
  for (int32_t j = 0; j < ny; ++j)
    for (int32_t i = 0; i < nx; ++i) {
      const int32_t a = j * (nx + 1) + i, b = a + 1, c = a + nx + 2, d = a + nx + 1;
      for (int32_t v : {a, b, c, a, c, d}) tri.push_back(v);
    }
  const int64_t V = (int64_t)xy.size() / 2, T = (int64_t)tri.size() / 3;
  swe::HostMesh m;
  if (swe::build_host_mesh(xy.data(), V, tri.data(), T, 1, banks ? 256 : 0, false, m, false, !banks) != 0)
    return 3;
  swe::HostMesh whole = m;
  swe::ResidentParts p;
  auto stage = [&](swe::HostMesh& on) {
    if (!banks) return swe::build_resident_parts(on, xy.data(), tri.data(), true, 152, p);
    swe::order_records_for_banks(on);
    return true;
  };
  g_count = 0;
  if (!stage(whole)) return 3;
  const long long need = g_count;
  int seen = 0;
  const long long fails = banks ? 12 : 60;
  for (long long f = 0; f < fails; ++f) {
    swe::HostMesh on = m;
    g_left = need * f / fails;
    const bool ok = stage(on);
    g_left = -1;
    if (!banks) {
      seen += !ok;
      continue;
    }
    bool left = false;
    for (int64_t t = 0; t < on.ntiles; ++t) {
      auto same = [&](const swe::HostMesh& as) {
        return std::equal(on.tA.begin() + on.toff[t], on.tA.begin() + on.toff[t + 1], as.tA.begin() + on.toff[t]) &&
               std::equal(on.tnx.begin() + on.toff[t], on.tnx.begin() + on.toff[t + 1], as.tnx.begin() + on.toff[t]);
      };
      if (!same(whole) && !same(m)) {
        std::printf("a tile in half an order\n");
        return 1;
      }
      left = left || !same(whole);
    }
    seen += left;
  }
  if (!stage(m)) return 3;
  std::printf("ok %d\n", seen);
  return 0;
}
