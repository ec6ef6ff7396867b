// Host side of the resident step kernel (swe_resident.cuh): which meshes take
// it, how they are cut into parts, and the launch.
#include <algorithm>
#include <cstring>
#include <vector>

#include "../../include/swe.h"
#include "mesh_build.h"
#include "swe_handles.cuh"
#include "swe_resident.cuh"

using namespace swe_host;

namespace {

#define cuda_failed(call) swe_host::cuda_failed_at((call), #call, __FILE__, __LINE__)

size_t word(const swe_mesh* m) { return m->prm.precision == SWE_F64 ? 8 : 4; }

// Shared memory of a part of `cells` compact cells: about 4 sqrt(cells) halo
// cells and half a record more per halo cell than 1.5 per cell.
int64_t part_bytes(size_t w, bool lo, int64_t cells) {
  int64_t root = 1;
  while (root * root < cells) ++root;
  const int64_t halos = 4 * root, recs = (3 * cells + halos) / 2 + 8;
  return swe::make_res_layout((uint32_t)w, lo, (uint32_t)cells, (uint32_t)halos, (uint32_t)recs).total;
}

template <typename Real, bool CH>
int occupancy(int threads, uint32_t smem) {
  auto k = swe::k_resident<Real, CH>;
  cudaFuncAttributes fa{};
  if (cudaFuncGetAttributes(&fa, k) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const int cap = smem_optin_bytes() - (int)fa.sharedSizeBytes;
  int n = 0;
  if (cap <= 0 || (int)smem > cap ||
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, cap) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

int occupancy_of(const swe_mesh* m, int threads, uint32_t smem) {
  if (m->prm.precision == SWE_F64) return occupancy<double, false>(threads, smem);
  return m->prm.compensated_depth ? occupancy<float, true>(threads, smem)
                                  : occupancy<float, false>(threads, smem);
}

template <typename Real>
swe::ResPlan<Real> res_plan(const swe_state* s) {
  const ResidentMesh& r = s->mesh->res;
  swe::ResPlan<Real> P{};
  P.blocks = (const swe::ResBlock*)(r.base + r.at_blocks);
  P.cells = (const int32_t*)(r.base + r.at_cells);
  P.pub = (const int32_t*)(r.base + r.at_pub);
  P.halo = (const int32_t*)(r.base + r.at_halo);
  P.halo_pub = (const int32_t*)(r.base + r.at_halo_pub);
  P.side = (const uint32_t*)(r.base + r.at_rec);
  P.rec = (const int4*)(r.base + r.at_rec);
  P.nx = (const Real*)(r.base + r.at_geo[0]);
  P.ny = (const Real*)(r.base + r.at_geo[1]);
  P.len = (const Real*)(r.base + r.at_geo[2]);
  P.xbuf = s->res_xbuf;
  P.slots = s->res_slots;
  P.epoch = s->res_epoch;
  P.npub = r.npub;
  return P;
}

template <typename Real, bool CH>
cudaError_t launch(const swe_state* s, int64_t n, cudaStream_t st) {
  const swe_mesh* m = s->mesh;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)m->res.nblocks);
  cfg.blockDim = dim3((unsigned)m->res.threads);
  cfg.dynamicSmemBytes = m->res.layout.total;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, swe::k_resident<Real, CH>, res_plan<Real>(s), dev_mesh<Real>(m),
                            dev_state<Real>(s), num_of(m), m->res.layout, (long long)n);
}

}  // namespace

namespace swe_host {

int64_t resident_max_cells(const swe_mesh* m) {
  const bool lo = m->prm.compensated_depth != 0;
  const int64_t cap = smem_optin_bytes() - 2048;
  int64_t c = 0;
  for (int64_t step = 4096; step > 0; step /= 2)
    while (part_bytes(word(m), lo, c + step) <= cap) c += step;
  return c;
}

static void build(swe_mesh* m, const std::vector<swe::HostMesh>& hm, const double* const* xy,
                  const int32_t* const* tri) {
  ResidentMesh& r = m->res;
  int coop = 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, m->device) != cudaSuccess || !coop) {
    cudaGetLastError();
    return;
  }
  const int n = nscen(m);
  const size_t w = word(m);
  const bool f64 = w == 8;
  // One part per SM (two or three smaller ones measured the same to 40 %
  // slower), none smaller than kMinPart: below that more parts only add
  // exchange (FP32 step of 1,058 cells: 2.2 us with parts of 16, 1.9 with 64;
  // FP64: 6.7 us with 16, 6.6 with 32, 6.9 with 64).
  const int64_t slots = m->sms, kMinPart = f64 ? 32 : 64;
  if (n > slots) return;
  int64_t per = std::max<int64_t>(kMinPart, (m->T + slots - 1) / slots);
  std::vector<int32_t> parts(n);
  for (;; ++per) {
    int64_t total = 0;
    for (int i = 0; i < n; ++i) {
      parts[i] = (int32_t)((m->scen[i].ncells + per - 1) / per);
      total += parts[i];
    }
    if (total <= slots) break;
  }
  std::vector<swe::ResidentParts> pt(n);
  std::vector<swe::ResBlock> blocks;
  int64_t cells = 0, halos = 0, recs = 0, npub = 0;
  int32_t cell_cap = 0, halo_cap = 0, rec_cap = 0;
  for (int i = 0; i < n; ++i) {
    if (!swe::build_resident_parts(hm[i], xy[i], tri[i], m->prm.order == SWE_ORDER_MORTON, parts[i],
                                   pt[i]))
      return;
    const int32_t block0 = (int32_t)blocks.size();
    for (int32_t b = 0; b < parts[i]; ++b) {
      swe::ResBlock k{};
      k.scen = i;
      k.cell0 = (int32_t)cells + pt[i].cell0[b];
      k.ncell = pt[i].cell0[b + 1] - pt[i].cell0[b];
      k.halo0 = (int32_t)halos + pt[i].halo0[b];
      k.nhalo = pt[i].halo0[b + 1] - pt[i].halo0[b];
      k.rec0 = (int32_t)recs + pt[i].rec0[b];
      k.nrec = pt[i].rec0[b + 1] - pt[i].rec0[b];
      k.block0 = block0;
      k.nblocks = parts[i];
      k.first = b == 0;
      blocks.push_back(k);
    }
    const int32_t c0 = (int32_t)m->scen[i].cell0, p0 = (int32_t)npub;
    for (int32_t& c : pt[i].cells) c += c0;
    for (int32_t& p : pt[i].pub)
      if (p >= 0) p += p0;
    for (int32_t& c : pt[i].halo) c += c0;
    for (int32_t& p : pt[i].halo_pub) p += p0;
    cells += (int64_t)pt[i].cells.size();
    halos += (int64_t)pt[i].halo.size();
    recs += (int64_t)pt[i].side.size();
    npub += pt[i].npub;
    cell_cap = std::max(cell_cap, pt[i].cell_cap);
    halo_cap = std::max(halo_cap, pt[i].halo_cap);
    rec_cap = std::max(rec_cap, pt[i].rec_cap);
  }
  r.layout = swe::make_res_layout((uint32_t)w, m->prm.compensated_depth != 0, (uint32_t)cell_cap,
                                  (uint32_t)halo_cap, (uint32_t)rec_cap);
  // Threads: one control warp, and enough others for the fewest even rounds
  // over the records. FP64: up to 12 warps, which fill the FP64 pipe (384
  // threads 30.1 us per step of 104,882 cells, 256 31.4, 512 31.3); FP32: as
  // many as the registers allow (249,498 cells: 992 threads 4.6 us, 512 5.1,
  // 256 6.5).
  const int max_warps =
      f64 ? 12 : (m->prm.compensated_depth ? swe::res_max_threads<float, true>()
                                           : swe::res_max_threads<float, false>()) / 32 - 1;
  const int chunks = (rec_cap + 31) / 32;
  const int rounds = (chunks + max_warps - 1) / max_warps;
  r.threads = 32 * ((chunks + rounds - 1) / rounds + 1);
  const int occ = occupancy_of(m, r.threads, r.layout.total);
  if ((int64_t)occ * m->sms < (int64_t)blocks.size()) return;

  // One blob, as it will lie on the device (resident_upload).
  auto add = [&](size_t bytes) {
    const size_t at = r.blob.size();
    r.blob.resize(at + align_up(bytes));
    return at;
  };
  r.at_blocks = add(sizeof(swe::ResBlock) * blocks.size());
  r.at_cells = add(4 * cells);
  r.at_pub = add(4 * cells);
  r.at_halo = add(4 * halos);
  r.at_halo_pub = add(4 * halos);
  r.at_rec = add((f64 ? 4 : 16) * recs);
  for (size_t& g : r.at_geo) g = add(f64 ? 8 * recs : 0);
  char* base = r.blob.data();
  std::memcpy(base + r.at_blocks, blocks.data(), sizeof(swe::ResBlock) * blocks.size());
  int64_t c = 0, h = 0, q = 0;
  for (const swe::ResidentParts& p : pt) {
    std::memcpy(base + r.at_cells + 4 * c, p.cells.data(), 4 * p.cells.size());
    std::memcpy(base + r.at_pub + 4 * c, p.pub.data(), 4 * p.pub.size());
    std::memcpy(base + r.at_halo + 4 * h, p.halo.data(), 4 * p.halo.size());
    std::memcpy(base + r.at_halo_pub + 4 * h, p.halo_pub.data(), 4 * p.halo_pub.size());
    if (f64) {
      std::memcpy(base + r.at_rec + 4 * q, p.side.data(), 4 * p.side.size());
      const std::vector<double>* g[3] = {&p.nx, &p.ny, &p.len};
      for (int k = 0; k < 3; ++k)
        std::memcpy(base + r.at_geo[k] + 8 * q, g[k]->data(), 8 * p.side.size());
    } else {
      uint32_t* rec = (uint32_t*)(base + r.at_rec) + 4 * q;
      for (size_t k = 0; k < p.side.size(); ++k) {
        const float f[3] = {(float)p.nx[k], (float)p.ny[k], (float)p.len[k]};
        rec[4 * k] = p.side[k];
        std::memcpy(rec + 4 * k + 1, f, sizeof f);
      }
    }
    c += (int64_t)p.cells.size();
    h += (int64_t)p.halo.size();
    q += (int64_t)p.side.size();
  }
  r.npub = (int32_t)npub;
  r.nblocks = (int32_t)blocks.size();
}

void resident_build(swe_mesh* m, const std::vector<swe::HostMesh>& hm, const double* const* xy,
                    const int32_t* const* tri) noexcept {
  m->res = ResidentMesh();
  try {
    build(m, hm, xy, tri);
  } catch (...) {  // no host memory: the mesh steps without its parts
    m->res = ResidentMesh();
  }
}

swe_status resident_upload(swe_mesh* m) {
  ResidentMesh& r = m->res;
  r.base = (char*)m->arena.take(r.blob.size());
  if (!r.base || cuda_failed(cudaMemcpyAsync(r.base, r.blob.data(), r.blob.size(),
                                             cudaMemcpyHostToDevice, m->stream)) ||
      cuda_failed(cudaStreamSynchronize(m->stream)))
    return SWE_ECUDA;
  std::vector<char>().swap(r.blob);
  return SWE_OK;
}

cudaError_t launch_resident(const swe_state* s, int64_t n, cudaStream_t st) {
  if (s->mesh->prm.precision == SWE_F64) return launch<double, false>(s, n, st);
  return s->hlo ? launch<float, true>(s, n, st) : launch<float, false>(s, n, st);
}

}  // namespace swe_host
