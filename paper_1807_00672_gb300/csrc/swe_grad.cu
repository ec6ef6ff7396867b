// Gradients through many steps (swe_grad_record / swe_grad, include/swe.h).
//
// swe_grad_record runs n steps forward on a state, as swe_run does, and
// keeps a tape: the dt of every step (held fixed for the derivative), the
// depths at the gauge cells after every step, and the state every K steps
// (checkpoints). The recorded steps write straight into the tape's buffers,
// the way a replay does: a segment's inner states into one of two rings (the
// last segment's into a buffer of their own), its end into the next
// checkpoint; the steps follow each other without copies or other launches
// between them (1.0M FP32 cells, K = 50: 27.1 us per recorded step when each
// was followed by a launch that noted its dt and gauges, and the last
// segment's by a copy; 21.3 now). swe_grad then runs the adjoint backwards
// through the steps: segment by segment, from the last checkpoint to the
// first. The inner states of the last three segments are still there from
// the recording; those of an earlier one are recomputed from its checkpoint
// with the forward kernel (the forward is deterministic, so the replay
// reproduces the recorded states bit for bit; the replay's dt is checked
// against the recorded one; the segment's last state is the next checkpoint,
// or the final state, and is not recomputed). The tiled adjoint kernel runs
// step by step, adding the gauge-loss seeds as it passes their steps. The
// replay of the next segment runs on a second stream while the current
// segment's adjoint steps run, each into its own ring of states. Memory:
// ceil(n / K) + 1 checkpoints, up to 3 (K - 1) inner states and two adjoint
// states. K = 1 keeps every state and replays nothing.
#include <algorithm>
#include <cmath>
#include <limits>
#include <numeric>
#include <vector>

#include "../../include/swe.h"
#include "swe_adjoint.cuh"
#include "mesh_build.h"
#include "swe_handles.cuh"
#include "swe_kernels.cuh"

using namespace swe_host;

namespace {

#define cuda_failed(call) swe_host::cuda_failed_at((call), #call, __FILE__, __LINE__)
#define CK(call)                              \
  do {                                        \
    if (cuda_failed(call)) return SWE_ECUDA;  \
  } while (0)

constexpr int kErrReplay = 8;  // a replayed step did not reproduce the recorded dt

// States of a tape, sb bytes each: checkpoint seg (U^{seg K}) at ck + seg sb,
// U^N behind the last one. Inner states U^{seg K + 1} .. of segment seg lie in
// ring seg % 2, so that the replay of the next segment (on the side stream)
// overlaps the adjoint steps of the current one, those of the last segment in
// `tail`.
struct TapeSlots {
  char *ck, *ring[2], *tail;
  int64_t N, K, nck;
  size_t sb;
  __host__ __device__ int64_t seg_len(int64_t seg) const {
    return (seg + 1) * K < N ? K : N - seg * K;
  }
  __host__ __device__ char* slot(int64_t seg, int64_t r) const {  // state U^{seg K + r}
    if (r == 0) return ck + seg * sb;
    if (r == seg_len(seg)) return ck + (seg + 1) * sb;
    if (seg == nck - 1) return tail + (r - 1) * sb;
    return ring[seg % 2] + (r - 1) * sb;
  }
  __host__ __device__ char* state(int64_t n) const {  // U^n
    if (n == 0) return ck;
    const int64_t seg = (n - 1) / K;
    return slot(seg, n - seg * K);
  }
};

// Gauge depths after steps k0 .. k1 - 1.
template <typename Real>
__global__ void __launch_bounds__(128)
    k_tape_gauges(TapeSlots s, int64_t k0, int64_t k1, const int32_t* cells, int G, double* gauge) {
  for (int64_t i = k0 * G + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < k1 * G;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = i / G;
    gauge[i] = (double)((const Real*)s.state(k + 1))[4 * (int64_t)cells[i - k * G]];
  }
}

// n interleaved cells: the state's current buffer to the tape's U^0, or the
// tape's newest state (steps0: the state's steps before the recording) back.
template <typename Real>
__global__ void __launch_bounds__(256)
    k_copy_state(const swe::Ctl* ctl, Real* b0, Real* b1, TapeSlots s, long long steps0, int to_tape,
                 int64_t n) {
  Real* own = ctl->cur ? b1 : b0;
  Real* tape = (Real*)s.state(to_tape ? 0 : ctl->steps - steps0);
  const Real* from = to_tape ? own : tape;
  Real* to = to_tape ? tape : own;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const swe::V4<Real> v = swe::ld4(from + 4 * i);
    swe::st4(to + 4 * i, v.x, v.y, v.z, v.w);
  }
}

// Caller cells -> internal cells, in place.
__global__ void k_internal_cells(const int32_t* iperm, int32_t* cells, int n) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
    cells[j] = iperm[cells[j]];
}

// Replay control word: buffer 0 current, the recorded dt, no end time.
__global__ void k_replay_begin(swe::Ctl* ctl, double dt, long long part0, long long nparts) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  swe::Ctl c{};
  c.t = 0.0;
  c.t_end = __longlong_as_double(0x7ff0000000000000ll);  // +inf
  c.dt = dt;
  c.dt_cfl = dt;
  c.part0 = part0;
  c.nparts = nparts;
  *ctl = c;
}

// The last replayed step must have used the recorded dt.
__global__ void k_replay_check(const swe::Ctl* ctl, double dt, int* err) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  if (ctl->dt_last != dt || ctl->err) atomicOr(err, kErrReplay | ctl->err);
}

// dL/dn = dL/d(g n^2) * 2 g n with n = sqrt(g n^2 / g) >= 0.
template <typename Real>
__global__ void k_finish_dn(const Real* dgn2, const Real* gn2, double g, Real* out, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = Real((double)dgn2[i] * 2.0 * sqrt(g * (double)gn2[i]));
}

// Programmatic dependent launch: a step's blocks fetch their first tiles'
// tape and mesh data while the previous adjoint step's last blocks finish,
// and wait for it (griddepcontrol.wait) before reading its output.
template <typename Real, int NT, int CPT>
void launch_adjoint_nt(const swe_mesh* m, const swe::DevMesh<Real>& dm, const swe::AdjArgs<Real>& a,
                       const swe::AdjLayout& L, int grid, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = L.total;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if constexpr (sizeof(Real) == 8) {
    if (a.split > 1) {
      cudaLaunchKernelEx(&cfg, swe::k_tiled_adjoint<Real, NT, 2, CPT, true>, dm, a, num_of(m), L);
      return;
    }
  }
  cudaLaunchKernelEx(&cfg, swe::k_tiled_adjoint<Real, NT, 2, CPT>, dm, a, num_of(m), L);
}

template <typename Real, int CPT>
void launch_adjoint_cpt(const swe_mesh* m, const swe::DevMesh<Real>& dm, const swe::AdjArgs<Real>& a,
                        const swe::AdjLayout& L, int grid, cudaStream_t st) {
  switch (m->tile / CPT) {
    case 32: launch_adjoint_nt<Real, 32, CPT>(m, dm, a, L, grid, st); break;
    case 64: launch_adjoint_nt<Real, 64, CPT>(m, dm, a, L, grid, st); break;
    case 128: launch_adjoint_nt<Real, 128, CPT>(m, dm, a, L, grid, st); break;
    default: launch_adjoint_nt<Real, 256, CPT>(m, dm, a, L, grid, st); break;
  }
}

// The adjoint runs on its own chunk table (one wave at its own occupancy).
template <typename Real>
void launch_adjoint(const swe_mesh* m, const swe::Chunk* chunks, int grid,
                    const swe::AdjArgs<Real>& a, const swe::AdjLayout& L, cudaStream_t st) {
  swe::DevMesh<Real> dm = dev_mesh<Real>(m);
  dm.chunks = chunks;
  if (m->cpt == 2) launch_adjoint_cpt<Real, 2>(m, dm, a, L, grid, st);
  else launch_adjoint_cpt<Real, 1>(m, dm, a, L, grid, st);
}

// Opts the adjoint kernel into its shared memory; resident blocks per SM.
template <typename Real, int NT, int CPT, bool Parts>
int adjoint_occupancy(const swe::AdjLayout& L) {
  auto k = swe::k_tiled_adjoint<Real, NT, 2, CPT, Parts>;
  // The limit is a property of the kernel, shared by every mesh that
  // launches it: set it to the device's largest opt-in size (not this
  // layout's), so that a later mesh with a smaller layout cannot lower it
  // below what an earlier one needs.
  cudaFuncAttributes fa{};
  if (cudaFuncGetAttributes(&fa, k) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const int cap = swe_host::smem_optin_bytes() - (int)fa.sharedSizeBytes;  // less its static part
  if (cap <= 0 || (int)L.total > cap ||
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, cap) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, NT, L.total) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

template <typename Real, int NT, int CPT>
int prepare_adjoint_nt(const swe::AdjLayout& L) {
  const int n = adjoint_occupancy<Real, NT, CPT, false>(L);
  if constexpr (sizeof(Real) == 8) return std::min(n, adjoint_occupancy<Real, NT, CPT, true>(L));
  return n;
}

template <typename Real, int CPT>
int prepare_adjoint_cpt(const swe_mesh* m, const swe::AdjLayout& L) {
  switch (m->tile / CPT) {
    case 32: return prepare_adjoint_nt<Real, 32, CPT>(L);
    case 64: return prepare_adjoint_nt<Real, 64, CPT>(L);
    case 128: return prepare_adjoint_nt<Real, 128, CPT>(L);
    default: return prepare_adjoint_nt<Real, 256, CPT>(L);
  }
}

template <typename Real>
int prepare_adjoint(const swe_mesh* m, const swe::AdjLayout& L) {
  return m->cpt == 2 ? prepare_adjoint_cpt<Real, 2>(m, L) : prepare_adjoint_cpt<Real, 1>(m, L);
}

// Parts per tile of the FP64 adjoint (k_tiled_adjoint): the least time on the
// busiest SM, in units of a tile's 23.5 us. As measured (256-cell tiles), a
// step costs 0.6 for its launch and latency, and a part its share of the tile
// and 0.15 for what every part does for the whole tile. us per step, whole
// tiles and parts: 400 cells (2 tiles, eighths) 32.0 and 20.5, 3,600 (15,
// eighths) 37.5 and 20.8, 10,000 (40, thirds) 37.6 and 26.5; 22,500 (88) 37.8
// and 38.3 in thirds, 79,806 (313) 83.2 and 84.0 in halves: whole. FP32 tiles
// stay whole (10,000 cells: 9.2 us per step, most of it the launch).
int adjoint_split(int64_t tiles, int sms, int tile_cells) {
  int best = 1;
  double least = 0.6 + (double)((tiles + sms - 1) / sms);
  for (int s = 2; s <= 8 && s <= tile_cells / 32; ++s) {
    const double part = (double)((tile_cells / 32 + s - 1) / s) * 32 / tile_cells;
    const double cost = 0.6 + (double)((tiles * s + sms - 1) / sms) * (part + 0.15);
    if (cost < 0.95 * least) {
      least = cost;
      best = s;
    }
  }
  return best;
}

int grid_for(int64_t n, int cap) {
  int64_t g = (n + 255) / 256;
  return (int)std::max<int64_t>(1, std::min<int64_t>(g, cap));
}

}  // namespace

struct swe_tape {
  swe_mesh* mesh = nullptr;
  cudaStream_t stream = nullptr;
  int64_t N = 0, K = 0, nck = 0;
  int G = 0;
  size_t w = 8;
  int64_t Tp = 0, T = 0;
  Arena arena;
  TapeSlots slots{};
  // The segment whose inner states each ring holds (-1: none): the recording
  // leaves the last but one and two there, a replay the one it recomputed.
  int64_t holds[2] = {-1, -1};
  cudaStream_t side = nullptr;
  cudaEvent_t replayed[2] = {nullptr, nullptr}, consumed[2] = {nullptr, nullptr};
  char* lam[2] = {nullptr, nullptr};
  void* gn2 = nullptr;   // copy of the state's g n^2
  void* dgn2 = nullptr;
  void* scratch = nullptr;
  double* stage = nullptr;  // T doubles
  double* dts_dev = nullptr;
  double* gauge_dev = nullptr;
  double* gseed_dev = nullptr;
  int32_t* gcells = nullptr;
  swe::GaugeSeeds gauges{};  // gseed_dev by distinct gauge cell
  swe::Chunk* chunks = nullptr;  // work of the adjoint kernel's blocks, in units of
  int64_t nchunks = 0;           // 1 / split tiles
  int split = 1;
  swe::Ctl* ctl = nullptr;      // two replay control words (one per ring)
  double* partial = nullptr;    // two arrays of per-chunk mass partials
  int* err = nullptr;
  std::vector<double> dts;
  swe::AdjLayout adj{};
  float record_ms = 0.f, grad_ms = 0.f;
  cudaEvent_t ev[2] = {nullptr, nullptr};

  size_t state_bytes() const { return 4 * w * (size_t)Tp; }
  int64_t seg_len(int64_t seg) const { return slots.seg_len(seg); }
  void* slot(int64_t seg, int64_t r) const { return slots.slot(seg, r); }
};

namespace {

void free_tape(swe_tape* t) {
  if (t->mesh && t->stream) cudaStreamSynchronize(t->stream);
  if (t->side) cudaStreamSynchronize(t->side);
  for (auto& e : t->ev)
    if (e) cudaEventDestroy(e);
  for (int i = 0; i < 2; ++i) {
    if (t->replayed[i]) cudaEventDestroy(t->replayed[i]);
    if (t->consumed[i]) cudaEventDestroy(t->consumed[i]);
  }
  if (t->side) cudaStreamDestroy(t->side);
  arena_free(t->arena);
  swe_mesh* m = t->mesh;
  delete t;
  if (m) release_mesh(m);
}

// Step r of segment seg on the tape's buffers: the current buffer (number
// cur when r is even) is its input slot, the other one its output slot.
template <typename Real>
void set_buffers(const swe_tape* t, int64_t seg, int64_t r, int cur, swe::DevState<Real>& d) {
  Real* in = (Real*)t->slot(seg, r);
  Real* out = (Real*)t->slot(seg, r + 1);
  for (int b = 0; b < 2; ++b) {
    Real* p = b == cur ? in : out;
    d.h[b] = p;
    d.hu[b] = p + 1;
    d.hv[b] = p + 2;
  }
  d.stride = 4;
  d.z = in + 3;
}

// Device state view of replay step r of segment seg (the replay control word
// starts with buffer 0 current).
template <typename Real>
swe::DevState<Real> replay_state(const swe_tape* t, int64_t seg, int64_t r) {
  swe::DevState<Real> d{};
  set_buffers(t, seg, r, (int)(r % 2), d);
  d.gn2 = (const Real*)t->gn2;
  d.partial = t->partial + (seg % 2) * std::max<int64_t>(1, t->mesh->nchunks);
  d.ctl = t->ctl + seg % 2;
  return d;
}

template <typename Real>
swe_status record_t(swe_state* s, swe_tape* t) {
  swe_mesh* m = s->mesh;
  cudaStream_t st = m->stream;
  const int gs = grid_for(t->Tp, m->sms * 8);
  Real* b0 = (Real*)s->h[0];
  Real* b1 = (Real*)s->h[1];
  const long long steps0 = s->host_ctl[0].steps;
  const int cur0 = s->host_ctl[0].cur;
  k_copy_state<Real><<<gs, 256, 0, st>>>(s->ctl, b0, b1, t->slots, steps0, 1, t->Tp);
  CK(cudaMemcpyAsync(t->gn2, s->gn2, t->w * t->Tp, cudaMemcpyDeviceToDevice, st));
  CK(cudaEventRecord(t->ev[0], st));
  auto gauges = [&](int64_t k0, int64_t k1) {
    if (t->G > 0)
      k_tape_gauges<Real><<<(int)std::min<int64_t>(((k1 - k0) * t->G + 127) / 128, m->sms * 8), 128, 0,
                            st>>>(t->slots, k0, k1, t->gcells, t->G, t->gauge_dev);
  };
  int64_t noted = 0;  // steps whose gauges are taken
  for (int64_t k = 0; k < t->N; ++k) {
    const int64_t seg = k / t->K;
    // a ring is about to be used again: take the gauges of the steps so far
    if (k == seg * t->K && t->K > 1 && seg >= 2 && seg < t->nck - 1) {
      gauges(noted, k);
      noted = k;
    }
    swe::DevState<Real> d = dev_state<Real>(s);
    set_buffers(t, seg, k - seg * t->K, (int)((cur0 + k) % 2), d);
    d.dt_log = t->dts_dev + k;
    launch_forward(m, d, st);
  }
  gauges(noted, t->N);
  k_copy_state<Real><<<gs, 256, 0, st>>>(s->ctl, b0, b1, t->slots, steps0, 0, t->Tp);
  CK(cudaEventRecord(t->ev[1], st));
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(st));
  CK(cudaEventElapsedTime(&t->record_ms, t->ev[0], t->ev[1]));
  for (int64_t seg = std::max<int64_t>(0, t->nck - 3); seg < t->nck - 1; ++seg) t->holds[seg % 2] = seg;
  return SWE_OK;
}

// Recomputes the inner states U^{j0+1} .. U^{j1-1} of segment seg into its
// ring, on stream st.
template <typename Real>
void replay_segment(swe_tape* t, int64_t seg, cudaStream_t st) {
  const swe_mesh* m = t->mesh;
  const Scenario& sc = m->scen[0];
  const int64_t j0 = seg * t->K, j1 = std::min(t->N, j0 + t->K);
  if (j1 - j0 <= 1) return;
  swe::Ctl* ctl = t->ctl + seg % 2;
  k_replay_begin<<<1, 1, 0, st>>>(ctl, t->dts[j0], sc.chunk0, sc.nchunks);
  for (int64_t r = 0; r + 1 < j1 - j0; ++r) launch_forward(m, replay_state<Real>(t, seg, r), st);
  k_replay_check<<<1, 1, 0, st>>>(ctl, t->dts[j1 - 2], t->err);
}

template <typename Real>
swe_status grad_t(swe_tape* t, bool seeds_gauge, int* lam_cur) {
  swe_mesh* m = t->mesh;
  cudaStream_t st = m->stream;
  int cur = 0;
  if (seeds_gauge)
    swe::k_inject_gauges<Real><<<1, 128, 0, st>>>((Real*)t->lam[cur], t->gauges, t->N - 1);
  swe::k_adjoint_start<Real><<<grid_for(t->Tp, m->sms * 8), 256, 0, st>>>(
      (const Real*)t->slot(t->nck - 1, t->seg_len(t->nck - 1)), (Real*)t->lam[cur], (const Real*)t->gn2,
      (Real*)t->dgn2, Real(t->dts[t->N - 1]), num_of(m), t->Tp);
  // Replays run one segment ahead on the side stream: segment seg - 1's
  // replay (ring (seg - 1) % 2) overlaps segment seg's adjoint steps; it
  // first waits for the adjoint of segment seg + 1, the ring's last user.
  // The last segment needs none (its states are in the tail), nor does one
  // whose states its ring still holds.
  CK(cudaEventRecord(t->consumed[0], st));
  CK(cudaEventRecord(t->consumed[1], st));
  for (int64_t seg = t->nck - 1; seg >= 0; --seg) {
    const int64_t j0 = seg * t->K, j1 = std::min(t->N, j0 + t->K);
    if (seg >= 1 && t->holds[(seg - 1) % 2] != seg - 1) {
      CK(cudaStreamWaitEvent(t->side, t->consumed[(seg - 1) % 2], 0));
      replay_segment<Real>(t, seg - 1, t->side);
      CK(cudaEventRecord(t->replayed[(seg - 1) % 2], t->side));
      t->holds[(seg - 1) % 2] = seg - 1;
    }
    if (seg < t->nck - 1) CK(cudaStreamWaitEvent(st, t->replayed[seg % 2], 0));
    for (int64_t j = j1 - 1; j >= j0; --j) {
      const int64_t r = j - j0;
      swe::AdjArgs<Real> a{};
      a.un = (const Real*)t->slot(seg, r);
      a.mu_in = (const Real*)t->lam[cur];
      a.mu_out = (Real*)t->lam[cur ^ 1];
      a.gn2 = (const Real*)t->gn2;
      a.dgn2 = (Real*)t->dgn2;
      a.dt = Real(t->dts[j]);
      a.dt_prev = j > 0 ? Real(t->dts[j - 1]) : Real(0);
      a.last = j == 0;
      a.split = t->split;
      a.err = t->err;
      a.gauges = t->gauges;
      a.gstep = (seeds_gauge && j >= 1) ? (long long)(j - 1) : -1ll;  // lambda^j gets dL/dh^j
      launch_adjoint<Real>(m, t->chunks, (int)t->nchunks, a, t->adj, st);
      cur ^= 1;
    }
    CK(cudaEventRecord(t->consumed[seg % 2], st));
  }
  CK(cudaGetLastError());
  *lam_cur = cur;
  return SWE_OK;
}

swe_status grad_record(swe_state* s, int64_t n_steps, int64_t checkpoint_every,
                       const int32_t* gauge_cells, int32_t n_gauges, double* gauge_h,
                       swe_tape** out) {
  if (!out) return SWE_EINVAL;
  *out = nullptr;
  if (!s || n_steps <= 0 || checkpoint_every <= 0 || n_gauges < 0 || (n_gauges > 0 && !gauge_cells))
    return SWE_EINVAL;
  swe_mesh* m = s->mesh;
  if (m->kernel != SWE_KERNEL_TILED || nscen(m) != 1 || m->ghosts || m->tile / m->cpt > 256 ||
      m->prm.compensated_depth)
    return SWE_ESTATE;
  for (int j = 0; j < n_gauges; ++j)
    if (gauge_cells[j] < 0 || gauge_cells[j] >= m->T) return SWE_EINVAL;
  swe_status st = read_ctl(s);
  if (st != SWE_OK) return st;
  if (s->host_ctl[0].err) return SWE_ESTATE;

  swe_tape* t = new swe_tape();
  t->mesh = m;
  retain_mesh(m);
  swe::OnThrow on_throw([t] { free_tape(t); });
  t->stream = m->stream;
  t->N = n_steps;
  t->K = std::min(checkpoint_every, n_steps);
  t->nck = (n_steps + t->K - 1) / t->K;
  t->G = n_gauges;
  t->w = m->prm.precision == SWE_F64 ? 8 : 4;
  t->Tp = m->Tp;
  t->T = m->T;
  const int geo_arrays = (m->prm.precision == SWE_F64) ? 3 : 2;
  t->adj = swe::make_adj_layout((uint32_t)t->w, (uint32_t)geo_arrays, (uint32_t)m->tile, 2u,
                                (uint32_t)m->layout.rec_cap, (uint32_t)m->layout.halo_cap);
  const int occ = m->prm.precision == SWE_F64 ? prepare_adjoint<double>(m, t->adj)
                                              : prepare_adjoint<float>(m, t->adj);
  if (occ < 1) {
    g_cuda_msg = "adjoint kernel layout does not fit in shared memory";
    free_tape(t);
    return SWE_ECUDA;
  }
  // Adjoint chunk table: one wave of resident blocks, one chunk for every
  // block slot (chunks of equal tile counts leave slots empty: 313 FP64 tiles
  // on 304 slots made 157 chunks of 2, some SMs with 4 tiles and others with 2).
  std::vector<swe::Chunk> chunks;
  {
    const Scenario& sc = m->scen[0];
    const int64_t resident = (int64_t)m->sms * occ;
    t->split = m->prm.precision == SWE_F64 ? adjoint_split(sc.ntiles, m->sms, m->tile) : 1;
    const int64_t units = sc.ntiles * t->split;
    const int64_t nc = std::min<int64_t>(units, resident);
    for (int64_t r = 0; r < nc; ++r) {
      swe::Chunk c{};
      c.scen = 0;
      c.tile0 = (int32_t)(sc.tile0 * t->split + r);
      c.ntiles = (int32_t)((units - r + nc - 1) / nc);
      c.stride = (int32_t)nc;
      c.part = (int32_t)r;
      c.cell_end = (int32_t)(sc.cell0 + sc.ncells);
      chunks.push_back(c);
    }
    t->nchunks = nc;
  }
  const size_t sb = t->state_bytes();
  Layout L;
  const size_t inner = sb * (size_t)(t->K - 1);  // a segment's inner states
  const int rings = (int)std::min<int64_t>(2, t->nck - 1);
  L.add(sb * (t->nck + 1));
  for (int i = 0; i <= rings; ++i) L.add(inner);  // the rings and the tail
  L.add(sb); L.add(sb);
  L.add(t->w * t->Tp);  // gn2
  L.add(t->w * t->Tp);  // dgn2
  L.add(t->w * t->Tp);  // scratch
  L.add(8 * t->T);      // stage
  L.add(8 * t->N);      // dts
  L.add(8 * t->N * std::max(1, t->G));  // gauge depths
  L.add(8 * t->N * std::max(1, t->G));  // gauge seeds
  L.add(4 * std::max(1, t->G));
  L.add(4 * (3 * (size_t)t->G + 1 + (size_t)m->ntiles + 1));  // gauges by cell and tile
  L.add(sizeof(swe::Chunk) * chunks.size());
  L.add(2 * sizeof(swe::Ctl));
  L.add(2 * 8 * (size_t)std::max<int64_t>(1, m->nchunks));
  L.add(sizeof(int));
  if (!arena_alloc(t->arena, L.total)) {
    free_tape(t);
    return SWE_ENOMEM;
  }
  t->slots.N = t->N;
  t->slots.K = t->K;
  t->slots.nck = t->nck;
  t->slots.sb = sb;
  t->slots.ck = (char*)t->arena.take(sb * (t->nck + 1));
  for (int i = 0; i < rings; ++i) t->slots.ring[i] = (char*)t->arena.take(inner);
  t->slots.tail = (char*)t->arena.take(inner);
  t->lam[0] = (char*)t->arena.take(sb);
  t->lam[1] = (char*)t->arena.take(sb);
  t->gn2 = t->arena.take(t->w * t->Tp);
  t->dgn2 = t->arena.take(t->w * t->Tp);
  t->scratch = t->arena.take(t->w * t->Tp);
  t->stage = (double*)t->arena.take(8 * t->T);
  t->dts_dev = (double*)t->arena.take(8 * t->N);
  t->gauge_dev = (double*)t->arena.take(8 * t->N * std::max(1, t->G));
  t->gseed_dev = (double*)t->arena.take(8 * t->N * std::max(1, t->G));
  t->gcells = (int32_t*)t->arena.take(4 * std::max(1, t->G));
  int32_t* by_cell = (int32_t*)t->arena.take(4 * (3 * (size_t)t->G + 1 + (size_t)m->ntiles + 1));
  t->chunks = (swe::Chunk*)t->arena.take(sizeof(swe::Chunk) * chunks.size());
  t->ctl = (swe::Ctl*)t->arena.take(2 * sizeof(swe::Ctl));
  t->partial = (double*)t->arena.take(2 * 8 * (size_t)std::max<int64_t>(1, m->nchunks));
  t->err = (int*)t->arena.take(sizeof(int));
  if (t->arena.overflow) {
    g_cuda_msg = "tape arena layout";
    free_tape(t);
    return SWE_ECUDA;
  }
  auto fail = [&](swe_status r) { free_tape(t); return r; };
  // The steps write every cell of a state; its padding (read by copies of
  // whole tiles, never used) is set once.
  auto zero_padding = [&](char* states, int64_t n) {
    const size_t used = 4 * t->w * (size_t)t->T;
    return n > 0 && sb > used &&
           cuda_failed(cudaMemset2DAsync(states + used, sb, 0, sb - used, (size_t)n, m->stream));
  };
  if (zero_padding(t->slots.ck, t->nck + 1) || zero_padding(t->slots.tail, t->K - 1) ||
      (rings > 0 && zero_padding(t->slots.ring[0], t->K - 1)) ||
      (rings > 1 && zero_padding(t->slots.ring[1], t->K - 1)) ||
      cuda_failed(cudaMemsetAsync(t->lam[0], 0, t->arena.base + L.total - t->lam[0], m->stream)) ||
      cuda_failed(cudaEventCreate(&t->ev[0])) || cuda_failed(cudaEventCreate(&t->ev[1])) ||
      cuda_failed(cudaStreamCreateWithFlags(&t->side, cudaStreamNonBlocking)))
    return fail(SWE_ECUDA);
  for (int i = 0; i < 2; ++i)
    if (cuda_failed(cudaEventCreateWithFlags(&t->replayed[i], cudaEventDisableTiming)) ||
        cuda_failed(cudaEventCreateWithFlags(&t->consumed[i], cudaEventDisableTiming)))
      return fail(SWE_ECUDA);
  if (cuda_failed(cudaMemcpyAsync(t->chunks, chunks.data(), sizeof(swe::Chunk) * chunks.size(),
                                  cudaMemcpyHostToDevice, m->stream)) ||
      cuda_failed(cudaStreamSynchronize(m->stream)))
    return fail(SWE_ECUDA);
  // gauge cells in internal order
  if (t->G > 0) {
    std::vector<int32_t> gi(t->G);
    if (cuda_failed(cudaMemcpyAsync(t->gcells, gauge_cells, 4 * t->G, cudaMemcpyHostToDevice, m->stream)))
      return fail(SWE_ECUDA);
    k_internal_cells<<<grid_for(t->G, m->sms), 256, 0, m->stream>>>(m->iperm, t->gcells, t->G);
    if (cuda_failed(cudaMemcpyAsync(gi.data(), t->gcells, 4 * t->G, cudaMemcpyDeviceToHost, m->stream)) ||
        cuda_failed(cudaStreamSynchronize(m->stream)))
      return fail(SWE_ECUDA);
    // the distinct cells, and each one's gauges in ascending order
    std::vector<int32_t> cells, first, index(t->G);
    std::iota(index.begin(), index.end(), 0);
    std::stable_sort(index.begin(), index.end(), [&](int32_t a, int32_t b) { return gi[a] < gi[b]; });
    for (int q = 0; q < t->G; ++q)
      if (q == 0 || gi[index[q]] != cells.back()) {
        cells.push_back(gi[index[q]]);
        first.push_back(q);
      }
    first.push_back(t->G);
    const int nc = (int)cells.size();
    std::vector<int32_t> tiles(m->ntiles + 1, 0);  // where each tile's cells start
    for (int32_t c : cells) tiles[c / m->tile + 1] += 1;
    for (int64_t k = 0; k < m->ntiles; ++k) tiles[k + 1] += tiles[k];
    t->gauges = {by_cell, by_cell + t->G, by_cell + 2 * t->G + 1, by_cell + 3 * t->G + 1, t->gseed_dev,
                 t->G, nc};
    auto put = [&](const int32_t* to, const std::vector<int32_t>& v) {
      return cuda_failed(cudaMemcpyAsync((void*)to, v.data(), 4 * v.size(), cudaMemcpyHostToDevice,
                                         m->stream));
    };
    if (put(t->gauges.cells, cells) || put(t->gauges.first, first) || put(t->gauges.index, index) ||
        put(t->gauges.tile_first, tiles) ||
        cuda_failed(cudaStreamSynchronize(m->stream)))
      return fail(SWE_ECUDA);
  }
  const int64_t steps0 = s->host_ctl[0].steps;
  st = make_open_ended(s);  // end time +inf: every step takes its CFL dt
  if (st != SWE_OK) return fail(st);
  st = m->prm.precision == SWE_F64 ? record_t<double>(s, t) : record_t<float>(s, t);
  if (st != SWE_OK) return fail(st);
  st = read_ctl(s);
  if (st != SWE_OK) return fail(st);
  if (s->host_ctl[0].err) {
    const int e = s->host_ctl[0].err;
    free_tape(t);
    return (e & swe::kErrTimeout) ? SWE_ETIMEOUT : (e & swe::kErrNan) ? SWE_ENAN : SWE_EDRY;
  }
  if (s->host_ctl[0].steps - steps0 != t->N) return fail(SWE_ESTATE);
  t->dts.resize(t->N);
  if (cuda_failed(cudaMemcpyAsync(t->dts.data(), t->dts_dev, 8 * t->N, cudaMemcpyDeviceToHost, m->stream)) ||
      (gauge_h && t->G > 0 &&
       cuda_failed(cudaMemcpyAsync(gauge_h, t->gauge_dev, 8 * t->N * t->G, cudaMemcpyDeviceToHost, m->stream))) ||
      cuda_failed(cudaStreamSynchronize(m->stream)))
    return fail(SWE_ECUDA);
  *out = t;
  return SWE_OK;
}


// swe_grad and swe_grad_device: seeds and outputs in host memory, or
// (on_device) in device memory ordered on caller_stream.
swe_status grad(swe_tape* t, const double* g_h, const double* g_hu, const double* g_hv,
                const double* g_gauge, double* d_h0, double* d_hu0, double* d_hv0, double* d_z,
                double* d_n, bool on_device, void* caller_stream) {
  if (!t) return SWE_EINVAL;
  swe_mesh* m = t->mesh;
  cudaStream_t st = m->stream;
  const size_t sb = t->state_bytes();
  if (on_device && caller_stream && (cudaStream_t)caller_stream != st) {
    // the seeds were written, and the outputs may still be read, on the
    // caller's stream
    cudaEvent_t ev = nullptr;
    CK(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    cudaError_t e = cudaEventRecord(ev, (cudaStream_t)caller_stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ev, 0);
    cudaEventDestroy(ev);
    CK(e);
  }
  const cudaMemcpyKind in_kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  CK(cudaMemsetAsync(t->lam[0], 0, sb, st));
  CK(cudaMemsetAsync(t->lam[1], 0, sb, st));
  CK(cudaMemsetAsync(t->err, 0, sizeof(int), st));
  const double* seeds[3] = {g_h, g_hu, g_hv};
  for (int c = 0; c < 3; ++c) {
    if (!seeds[c]) continue;
    const double* from = seeds[c];
    if (!on_device) {
      CK(cudaMemcpyAsync(t->stage, seeds[c], 8 * t->T, cudaMemcpyHostToDevice, st));
      from = t->stage;
    }
    gather_any(m, from, t->lam[0] + c * t->w, 4);
  }
  const bool gseed = g_gauge && t->G > 0;
  if (gseed) CK(cudaMemcpyAsync(t->gseed_dev, g_gauge, 8 * t->N * t->G, in_kind, st));
  CK(cudaEventRecord(t->ev[0], st));
  int cur = 0;
  swe_status r = m->prm.precision == SWE_F64 ? grad_t<double>(t, gseed, &cur)
                                             : grad_t<float>(t, gseed, &cur);
  if (r != SWE_OK) return r;
  CK(cudaEventRecord(t->ev[1], st));
  double* outs[4] = {d_h0, d_hu0, d_hv0, d_z};
  for (int c = 0; c < 4; ++c) {
    if (!outs[c]) continue;
    if (on_device) {
      scatter_any(m, t->lam[cur] + c * t->w, outs[c], 4);
      continue;
    }
    scatter_any(m, t->lam[cur] + c * t->w, t->stage, 4);
    CK(cudaMemcpyAsync(outs[c], t->stage, 8 * t->T, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
  }
  if (d_n) {
    const int gs = grid_for(t->Tp, m->sms * 8);
    if (m->prm.precision == SWE_F64)
      k_finish_dn<double><<<gs, 256, 0, st>>>((const double*)t->dgn2, (const double*)t->gn2,
                                              m->prm.g, (double*)t->scratch, t->Tp);
    else
      k_finish_dn<float><<<gs, 256, 0, st>>>((const float*)t->dgn2, (const float*)t->gn2, m->prm.g,
                                             (float*)t->scratch, t->Tp);
    if (on_device) {
      scatter_any(m, t->scratch, d_n, 1);
    } else {
      scatter_any(m, t->scratch, t->stage, 1);
      CK(cudaMemcpyAsync(d_n, t->stage, 8 * t->T, cudaMemcpyDeviceToHost, st));
    }
  }
  int err = 0;
  CK(cudaMemcpyAsync(&err, t->err, sizeof(int), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  CK(cudaGetLastError());
  CK(cudaEventElapsedTime(&t->grad_ms, t->ev[0], t->ev[1]));
  if (err) t->holds[0] = t->holds[1] = -1;  // no ring to rely on
  if (err & swe::kErrTimeout) return SWE_ETIMEOUT;
  if (err) return SWE_ESTATE;  // the replay did not reproduce the recorded steps
  return SWE_OK;
}

}  // namespace

extern "C" {

swe_status swe_grad_record(swe_state* s, int64_t n_steps, int64_t checkpoint_every,
                           const int32_t* gauge_cells, int32_t n_gauges, double* gauge_h,
                           swe_tape** out) {
  if (out) *out = nullptr;
  return swe::guarded(
      [&] { return grad_record(s, n_steps, checkpoint_every, gauge_cells, n_gauges, gauge_h, out); });
}

swe_status swe_grad(swe_tape* t, const double* g_h, const double* g_hu, const double* g_hv,
                    const double* g_gauge, double* d_h0, double* d_hu0, double* d_hv0, double* d_z,
                    double* d_n) {
  return grad(t, g_h, g_hu, g_hv, g_gauge, d_h0, d_hu0, d_hv0, d_z, d_n, false, nullptr);
}

swe_status swe_grad_device(swe_tape* t, const double* g_h, const double* g_hu, const double* g_hv,
                           const double* g_gauge, double* d_h0, double* d_hu0, double* d_hv0,
                           double* d_z, double* d_n, void* cuda_stream) {
  return grad(t, g_h, g_hu, g_hv, g_gauge, d_h0, d_hu0, d_hv0, d_z, d_n, true, cuda_stream);
}

swe_status swe_tape_gauges_device(const swe_tape* t, double* gauge_h, void* cuda_stream) {
  if (!t || (!gauge_h && t->G > 0)) return SWE_EINVAL;
  if (t->G == 0) return SWE_OK;
  cudaStream_t st = t->mesh->stream;
  if (cuda_stream && (cudaStream_t)cuda_stream != st) {
    cudaEvent_t ev = nullptr;
    CK(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    cudaError_t e = cudaEventRecord(ev, (cudaStream_t)cuda_stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ev, 0);
    cudaEventDestroy(ev);
    CK(e);
  }
  CK(cudaMemcpyAsync(gauge_h, t->gauge_dev, 8 * t->N * t->G, cudaMemcpyDeviceToDevice, st));
  CK(cudaStreamSynchronize(st));
  return SWE_OK;
}

swe_status swe_tape_info(const swe_tape* t, double* info) {
  if (!t || !info) return SWE_EINVAL;
  info[0] = (double)t->N;
  info[1] = (double)t->K;
  info[2] = (double)t->record_ms;
  info[3] = (double)t->grad_ms;
  info[4] = (double)t->arena.size;
  return SWE_OK;
}

void swe_tape_destroy(swe_tape* t) {
  if (!t) return;
  free_tape(t);
}

}  // extern "C"
