// Resident step kernel: several explicit steps of a small mesh in one launch
// (Sec. 2.2 of Zaoui's paper, the arithmetic of k_tiled_step).
//
// A mesh whose cells, face records and face slots fit in the shared memory
// of the whole chip needs no HBM or L2 traffic between steps, and at that
// size a step launched by itself is bound by latency: the launch, the first
// copies, the hand-over of the control word. Here each block keeps one part
// of the mesh (consecutive cells of the Morton order) in its shared memory
// for all the steps of a call, and the blocks of one scenario exchange, per
// step, only
//   - the cells that another block's faces read, published as 16-byte words
//     that carry their values and the step's epoch together: a reader polls
//     the word itself, so neither a fence nor a flag is needed;
//   - one 16-byte slot per block with its largest CFL rate: every block reads
//     all slots of its scenario and forms the next dt, whose latency hides
//     behind the faces (only the cell updates need dt). (A copy of the rate
//     written to each reader instead of one slot that all poll: 2.5 against
//     2.3 us per FP32 step of 10,082 cells.)
// The grid is launched cooperatively (all blocks resident at once); every
// poll is bounded and latches kErrTimeout when it gives up.
//
// Reuse of the exchange words: the words of epochs e and e + 2 share memory.
// A block publishes epoch e + 2 only after it has read every slot of epoch
// e + 1, and a block writes its slot of epoch e + 1 only after its faces have
// read every word of epoch e and its control warp every slot of epoch e.
// Epochs grow over the life of a state (Ctl resets do not touch them): every
// launch advances the epoch past every word it could publish, whether it
// steps, stops or gives up (pass_entry), so no word of an earlier launch can
// be taken for a new one.
//
// A block that gives up may do so, and set the stop flag, before others have
// started: one thread of each block reads the flag and the epoch, so a block
// goes on or leaves as a whole. A launch in which a block gave up cannot end
// well for the scenario (its rate never comes), whoever still joined it.
#pragma once

#include "swe_kernels.cuh"

namespace swe {

// One block's part. Offsets into the concatenated plan arrays.
struct ResBlock {
  int32_t scen, cell0, ncell, halo0, nhalo, rec0, nrec;
  int32_t block0, nblocks;  // the scenario's blocks
  int32_t first;          // 1: this block writes the scenario's control word
};

template <typename Real>
struct ResPlan {
  const ResBlock* blocks;
  const int32_t* cells;     // internal index of each part's cells
  const int32_t* pub;       // publication number of the cell, or -1
  const int32_t* halo;      // internal index of each part's halo cells
  const int32_t* halo_pub;  // and their publication numbers
  const uint32_t* side;     // FP64 records: side codes and geometry arrays
  const Real* nx;
  const Real* ny;
  const Real* len;
  const int4* rec;          // FP32 records {side codes, nx, ny, l}
  unsigned char* xbuf;      // [2][npub] published cells (kPubBytes each)
  unsigned char* slots;     // [2][blocks] 16-byte rate slots
  uint32_t* epoch;          // per scenario: last epoch of the latest launch
  int32_t npub;
};

// Side code: face k of the part's cell idx as k << 14 | idx; k = 3 names the
// halo cell idx; 0xffff a wall. A record holds side A's code in the high
// half, side B's in the low half.
constexpr uint32_t kResWall = 0xffffu;

template <typename Real>
__host__ __device__ constexpr int pub_bytes() { return sizeof(Real) == 4 ? 16 : 32; }

// Shared-memory plan (offsets in bytes), from the largest part.
struct ResLayout {
  uint32_t ncs;  // slot stride between faces k, in slots
  uint32_t off_rec, off_nx, off_ny, off_len, off_sq, off_slots, off_ra, off_irp, off_gn2, off_lo,
      off_pub, off_hz, off_hpub, total;
};

inline ResLayout make_res_layout(uint32_t w, bool with_lo, uint32_t cells, uint32_t halos,
                                 uint32_t recs) {
  auto a16 = [](uint32_t x) { return (x + 15u) & ~15u; };
  ResLayout L{};
  uint32_t o = a16(cells * 4 * w);  // cells (h, hu, hv, z), FP64 (h, u, v, z), at 0
  L.ncs = cells + (w == 4 ? 3u : 1u);
  L.off_rec = o; o += a16(recs * (w == 4 ? 16u : 4u));
  if (w == 8) {
    L.off_nx = o; o += a16(recs * 8);
    L.off_ny = o; o += a16(recs * 8);
    L.off_len = o; o += a16(recs * 8);
    L.off_sq = o; o += a16(cells * 16);  // (hu, hv)
  }
  L.off_slots = o; o += a16(3 * L.ncs * (w == 4 ? 16u : 24u));
  L.off_ra = o; o += a16(cells * w);
  L.off_irp = o; o += a16(cells * w);
  L.off_gn2 = o; o += a16(cells * w);
  L.off_lo = o; o += with_lo ? a16(cells * 4) : 0u;
  L.off_pub = o; o += a16(cells * 4);
  L.off_hz = o; o += a16(halos * w);
  L.off_hpub = o; o += a16(halos * 4);
  L.total = o;
  return L;
}

// 16-byte words read and written as one access at GPU scope.
__device__ __forceinline__ void st_word(void* p, unsigned long long a, unsigned long long b) {
  asm volatile(
      "{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n}" ::"l"(p),
      "l"(a), "l"(b)
      : "memory");
}
__device__ __forceinline__ void ld_word(const void* p, unsigned long long& a, unsigned long long& b) {
  asm volatile(
      "{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n}"
      : "=l"(a), "=l"(b)
      : "l"(p)
      : "memory");
}

// Whether a block of the scenario has given up.
__device__ __forceinline__ bool timed_out(const Ctl* ctl) {
  return *(const volatile int*)&ctl->err & kErrTimeout;
}

// One thread of each block calls this once the block has read the epoch of
// the launch. The last of the scenario's nblocks blocks advances it to `next`,
// which nothing but the next launch reads.
__device__ __forceinline__ void pass_entry(Ctl* ctl, uint32_t* epoch, uint32_t next, int nblocks) {
  __threadfence();
  if (atomicAdd(&ctl->ticket, 1u) != (unsigned)nblocks - 1u) return;
  __threadfence();
  ctl->ticket = 0u;
  *epoch = next;
}

// Polls a word until the epoch in its last 4 bytes is e; false after `limit`
// reads, or once another block has given up.
__device__ __forceinline__ bool poll_word(const void* p, uint32_t e, uint32_t limit, const Ctl* ctl,
                                          unsigned long long& a, unsigned long long& b) {
  for (uint32_t i = 0; i < limit; ++i) {
    ld_word(p, a, b);
    if ((uint32_t)(b >> 32) == e) return true;
    if ((i & 1023u) == 1023u && timed_out(ctl)) return false;
  }
  return false;
}

// A published cell: (h, hu, hv) in FP32, (h, u, v) in FP64.
__device__ __forceinline__ void publish_cell(unsigned char* w, uint32_t e, float x, float y, float z) {
  const unsigned long long a =
      (unsigned long long)__float_as_uint(x) | (unsigned long long)__float_as_uint(y) << 32;
  st_word(w, a, (unsigned long long)__float_as_uint(z) | (unsigned long long)e << 32);
}
__device__ __forceinline__ void publish_cell(unsigned char* w, uint32_t e, double x, double y,
                                             double z) {
  const unsigned long long yb = (unsigned long long)__double_as_longlong(y);
  const unsigned long long ee = (unsigned long long)e << 32;
  st_word(w, (unsigned long long)__double_as_longlong(x), (yb & 0xffffffffull) | ee);
  st_word(w + 16, (unsigned long long)__double_as_longlong(z), (yb >> 32) | ee);
}
__device__ __forceinline__ bool read_cell(const unsigned char* w, uint32_t e, uint32_t limit,
                                          const Ctl* ctl, V4<float>& c) {
  unsigned long long a = 0, b = 0;
  const bool ok = poll_word(w, e, limit, ctl, a, b);
  c.x = __uint_as_float((uint32_t)a);
  c.y = __uint_as_float((uint32_t)(a >> 32));
  c.z = __uint_as_float((uint32_t)b);
  return ok;
}
__device__ __forceinline__ bool read_cell(const unsigned char* w, uint32_t e, uint32_t limit,
                                          const Ctl* ctl, V4<double>& c) {
  unsigned long long a = 0, b = 0, d = 0, f = 0;
  bool ok = false;
  for (uint32_t i = 0; i < limit; ++i) {  // both words in flight at once
    ld_word(w, a, b);
    ld_word(w + 16, d, f);
    ok = (uint32_t)(b >> 32) == e && (uint32_t)(f >> 32) == e;
    if (ok || ((i & 1023u) == 1023u && timed_out(ctl))) break;
  }
  c.x = __longlong_as_double((long long)a);
  c.y = __longlong_as_double((long long)((b & 0xffffffffull) | f << 32));
  c.z = __longlong_as_double((long long)d);
  return ok;
}

// Largest of 32 non-negative values, as the IEEE bits of a double.
__device__ __forceinline__ unsigned long long warp_max_bits(float v) {
  const unsigned r = __reduce_max_sync(0xffffffffu, __float_as_uint(v));
  return (unsigned long long)__double_as_longlong((double)__uint_as_float(r));
}
__device__ __forceinline__ unsigned long long warp_max_bits(unsigned long long v) {
  const unsigned hi = (unsigned)(v >> 32);
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)v : 0u);
  return (unsigned long long)mh << 32 | ml;
}
__device__ __forceinline__ unsigned long long warp_max_bits(double v) {
  return warp_max_bits((unsigned long long)__double_as_longlong(v));
}

// Most threads per block: the register budget (one block per SM at this
// size, or several smaller ones).
template <typename Real, bool CH>
constexpr int res_max_threads() { return sizeof(Real) == 8 ? 544 : CH ? 800 : 1024; }

// Polls per round of swe_params.wait_rounds (a round is at most about 20 us),
// on top of kLeastPolls (about 45 ms). A block's own copies take microseconds,
// which one round covers; here it waits for other blocks, which may start tens
// of microseconds apart and take a step of up to 50.
constexpr uint32_t kPollsPerRound = 32, kLeastPolls = 1u << 16;
__device__ __forceinline__ uint32_t most_polls(uint32_t rounds) {
  if (rounds == 0u) return 0u;  // the caller asked for no wait at all
  return rounds < (0xffffffffu - kLeastPolls) / kPollsPerRound ? kLeastPolls + rounds * kPollsPerRound
                                                              : 0xffffffffu;
}

// Up to n_steps steps of every scenario (fewer where one reaches its end time
// or an error). The last warp of a block is its control warp: while the
// others compute the faces of step s it reads the scenario's rate slots and
// forms dt and the clock. Two block barriers per step. CH: FP32 with a depth
// residual per cell.
template <typename Real, bool CH>
__global__ void __launch_bounds__(res_max_threads<Real, CH>(), 1)
    k_resident(ResPlan<Real> P, DevMesh<Real> m, DevState<Real> s, Num num, ResLayout L,
               long long n_steps) {
  constexpr bool kF64 = sizeof(Real) == 8;
  constexpr bool kComp = !kF64;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ unsigned long long s_wrate[32];
  __shared__ unsigned s_wbad[32], s_count;
  __shared__ Real s_dt;
  __shared__ int s_stop, s_fail, s_leave;
  __shared__ uint32_t s_epoch;
  Real* sc = reinterpret_cast<Real*>(smem);
  const int4* srec = reinterpret_cast<const int4*>(smem + L.off_rec);
  uint32_t* sside = reinterpret_cast<uint32_t*>(smem + L.off_rec);
  Real* snx = reinterpret_cast<Real*>(smem + L.off_nx);
  Real* sny = reinterpret_cast<Real*>(smem + L.off_ny);
  Real* slen = reinterpret_cast<Real*>(smem + L.off_len);
  double2* sq = reinterpret_cast<double2*>(smem + L.off_sq);
  Real* sslot = reinterpret_cast<Real*>(smem + L.off_slots);
  Real* sra = reinterpret_cast<Real*>(smem + L.off_ra);
  Real* sirp = reinterpret_cast<Real*>(smem + L.off_irp);
  Real* sgn2 = reinterpret_cast<Real*>(smem + L.off_gn2);
  float* slo = reinterpret_cast<float*>(smem + L.off_lo);
  int32_t* spub = reinterpret_cast<int32_t*>(smem + L.off_pub);
  Real* shz = reinterpret_cast<Real*>(smem + L.off_hz);
  int32_t* shpub = reinterpret_cast<int32_t*>(smem + L.off_hpub);
  const int ncs = (int)L.ncs;

  const ResBlock blk = P.blocks[blockIdx.x];
  Ctl* ctl = s.ctl + blk.scen;
  const int tid = threadIdx.x, nthr = blockDim.x, nct = nthr - 32, lane = tid & 31;
  const bool control = tid >= nct;
  const int cur = ctl->cur;  // written only once every block has stepped
  if (tid == 0) {
    s_epoch = P.epoch[blk.scen] + 1u;
    s_leave = *(const volatile int*)&ctl->done | (int)timed_out(ctl);
  }
  __syncthreads();
  const uint32_t e0 = s_epoch;  // epoch of the state at entry
  const uint32_t e_next = e0 + (uint32_t)n_steps + 1u;
  if (s_leave) {
    if (tid == 0) pass_entry(ctl, P.epoch + blk.scen, e_next, blk.nblocks);
    return;
  }
  const uint32_t limit = most_polls(num.wait_rounds);
  auto pub_word = [&](uint32_t e, int p) {
    return P.xbuf + ((size_t)(e & 1u) * P.npub + p) * pub_bytes<Real>();
  };
  auto rate_slot = [&](uint32_t e, int b) {
    return P.slots + ((size_t)(e & 1u) * gridDim.x + b) * 16;
  };

  // The part's cells, constants and records.
  const Real* h = cur ? s.h[1] : s.h[0];
  const Real* hu = cur ? s.hu[1] : s.hu[0];
  const Real* hv = cur ? s.hv[1] : s.hv[0];
  const int64_t sd = s.stride;
  auto z_of = [&](int64_t i) { return sd == 4 ? h[4 * i + 3] : s.z[i]; };
  for (int j = tid; j < blk.ncell; j += nthr) {
    const int64_t i = P.cells[blk.cell0 + j];
    const int p = P.pub[blk.cell0 + j];
    const Real hh = h[i * sd], qx = hu[i * sd], qy = hv[i * sd], z = z_of(i);
    Real x = qx, y = qy;
    if constexpr (kF64) {
      velocity(hh, qx, qy, num, x, y);
      sq[j] = make_double2(qx, qy);
      sra[j] = m.rarea ? m.rarea[i] : __ddiv_rn(1.0, m.area[i]);
    } else {
      sra[j] = rcp_approx(m.area[i]);
    }
    st4(sc + 4 * j, hh, x, y, z);
    sirp[j] = m.irP[i];
    sgn2[j] = s.gn2[i];
    if constexpr (CH) slo[j] = s.hlo[i];
    spub[j] = p;
    if (p >= 0) publish_cell(pub_word(e0, p), e0, hh, x, y);
  }
  for (int q = tid; q < blk.nhalo; q += nthr) {
    shz[q] = z_of(P.halo[blk.halo0 + q]);
    shpub[q] = P.halo_pub[blk.halo0 + q];
  }
  for (int r = tid; r < blk.nrec; r += nthr) {
    if constexpr (kF64) {
      sside[r] = P.side[blk.rec0 + r];
      snx[r] = P.nx[blk.rec0 + r];
      sny[r] = P.ny[blk.rec0 + r];
      slen[r] = P.len[blk.rec0 + r];
    } else {
      const_cast<int4*>(srec)[r] = P.rec[blk.rec0 + r];
    }
  }
  // The scenario's clock (control warp, lane 0).
  double t = ctl->t, dt_now = ctl->dt, dt_cfl = ctl->dt_cfl, dt_last = ctl->dt_last;
  const double t_end = ctl->t_end;
  int clamped = ctl->clamped, done = 0, err = 0;
  long long taken = 0;
  if (tid == 0) {
    s_count = 0;
    s_stop = 0;
    s_fail = 0;
    s_dt = Real(dt_now);
  }
  __syncthreads();

  // Control warp: the largest rate of the state of epoch e over the
  // scenario's blocks, then the clock after the step that made it (as
  // finish_launch sets it). What does not need the rate is formed before it
  // is there, and a lane's slots are read kBatch at a time. False if a slot
  // did not come.
  constexpr int kBatch = 5;
  auto next_clock = [&](uint32_t e) -> bool {
    dt_last = dt_now;
    t = clamped ? t_end : t + dt_now;
    const double rest = t_end - t;
    const bool at_end = t >= t_end;
    taken += 1;
    unsigned long long top = 0;
    unsigned bad = 0;
    bool ok = true;
    for (int i0 = lane; i0 < blk.nblocks && ok; i0 += 32 * kBatch) {
      unsigned long long a[kBatch], b[kBatch];
      ok = false;
      for (uint32_t n = 0; n < limit && !ok; ++n) {
#pragma unroll
        for (int q = 0; q < kBatch; ++q)
          ld_word(rate_slot(e, blk.block0 + min(i0 + 32 * q, blk.nblocks - 1)), a[q], b[q]);
        ok = true;
#pragma unroll
        for (int q = 0; q < kBatch; ++q) ok = ok && (uint32_t)(b[q] >> 32) == e;
        if (!ok && (n & 1023u) == 1023u && timed_out(ctl)) break;
      }
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        top = max(top, a[q]);
        bad |= (unsigned)b[q];
      }
    }
    if (__any_sync(0xffffffffu, !ok)) return false;
    top = warp_max_bits(top);
    err |= (int)__reduce_or_sync(0xffffffffu, bad);
    if (top == 0ull) err |= kErrDry;
    err |= rate_error(__longlong_as_double((long long)top));
    if (err) {
      done = 1;
      dt_now = 0.0;
      dt_cfl = 0.0;
    } else {
      dt_cfl = cfl_dt(num.courant, __longlong_as_double((long long)top));
      done = at_end;
      clamped = dt_cfl >= rest;
      dt_now = clamped ? rest : dt_cfl;
    }
    return true;
  };

  int neg = 0;
  Real chk = Real(0);
  bool timeout = false;
  long long k = 0;
  for (; k < n_steps; ++k) {
    const uint32_t e = e0 + (uint32_t)k;
    if (control) {
      if (k > 0) {
        const bool ok = next_clock(e);
        if (lane == 0) {
          s_dt = Real(dt_now);
          if (done) s_stop = 1;
          if (!ok) s_fail = 1;
        }
      } else if (lane == 0) {  // idle otherwise
        pass_entry(ctl, P.epoch + blk.scen, e_next, blk.nblocks);
      }
    } else {
      // A warp's 32 records together: its lanes meet again after the polls,
      // whose lengths differ (left to themselves they went through the face
      // in up to four groups, 2 us of an FP64 step).
      for (int r0 = tid & ~31; r0 < blk.nrec; r0 += nct) {
        const int r = r0 + lane;
        const bool live = r < blk.nrec;
        uint32_t packed = 0xffffffffu;
        Real nx = Real(0), ny = Real(0), len = Real(0);
        if (live) {
          if constexpr (kF64) {
            packed = sside[r];
            nx = snx[r];
            ny = sny[r];
            len = slen[r];
          } else {
            int32_t w;
            rec_f32(srec, r, w, nx, ny, len);
            packed = (uint32_t)w;
          }
        }
        const uint32_t a = packed >> 16, b = packed & 0xffffu;
        const int ka = a >> 14, kb = b >> 14, ia = a & 0x3fff, ib = b & 0x3fff;
        const bool wall = b == kResWall;
        V4<Real> A{}, B{};
        if (live) {
          if (ka != 3) A = ld4(sc + 4 * ia);
          if (kb != 3) B = ld4(sc + 4 * ib);
          if (!wall && (ka == 3 || kb == 3)) {  // one side is a halo cell
            const int q = ka == 3 ? ia : ib;
            V4<Real> H;
            if (!read_cell(pub_word(e, shpub[q]), e, limit, ctl, H)) s_fail = 1;
            H.w = shz[q];
            if (ka == 3) A = H;
            else B = H;
          }
        }
        __syncwarp();
        if (!live) continue;
        Real c0, cA1, cA2, cB1, cB2;
        if (wall) {
          if constexpr (kF64) face_flux_f64<true>(A, A, nx, ny, len, num, c0, cA1, cA2, cB1, cB2);
          else face_flux_f32<true>(A, A, nx, ny, len, num, c0, cA1, cA2, cB1, cB2);
        } else {
          if constexpr (kF64) face_flux_f64<false>(A, B, nx, ny, len, num, c0, cA1, cA2, cB1, cB2);
          else face_flux_f32<false>(A, B, nx, ny, len, num, c0, cA1, cA2, cB1, cB2);
        }
        // FP32 forms side B's contributions negated
        if (ka != 3) {
          const int q = ka * ncs + ia;
          if constexpr (kF64) {
            sslot[q] = c0;
            sslot[3 * ncs + q] = cA1;
            sslot[6 * ncs + q] = cA2;
          } else {
            st4(sslot + 4 * q, c0, 0.0f, cA1, cA2);
          }
        }
        if (kb != 3) {
          const int q = kb * ncs + ib;
          if constexpr (kF64) {
            sslot[q] = -c0;
            sslot[3 * ncs + q] = -cB1;
            sslot[6 * ncs + q] = -cB2;
          } else {
            st4(sslot + 4 * q, -c0, 0.0f, cB1, cB2);
          }
        }
      }
    }
    __syncthreads();
    if (s_stop) break;
    if (s_fail) {
      timeout = true;
      break;
    }
    if (!control) {
      const Real dt = s_dt;
      const bool last = k + 1 == n_steps;
      Real rate = Real(0);
      NoMass<Real> mass;
      for (int j = tid; j < blk.ncell; j += nct) {
        Real R[3];
        const V4<Real> c = ld4(sc + 4 * j);
        Real qx = c.y, qy = c.z, lo = Real(0);
        if constexpr (kF64) {
#pragma unroll
          for (int q = 0; q < 3; ++q)
            R[q] = sslot[3 * q * ncs + j] + sslot[(3 * q + 1) * ncs + j] + sslot[(3 * q + 2) * ncs + j];
          const double2 q2 = sq[j];
          qx = q2.x;
          qy = q2.y;
        } else {
          sum_faces_f32(ld4(sslot + 4 * j), ld4(sslot + 4 * (ncs + j)), ld4(sslot + 4 * (2 * ncs + j)),
                        R);
        }
        if constexpr (CH) lo = slo[j];
        Real a1, b1, c1, rh;
        cell_finish<Real, kComp, NoMass<Real>, true, CH>(c.x, qx, qy, sra[j], sirp[j], sgn2[j], dt, R,
                                                         num, a1, b1, c1, mass, rate, chk, neg, &lo, &rh);
        Real x = b1, y = c1;
        if constexpr (kF64) {
          x = mul_rn(b1, rh);
          y = mul_rn(c1, rh);
          sq[j] = make_double2(b1, c1);
        }
        if constexpr (CH) slo[j] = lo;
        st4(sc + 4 * j, a1, x, y, c.w);
        const int p = spub[j];
        if (p >= 0 && !last) publish_cell(pub_word(e + 1, p), e + 1, a1, x, y);
      }
      // The block's largest rate, published by the last of its warps to
      // get here.
      const unsigned long long wr = warp_max_bits(rate);
      const unsigned wb = __any_sync(0xffffffffu, chk != Real(0)) ? (unsigned)kErrNan : 0u;
      const int wid = tid >> 5, nw = nct >> 5;
      unsigned n = 0;
      if (lane == 0) {
        s_wrate[wid] = wr;
        s_wbad[wid] = wb;
        __threadfence_block();
        n = atomicAdd(&s_count, 1u);
      }
      n = __shfl_sync(0xffffffffu, n, 0);
      if (n == (unsigned)nw - 1u) {
        __threadfence_block();
        const unsigned long long br =
            warp_max_bits(lane < nw ? *(volatile unsigned long long*)&s_wrate[lane] : 0ull);
        const unsigned bb =
            __reduce_or_sync(0xffffffffu, lane < nw ? *(volatile unsigned*)&s_wbad[lane] : 0u);
        if (lane == 0) {
          st_word(rate_slot(e + 1, blockIdx.x), br,
                  (unsigned long long)bb | (unsigned long long)(e + 1) << 32);
          s_count = 0;
        }
      }
    }
    __syncthreads();
  }

  // After the last step its rate gives the next dt (the scenario's first
  // block needs it); a step that ended the run has set the clock already.
  if (!timeout && k == n_steps && control && blk.first) timeout = !next_clock(e0 + (uint32_t)k);
  if (control && lane == 0) {
    if (timeout) {
      atomicOr(&ctl->err, kErrTimeout);
      ctl->done = 1;
      ctl->dt = 0.0;
      ctl->dt_cfl = 0.0;
    } else if (blk.first) {
      ctl->t = t;
      ctl->dt = dt_now;
      ctl->dt_cfl = dt_cfl;
      ctl->dt_last = dt_last;
      ctl->steps += taken;
      if (taken > 0) ctl->cur = cur ^ 1;
      ctl->clamped = clamped;
      if (err) atomicOr(&ctl->err, err);
      if (done) ctl->done = 1;
    }
  }
  // State after the step(s), into the other buffer: until the buffer number
  // changes, the one read at entry is the state.
  if (!timeout && k > 0) {
    Real* oh = cur ? s.h[0] : s.h[1];
    Real* ohu = cur ? s.hu[0] : s.hu[1];
    Real* ohv = cur ? s.hv[0] : s.hv[1];
    for (int j = tid; j < blk.ncell; j += nthr) {
      const int64_t i = P.cells[blk.cell0 + j];
      const V4<Real> c = ld4(sc + 4 * j);
      Real qx = c.y, qy = c.z;
      if constexpr (kF64) {
        qx = sq[j].x;
        qy = sq[j].y;
      }
      if (sd == 4) {
        st4(oh + 4 * i, c.x, qx, qy, c.w);
      } else {
        oh[i] = c.x;
        ohu[i] = qx;
        ohv[i] = qy;
      }
      if constexpr (CH) s.hlo[i] = slo[j];
    }
  }
  const int wneg = __reduce_add_sync(0xffffffffu, neg);
  if (lane == 0 && wneg) atomicAdd((unsigned long long*)&ctl->neg, (unsigned long long)wneg);
}

}  // namespace swe
