// qed_step.cu -- the per-macroparticle QED Monte Carlo step on sm_103a: the push,
// the multi-pass lepton step (FP64 contexts, Methods II and III, the learned
// sampler with ordered appends; the others take the single pass of
// qed_onepass.cu), compaction, the isolated sampler and the parity hooks.  The
// photons' stage is qed_photon.cu's.
//
// What is computed per lepton: field gather (uniform / per-particle / CIC) ->
// Boris push -> chi_e (Eq. 2) -> W_rad from the tables (Eq. 1 with the xi_min
// cut) -> N = max(1, ceil(W Dt / 0.2)) sub-steps -> Method I events with Philox
// draws -> xi from Eq. (7) -> recoil; photons appended.
// How the multi-pass step is laid out: a streaming pass reads every particle
// once (coalesced), pushes it and evaluates the rate and the first draw; those
// with one sub-step and no event (most) are finished there.  The rest are
// staged as 64-byte records, ordered by a class list (binned by N so that
// lanes of a warp do similar work), and run through a counting pass, a scan
// and a writing pass that append their photons in list order.  Appends keep a
// deterministic order (and sub-step order within a particle); the scan works
// within the block and across tiles by a single-pass decoupled look-back, so
// slot = count at launch + global prefix.
// Particle state is structure-of-arrays; loads and stores of a tile are
// coalesced 4-byte (FP32) or 8-byte (FP64) accesses.
#include <cstdio>

#include "qed_internal.h"
#include "qed_kernels.cuh"
#include "qed_mlp.cuh"

namespace qed {


// ---------------------------------------------------------------------------
// Lepton kernel (electrons and positrons in one launch)
// ---------------------------------------------------------------------------
// Pushed state of a flagged lepton, written once by the streaming pass so the
// later passes read 64 (FP32) or 128 (FP64) contiguous bytes per particle
// instead of gathering a 4- or 8-byte word from each of 14 arrays.
template <class Real> struct alignas(16) Stage {
  Real p[3], e[3], b[3];
  uint32_t id_lo, id_hi;
  Real w;
  Real x[3];
  uint32_t slot;
};
static_assert(sizeof(Stage<float>) == 64, "FP32 staging record");
static_assert(sizeof(Stage<double>) == 128, "FP64 staging record");
constexpr uint32_t STAGE_BATCH = 256;  // records a warp reserves at a time

template <class Real> struct LeptonArgs {
  Sp<Real> sp[2];
  int nsp;
  Sp<Real> ph;
  Fld<Real> f;
  Consts C;
  Tables<Real> T;  // R, F staged to shared memory; Y read through L1/L2
  Out o;
  int64_t step;
  uint8_t *heavy_flags;     // [streaming-pass slot] class flag (0 = finished)
  const int *heavy_list;    // class list: staging record or -(slot + 1), class-major
  const int64_t *d_step;    // if set, the step index is read here (graph replay)
  const int64_t *cls_off;   // class list: class c occupies [cls_off[c-1], cls_off[c])
  Stage<Real> *stage;       // pushed state of the flagged leptons (streaming pass)
  uint32_t *stage_tag;      // their tags (species with tags)
  int32_t *stage_idx;       // [slot] staging index of a flagged slot, -1 if not staged
  unsigned int *stage_n;    // staging allocation counter (reset by the class-list scan)
  int64_t stage_cap;
  uint32_t *sub_cnt;        // sub-step passes: photons per class-2..5 entry
  Real *sub_gf;             // final gamma per entry (entries < rec_cap)
  Real *rec_e;              // [REC][rec_cap] photon energies
  uint32_t *rec_k;          // [REC][rec_cap] their sub-step indices
  int64_t rec_cap;
  const int64_t *sub_meta;  // [0] photons of the sub-step entries, [1] photon count before them
  int32_t *replay_list;     // entries whose chains the replay launch redoes
  unsigned int *replay_n;   // their number (reset by the scan)
  const uint32_t *mlp_frag; // learned inverse CDF (used when use_mlp)
  const float *mlp_w;
  int use_mlp;
  int emit_lanes, scan_draws;  // chain scheduling (QED_SCHED_EMIT_LANES, _SCAN_DRAWS)
};


// First slot of a thread.  FP64: consecutive slices of 32 go to different CTAs, so
// that a small species is spread over the SMs, which run FP64 at 2 FMAs per clock
// (10^4 electrons in 40 CTAs of 256 took 26 us, over all SMs 11).  FP32 is bound by
// memory, and a CTA's 256 slots stay together: the push of 4.2M electrons with
// fields 49.7 us, 52.8 spread; 16.8M 182, 190.
template <class Real> __device__ __forceinline__ int64_t first_slot() {
  return sizeof(Real) == 8 ? ((int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31)
                           : (int64_t)blockIdx.x * TILE + threadIdx.x;
}

// ---------------------------------------------------------------------------
// Push-only pass (qed_gather_push): field gather, Boris push and position
// update of every lepton; no emission, so no ordering is needed.
// ---------------------------------------------------------------------------
template <class Real, int FM>
__global__ void __launch_bounds__(TILE) k_lepton_push(LeptonArgs<Real> A) {
  __shared__ long long s_meta[2];
  if (threadIdx.x == 0) {
    s_meta[0] = *(volatile int64_t *)A.sp[0].d_n;
    s_meta[1] = A.nsp > 1 ? *(volatile int64_t *)A.sp[1].d_n : 0;
  }
  __syncthreads();
  const int64_t n0 = s_meta[0], n1 = s_meta[1];
  const Real dt = sel<Real>(A.C.dt, A.C.f_dt);
  uint32_t status = 0;
  for (int64_t g = first_slot<Real>(); g < n0 + n1; g += (int64_t)gridDim.x * TILE) {
    const int si = g < n0 ? 0 : 1;
    const Sp<Real> &S = A.sp[si];
    const int64_t i = si ? g - n0 : g;
    Real x = S.x[i], y = S.y[i], z = S.z[i];
    Real px = S.px[i], py = S.py[i], pz = S.pz[i];
    Real E[3], B[3];
    get_fields<Real, FM>(S, A.f, i, x, y, z, E, B);
    const Real gm = boris(px, py, pz, E, B, S.q, dt);
    if (!(gm < (Real)1e30)) {  // non-finite state: left as it was
      status |= QED_STATUS_NONFINITE;
      continue;
    }
    const Real ig = r_div(dt, gm);
    S.x[i] = x + px * ig; S.y[i] = y + py * ig; S.z[i] = z + pz * ig;
    S.px[i] = px; S.py[i] = py; S.pz[i] = pz;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) status |= __shfl_xor_sync(0xFFFFFFFFu, status, o);
  if ((threadIdx.x & 31) == 0 && status) atomicOr(&A.o.cnt->status, status);
}

// ---------------------------------------------------------------------------
// Streaming pass over all leptons: gather, push, chi, rate and the first
// Method I draw, with no block-wide synchronisation.  A particle that needs
// one sub-step and draws no event is finished here (its new position and
// momentum are written); the rest are only flagged -- 1: one sub-step with an
// event, 2: more than one sub-step -- and are redone, from their unchanged
// stored state, by the ordered passes that append photons.
// ---------------------------------------------------------------------------

template <class Real, int FM, int MODE>
__global__ void __launch_bounds__(TILE, sizeof(Real) == 4 ? 3 : 2) k_lepton_stream(LeptonArgs<Real> A) {
  const int64_t step_ = A.d_step ? *A.d_step : A.step;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr bool kSmem = sizeof(Real) == 4;
  constexpr int NV = stream_words<FM>();
  Real *sR = kSmem ? reinterpret_cast<Real *>(smem_raw) : const_cast<Real *>(A.T.R);
  Real *sF = kSmem ? sR + A.T.gl.n : const_cast<Real *>(A.T.F);
  // prefetch buffers after the tables: [2][NV][TILE] words, then [2][TILE] ids
  const size_t tab_bytes = kSmem ? (((size_t)A.T.gl.n * (1 + A.T.gy.n) * sizeof(Real) + 15) & ~(size_t)15) : 0;
  Real *pf = reinterpret_cast<Real *>(smem_raw + tab_bytes);
  uint64_t *pf_id = reinterpret_cast<uint64_t *>(pf + 2 * NV * TILE);
  __shared__ long long s_meta[4];
  __shared__ BlockTally bt;
  if (kSmem) {
    load_tables_smem(sR, A.T.R, A.T.gl.n);
    load_tables_smem(sF, A.T.F, A.T.gl.n * A.T.gy.n);
  }
  block_tally_init(&bt);
  if (threadIdx.x == 0) {
    s_meta[0] = *(volatile int64_t *)A.sp[0].d_n;
    s_meta[1] = A.nsp > 1 ? *(volatile int64_t *)A.sp[1].d_n : 0;
  }
  __syncthreads();
  const int64_t n0 = s_meta[0], n1 = s_meta[1];
  const int64_t T0 = (n0 + TILE - 1) / TILE, T1 = (n1 + TILE - 1) / TILE;
  const int64_t nslots = (T0 + T1) * TILE;
  const Real inv_aS = sel<Real>(A.C.inv_aS, A.C.f_inv_aS);
  const Real dt = sel<Real>(A.C.dt, A.C.f_dt), wdt_max = sel<Real>(A.C.wdt_max, A.C.f_wdt_max);
  const int lane = threadIdx.x & 31;
  const int t = threadIdx.x;
  // this warp's current batch of staging records (warp-uniform)
  uint32_t batch_base = 0, batch_used = STAGE_BATCH;
  Tally tl;
  tl.clear();
  // issue the copies of slot `sl`'s particle into buffer b
  auto prefetch = [&](int64_t sl, int b) {
    const int64_t tile = sl / TILE;
    const int si = tile < T0 ? 0 : 1;
    const Sp<Real> &S = A.sp[si];
    const int64_t i = (tile - (si ? T0 : 0)) * TILE + (sl % TILE);
    if (i >= (si ? n1 : n0)) return;
    Real *d = pf + (size_t)b * NV * TILE + t;
    const Real *src[12] = {S.x, S.y, S.z, S.px, S.py, S.pz, S.ex, S.ey, S.ez, S.bx, S.by, S.bz};
#pragma unroll
    for (int c = 0; c < NV; ++c) cp_async<sizeof(Real)>(d + c * TILE, src[c] + i);
    cp_async<8>(pf_id + b * TILE + t, S.id + i);
  };
  const int64_t stride = (int64_t)gridDim.x * TILE;
  int buf = 0;
  int64_t slot = first_slot<Real>();
  if (slot < nslots) prefetch(slot, 0);
  cp_async_commit();
  // nslots is a multiple of TILE: every lane of a warp runs the same iterations
  for (; slot < nslots; slot += stride, buf ^= 1) {
    if (slot + stride < nslots) prefetch(slot + stride, buf ^ 1);
    cp_async_commit();
    cp_async_wait<1>();  // this slot's copies have landed
    const int64_t tile = slot / TILE;
    const int si = tile < T0 ? 0 : 1;
    const Sp<Real> &S = A.sp[si];
    const int64_t i = (tile - (si ? T0 : 0)) * TILE + (slot % TILE);
    uint8_t flag = 0;
    Real x = 0, y = 0, z = 0, px = 0, py = 0, pz = 0;
    Real E[3] = {0, 0, 0}, B[3] = {0, 0, 0};
    uint64_t pid = 0;
    if (i < (si ? n1 : n0)) {
      const Real *v = pf + (size_t)buf * NV * TILE + t;
      x = v[0]; y = v[TILE]; z = v[2 * TILE];
      px = v[3 * TILE]; py = v[4 * TILE]; pz = v[5 * TILE];
      if (FM == FM_PER_PARTICLE) {
        E[0] = v[6 * TILE]; E[1] = v[7 * TILE]; E[2] = v[8 * TILE];
        B[0] = v[9 * TILE]; B[1] = v[10 * TILE]; B[2] = v[11 * TILE];
      } else {
        get_fields<Real, FM>(S, A.f, i, x, y, z, E, B);
      }
      pid = pf_id[buf * TILE + t];
      Real g;
      if (MODE != MODE_EMIT) {
        g = boris(px, py, pz, E, B, S.q, dt);
        Real ig = r_div(dt, g);
        x += px * ig; y += py * ig; z += pz * ig;
      } else {
        g = m_sqrt((Real)1 + px * px + py * py + pz * pz);
      }
      if (!(g < (Real)1e30)) {
        tl.status |= QED_STATUS_NONFINITE;
      } else {
        Real chi = chi_lepton(px, py, pz, g, E[0], E[1], E[2], B[0], B[1], B[2], inv_aS);
        Tally t0;
        t0.clear();
        RateOut<Real> ro = photon_rate(sR, sF, A.T, A.C, chi, g, t0);
        const Real wdt = ro.W * dt;
        if (A.C.generator != GEN_METHOD_I) {
          // Methods II/III: P_cum += W Dt; an event when 1 - exp(-P_cum) > r3
          // (II) or P_cum > r3 (III); r3 is word 3 of the emission draw when
          // not drawn yet.  The emission itself (and the new P_cum, r3) is the
          // counting pass's, as a one-sub-step particle with an event.
          const U4 r = draw(A.C, pid, step_, 0, STREAM_EMIT);
          Real r3 = S.od_r[i];
          const bool fresh = !(r3 > (Real)0);
          if (fresh) r3 = unif<Real>(r.w);
          const Real P = S.od_p[i] + wdt;
          const bool ev = A.C.generator == GEN_METHOD_II ? -m_expm1(-P) > r3 : P > r3;
          if (ev) {
            flag = 1;
          } else {
            S.od_p[i] = P;
            if (fresh) S.od_r[i] = r3;
          }
        } else if (wdt > wdt_max) {
          // classes by sub-step count N = ceil(W Dt / wdt_max): 2: N <= 3, 3: N <= 7,
          // 4: N <= 15, 5: N >= 16 (lanes of a warp then do similar amounts of work)
          const Real q = r_div(wdt, wdt_max);
          flag = q <= (Real)3 ? 2 : (q <= (Real)7 ? 3 : (q <= (Real)15 ? 4 : 5));
        } else {
          U4 r = draw(A.C, pid, step_, 0, STREAM_EMIT);
          if (wdt > unif<Real>(r.x)) flag = 1;  // one sub-step with an event
        }
        if (flag == 0) {
          tl.status |= t0.status;
          tl.domain += t0.domain;
          tl.substeps += 1;
          if (MODE != MODE_EMIT) {
            S.x[i] = x; S.y[i] = y; S.z[i] = z;
            S.px[i] = px; S.py[i] = py; S.pz[i] = pz;
          }
        }
      }
    }
    A.heavy_flags[slot] = flag;
    // stage the pushed state of the flagged particles (warp-collective)
    const unsigned m = __ballot_sync(0xFFFFFFFFu, flag != 0);
    if (m) {
      const uint32_t cm = __popc(m);
      if (batch_used + cm > STAGE_BATCH) {
        uint32_t nb = 0;
        if (lane == 0) nb = atomicAdd(A.stage_n, STAGE_BATCH);
        batch_base = __shfl_sync(0xFFFFFFFFu, nb, 0);
        batch_used = 0;
      }
      if (flag) {
        const uint64_t pos = (uint64_t)batch_base + batch_used + __popc(m & ((1u << lane) - 1u));
        int32_t sidx = -1;
        if (pos < (uint64_t)A.stage_cap) {
          sidx = (int32_t)pos;
          Stage<Real> r;
          r.p[0] = px; r.p[1] = py; r.p[2] = pz;
          r.e[0] = E[0]; r.e[1] = E[1]; r.e[2] = E[2];
          r.b[0] = B[0]; r.b[1] = B[1]; r.b[2] = B[2];
          r.id_lo = (uint32_t)pid; r.id_hi = (uint32_t)(pid >> 32);
          r.w = S.w[i];
          r.x[0] = x; r.x[1] = y; r.x[2] = z;
          r.slot = (uint32_t)slot;
          const uint4 *src = reinterpret_cast<const uint4 *>(&r);
          uint4 *dst = reinterpret_cast<uint4 *>(A.stage + pos);
#pragma unroll
          for (int q = 0; q < (int)(sizeof(Stage<Real>) / 16); ++q) dst[q] = src[q];
          if (S.tag) A.stage_tag[pos] = S.tag[i];
          // the later passes read the staged copy; the pushed position and
          // momentum go to the arrays now, with the rest of the tile
          if (MODE != MODE_EMIT) {
            S.x[i] = x; S.y[i] = y; S.z[i] = z;
            S.px[i] = px; S.py[i] = py; S.pz[i] = pz;
          }
        }
        A.stage_idx[slot] = sidx;
      }
      batch_used += cm;
    }
  }
  cp_async_wait<0>();
  tally_flush(&bt, tl);
  __syncthreads();
  block_tally_commit(&bt, A.o.cnt, 0);
}

// ---------------------------------------------------------------------------
// Emission passes over the class list: every lepton the streaming pass could
// not finish (an event possible, or N > 1 by the rate bound).  The work is
// split so that no emission chain ever waits on another:
//   counting pass: the exact rate (with the xi_min cut) and N, then the
//     particle's Method I chain -- per sub-step one Philox draw, on an event
//     kappa from r2, ln delta from the inverse table (or the learned sampler
//     for N = 1), xi (Eq. 7) and the recoil -- writing only the number of
//     photons, the final gamma and the first REC emission records (photon
//     energy, sub-step index).  Particles are independent: no scan, no order.
//   scan: an in-place exclusive scan of the counts (one pass, decoupled
//     look-back over 4096-entry tiles of uniform cost) gives every particle
//     its first photon slot.
//   writing pass: the photons of each particle, from its records -- or, for a
//     particle with more than REC photons, from a replay of its chain -- and
//     its final momentum.
// Within a warp the chain is split into a scan phase (each lane draws until
// its next event) and an emission phase that the lanes with an event execute
// together, so lanes of different event counts stay converged.
// ---------------------------------------------------------------------------
constexpr int REC = SUB_REC;
// Work scheduling of the counting pass: a lane is idle (no particle), scanning
// (drawing sub-steps) or pending (an event found, its emission not yet done).
enum { LS_IDLE = 0, LS_SCAN = 1, LS_PEND = 2 };
constexpr int CNT_CHUNK = 64, CNT_CHUNK_MIN = 16;  // entries per queue chunk of a warp
// An emission round waits for A.emit_lanes lanes with an event, a refill
// round for CNT_MIN_INIT idle lanes; a scanning round draws A.scan_draws
// sub-steps per lane.
constexpr int CNT_MIN_INIT = 20;

// A class-list entry's particle after the push.  Entry e >= 0 is staging
// record e (written by the streaming pass, which has also stored the pushed
// position and momentum); e < 0 is slot -e-1, a particle the staging area had
// no room for, gathered and pushed again from its unchanged stored state.
template <class Real> struct Entry {
  Real x, y, z, px, py, pz, g, w;
  Real E[3], B[3];
  uint64_t id;
  uint32_t tag;
  int64_t i;     // index in species si
  int si;
  bool staged;
};

template <class Real, int FM, int MODE>
__device__ __forceinline__ void load_entry(const LeptonArgs<Real> &A, int32_t e, int64_t T0,
                                           Real dt, Entry<Real> &P) {
  int64_t slot;
  P.staged = e >= 0;
  if (P.staged) {
    Stage<Real> r;
    const uint4 *src = reinterpret_cast<const uint4 *>(A.stage + e);
    uint4 *dst = reinterpret_cast<uint4 *>(&r);
#pragma unroll
    for (int q = 0; q < (int)(sizeof(Stage<Real>) / 16); ++q) dst[q] = __ldcs(src + q);
    P.px = r.p[0]; P.py = r.p[1]; P.pz = r.p[2];
#pragma unroll
    for (int c = 0; c < 3; ++c) { P.E[c] = r.e[c]; P.B[c] = r.b[c]; }
    P.id = (uint64_t)r.id_lo | ((uint64_t)r.id_hi << 32);
    P.w = r.w;
    P.x = r.x[0]; P.y = r.x[1]; P.z = r.x[2];
    slot = r.slot;
  } else {
    slot = -(int64_t)e - 1;
  }
  const int64_t tile = slot / TILE;
  P.si = tile < T0 ? 0 : 1;
  P.i = (tile - (P.si ? T0 : 0)) * TILE + (slot % TILE);
  const Sp<Real> &S = A.sp[P.si];
  if (P.staged) {
    P.tag = S.tag ? A.stage_tag[e] : 0u;
    P.g = m_sqrt((Real)1 + P.px * P.px + P.py * P.py + P.pz * P.pz);
    return;
  }
  const int64_t i = P.i;
  P.x = S.x[i]; P.y = S.y[i]; P.z = S.z[i];
  P.px = S.px[i]; P.py = S.py[i]; P.pz = S.pz[i];
  get_fields<Real, FM>(S, A.f, i, P.x, P.y, P.z, P.E, P.B);
  P.id = S.id[i];
  P.w = S.w[i];
  P.tag = S.tag ? S.tag[i] : 0u;
  if (MODE != MODE_EMIT) {
    P.g = boris(P.px, P.py, P.pz, P.E, P.B, S.q, dt);
    Real ig = r_div(dt, P.g);
    P.x += P.px * ig; P.y += P.py * ig; P.z += P.pz * ig;
  } else {
    P.g = m_sqrt((Real)1 + P.px * P.px + P.py * P.py + P.pz * P.pz);
  }
}

// Final state of an entry after its emissions (final gamma g, unit direction
// n): a staged particle already has its pushed position stored.
template <class Real, int MODE>
__device__ __forceinline__ void store_entry(const LeptonArgs<Real> &A, const Entry<Real> &P,
                                            Real g, Real nx, Real ny, Real nz) {
  const Sp<Real> &S = A.sp[P.si];
  const int64_t i = P.i;
  const Real pm = m_sqrt((g - (Real)1) * (g + (Real)1));
  if (MODE != MODE_EMIT && !P.staged) { S.x[i] = P.x; S.y[i] = P.y; S.z[i] = P.z; }
  S.px[i] = pm * nx; S.py[i] = pm * ny; S.pz[i] = pm * nz;
}

template <class Real>
__device__ __forceinline__ void unit_dir(const Entry<Real> &P, Real &nx, Real &ny, Real &nz) {
  nx = ny = nz = 0;
  const Real pm = m_sqrt(P.px * P.px + P.py * P.py + P.pz * P.pz);
  if (pm > (Real)0) { Real ip = (Real)1 / pm; nx = P.px * ip; ny = P.py * ip; nz = P.pz * ip; }
}

// Sub-step count of a particle (Method I: N = max(1, ceil(W Dt / wdt_max))).
template <class Real>
__device__ __forceinline__ int64_t substep_count(const Consts &C, Real W, Real dt, Real wdt_max,
                                                 uint32_t &status) {
  const Real wdt = W * dt;
  if (!(wdt > wdt_max)) return 1;
  Real nn = m_ceil(wdt / wdt_max);
  if (nn > (Real)C.max_substeps) {
    nn = (Real)C.max_substeps;
    status |= QED_STATUS_SUBSTEPS;
  }
  return (int64_t)nn;
}

template <class Real, int FM, int MODE, bool MLP>
__global__ void __launch_bounds__(TILE, sizeof(Real) == 4 && !MLP ? 3 : 2) k_substep_count(LeptonArgs<Real> A) {
  const int64_t step_ = A.d_step ? *A.d_step : A.step;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr bool kSmem = sizeof(Real) == 4;
  Real *sR = kSmem ? reinterpret_cast<Real *>(smem_raw) : const_cast<Real *>(A.T.R);
  Real *sF = kSmem ? sR + A.T.gl.n : const_cast<Real *>(A.T.F);
  // learned sampler image after the tables (FP32 contexts only)
  uint32_t *s_frag = reinterpret_cast<uint32_t *>(
      smem_raw + (kSmem ? (((size_t)A.T.gl.n * (1 + A.T.gy.n) * sizeof(Real) + 15) & ~(size_t)15) : 0));
  float *s_fw = reinterpret_cast<float *>(s_frag + MLP_FRAG_WORDS);
  constexpr bool use_mlp = kSmem && MLP;
  if (use_mlp) mlp_stage(s_frag, s_fw, A.mlp_frag, A.mlp_w);
  __shared__ long long s_meta[4];
  __shared__ BlockTally bt;
  if (kSmem) {
    load_tables_smem(sR, A.T.R, A.T.gl.n);
    load_tables_smem(sF, A.T.F, A.T.gl.n * A.T.gy.n);
  }
  block_tally_init(&bt);
  if (threadIdx.x == 0) {
    s_meta[0] = *(volatile int64_t *)A.sp[0].d_n;
    s_meta[1] = 0;  // the whole class list
    s_meta[2] = A.cls_off[NCLS];
  }
  __syncthreads();
  const int64_t T0 = (s_meta[0] + TILE - 1) / TILE;
  const int64_t begin = s_meta[1], nh = s_meta[2] - s_meta[1];
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  const Real inv_aS = sel<Real>(A.C.inv_aS, A.C.f_inv_aS);
  const Real dt = sel<Real>(A.C.dt, A.C.f_dt);
  const Real wdt_max = sel<Real>(A.C.wdt_max, A.C.f_wdt_max);
  const int64_t rc = A.rec_cap;
  Tally tl;
  tl.clear();
  // This warp's queue: chunks w, w + W, w + 2W, ... of `chunk` entries, counted
  // from the end of the list (the heaviest classes first).  The first chunks
  // go to different CTAs, and a short list is cut into smaller ones, so that
  // its chains run on all SMs (250 FP64 entries: 62 us on one SM).
  const int64_t W = (int64_t)gridDim.x * (TILE / 32);
  const int64_t w = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const int chunk = nh >= W * CNT_CHUNK ? CNT_CHUNK : CNT_CHUNK_MIN;
  const int64_t nchunks = (nh + chunk - 1) / chunk;
  const int64_t qend = w < nchunks ? ((nchunks - 1 - w) / W + 1) * chunk : 0;
  int64_t next = 0;  // queue position (warp-uniform)
  // lane state
  int state = LS_IDLE;
  int64_t h = 0, N = 0, k = 0;
  uint32_t cnt = 0, wy = 0;
  Real px = 0, py = 0, pz = 1, g = 1, chi = 0, dts = 0, nx = 0, ny = 0, nz = 0;
  Real E[3] = {0, 0, 0}, B[3] = {0, 0, 0};
  uint64_t pid = 0;
  RateOut<Real> ro{(Real)0, (Real)-1e30, (Real)0};
  // Methods II/III: the particle's species, index and the word for its next r3
  int psi = 0;
  int64_t pi = 0;
  uint32_t w3 = 0;
  auto finish = [&]() {
    tl.events += cnt;
    A.sub_cnt[h] = cnt;
    if (h < rc) A.sub_gf[h] = g;
    if (A.C.generator != GEN_METHOD_I) {  // P_cum restarts with a fresh r3 (word 2)
      A.sp[psi].od_p[pi] = (Real)0;
      A.sp[psi].od_r[pi] = unif<Real>(w3);
    }
    state = LS_IDLE;
  };
  for (;;) {
    const unsigned idle = __ballot_sync(0xFFFFFFFFu, state == LS_IDLE);
    const unsigned pend = __ballot_sync(0xFFFFFFFFu, state == LS_PEND);
    const unsigned scan = __ballot_sync(0xFFFFFFFFu, state == LS_SCAN);
    const bool more = next < qend;
    // one phase per round, run by every lane in that state: emission once
    // enough lanes wait for it, refills once enough lanes are idle, else
    // draws; the fall-backs guarantee progress
    int phase;
    if (__popc(pend) >= A.emit_lanes) phase = LS_PEND;
    else if (more && __popc(idle) >= CNT_MIN_INIT) phase = LS_IDLE;
    else if (scan) phase = LS_SCAN;
    else if (pend) phase = LS_PEND;
    else if (more && idle) phase = LS_IDLE;
    else break;
    if (phase == LS_IDLE) {
      // refill: the idle lanes take the next queue positions, in lane order
      if (state == LS_IDLE) {
        const int64_t q = next + __popc(idle & lt_mask);
        const int64_t hr = q < qend ? (w + (q / chunk) * W) * chunk + (q % chunk) : nh;
        if (hr < nh) {
          h = nh - 1 - hr;
          Entry<Real> P;
          load_entry<Real, FM, MODE>(A, A.heavy_list[begin + h], T0, dt, P);
          px = P.px; py = P.py; pz = P.pz; g = P.g;
#pragma unroll
          for (int c = 0; c < 3; ++c) { E[c] = P.E[c]; B[c] = P.B[c]; }
          pid = P.id;
          unit_dir(P, nx, ny, nz);
          chi = chi_lepton(px, py, pz, g, E[0], E[1], E[2], B[0], B[1], B[2], inv_aS);
          ro = photon_rate(sR, sF, A.T, A.C, chi, g, tl);
          k = 0;
          cnt = 0;
          if (A.C.generator != GEN_METHOD_I) {
            // Methods II/III: the streaming pass found the event; one photon,
            // its xi from word 1 of the step's emission draw
            const U4 r = draw(A.C, pid, step_, 0, STREAM_EMIT);
            N = 1;
            dts = dt;
            wy = r.y;
            w3 = r.z;
            psi = P.si;
            pi = P.i;
            tl.substeps += 1;
            state = LS_PEND;
          } else {
            N = substep_count(A.C, ro.W, dt, wdt_max, tl.status);
            tl.substeps += N;
            dts = dt / (Real)N;
            state = LS_SCAN;
          }
        }
      }
      next += __popc(idle);
    } else if (phase == LS_SCAN) {
      // Method I draws until an event or the last sub-step; one Philox call
      // gives the words of two sub-steps (2j and 2j+1)
      if (state == LS_SCAN) {
        const Real thr = ro.W * dts;
        for (int s = 0; s < A.scan_draws; s += 2) {
          const U4 r = draw(A.C, pid, step_, k >> 1, STREAM_EMIT);
          if (!(k & 1)) {
            if (thr > unif<Real>(r.x)) { wy = r.y; state = LS_PEND; break; }
            if (++k >= N) { finish(); break; }
          }
          if (thr > unif<Real>(r.z)) { wy = r.w; state = LS_PEND; break; }
          if (++k >= N) { finish(); break; }
        }
      }
    } else {
      // emission, by every lane with an event: kappa from r2 (Eq. 7), then
      // ln delta from the inverse table -- or, for a particle with N = 1 in a
      // context with the learned sampler, from the network (a warp-collective
      // call, made by every lane, only in rounds where some lane needs it)
      const bool ev = state == LS_PEND;
      const Real kap = ev ? photon_kappa(ro.kmin, unif<Real>(wy), unif<Real>(~wy)) : (Real)0;
      Real Y = (Real)0;
      bool in_mlp = false;
      if (use_mlp && __any_sync(0xFFFFFFFFu, ev && N == 1)) {
        const float lchi = chi > (Real)0 ? (float)m_log(chi) : MLP_L_LO - 1.0f;
        in_mlp = ev && N == 1 && lchi >= MLP_L_LO && lchi <= MLP_L_HI && (float)kap >= MLP_K_LO &&
                 (float)kap <= MLP_K_HI;
        const float zz = mlp_infer_warp(s_frag, s_fw, (lchi - MLP_LC) / MLP_LS,
                                        ((float)kap - MLP_KC) / MLP_KS);
        Y = (Real)(zz + mlp_baseline((float)kap));
      }
      if (ev) {
        if (!in_mlp) Y = photon_lndelta_table(A.T.Y, A.T, ro.l, kap, tl);
        XiOut<Real> xo = xi_from_lndelta(chi, Y);
        Real g2 = g * xo.omxi, eph = g * xo.xi;
        if (g2 < (Real)1) { g2 = (Real)1; eph = g - (Real)1; }
        if (cnt < REC && h < rc) {
          A.rec_e[cnt * rc + h] = eph;
          A.rec_k[cnt * rc + h] = (uint32_t)k;
        }
        ++cnt;
        int b = spec_bin(A.C, eph);
        {  // one shared atomic per distinct bin among the emitting lanes
          const unsigned em = __activemask();
          const unsigned same = __match_any_sync(em, b);
          if (b >= 0 && lane == __ffs(same) - 1) atomicAdd(&bt.hist[b], (unsigned long long)__popc(same));
        }
        Real pm2 = m_sqrt((g2 - (Real)1) * (g2 + (Real)1));
        px = pm2 * nx; py = pm2 * ny; pz = pm2 * nz;
        g = g2;
        if (++k >= N) {
          finish();
        } else {  // the rate for the remaining sub-steps
          chi = chi_lepton(px, py, pz, g, E[0], E[1], E[2], B[0], B[1], B[2], inv_aS);
          ro = photon_rate(sR, sF, A.T, A.C, chi, g, tl);
          state = LS_SCAN;
        }
      }
    }
  }
  tally_flush(&bt, tl);
  __syncthreads();
  block_tally_commit(&bt, A.o.cnt, 0);
}

// Writing pass, warp-cooperative: a warp takes 32 consecutive entries; each
// lane stores its own particle's final state, and then the warp's photons are
// written by consecutive lanes -- one photon per lane, its parent's data
// fetched by shuffles -- so the 15 per-photon stores (state, id, alive flag,
// fields) are coalesced and every lane has a photon to write.  Particles whose
// photons are not all recorded are listed for the replay launch
// (k_substep_replay).
template <class Real, int FM, int MODE>
__global__ void __launch_bounds__(TILE, sizeof(Real) == 4 ? 4 : 2) k_substep_write_coop(LeptonArgs<Real> A) {
  const int64_t step_ = A.d_step ? *A.d_step : A.step;
  __shared__ uint8_t s_parent[TILE / 32][32 * REC];  // warp photon -> parent lane
  __shared__ long long s_meta[4];
  __shared__ BlockTally bt;
  block_tally_init(&bt);
  if (threadIdx.x == 0) {
    s_meta[0] = *(volatile int64_t *)A.sp[0].d_n;
    s_meta[1] = A.cls_off[NCLS];
    s_meta[2] = A.sub_meta[0];  // photons of all entries
    s_meta[3] = A.sub_meta[1];  // photon count before them
  }
  __syncthreads();
  const int64_t T0 = (s_meta[0] + TILE - 1) / TILE;
  const int64_t nh = s_meta[1];
  const uint32_t total = (uint32_t)s_meta[2];
  const int64_t nph = s_meta[3];
  const Real dt = sel<Real>(A.C.dt, A.C.f_dt);
  const int64_t rc = A.rec_cap;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint8_t *par = s_parent[wid];
  Tally tl;
  tl.clear();
  const int64_t nwarps = (int64_t)gridDim.x * (TILE / 32);
  for (int64_t wb = (blockIdx.x * (int64_t)(TILE / 32) + wid) * 32; wb < nh; wb += nwarps * 32) {
    const int64_t h = wb + lane;
    const bool act = h < nh;
    uint32_t off = 0, cnt = 0;
    int32_t e = 0;
    if (act) {
      off = A.sub_cnt[h];  // exclusive prefix of the counts now
      cnt = (h + 1 < nh ? A.sub_cnt[h + 1] : total) - off;
      e = A.heavy_list[h];
    }
    const bool rep = act && cnt > 0 && (cnt > REC || h >= rc);
    if (rep) A.replay_list[atomicAdd(A.replay_n, 1u)] = (int32_t)h;
    const uint32_t mine = (act && !rep) ? cnt : 0u;  // photons this lane's entry gives the warp
    // the particle: staged with no photon needs nothing (the streaming pass
    // stored it); otherwise its final state is stored here
    Entry<Real> P;
    P.x = P.y = P.z = P.px = P.py = P.w = (Real)0;
    P.pz = P.g = (Real)1;
#pragma unroll
    for (int c = 0; c < 3; ++c) { P.E[c] = (Real)0; P.B[c] = (Real)0; }
    P.id = 0;
    P.tag = 0;
    Real nx = 0, ny = 0, nz = 0;
    const bool need = act && !rep && (cnt > 0 || e < 0);
    if (need) {
      Real gfin = (Real)0;
      if (cnt > 0) gfin = A.sub_gf[h];
      load_entry<Real, FM, MODE>(A, e, T0, dt, P);
      unit_dir(P, nx, ny, nz);
      store_entry<Real, MODE>(A, P, cnt > 0 ? gfin : P.g, nx, ny, nz);
    }
    // the warp's photons, in entry order
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += v;
    }
    const uint32_t excl = incl - mine;
    const uint32_t T = __shfl_sync(0xFFFFFFFFu, incl, 31);
    for (uint32_t j = 0; j < mine; ++j) par[excl + j] = (uint8_t)lane;
    __syncwarp();
    for (uint32_t q0 = 0; q0 < T; q0 += 32) {
      const uint32_t q = q0 + lane;
      const bool valid = q < T;
      const int L = valid ? par[q] : 0;
      // the parent's data, by shuffles (every lane takes part)
      const Real x = __shfl_sync(0xFFFFFFFFu, P.x, L), y = __shfl_sync(0xFFFFFFFFu, P.y, L),
                 z = __shfl_sync(0xFFFFFFFFu, P.z, L);
      const Real ux = __shfl_sync(0xFFFFFFFFu, nx, L), uy = __shfl_sync(0xFFFFFFFFu, ny, L),
                 uz = __shfl_sync(0xFFFFFFFFu, nz, L);
      const Real w = __shfl_sync(0xFFFFFFFFu, P.w, L);
      Real E[3], B[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        E[c] = __shfl_sync(0xFFFFFFFFu, P.E[c], L);
        B[c] = __shfl_sync(0xFFFFFFFFu, P.B[c], L);
      }
      const uint64_t pid = (uint64_t)__shfl_sync(0xFFFFFFFFu, (unsigned long long)P.id, L);
      const uint32_t ptag = __shfl_sync(0xFFFFFFFFu, P.tag, L);
      const uint32_t poff = __shfl_sync(0xFFFFFFFFu, off, L);
      const uint32_t pex = __shfl_sync(0xFFFFFFFFu, excl, L);
      const int64_t ph = wb + L;
      if (!valid) continue;
      const uint32_t j = q - pex;  // the parent's j-th photon
      const Real eph = A.rec_e[j * rc + ph];
      const int64_t kk = A.rec_k[j * rc + ph];
      const int64_t out = nph + (int64_t)poff + j;
      if (out >= A.ph.cap) {
        tl.dropped += 1;
        tl.status |= QED_STATUS_CAPACITY;
        continue;
      }
      const U4 cid = draw(A.C, pid, step_, kk, STREAM_PHOTON_ID);
      write_child(A.ph, out, x, y, z, eph * ux, eph * uy, eph * uz, w,
                  (uint64_t)cid.x | ((uint64_t)cid.y << 32), E, B, ptag);
    }
    __syncwarp();  // par is rewritten by the next window
  }
  tally_flush(&bt, tl);
  __syncthreads();
  block_tally_commit(&bt, A.o.cnt, 0);
}

// Exclusive scan, in place, of the sub-step entries' photon counts (single
// pass, decoupled look-back over 4096-entry tiles).  The total and the photon
// count at launch go to sub_meta[0] and sub_meta[1]; the last tile publishes
// the new photon count.
struct SubScanArgs {
  uint32_t *cnt;
  unsigned int *replay_n;  // reset here for the writing pass
  const int64_t *n_entries;
  int64_t *sub_meta;       // [0] total, [1] photon count before
  int64_t *out_n;          // the photon count, advanced by the total
  int64_t out_cap;
  Out o;
};
constexpr int SCAN_ITEMS = 16;

__global__ void __launch_bounds__(TILE) k_sub_scan(SubScanArgs A) {
  __shared__ uint32_t scan_sm[33];
  __shared__ long long s_meta[6];
  if (threadIdx.x == 0) {
    s_meta[2] = *(volatile const int64_t *)A.n_entries;
    s_meta[3] = *(volatile int64_t *)A.out_n;
    s_meta[4] = (long long)A.o.scan.sync[2];
  }
  __syncthreads();
  const int64_t nh = s_meta[2], nph = s_meta[3];
  const uint32_t epoch = (uint32_t)s_meta[4];
  const int64_t per_tile = (int64_t)TILE * SCAN_ITEMS;
  const int64_t ntiles = (nh + per_tile - 1) / per_tile;
  uint32_t status = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *A.replay_n = 0u;
    if (ntiles == 0) {
      A.sub_meta[0] = 0;
      A.sub_meta[1] = nph;
    }
  }
  for (;;) {
    if (threadIdx.x == 0) s_meta[0] = (long long)atomicAdd(&A.o.scan.sync[0], 1u);
    __syncthreads();
    const int64_t t = s_meta[0];
    __syncthreads();
    if (t >= ntiles) break;
    const int64_t first = t * per_tile + (int64_t)threadIdx.x * SCAN_ITEMS;
    uint32_t v[SCAN_ITEMS];
    uint32_t sum = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
      v[j] = first + j < nh ? A.cnt[first + j] : 0u;
      sum += v[j];
    }
    const uint32_t excl = block_excl_scan(sum, scan_sm);
    const uint32_t agg = scan_sm[32];
    if (threadIdx.x < 32) {
      const uint32_t pre = lookback_warp(A.o.scan, t, epoch, agg, status);
      if (threadIdx.x == 0) {
        s_meta[1] = pre;
        if (t == ntiles - 1) {
          const int64_t tot = (int64_t)pre + agg;
          A.sub_meta[0] = tot;
          A.sub_meta[1] = nph;
          *A.out_n = nph + tot < A.out_cap ? nph + tot : A.out_cap;
        }
      }
    }
    __syncthreads();
    uint32_t run = (uint32_t)s_meta[1] + excl;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
      if (first + j < nh) A.cnt[first + j] = run;
      run += v[j];
    }
  }
  if (threadIdx.x == 0 && status) atomicOr(&A.o.cnt->status, status);
  launch_epilogue(A.o.scan, epoch);
}

// Replay launch of the writing pass: the particles k_substep_write_coop listed
// (more than REC photons, or past the record capacity, both rare) redo their
// emission chains -- same draws, same tables -- and write their photons and
// final momenta.  It is separate so that the common case carries neither the
// tables nor the chain's registers, and dense, so that the rare long replays
// share warps.  BY_SLOT: the list is of slots, leptons of the single pass
// whose momentum (with grid fields also position) is stored as before the
// step; sub_cnt is per slot then, and rec_k holds the photons of every list entry.
template <class Real, int FM, int MODE, bool BY_SLOT>
__global__ void __launch_bounds__(TILE, 2) k_substep_replay(LeptonArgs<Real> A) {
  const int64_t step_ = A.d_step ? *A.d_step : A.step;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr bool kSmem = sizeof(Real) == 4;
  Real *sR = kSmem ? reinterpret_cast<Real *>(smem_raw) : const_cast<Real *>(A.T.R);
  Real *sF = kSmem ? sR + A.T.gl.n : const_cast<Real *>(A.T.F);
  __shared__ long long s_meta[4];
  __shared__ BlockTally bt;
  // a block with nothing to replay leaves before staging the tables
  const int64_t n_iter = (int64_t)*(volatile unsigned int *)A.replay_n;
  if ((int64_t)blockIdx.x * TILE >= n_iter) return;
  if (kSmem) {
    load_tables_smem(sR, A.T.R, A.T.gl.n);
    load_tables_smem(sF, A.T.F, A.T.gl.n * A.T.gy.n);
  }
  block_tally_init(&bt);
  if (threadIdx.x == 0) {
    s_meta[0] = *(volatile int64_t *)A.sp[0].d_n;
    s_meta[1] = BY_SLOT ? 0 : A.cls_off[NCLS];
    s_meta[2] = A.sub_meta[0];  // photons of all entries
    s_meta[3] = A.sub_meta[1];  // photon count before them
  }
  __syncthreads();
  const int64_t T0 = (s_meta[0] + TILE - 1) / TILE;
  const int64_t nh = s_meta[1];
  const uint32_t total = (uint32_t)s_meta[2];
  const int64_t nph = s_meta[3];
  const Real inv_aS = sel<Real>(A.C.inv_aS, A.C.f_inv_aS);
  const Real dt = sel<Real>(A.C.dt, A.C.f_dt);
  const Real wdt_max = sel<Real>(A.C.wdt_max, A.C.f_wdt_max);
  Tally tl;
  tl.clear();
  for (int64_t q = blockIdx.x * (int64_t)TILE + threadIdx.x; q < n_iter; q += (int64_t)gridDim.x * TILE) {
    const int64_t h = (int64_t)A.replay_list[q];
    // sub_cnt holds the exclusive prefix of the counts now
    const uint32_t off = A.sub_cnt[h];
    // the photons the lepton has places for (by slot: as the single pass counted them)
    const uint32_t cnt = BY_SLOT ? A.rec_k[q] : (h + 1 < nh ? A.sub_cnt[h + 1] : total) - off;
    const int32_t e = BY_SLOT ? -(int32_t)h - 1 : A.heavy_list[h];
    const int64_t out0 = nph + (int64_t)off;
    Entry<Real> P;
    load_entry<Real, FM, MODE>(A, e, T0, dt, P);
    if (BY_SLOT && MODE != MODE_EMIT && FM != FM_GRID) {  // its stored position is the pushed one already
      const Sp<Real> &S = A.sp[P.si];
      P.x = S.x[P.i]; P.y = S.y[P.i]; P.z = S.z[P.i];
    }
    Real nx, ny, nz;
    unit_dir(P, nx, ny, nz);
    Real g = P.g;
    auto put = [&](uint32_t j, Real eph, int64_t kk) {
      const int64_t out = out0 + j;
      if (out >= A.ph.cap) {
        if (!BY_SLOT) {  // (by slot: the scan counted them)
          tl.dropped += 1;
          tl.status |= QED_STATUS_CAPACITY;
        }
        return;
      }
      U4 cid = draw(A.C, P.id, step_, kk, STREAM_PHOTON_ID);
      write_child(A.ph, out, P.x, P.y, P.z, eph * nx, eph * ny, eph * nz, P.w,
                  (uint64_t)cid.x | ((uint64_t)cid.y << 32), P.E, P.B, P.tag);
    };
    // the chain again (its counters went to the counting pass's tally)
    Tally dummy;
    dummy.clear();
    const Real *E = P.E, *B = P.B;
    Real chi = chi_lepton(P.px, P.py, P.pz, g, E[0], E[1], E[2], B[0], B[1], B[2], inv_aS);
    RateOut<Real> ro = photon_rate(sR, sF, A.T, A.C, chi, g, dummy);
    const bool forced = A.C.generator != GEN_METHOD_I;  // Methods II/III: one photon at k = 0
    const int64_t N = forced ? 1 : substep_count(A.C, ro.W, dt, wdt_max, dummy.status);
    const Real dts = dt / (Real)N;
    uint32_t j = 0;
    for (int64_t kk = 0; kk < N && j < cnt; ++kk) {
      const EmitWords r = emit_words(A.C, P.id, step_, kk);
      if (!forced && !(ro.W * dts > unif<Real>(r.r1))) continue;
      XiOut<Real> xo = photon_xi(A.T.Y, A.T, ro.l, chi, ro.kmin, unif<Real>(r.r2), unif<Real>(~r.r2), dummy);
      Real g2 = g * xo.omxi, eph = g * xo.xi;
      if (g2 < (Real)1) { g2 = (Real)1; eph = g - (Real)1; }
      put(j++, eph, kk);
      Real pm2 = m_sqrt((g2 - (Real)1) * (g2 + (Real)1));
      g = g2;
      chi = chi_lepton(pm2 * nx, pm2 * ny, pm2 * nz, g, E[0], E[1], E[2], B[0], B[1], B[2], inv_aS);
      ro = photon_rate(sR, sF, A.T, A.C, chi, g, dummy);
    }
    if (j != cnt) {  // the replay disagreed with the count: zero-energy photons fill the slots
      tl.status |= QED_STATUS_REPLAY;
      for (; j < cnt; ++j) put(j, (Real)0, 0);
    }
    store_entry<Real, MODE>(A, P, g, nx, ny, nz);
  }
  tally_flush(&bt, tl);
  __syncthreads();
  block_tally_commit(&bt, A.o.cnt, 0);
}

// ---------------------------------------------------------------------------
// Class list of the streaming pass's flagged leptons: one ordered list,
// class-major (all class-1 slots in slot order, then class 2, ..., class 5),
// built by a count, a scan and a scatter pass -- no CTA waits on another.
// off[c - 1] is the first list position of class c and off[NCLS] the length.
// Flags are read 8 per thread (one 8-byte load), 2048 per chunk; a chunk's
// per-class counts (<= 2048 each) are packed 12 bits per class in a uint64.
// ---------------------------------------------------------------------------
constexpr int CLS_ITEMS = 8;
constexpr int CLS_CHUNK = TILE * CLS_ITEMS;
static_assert(CLS_CHUNK == CLS_CHUNK_FLAGS, "class-list chunk size");
constexpr int CLS_SCAN_THREADS = 1024;
constexpr int CLS_SCAN_PER_THREAD = 8;  // chunks per thread per round of the scan

struct ClassListArgs {
  const uint8_t *flags;
  const int64_t *n0, *n1;  // species counts (size the streaming pass's slot range)
  int *list;
  unsigned long long *chunk_cnt;  // [chunks] packed per-class counts
  uint32_t *chunk_off;            // [chunks][NCLS] first list position per class
  int64_t *off;                   // [NCLS + 1]
  const int32_t *stage_idx;       // [slot] staging record of a flagged slot (-1: none)
  unsigned int *stage_n;          // staging counter, reset by the scan for the next step
  qed_counters *cnt;              // deferred += list length
};

__device__ __forceinline__ int64_t cls_nslots(const ClassListArgs &A) {
  const int64_t n0 = *(volatile const int64_t *)A.n0;
  const int64_t n1 = A.n1 ? *(volatile const int64_t *)A.n1 : 0;
  return ((n0 + TILE - 1) / TILE + (n1 + TILE - 1) / TILE) * TILE;
}

// This thread's 8 flags of chunk c and their packed per-class counts.  The
// slot range is a multiple of TILE, so a group of 8 is all in or all out.
__device__ __forceinline__ unsigned long long cls_load(const ClassListArgs &A, int64_t c,
                                                       int64_t nslots, uint2 &raw) {
  const int64_t first = c * CLS_CHUNK + (int64_t)threadIdx.x * CLS_ITEMS;
  raw = make_uint2(0u, 0u);
  if (first < nslots) raw = *reinterpret_cast<const uint2 *>(A.flags + first);
  const uint8_t *fl = reinterpret_cast<const uint8_t *>(&raw);
  unsigned long long packed = 0;
#pragma unroll
  for (int j = 0; j < CLS_ITEMS; ++j)
    if (fl[j] >= 1 && fl[j] <= NCLS) packed += 1ull << (12 * (fl[j] - 1));
  return packed;
}

// Block-wide exclusive scan of a uint64 per thread; sm needs 33 words and
// receives the block total in sm[32].
__device__ __forceinline__ unsigned long long block_excl_scan64(unsigned long long v,
                                                               unsigned long long *sm) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned long long incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    unsigned long long u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) sm[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    unsigned long long w = lane < nw ? sm[lane] : 0ull, wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      unsigned long long u = __shfl_up_sync(0xFFFFFFFFu, wi, o);
      if (lane >= o) wi += u;
    }
    if (lane < nw) sm[lane] = wi - w;
    if (lane == nw - 1) sm[32] = wi;
  }
  __syncthreads();
  const unsigned long long r = sm[wid] + incl - v;
  __syncthreads();
  return r;
}

__device__ __forceinline__ uint32_t cls_field(unsigned long long p, int c) {
  return (uint32_t)(p >> (12 * c)) & 0xFFFu;
}

__global__ void __launch_bounds__(TILE) k_cls_count(ClassListArgs A) {
  __shared__ unsigned long long sm[33];
  const int64_t nslots = cls_nslots(A);
  const int64_t nchunks = (nslots + CLS_CHUNK - 1) / CLS_CHUNK;
  for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
    uint2 raw;
    const unsigned long long p = cls_load(A, c, nslots, raw);
    block_excl_scan64(p, sm);
    if (threadIdx.x == 0) A.chunk_cnt[c] = sm[32];
  }
}

// One CTA: class totals, class starts, and every chunk's per-class offset.
__global__ void __launch_bounds__(CLS_SCAN_THREADS) k_cls_scan(ClassListArgs A) {
  __shared__ unsigned long long tot[NCLS];
  __shared__ unsigned long long sm[33];
  __shared__ int64_t base[NCLS];
  const int64_t nslots = cls_nslots(A);
  const int64_t nchunks = (nslots + CLS_CHUNK - 1) / CLS_CHUNK;
  if (threadIdx.x < NCLS) tot[threadIdx.x] = 0;
  if (threadIdx.x == 0) *A.stage_n = 0u;  // the streaming pass of this step is done with it
  __syncthreads();
  unsigned long long mine[NCLS] = {0, 0, 0, 0, 0};
  for (int64_t c = threadIdx.x; c < nchunks; c += blockDim.x) {
    const unsigned long long p = A.chunk_cnt[c];
#pragma unroll
    for (int k = 0; k < NCLS; ++k) mine[k] += cls_field(p, k);
  }
#pragma unroll
  for (int k = 0; k < NCLS; ++k) {
    unsigned long long v = mine[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(&tot[k], v);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int64_t b = 0;
    for (int k = 0; k < NCLS; ++k) {
      base[k] = b;
      A.off[k] = b;
      b += (int64_t)tot[k];
    }
    A.off[NCLS] = b;
    if (b) atomicAdd(reinterpret_cast<unsigned long long *>(&A.cnt->deferred), (unsigned long long)b);
  }
  __syncthreads();
  // per-class running prefix over chunks; each round a thread takes
  // CLS_SCAN_PER_THREAD consecutive chunks.  A round's prefixes stay below
  // 2^25 per class (2048 * 8 * 1024), so two classes share a packed scan.
  int64_t carry[NCLS];
#pragma unroll
  for (int k = 0; k < NCLS; ++k) carry[k] = base[k];
  const int64_t per_round = (int64_t)blockDim.x * CLS_SCAN_PER_THREAD;
  for (int64_t r0 = 0; r0 < nchunks; r0 += per_round) {
    const int64_t c0 = r0 + (int64_t)threadIdx.x * CLS_SCAN_PER_THREAD;
    uint32_t t[NCLS + 1] = {0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < CLS_SCAN_PER_THREAD; ++j) {
      const int64_t c = c0 + j;
      if (c < nchunks) {
        const unsigned long long p = A.chunk_cnt[c];
#pragma unroll
        for (int k = 0; k < NCLS; ++k) t[k] += cls_field(p, k);
      }
    }
    uint32_t run[NCLS + 1], rtot[NCLS + 1];
#pragma unroll
    for (int q = 0; q < (NCLS + 1) / 2; ++q) {
      const unsigned long long v = (unsigned long long)t[2 * q] | ((unsigned long long)t[2 * q + 1] << 32);
      const unsigned long long e = block_excl_scan64(v, sm), tt = sm[32];
      run[2 * q] = (uint32_t)e;
      run[2 * q + 1] = (uint32_t)(e >> 32);
      rtot[2 * q] = (uint32_t)tt;
      rtot[2 * q + 1] = (uint32_t)(tt >> 32);
    }
#pragma unroll
    for (int j = 0; j < CLS_SCAN_PER_THREAD; ++j) {
      const int64_t c = c0 + j;
      if (c < nchunks) {
        const unsigned long long p = A.chunk_cnt[c];
#pragma unroll
        for (int k = 0; k < NCLS; ++k) {
          A.chunk_off[c * NCLS + k] = (uint32_t)(carry[k] + run[k]);
          run[k] += cls_field(p, k);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < NCLS; ++k) carry[k] += (int64_t)rtot[k];
  }
}

__global__ void __launch_bounds__(TILE) k_cls_scatter(ClassListArgs A) {
  __shared__ unsigned long long sm[33];
  const int64_t nslots = cls_nslots(A);
  const int64_t nchunks = (nslots + CLS_CHUNK - 1) / CLS_CHUNK;
  for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
    uint2 raw;
    const unsigned long long p = cls_load(A, c, nslots, raw);
    unsigned long long ex = block_excl_scan64(p, sm);
    if (!p) continue;
    const uint8_t *fl = reinterpret_cast<const uint8_t *>(&raw);
    const int64_t first = c * CLS_CHUNK + (int64_t)threadIdx.x * CLS_ITEMS;
#pragma unroll
    for (int j = 0; j < CLS_ITEMS; ++j) {
      const int k = (int)fl[j] - 1;
      if (k < 0 || k >= NCLS) continue;
      // list entry: the staging record, or -(slot + 1) for an unstaged slot
      const int32_t sidx = A.stage_idx[first + j];
      A.list[A.chunk_off[c * NCLS + k] + cls_field(ex, k)] = sidx >= 0 ? sidx : -(int32_t)(first + j) - 1;
      ex += 1ull << (12 * k);
    }
  }
}

// ---------------------------------------------------------------------------
// Stable in-place compaction of dead particles (alive == 0): the live particles
// of every tile are counted (from the flags alone), the counts scanned, and the
// tiles moved.  The warps of a moving tile read its particles into registers and
// publish that; the tile then waits until the tiles whose range it writes to --
// at most two, which lie before it by the particles dead so far -- have published
// too, and writes: no word is overwritten before it has been read.  Tiles are
// taken in order, so the ones waited for are under way, and have mostly published
// by the time this tile's own words arrive.  The wait is bounded.  (8.4M photons
// of 61 bytes, one in ten dead: 268 us with the positions from a look-back, which
// had each tile wait for the sums of all before it, one 2048-particle tile of
// 1024 threads in flight per SM; 198 with counts and a scan of their own launch,
// and the CTA's barrier before it published; 185 this way, 135 at the copy
// rate.  900,000: 31 -> 28 us.)
// ---------------------------------------------------------------------------
constexpr int COMPACT_THREADS = 256;
template <class Real> __host__ __device__ constexpr int compact_items() { return sizeof(Real) == 4 ? 2 : 1; }
template <class Real> __host__ __device__ constexpr int compact_tile() { return COMPACT_THREADS * compact_items<Real>(); }

template <class Real> struct CompactArgs {
  Sp<Real> s;
  uint32_t *off;        // [tile] live particles, then its first one's destination
  uint32_t *read;       // [tile] warps whose part of the tile is in registers
  uint32_t *total;      // live particles
  uint32_t *one;        // [COMPACT_ONE] the single launch: live particles + 1 (zero between calls)
  uint32_t *group;      // [COMPACT_ONE / 32] live particles and, from bit 20, tiles of 32 (zero between calls)
  unsigned int *ticket; // [0] tiles taken, [1] CTAs done, [2] waits that ran out, [3] counting CTAs done (zero between calls)
  qed_counters *cnt;
};

// nonzero bytes of a word
__device__ __forceinline__ uint32_t live_bytes(uint32_t w) { return (uint32_t)__popc(__vsetne4(w, 0u)); }

// Eight words at a 32-byte boundary.
__device__ __forceinline__ void load8(uint32_t (&v)[8], const uint32_t *p) {
  asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "l"(p) : "memory");
}
__device__ __forceinline__ void store8(uint32_t *p, const uint32_t (&v)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]),
               "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}

// The tiles' counts, a warp per tile; the CTA that finishes last scans them, 8
// tiles per thread by one load of 32 bytes (16M photons, 31250 tiles: 29 us with
// a launch of its own for the scan and a word per load, 13 this way).
template <class Real>
__global__ void __launch_bounds__(CLS_SCAN_THREADS) k_compact_count(CompactArgs<Real> A) {
  constexpr int TP = compact_tile<Real>(), PER = TP / 32;  // flags per lane: 16 or 8
  asm volatile("griddepcontrol.launch_dependents;");
  __shared__ uint32_t sm[33];
  __shared__ bool s_last;
  const int64_t n = *(volatile int64_t *)A.s.d_n;
  const int64_t ntiles = (n + TP - 1) / TP;
  const int lane = threadIdx.x & 31;
  const bool aligned = (reinterpret_cast<uintptr_t>(A.s.alive) & 15) == 0;
  for (int64_t t = ((int64_t)blockIdx.x * CLS_SCAN_THREADS + threadIdx.x) >> 5; t < ntiles;
       t += ((int64_t)gridDim.x * CLS_SCAN_THREADS) >> 5) {
    const int64_t first = t * TP + lane * PER;
    uint32_t c = 0;
    if (aligned && first + PER <= n) {
      const uint2 *p = reinterpret_cast<const uint2 *>(A.s.alive + first);
#pragma unroll
      for (int q = 0; q < PER / 8; ++q) c += live_bytes(p[q].x) + live_bytes(p[q].y);
    } else {
      for (int j = 0; j < PER; ++j) c += first + j < n && A.s.alive[first + j] ? 1u : 0u;
    }
    c = __reduce_add_sync(0xFFFFFFFFu, c);
    if (lane == 0) {
      A.off[t] = c;
      A.read[t] = 0u;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(&A.ticket[3], 1u) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  if (!s_last) return;
  uint32_t carry = 0;
  for (int64_t r0 = 0; r0 < ntiles; r0 += CLS_SCAN_THREADS * 8) {
    const int64_t c0 = r0 + (int64_t)threadIdx.x * 8;
    uint32_t v[8], t = 0;
    if (c0 + 8 <= ntiles) {
      load8(v, A.off + c0);
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = c0 + j < ntiles ? A.off[c0 + j] : 0u;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) t += v[j];
    uint32_t run = carry + block_excl_scan(t, sm);
    carry += sm[32];
    __syncthreads();  // sm[32] is read
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t q = v[j];
      v[j] = run;
      run += q;
    }
    if (c0 + 8 <= ntiles) {
      store8(A.off + c0, v);
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (c0 + j < ntiles) A.off[c0 + j] = v[j];
    }
  }
  if (threadIdx.x == 0) {
    *A.total = carry;
    A.ticket[3] = 0u;
  }
}

__device__ __forceinline__ uint32_t word_hash(float v) { return __float_as_uint(v); }
__device__ __forceinline__ uint32_t word_hash(double v) { return (uint32_t)__double2loint(v) ^ (uint32_t)__double2hiint(v); }

// What a thread holds of a tile.
template <class Real> struct CompactPart {
  static constexpr int CI = compact_items<Real>();
  bool keep[CI];
  Real v[CI][13];
  uint64_t id[CI];
  uint32_t tg[CI];
};

template <class Real>
__device__ __forceinline__ void compact_load(const Sp<Real> &S, int64_t t, int64_t n, CompactPart<Real> &r) {
  const bool fields = S.ex != nullptr;
#pragma unroll
  for (int k = 0; k < r.CI; ++k) {  // (the words do not wait for the flag)
    const int64_t i = t * compact_tile<Real>() + k * COMPACT_THREADS + threadIdx.x;
    r.keep[k] = false;
    r.id[k] = 0;
    r.tg[k] = 0;
#pragma unroll
    for (int q = 0; q < 13; ++q) r.v[k][q] = (Real)0;
    if (i < n) {
      r.keep[k] = S.alive[i];
      r.v[k][0] = S.x[i]; r.v[k][1] = S.y[i]; r.v[k][2] = S.z[i];
      r.v[k][3] = S.px[i]; r.v[k][4] = S.py[i]; r.v[k][5] = S.pz[i]; r.v[k][6] = S.w[i];
      r.id[k] = S.id[i];
      if (S.tag) r.tg[k] = S.tag[i];
      if (fields) {
        r.v[k][7] = S.ex[i]; r.v[k][8] = S.ey[i]; r.v[k][9] = S.ez[i];
        r.v[k][10] = S.bx[i]; r.v[k][11] = S.by[i]; r.v[k][12] = S.bz[i];
      }
    }
  }
}

// The warp's live particles of each item into s_warp; the value is a use of
// every word, which therefore have arrived where it is known.
template <class Real>
__device__ __forceinline__ uint32_t compact_arrived(const CompactPart<Real> &r,
                                                    uint32_t (*s_warp)[COMPACT_THREADS / 32]) {
  uint32_t h = 0;
#pragma unroll
  for (int k = 0; k < r.CI; ++k) {
    const unsigned m = __ballot_sync(0xFFFFFFFFu, r.keep[k]);
    if ((threadIdx.x & 31) == 0) s_warp[k][threadIdx.x >> 5] = __popc(m);
    h ^= (uint32_t)r.id[k] ^ (uint32_t)(r.id[k] >> 32) ^ r.tg[k];
#pragma unroll
    for (int q = 0; q < 13; ++q) h ^= word_hash(r.v[k][q]);
  }
  return h;
}

// The live particles to their places from `off` on.
template <class Real>
__device__ __forceinline__ void compact_store(const Sp<Real> &S, const CompactPart<Real> &r, uint32_t off,
                                              const uint32_t (*s_warp)[COMPACT_THREADS / 32]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const bool fields = S.ex != nullptr;
  uint32_t before = off;
#pragma unroll
  for (int k = 0; k < r.CI; ++k) {
    uint32_t base = before;
#pragma unroll
    for (int w = 0; w < COMPACT_THREADS / 32; ++w) {
      if (w < wid) base += s_warp[k][w];
      before += s_warp[k][w];
    }
    const unsigned m = __ballot_sync(0xFFFFFFFFu, r.keep[k]);
    if (!r.keep[k]) continue;
    const int64_t d = base + __popc(m & ((1u << lane) - 1u));
    S.x[d] = r.v[k][0]; S.y[d] = r.v[k][1]; S.z[d] = r.v[k][2];
    S.px[d] = r.v[k][3]; S.py[d] = r.v[k][4]; S.pz[d] = r.v[k][5]; S.w[d] = r.v[k][6];
    S.id[d] = r.id[k];
    S.alive[d] = 1;
    if (S.tag) S.tag[d] = r.tg[k];
    if (fields) {
      S.ex[d] = r.v[k][7]; S.ey[d] = r.v[k][8]; S.ez[d] = r.v[k][9];
      S.bx[d] = r.v[k][10]; S.by[d] = r.v[k][11]; S.bz[d] = r.v[k][12];
    }
  }
}

// Up to COMPACT_ONE tiles, one per CTA, in one launch: every tile publishes its
// live particles once its words have arrived, for itself and for its group of
// 32 tiles, and one warp adds up those of the groups and tiles before it, whose
// words have then been read as well.  (24,000 FP32 photons: kernel 10 us with the
// look-back, 12 and a launch gap in two launches, 7 this way; 200,000: 13, 15,
// 11; 524,288, the most: 23, 22, 22.  All 256 threads polling the tiles before
// it took 20 for 200,000.)
template <class Real>
__global__ void __launch_bounds__(COMPACT_THREADS, sizeof(Real) == 4 ? 4 : 3) k_compact_small(CompactArgs<Real> A) {
  constexpr int CI = compact_items<Real>(), TP = compact_tile<Real>(), WARPS = COMPACT_THREADS / 32;
  __shared__ uint32_t s_warp[CI][WARPS], s_off, s_tile;
  const int64_t n = *(volatile int64_t *)A.s.d_n;
  const int64_t ntiles = (n + TP - 1) / TP;
  if (threadIdx.x == 0) s_tile = atomicAdd(&A.ticket[0], 1u);
  __syncthreads();
  const int64_t t = s_tile;
  bool gave_up = false;
  if (t < ntiles) {
    CompactPart<Real> r;
    compact_load(A.s, t, n, r);
    __syncthreads_or((int)compact_arrived(r, s_warp));
    uint32_t cnt = 0;
#pragma unroll
    for (int k = 0; k < CI; ++k)
#pragma unroll
      for (int w = 0; w < WARPS; ++w) cnt += s_warp[k][w];
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x, g = (int)t >> 5;
      if (lane == 0) {
        __threadfence();
        *(volatile uint32_t *)&A.one[t] = cnt + 1;
        atomicAdd(&A.group[g], (1u << 20) + cnt);
      }
      uint32_t a = lane < g ? 0u : 32u << 20, o = lane < (t & 31) ? 0u : 1u;
      long long spins = 0;
      while (a >> 20 != 32u || o == 0u) {
        if (lane < g) a = *(volatile uint32_t *)&A.group[lane];
        if (lane < (t & 31)) o = *(volatile uint32_t *)&A.one[(t & ~(int64_t)31) + lane];
        if (++spins > LOOKBACK_SPIN_LIMIT) {
          gave_up = true;
          break;
        }
      }
      __threadfence();
      const uint32_t sum = __reduce_add_sync(0xFFFFFFFFu, (a & 0xFFFFFu) + o - 1u);
      if (lane == 0) s_off = sum;
    }
    gave_up = __syncthreads_or(gave_up) != 0;
    const uint32_t off = s_off;
    if (!gave_up && (off != t * TP || cnt != (t + 1 < ntiles ? TP : n - t * TP))) compact_store(A.s, r, off, s_warp);
    if (t == ntiles - 1 && threadIdx.x == 0) *A.total = off + cnt;
  }
  __syncthreads();
  // the last CTA publishes the count, unless a tile gave up, and leaves zeros
  if (threadIdx.x == 0) {
    if (gave_up) {
      atomicOr(&A.cnt->status, (unsigned)QED_STATUS_TIMEOUT);
      atomicAdd(&A.ticket[2], 1u);
    }
    __threadfence();
    s_tile = atomicAdd(&A.ticket[1], 1u) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  if (!s_tile) return;
  for (int64_t s = threadIdx.x; s < ntiles; s += COMPACT_THREADS) A.one[s] = 0u;
  if (threadIdx.x < COMPACT_ONE / 32) A.group[threadIdx.x] = 0u;
  if (threadIdx.x == 0) {
    if (ntiles > 0 && *(volatile unsigned *)&A.ticket[2] == 0u) *A.s.d_n = *(volatile uint32_t *)A.total;
    A.ticket[0] = A.ticket[1] = A.ticket[2] = 0u;
  }
}

template <class Real>
__global__ void __launch_bounds__(COMPACT_THREADS, sizeof(Real) == 4 ? 4 : 3) k_compact_move(CompactArgs<Real> A) {
  constexpr int CI = compact_items<Real>(), TP = compact_tile<Real>(), WARPS = COMPACT_THREADS / 32;
  __shared__ uint32_t s_warp[2][CI][WARPS];  // (what a tile leaves here alternates between two places)
  __shared__ uint32_t s_tile[2], s_off[2], s_end[2], s_go[2];
  const int lane = threadIdx.x & 31;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the counting pass is done, its results visible
  const int64_t n = *(volatile int64_t *)A.s.d_n;
  const int64_t ntiles = (n + TP - 1) / TP;
  bool gave_up = false;
  // (thread 0) takes a tile
  auto take = [&](int p) {
    const uint32_t t = atomicAdd(&A.ticket[0], 1u);
    s_tile[p] = t;
    if (t < ntiles) {
      s_off[p] = A.off[t];
      s_end[p] = t + 1 < ntiles ? A.off[t + 1] : *A.total;
    }
  };
  if (threadIdx.x == 0) take(0);
  __syncthreads();
  for (int p = 0;; p ^= 1) {
    const int64_t t = s_tile[p];
    if (t >= ntiles) break;
    const uint32_t off = s_off[p], cnt = s_end[p] - off;
    const bool whole = cnt == (uint32_t)(t + 1 < ntiles ? TP : n - t * TP);
    if ((int64_t)off == t * TP && whole) {
      // a tile that stays where it is moves nothing, and none writes into it
      if (threadIdx.x == 0) take(p ^ 1);
      __syncthreads();
      continue;
    }
    CompactPart<Real> r;
    compact_load(A.s, t, n, r);
    // (thread 0, while its words are on their way) the tiles before this one
    // that it writes to: at most two
    const int64_t s0 = off / TP, s1 = cnt ? (int64_t)((off + cnt - 1) / TP) : -1;
    uint32_t f0 = WARPS, f1 = WARPS;
    if (threadIdx.x == 0) {
      if (s0 <= s1 && s0 < t) f0 = *(volatile uint32_t *)&A.read[s0];
      if (s0 < s1 && s1 < t) f1 = *(volatile uint32_t *)&A.read[s1];
    }
    // the warp publishes when its words have arrived
    const uint32_t h = __reduce_or_sync(0xFFFFFFFFu, compact_arrived(r, s_warp[p]));
    if (lane == 0) {
      __threadfence();
      asm volatile("red.relaxed.gpu.global.add.u32 [%0], %1;" ::"l"(A.read + t), "r"(1u), "r"(h) : "memory");
    }
    if (threadIdx.x == 0) {
      // a CTA waits with no other tile in hand, after publishing its own, and
      // only for tiles before it
      uint32_t go = 1;
      for (int64_t s = s0; s <= s1 && s < t; ++s) {
        uint32_t f = s == s0 ? f0 : f1;
        long long spins = 0;
        while (f != WARPS && (f = *(volatile uint32_t *)&A.read[s]) != WARPS)
          if (++spins > LOOKBACK_SPIN_LIMIT) {
            go = 0;
            break;
          }
      }
      __threadfence();
      s_go[p] = go;
      take(p ^ 1);
    }
    __syncthreads();
    if (!s_go[p]) {
      gave_up = true;
      continue;
    }
    compact_store(A.s, r, off, s_warp[p]);
  }
  // the last CTA publishes the count -- unless a tile gave up, and so wrote
  // nothing -- and leaves the counters at zero
  if (threadIdx.x == 0) {
    if (gave_up) {
      atomicOr(&A.cnt->status, (unsigned)QED_STATUS_TIMEOUT);
      atomicAdd(&A.ticket[2], 1u);
    }
    __threadfence();
    if (atomicAdd(&A.ticket[1], 1u) == gridDim.x - 1) {
      __threadfence();
      if (*(volatile unsigned *)&A.ticket[2] == 0u) *A.s.d_n = *A.total;
      A.ticket[0] = A.ticket[1] = A.ticket[2] = 0u;
    }
  }
}

// ---------------------------------------------------------------------------
// Hole-filling compaction.  With a live particles among n, every dead slot
// below a (a hole) receives a live particle from [a, n) (a tail): the k-th
// hole in index order takes the k-th tail in index order.  Only as many
// particles move as there are holes, and every live particle below a keeps
// its index.  Count, scan, hole-list and move passes; no CTA waits on another.
// ---------------------------------------------------------------------------
constexpr int FILL_ITEMS = 8;
constexpr int FILL_CHUNK = TILE * FILL_ITEMS;
static_assert(FILL_CHUNK == CLS_CHUNK_FLAGS, "fill chunks use the class-list scratch");

template <class Real> struct FillArgs {
  Sp<Real> s;
  unsigned long long *chunk_alive;  // [chunks]
  uint32_t *chunk_off;              // [chunks][NCLS]: [0] holes before, [1] tails before
  int64_t *meta;                    // [0] n, [1] a, [2] holes (as many as tails)
  int *holes, *tails;               // their slots in index order
};

// live flags of this thread's 8 slots of chunk c (bit j: slot first + j)
__device__ __forceinline__ uint32_t fill_bits(const uint8_t *alive, int64_t c, int64_t n,
                                              int64_t &first) {
  first = c * FILL_CHUNK + (int64_t)threadIdx.x * FILL_ITEMS;
  uint32_t bits = 0;
  if (first + FILL_ITEMS <= n && (reinterpret_cast<uintptr_t>(alive) & 7) == 0) {
    const uint2 w = *reinterpret_cast<const uint2 *>(alive + first);
#pragma unroll
    for (int j = 0; j < FILL_ITEMS; ++j)
      if ((j < 4 ? w.x >> 8 * j : w.y >> 8 * (j - 4)) & 0xFFu) bits |= 1u << j;
    return bits;
  }
#pragma unroll
  for (int j = 0; j < FILL_ITEMS; ++j)
    if (first + j < n && alive[first + j]) bits |= 1u << j;
  return bits;
}

template <class Real>
__global__ void __launch_bounds__(TILE) k_fill_count(FillArgs<Real> A) {
  __shared__ uint32_t scan_sm[33];
  const int64_t n = *(volatile const int64_t *)A.s.d_n;
  const int64_t nchunks = (n + FILL_CHUNK - 1) / FILL_CHUNK;
  for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
    int64_t first;
    const uint32_t bits = fill_bits(A.s.alive, c, n, first);
    block_excl_scan(__popc(bits), scan_sm);
    if (threadIdx.x == 0) A.chunk_alive[c] = scan_sm[32];
    __syncthreads();
  }
}

// One CTA: a, the boundary chunk's split, and each chunk's hole and tail offsets.
__global__ void __launch_bounds__(CLS_SCAN_THREADS) k_fill_scan(const uint8_t *alive,
                                                                 int64_t *d_n,
                                                                 FillArgs<float> A) {
  __shared__ unsigned long long tot;
  __shared__ unsigned long long sm[33];
  __shared__ uint32_t xs;
  const int64_t n = *(volatile const int64_t *)d_n;
  const int64_t nchunks = (n + FILL_CHUNK - 1) / FILL_CHUNK;
  if (threadIdx.x == 0) { tot = 0; xs = 0; }
  __syncthreads();
  unsigned long long mine = 0;
  for (int64_t c = threadIdx.x; c < nchunks; c += blockDim.x) mine += A.chunk_alive[c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xFFFFFFFFu, mine, o);
  if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&tot, mine);
  __syncthreads();
  const int64_t a = (int64_t)tot;
  // live particles of the boundary chunk below a
  const int64_t cb = a / FILL_CHUNK, b0 = cb * FILL_CHUNK;
  uint32_t xl = 0;
  for (int64_t i = b0 + threadIdx.x; i < a; i += blockDim.x) xl += alive[i] ? 1u : 0u;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) xl += __shfl_xor_sync(0xFFFFFFFFu, xl, o);
  if ((threadIdx.x & 31) == 0 && xl) atomicAdd(&xs, xl);
  __syncthreads();
  const uint32_t x = xs;
  if (threadIdx.x == 0) {
    A.meta[0] = n;
    A.meta[1] = a;
    *d_n = a;
  }
  int64_t carry_h = 0, carry_t = 0;
  const int64_t per_round = (int64_t)blockDim.x * CLS_SCAN_PER_THREAD;
  for (int64_t r0 = 0; r0 < nchunks; r0 += per_round) {
    const int64_t c0 = r0 + (int64_t)threadIdx.x * CLS_SCAN_PER_THREAD;
    uint32_t hv[CLS_SCAN_PER_THREAD], tv[CLS_SCAN_PER_THREAD];
    uint32_t hs = 0, ts = 0;
#pragma unroll
    for (int j = 0; j < CLS_SCAN_PER_THREAD; ++j) {
      const int64_t c = c0 + j;
      hv[j] = tv[j] = 0;
      if (c < nchunks) {
        const int64_t lo = c * FILL_CHUNK, hi = lo + FILL_CHUNK < n ? lo + FILL_CHUNK : n;
        const uint32_t al = (uint32_t)A.chunk_alive[c];
        if (hi <= a) {
          hv[j] = (uint32_t)(hi - lo) - al;
        } else if (lo >= a) {
          tv[j] = al;
        } else {
          hv[j] = (uint32_t)(a - lo) - x;
          tv[j] = al - x;
        }
      }
      hs += hv[j];
      ts += tv[j];
    }
    const unsigned long long v = (unsigned long long)hs | ((unsigned long long)ts << 32);
    const unsigned long long e = block_excl_scan64(v, sm), tt = sm[32];
    uint32_t rh = (uint32_t)e, rt = (uint32_t)(e >> 32);
#pragma unroll
    for (int j = 0; j < CLS_SCAN_PER_THREAD; ++j) {
      const int64_t c = c0 + j;
      if (c < nchunks) {
        A.chunk_off[c * NCLS + 0] = (uint32_t)(carry_h + rh);
        A.chunk_off[c * NCLS + 1] = (uint32_t)(carry_t + rt);
      }
      rh += hv[j];
      rt += tv[j];
    }
    carry_h += (int64_t)(uint32_t)tt;
    carry_t += (int64_t)(uint32_t)(tt >> 32);
  }
  if (threadIdx.x == 0) A.meta[2] = carry_h;
}

// The holes' and the tails' slots.  (A chunk is below a, above it, or the one
// that a lies in.)
template <class Real>
__global__ void __launch_bounds__(TILE) k_fill_holes(FillArgs<Real> A) {
  __shared__ uint32_t scan_sm[33];
  const int64_t n = A.meta[0], a = A.meta[1];
  if (A.meta[2] == 0) return;
  const int64_t nchunks = (n + FILL_CHUNK - 1) / FILL_CHUNK;
  for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
    int64_t first;
    const uint32_t bits = fill_bits(A.s.alive, c, n, first);
    uint32_t hole = 0, tail = 0;
#pragma unroll
    for (int j = 0; j < FILL_ITEMS; ++j) {
      if (first + j < a && !(bits & (1u << j))) hole |= 1u << j;
      if (first + j >= a && (bits & (1u << j))) tail |= 1u << j;
    }
    // (at most 2048 of each: two counts in a word)
    const uint32_t ex = block_excl_scan(__popc(hole) | (uint32_t)__popc(tail) << 16, scan_sm);
    uint32_t k = A.chunk_off[c * NCLS + 0] + (ex & 0xFFFFu);
    __syncthreads();
    while (hole) {
      const int j = __ffs(hole) - 1;
      hole &= hole - 1;
      A.holes[k++] = (int)(first + j);
    }
    k = A.chunk_off[c * NCLS + 1] + (ex >> 16);
    while (tail) {
      const int j = __ffs(tail) - 1;
      tail &= tail - 1;
      A.tails[k++] = (int)(first + j);
    }
  }
}

// A particle per thread: all its words are read before any is written (2000
// moves of 15 arrays: 22 us with each chunk's threads moving their own tails
// word by word, 5 this way).
template <class Real>
__global__ void __launch_bounds__(TILE) k_fill_move(FillArgs<Real> A) {
  const int64_t m = A.meta[2];
  const Sp<Real> &S = A.s;
  const bool fields = S.ex != nullptr;
  for (int64_t k = blockIdx.x * (int64_t)TILE + threadIdx.x; k < m; k += (int64_t)gridDim.x * TILE) {
    const int64_t i = A.tails[k], d = A.holes[k];
    const Real v[7] = {S.x[i], S.y[i], S.z[i], S.px[i], S.py[i], S.pz[i], S.w[i]};
    const uint64_t id = S.id[i];
    const uint32_t tag = S.tag ? S.tag[i] : 0u;
    Real f[6] = {0, 0, 0, 0, 0, 0};
    if (fields) {
      f[0] = S.ex[i]; f[1] = S.ey[i]; f[2] = S.ez[i];
      f[3] = S.bx[i]; f[4] = S.by[i]; f[5] = S.bz[i];
    }
    S.x[d] = v[0]; S.y[d] = v[1]; S.z[d] = v[2];
    S.px[d] = v[3]; S.py[d] = v[4]; S.pz[d] = v[5]; S.w[d] = v[6];
    S.id[d] = id;
    if (S.tag) S.tag[d] = tag;
    if (fields) {
      S.ex[d] = f[0]; S.ey[d] = f[1]; S.ez[d] = f[2];
      S.bx[d] = f[3]; S.by[d] = f[4]; S.bz[d] = f[5];
    }
    S.alive[d] = 1;
  }
}

// ---------------------------------------------------------------------------
// Number of live particles (alive != 0) among the first *d_n, added to *out.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(TILE) k_count_alive(const uint8_t *alive, const int64_t *d_n,
                                                      unsigned long long *out) {
  const int64_t n = *(volatile const int64_t *)d_n;
  unsigned long long c = 0;
  for (int64_t i = blockIdx.x * (int64_t)TILE + threadIdx.x; i < n; i += (int64_t)gridDim.x * TILE)
    c += alive[i] ? 1u : 0u;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

// ---------------------------------------------------------------------------
// Snapshot of the photon count at the start of a fused step.
// ---------------------------------------------------------------------------
__global__ void k_snapshot(const int64_t *src, int64_t *dst) { *dst = *src; }

// ---------------------------------------------------------------------------
// Isolated sampler (xi at given chi, gamma; r2 from Philox(i, step)).
// ---------------------------------------------------------------------------
struct SampleArgs {
  const float *chi, *gamma;
  float *xi;
  int64_t n, step;
  Consts C;
  Tables<float> T;
  Out o;
  const uint32_t *mlp_frag;
  const float *mlp_w;
  int use_mlp;
  int emit_lanes, scan_draws;  // chain scheduling (QED_SCHED_EMIT_LANES, _SCAN_DRAWS)
};

__global__ void __launch_bounds__(TILE) k_sample_xi(SampleArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float *sR = reinterpret_cast<float *>(smem_raw);
  float *sF = sR + A.T.gl.n;
  uint32_t *s_frag = reinterpret_cast<uint32_t *>(
      smem_raw + (((size_t)A.T.gl.n * (1 + A.T.gy.n) * sizeof(float) + 15) & ~(size_t)15));
  float *s_fw = reinterpret_cast<float *>(s_frag + MLP_FRAG_WORDS);
  load_tables_smem(sR, A.T.R, A.T.gl.n);
  load_tables_smem(sF, A.T.F, A.T.gl.n * A.T.gy.n);
  if (A.use_mlp) mlp_stage(s_frag, s_fw, A.mlp_frag, A.mlp_w);
  __syncthreads();
  Tally tl;
  tl.clear();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // warp-uniform loop (the learned sampler is a warp-collective call)
  for (int64_t ib = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); ib < A.n; ib += stride) {
    const int64_t i = ib + (threadIdx.x & 31);
    const bool active = i < A.n;
    float chi = active ? __ldcs(A.chi + i) : 1.f, g = active ? __ldcs(A.gamma + i) : 1e3f;
    RateOut<float> ro = photon_rate(sR, sF, A.T, A.C, chi, g, tl);
    U4 r = draw(A.C, (uint64_t)i, A.step, 0, STREAM_EMIT);
    const float kap = photon_kappa(ro.kmin, unif<float>(r.y), unif<float>(~r.y));
    float Y = 0.f;
    bool in_mlp = false;
    if (A.use_mlp) {
      const float lchi = logf(chi);
      in_mlp = lchi >= MLP_L_LO && lchi <= MLP_L_HI && kap >= MLP_K_LO && kap <= MLP_K_HI;
      Y = mlp_infer_warp(s_frag, s_fw, (lchi - MLP_LC) / MLP_LS, (kap - MLP_KC) / MLP_KS) +
          mlp_baseline(kap);
    }
    if (!active) continue;
    float xi = 0.f;
    if (ro.W > 0.f) {
      if (!in_mlp) Y = photon_lndelta_table(A.T.Y, A.T, ro.l, kap, tl);
      xi = xi_from_lndelta(chi, Y).xi;
    }
    __stcs(A.xi + i, xi);
  }
  if (tl.status) atomicOr(&A.o.cnt->status, tl.status);
}

// ---------------------------------------------------------------------------
// Parity helpers: rates and inverse CDF at given inputs (tables in global).
// ---------------------------------------------------------------------------
template <class Real> struct EvalArgs {
  int which;
  const double *chi, *gamma;
  const uint32_t *word;
  double *out;
  int64_t n;
  Consts C;
  Tables<Real> T;
};

template <class Real> __global__ void k_eval_rates(EvalArgs<Real> A) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= A.n) return;
  Tally tl;
  tl.clear();
  Real chi = (Real)A.chi[i], g = (Real)A.gamma[i];
  if (A.which == 0)
    A.out[i] = (double)photon_rate(A.T.R, A.T.F, A.T, A.C, chi, g, tl).W;
  else
    A.out[i] = (double)pair_rate(A.T.P, A.T, A.C, chi, g, tl).W;
}

template <class Real> __global__ void k_eval_xi(EvalArgs<Real> A) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= A.n) return;
  Tally tl;
  tl.clear();
  Real chi = (Real)A.chi[i];
  uint32_t w = A.word[i];
  if (A.which == 0) {
    Real g = (Real)A.gamma[i];
    RateOut<Real> ro = photon_rate(A.T.R, A.T.F, A.T, A.C, chi, g, tl);
    XiOut<Real> xo = photon_xi(A.T.Y, A.T, ro.l, chi, ro.kmin, unif<Real>(w), unif<Real>(~w), tl);
    A.out[i] = (double)xo.xi;
  } else {
    RateOut<Real> ro = pair_rate(A.T.P, A.T, A.C, chi, (Real)1e6, tl);
    Real l = ro.l;
    if (!(chi >= sel<Real>(A.C.chi_pair_min, A.C.f_chi_pair_min))) l = A.T.glp.lo;
    XiOut<Real> xo = pair_xi(A.T.Yp, A.T, l, unif<Real>(w), unif<Real>(~w));
    A.out[i] = (double)xo.xi;
  }
}

// chi of every particle of a species from its momentum and per-particle
// fields (Eq. 2 for leptons, Eq. 3 for photons), in the context's precision,
// by the same functions the step kernels use (parity hook).
template <class Real> __global__ void k_eval_chi(Sp<Real> S, Real inv_aS, double *out) {
  const int64_t n = *(volatile const int64_t *)S.d_n;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const Real px = S.px[i], py = S.py[i], pz = S.pz[i];
    Real chi;
    if (S.q == (Real)0) {
      chi = chi_photon(px, py, pz, S.ex[i], S.ey[i], S.ez[i], S.bx[i], S.by[i], S.bz[i], inv_aS);
    } else {
      const Real g = m_sqrt((Real)1 + px * px + py * py + pz * pz);
      chi = chi_lepton(px, py, pz, g, S.ex[i], S.ey[i], S.ez[i], S.bx[i], S.by[i], S.bz[i], inv_aS);
    }
    out[i] = (double)chi;
  }
}

// Learned inverse CDF at given inputs (parity and spectral-error hook): xi
// of the photon sampler at (chi, gamma) for the uniform word w, through the
// network where (ln chi, kappa) lies in its domain, else through the inverse
// table -- exactly the choice the step kernels make.  Warp-uniform loop (the
// network is a warp-collective call); rates from the global-memory tables.
__global__ void __launch_bounds__(TILE) k_eval_xi_mlp(EvalArgs<float> A, const uint32_t *frag,
                                                      const float *w) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t *s_frag = reinterpret_cast<uint32_t *>(smem_raw);
  float *s_fw = reinterpret_cast<float *>(s_frag + MLP_FRAG_WORDS);
  mlp_stage(s_frag, s_fw, frag, w);
  __syncthreads();
  Tally tl;
  tl.clear();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t ib = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); ib < A.n; ib += stride) {
    const int64_t i = ib + (threadIdx.x & 31);
    const bool active = i < A.n;
    const float chi = active ? (float)A.chi[i] : 1.f, g = active ? (float)A.gamma[i] : 1e3f;
    const uint32_t wd = active ? A.word[i] : 0u;
    RateOut<float> ro = photon_rate(A.T.R, A.T.F, A.T, A.C, chi, g, tl);
    const float kap = photon_kappa(ro.kmin, unif<float>(wd), unif<float>(~wd));
    const float lchi = logf(chi);
    const bool in_mlp = lchi >= MLP_L_LO && lchi <= MLP_L_HI && kap >= MLP_K_LO && kap <= MLP_K_HI;
    float Y = mlp_infer_warp(s_frag, s_fw, (lchi - MLP_LC) / MLP_LS, (kap - MLP_KC) / MLP_KS) +
              mlp_baseline(kap);
    if (!active) continue;
    double xi = 0.0;
    if (ro.W > 0.f) {
      if (!in_mlp) Y = photon_lndelta_table(A.T.Y, A.T, ro.l, kap, tl);
      xi = (double)xi_from_lndelta(chi, Y).xi;
    }
    A.out[i] = xi;
  }
}

// ---------------------------------------------------------------------------
// Standing wave E = 2 a0 cos x (0, cos t, sin t), B = 2 a0 sin x (0, cos t,
// sin t) on grid[nz][ny][nx][8].  Each block computes the nx node values of
// one x-row once (FP64 cos/sin) and streams them over its (y, z) rows.
// ---------------------------------------------------------------------------
__global__ void k_fill_standing_wave(float *grid, int nx, int ny, int nz, double x0, double dx,
                                     double a0, double t) {
  extern __shared__ __align__(16) float4 srow[];  // [nx][2]
  const double ct = cos(t), st = sin(t);
  for (int i = threadIdx.x; i < nx; i += blockDim.x) {
    double x = x0 + (double)i * dx;
    double cx = 2.0 * a0 * cos(x), sx = 2.0 * a0 * sin(x);
    srow[2 * i] = make_float4(0.f, (float)(cx * ct), (float)(cx * st), 0.f);
    srow[2 * i + 1] = make_float4((float)(sx * ct), (float)(sx * st), 0.f, 0.f);
  }
  __syncthreads();
  const int64_t rows = (int64_t)ny * nz;
  const int64_t total = rows * nx * 2;  // float4 units
  float4 *g4 = reinterpret_cast<float4 *>(grid);
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    int64_t within = q % (2 * (int64_t)nx);
    __stcs(g4 + q, srow[within]);
  }
}

// ---------------------------------------------------------------------------
// Host-side launch helpers
// ---------------------------------------------------------------------------
Consts consts_of(const qed_ctx *c) {
  Consts k{};
  k.a_S = c->cfg.a_S;
  k.alpha = c->cfg.alpha;
  k.dt = c->cfg.dt;
  k.wdt_max = c->cfg.wdt_max;
  k.xi_min_energy = c->cfg.xi_min_energy;
  k.generator = c->cfg.generator;
  k.chi_pair_min = c->cfg.chi_pair_min;
  k.spec_lo = c->cfg.spec_lo;
  k.spec_scale = 64.0 / log(c->cfg.spec_hi / c->cfg.spec_lo);
  k.seed = c->cfg.seed;
  k.max_substeps = c->cfg.max_substeps;
  k.pair_sign = c->cfg.pair_sign;
  k.inv_aS = 1.0 / c->cfg.a_S;
  k.alpha_aS = c->cfg.alpha * c->cfg.a_S;
  k.f_dt = (float)k.dt;
  k.f_wdt_max = (float)k.wdt_max;
  k.f_xi_min_energy = (float)k.xi_min_energy;
  k.f_chi_pair_min = (float)k.chi_pair_min;
  k.f_spec_lo = (float)k.spec_lo;
  k.f_spec_scale = (float)k.spec_scale;
  k.f_inv_aS = (float)k.inv_aS;
  k.f_alpha_aS = (float)k.alpha_aS;
  for (int r = 0; r < 10; ++r) {
    k.rk[2 * r] = (uint32_t)k.seed + (uint32_t)r * 0x9E3779B9u;
    k.rk[2 * r + 1] = (uint32_t)(k.seed >> 32) + (uint32_t)r * 0xBB67AE85u;
  }
  return k;
}

Out out_of(const qed_ctx *c) {
  return Out{c->d_counters, ScanState{c->tile_state, c->sync, c->max_tiles}};
}

template <class Real> size_t lepton_smem(const qed_ctx *c) {
  return sizeof(Real) * ((size_t)c->gl.n + (size_t)c->gl.n * c->gy.n);
}

template <class Real, int FM>
static cudaError_t launch_push(qed_ctx *c, const LeptonArgs<Real> &a, cudaStream_t st) {
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lepton_push<Real, FM>, TILE, 0);
  if (e != cudaSuccess) return e;
  per_sm = persistent_blocks_per_sm(c, per_sm, QED_TUNE_STREAM);
  k_lepton_push<Real, FM><<<c->num_sms * per_sm, TILE, 0, st>>>(a);
  c->launches += 1;
  return cudaGetLastError();
}

// A persistent launch of an emission kernel that stages the FP32 rate and
// forward tables (and, when `mlp` is set, the learned sampler) in shared memory.
template <class Real, class Kern>
static cudaError_t launch_tables_kernel(qed_ctx *c, Kern kern, const LeptonArgs<Real> &a, bool mlp,
                                        int group, cudaStream_t st, size_t extra = 0) {
  size_t sm = sizeof(Real) == 8 ? 0 : lepton_smem<Real>(c);
  if (sm && mlp) sm = ((sm + 15) & ~(size_t)15) + MLP_SMEM_BYTES;
  if (extra) sm = ((sm + 15) & ~(size_t)15) + extra;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, TILE, sm);
  if (e != cudaSuccess) return e;
  per_sm = persistent_blocks_per_sm(c, per_sm, group);
  kern<<<c->num_sms * per_sm, TILE, sm, st>>>(a);
  c->launches += 1;
  return cudaGetLastError();
}

// A persistent launch of a kernel without dynamic shared memory.
template <class Real, class Kern>
static cudaError_t launch_plain_kernel(qed_ctx *c, Kern kern, const LeptonArgs<Real> &a,
                                       cudaStream_t st) {
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, TILE, 0);
  if (e != cudaSuccess) return e;
  per_sm = persistent_blocks_per_sm(c, per_sm, QED_TUNE_ORDER);
  kern<<<c->num_sms * per_sm, TILE, 0, st>>>(a);
  c->launches += 1;
  return cudaGetLastError();
}

// The class list of the streaming pass's flags (three launches).
static cudaError_t launch_class_lists(qed_ctx *c, const int64_t *n0, const int64_t *n1,
                                      cudaStream_t st) {
  ClassListArgs a{};
  a.flags = c->heavy_flags;
  a.n0 = n0;
  a.n1 = n1;
  a.list = c->heavy_list;
  a.chunk_cnt = c->cls_chunk_cnt;
  a.chunk_off = c->cls_chunk_off;
  a.off = c->cls_off;
  a.stage_idx = c->stage_idx;
  a.stage_n = c->stage_n;
  a.cnt = c->d_counters;
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_cls_count, TILE, 0);
  if (e != cudaSuccess) return e;
  const int grid = c->num_sms * (per_sm > 0 ? per_sm : 1);
  k_cls_count<<<grid, TILE, 0, st>>>(a);
  k_cls_scan<<<1, CLS_SCAN_THREADS, 0, st>>>(a);
  k_cls_scatter<<<grid, TILE, 0, st>>>(a);
  c->launches += 3;
  return cudaGetLastError();
}

static cudaError_t launch_sub_scan(qed_ctx *c, const int64_t *n_entries, int64_t *out_n, int64_t out_cap,
                                   cudaStream_t st) {
  SubScanArgs a{};
  a.cnt = c->sub_cnt;
  a.replay_n = c->replay_n;
  a.n_entries = n_entries;
  a.sub_meta = c->sub_meta;
  a.out_n = out_n;
  a.out_cap = out_cap;
  a.o = out_of(c);
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sub_scan, TILE, 0);
  if (e != cudaSuccess) return e;
  per_sm = persistent_blocks_per_sm(c, per_sm, QED_TUNE_ORDER);
  k_sub_scan<<<c->num_sms * per_sm, TILE, 0, st>>>(a);
  c->launches += 1;
  return cudaGetLastError();
}

// Emission: the streaming pass finishes the particles that surely have one
// sub-step and no event and classes the rest; the class list orders them
// (class 1 first, each class in particle order); the counting pass, the scan
// and the writing pass append their photons in that order.
template <class Real, int FM, int MODE>
static cudaError_t launch_lepton_t(qed_ctx *c, const LeptonArgs<Real> &a, cudaStream_t st) {
  if (MODE == MODE_PUSH) return launch_push<Real, FM>(c, a, st);
  cudaError_t e = launch_tables_kernel<Real>(c, k_lepton_stream<Real, FM, MODE>, a, false,
                                             QED_TUNE_STREAM, st, stream_prefetch_bytes<Real, FM>());
  if (e == cudaSuccess) e = prof_mark(c, 1, st);
  if (e == cudaSuccess) e = launch_class_lists(c, a.sp[0].d_n, a.nsp > 1 ? a.sp[1].d_n : nullptr, st);
  if (e == cudaSuccess) e = prof_mark(c, 2, st);
  if (e == cudaSuccess)
    e = a.use_mlp && sizeof(Real) == 4
            ? launch_tables_kernel<Real>(c, k_substep_count<Real, FM, MODE, true>, a, true,
                                         QED_TUNE_CHAINS, st)
            : launch_tables_kernel<Real>(c, k_substep_count<Real, FM, MODE, false>, a, false,
                                         QED_TUNE_CHAINS, st);
  if (e == cudaSuccess) e = prof_mark(c, 3, st);
  if (e == cudaSuccess) e = launch_sub_scan(c, c->cls_off + NCLS, a.ph.d_n, a.ph.cap, st);
  if (e == cudaSuccess) e = prof_mark(c, 4, st);
  if (e == cudaSuccess) e = launch_plain_kernel<Real>(c, k_substep_write_coop<Real, FM, MODE>, a, st);
  if (e == cudaSuccess)
    e = launch_tables_kernel<Real>(c, k_substep_replay<Real, FM, MODE, false>, a, false, QED_TUNE_CHAINS, st);
  if (e == cudaSuccess) e = prof_mark(c, 5, st);
  return e;
}

template <class Real, int MODE>
static cudaError_t launch_lepton_m(qed_ctx *c, const LeptonArgs<Real> &a, int fm, cudaStream_t st) {
  if (fm == QED_FIELDS_UNIFORM) return launch_lepton_t<Real, FM_UNIFORM, MODE>(c, a, st);
  if (fm == QED_FIELDS_PER_PARTICLE) return launch_lepton_t<Real, FM_PER_PARTICLE, MODE>(c, a, st);
  return launch_lepton_t<Real, FM_GRID, MODE>(c, a, st);
}

cudaError_t launch_lepton_onepass(qed_ctx *c, const qed_species *s0, const qed_species *s1,
                                  const qed_species *ph, const qed_fields *f, int64_t step,
                                  int mode, bool ordered, cudaStream_t st);

// The replay of a single pass with ordered appends: the leptons whose records
// found no room.  16 stage_cap floats hold the records, so they run out past
// max_particles / 2 photons in a step, or max_particles / 3 where the photons take
// fields of their own.
template <int MODE>
static cudaError_t launch_replay_by_slot(qed_ctx *c, const LeptonArgs<float> &a, int fm, cudaStream_t st) {
  if (fm == QED_FIELDS_UNIFORM)
    return launch_tables_kernel<float>(c, k_substep_replay<float, FM_UNIFORM, MODE, true>, a, false, QED_TUNE_CHAINS, st);
  if (fm == QED_FIELDS_PER_PARTICLE)
    return launch_tables_kernel<float>(c, k_substep_replay<float, FM_PER_PARTICLE, MODE, true>, a, false, QED_TUNE_CHAINS, st);
  return launch_tables_kernel<float>(c, k_substep_replay<float, FM_GRID, MODE, true>, a, false, QED_TUNE_CHAINS, st);
}

template <class Real>
cudaError_t launch_lepton(qed_ctx *c, const qed_species *s0, const qed_species *s1,
                          const qed_species *ph, const qed_fields *f, int64_t step, int mode,
                          cudaStream_t st) {
  // FP32 contexts under Method I take the single pass; with ordered appends the
  // learned sampler keeps the multi-pass path
  const bool ordered = c->cfg.append_order == QED_APPEND_ORDERED;
  const bool single = sizeof(Real) == 4 && mode != MODE_PUSH && c->cfg.generator == QED_GEN_METHOD_I &&
                      !(ordered && c->cfg.sampler == QED_SAMPLER_MLP && c->mlp_ready);
  if (single) {
    // marks: 1 after the single-pass kernel (recorded by it), 2..5 after the
    // learned sampler's dense pass or the ordered writes, if any
    cudaError_t e = launch_lepton_onepass(c, s0, s1, ph, f, step, mode, ordered, st);
    if (!ordered) {
      for (int k = 2; k <= 5 && e == cudaSuccess; ++k) e = prof_mark(c, k, st);
      return e;
    }
    if (e != cudaSuccess) return e;
  }
  LeptonArgs<Real> a{};
  a.sp[0] = to_sp<Real>(s0);
  a.nsp = s1 ? 2 : 1;
  if (s1) a.sp[1] = to_sp<Real>(s1);
  a.ph = to_sp<Real>(ph);
  a.f = to_fld<Real>(f);
  a.C = consts_of(c);
  a.T = tables_of<Real>(c);
  a.o = out_of(c);
  a.step = step;
  a.heavy_flags = c->heavy_flags;
  a.heavy_list = c->heavy_list;
  a.cls_off = c->cls_off;
  a.sub_cnt = c->sub_cnt;
  a.sub_gf = static_cast<Real *>(c->sub_gf);
  a.rec_e = static_cast<Real *>(c->rec_e);
  a.rec_k = c->rec_k;
  a.rec_cap = c->rec_cap;
  a.stage = static_cast<Stage<Real> *>(c->stage);
  a.stage_tag = c->stage_tag;
  a.stage_idx = c->stage_idx;
  a.stage_n = c->stage_n;
  a.stage_cap = c->stage_cap;
  a.sub_meta = c->sub_meta;
  a.replay_list = c->stage_idx;  // free once the class list is built
  a.replay_n = c->replay_n;
  a.mlp_frag = c->mlp_frag;
  a.mlp_w = c->mlp_w;
  a.use_mlp = c->cfg.sampler == QED_SAMPLER_MLP && c->mlp_ready;
  a.emit_lanes = sched_param(c, QED_SCHED_EMIT_LANES);
  a.scan_draws = sched_param(c, QED_SCHED_SCAN_DRAWS);
  a.d_step = c->use_dstep ? c->d_step : nullptr;
  if constexpr (sizeof(Real) == 4) {
    if (single) {
      a.replay_n = c->ord_n + 3;
      a.C.f_alpha_aS *= (float)c->replay_rate;
      cudaError_t e = mode == MODE_EMIT ? launch_replay_by_slot<MODE_EMIT>(c, a, f->mode, st)
                                        : launch_replay_by_slot<MODE_FUSED>(c, a, f->mode, st);
      for (int k = 2; k <= 5 && e == cudaSuccess; ++k) e = prof_mark(c, k, st);
      return e;
    }
  }
  if (mode == MODE_PUSH) return launch_lepton_m<Real, MODE_PUSH>(c, a, f->mode, st);
  if (mode == MODE_EMIT) return launch_lepton_m<Real, MODE_EMIT>(c, a, f->mode, st);
  return launch_lepton_m<Real, MODE_FUSED>(c, a, f->mode, st);
}

template <class Real>
cudaError_t launch_compact(qed_ctx *c, const qed_species *s, cudaStream_t st) {
  CompactArgs<Real> a{};
  constexpr int TP = compact_tile<Real>();
  const int64_t tiles = (s->capacity + TP - 1) / TP;
  a.s = to_sp<Real>(s);
  a.off = c->sub_cnt;  // (scratch of the step, one word per slot)
  a.read = c->sub_cnt + tiles;
  a.total = c->sub_cnt + 2 * tiles;
  a.ticket = c->compact_n;
  a.one = c->compact_n + 4;
  a.cnt = c->d_counters;
  if (tiles <= COMPACT_ONE) {
    a.group = a.one + COMPACT_ONE;
    a.total = a.group + COMPACT_ONE / 32;
    k_compact_small<Real><<<(unsigned)(tiles < 1 ? 1 : tiles), COMPACT_THREADS, 0, st>>>(a);
    c->launches += 1;
    return cudaGetLastError();
  }
  const int64_t count_need = (tiles * 32 + CLS_SCAN_THREADS - 1) / CLS_SCAN_THREADS, count_most = (int64_t)c->num_sms * 2;
  k_compact_count<Real><<<(unsigned)(count_need < 1 ? 1 : count_need < count_most ? count_need : count_most),
                          CLS_SCAN_THREADS, 0, st>>>(a);
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_compact_move<Real>, COMPACT_THREADS, 0);
  if (e != cudaSuccess) return e;
  per_sm = persistent_blocks_per_sm(c, per_sm, QED_TUNE_COMPACT);
  const int64_t most = (int64_t)c->num_sms * per_sm;
  // (launched while the counting pass runs, so that its CTAs are in place when that
  // ends: two launches one behind the other lost to a single one with a look-back
  // at 260,000 to 800,000 photons; 524,289 FP32 23.2 with the look-back, 25.2, 23.6
  // this way, 300,001 FP64 21.1, 25.1, 22.9, 2M FP32 55.9, 45.3, 43.2 us)
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(tiles < 1 ? 1 : tiles < most ? tiles : most));
  cfg.blockDim = dim3(COMPACT_THREADS);
  cfg.stream = st;
  cudaLaunchAttribute early{};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  c->launches += 2;
  return cudaLaunchKernelEx(&cfg, k_compact_move<Real>, a);
}

template <class Real>
cudaError_t launch_compact_fill(qed_ctx *c, const qed_species *s, cudaStream_t st) {
  FillArgs<Real> a{};
  a.s = to_sp<Real>(s);
  a.chunk_alive = c->cls_chunk_cnt;
  a.chunk_off = c->cls_chunk_off;
  a.meta = c->fill_meta;
  a.holes = c->heavy_list;
  a.tails = c->stage_idx;
  FillArgs<float> af{};  // the scan reads only the shared scratch
  af.chunk_alive = a.chunk_alive;
  af.chunk_off = a.chunk_off;
  af.meta = a.meta;
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fill_count<Real>, TILE, 0);
  if (e != cudaSuccess) return e;
  // no more CTAs than the capacity has chunks
  const int64_t chunks = (s->capacity + FILL_CHUNK - 1) / FILL_CHUNK, most = (int64_t)c->num_sms * (per_sm > 0 ? per_sm : 1);
  const unsigned grid = (unsigned)(chunks < 1 ? 1 : chunks < most ? chunks : most);
  k_fill_count<Real><<<grid, TILE, 0, st>>>(a);
  k_fill_scan<<<1, CLS_SCAN_THREADS, 0, st>>>(s->alive, s->d_n, af);
  k_fill_holes<Real><<<grid, TILE, 0, st>>>(a);
  k_fill_move<Real><<<grid, TILE, 0, st>>>(a);
  c->launches += 4;
  return cudaGetLastError();
}

cudaError_t launch_count_alive(qed_ctx *c, const qed_species *s, int64_t *out, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(int64_t), st);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_count_alive, TILE, 0);
  if (e != cudaSuccess) return e;
  k_count_alive<<<c->num_sms * (per_sm > 0 ? per_sm : 1), TILE, 0, st>>>(
      s->alive, s->d_n, reinterpret_cast<unsigned long long *>(out));
  c->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_snapshot(qed_ctx *c, const int64_t *src, int64_t *dst, cudaStream_t st) {
  k_snapshot<<<1, 1, 0, st>>>(src, dst);
  c->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_sample_xi(qed_ctx *c, const float *chi, const float *gamma, float *xi,
                             int64_t n, int64_t step, cudaStream_t st) {
  SampleArgs a{};
  a.chi = chi; a.gamma = gamma; a.xi = xi; a.n = n; a.step = step;
  a.C = consts_of(c);
  a.T = tables_of<float>(c);
  a.o = out_of(c);
  a.mlp_frag = c->mlp_frag;
  a.mlp_w = c->mlp_w;
  a.use_mlp = c->cfg.sampler == QED_SAMPLER_MLP && c->mlp_ready;
  size_t sm = lepton_smem<float>(c);
  if (a.use_mlp) sm = ((sm + 15) & ~(size_t)15) + MLP_SMEM_BYTES;
  cudaError_t e = cudaFuncSetAttribute(k_sample_xi, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sample_xi, TILE, sm);
  if (e != cudaSuccess) return e;
  per_sm = persistent_blocks_per_sm(c, per_sm, QED_TUNE_COMPACT);
  k_sample_xi<<<c->num_sms * per_sm, TILE, sm, st>>>(a);
  c->launches += 1;
  return cudaGetLastError();
}

template <class Real>
cudaError_t launch_eval(qed_ctx *c, int kind, int which, const double *chi, const double *gamma,
                        const uint32_t *word, double *out, int64_t n, cudaStream_t st) {
  EvalArgs<Real> a{};
  a.which = which; a.chi = chi; a.gamma = gamma; a.word = word; a.out = out; a.n = n;
  a.C = consts_of(c);
  a.T = tables_of<Real>(c);
  unsigned blocks = (unsigned)((n + 255) / 256);
  if (blocks == 0) return cudaSuccess;
  if (kind == 0) k_eval_rates<Real><<<blocks, 256, 0, st>>>(a);
  else k_eval_xi<Real><<<blocks, 256, 0, st>>>(a);
  c->launches += 1;
  return cudaGetLastError();
}

template <class Real> cudaError_t launch_eval_chi(qed_ctx *c, const qed_species *s, double *out,
                                                   cudaStream_t st) {
  const Consts C = consts_of(c);
  k_eval_chi<Real><<<c->num_sms * 4, 256, 0, st>>>(to_sp<Real>(s), sizeof(Real) == 8 ? (Real)C.inv_aS : (Real)C.f_inv_aS,
                                                   out);
  c->launches += 1;
  return cudaGetLastError();
}
template cudaError_t launch_eval_chi<float>(qed_ctx *, const qed_species *, double *, cudaStream_t);
template cudaError_t launch_eval_chi<double>(qed_ctx *, const qed_species *, double *, cudaStream_t);

cudaError_t launch_eval_xi_mlp(qed_ctx *c, const double *chi, const double *gamma,
                               const uint32_t *word, double *out, int64_t n, cudaStream_t st) {
  EvalArgs<float> a{};
  a.which = 0; a.chi = chi; a.gamma = gamma; a.word = word; a.out = out; a.n = n;
  a.C = consts_of(c);
  a.T = tables_of<float>(c);
  if (n == 0) return cudaSuccess;
  const size_t sm = MLP_SMEM_BYTES;
  cudaError_t e = cudaFuncSetAttribute(k_eval_xi_mlp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  int64_t blocks = (n + TILE - 1) / TILE;
  if (blocks > (int64_t)c->num_sms * 8) blocks = (int64_t)c->num_sms * 8;
  k_eval_xi_mlp<<<(unsigned)blocks, TILE, sm, st>>>(a, c->mlp_frag, c->mlp_w);
  c->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_fill(qed_ctx *c, float *grid, int nx, int ny, int nz, double x0, double dx,
                        double a0, double t, cudaStream_t st) {
  size_t sm = sizeof(float4) * 2 * (size_t)nx;
  cudaError_t e = cudaFuncSetAttribute(k_fill_standing_wave,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k_fill_standing_wave<<<c->num_sms * 4, 256, sm, st>>>(grid, nx, ny, nz, x0, dx, a0, t);
  c->launches += 1;
  return cudaGetLastError();
}

template cudaError_t launch_lepton<float>(qed_ctx *, const qed_species *, const qed_species *,
                                          const qed_species *, const qed_fields *, int64_t, int,
                                          cudaStream_t);
template cudaError_t launch_lepton<double>(qed_ctx *, const qed_species *, const qed_species *,
                                           const qed_species *, const qed_fields *, int64_t, int,
                                           cudaStream_t);
template cudaError_t launch_compact<float>(qed_ctx *, const qed_species *, cudaStream_t);
template cudaError_t launch_compact<double>(qed_ctx *, const qed_species *, cudaStream_t);
template cudaError_t launch_compact_fill<float>(qed_ctx *, const qed_species *, cudaStream_t);
template cudaError_t launch_compact_fill<double>(qed_ctx *, const qed_species *, cudaStream_t);
template cudaError_t launch_eval<float>(qed_ctx *, int, int, const double *, const double *,
                                        const uint32_t *, double *, int64_t, cudaStream_t);
template cudaError_t launch_eval<double>(qed_ctx *, int, int, const double *, const double *,
                                         const uint32_t *, double *, int64_t, cudaStream_t);

}  // namespace qed
