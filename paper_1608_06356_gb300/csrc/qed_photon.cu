// qed_photon.cu -- the photon stage of a step (qed_pair, and the photons of
// qed_step_fused): ballistic push, chi_ph (Eq. 3), pair rate (Eq. 6), Method I,
// the e-/e+ of each event appended in photon order.
//
// Three launches:
//   k_photon_stream  every live photon once: push, rate and the first draw.  A
//     photon with one sub-step and no event is finished there.  The others
//     (an event, or several sub-steps to draw) enter the warp's pool in
//     shared memory -- of scanning and of pending photons, any lane running
//     any entry, as in the lepton step -- so that one long chain does not hold
//     its warp.  An event leaves a record (the pair's energies), the photon's
//     bit in a mask, and one on the count of its chunk of 2048 photons.
//   k_pair_scan      the chunks' first positions (one CTA) and the new counts.
//   k_pair_write     per record: its position (chunk, and the mask's bits
//     before it in the chunk) and the two leptons there.
// At 2^20 photons of which 2000 convert: 64 us in six launches (a memset, the
// stream, a list of the flagged photons, a counting pass, a scan and a writing
// pass) -> 40 us (27, 3, 10): the stream is bound by instruction issue (490
// per 32 photons, 9 us at the copy rate), the pairs by the latency of the few
// photons concerned.  With no photons 20 -> 7.
#include <cstdio>

#include "qed_internal.h"
#include "qed_kernels.cuh"

namespace qed {
namespace {

constexpr int CHUNK = CLS_CHUNK_FLAGS;      // photons per chunk
constexpr int CHUNK_WORDS = CHUNK / 32;     // mask words per chunk
constexpr int PH_THREADS = 256, PH_WARPS = PH_THREADS / 32;
constexpr int PH_POOL = 64;                 // pool entries per warp

// lists of pool entries: scanning (up) and pending (down) share an array, the
// free entries (up) have their own
enum { P_SCAN = 0, P_PEND = 1, P_FREE = 2 };
__device__ __forceinline__ constexpr int plist_at(int l, int k) {
  return l == P_PEND ? PH_POOL - 1 - k : l == P_SCAN ? k : PH_POOL + k;
}

// A photon in the pool.  r2 is the word of a pending event, found at sub-step s.
template <class Real, int FM> struct PoolEntry {
  uint32_t i, id0, id1, N, s, r2;
  Real thr, l, k;  // event threshold W Dt / N, ln chi (clamped), |p|
  Real f[FM == FM_GRID ? 6 : 1];
};

template <class Real> struct PhotonArgs {
  Sp<Real> ph, el, po;
  const int64_t *n_active;  // photons [0, *n_active) are processed
  Fld<Real> f;
  Consts C;
  Tables<Real> T;
  qed_counters *cnt;
  int64_t step;
  const int64_t *d_step;  // if set, the step index is read here (graph replay)
  uint32_t *mask;         // [photon / 32] bits of the photons that convert
  uint32_t *sum, *off;    // [chunk] pairs (zero between steps), then the first pair's position
  uint2 *rec_i;           // [record] photon, sub-step (records for every photon: holds_pairs)
  Real *rec;              // [record][8] gamma_e, gamma_p, E, B (E, B with grid fields)
  unsigned int *n;        // [0] records, [1] those of the pass being written
  int64_t *meta;          // [1], [2] electron and positron counts before
};

// dynamic shared memory: the pools, their lists and the pair-rate table
template <class Real, int FM> size_t photon_smem(const qed_ctx *c) {
  return PH_WARPS * PH_POOL * (sizeof(PoolEntry<Real, FM>) + 2) + sizeof(Real) * (size_t)c->glp.n;
}

// Photons of the pass: never more than the species holds, so never more pairs
// than there are records.
__device__ __forceinline__ int64_t photons_of(const int64_t *n_active, int64_t cap) {
  const int64_t n = *(volatile const int64_t *)n_active;
  return n < cap ? n : cap;
}

template <class Real, int FM>
__global__ void __launch_bounds__(PH_THREADS, sizeof(Real) == 4 ? 4 : 2) k_photon_stream(PhotonArgs<Real> A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PoolEntry<Real, FM> *const s_pool = reinterpret_cast<PoolEntry<Real, FM> *>(smem_raw);
  uint8_t *const s_list = reinterpret_cast<uint8_t *>(s_pool + PH_WARPS * PH_POOL);
  Real *const sP = reinterpret_cast<Real *>(s_list + PH_WARPS * 2 * PH_POOL);
  __shared__ BlockTally bt;
  const int64_t n = photons_of(A.n_active, A.ph.cap);
  const int64_t nslices = (n + 31) / 32;
  if (blockIdx.x >= nslices) return;  // (slice w of warp wid is wid * gridDim + blockIdx, so none here)
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int64_t step_ = A.d_step ? *A.d_step : A.step;
  load_tables_smem(sP, A.T.P, A.T.glp.n);
  block_tally_init(&bt);
  PoolEntry<Real, FM> *const pool = s_pool + wid * PH_POOL;
  uint8_t *const list = s_list + wid * 2 * PH_POOL;
  int len[3] = {0, 0, PH_POOL};
  for (int q = lane; q < PH_POOL; q += 32) list[plist_at(P_FREE, q)] = (uint8_t)q;
  __syncthreads();
  const Real inv_aS = sel<Real>(A.C.inv_aS, A.C.f_inv_aS);
  const Real dt = sel<Real>(A.C.dt, A.C.f_dt), wdt_max = sel<Real>(A.C.wdt_max, A.C.f_wdt_max);
  Tally tl;
  tl.clear();
  auto file = [&](int s, bool in, int e) {
    const unsigned m = __ballot_sync(0xFFFFFFFFu, in);
    if (in) list[plist_at(s, len[s] + __popc(m & lt_mask))] = (uint8_t)e;
    len[s] += __popc(m);
  };
  // consecutive slices go to different CTAs
  int64_t slice = (int64_t)wid * gridDim.x + blockIdx.x;
  const int64_t stride = (int64_t)gridDim.x * PH_WARPS;
  for (;;) {
    const bool streaming = slice < nslices;
    const int phase = len[P_PEND] >= len[P_SCAN] ? P_PEND : P_SCAN;
    const int most = len[P_PEND] >= len[P_SCAN] ? len[P_PEND] : len[P_SCAN];
    if (streaming && most < 32 && len[P_FREE] >= 32) {
      const int64_t i = slice * 32 + lane;
      if (lane == 0) A.mask[slice] = 0u;
      int st = -1;
      Real k = 0, E[3] = {0, 0, 0}, B[3] = {0, 0, 0};
      RateOut<Real> ro{(Real)0, (Real)0, (Real)0};
      uint64_t pid = 0;
      uint32_t r2 = 0;
      int64_t N = 1;
      // (the words do not wait for the flag; 8.4M photons with fields, all alive,
      // half or all dead: 204, 203 and 73 us, against 240, 247 and 96 in the stream
      // and list that read the flag first)
      uint8_t alive = 0;
      Real x = 0, y = 0, z = 0, px = 0, py = 0, pz = 0;
      if (i < n) {
        alive = A.ph.alive[i];
        x = A.ph.x[i]; y = A.ph.y[i]; z = A.ph.z[i];
        px = A.ph.px[i]; py = A.ph.py[i]; pz = A.ph.pz[i];
        if (FM == FM_PER_PARTICLE) get_fields<Real, FM>(A.ph, A.f, i, x, y, z, E, B);
      }
      if (alive) {
        if (FM != FM_PER_PARTICLE) get_fields<Real, FM>(A.ph, A.f, i, x, y, z, E, B);
        k = m_sqrt(px * px + py * py + pz * pz);
        const Real chi = chi_photon(px, py, pz, E[0], E[1], E[2], B[0], B[1], B[2], inv_aS);
        ro = pair_rate(sP, A.T, A.C, chi, k, tl);
        const Real wdt = ro.W * dt;
        if (ro.W > (Real)0) {  // (most soft photons have W = 0: no id read)
          pid = A.ph.id[i];
          if (wdt > wdt_max) {
            Real nn = m_ceil(wdt / wdt_max);
            if (nn > (Real)A.C.max_substeps) {
              nn = (Real)A.C.max_substeps;
              tl.status |= QED_STATUS_SUBSTEPS;
            }
            N = (int64_t)nn;
            st = P_SCAN;
          } else {
            const U4 r = draw(A.C, pid, step_, 0, STREAM_PAIR);
            if (wdt > unif<Real>(r.x)) {  // one sub-step with an event
              st = P_PEND;
              r2 = r.y;
            }
          }
        }
        tl.substeps += N;
        if (k > (Real)0) {
          const Real ik = dt / k;
          A.ph.x[i] = x + px * ik; A.ph.y[i] = y + py * ik; A.ph.z[i] = z + pz * ik;
        }
      }
      const unsigned m = __ballot_sync(0xFFFFFFFFu, st >= 0);
      int e = 0;
      if (st >= 0) {
        e = list[plist_at(P_FREE, len[P_FREE] - 1 - __popc(m & lt_mask))];
        PoolEntry<Real, FM> &P = pool[e];
        P.i = (uint32_t)i;
        P.id0 = (uint32_t)pid; P.id1 = (uint32_t)(pid >> 32);
        P.N = (uint32_t)N; P.s = 0; P.r2 = r2;
        P.thr = ro.W * (dt / (Real)N); P.l = ro.l; P.k = k;
        if constexpr (FM == FM_GRID) {
#pragma unroll
          for (int c = 0; c < 3; ++c) { P.f[c] = E[c]; P.f[3 + c] = B[c]; }
        }
      }
      __syncwarp();
      len[P_FREE] -= __popc(m);
      file(P_SCAN, st == P_SCAN, e);
      file(P_PEND, st == P_PEND, e);
      __syncwarp();
      slice += stride;
      continue;
    }
    if (most == 0) break;
    const int take = min(most, 32);
    const bool act = lane < take;
    const int e = act ? list[plist_at(phase, most - 1 - lane)] : 0;
    __syncwarp();
    int st = -1;
    if (phase == P_SCAN) {
      len[P_SCAN] -= take;
      // ---- the next sub-steps, one draw each
      if (act) {
        const uint64_t pid = (uint64_t)pool[e].id0 | ((uint64_t)pool[e].id1 << 32);
        const uint32_t N = pool[e].N;
        uint32_t s = pool[e].s;
        const Real thr = pool[e].thr;
        st = P_SCAN;
#pragma unroll 1
        for (int u = 0; u < 4 && st == P_SCAN; ++u) {
          const U4 r = draw(A.C, pid, step_, s, STREAM_PAIR);
          if (thr > unif<Real>(r.x)) {
            st = P_PEND;
            pool[e].r2 = r.y;
          } else if (++s >= N) {
            st = P_FREE;
          }
        }
        pool[e].s = s;
      }
    } else {
      len[P_PEND] -= take;
      // ---- the pair: energies, record, mask and counts
      unsigned base = 0;
      if (lane == 0) base = atomicAdd(A.n, (unsigned)take);
      Real ge = 0, gp = 0;
      if (act) {
        const uint32_t r2 = pool[e].r2;
        const Real k = pool[e].k;
        const XiOut<Real> xo = pair_xi(A.T.Yp, A.T, pool[e].l, unif<Real>(r2), unif<Real>(~r2));
        ge = xo.xi * k;
        gp = xo.omxi * k;
        if (ge < (Real)1) { ge = (Real)1; gp = k - (Real)1; }
        if (gp < (Real)1) { gp = (Real)1; ge = k - (Real)1; }
      }
      base = __shfl_sync(0xFFFFFFFFu, base, 0);
      if (act) {
        const uint32_t i = pool[e].i, r = base + lane;
        A.ph.alive[i] = 0;
        atomicOr(&A.mask[i / 32], 1u << (i & 31));
        atomicAdd(&A.sum[i / CHUNK], 1u);
        A.rec_i[r] = make_uint2(i, pool[e].s);
        Real *R = A.rec + 8 * (size_t)r;
        R[0] = ge;
        R[1] = gp;
        if constexpr (FM == FM_GRID) {
#pragma unroll
          for (int c = 0; c < 6; ++c) R[2 + c] = pool[e].f[c];
        }
        tl.events += 1;
        st = P_FREE;
      }
    }
    if (phase == P_SCAN) {
      file(P_SCAN, st == P_SCAN, e);
      file(P_PEND, st == P_PEND, e);
    }
    file(P_FREE, st == P_FREE, e);
    __syncwarp();
  }
  tally_flush(&bt, tl);
  __syncthreads();
  block_tally_commit(&bt, A.cnt, 1);
}

// One CTA: the chunks' first positions in photon order, the lepton counts, and
// the start of the next pass (counts and sums zero).
constexpr int PSCAN_THREADS = 1024, PSCAN_CHUNKS = 4;
struct PairScanArgs {
  const int64_t *n_active;
  int64_t ph_cap;
  uint32_t *sum, *off;
  unsigned int *n;
  int64_t *el_n, *po_n, *meta;
  int64_t el_cap, po_cap;
  qed_counters *cnt;
};
__global__ void __launch_bounds__(PSCAN_THREADS) k_pair_scan(PairScanArgs A) {
  __shared__ uint32_t sm[33];
  const unsigned pairs = *(volatile unsigned *)A.n;
  if (threadIdx.x == 0) A.n[1] = pairs;
  if (pairs == 0) return;
  const int64_t nchunks = (photons_of(A.n_active, A.ph_cap) + CHUNK - 1) / CHUNK;
  uint32_t carry = 0;
  for (int64_t r0 = 0; r0 < nchunks; r0 += PSCAN_THREADS * PSCAN_CHUNKS) {
    const int64_t c0 = r0 + (int64_t)threadIdx.x * PSCAN_CHUNKS;
    uint32_t v[PSCAN_CHUNKS], t = 0;
#pragma unroll
    for (int j = 0; j < PSCAN_CHUNKS; ++j) {
      v[j] = c0 + j < nchunks ? A.sum[c0 + j] : 0u;
      t += v[j];
    }
    uint32_t run = carry + block_excl_scan(t, sm);
    carry += sm[32];
    __syncthreads();  // sm[32] is read
#pragma unroll
    for (int j = 0; j < PSCAN_CHUNKS; ++j) {
      if (c0 + j < nchunks) {
        A.off[c0 + j] = run;
        if (v[j]) A.sum[c0 + j] = 0u;
      }
      run += v[j];
    }
  }
  if (threadIdx.x == 0) {
    A.n[0] = 0u;
    unsigned long long dropped = 0;
    int64_t *const cn[2] = {A.el_n, A.po_n};
    const int64_t cap[2] = {A.el_cap, A.po_cap};
    for (int q = 0; q < 2; ++q) {
      const int64_t before = *cn[q], after = before + pairs < cap[q] ? before + pairs : cap[q];
      const int64_t written = after > before ? after - before : 0;
      A.meta[1 + q] = before;
      *cn[q] = after;
      dropped += (unsigned long long)(pairs - written);
    }
    if (dropped) {
      atomicAdd(reinterpret_cast<unsigned long long *>(&A.cnt->dropped), dropped);
      atomicOr(&A.cnt->status, (unsigned)QED_STATUS_CAPACITY);
    }
  }
}

template <class Real, int FM>
__global__ void __launch_bounds__(PH_THREADS) k_pair_write(PhotonArgs<Real> A) {
  const unsigned pairs = *(volatile unsigned *)&A.n[1];
  if (blockIdx.x * PH_THREADS >= pairs) return;
  const int64_t step_ = A.d_step ? *A.d_step : A.step;
  const int64_t ne = A.meta[1], np = A.meta[2];
  for (unsigned r = blockIdx.x * PH_THREADS + threadIdx.x; r < pairs; r += gridDim.x * PH_THREADS) {
    const uint2 ri = A.rec_i[r];
    const int64_t i = ri.x;
    // (the photon's words are on their way while its position is counted)
    const Real *R = A.rec + 8 * (size_t)r;
    const Real ge = R[0], gp = R[1];
    const Real px = A.ph.px[i], py = A.ph.py[i], pz = A.ph.pz[i];
    const Real x = A.ph.x[i], y = A.ph.y[i], z = A.ph.z[i], w = A.ph.w[i];
    const uint64_t pid = A.ph.id[i];
    const uint32_t tag = A.ph.tag ? A.ph.tag[i] : 0u;
    Real E[3] = {0, 0, 0}, B[3] = {0, 0, 0};
    if (A.el.ex || A.po.ex) {
      if constexpr (FM == FM_GRID) {
#pragma unroll
        for (int q = 0; q < 3; ++q) { E[q] = R[2 + q]; B[q] = R[5 + q]; }
      } else {
        get_fields<Real, FM>(A.ph, A.f, i, (Real)0, (Real)0, (Real)0, E, B);
      }
    }
    const int64_t c = i / CHUNK;
    uint32_t pos = A.off[c];
    const uint4 *m4 = reinterpret_cast<const uint4 *>(A.mask + c * CHUNK_WORDS);
    const int at = (int)(i % CHUNK) / 32;
#pragma unroll 8
    for (int q = 0; q <= at / 4; ++q) {
      const uint4 m = m4[q];
      const uint32_t bits[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        pos += __popc(q * 4 + j < at ? bits[j] : q * 4 + j == at ? bits[j] & ((1u << (i & 31)) - 1u) : 0u);
    }
    const Real k = m_sqrt(px * px + py * py + pz * pz);
    const Real ik = (Real)1 / k;
    const Real nx = px * ik, ny = py * ik, nz = pz * ik;
    const U4 cid = draw(A.C, pid, step_, ri.y, STREAM_PAIR_ID);
    const Real pe = m_sqrt((ge - (Real)1) * (ge + (Real)1));
    const Real pp = m_sqrt((gp - (Real)1) * (gp + (Real)1));
    if (ne + pos < A.el.cap)
      write_child(A.el, ne + pos, x, y, z, pe * nx, pe * ny, pe * nz, w, (uint64_t)cid.x | ((uint64_t)cid.y << 32), E, B, tag);
    if (np + pos < A.po.cap)
      write_child(A.po, np + pos, x, y, z, pp * nx, pp * ny, pp * nz, w, (uint64_t)cid.z | ((uint64_t)cid.w << 32), E, B, tag);
  }
}

template <class Real, int FM>
cudaError_t launch_photon_t(qed_ctx *c, const PhotonArgs<Real> &a, cudaStream_t st) {
  const size_t sm = photon_smem<Real, FM>(c);
  int per_sm = 0;
  cudaError_t e = cudaFuncSetAttribute(k_photon_stream<Real, FM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_photon_stream<Real, FM>, PH_THREADS, sm);
  if (e != cudaSuccess) return e;
  per_sm = persistent_blocks_per_sm(c, per_sm, QED_TUNE_PHOTON);
  // no more CTAs than the capacity has slices
  const int64_t slices = (a.ph.cap + 31) / 32, most = (int64_t)c->num_sms * per_sm;
  const unsigned grid = (unsigned)(slices < 1 ? 1 : slices < most ? slices : most);
  k_photon_stream<Real, FM><<<grid, PH_THREADS, sm, st>>>(a);
  c->launches += 1;
  e = cudaGetLastError();
  if (e == cudaSuccess) e = prof_mark(c, 6, st);
  if (e != cudaSuccess) return e;
  PairScanArgs s{a.n_active, a.ph.cap, a.sum, a.off, a.n, a.el.d_n, a.po.d_n, a.meta, a.el.cap, a.po.cap, a.cnt};
  k_pair_scan<<<1, PSCAN_THREADS, 0, st>>>(s);
  k_pair_write<Real, FM><<<grid, PH_THREADS, 0, st>>>(a);
  c->launches += 2;
  return cudaGetLastError();
}

}  // namespace

template <class Real>
cudaError_t launch_photon(qed_ctx *c, const qed_species *g, const qed_species *e,
                          const qed_species *p, const int64_t *n_active, const qed_fields *f,
                          int64_t step, cudaStream_t st) {
  PhotonArgs<Real> a{};
  a.ph = to_sp<Real>(g);
  a.el = to_sp<Real>(e);
  a.po = to_sp<Real>(p);
  a.n_active = n_active;
  a.f = to_fld<Real>(f);
  a.C = consts_of(c);
  a.T = tables_of<Real>(c);
  a.cnt = c->d_counters;
  a.step = step;
  a.d_step = c->use_dstep ? c->d_step : nullptr;
  a.mask = reinterpret_cast<uint32_t *>(c->heavy_flags);
  a.sum = c->pair_sum;
  a.off = c->cls_chunk_off;
  a.rec_i = reinterpret_cast<uint2 *>(c->rec_k);
  a.rec = static_cast<Real *>(c->stage);
  a.n = c->pair_n;
  a.meta = c->sub_meta;
  if (f->mode == QED_FIELDS_UNIFORM) return launch_photon_t<Real, FM_UNIFORM>(c, a, st);
  if (f->mode == QED_FIELDS_PER_PARTICLE) return launch_photon_t<Real, FM_PER_PARTICLE>(c, a, st);
  return launch_photon_t<Real, FM_GRID>(c, a, st);
}
template cudaError_t launch_photon<float>(qed_ctx *, const qed_species *, const qed_species *,
                                          const qed_species *, const int64_t *, const qed_fields *,
                                          int64_t, cudaStream_t);
template cudaError_t launch_photon<double>(qed_ctx *, const qed_species *, const qed_species *,
                                           const qed_species *, const int64_t *, const qed_fields *,
                                           int64_t, cudaStream_t);

}  // namespace qed
