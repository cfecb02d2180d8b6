// qed_onepass.cu -- the lepton step in a single pass (FP32 contexts, event
// generator Method I): photons appended in no particular order
// (qed_config.append_order = QED_APPEND_ANY), or in the multi-pass path's order
// (QED_APPEND_ORDERED with the table sampler; the passes after the kernel).
//
// What is computed is the multi-pass path's: per lepton, field gather, Boris
// push, chi_e (Eq. 2), W_rad (Eq. 1 above the xi_min cut), N = max(1,
// ceil(W Dt / 0.2)) sub-steps of Method I with Philox draws keyed by (id,
// step, sub-step / 2) -- one draw serves two sub-steps --, xi from the inverse
// CDF (Eq. 7) on an event, the recoil and the photon.  Every particle, photon
// id and photon energy is the same; under QED_APPEND_ANY only the order of the
// appended photons differs (it depends on the scheduling of the warps), so the
// photon buffer is the same set in another order.
//
// How the work is laid out, per warp of a persistent grid (one CTA of OP_WARPS
// warps per SM):
//   streaming: each lane takes one particle of a 32-particle slice (the next
//     slice's words are in flight into shared memory, cp.async), pushes it and
//     computes chi.  The rate bound W <= w_j chi / gamma (w_j = alpha a_S
//     times the largest value of int_0^1 dW/dxi / chi in the rate table at
//     and above the row j at or below ln chi, so it holds with the xi_min cut)
//     settles most particles without the 2-D tables: if w_j chi Dt / gamma <=
//     0.2 the particle has one sub-step, and if its first draw r1 is not
//     below that bound it has no event -- it is finished (its pushed state
//     written).  The others enter the warp's pool.
//   pool: PCAP chains in shared memory, each in one of three states: rate due
//     (chi and the exact rate; a new particle also gets N), scanning (Method I
//     draws due), or event pending (xi, the recoil, the photon).  A round
//     takes up to 32 chains of one state -- any lane runs any chain -- and
//     files each under its next state; a chain that ends frees its entry.  The
//     warp streams while the pool has room for a slice, and otherwise runs the
//     fullest state (19 chains at least then), where a lane that keeps its own
//     chain in registers waits for its neighbours' states: 26 of 32 lanes
//     active over the whole kernel instead of 22.  After the last slice the
//     pool is drained.
//   photons: an emission round reserves slots for its photons with one atomic
//     on the photon count and writes them there.  Ordered appends: it writes
//     records instead, with all a photon takes from its parent; three short
//     passes then turn each emitting lepton's count into the position of its
//     first photon, list the record of every position and write the photons in
//     position order.  (4M electrons: 417 us of kernels for the multi-pass
//     path, with its 64-byte staging of every deferred lepton and its replay
//     of the long chains; 262 us this way: 182, scan 11, offsets 20, index 21,
//     photons 25.  Photons written in record order, gathering their parents:
//     139 instead of 46.)
//   learned sampler: an event of a one-sub-step lepton inside the network's
//     domain ends its chain with a 16-byte record instead of an emission; the
//     dense pass k_net_emit (below) finishes those emissions, 32 per warp.
// No particle waits on another and nothing is staged in global memory: a
// particle is read once and its slot written once or twice (the pushed state,
// then the recoiled momentum of one that emitted, shortly after, while the
// line is still in L2).
//
// What bounds it: instruction issue, 62% of the slots of 20 warps an SM (the
// rest is the latency of dependent arithmetic); DRAM moves little more than the
// algorithmic bytes.  The 64M-electron ensemble: 2.93 -> 2.04 ms per launch
// (2.18 -> 3.13 TB/s algorithmic), at 16M 735 -> 544 us, of which streaming
// alone 239 (198 at the copy rate).  Steps and choices measured at 16M: chains in
// a pool (20 warps of 96 entries, tables in shared memory) 647; fewer entries
// leave more L1 to the inverse table and fewer lanes to a round (80: 601, 72:
// 629, 64: 682), and the tables are as fast through L1, which leaves room for 88
// entries: 594; 16 warps of 120 entries 692, 24 of 80 entries (80 registers)
// 630; E and B left in global memory for larger pools 651; the parent's words
// and the photon slots requested before the inverse look-up 563; slices by
// 16-byte copies past L1 544.
#include <cstdio>

#include "qed_internal.h"
#include "qed_kernels.cuh"
#include "qed_mlp.cuh"

namespace qed {

namespace {

// one CTA per SM; 20 warps leave 96 registers to a thread
constexpr int OP_WARPS = 20;
constexpr int OP_THREADS = OP_WARPS * 32;
// Chains per warp's pool.
template <int FM, bool ORD> __host__ __device__ constexpr int pool_cap() { return ORD && FM == FM_GRID ? 80 : 88; }
// Words of a pool entry: the slot, the id, the pushed momentum until the first
// emission and then the unit direction, gamma, chi, the event threshold W Dt / N
// (of a pending event its word r2), kappa_min, N (0: new), the sub-step (top
// bits: below) and, unless the field is uniform, E and B; ORD (photons in the
// ordered path's order, below): the photons so far and, with grid fields, the
// pushed position.
enum { W_SLOT, W_ID0, W_ID1, W_VX, W_VY, W_VZ, W_G, W_CHI, W_THR, W_KMIN, W_N, W_K, W_FIELDS, W_R2 = W_THR };
constexpr uint32_t EMITTED = 0x80000000u;  // it has emitted
constexpr uint32_t LOST = 0x40000000u;     // ORD: the record of one of its photons found no room
constexpr uint32_t K_MASK = 0x3FFFFFFFu;
template <int FM> __host__ __device__ constexpr int w_cnt() { return FM == FM_UNIFORM ? W_FIELDS : W_FIELDS + 6; }
template <int FM, bool ORD> __host__ __device__ constexpr int pool_words() {
  return w_cnt<FM>() + (ORD ? (FM == FM_GRID ? 4 : 1) : 0);
}
// The states of a chain, and the free entries.  An entry is in one list, so two
// lists share an array of bytes from its two ends: rate (up) and scan (down),
// pending (up) and free (down).  ORD: a third array holds the entries' classes.
enum { L_RATE = 0, L_SCAN = 1, L_PEND = 2, L_FREE = 3 };
template <int PCAP> __device__ __forceinline__ constexpr int list_at(int l, int k) {
  return (l >> 1) * PCAP + ((l & 1) ? PCAP - 1 - k : k);
}

// ---- ordered appends (QED_APPEND_ORDERED): what the single pass leaves to
// the writing pass.  The photons' order is by class of their lepton's sub-step
// count (1: one sub-step; 2-5: N <= 3, <= 7, <= 15, more), then slot, then
// sub-step.
struct OrdArgs {
  uint8_t *flags;    // [slot] class of a lepton with photons (top bit: replayed), else 0
  uint32_t *cnt;     // [slot] its photons; then the position of its first photon
  uint32_t *sum;     // [chunk of CLS_CHUNK_FLAGS slots][NCLS] photons; then the position of their first
  float *rec;        // records of rec_words floats: slot, sub-step, index, tag; position, weight; id,
                     // photon momentum (; E, B at 16), so that the writing pass reads its parent in one
                     // piece and not from 15 arrays
  uint32_t rec_cap;  // records
  int rec_words;     // 16, or 24 where the photons take fields of their own
  uint32_t *idx;     // [position] its record
  unsigned int *n;   // [0] records asked for, [1] leptons to replay, [2], [3] of the pass being written
  int32_t *replay;   // slots of the leptons whose records found no room
  uint32_t *replay_cnt;  // their photons
};
constexpr uint8_t FLAG_REPLAY = 0x80;

struct OnePassArgs {
  Sp<float> sp[2];
  int nsp;
  Sp<float> ph;
  Fld<float> f;
  Consts C;
  Tables<float> T;
  Out o;
  int64_t step;
  const int64_t *d_step;
  const float *w_up_row;       // W_rad <= w_up_row[j] chi / gamma for ln chi >= row j
  float chi_tab_lo, chi_tab_hi;  // chi range of the rate tables
  float delta_tab_lo;            // lower end of the forward table in delta
  const uint32_t *mlp_frag;  // learned sampler: BF16 fragments and the FP32 small
  const float *mlp_fw;       // layers, in global memory (read through L1)
  float4 *net_rec;           // records of the deferred network emissions
  unsigned long long *net_n; // their count
  int64_t net_cap;
  bool aligned16;  // every array a slice is read from starts on a 16-byte boundary
  OrdArgs ord;
};

// Dynamic shared memory per warp: the prefetch words and ids of a slice, the
// pool and its lists.  The tables are read through L1.
template <int FM, bool ORD> __host__ __device__ constexpr size_t warp_smem() {
  const size_t b = 32 * ((size_t)stream_words<FM>() * 4 + 8) +
                   (size_t)pool_cap<FM, ORD>() * (4 * pool_words<FM, ORD>() + (ORD ? 3 : 2));
  return (b + 15) & ~(size_t)15;  // (cp.async)
}

// Learned-sampler emissions deferred to the dense pass: one record per
// emission, 16 bytes -- the lepton's index (species in the top bit) and kappa
// -- plus, with grid fields, its position before the push (so that the dense
// pass gathers the same fields), 32 bytes.  Everything else (the pushed
// momentum, gamma, the direction, chi, the id) the dense pass reads or
// recomputes with the same expressions.
template <int FM> __host__ __device__ constexpr int net_stride() { return FM == FM_GRID ? 3 : 1; }  // float4 per record

// gamma and the unit direction of a pushed momentum, as a deferred particle
// gets them in the heavy phase and in the dense pass alike
__device__ __forceinline__ void gamma_dir(float px, float py, float pz, float &g, float &nx, float &ny,
                                          float &nz) {
  g = sqrtf(1.f + px * px + py * py + pz * pz);
  const float pm = sqrtf(px * px + py * py + pz * pz);
  nx = ny = nz = 0.f;
  if (pm > 0.f) {
    const float ip = 1.f / pm;
    nx = px * ip; ny = py * ip; nz = pz * ip;
  }
}


// N = max(1, ceil(W Dt / wdt_max)), capped at max_substeps (status bit).
__device__ __forceinline__ int64_t substep_count_op(const Consts &C, float W, float dt, float wdt_max,
                                                    uint32_t &status) {
  const float wdt = W * dt;
  if (!(wdt > wdt_max)) return 1;
  float nn = ceilf(wdt / wdt_max);
  if (nn > (float)C.max_substeps) {
    nn = (float)C.max_substeps;
    status |= QED_STATUS_SUBSTEPS;
  }
  return (int64_t)nn;
}

__device__ __forceinline__ void put8(float *p, float a, float b, float c, float d, float e, float f, float g, float h) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d),
               "f"(e), "f"(f), "f"(g), "f"(h)
               : "memory");
}

// Method I on the sub-steps that a draw serves (2j and 2j + 1; a chain may
// enter at the odd one): the next state, L_FREE at the end of the chain.
__device__ __forceinline__ int draw_two(const U4 &r, float thr, int N, int &k, uint32_t &r2) {
  if (!(k & 1)) {
    if (thr > unif<float>(r.x)) { r2 = r.y; return L_PEND; }
    if (++k >= N) return L_FREE;
  }
  if (thr > unif<float>(r.z)) { r2 = r.w; return L_PEND; }
  return ++k >= N ? L_FREE : L_SCAN;
}

template <int FM, int MODE, bool MLP, bool ORD>
__global__ void __launch_bounds__(OP_THREADS, 1) k_lepton_onepass(OnePassArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t s_hist[64];
  __shared__ BlockTally bt;
  __shared__ long long s_meta[4];
  __shared__ unsigned long long s_deferred;
  __shared__ unsigned long long s_src[2][13];  // the arrays a slice is read from
  constexpr int NV = stream_words<FM>(), PCAP = pool_cap<FM, ORD>(), W_CNT = w_cnt<FM>(), W_POS = W_CNT + 1;
  constexpr bool KEEP_X = ORD && FM == FM_GRID;  // the stored position stays until the chain's end
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  unsigned char *const mine = smem_raw + (size_t)wid * warp_smem<FM, ORD>();
  uint64_t *const pf_id = reinterpret_cast<uint64_t *>(mine);                 // [32]
  float *const pf = reinterpret_cast<float *>(mine + 256);                    // [NV][32]
  uint32_t *const pool = reinterpret_cast<uint32_t *>(pf + NV * 32);          // [words][PCAP]
  uint8_t *const list = reinterpret_cast<uint8_t *>(pool + pool_words<FM, ORD>() * PCAP);  // [2][PCAP]
  uint8_t *const cls = list + 2 * PCAP;  // ORD: [PCAP]
  block_tally_init(&bt);
  if (threadIdx.x < 64) s_hist[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    s_meta[0] = *(volatile int64_t *)A.sp[0].d_n;
    s_meta[1] = A.nsp > 1 ? *(volatile int64_t *)A.sp[1].d_n : 0;
    s_meta[2] = (long long)A.o.scan.sync[2];
    s_deferred = 0;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const Sp<float> &S = A.sp[k];
      const void *src[13] = {S.x, S.y, S.z, S.px, S.py, S.pz, S.ex, S.ey, S.ez, S.bx, S.by, S.bz, S.id};
#pragma unroll
      for (int c = 0; c < 13; ++c) s_src[k][c] = reinterpret_cast<unsigned long long>(src[c]);
    }
  }
  __syncthreads();
  const int64_t step_ = A.d_step ? *A.d_step : A.step;
  // slots fit 32 bits: a species holds at most 2^30 - 4096 particles
  const uint32_t n0 = (uint32_t)s_meta[0], n1 = (uint32_t)s_meta[1];
  const uint32_t epoch = (uint32_t)s_meta[2];
  const uint32_t slots0 = (n0 + TILE - 1) / TILE * TILE, nslots = slots0 + (n1 + TILE - 1) / TILE * TILE;
  // consecutive slices go to different SMs
  const uint32_t stride = gridDim.x * OP_THREADS;
  uint32_t slot = (wid * gridDim.x + blockIdx.x) * 32 + lane;
  const float inv_aS = A.C.f_inv_aS, dt = A.C.f_dt, wdt_max = A.C.f_wdt_max;
  Tally tl;
  tl.clear();
  uint32_t deferred = 0;  // new particles taken by this lane

  // species and index of a slot (species 1 starts at a tile of its own)
  auto slot_index = [&](uint32_t sl, int &si, uint32_t &i) {
    si = sl < slots0 ? 0 : 1;
    i = si ? sl - slots0 : sl;
  };
  // ---- the pool's lists: entries of a state in any order (lengths warp-uniform)
  int len[4] = {0, 0, 0, PCAP};
  for (int q = lane; q < PCAP; q += 32) list[list_at<PCAP>(L_FREE, q)] = (uint8_t)q;
  __syncwarp();
  auto word = [&](int w, int e) -> uint32_t & { return pool[w * PCAP + e]; };
  auto real = [&](int w, int e) -> float & { return reinterpret_cast<float *>(pool)[w * PCAP + e]; };
  // file entry e of each lane whose next state is s
  auto file = [&](int s, bool in, int e) {
    const unsigned m = __ballot_sync(0xFFFFFFFFu, in);
    if (in) list[list_at<PCAP>(s, len[s] + __popc(m & lt_mask))] = (uint8_t)e;
    len[s] += __popc(m);
  };
  auto fields_of = [&](int e, float E[3], float B[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      E[c] = FM == FM_UNIFORM ? A.f.e[c] : real(W_FIELDS + c, e);
      B[c] = FM == FM_UNIFORM ? A.f.b[c] : real(W_FIELDS + 3 + c, e);
    }
  };
  // The end of a chain: its lepton's state -- the recoiled momentum (direction
  // n and g) if it has emitted, else nothing more (its pushed state is stored).
  // ORD: the pushed momentum (and with grid fields the position) too, which
  // only this stores -- unless a photon's record was lost: what is stored then
  // stays as it was for the replay.
  auto finish = [&](int e, uint32_t kw, float g, float nx, float ny, float nz) {
    if (!ORD && !(kw & EMITTED)) return;
    const uint32_t sl = word(W_SLOT, e);
    int si;
    uint32_t i;
    slot_index(sl, si, i);
    const Sp<float> &S = A.sp[si];
    if (ORD) {
      if (kw & EMITTED) {
        A.ord.flags[sl] = cls[e] | (kw & LOST ? FLAG_REPLAY : 0);
        const uint32_t cnt = word(W_CNT, e);
        A.ord.cnt[sl] = cnt;
        atomicAdd(&A.ord.sum[sl / CLS_CHUNK_FLAGS * NCLS + cls[e] - 1], cnt);
        if (kw & LOST) {
          const unsigned r = atomicAdd(&A.ord.n[1], 1u);
          A.ord.replay[r] = (int32_t)sl;
          A.ord.replay_cnt[r] = cnt;
          return;
        }
      }
      if (MODE != MODE_EMIT && KEEP_X) {
        S.x[i] = real(W_POS, e); S.y[i] = real(W_POS + 1, e); S.z[i] = real(W_POS + 2, e);
      }
      if (!(kw & EMITTED)) {  // n is the pushed momentum
        if (MODE != MODE_EMIT) { S.px[i] = nx; S.py[i] = ny; S.pz[i] = nz; }
        return;
      }
    }
    const float pm = sqrtf((g - 1.f) * (g + 1.f));
    S.px[i] = pm * nx; S.py[i] = pm * ny; S.pz[i] = pm * nz;
  };

  // The next slice's words are copied into shared memory (cp.async) as soon as
  // the current ones have been read from there: 16 bytes per lane and copy
  // where the arrays are aligned (a slice is 8 such pieces of each float array
  // and 16 of the ids; past L1, which the tables need), else each lane its
  // own particle's words.
  constexpr int PIECES = (NV * 8 + 31) / 32;  // 16-byte pieces of a slice per lane
  const float *piece[PIECES];
  const uint64_t *piece_id = nullptr;
  int piece_si = -1;
  auto prefetch = [&](uint32_t sl) {
    const int si = sl < slots0 ? 0 : 1;
    const uint32_t i = si ? sl - slots0 : sl, n = si ? n1 : n0, q0 = i - lane;
    if (A.aligned16) {
      if (si != piece_si) {  // this lane's pieces of the species' arrays
        piece_si = si;
#pragma unroll
        for (int t = 0; t < PIECES; ++t) {
          const int q = t * 32 + lane;
          piece[t] = reinterpret_cast<const float *>(s_src[si][q < NV * 8 ? q >> 3 : 0]) + (q & 7) * 4;
        }
        piece_id = reinterpret_cast<const uint64_t *>(s_src[si][12]) + 2 * (lane & 15);
      }
      if (q0 + 32 <= n) {
#pragma unroll
        for (int t = 0; t < PIECES; ++t)
          if (t * 32 + lane < NV * 8) cp_async16(pf + (t * 32 + lane) * 4, piece[t] + q0, 16);
        if (lane < 16) cp_async16(pf_id + 2 * lane, piece_id + q0, 16);
      } else if (q0 < n) {  // the species' last slice
        const int left = (int)(n - q0), p = (lane & 7) * 4;
#pragma unroll
        for (int t = 0; t < PIECES; ++t)
          if (t * 32 + lane < NV * 8 && p < left)
            cp_async16(pf + (t * 32 + lane) * 4, piece[t] + q0, min(left - p, 4) * 4);
        if (lane < 16 && 2 * lane < left) cp_async16(pf_id + 2 * lane, piece_id + q0, min(left - 2 * lane, 2) * 8);
      }
    } else if (i < n) {
#pragma unroll
      for (int c = 0; c < NV; ++c) cp_async<4>(pf + c * 32 + lane, reinterpret_cast<const float *>(s_src[si][c]) + i);
      cp_async<8>(pf_id + lane, reinterpret_cast<const uint64_t *>(s_src[si][12]) + i);
    }
    cp_async_commit();
  };
  // the pushed state of a slice's lepton (ORD: of a deferred one, `keep`, what
  // finish does not store)
  auto store_pushed = [&](const Sp<float> &S, uint32_t i, bool keep, float x, float y, float z, float px, float py,
                          float pz) {
    if (!(KEEP_X && keep)) { S.x[i] = x; S.y[i] = y; S.z[i] = z; }
    if (!(ORD && keep)) { S.px[i] = px; S.py[i] = py; S.pz[i] = pz; }
  };
  if (slot < nslots) prefetch(slot);

  for (;;) {
    // nslots is a multiple of 32: every lane of a warp sees the same
    const bool streaming = slot < nslots;
    // the fullest state (ties to the later one, which is nearer its end)
    int phase = L_RATE, most = len[L_RATE];
    if (len[L_SCAN] >= most) { phase = L_SCAN; most = len[L_SCAN]; }
    if (len[L_PEND] >= most) { phase = L_PEND; most = len[L_PEND]; }
    if (streaming && most < 32 && len[L_FREE] >= 32) {
      // ---- a slice of leptons
      cp_async_wait<0>();
      __syncwarp();
      int si;
      uint32_t i;
      slot_index(slot, si, i);
      bool heavy = false;
      if (ORD) A.ord.flags[slot] = 0;
      float x = pf[lane], y = pf[32 + lane], z = pf[64 + lane];
      float px = pf[96 + lane], py = pf[128 + lane], pz = pf[160 + lane];
      float E[3] = {0.f, 0.f, 0.f}, B[3] = {0.f, 0.f, 0.f};
      if (FM == FM_PER_PARTICLE) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          E[c] = pf[(6 + c) * 32 + lane];
          B[c] = pf[(9 + c) * 32 + lane];
        }
      }
      const uint64_t pid = pf_id[lane];
      const uint32_t next = slot + stride;
      __syncwarp();  // the words are read by all lanes
      if (next < nslots) prefetch(next);
      if (i < (si ? n1 : n0)) {
        if (FM != FM_PER_PARTICLE) get_fields<float, FM>(A.sp[0], A.f, i, x, y, z, E, B);
        float g;
        if (MODE != MODE_EMIT) {
          g = boris(px, py, pz, E, B, si ? A.sp[1].q : A.sp[0].q, dt);
          const float ig = r_div(dt, g);
          x += px * ig; y += py * ig; z += pz * ig;
        } else {
          g = sqrtf(1.f + px * px + py * py + pz * pz);
        }
        if (!(g < 1e30f)) {
          tl.status |= QED_STATUS_NONFINITE;  // left as it was
        } else {
          const float chi = chi_lepton(px, py, pz, g, E[0], E[1], E[2], B[0], B[1], B[2], inv_aS);
          // one sub-step and no event, for sure, from the rate bound of the
          // table row at or below ln chi, and r1
          const float fj = (r_log(chi) - A.T.gl.x0) * A.T.gl.inv_h;
          const int j = fj >= 0.f ? (fj < (float)(A.T.gl.n - 1) ? (int)fj : A.T.gl.n - 1) : 0;
          const float wdt_up = r_div(__ldg(A.w_up_row + j) * dt * chi, g);
          heavy = true;
          if (wdt_up <= wdt_max) {
            const U4 r = draw(A.C, pid, step_, 0, STREAM_EMIT);
            heavy = wdt_up > unif<float>(r.x);
          }
          if (!heavy) {
            tl.substeps += 1;
            // (ORD: as photon_rate counts, the cut below the forward table too)
            const float c = A.C.f_xi_min_energy;
            if (chi > 0.f && (chi < A.chi_tab_lo || chi > A.chi_tab_hi) && (!ORD || g > c)) {
              tl.domain += 1;
              tl.status |= QED_STATUS_DOMAIN;
            }
            if (ORD && c > 0.f && g > c && c * (2.f / 3.f) < A.delta_tab_lo * fminf(chi, A.chi_tab_hi) * (g - c)) {
              tl.domain += 1;
              tl.status |= QED_STATUS_DOMAIN;
            }
          }
          if (MODE != MODE_EMIT) {
            if (si == 0) store_pushed(A.sp[0], i, heavy, x, y, z, px, py, pz);
            else store_pushed(A.sp[1], i, heavy, x, y, z, px, py, pz);
          }
        }
      }
      // the deferred ones take free entries
      const unsigned hm = __ballot_sync(0xFFFFFFFFu, heavy);
      if (heavy) {
        const int r = __popc(hm & lt_mask);
        const int e = list[list_at<PCAP>(L_FREE, len[L_FREE] - 1 - r)];
        word(W_SLOT, e) = slot;
        word(W_ID0, e) = (uint32_t)pid;
        word(W_ID1, e) = (uint32_t)(pid >> 32);
        real(W_VX, e) = px; real(W_VY, e) = py; real(W_VZ, e) = pz;
        word(W_N, e) = 0u;
        word(W_K, e) = 0u;
        if (ORD) word(W_CNT, e) = 0u;
        if (KEEP_X) { real(W_POS, e) = x; real(W_POS + 1, e) = y; real(W_POS + 2, e) = z; }
        if (FM != FM_UNIFORM) {
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            real(W_FIELDS + c, e) = E[c];
            real(W_FIELDS + 3 + c, e) = B[c];
          }
        }
        list[list_at<PCAP>(L_RATE, len[L_RATE] + r)] = (uint8_t)e;
      }
      const int nh = __popc(hm);
      len[L_FREE] -= nh;
      len[L_RATE] += nh;
      slot = next;
      __syncwarp();  // the entries, and the pushed state written above, are visible to the warp
      continue;
    }
    if (most == 0) break;  // (a pool with nothing to run has room, so nothing is left to stream)
    const int take = min(most, 32);
    const bool act = lane < take;
    const int e = act ? list[list_at<PCAP>(phase, most - 1 - lane)] : 0;
    __syncwarp();  // the entries are taken before others are filed
    int st = -1;
    if (phase == L_RATE) {
      len[L_RATE] -= take;
      // ---- chi (Eq. 2) and the exact rate; a new particle also gets N; then
      // the first draw
      float kap = 0.f;
      bool net = false;
      float E[3], B[3];
      if (act) {
        fields_of(e, E, B);
        const float vx = real(W_VX, e), vy = real(W_VY, e), vz = real(W_VZ, e);
        float px = vx, py = vy, pz = vz, g;
        int N = (int)word(W_N, e);
        const uint32_t kw = word(W_K, e);
        const bool fresh = N == 0;
        if (fresh) {
          g = sqrtf(1.f + px * px + py * py + pz * pz);
        } else {  // after an emission: (vx, vy, vz) is the direction
          g = real(W_G, e);
          const float pm = sqrtf((g - 1.f) * (g + 1.f));
          px = pm * vx; py = pm * vy; pz = pm * vz;
        }
        const float chi = chi_lepton(px, py, pz, g, E[0], E[1], E[2], B[0], B[1], B[2], inv_aS);
        const RateOut<float> ro = photon_rate(A.T.R, A.T.F, A.T, A.C, chi, g, tl);
        if (fresh) {
          N = (int)substep_count_op(A.C, ro.W, dt, wdt_max, tl.status);
          tl.substeps += N;
          word(W_N, e) = (uint32_t)N;
          real(W_G, e) = g;
          if (ORD) {  // the class, as the ordered path bins W Dt
            const float wdt = ro.W * dt, q = r_div(wdt, wdt_max);
            cls[e] = !(wdt > wdt_max) ? 1 : q <= 3.f ? 2 : q <= 7.f ? 3 : q <= 15.f ? 4 : 5;
          }
        }
        const float thr = ro.W * (dt / (float)N);
        real(W_CHI, e) = chi;
        real(W_THR, e) = thr;
        real(W_KMIN, e) = ro.kmin;
        int k = (int)(kw & K_MASK);
        uint32_t r2 = 0;
        const uint64_t pid = (uint64_t)word(W_ID0, e) | ((uint64_t)word(W_ID1, e) << 32);
        st = draw_two(draw(A.C, pid, step_, k >> 1, STREAM_EMIT), thr, N, k, r2);
        // ORD counts as deferred what the multi-pass path does: an event or W Dt > wdt_max
        if (fresh) deferred += !ORD || cls[e] > 1 || st == L_PEND ? 1 : 0;
        word(W_K, e) = (uint32_t)k | (kw & ~K_MASK);
        if (st == L_PEND) word(W_R2, e) = r2;
        if (st == L_FREE) finish(e, kw, g, vx, vy, vz);
        if (MLP && st == L_PEND && N == 1) {
          // an event of a one-sub-step particle inside the network's domain
          // takes its xi from the learned sampler, in the dense pass that
          // follows this kernel: a record here (one per such particle: at
          // most n0 + n1, which the records hold), no photon yet
          kap = photon_kappa(ro.kmin, unif<float>(r2), unif<float>(~r2));
          const float lchi = chi > 0.f ? logf(chi) : MLP_L_LO - 1.f;
          net = lchi >= MLP_L_LO && lchi <= MLP_L_HI && kap >= MLP_K_LO && kap <= MLP_K_HI;
        }
      }
      if (MLP) {
        const unsigned nm = __ballot_sync(0xFFFFFFFFu, net);
        if (nm) {
          const int leader = __ffs(nm) - 1;
          unsigned long long base = 0;
          if (lane == leader) base = atomicAdd(A.net_n, (unsigned long long)__popc(nm));
          base = __shfl_sync(0xFFFFFFFFu, base, leader);
          if (net) {
            constexpr int RS = net_stride<FM>();
            const unsigned long long r = base + __popc(nm & lt_mask);
            if (r < (unsigned long long)(A.net_cap / RS)) {
              int si;
              uint32_t i;
              slot_index(word(W_SLOT, e), si, i);
              float4 *R = A.net_rec + RS * r;
              R[0] = make_float4(__uint_as_float(i), __uint_as_float((uint32_t)si << 31), kap, E[0]);
              if (FM == FM_GRID) {
                R[1] = make_float4(E[1], E[2], B[0], B[1]);
                R[2] = make_float4(B[2], 0.f, 0.f, 0.f);
              }
            } else {  // only with counts beyond the species' capacities
              tl.dropped += 1;
              tl.status |= QED_STATUS_CAPACITY;
            }
            st = L_FREE;
          }
        }
      }
    } else if (phase == L_SCAN) {
      len[L_SCAN] -= take;
      // ---- the next four sub-steps, from two independent draws
      if (act) {
        const uint64_t pid = (uint64_t)word(W_ID0, e) | ((uint64_t)word(W_ID1, e) << 32);
        const uint32_t kw = word(W_K, e);
        const int N = (int)word(W_N, e);
        const float thr = real(W_THR, e);
        int k = (int)(kw & K_MASK);
        uint32_t r2 = 0;
        const U4 ra = draw(A.C, pid, step_, k >> 1, STREAM_EMIT);
        const U4 rb = draw(A.C, pid, step_, (k >> 1) + 1, STREAM_EMIT);
        st = draw_two(ra, thr, N, k, r2);
        if (st == L_SCAN) st = draw_two(rb, thr, N, k, r2);
        word(W_K, e) = (uint32_t)k | (kw & ~K_MASK);
        if (st == L_PEND) word(W_R2, e) = r2;
        if (st == L_FREE && (ORD || (kw & EMITTED)))
          finish(e, kw, real(W_G, e), real(W_VX, e), real(W_VY, e), real(W_VZ, e));
      }
    } else {
      len[L_PEND] -= take;
      // ---- emission: kappa and ln delta from the inverse table (Eq. 7), xi,
      // the recoil and the photon, whose slots come from one atomic (ORD: its
      // record, likewise)
      unsigned long long base = 0;
      if (lane == 0)
        base = ORD ? atomicAdd(A.ord.n, (unsigned)take)
                   : atomicAdd(reinterpret_cast<unsigned long long *>(A.ph.d_n), (unsigned long long)take);
      float x = 0.f, y = 0.f, z = 0.f, w = 0.f, eph = 0.f, g2 = 1.f, nx = 0.f, ny = 0.f, nz = 0.f;
      uint32_t sl = 0, tag = 0, kw = 0;
      if (act) {  // (the parent's words and the slots are on their way during the look-up)
        sl = word(W_SLOT, e);
        int si;
        uint32_t i;
        slot_index(sl, si, i);
        const Sp<float> &S = A.sp[si];
        if (KEEP_X) { x = real(W_POS, e); y = real(W_POS + 1, e); z = real(W_POS + 2, e); }
        else { x = S.x[i]; y = S.y[i]; z = S.z[i]; }
        w = S.w[i];
        if (S.tag) tag = S.tag[i];
        const float chi = real(W_CHI, e), g = real(W_G, e);
        const uint32_t r2 = word(W_R2, e);
        kw = word(W_K, e);
        const float kap = photon_kappa(real(W_KMIN, e), unif<float>(r2), unif<float>(~r2));
        float l = r_log(chi);  // (clamped as in photon_rate)
        l = l < A.T.gl.lo ? A.T.gl.lo : l > A.T.gl.hi ? A.T.gl.hi : l;
        const XiOut<float> xo = xi_from_lndelta(chi, photon_lndelta_table(A.T.Y, A.T, l, kap, tl));
        g2 = g * xo.omxi;
        eph = g * xo.xi;
        if (g2 < 1.f) { g2 = 1.f; eph = g - 1.f; }
        const int b = spec_bin(A.C, eph);
        if (b >= 0) atomicAdd(&s_hist[b], 1u);
        nx = real(W_VX, e); ny = real(W_VY, e); nz = real(W_VZ, e);
        if (!(kw & EMITTED)) {  // the direction, from the pushed momentum
          float gg;
          gamma_dir(nx, ny, nz, gg, nx, ny, nz);
          real(W_VX, e) = nx; real(W_VY, e) = ny; real(W_VZ, e) = nz;
        }
      }
      base = __shfl_sync(0xFFFFFFFFu, base, 0);
      if (act) {
        int k = (int)(kw & K_MASK);
        const int64_t pos = (int64_t)base + lane;
        if (ORD) {
          const uint32_t j = word(W_CNT, e);
          word(W_CNT, e) = j + 1;
          if (pos < (int64_t)A.ord.rec_cap) {
            float *r = A.ord.rec + pos * A.ord.rec_words;
            put8(r, __uint_as_float(sl), __uint_as_float((uint32_t)k), __uint_as_float(j), __uint_as_float(tag), x, y, z, w);
            put8(r + 8, real(W_ID0, e), real(W_ID1, e), eph * nx, eph * ny, eph * nz, 0.f, 0.f, 0.f);
            if (A.ord.rec_words > 16) {
              float E[3], B[3];
              fields_of(e, E, B);
              put8(r + 16, E[0], E[1], E[2], B[0], B[1], B[2], 0.f, 0.f);
            }
          } else {
            kw |= LOST;
          }
        } else if (pos >= A.ph.cap) {
          tl.dropped += 1;
          tl.status |= QED_STATUS_CAPACITY;
        } else {
          const uint64_t pid = (uint64_t)word(W_ID0, e) | ((uint64_t)word(W_ID1, e) << 32);
          const U4 cid = draw(A.C, pid, step_, k, STREAM_PHOTON_ID);
          float E[3], B[3];
          fields_of(e, E, B);
          write_child(A.ph, pos, x, y, z, eph * nx, eph * ny, eph * nz, w,
                      (uint64_t)cid.x | ((uint64_t)cid.y << 32), E, B, tag);
        }
        tl.events += 1;
        // the rate for the remaining sub-steps, or the end of the chain
        st = ++k >= (int)word(W_N, e) ? L_FREE : L_RATE;
        kw = (uint32_t)k | (kw & ~K_MASK) | EMITTED;
        real(W_G, e) = g2;
        word(W_K, e) = kw;
        if (st == L_FREE) finish(e, kw, g2, nx, ny, nz);
      }
    }
    if (phase == L_PEND) {
      file(L_RATE, st == L_RATE, e);
    } else {
      file(L_SCAN, st == L_SCAN, e);
      file(L_PEND, st == L_PEND, e);
    }
    file(L_FREE, st == L_FREE, e);
    __syncwarp();
  }
  cp_async_wait<0>();

  tally_flush(&bt, tl);
  {
    uint32_t d = deferred;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xFFFFFFFFu, d, o);
    if (lane == 0 && d) atomicAdd(&s_deferred, (unsigned long long)d);
  }
  __syncthreads();
  if (threadIdx.x < 64) bt.hist[threadIdx.x] = s_hist[threadIdx.x];
  __syncthreads();
  block_tally_commit(&bt, A.o.cnt, 0);
  if (threadIdx.x == 0) {
    if (s_deferred) atomicAdd(reinterpret_cast<unsigned long long *>(&A.o.cnt->deferred), s_deferred);
    // the last CTA to finish clamps the photon count to the capacity (the
    // slots past it were counted as dropped) and resets the shared counters
    __threadfence();
    const unsigned int prev = atomicAdd(&A.o.scan.sync[1], 1u);
    if (prev == gridDim.x - 1) {
      __threadfence();
      if (!ORD) {
        int64_t *dn = A.ph.d_n;
        if (*(volatile int64_t *)dn > A.ph.cap) *dn = A.ph.cap;
      }
      A.o.scan.sync[0] = 0u;
      A.o.scan.sync[1] = 0u;
      A.o.scan.sync[2] = epoch + 1u;
      __threadfence();
    }
  }
}

// ---- ordered appends: positions and photons ------------------------------
// Positions: the class totals, then every chunk's first position per class (one
// CTA).  Publishes the photon count; what does not fit is counted as dropped.
constexpr int ORD_SCAN_THREADS = 1024, ORD_SCAN_CHUNKS = 2;  // chunks per thread and round
struct OrdScanArgs {
  OrdArgs ord;
  const int64_t *n0, *n1;
  int64_t *ph_n, *meta;  // meta: [0] photons of the pass, [1] photon count before
  int64_t ph_cap;
  qed_counters *cnt;
};

// Exclusive scan over the CTA of a pair of sums in one word; sm: 33 words, the
// totals in sm[32].
__device__ __forceinline__ unsigned long long scan_pair(unsigned long long v, unsigned long long *sm) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned long long incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) sm[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    const unsigned long long w = lane < nw ? sm[lane] : 0ull;
    unsigned long long wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long u = __shfl_up_sync(0xFFFFFFFFu, wi, o);
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

__device__ __forceinline__ uint32_t ord_slots(const int64_t *n0, const int64_t *n1) {
  const uint32_t a = (uint32_t)*(volatile const int64_t *)n0, b = n1 ? (uint32_t)*(volatile const int64_t *)n1 : 0u;
  return (a + TILE - 1) / TILE * TILE + (b + TILE - 1) / TILE * TILE;
}

__global__ void __launch_bounds__(ORD_SCAN_THREADS) k_ord_scan(OrdScanArgs A) {
  __shared__ unsigned long long sm[33];
  __shared__ uint32_t s_tot[NCLS];
  const unsigned asked = *(volatile unsigned *)A.ord.n;
  const int64_t nph = *(volatile int64_t *)A.ph_n;
  if (threadIdx.x < NCLS) s_tot[threadIdx.x] = 0;
  __syncthreads();
  uint32_t total = 0;
  if (asked) {
    const uint32_t nchunks = (ord_slots(A.n0, A.n1) + CLS_CHUNK_FLAGS - 1) / CLS_CHUNK_FLAGS;
    uint32_t mine[NCLS] = {0, 0, 0, 0, 0};
    for (uint32_t c = threadIdx.x; c < nchunks; c += ORD_SCAN_THREADS)
#pragma unroll
      for (int k = 0; k < NCLS; ++k) mine[k] += A.ord.sum[c * NCLS + k];
#pragma unroll
    for (int k = 0; k < NCLS; ++k) {
      const uint32_t v = __reduce_add_sync(0xFFFFFFFFu, mine[k]);
      if ((threadIdx.x & 31) == 0 && v) atomicAdd(&s_tot[k], v);
    }
    __syncthreads();
    uint32_t carry[NCLS + 1];
#pragma unroll
    for (int k = 0; k < NCLS; ++k) {
      carry[k] = total;
      total += s_tot[k];
    }
    carry[NCLS] = 0;
    for (uint32_t r0 = 0; r0 < nchunks; r0 += ORD_SCAN_THREADS * ORD_SCAN_CHUNKS) {
      const uint32_t c0 = r0 + threadIdx.x * ORD_SCAN_CHUNKS;
      uint32_t t[NCLS + 1] = {0, 0, 0, 0, 0, 0};
#pragma unroll
      for (int j = 0; j < ORD_SCAN_CHUNKS; ++j)
        if (c0 + j < nchunks)
#pragma unroll
          for (int k = 0; k < NCLS; ++k) t[k] += A.ord.sum[(c0 + j) * NCLS + k];
#pragma unroll
      for (int q = 0; q < (NCLS + 1) / 2; ++q) {  // (sums of photons stay below 2^32)
        const unsigned long long v = (unsigned long long)t[2 * q] | ((unsigned long long)t[2 * q + 1] << 32);
        const unsigned long long ex = scan_pair(v, sm), tt = sm[32];
        t[2 * q] = carry[2 * q] + (uint32_t)ex;
        t[2 * q + 1] = carry[2 * q + 1] + (uint32_t)(ex >> 32);
        carry[2 * q] += (uint32_t)tt;
        carry[2 * q + 1] += (uint32_t)(tt >> 32);
        __syncthreads();  // sm[32] is read
      }
#pragma unroll
      for (int j = 0; j < ORD_SCAN_CHUNKS; ++j)
        if (c0 + j < nchunks)
#pragma unroll
          for (int k = 0; k < NCLS; ++k) {
            const uint32_t v = A.ord.sum[(c0 + j) * NCLS + k];
            A.ord.sum[(c0 + j) * NCLS + k] = t[k];
            t[k] += v;
          }
    }
  }
  if (threadIdx.x == 0) {
    A.meta[0] = total;
    A.meta[1] = nph;
    const int64_t after = nph + total < A.ph_cap ? nph + total : A.ph_cap;
    const int64_t written = after > nph ? after - nph : 0;
    *A.ph_n = after;
    if (written < total) {
      atomicAdd(reinterpret_cast<unsigned long long *>(&A.cnt->dropped), (unsigned long long)(total - written));
      atomicOr(&A.cnt->status, (unsigned)QED_STATUS_CAPACITY);
    }
    // the counts of this pass for the writing pass, and the next one's start
    A.ord.n[2] = asked;
    A.ord.n[3] = A.ord.n[1];
    A.ord.n[0] = A.ord.n[1] = 0u;
  }
}

// Every emitting lepton's first position: its chunk's of its class, and the
// photons of the class before it in the chunk.
__global__ void __launch_bounds__(TILE) k_ord_offsets(OrdArgs O, const int64_t *n0, const int64_t *n1) {
  constexpr int ITEMS = CLS_CHUNK_FLAGS / TILE;  // 8 flags, one 8-byte load
  constexpr int WARPS = TILE / 32;
  __shared__ uint32_t s_warp[2][WARPS][NCLS];  // (two, so that one barrier a chunk does)
  if (*(volatile unsigned *)&O.n[2] == 0) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t nslots = ord_slots(n0, n1), nchunks = (nslots + CLS_CHUNK_FLAGS - 1) / CLS_CHUNK_FLAGS;
  int buf = 0;
  for (uint32_t c = blockIdx.x; c < nchunks; c += gridDim.x, buf ^= 1) {
    const uint32_t first = c * CLS_CHUNK_FLAGS + threadIdx.x * ITEMS;
    uint2 raw = make_uint2(0u, 0u);
    if (first < nslots) raw = *reinterpret_cast<const uint2 *>(O.flags + first);  // (slots come in tiles)
    uint32_t n[ITEMS], t[NCLS] = {0, 0, 0, 0, 0};
    int k[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      k[j] = (int)((j < 4 ? raw.x >> 8 * j : raw.y >> 8 * (j - 4)) & 0x7Fu);  // class, 0: none
      n[j] = k[j] ? O.cnt[first + j] : 0u;
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
#pragma unroll
      for (int q = 0; q < NCLS; ++q) t[q] += k[j] == q + 1 ? n[j] : 0u;
#pragma unroll
    for (int q = 0; q < NCLS; ++q) {  // the lanes before, and the warp's total
      uint32_t incl = t[q];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += u;
      }
      if (lane == 31) s_warp[buf][wid][q] = incl;
      t[q] = incl - t[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NCLS; ++q) {
      t[q] += O.sum[c * NCLS + q];
      for (int w = 0; w < wid; ++w) t[q] += s_warp[buf][w][q];
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
#pragma unroll
      for (int q = 0; q < NCLS; ++q)
        if (k[j] == q + 1) {
          O.cnt[first + j] = t[q];
          t[q] += n[j];
        }
  }
}

// The record of every position (its lepton's first position plus its index),
// so that the writing pass runs in position order and its stores to the
// photons' arrays are contiguous.
__global__ void __launch_bounds__(TILE) k_ord_index(OrdArgs O, const int64_t *meta, int64_t ph_cap) {
  const unsigned asked = *(volatile unsigned *)&O.n[2];
  const unsigned nrec = asked < O.rec_cap ? asked : O.rec_cap;
  const int64_t room = ph_cap - meta[1];
  for (unsigned r = blockIdx.x * TILE + threadIdx.x; r < nrec; r += gridDim.x * TILE) {
    const float4 a = *reinterpret_cast<const float4 *>(O.rec + (size_t)r * O.rec_words);
    const uint32_t sl = __float_as_uint(a.x), q = O.cnt[sl] + __float_as_uint(a.z);
    if (q < room && !(O.flags[sl] & FLAG_REPLAY)) O.idx[q] = r;
  }
}

struct OrdWriteArgs {
  Sp<float> ph;
  Fld<float> f;
  Consts C;
  OrdArgs ord;
  const int64_t *meta;
  int64_t step;
  const int64_t *d_step;
};
__global__ void __launch_bounds__(TILE) k_ord_write(OrdWriteArgs A) {
  const unsigned asked = *(volatile unsigned *)&A.ord.n[2];
  if (asked == 0) return;
  const unsigned nrec = asked < A.ord.rec_cap ? asked : A.ord.rec_cap;
  const bool replays = *(volatile unsigned *)&A.ord.n[3] != 0;
  const int64_t step_ = A.d_step ? *A.d_step : A.step, nph = A.meta[1];
  int64_t total = A.meta[0];
  if (total > A.ph.cap - nph) total = A.ph.cap - nph;
  for (int64_t q = blockIdx.x * (int64_t)TILE + threadIdx.x; q < total; q += (int64_t)gridDim.x * TILE) {
    const unsigned r = A.ord.idx[q];
    if (replays && r >= nrec) continue;
    const float4 *R = reinterpret_cast<const float4 *>(A.ord.rec + (size_t)r * A.ord.rec_words);
    const float4 a = __ldcs(R), x = __ldcs(R + 1), b = __ldcs(R + 2), c = __ldcs(R + 3);
    if (replays) {  // a position the replay fills holds an old step's index
      const uint32_t sl = __float_as_uint(a.x);
      if ((A.ord.flags[sl] & FLAG_REPLAY) || A.ord.cnt[sl] + __float_as_uint(a.z) != q) continue;
    }
    float E[3] = {A.f.e[0], A.f.e[1], A.f.e[2]}, B[3] = {A.f.b[0], A.f.b[1], A.f.b[2]};
    if (A.ord.rec_words > 16) {
      const float4 u = __ldcs(R + 4), v = __ldcs(R + 5);
      E[0] = u.x; E[1] = u.y; E[2] = u.z;
      B[0] = u.w; B[1] = v.x; B[2] = v.y;
    }
    const uint64_t pid = (uint64_t)__float_as_uint(b.x) | ((uint64_t)__float_as_uint(b.y) << 32);
    const U4 cid = draw(A.C, pid, step_, __float_as_uint(a.y), STREAM_PHOTON_ID);
    write_child(A.ph, nph + q, x.x, x.y, x.z, b.z, b.w, c.x, x.w, (uint64_t)cid.x | ((uint64_t)cid.y << 32), E, B,
                __float_as_uint(a.w));
  }
}

cudaError_t launch_ordered_writes(qed_ctx *c, const OnePassArgs &a, cudaStream_t st) {
  const int64_t *n0 = a.sp[0].d_n, *n1 = a.nsp > 1 ? a.sp[1].d_n : nullptr;
  OrdScanArgs sc{a.ord, n0, n1, a.ph.d_n, c->sub_meta, a.ph.cap, c->d_counters};
  k_ord_scan<<<1, ORD_SCAN_THREADS, 0, st>>>(sc);
  // no more CTAs than the capacities need
  const int64_t slots = (a.sp[0].cap + TILE - 1) / TILE + (a.nsp > 1 ? (a.sp[1].cap + TILE - 1) / TILE : 0);
  const int64_t chunks = (slots * TILE + CLS_CHUNK_FLAGS - 1) / CLS_CHUNK_FLAGS;
  const int64_t most = (int64_t)c->num_sms * 8;
  k_ord_offsets<<<(unsigned)(chunks < 1 ? 1 : chunks < most ? chunks : most), TILE, 0, st>>>(a.ord, n0, n1);
  const int64_t need = (a.ph.cap + TILE - 1) / TILE;
  const unsigned grid = (unsigned)(need < 1 ? 1 : need < most ? need : most);
  k_ord_index<<<grid, TILE, 0, st>>>(a.ord, c->sub_meta, a.ph.cap);
  OrdWriteArgs w{a.ph, a.f, a.C, a.ord, c->sub_meta, a.step, a.d_step};
  k_ord_write<<<grid, TILE, 0, st>>>(w);
  c->launches += 4;
  return cudaGetLastError();
}

// ---- the learned sampler's dense pass ----------------------------------
// The deferred emissions of one-sub-step leptons (records written by the
// single-pass kernel): every warp takes 32 records at a time, evaluates the
// network for all of them at once (tensor cores, weights in shared memory),
// and finishes each emission with the heavy phase's expressions: gamma, the
// direction and chi of the pushed lepton, xi (Eq. 7 through ln delta), the
// recoiled momentum, the spectrum bin and the photon.
struct NetArgs {
  Sp<float> sp[2];
  Sp<float> ph;
  Fld<float> f;
  Consts C;
  Out o;
  int64_t step;
  const int64_t *d_step;
  const uint32_t *mlp_frag;
  const float *mlp_fw;
  const float4 *net_rec;
  unsigned long long *net_n;  // [0] records written, [1] CTAs of this pass done
  int64_t net_cap;            // float4 units of net_rec
};
constexpr int NET_THREADS = 256;

template <int FM>
__global__ void __launch_bounds__(NET_THREADS) k_net_emit(NetArgs A) {
  constexpr int RS = net_stride<FM>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ BlockTally bt;
  __shared__ long long s_n;
  uint32_t *s_frag = reinterpret_cast<uint32_t *>(smem_raw);
  float *s_fw = reinterpret_cast<float *>(s_frag + MLP_FRAG_WORDS);
  for (int k = threadIdx.x; k < MLP_FRAG_WORDS; k += blockDim.x) s_frag[k] = A.mlp_frag[k];
  for (int k = threadIdx.x; k < MLP_SMEM_FLOATS; k += blockDim.x) s_fw[k] = A.mlp_fw[k];
  block_tally_init(&bt);
  if (threadIdx.x == 0) {
    const unsigned long long n = *(volatile unsigned long long *)A.net_n;
    const unsigned long long cap = (unsigned long long)(A.net_cap / RS);
    s_n = (long long)(n < cap ? n : cap);
  }
  __syncthreads();
  const int64_t n = s_n;
  const int64_t step_ = A.d_step ? *A.d_step : A.step;
  const float inv_aS = A.C.f_inv_aS;
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  Tally tl;
  tl.clear();
  for (int64_t base = w * 32; base < n; base += nw * 32) {  // warp-uniform
    const int64_t r = base + lane;
    const bool ok = r < n;
    int si = 0;
    int64_t i = 0;
    float kap = 0.f, g = 1.f, nx = 0.f, ny = 0.f, nz = 0.f, chi = 1.f;
    float E[3] = {0.f, 0.f, 0.f}, B[3] = {0.f, 0.f, 0.f};
    if (ok) {
      const float4 *R = A.net_rec + RS * r;
      const float4 R0 = R[0];
      const uint32_t hi = __float_as_uint(R0.y);
      i = (int64_t)(((uint64_t)(hi & 0x7FFFFFFFu) << 32) | __float_as_uint(R0.x));
      si = (int)(hi >> 31);
      kap = R0.z;
      const Sp<float> &S = A.sp[si];
      if (FM == FM_GRID) {
        const float4 R1 = R[1], R2 = R[2];
        E[0] = R0.w; E[1] = R1.x; E[2] = R1.y;
        B[0] = R1.z; B[1] = R1.w; B[2] = R2.x;
      } else {
        get_fields<float, FM>(S, A.f, i, 0.f, 0.f, 0.f, E, B);
      }
      const float px = S.px[i], py = S.py[i], pz = S.pz[i];
      gamma_dir(px, py, pz, g, nx, ny, nz);
      chi = chi_lepton(px, py, pz, g, E[0], E[1], E[2], B[0], B[1], B[2], inv_aS);
    }
    const float lchi = ok ? logf(chi) : 0.f;
    const float zz = mlp_infer_warp(s_frag, s_fw, (lchi - MLP_LC) / MLP_LS, (kap - MLP_KC) / MLP_KS);
    float eph = 0.f, g2 = g;
    if (ok) {
      const float Y = zz + mlp_baseline(kap);
      const XiOut<float> xo = xi_from_lndelta(chi, Y);
      g2 = g * xo.omxi;
      eph = g * xo.xi;
      if (g2 < 1.f) { g2 = 1.f; eph = g - 1.f; }
      const int b = spec_bin(A.C, eph);
      const unsigned same = __match_any_sync(__activemask(), b);
      if (b >= 0 && lane == __ffs(same) - 1) atomicAdd(&bt.hist[b], (unsigned long long)__popc(same));
    }
    const unsigned em = __ballot_sync(0xFFFFFFFFu, ok);
    const int leader = __ffs(em) - 1;
    unsigned long long pbase = 0;
    if (lane == leader)
      pbase = atomicAdd(reinterpret_cast<unsigned long long *>(A.ph.d_n), (unsigned long long)__popc(em));
    pbase = __shfl_sync(0xFFFFFFFFu, pbase, leader < 0 ? 0 : leader);
    if (ok) {
      const Sp<float> &S = A.sp[si];
      const int64_t pos = (int64_t)pbase + __popc(em & lt_mask);
      if (pos >= A.ph.cap) {
        tl.dropped += 1;
        tl.status |= QED_STATUS_CAPACITY;
      } else {
        const U4 cid = draw(A.C, S.id[i], step_, 0, STREAM_PHOTON_ID);
        write_child(A.ph, pos, S.x[i], S.y[i], S.z[i], eph * nx, eph * ny, eph * nz, S.w[i],
                    (uint64_t)cid.x | ((uint64_t)cid.y << 32), E, B, S.tag ? S.tag[i] : 0u);
      }
      const float pm = sqrtf((g2 - 1.f) * (g2 + 1.f));
      S.px[i] = pm * nx; S.py[i] = pm * ny; S.pz[i] = pm * nz;
      tl.events += 1;
    }
  }
  tally_flush(&bt, tl);
  __syncthreads();
  block_tally_commit(&bt, A.o.cnt, 0);
  if (threadIdx.x == 0) {
    // the last CTA clamps the photon count to the capacity and clears the
    // record count for the next step
    __threadfence();
    const unsigned long long prev = atomicAdd(A.net_n + 1, 1ull);
    if (prev == gridDim.x - 1) {
      __threadfence();
      int64_t *dn = A.ph.d_n;
      if (*(volatile int64_t *)dn > A.ph.cap) *dn = A.ph.cap;
      A.net_n[0] = 0ull;
      A.net_n[1] = 0ull;
      __threadfence();
    }
  }
}

template <int FM>
cudaError_t launch_net_emit_t(qed_ctx *c, const NetArgs &n, cudaStream_t st) {
  const size_t sm = MLP_SMEM_BYTES;
  auto kern = k_net_emit<FM>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NET_THREADS, sm);
  if (e != cudaSuccess) return e;
  per_sm = persistent_blocks_per_sm(c, per_sm, QED_TUNE_COMPACT);
  kern<<<c->num_sms * per_sm, NET_THREADS, sm, st>>>(n);
  c->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_net_emit(qed_ctx *c, const OnePassArgs &a, int fm, cudaStream_t st) {
  NetArgs n{};
  n.sp[0] = a.sp[0];
  n.sp[1] = a.nsp > 1 ? a.sp[1] : a.sp[0];
  n.ph = a.ph;
  n.f = a.f;
  n.C = a.C;
  n.o = a.o;
  n.step = a.step;
  n.d_step = a.d_step;
  n.mlp_frag = a.mlp_frag;
  n.mlp_fw = a.mlp_fw;
  n.net_rec = a.net_rec;
  n.net_n = a.net_n;
  n.net_cap = a.net_cap;
  if (fm == QED_FIELDS_UNIFORM) return launch_net_emit_t<FM_UNIFORM>(c, n, st);
  if (fm == QED_FIELDS_PER_PARTICLE) return launch_net_emit_t<FM_PER_PARTICLE>(c, n, st);
  return launch_net_emit_t<FM_GRID>(c, n, st);
}

template <int FM> bool slices_aligned(const OnePassArgs &a) {
  uintptr_t all = 0;
  for (int k = 0; k < a.nsp; ++k) {
    const Sp<float> &S = a.sp[k];
    const void *src[13] = {S.id, S.x, S.y, S.z, S.px, S.py, S.pz, S.ex, S.ey, S.ez, S.bx, S.by, S.bz};
    for (int c = 0; c <= stream_words<FM>(); ++c) all |= reinterpret_cast<uintptr_t>(src[c]);
  }
  return (all & 15) == 0;
}

template <int FM, int MODE, bool MLP, bool ORD>
cudaError_t launch_onepass_t(qed_ctx *c, OnePassArgs a, cudaStream_t st) {
  a.aligned16 = slices_aligned<FM>(a);
  const size_t sm = OP_WARPS * warp_smem<FM, ORD>();
  auto kern = k_lepton_onepass<FM, MODE, MLP, ORD>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  kern<<<c->num_sms, OP_THREADS, sm, st>>>(a);
  c->launches += 1;
  return cudaGetLastError();
}

template <int MODE, bool MLP, bool ORD>
cudaError_t launch_onepass_m(qed_ctx *c, const OnePassArgs &a, int fm, cudaStream_t st) {
  if (fm == QED_FIELDS_UNIFORM) return launch_onepass_t<FM_UNIFORM, MODE, MLP, ORD>(c, a, st);
  if (fm == QED_FIELDS_PER_PARTICLE) return launch_onepass_t<FM_PER_PARTICLE, MODE, MLP, ORD>(c, a, st);
  return launch_onepass_t<FM_GRID, MODE, MLP, ORD>(c, a, st);
}

}  // namespace

// The lepton step of an FP32 context under Method I (electrons s0 and, if
// given, positrons s1; photons appended to ph).  mode: 1 emission only
// (qed_emit), 2 push and emission (qed_step_fused).  ordered: photons in the
// ordered path's order (the table sampler's; the caller launches the replay of
// the leptons whose records found no room).
cudaError_t launch_lepton_onepass(qed_ctx *c, const qed_species *s0, const qed_species *s1,
                                  const qed_species *ph, const qed_fields *f, int64_t step,
                                  int mode, bool ordered, cudaStream_t st) {
  OnePassArgs a{};
  a.sp[0] = to_sp<float>(s0);
  a.nsp = s1 ? 2 : 1;
  if (s1) a.sp[1] = to_sp<float>(s1);
  a.ph = to_sp<float>(ph);
  a.f = to_fld<float>(f);
  a.C = consts_of(c);
  a.T = tables_of<float>(c);
  a.o = out_of(c);
  a.step = step;
  a.d_step = c->use_dstep ? c->d_step : nullptr;
  a.w_up_row = c->w_up_row;
  a.chi_tab_lo = (float)exp(c->gl.lo);
  a.chi_tab_hi = (float)exp(c->gl.hi);
  a.delta_tab_lo = (float)exp(c->gy.lo);
  a.mlp_frag = c->mlp_frag;
  a.mlp_fw = c->mlp_fw;
  a.net_rec = c->net_rec;
  a.net_n = c->net_n;
  a.net_cap = c->net_cap;
  const bool mlp = c->cfg.sampler == QED_SAMPLER_MLP && c->mlp_ready && c->net_rec;
  cudaError_t e = cudaSuccess;
  if (ordered) {
    a.ord.flags = c->heavy_flags;
    a.ord.cnt = c->sub_cnt;
    a.ord.sum = c->cls_chunk_off;
    a.ord.rec = static_cast<float *>(c->stage);
    a.ord.rec_words = f->mode != QED_FIELDS_UNIFORM && ph->ex ? 24 : 16;
    const int64_t cap = 16 * c->stage_cap / a.ord.rec_words;  // (a staging record is 16 floats)
    a.ord.rec_cap = (uint32_t)(cap < 0x7fffffff ? cap : 0x7fffffff);
    a.ord.idx = reinterpret_cast<uint32_t *>(c->heavy_list);
    a.ord.n = c->ord_n;
    a.ord.replay = c->stage_idx;
    a.ord.replay_cnt = c->rec_k;
    // the chunks of the slots that the capacities allow
    const int64_t tiles = (s0->capacity + TILE - 1) / TILE + (s1 ? (s1->capacity + TILE - 1) / TILE : 0);
    const int64_t chunks = (tiles * TILE + CLS_CHUNK_FLAGS - 1) / CLS_CHUNK_FLAGS;
    e = cudaMemsetAsync(a.ord.sum, 0, sizeof(uint32_t) * NCLS * (size_t)chunks, st);
    if (e == cudaSuccess)
      e = mode == MODE_EMIT ? launch_onepass_m<MODE_EMIT, false, true>(c, a, f->mode, st)
                            : launch_onepass_m<MODE_FUSED, false, true>(c, a, f->mode, st);
    if (e == cudaSuccess) e = prof_mark(c, 1, st);
    if (e == cudaSuccess) e = launch_ordered_writes(c, a, st);
    return e;
  }
  if (mode == MODE_EMIT)
    e = mlp ? launch_onepass_m<MODE_EMIT, true, false>(c, a, f->mode, st)
            : launch_onepass_m<MODE_EMIT, false, false>(c, a, f->mode, st);
  else
    e = mlp ? launch_onepass_m<MODE_FUSED, true, false>(c, a, f->mode, st)
            : launch_onepass_m<MODE_FUSED, false, false>(c, a, f->mode, st);
  if (e == cudaSuccess) e = prof_mark(c, 1, st);
  if (e == cudaSuccess && mlp) e = launch_net_emit(c, a, f->mode, st);
  return e;
}

}  // namespace qed
