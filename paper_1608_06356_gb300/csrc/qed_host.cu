// qed_host.cu -- the lepton stage of the QED step for leptons held in host
// memory: the ensemble is streamed through the GPU in chunks, with the copies
// of one chunk overlapping the step of another.
//
// Three device staging buffers of `chunk` leptons rotate through three
// streams: chunk k is copied in on the input stream (once its buffer's
// previous chunk has been copied out), stepped on the caller's stream -- the
// same launches as qed_step_fused's lepton stage, appending photons to the
// device photon species -- and its positions and momenta copied back on the
// output stream, together with the photons the chunk appended for the host
// mirror of the photon species.  Both ways a copy kernel works through
// host-mapped pointers; the photons' range is read on the device, so that
// every chunk is queued at once and the host waits only at the end.  Memory the
// device cannot map goes by copies per array, the photons' after the host has
// read their range.  Particle ids key the random
// streams, so chunking changes no result, only the order of the photons
// (chunks in order; within a chunk as the lepton step appends them).
#include <cstdio>
#include <cstring>

#include <cuda.h>

#include "qed_internal.h"

namespace qed {
template <class Real>
cudaError_t launch_lepton(qed_ctx *, const qed_species *, const qed_species *, const qed_species *,
                          const qed_fields *, int64_t, int, cudaStream_t);

namespace {

constexpr int MODE_FUSED_ = 2;  // gather, push and emission (the lepton stage of qed_step_fused)

int cuda_fail(cudaError_t e, const char *what) {
  if (e == cudaSuccess) return QED_OK;
  fprintf(stderr, "libqed: %s: %s\n", what, cudaGetErrorString(e));
  return QED_ERR_CUDA;
}

__global__ void k_set_count(int64_t *d_n, int64_t v) { *d_n = v; }
__global__ void k_mark_count(int64_t *dst, const int64_t *src) { *dst = *src; }

// One chunk's arrays between host memory and the GPU, copied by the SMs through
// host-mapped pointers: arrays [0, nl) over n elements, and arrays [nl, na)
// over the photons a chunk appended, [*lo, *hi) clamped to the capacity -- a
// range read on the device, so no host round trip is needed between chunks.
//
// The host link bounds the host step.  A copy engine takes one array at a time
// and idles between them: 120 copies of 2 MB ran at 173 GB/s in, and at 146
// with the copies out beside them (58); a launch per chunk each way gives 211
// alone, 197 beside 79.  4M leptons in 8 chunks: 2012 -> 1660 us, 1195 of them
// the link's for what comes in; 64M in 16, where a copy is 16 MB: 23.85 -> 23.2 ms.
// The copies must run beside the lepton kernel, which leaves 4096 registers of
// an SM: a CTA is 128 threads of at most 32 registers (units of 8 KB, round
// robin over the arrays, 64 bytes in flight per thread), and it asks for the
// shared memory carve-out the lepton kernel needs -- an SM changes its carve-out
// only when it is empty, so with the default the lepton kernel waited for the
// copies to end (1860 us).  One CTA per SM in: with half as many, 1700.  Three
// in eight of the SMs out, so that what goes out takes its share of the link over
// the whole of the next chunk: a quarter 1580 us for the 4M but 25.1 ms for the
// 64M, half of them 24.4 ms.
constexpr int MAX_LANES = 17;     // of a lepton species
constexpr int MAX_PARRAYS = 16;   // of a photon species
constexpr int MAX_COPY = MAX_LANES + MAX_PARRAYS;
constexpr int COPY_THREADS = 128, COPY_UNIT = 4 * COPY_THREADS;  // 16-byte words per unit
struct CopyArgs {
  const char *src[MAX_COPY];
  char *dst[MAX_COPY];
  int esz[MAX_COPY];
  int wide[MAX_COPY];  // 16: both bases 16-byte aligned; 4: 4-byte aligned; else bytes
  int skip[MAX_LANES];  // (leptons) bytes from the bases to the chunk's first element, below 16
  int nl, na;
  int64_t n;
  const int64_t *lo, *hi;
  int64_t cap;
  int64_t *set_n;  // where n is left as the chunk's count, or null
};

// Array between offsets b0 and b1 of its bytes: bytes up to a 16-byte boundary,
// units of 16-byte words, and the rest (by words or bytes if the bases are not so
// aligned).  base = units handed out so far.
__device__ __forceinline__ void copy_array(const char *src, char *dst, int esz, int wide, int64_t b0,
                                           int64_t b1, int64_t &base) {
  const int64_t t0 = (int64_t)blockIdx.x * COPY_THREADS + threadIdx.x;
  const int64_t nt = (int64_t)gridDim.x * COPY_THREADS;
  if (b1 <= b0) return;
  const int64_t m0 = (b0 + 15) & ~(int64_t)15, m1 = b1 & ~(int64_t)15;
  if (m0 >= m1 || wide < 16) {
    if (esz % 4 || wide < 4) {
      for (int64_t q = b0 + t0; q < b1; q += nt) dst[q] = src[q];
    } else {
      const uint32_t *s4 = reinterpret_cast<const uint32_t *>(src);
      uint32_t *d4 = reinterpret_cast<uint32_t *>(dst);
      for (int64_t q = b0 / 4 + t0; q < b1 / 4; q += nt) d4[q] = s4[q];
    }
    return;
  }
  if (t0 < 15) {  // at most 15 bytes on either side
    if (b0 + t0 < m0) dst[b0 + t0] = src[b0 + t0];
    if (m1 + t0 < b1) dst[m1 + t0] = src[m1 + t0];
  }
  const uint4 *s = reinterpret_cast<const uint4 *>(src + m0);
  uint4 *d = reinterpret_cast<uint4 *>(dst + m0);
  const int64_t nw = (m1 - m0) / 16, nu = (nw + COPY_UNIT - 1) / COPY_UNIT;
  const int grid = (int)gridDim.x, r = (int)(base % grid);
  for (int64_t u = (int)blockIdx.x >= r ? blockIdx.x - r : blockIdx.x - r + grid; u < nu; u += grid) {
    const int64_t w = u * COPY_UNIT + threadIdx.x;
    uint4 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (w + k * COPY_THREADS < nw) v[k] = s[w + k * COPY_THREADS];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (w + k * COPY_THREADS < nw) d[w + k * COPY_THREADS] = v[k];
  }
  base += nu;
}

__global__ void __launch_bounds__(COPY_THREADS, 16) k_copy_chunk(const __grid_constant__ CopyArgs A) {
  if (A.set_n && blockIdx.x == 0 && threadIdx.x == 0) *A.set_n = A.n;
  int64_t base = 0;
  for (int a = 0; a < A.nl; ++a)
    copy_array(A.src[a], A.dst[a], A.esz[a], A.wide[a], A.skip[a], A.skip[a] + A.n * A.esz[a], base);
  if (A.na == A.nl) return;
  int64_t lo = *A.lo, hi = *A.hi;
  lo = lo < A.cap ? lo : A.cap;
  hi = hi < A.cap ? hi : A.cap;
  for (int a = A.nl; a < A.na; ++a)
    copy_array(A.src[a], A.dst[a], A.esz[a], A.wide[a], lo * A.esz[a], hi * A.esz[a], base);
}

int width_of(const void *a, const void *b) {
  const uintptr_t al = reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b);
  return al % 16 == 0 ? 16 : al % 4 == 0 ? 4 : 1;
}

// The device pointer of `bytes` bytes of host memory that the device can map
// (page-locked memory allocated by the CUDA runtime is), or null: the whole
// range must lie in one allocation or registration.
char *map_host(void *h, size_t bytes) {
  static const auto query = [] {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess || q != cudaDriverEntryPointSuccess)
      fn = nullptr;
    return reinterpret_cast<CUresult (*)(unsigned int, CUpointer_attribute *, void **, CUdeviceptr)>(fn);
  }();
  CUpointer_attribute what[3] = {CU_POINTER_ATTRIBUTE_DEVICE_POINTER, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                 CU_POINTER_ATTRIBUTE_RANGE_SIZE};
  CUdeviceptr d = 0, start = 0;
  size_t size = 0;
  void *out[3] = {&d, &start, &size};
  // (what is not known of a pointer reads as zero)
  if (!query || query(3, what, out, reinterpret_cast<CUdeviceptr>(h)) != CUDA_SUCCESS || !d) return nullptr;
  if (d < start || d - start > size || size - (d - start) < bytes) return nullptr;
  return reinterpret_cast<char *>(d);
}

// One array of the lepton species as the host step moves it: host pointer,
// bytes per element, device staging offset, and whether it is copied back.
struct Lane {
  char *host;
  size_t esz;
  size_t off;
  bool back;
};

constexpr int NBUF = 3;

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// The arrays of a lepton species, in staging order; *per_buf = staging bytes
// of one buffer for `chunk` leptons.
int lanes_of(const qed_species *s, size_t real, int64_t chunk, Lane out[MAX_LANES], size_t *per_buf) {
  int n = 0;
  size_t off = 0;
  auto add = [&](void *p, size_t esz, bool back) {
    out[n++] = Lane{static_cast<char *>(p), esz, off, back};
    off += align256(esz * (size_t)chunk + 16);
  };
  void *state[6] = {s->x, s->y, s->z, s->px, s->py, s->pz};
  for (void *p : state) add(p, real, true);
  add(s->w, real, false);
  add(s->id, sizeof(uint64_t), false);
  void *fld[6] = {s->ex, s->ey, s->ez, s->bx, s->by, s->bz};
  if (s->ex)
    for (void *p : fld) add(p, real, false);
  if (s->od_p) {
    add(s->od_p, real, true);
    add(s->od_r, real, true);
  }
  if (s->tag) add(s->tag, sizeof(uint32_t), false);
  *per_buf = off;
  return n;
}

// Bytes that element `off` of a host array lies past a 16-byte boundary of it; a
// chunk copied by the SMs lies as far past one in its staging buffer, so that
// the words of both sides agree whatever the chunk's size.  (The lepton kernel
// then takes its words one by one: 4M leptons in chunks of 2^19 1675 us, of
// 2^19 + 1 1932; 2343 by copies per array.)
int past16(const Lane &L, int64_t off) { return (int)((size_t)off * L.esz & 15); }

// The device species of staging buffer b, of a chunk from element `off` on.
qed_species staging_species(qed_ctx *c, const qed_species *h, const Lane *L, int64_t off, int b,
                            int64_t chunk) {
  char *base = static_cast<char *>(c->hs_mem) + (size_t)b * c->hs_per_buf;
  auto at = [&](int k) { return base + L[k].off + past16(L[k], off); };
  qed_species s{};
  void **dst[6] = {&s.x, &s.y, &s.z, &s.px, &s.py, &s.pz};
  int k = 0;
  for (int i = 0; i < 6; ++i) *dst[i] = at(k++);
  s.w = at(k++);
  s.id = reinterpret_cast<uint64_t *>(at(k++));
  if (h->ex) {
    void **fd[6] = {&s.ex, &s.ey, &s.ez, &s.bx, &s.by, &s.bz};
    for (int i = 0; i < 6; ++i) *fd[i] = at(k++);
  }
  if (h->od_p) {
    s.od_p = at(k++);
    s.od_r = at(k++);
  }
  if (h->tag) s.tag = reinterpret_cast<uint32_t *>(at(k++));
  s.d_n = c->hs_dn + b;
  s.capacity = chunk;
  s.q = h->q;
  return s;
}

// The arrays of a photon species and of its host mirror (the mirror must have
// every array the device species has).
int photon_arrays(const qed_species *g, const qed_species *gh, size_t real, void *dev[16],
                  void *host[16], size_t esz[16]) {
  int n = 0;
  auto add = [&](void *d, void *h, size_t e) {
    if (!d) return true;
    if (!h) return false;
    dev[n] = d; host[n] = h; esz[n] = e; ++n;
    return true;
  };
  bool ok = add(g->x, gh->x, real) && add(g->y, gh->y, real) && add(g->z, gh->z, real) &&
            add(g->px, gh->px, real) && add(g->py, gh->py, real) && add(g->pz, gh->pz, real) &&
            add(g->w, gh->w, real) && add(g->id, gh->id, sizeof(uint64_t)) &&
            add(g->alive, gh->alive, 1) && add(g->ex, gh->ex, real) && add(g->ey, gh->ey, real) &&
            add(g->ez, gh->ez, real) && add(g->bx, gh->bx, real) && add(g->by, gh->by, real) &&
            add(g->bz, gh->bz, real) && add(g->tag, gh->tag, sizeof(uint32_t));
  return ok ? n : -1;
}

int ensure_host_step(qed_ctx *c, size_t per_buf) {
  if (!c->hs_in) {
    if (cudaStreamCreateWithFlags(&c->hs_in, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&c->hs_out, cudaStreamNonBlocking) != cudaSuccess)
      return QED_ERR_CUDA;
    for (int i = 0; i < 3 * NBUF; ++i)
      if (cudaEventCreateWithFlags(&c->hs_ev[i], cudaEventDisableTiming) != cudaSuccess)
        return QED_ERR_CUDA;
    if (cudaMalloc(&c->hs_dn, (2 * NBUF + 1) * sizeof(int64_t)) != cudaSuccess) return QED_ERR_NOMEM;
    if (cudaHostAlloc(reinterpret_cast<void **>(&c->hs_cnt), 2 * NBUF * sizeof(int64_t),
                      cudaHostAllocDefault) != cudaSuccess)
      return QED_ERR_NOMEM;
  }
  if (per_buf > c->hs_per_buf) {
    if (c->hs_mem) {
      cudaFree(c->hs_mem);
      c->hs_mem = nullptr;
      c->hs_per_buf = 0;
    }
    if (cudaMalloc(&c->hs_mem, NBUF * per_buf) != cudaSuccess) return QED_ERR_NOMEM;
    c->hs_per_buf = per_buf;
  }
  return QED_OK;
}

}  // namespace

void free_host_step(qed_ctx *c) {
  if (c->hs_mem) cudaFree(c->hs_mem);
  if (c->hs_dn) cudaFree(c->hs_dn);
  if (c->hs_cnt) cudaFreeHost(c->hs_cnt);
  for (int i = 0; i < 3 * NBUF; ++i)
    if (c->hs_ev[i]) cudaEventDestroy(c->hs_ev[i]);
  if (c->hs_in) cudaStreamDestroy(c->hs_in);
  if (c->hs_out) cudaStreamDestroy(c->hs_out);
}

int lepton_step_host(qed_ctx *c, const qed_species *lh, const qed_species *g,
                     const qed_species *gh, const qed_fields *f, int64_t step, int64_t chunk,
                     cudaStream_t st) {
  const bool f64 = c->cfg.precision == QED_FP64;
  const size_t real = f64 ? sizeof(double) : sizeof(float);
  const int64_t n = *lh->d_n;
  if (n < 0 || n > lh->capacity) return QED_ERR_ARG;
  Lane L[MAX_LANES];
  size_t per_buf = 0;
  const int nl = lanes_of(lh, real, chunk, L, &per_buf);
  void *pdev[16], *phost[16];
  size_t pesz[16];
  const int np = gh ? photon_arrays(g, gh, real, pdev, phost, pesz) : 0;
  if (np < 0) return QED_ERR_ARG;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone)
    return QED_ERR_UNSUPPORTED;
  int rc = ensure_host_step(c, per_buf);
  if (rc != QED_OK) return rc;
  // The arrays are copied by k_copy_chunk where the device can map them all:
  // the leptons if they are 16-byte aligned too, else by a copy per array; the
  // photons else by copies whose ranges the host reads after each chunk.
  char *lmap[MAX_LANES];
  bool lmapped = true;
  for (int a = 0; a < nl && lmapped; ++a) {
    lmap[a] = map_host(L[a].host, (size_t)n * L[a].esz);
    lmapped = lmap[a] && width_of(lmap[a], L[a].host) == 16;
  }
  CopyArgs pc{};
  bool mapped = gh != nullptr && np > 0;
  for (int a = 0; a < np && mapped; ++a) {
    char *dp = map_host(phost[a], (size_t)g->capacity * pesz[a]);
    mapped = dp != nullptr;
    pc.src[a] = static_cast<const char *>(pdev[a]);
    pc.dst[a] = dp;
    pc.esz[a] = (int)pesz[a];
    pc.wide[a] = width_of(pdev[a], dp);
  }
  pc.na = mapped ? np : 0;
  pc.cap = g->capacity;
  const int in_blocks = c->num_sms, out_blocks = lmapped ? (c->num_sms * 3 + 7) / 8 : 4 * c->num_sms;
  constexpr int R = NBUF + 1;  // device ring of photon counts after each chunk
  int64_t *ring = c->hs_dn + NBUF;
  cudaEvent_t *in_done = c->hs_ev, *comp_done = c->hs_ev + NBUF, *out_done = c->hs_ev + 2 * NBUF;
  int64_t *cnt = c->hs_cnt;  // [0, NBUF): photon count after chunk k (slot k % NBUF); [NBUF]: at start
  cudaError_t e = cudaFuncSetAttribute(k_copy_chunk, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return cuda_fail(e, "qed_lepton_step_host");
  int64_t m_done = 0;  // (host-read ranges) photons already on the host mirror
  if (mapped) {
    k_mark_count<<<1, 1, 0, st>>>(ring, g->d_n);
    c->launches += 1;
    e = cudaGetLastError();
  } else {
    e = cudaMemcpyAsync(cnt + NBUF, g->d_n, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    m_done = cnt[NBUF];
  }
  if (e != cudaSuccess) return cuda_fail(e, "qed_lepton_step_host");
  const int64_t gcap = g->capacity;
  auto copy_photons = [&](int64_t upto) -> cudaError_t {
    upto = upto < gcap ? upto : gcap;
    if (!gh || upto <= m_done) return cudaSuccess;
    for (int a = 0; a < np; ++a) {
      const size_t o = (size_t)m_done * pesz[a], b = (size_t)(upto - m_done) * pesz[a];
      cudaError_t r = cudaMemcpyAsync(static_cast<char *>(phost[a]) + o,
                                      static_cast<char *>(pdev[a]) + o, b, cudaMemcpyDeviceToHost,
                                      c->hs_out);
      if (r != cudaSuccess) return r;
    }
    m_done = upto;
    return cudaSuccess;
  };
  const int64_t K = (n + chunk - 1) / chunk;
  for (int64_t k = 0; k < K && e == cudaSuccess; ++k) {
    const int b = (int)(k % NBUF);
    const int64_t off = k * chunk, nk = n - off < chunk ? n - off : chunk;
    qed_species sb = staging_species(c, lh, L, lmapped ? off : 0, b, chunk);
    char *base = static_cast<char *>(c->hs_mem) + (size_t)b * c->hs_per_buf;
    // in: once the buffer's previous chunk has been copied out
    if (k >= NBUF) e = cudaStreamWaitEvent(c->hs_in, out_done[b], 0);
    if (e == cudaSuccess && lmapped) {
      CopyArgs in{};
      for (int a = 0; a < nl; ++a) {
        in.skip[a] = past16(L[a], off);
        in.src[a] = lmap[a] + (size_t)off * L[a].esz - in.skip[a];
        in.dst[a] = base + L[a].off;
        in.esz[a] = (int)L[a].esz;
        in.wide[a] = 16;
      }
      in.nl = in.na = nl;
      in.n = nk;
      in.set_n = c->hs_dn + b;
      k_copy_chunk<<<in_blocks, COPY_THREADS, 0, c->hs_in>>>(in);
      c->launches += 1;
      e = cudaGetLastError();
    } else {
      for (int a = 0; a < nl && e == cudaSuccess; ++a)
        e = cudaMemcpyAsync(base + L[a].off, L[a].host + (size_t)off * L[a].esz,
                            (size_t)nk * L[a].esz, cudaMemcpyHostToDevice, c->hs_in);
      if (e == cudaSuccess) {
        k_set_count<<<1, 1, 0, c->hs_in>>>(c->hs_dn + b, nk);
        c->launches += 1;
        e = cudaGetLastError();
      }
    }
    if (e == cudaSuccess) e = cudaEventRecord(in_done[b], c->hs_in);
    // step on the caller's stream, then the photon count after it
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, in_done[b], 0);
    if (e == cudaSuccess)
      e = f64 ? launch_lepton<double>(c, &sb, nullptr, g, f, step, MODE_FUSED_, st)
              : launch_lepton<float>(c, &sb, nullptr, g, f, step, MODE_FUSED_, st);
    if (e == cudaSuccess) {
      if (mapped) {
        k_mark_count<<<1, 1, 0, st>>>(ring + (k + 1) % R, g->d_n);
        c->launches += 1;
        e = cudaGetLastError();
      } else {
        e = cudaMemcpyAsync(cnt + b, g->d_n, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
      }
    }
    if (e == cudaSuccess) e = cudaEventRecord(comp_done[b], st);
    // out: the updated positions and momenta (and event-generator state), and
    // with mapped mirrors the chunk's photons
    if (e == cudaSuccess) e = cudaStreamWaitEvent(c->hs_out, comp_done[b], 0);
    if (!lmapped)
      for (int a = 0; a < nl && e == cudaSuccess; ++a)
        if (L[a].back)
          e = cudaMemcpyAsync(L[a].host + (size_t)off * L[a].esz, base + L[a].off,
                              (size_t)nk * L[a].esz, cudaMemcpyDeviceToHost, c->hs_out);
    if (e == cudaSuccess && (lmapped || mapped)) {
      CopyArgs out{};
      int m = 0;
      auto add = [&](const char *src, char *dst, int esz, int wide) {
        out.src[m] = src; out.dst[m] = dst; out.esz[m] = esz; out.wide[m] = wide; ++m;
      };
      for (int a = 0; a < nl && lmapped; ++a)
        if (L[a].back) {
          out.skip[m] = past16(L[a], off);
          add(base + L[a].off, lmap[a] + (size_t)off * L[a].esz - out.skip[m], (int)L[a].esz, 16);
        }
      out.nl = m;
      for (int a = 0; a < pc.na; ++a) add(pc.src[a], pc.dst[a], pc.esz[a], pc.wide[a]);
      out.na = m;
      out.n = nk;
      // ring slot k % R is rewritten only by chunk k + NBUF, whose input copy
      // waits for this buffer's out_done (recorded after this copy)
      out.lo = ring + k % R;
      out.hi = ring + (k + 1) % R;
      out.cap = pc.cap;
      k_copy_chunk<<<out_blocks, COPY_THREADS, 0, c->hs_out>>>(out);
      c->launches += 1;
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaEventRecord(out_done[b], c->hs_out);
    // (host-read ranges) the previous chunk's photons, now that the next
    // chunks are queued
    if (e == cudaSuccess && !mapped && k >= 1) {
      const int pb = (int)((k - 1) % NBUF);
      e = cudaEventSynchronize(comp_done[pb]);
      if (e == cudaSuccess) e = copy_photons(cnt[pb]);
    }
  }
  if (e == cudaSuccess && !mapped && K >= 1) {
    const int lb = (int)((K - 1) % NBUF);
    e = cudaEventSynchronize(comp_done[lb]);
    if (e == cudaSuccess) e = copy_photons(cnt[lb]);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->hs_out);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->hs_in);
  if (e == cudaSuccess && gh && gh->d_n)
    e = cudaMemcpyAsync(cnt + NBUF, g->d_n, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "qed_lepton_step_host");
  if (gh && gh->d_n) *gh->d_n = cnt[NBUF] < gcap ? cnt[NBUF] : gcap;
  return QED_OK;
}

}  // namespace qed
