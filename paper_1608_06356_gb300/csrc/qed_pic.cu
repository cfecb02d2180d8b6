// qed_pic.cu -- the particle-in-cell loop around the QED step: current
// deposition, the Yee field update and the node grid the particle gather
// reads (qed_pic_deposit, qed_pic_fields, qed_pic_step).
//
// The paper adds its QED module to a PIC code (introduction) whose field
// solver it does not describe; this is the standard explicit scheme.  Fields
// live on Yee's staggered grid in float, [nz][ny][nx] per component (x
// fastest), periodic:
//   ex, jx at (i+1/2, j, k)     bx at (i, j+1/2, k+1/2)
//   ey, jy at (i, j+1/2, k)     by at (i+1/2, j, k+1/2)
//   ez, jz at (i, j, k+1/2)     bz at (i+1/2, j+1/2, k)
// and are advanced by the leapfrog of dB/dt = -curl E, dE/dt = curl B - J in
// the units of the library (J in e n_c c).
//
// Kernels.  The field kernels are stencils bound by HBM bandwidth: a thread
// takes one or four cells along x (coalesced), the y/z neighbours coming from
// planes that L2 still holds.  One step is four passes -- B half-step, E step (which zeroes J behind it), B half-step, node
// grid -- because each needs its neighbours' results of the one before.  The
// deposit adds 8 CIC weights x 3 components per particle at their staggered
// positions: few particles directly, one thread each, by atomics in L2 -- the
// two x-neighbours of each stencil row by one 16-byte vector atomic where they
// share an aligned group of four floats (3 rows in 4), so about 15 atomic
// operations per particle instead of 24 -- and many by tiles of cells that
// are summed on chip.
#include <cmath>
#include <cstdio>

#include "qed_internal.h"

namespace qed {
namespace {

int cuda_fail(cudaError_t e, const char *what) {
  if (e == cudaSuccess) return QED_OK;
  fprintf(stderr, "libqed: %s: %s\n", what, cudaGetErrorString(e));
  return QED_ERR_CUDA;
}

constexpr int FIELD_THREADS = 128;
constexpr int DEPOSIT_THREADS = 256;

struct YeeArgs {
  float *ex, *ey, *ez, *bx, *by, *bz, *jx, *jy, *jz;
  float4 *nodes;
  int nx, ny, nz;
  float idx, idy, idz;  // inverse spacings
  bool nodes32;         // the nodes start on a 32-byte boundary
  uint32_t row0, rows;  // rows (j, k) of this launch
};

YeeArgs yee_args(const qed_yee *y) {
  YeeArgs a;
  a.ex = y->ex; a.ey = y->ey; a.ez = y->ez;
  a.bx = y->bx; a.by = y->by; a.bz = y->bz;
  a.jx = y->jx; a.jy = y->jy; a.jz = y->jz;
  a.nodes = reinterpret_cast<float4 *>(y->nodes);
  a.nx = y->nx; a.ny = y->ny; a.nz = y->nz;
  a.nodes32 = (reinterpret_cast<uintptr_t>(y->nodes) & 31) == 0;
  a.idx = (float)(1.0 / y->dx); a.idy = (float)(1.0 / y->dy); a.idz = (float)(1.0 / y->dz);
  return a;
}

// V consecutive cells along x of one thread, (i .. i + V - 1, j, k), and its
// neighbours: `c` the first cell, `l` and `r` the cells before the first and
// after the last, the rest offsets from a cell to its neighbours along y and z.
// All periodic.  A field kernel is a stream of arrays bound by HBM bandwidth;
// with a cell per thread each load is 4 bytes and too few are in flight, so rows
// of a multiple of four cells (every array starts on a 16-byte boundary) take
// four cells a thread: 256^3 cells, B half-step 133 -> 86 us, E step 179 -> 141
// (89 and 149 at the copy rate).
template <int V> struct Cells {
  int64_t c, l, r, yp, ym, zp, zm;
  __device__ __forceinline__ bool at(const YeeArgs &A) {
    const uint32_t per_row = (uint32_t)A.nx / V;
    const uint32_t t = blockIdx.x * FIELD_THREADS + threadIdx.x;
    uint32_t row = t / per_row;
    if (row >= A.rows) return false;
    const int i = (int)(t - row * per_row) * V;
    row += A.row0;
    const int j = (int)(row % (uint32_t)A.ny), k = (int)(row / (uint32_t)A.ny);
    const int64_t nx = A.nx, plane = (int64_t)A.nx * A.ny, base = (int64_t)row * nx;
    c = base + i;
    l = base + (i == 0 ? A.nx - 1 : i - 1);
    r = base + (i + V == A.nx ? 0 : i + V);
    yp = j + 1 == A.ny ? -(int64_t)j * nx : nx;
    ym = j == 0 ? (int64_t)(A.ny - 1) * nx : -nx;
    zp = k + 1 == A.nz ? -(int64_t)k * plane : plane;
    zm = k == 0 ? (int64_t)(A.nz - 1) * plane : -plane;
    return true;
  }
};

template <int V> struct Vals {
  float v[V];
  __device__ __forceinline__ void load(const float *p) {
    if constexpr (V == 4) {
      const float4 q = *reinterpret_cast<const float4 *>(p);
      v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
      v[0] = *p;
    }
  }
  __device__ __forceinline__ void store(float *p) const {
    if constexpr (V == 4) *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else *p = v[0];
  }
};
template <int V> __device__ __forceinline__ Vals<V> vals(const float *p) {
  Vals<V> r;
  r.load(p);
  return r;
}

// B -= h curl E at the B positions (forward differences of E).
template <int V> __global__ void __launch_bounds__(FIELD_THREADS) k_yee_b_half(YeeArgs A, float h) {
  Cells<V> q;
  if (!q.at(A)) return;
  const Vals<V> ex = vals<V>(A.ex + q.c), ey = vals<V>(A.ey + q.c), ez = vals<V>(A.ez + q.c);
  const Vals<V> exy = vals<V>(A.ex + q.c + q.yp), exz = vals<V>(A.ex + q.c + q.zp);
  const Vals<V> eyz = vals<V>(A.ey + q.c + q.zp), ezy = vals<V>(A.ez + q.c + q.yp);
  Vals<V> bx = vals<V>(A.bx + q.c), by = vals<V>(A.by + q.c), bz = vals<V>(A.bz + q.c);
  const float eyr = A.ey[q.r], ezr = A.ez[q.r];
#pragma unroll
  for (int m = 0; m < V; ++m) {
    const float eyx = m + 1 < V ? ey.v[m + 1 < V ? m + 1 : 0] : eyr, ezx = m + 1 < V ? ez.v[m + 1 < V ? m + 1 : 0] : ezr;
    const float cx = (ezy.v[m] - ez.v[m]) * A.idy - (eyz.v[m] - ey.v[m]) * A.idz;
    const float cy = (exz.v[m] - ex.v[m]) * A.idz - (ezx - ez.v[m]) * A.idx;
    const float cz = (eyx - ey.v[m]) * A.idx - (exy.v[m] - ex.v[m]) * A.idy;
    bx.v[m] -= h * cx;
    by.v[m] -= h * cy;
    bz.v[m] -= h * cz;
  }
  bx.store(A.bx + q.c);
  by.store(A.by + q.c);
  bz.store(A.bz + q.c);
}

// E += dt (curl B - J) at the E positions (backward differences of B); J is
// zeroed for the next deposit.
template <int V> __global__ void __launch_bounds__(FIELD_THREADS) k_yee_e(YeeArgs A, float dt) {
  Cells<V> q;
  if (!q.at(A)) return;
  const Vals<V> bx = vals<V>(A.bx + q.c), by = vals<V>(A.by + q.c), bz = vals<V>(A.bz + q.c);
  const Vals<V> bxy = vals<V>(A.bx + q.c + q.ym), bxz = vals<V>(A.bx + q.c + q.zm);
  const Vals<V> byz = vals<V>(A.by + q.c + q.zm), bzy = vals<V>(A.bz + q.c + q.ym);
  const Vals<V> jx = vals<V>(A.jx + q.c), jy = vals<V>(A.jy + q.c), jz = vals<V>(A.jz + q.c);
  Vals<V> ex = vals<V>(A.ex + q.c), ey = vals<V>(A.ey + q.c), ez = vals<V>(A.ez + q.c), zero;
  const float byl = A.by[q.l], bzl = A.bz[q.l];
#pragma unroll
  for (int m = 0; m < V; ++m) {
    const float byx = m > 0 ? by.v[m > 0 ? m - 1 : 0] : byl, bzx = m > 0 ? bz.v[m > 0 ? m - 1 : 0] : bzl;
    const float cx = (bz.v[m] - bzy.v[m]) * A.idy - (by.v[m] - byz.v[m]) * A.idz;
    const float cy = (bx.v[m] - bxz.v[m]) * A.idz - (bz.v[m] - bzx) * A.idx;
    const float cz = (by.v[m] - byx) * A.idx - (bx.v[m] - bxy.v[m]) * A.idy;
    ex.v[m] += dt * (cx - jx.v[m]);
    ey.v[m] += dt * (cy - jy.v[m]);
    ez.v[m] += dt * (cz - jz.v[m]);
    zero.v[m] = 0.f;
  }
  ex.store(A.ex + q.c);
  ey.store(A.ey + q.c);
  ez.store(A.ez + q.c);
  zero.store(A.jx + q.c);
  zero.store(A.jy + q.c);
  zero.store(A.jz + q.c);
}

// Node (i, j, k): E components the mean of their two staggered neighbours
// along their own axis, B components the mean of their four neighbours in
// the plane normal to them.
// A cell per thread: its node is a 32-byte sector, written as one where the
// nodes are so aligned: 256^3 cells, 204 -> 171 us (139 at the copy rate; in
// halves 195, and with four cells a thread, whose halves lie 128 bytes apart,
// 203).
__global__ void __launch_bounds__(FIELD_THREADS) k_yee_nodes(YeeArgs A) {
  Cells<1> q;
  if (!q.at(A)) return;
  float4 a, b;
  a.x = 0.5f * (A.ex[q.c] + A.ex[q.l]);
  a.y = 0.5f * (A.ey[q.c] + A.ey[q.c + q.ym]);
  a.z = 0.5f * (A.ez[q.c] + A.ez[q.c + q.zm]);
  a.w = 0.25f * (A.bx[q.c] + A.bx[q.c + q.ym] + A.bx[q.c + q.zm] + A.bx[q.c + q.ym + q.zm]);
  b.x = 0.25f * (A.by[q.c] + A.by[q.l] + A.by[q.c + q.zm] + A.by[q.l + q.zm]);
  b.y = 0.25f * (A.bz[q.c] + A.bz[q.l] + A.bz[q.c + q.ym] + A.bz[q.l + q.ym]);
  b.z = 0.f;
  b.w = 0.f;
  float4 *const p = A.nodes + 2 * q.c;
  if (A.nodes32) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z),
                 "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
  } else {
    p[0] = a;
    p[1] = b;
  }
}

template <class Real> struct DepArgs {
  const Real *x, *y, *z, *px, *py, *pz, *w;
  const int64_t *d_n, *d_lim;
  int64_t cap;
  float *jx, *jy, *jz;
  int nx, ny, nz;
  Real idx, idy, idz, x0, y0, z0;
  Real scale;   // q weight_unit / (dx dy dz)
  Real half_dt;
  qed_counters *cnt;
};

// The two x-neighbours a0, a1 of one row of the stencil: one 16-byte vector
// atomic (the other two lanes add zero) when both lie in one aligned group of
// four floats inside the array, else a scalar atomic each (a row wrapping
// around the periodic boundary, a pair across a group, or nx = 1, where
// a1 == a0).
__device__ __forceinline__ void add_pair(float *J, int64_t ncell, int64_t a0, int64_t a1, float v0,
                                         float v1) {
  const int64_t g = a0 & ~(int64_t)3;
  const int l = (int)(a0 & 3);
  if (a1 == a0 + 1 && l != 3 && g + 3 < ncell) {
    const float4 v = l == 0 ? make_float4(v0, v1, 0.f, 0.f)
                   : l == 1 ? make_float4(0.f, v0, v1, 0.f)
                            : make_float4(0.f, 0.f, v0, v1);
    atomicAdd(reinterpret_cast<float4 *>(J + g), v);
  } else {
    atomicAdd(J + a0, v0);
    atomicAdd(J + a1, v1);
  }
}

// CIC spread of `amount` at reduced coordinates (fx, fy, fz) (cells from the
// origin of the component's staggered lattice).
template <class Real>
__device__ __forceinline__ void spread(float *J, const DepArgs<Real> &A, Real fx, Real fy, Real fz,
                                       Real amount) {
  const Real ix = floor(fx), iy = floor(fy), iz = floor(fz);
  const Real wx = fx - ix, wy = fy - iy, wz = fz - iz;
  int64_t i0 = (int64_t)ix % A.nx, j0 = (int64_t)iy % A.ny, k0 = (int64_t)iz % A.nz;
  if (i0 < 0) i0 += A.nx;
  if (j0 < 0) j0 += A.ny;
  if (k0 < 0) k0 += A.nz;
  const int64_t i1 = i0 + 1 == A.nx ? 0 : i0 + 1;
  const int64_t j1 = j0 + 1 == A.ny ? 0 : j0 + 1;
  const int64_t k1 = k0 + 1 == A.nz ? 0 : k0 + 1;
  const int64_t nx = A.nx, plane = (int64_t)A.nx * A.ny, ncell = plane * A.nz;
#pragma unroll
  for (int dk = 0; dk < 2; ++dk)
#pragma unroll
    for (int dj = 0; dj < 2; ++dj) {
      const Real wr = amount * (dj ? wy : (Real)1 - wy) * (dk ? wz : (Real)1 - wz);
      const int64_t row = (dk ? k1 : k0) * plane + (dj ? j1 : j0) * nx;
      add_pair(J, ncell, row + i0, row + i1, (float)(wr * ((Real)1 - wx)), (float)(wr * wx));
    }
}

// Velocity times dt-independent parts of one particle's deposit: reduced
// coordinates (cells) of its mid-step position and its velocity.  The
// products are written with explicit fused operations so that every kernel
// that calls this rounds alike.
template <class Real> struct DepPoint { Real f[3], j[3]; };

// 1 / sqrt(x), x >= 1: the fast reciprocal root and one Newton step on its
// residual (the IEEE root and division are a third of the instructions of a
// binning kernel, which issue bounds).  Over all floats, in units of 2^-24, at
// most 1.24 and 0.48 rms off; the IEEE root and division 1.50 and 0.60, the step
// as y (1.5 - x y y / 2), of as many operations, 2.03 and 0.58.  0 where x has
// overflowed, as the division gives.
__device__ __forceinline__ float dep_rsqrt(float x) {
  const float y = rsqrtf(x), r = fmaf(0.5f * y, fmaf(-x * y, y, 1.f), y);
  return x == INFINITY ? 0.f : r;
}
__device__ __forceinline__ double dep_rsqrt(double x) { return 1.0 / sqrt(x); }

template <class Real>
__device__ __forceinline__ bool dep_point(const DepArgs<Real> &A, int64_t p, DepPoint<Real> &d) {
  const Real px = A.px[p], py = A.py[p], pz = A.pz[p];
  const Real ig = dep_rsqrt(fma(pz, pz, fma(py, py, fma(px, px, (Real)1))));
  const Real vx = px * ig, vy = py * ig, vz = pz * ig;
  d.f[0] = (fma(-A.half_dt, vx, A.x[p]) - A.x0) * A.idx;
  d.f[1] = (fma(-A.half_dt, vy, A.y[p]) - A.y0) * A.idy;
  d.f[2] = (fma(-A.half_dt, vz, A.z[p]) - A.z0) * A.idz;
  d.j[0] = vx; d.j[1] = vy; d.j[2] = vz;
  const Real lim = (Real)4.0e15;  // reduced coordinates beyond this are not finite cells
  return fabs(d.f[0]) < lim && fabs(d.f[1]) < lim && fabs(d.f[2]) < lim;  // also false for NaN
}

template <class Real>
__device__ __forceinline__ void dep_direct(const DepArgs<Real> &A, const DepPoint<Real> &d, Real a) {
  // (a v in place: scaled beforehand, FP64 took 16 operations a particle more,
  // 1209 us for 1088 at 180^3 and 2^22)
  spread(A.jx, A, d.f[0] - (Real)0.5, d.f[1], d.f[2], a * d.j[0]);
  spread(A.jy, A, d.f[0], d.f[1] - (Real)0.5, d.f[2], a * d.j[1]);
  spread(A.jz, A, d.f[0], d.f[1], d.f[2] - (Real)0.5, a * d.j[2]);
}

template <class Real> __device__ __forceinline__ int64_t dep_count(const DepArgs<Real> &A) {
  int64_t n = *A.d_n;
  if (A.d_lim && *A.d_lim < n) n = *A.d_lim;
  return n > A.cap ? A.cap : n;
}

// Scratch of the tiled path.  A tile's records are a segment, or one of `ways`
// segments: the particles of a grid with few tiles spread their atomics over
// that many counters.  A counter has a sector of its own: neighbours in one
// sector would share its queue.
constexpr int SECTOR = 8;  // words
struct TileArgs {
  uint32_t *cnt;     // [segment * SECTOR] particles counted (zero between calls)
  uint32_t *cursor;  // [segment * SECTOR] next record
  uint32_t *meta;    // [0] records, [1] parts, [2] whether this call is tiled
  uint4 *part;       // [ntiles + rec_cap / DEP_PART_MIN] parts of tiles: tile, first record, last + 1, batches with heavy cells
  uint32_t ntiles, ways, rec_cap;
  uint32_t most_ctas;  // CTAs of k_dep_tile that fill the chip twice
  uint32_t ntx, nty;
  // particles from min_n on are deposited by tiles if their order is scattered,
  // from min_sorted on in any order, above max_n directly
  int64_t min_n, min_sorted, max_n, cells;
};

// Direct deposit: a particle's 24 contributions as atomics.
template <class Real> __device__ __forceinline__ void deposit_direct(const DepArgs<Real> &A, int64_t n) {
  unsigned bad = 0;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
       p += (int64_t)gridDim.x * blockDim.x) {
    DepPoint<Real> d;
    if (!dep_point(A, p, d)) {
      bad = 1;
      continue;
    }
    dep_direct(A, d, A.scale * A.w[p]);
  }
  if (bad) atomicOr(&A.cnt->status, (unsigned)QED_STATUS_NONFINITE);
}

// (calls too small for the tiled path by their capacity)
template <class Real>
__global__ void __launch_bounds__(DEPOSIT_THREADS) k_pic_deposit(DepArgs<Real> A) {
  deposit_direct(A, dep_count(A));
}

// ---------------------------------------------------------------------------
// Tiled deposit.  The direct deposit is bound by atomics in L2: 15 per
// particle, on lines that a random particle order brings from HBM each time
// once J is larger than L2.  Here the particles are first binned by tile of
// 8 x 8 x 4 cells (count, segment allocation, scatter of 32-byte records -- one
// 256-bit store each, which a scattered order takes at twice the rate of two of
// 128 bits: 434 against 794 us for 16.8M), then a CTA sums a tile's currents on
// chip: one thread per cell, the particles of a batch ordered by cell, 36 sums
// in registers (3 x 2 x 2 positions per component around the cell), added up
// in a shared (8+2) x (8+2) x (4+2) halo tile; only that tile goes to J, by
// atomics that are contiguous along x.  16.8M particles: 256^3 cells in random
// order 5.00 -> 1.34 ms (count 0.14, scatter 0.42, tiles 0.78: bound by the
// scattered stores and by instruction issue in the tiles), 128^3 by cell 1.44
// -> 0.59 ms (0.09, 0.24, 0.26).  FP32 contexts only.
// ---------------------------------------------------------------------------
constexpr int TLX = 8, TLY = 8, TLZ = 4, TL_CELLS = TLX * TLY * TLZ;
constexpr int HLX = TLX + 2, HLY = TLY + 2, HLZ = TLZ + 2, HL_CELLS = HLX * HLY * HLZ;
constexpr int TILE_THREADS = TL_CELLS;  // a thread per cell

struct alignas(32) DepRec {
  float w[3], key, j[3], pad;  // offsets in the cell; cell of the tile (a small integer); a v
};

// A record is written and read by one 32-byte sector.
__device__ __forceinline__ void put_rec(DepRec *p, const DepRec &r) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(p), "f"(r.w[0]), "f"(r.w[1]),
               "f"(r.w[2]), "f"(r.key), "f"(r.j[0]), "f"(r.j[1]), "f"(r.j[2]), "f"(r.pad)
               : "memory");
}
__device__ __forceinline__ DepRec get_rec(const DepRec *p) {
  DepRec r;
  asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
               : "=f"(r.w[0]), "=f"(r.w[1]), "=f"(r.w[2]), "=f"(r.key), "=f"(r.j[0]), "=f"(r.j[1]), "=f"(r.j[2]),
                 "=f"(r.pad)
               : "l"(p));
  return r;
}

// Periodic cell index of an integral reduced coordinate.
__device__ __forceinline__ uint32_t dep_wrap(float f, int n) {
  if (f >= 0.f && f < (float)n) return (uint32_t)f;
  int64_t i = (int64_t)f % n;
  return (uint32_t)(i < 0 ? i + n : i);
}

// Tile of a particle, its cell in the tile and its offsets in the cell.
__device__ __forceinline__ uint32_t dep_tile(const DepArgs<float> &A, const TileArgs &T,
                                             const DepPoint<float> &d, float w[3], uint32_t &cell) {
  const float ix = floor(d.f[0]), iy = floor(d.f[1]), iz = floor(d.f[2]);
  w[0] = d.f[0] - ix; w[1] = d.f[1] - iy; w[2] = d.f[2] - iz;
  const uint32_t i = dep_wrap(ix, A.nx), j = dep_wrap(iy, A.ny), k = dep_wrap(iz, A.nz);
  cell = ((k % TLZ) * TLY + j % TLY) * TLX + i % TLX;
  return ((k / TLZ) * T.nty + j / TLY) * T.ntx + i / TLX;
}

// Part of its tile's segment that a particle is counted in: a CTA's particles
// share one, the CTAs running at a time spread over all.
__device__ __forceinline__ uint32_t dep_way(const TileArgs &T, int64_t p) {
  return (uint32_t)(p / DEPOSIT_THREADS) & (T.ways - 1);
}

constexpr uint32_t NO_TILE = 0xFFFFFFFFu;
// Most records of a tile that one CTA sums; fewer where they would not fill the
// chip twice over.  The CTAs take the parts from a list: with the tiles' own
// numbers and a stride a sheet's tiles all fell to one CTA in 32.
constexpr uint32_t DEP_PART = 8192, DEP_PART_MIN = 2048;

// Whether the particles' order is scattered enough for tiles, from eight samples
// of 32 consecutive ones (the same for every CTA): by the tiles a sample lies in,
// 4 cells / n + 1 of them in an order by cell, which drift adds to.  The line is
// where both sides measured the same: 256^3 cells, one a cell 6.4 tiles (drift by
// 0.2 cells; by none 1051 us directly, 1131 by tiles, by two cells 1519, 1161), half
// of one 18.9 (583, 884; 909, 908); 320^3, half 14.3 (1128, 1685; 2229, 1728).
__device__ __forceinline__ bool dep_scattered(const DepArgs<float> &A, const TileArgs &T, int64_t n) {
  constexpr int SAMPLES = DEPOSIT_THREADS / 32;
  __shared__ uint32_t s_tiles[SAMPLES];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  DepPoint<float> d;
  float w[3];
  uint32_t t = 0xFFFFFFFFu, cell;
  const int64_t p = n / SAMPLES * wid + lane;
  if (p < n && dep_point(A, p, d)) t = dep_tile(A, T, d, w, cell);
  const unsigned first = __ballot_sync(0xFFFFFFFFu, lane == __ffs(__match_any_sync(0xFFFFFFFFu, t)) - 1);
  if (lane == 0) s_tiles[wid] = __popc(first);
  __syncthreads();
  uint32_t tiles = 0;
#pragma unroll
  for (int q = 0; q < SAMPLES; ++q) tiles += s_tiles[q];
  return tiles * n > SAMPLES * (10 * T.cells - 4 * n);
}

// Particles per tile, one atomic per distinct tile of a warp: the
// atomics of particles stored by cell would otherwise queue up on the counters
// of a few tiles.
__global__ void __launch_bounds__(DEPOSIT_THREADS) k_dep_count(DepArgs<float> A, TileArgs T) {
  const int64_t n = dep_count(A);
  const bool tiled = n >= T.min_n && n <= T.max_n && (n >= T.min_sorted || dep_scattered(A, T, n));
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // for the launches that follow
    T.meta[0] = T.meta[1] = 0u;
    T.meta[2] = tiled;
  }
  if (!tiled) return;
  const int lane = threadIdx.x & 31;
  unsigned bad = 0;
  // warp-uniform loop
  for (int64_t b = (int64_t)blockIdx.x * DEPOSIT_THREADS + (threadIdx.x & ~31); b < n;
       b += (int64_t)gridDim.x * DEPOSIT_THREADS) {
    const int64_t p = b + lane;
    uint32_t t = NO_TILE;
    DepPoint<float> d;
    if (p < n) {
      if (dep_point(A, p, d)) {
        float w[3];
        uint32_t cell;
        t = dep_tile(A, T, d, w, cell) * T.ways + dep_way(T, p);
      } else {
        bad = 1;
      }
    }
    const unsigned same = __match_any_sync(0xFFFFFFFFu, t);
    if (t != NO_TILE && lane == __ffs(same) - 1) atomicAdd(&T.cnt[t * SECTOR], (uint32_t)__popc(same));
  }
  if (bad) atomicOr(&A.cnt->status, (unsigned)QED_STATUS_NONFINITE);
}

// Record segments: any order of the tiles does, so a CTA takes room for its
// segments with one atomic (the parts of a tile stay next to each other: ways
// divides ALLOC_THREADS).
constexpr int ALLOC_THREADS = 256;
__global__ void __launch_bounds__(ALLOC_THREADS) k_dep_alloc(DepArgs<float> A, TileArgs T) {
  __shared__ uint32_t sm[33], s_start[ALLOC_THREADS];
  __shared__ uint32_t s_base;
  if (*(volatile uint32_t *)&T.meta[2] == 0u) return;
  const uint32_t t = blockIdx.x * ALLOC_THREADS + threadIdx.x, nseg = T.ntiles * T.ways;
  const uint32_t c = t < nseg ? T.cnt[t * SECTOR] : 0u;
  const uint32_t ex = block_excl_scan(c, sm);
  if (threadIdx.x == 0) s_base = sm[32] ? atomicAdd(&T.meta[0], sm[32]) : 0u;
  __syncthreads();
  s_start[threadIdx.x] = s_base + ex;
  if (c) {
    T.cursor[t * SECTOR] = s_base + ex;
    T.cnt[t * SECTOR] = 0u;
  }
  __syncthreads();
  // the tiles with records, in parts of (nearly) equal numbers
  uint32_t beg = 0, len = 0;
  if (t < nseg && t % T.ways == T.ways - 1) {
    beg = s_start[threadIdx.x - (T.ways - 1)];
    uint32_t end = s_base + ex + c;
    if (end > T.rec_cap) end = T.rec_cap;
    len = end > beg ? end - beg : 0;
  }
  const uint32_t fill = (uint32_t)dep_count(A) / T.most_ctas;
  const uint32_t most = fill < DEP_PART_MIN ? DEP_PART_MIN : fill > DEP_PART ? DEP_PART : fill;
  const uint32_t k = len <= most ? len > 0 : (len + most - 1) / most;
  const uint32_t at = block_excl_scan(k, sm);
  if (threadIdx.x == 0) s_base = sm[32] ? atomicAdd(&T.meta[1], sm[32]) : 0u;
  __syncthreads();
  if (k == 1) T.part[s_base + at] = make_uint4(t / T.ways, beg, beg + len, 0u);
  for (uint32_t q = 0; k > 1 && q < k; ++q)
    T.part[s_base + at + q] = make_uint4(t / T.ways, beg + (uint32_t)((uint64_t)len * q / k),
                                         beg + (uint32_t)((uint64_t)len * (q + 1) / k), 0u);
}

__global__ void __launch_bounds__(DEPOSIT_THREADS, 4)
k_dep_scatter(DepArgs<float> A, TileArgs T, DepRec *rec) {
  const int64_t n = dep_count(A);
  if (*(volatile uint32_t *)&T.meta[2] == 0u) {
    deposit_direct(A, n);
    return;
  }
  const int lane = threadIdx.x & 31;
  for (int64_t b = (int64_t)blockIdx.x * DEPOSIT_THREADS + (threadIdx.x & ~31); b < n;
       b += (int64_t)gridDim.x * DEPOSIT_THREADS) {
    const int64_t p = b + lane;
    uint32_t t = NO_TILE;
    DepRec r;
    bool direct = false;
    if (p < n) {
      const float a = A.scale * A.w[p];
      DepPoint<float> d;
      if (dep_point(A, p, d)) {
        uint32_t cell;
        t = dep_tile(A, T, d, r.w, cell) * T.ways + dep_way(T, p);
        r.key = (float)cell;
        r.pad = 0.f;
        direct = !isfinite(a);  // reaches its own eight nodes per component and no others
#pragma unroll
        for (int c = 0; c < 3; ++c) r.j[c] = direct ? 0.f : d.j[c] * a;
      }
    }
    const unsigned same = __match_any_sync(0xFFFFFFFFu, t);
    const int leader = __ffs(same) - 1;
    uint32_t pos = 0;
    if (t != NO_TILE && lane == leader) pos = atomicAdd(&T.cursor[t * SECTOR], (uint32_t)__popc(same));
    pos = __shfl_sync(0xFFFFFFFFu, pos, leader) + __popc(same & ((1u << lane) - 1u));
    if (t != NO_TILE) {
      if (pos < T.rec_cap) put_rec(rec + pos, r);
      else direct = true;  // no room for its record
    }
    if (direct) {
      DepPoint<float> d;
      dep_point(A, p, d);
      dep_direct(A, d, A.scale * A.w[p]);
    }
  }
}

// weights at the half-integer positions cell - 1/2, + 1/2, + 3/2
__device__ __forceinline__ void dep_half(float w, float s[3]) {
  const bool lo = w < 0.5f;
  const float u = lo ? w + 0.5f : w - 0.5f;
  s[0] = lo ? 1.f - u : 0.f;
  s[1] = lo ? u : 1.f - u;
  s[2] = lo ? 0.f : u;
}

// The sums of one cell's particles over the positions around it, [z][y][x] of
// each component: 12 of jx (2 x 2 x 3), of jy (2 x 3 x 2) and of jz (3 x 2 x 2).
template <int COMP> __device__ __forceinline__ void cell_add(const DepRec &r, float (&v)[12]) {
  const float wx = r.w[0], wy = r.w[1], wz = r.w[2];
  const float X[2] = {1.f - wx, wx}, Y[2] = {1.f - wy, wy}, Z[2] = {1.f - wz, wz};
  float h[3];
  dep_half(COMP == 0 ? wx : COMP == 1 ? wy : wz, h);
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const float f = COMP == 0 ? r.j[0] * Y[b] * Z[a] : COMP == 1 ? r.j[1] * X[b] * Z[a] : r.j[2] * X[b] * Y[a];
#pragma unroll
      for (int k = 0; k < 3; ++k) v[COMP == 0 ? (a * 2 + b) * 3 + k : COMP == 1 ? (a * 3 + k) * 2 + b : (k * 2 + a) * 2 + b] += f * h[k];
    }
}
struct CellSums {
  float vx[12], vy[12], vz[12];
  __device__ __forceinline__ float x(int z, int y, int i) const { return vx[(z * 2 + y) * 3 + i]; }
  __device__ __forceinline__ float y(int z, int j, int i) const { return vy[(z * 3 + j) * 2 + i]; }
  __device__ __forceinline__ float z(int k, int y, int i) const { return vz[(k * 2 + y) * 2 + i]; }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int q = 0; q < 12; ++q) vx[q] = vy[q] = vz[q] = 0.f;
  }
  __device__ __forceinline__ void add(const DepRec &r) {
    cell_add<0>(r, vx);
    cell_add<1>(r, vy);
    cell_add<2>(r, vz);
  }
};

// Place of a tile's cell in its halo tile.
__device__ __forceinline__ int cell_place(int c) {
  return ((c / (TLX * TLY) + 1) * HLY + c / TLX % TLY + 1) * HLX + c % TLX + 1;
}
// One component of a heavy cell's chunk by eight lanes, added to the halo tile J
// around the cell: lane by lane, then over the lanes by an exchange in which a
// lane keeps half of its sums at a time and is left with three.
template <int COMP>
__device__ __forceinline__ void chunk_add(const DepRec *rec, const uint16_t *perm, uint32_t len, float *J) {
  const int l = threadIdx.x & 7;
  float v[12] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (uint32_t i = l; i < len; i += 8) cell_add<COMP>(get_rec(rec + perm[i]), v);
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const float send = l & 4 ? v[i] : v[i + 6];
    v[i] = (l & 4 ? v[i + 6] : v[i]) + __shfl_xor_sync(0xFFFFFFFFu, send, 4);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float send = l & 2 ? v[i] : v[i + 3];
    v[i] = (l & 2 ? v[i + 3] : v[i]) + __shfl_xor_sync(0xFFFFFFFFu, send, 2);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) v[i] += __shfl_xor_sync(0xFFFFFFFFu, v[i], 1);
  // sums 3 (l / 2) .. + 2: the even lane adds the first and the last, the odd one the second
  auto add = [&](int q, float a) {
    const int x = COMP == 0 ? q % 3 - 1 : q % 2;
    const int y = COMP == 0 ? q / 3 % 2 : COMP == 1 ? q / 2 % 3 - 1 : q / 2 % 2;
    const int z = COMP == 2 ? q / 4 - 1 : q / 6;
    atomicAdd(J + COMP * HL_CELLS + (z * HLY + y) * HLX + x, a);
  };
  if (len) {
    const int q = 3 * (l >> 2) * 2 + 3 * (l >> 1 & 1);
    add(q + (l & 1), l & 1 ? v[1] : v[0]);
    if (!(l & 1)) add(q + 2, v[2]);
  }
}

// particles of a tile ordered by cell at a time (a warp's threads do as many
// turns as its fullest cell, so the more at a time the better they are used)
constexpr int DEP_BATCH = 2048;
// A cell with more particles of a batch (8 a cell in a full batch of a uniform
// plasma) is left to a second pass, which sums it by eight lanes per DEP_CHUNK
// particles: one thread's turns would hold up the CTA.  16.8M particles, 256^3
// cells, ms directly / all cells by threads / this way: half of them in one cell
// 19 / 1095 / 1.9, in a ball of 8 cells' deviation 1.5 / 3.2 / 1.2, a sheet of one
// cell 1.2 / 2.8 / 1.1, of two 1.1 / 1.9 / 1.2.  (A second pass, and not a branch of
// the first: with the sums of both live the registers spill, uniform plasma 5%.
// Chunks by whole warps: 10-30% slower; DEP_HEAVY 16 and 24 within 3%.)
constexpr int DEP_HEAVY = 32, DEP_CHUNK = 64;
constexpr int DEP_CHUNKS = DEP_BATCH / (DEP_HEAVY + 1) + DEP_BATCH / DEP_CHUNK + 1;  // most of a batch
static_assert(DEP_BATCH <= 1 << 11 && DEP_CHUNK <= 1 << 8 && TL_CELLS <= 1 << 8, "a chunk in one word");

// The chunks of a batch's heavy cells, eight lanes each (warp-uniform loop).
__device__ __forceinline__ void dep_chunks(const DepRec *rec, const uint16_t *perm, const uint32_t *chunk, uint32_t nchunks,
                                           float *J) {
  for (uint32_t q0 = threadIdx.x >> 5 << 2; q0 < nchunks; q0 += TILE_THREADS / 8) {
    const uint32_t q = q0 + (threadIdx.x >> 3 & 3), w = q < nchunks ? chunk[q] : 0u;
    const uint32_t len = q < nchunks ? (w >> 19) + 1 : 0u;
    const uint16_t *p = perm + (w >> 8 & 2047u);
    float *const base = J + cell_place((int)(w & 255u));
    chunk_add<0>(rec, p, len, base);
    chunk_add<1>(rec, p, len, base);
    chunk_add<2>(rec, p, len, base);
  }
}

struct TileSmem {
  uint16_t perm[DEP_BATCH];  // the batch's records by cell
  uint32_t cnt[TL_CELLS];
  uint32_t scan[33];
  uint32_t heavy, light;     // whether any batch has heavy cells, and the part others
  uint32_t chunk[DEP_CHUNKS], nchunks;  // chunks of heavy cells: cell, first, length - 1
  float J[3][HL_CELLS];
  int64_t row[HLY * HLZ];  // first element of J's row of each halo row
};

// The halo tile's rows of J, and the tile's zeros.
__device__ __forceinline__ void dep_begin(const DepArgs<float> &A, const TileArgs &T, uint32_t t, TileSmem &s) {
  const int c = threadIdx.x;
  if (c < HLY * HLZ) {
    int y = ((int)(t / T.ntx % T.nty * TLY) - 1 + c % HLY) % A.ny;
    int z = ((int)(t / (T.ntx * T.nty) * TLZ) - 1 + c / HLY) % A.nz;
    if (y < 0) y += A.ny;
    if (z < 0) z += A.nz;
    s.row[c] = ((int64_t)z * A.ny + y) * A.nx;
  }
  for (int q = threadIdx.x; q < 3 * HL_CELLS; q += TILE_THREADS) (&s.J[0][0])[q] = 0.f;
}

// The halo tile to J: 16 lanes per row, 10 of them with a column.
__device__ __forceinline__ void dep_end(const DepArgs<float> &A, const TileArgs &T, uint32_t t, TileSmem &s) {
  __syncthreads();
  const int hx = threadIdx.x & 15;
  int x = (int)(t % T.ntx * TLX) - 1 + hx;
  if (x < 0 || x >= A.nx) {
    x %= A.nx;
    if (x < 0) x += A.nx;
  }
  if (hx < HLX)
    for (int r = threadIdx.x >> 4; r < 3 * HLY * HLZ; r += TILE_THREADS / 16) {
      const float v = (&s.J[0][0])[r * HLX + hx];
      if (v == 0.f) continue;
      const int comp = r / (HLY * HLZ);
      atomicAdd((comp == 0 ? A.jx : comp == 1 ? A.jy : A.jz) + s.row[r - comp * (HLY * HLZ)] + x, v);
    }
  __syncthreads();  // the shared arrays are the next part's
}

// The order by cell of a batch of m records; the CTA's thread c gets cell c's
// records, `mine` of them from the return value on, and whether any cell has more
// than DEP_HEAVY.
__device__ __forceinline__ uint32_t dep_sort(const DepRec *rec, uint32_t m, TileSmem &s, uint32_t &mine, bool &heavy) {
  constexpr int PER = DEP_BATCH / TILE_THREADS;
  s.cnt[threadIdx.x] = 0;
  __syncthreads();
  // a record's rank among its cell's, then its place in cell order
  uint32_t place[PER];  // cell | rank << 8
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    if (q * TILE_THREADS >= m) break;
    const uint32_t i = q * TILE_THREADS + threadIdx.x;
    if (i < m) {
      const uint32_t cell = (uint32_t)rec[i].key & (TL_CELLS - 1);
      place[q] = cell | atomicAdd(&s.cnt[cell], 1u) << 8;
    }
  }
  __syncthreads();
  mine = s.cnt[threadIdx.x];
  const uint32_t first = block_excl_scan(mine, s.scan);
  s.cnt[threadIdx.x] = first;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    if (q * TILE_THREADS >= m) break;
    const uint32_t i = q * TILE_THREADS + threadIdx.x;
    if (i < m) s.perm[s.cnt[place[q] & (TL_CELLS - 1)] + (place[q] >> 8)] = (uint16_t)i;
  }
  heavy = __syncthreads_or(mine > DEP_HEAVY) != 0;
  return first;
}

__global__ void __launch_bounds__(TILE_THREADS, 4)
k_dep_tile(DepArgs<float> A, TileArgs T, const DepRec *rec) {
  __shared__ TileSmem s;
  if (*(volatile uint32_t *)&T.meta[2] == 0u) return;
  const int c = threadIdx.x;
  // (little is kept over the sums: 36 of the 64 registers are theirs)
  const volatile uint32_t *const parts = &T.meta[1];
  if (c == 0) s.heavy = 0;
  for (uint32_t part = blockIdx.x; part < *parts; part += gridDim.x) {
    dep_begin(A, T, T.part[part].x, s);
    if (c == 0) s.light = 0;  // (set after the sort's barriers)
    CellSums S;
    S.clear();
    const uint32_t end = T.part[part].z;
    for (uint32_t b = T.part[part].y; b < end; b += DEP_BATCH) {
      uint32_t mine;
      bool heavy;
      const uint32_t first = dep_sort(rec + b, end - b < DEP_BATCH ? end - b : DEP_BATCH, s, mine, heavy);
      if (heavy) {
        if (c == 0) {
          s.heavy = 1;
          T.part[part].w |= 1u << (b - T.part[part].y) / DEP_BATCH;
        }
        if (mine > DEP_HEAVY) mine = 0;
        else if (mine) s.light = 1;
      } else if (c == 0) {
        s.light = 1;
      }
      for (uint32_t i = first; i < first + mine; ++i) S.add(get_rec(rec + b + s.perm[i]));
      __syncthreads();
    }
    if (!s.light) continue;
    // the cells' sums into the halo tile.  Along x (8 consecutive lanes) by
    // shuffles: a lane keeps what lies on its own column, the row's first and
    // last lane also the columns beside the tile; then in rounds in which every
    // thread adds at the same offset from its own cell, so that no two add to
    // one place
    const int lx = c % TLX, h0 = cell_place(c);
    const bool first_x = lx == 0, last_x = lx == TLX - 1;
    auto up = [&](float v) { const float r = __shfl_up_sync(0xFFFFFFFFu, v, 1, TLX); return first_x ? 0.f : r; };
    auto down = [&](float v) { const float r = __shfl_down_sync(0xFFFFFFFFu, v, 1, TLX); return last_x ? 0.f : r; };
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int w = 0; w < 3; ++w) {
        __syncthreads();
        if (w < 2) {
          const int h = h0 + (u * HLY + w) * HLX;
          const float v = S.x(u, w, 1) + up(S.x(u, w, 2)) + down(S.x(u, w, 0));
          s.J[0][h] += v;
          if (first_x) s.J[0][h - 1] += S.x(u, w, 0);
          if (last_x) s.J[0][h + 1] += S.x(u, w, 2);
        }
        const int hy = h0 + (u * HLY + w - 1) * HLX, hz = h0 + ((w - 1) * HLY + u) * HLX;
        const float vy = S.y(u, w, 0) + up(S.y(u, w, 1)), vz = S.z(w, u, 0) + up(S.z(w, u, 1));
        s.J[1][hy] += vy;
        s.J[2][hz] += vz;
        if (last_x) {
          s.J[1][hy + 1] += S.y(u, w, 1);
          s.J[2][hz + 1] += S.z(w, u, 1);
        }
      }
    dep_end(A, T, T.part[part].x, s);
  }
  __syncthreads();  // (a CTA without parts)
  if (!s.heavy) return;
  // the heavy cells of this CTA's parts, their batches sorted again (apart from
  // the threads' sums, which fill the registers)
  for (uint32_t part = blockIdx.x; part < *parts; part += gridDim.x) {
    const uint4 range = T.part[part];
    if (range.w == 0) continue;
    dep_begin(A, T, range.x, s);
    for (uint32_t h = range.w; h; h &= h - 1) {
      const uint32_t b = range.y + (__ffs(h) - 1) * DEP_BATCH;
      if (c == 0) s.nchunks = 0;
      uint32_t mine;
      bool heavy;
      const uint32_t first = dep_sort(rec + b, range.z - b < DEP_BATCH ? range.z - b : DEP_BATCH, s, mine, heavy);
      if (mine > DEP_HEAVY) {
        const uint32_t k = (mine + DEP_CHUNK - 1) / DEP_CHUNK, at = atomicAdd(&s.nchunks, k);
        for (uint32_t q = 0; q < k; ++q) {
          const uint32_t left = mine - q * DEP_CHUNK, len = left < DEP_CHUNK ? left : DEP_CHUNK;
          s.chunk[at + q] = (uint32_t)c | (first + q * DEP_CHUNK) << 8 | (len - 1) << 19;
        }
      }
      __syncthreads();
      dep_chunks(rec + b, s.perm, s.chunk, s.nchunks, &s.J[0][0]);
      __syncthreads();
    }
    dep_end(A, T, range.x, s);
  }
}

bool yee_ok(const qed_yee *y) {
  if (!y || y->nx < 1 || y->ny < 1 || y->nz < 1 || y->nx > 65536 || y->ny > 65536 ||
      y->nz > 65536 || (int64_t)y->ny * y->nz > 0x7fffffffLL)
    return false;
  if (!(y->dx > 0) || !(y->dy > 0) || !(y->dz > 0) || !std::isfinite(y->dx) ||
      !std::isfinite(y->dy) || !std::isfinite(y->dz) || !std::isfinite(y->x0) ||
      !std::isfinite(y->y0) || !std::isfinite(y->z0))
    return false;
  const void *p[] = {y->ex, y->ey, y->ez, y->bx, y->by, y->bz, y->jx, y->jy, y->jz, y->nodes};
  for (const void *q : p)
    if (!q || (reinterpret_cast<uintptr_t>(q) & 15) != 0) return false;
  return true;
}

bool courant_ok(const qed_yee *y, double dt) {
  double s = 0;
  if (y->nx > 1) s += 1.0 / (y->dx * y->dx);
  if (y->ny > 1) s += 1.0 / (y->dy * y->dy);
  if (y->nz > 1) s += 1.0 / (y->dz * y->dz);
  return dt * std::sqrt(s) < 1.0;
}

// A pass of V cells a thread over all rows: one launch, or one per slab of rows
// where the threads' numbers would not fit 32 bits (beyond 4.2e9 cells).
template <int V, class Launch> void field_pass(qed_ctx *c, YeeArgs A, Launch launch) {
  const int64_t rows = (int64_t)A.ny * A.nz, per_row = A.nx / V, slab = slab_rows(per_row, FIELD_THREADS);
  for (int64_t r = 0; r < rows; r += slab) {
    A.row0 = (uint32_t)r;
    A.rows = (uint32_t)(rows - r < slab ? rows - r : slab);
    launch(A, (unsigned)((A.rows * per_row + FIELD_THREADS - 1) / FIELD_THREADS));
    c->launches += 1;
  }
}

template <int V> void launch_advance(qed_ctx *c, const YeeArgs &A, float dt, cudaStream_t st) {
  auto b_half = [&](const YeeArgs &a, unsigned grid) { k_yee_b_half<V><<<grid, FIELD_THREADS, 0, st>>>(a, 0.5f * dt); };
  field_pass<V>(c, A, b_half);
  field_pass<V>(c, A, [&](const YeeArgs &a, unsigned grid) { k_yee_e<V><<<grid, FIELD_THREADS, 0, st>>>(a, dt); });
  field_pass<V>(c, A, b_half);
}

cudaError_t launch_fields(qed_ctx *c, const qed_yee *y, bool advance, cudaStream_t st) {
  const YeeArgs A = yee_args(y);
  if (advance) {
    if (A.nx % 4 == 0) launch_advance<4>(c, A, (float)c->cfg.dt, st);
    else launch_advance<1>(c, A, (float)c->cfg.dt, st);
  }
  field_pass<1>(c, A, [&](const YeeArgs &a, unsigned grid) { k_yee_nodes<<<grid, FIELD_THREADS, 0, st>>>(a); });
  return cudaGetLastError();
}

// Persistent grid over `capacity` particles: no more CTAs than they need.
template <class Kern>
cudaError_t particle_grid(const qed_ctx *c, Kern kern, int64_t capacity, unsigned *blocks) {
  int per_sm = 0;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, DEPOSIT_THREADS, 0);
  if (e != cudaSuccess) return e;
  const int64_t need = (capacity + DEPOSIT_THREADS - 1) / DEPOSIT_THREADS;
  int64_t b = (int64_t)c->num_sms * (per_sm < 1 ? 1 : per_sm);
  if (need < b) b = need;
  *blocks = (unsigned)(b < 1 ? 1 : b);
  return cudaSuccess;
}

// When the tiled path is taken.  The rule is on the number of particles on the
// device; the host sees only capacities, so where the capacity allows the
// tiled path its four kernels are launched and for fewer particles the scatter
// pass deposits them directly, the others return at once (1000 particles, room
// for 2^24: 24.7 us a call; 29.4 with a launch of its own for the direct deposit
// and a clear of the counters, 13.7 by one kernel).
// Measured on the device, tiled / direct in us (stored by cell; random order):
//   32^3 cells:  2^18 particles 28/37; 32/28    3 2^17 31/66; 34/42   2^20 62/177; 58/111
//   64^3:        3 2^17 33/32; 39/33            2^19 36/42; 44/43     2^23 407/917; 368/657
//   128^3:       2^21 148/139; 165/157          2^22 214/284; 246/323 2^24 580/1455; 834/1268
//   180^3:       2^22 350/275; 381/331          2^23 479/534; 550/651
//   200^3:       2^22 420/284; 449/501          2^23 546/535; 617/898
//   256^3:       2^23 852/556; 919/2538         2^24 1094/1026; 1349/5055
// so two particles per cell and 3 2^17 pay for a tile's fixed work.  Where J (12
// bytes a cell) no longer fits L2 a direct deposit in random order fetches its
// lines each time, and half a particle per cell pays; stored by cell it takes one
// and a half (200^3: 679/776), in between as the order goes (dep_scattered, which
// makes the 1026 above 1040).
// Grids of few tiles and more than 64 particles a cell are not taken.
// FP64 contexts deposit directly: GB300 adds and multiplies doubles at a small
// fraction of its float rate, and a tile is that work (128^3, 2^22 random: 1093 us
// directly, 2369 by tiles; 64^3, 2^19: 161, 352).
constexpr int64_t TILED_MIN_PARTICLES = 3 << 17, TILED_MIN_TILES = 128, TILED_MAX_PER_CELL = 64;
constexpr int64_t L2_CELLS = 6 << 20;
// counters of a grid with few tiles: a ball of particles queues on few of them
// (128^3, 2^22: 470 us with 4096, 370 with 16384; uniform 288, 281)
constexpr int64_t DEP_SEGMENTS = 16384;

// The launches of a deposit where the capacities allow the tiled path, else
// *done is left false.  The scratch is the step's (free between steps, and calls
// that share a context are ordered): records in the staging area, cursors and
// parts in the per-entry counts.
cudaError_t launch_deposit_tiled(qed_ctx *c, const DepArgs<float> &A, const qed_yee *y, bool *done, cudaStream_t st) {
  TileArgs T;
  T.ntx = (y->nx + TLX - 1) / TLX;
  T.nty = (y->ny + TLY - 1) / TLY;
  const int64_t cells = (int64_t)y->nx * y->ny * y->nz;
  const int64_t ntiles = (int64_t)T.ntx * T.nty * ((y->nz + TLZ - 1) / TLZ);
  T.ways = 1;
  while (ntiles * T.ways < DEP_SEGMENTS && T.ways < 64) T.ways *= 2;
  const int64_t nseg = ntiles * T.ways;
  const bool large = cells > L2_CELLS;
  T.min_n = large ? cells / 2 : 2 * cells;
  if (T.min_n < TILED_MIN_PARTICLES) T.min_n = TILED_MIN_PARTICLES;
  T.min_sorted = large ? 3 * cells / 2 : T.min_n;
  T.cells = cells;
  T.max_n = ntiles < TILED_MIN_TILES ? 0 : cells * TILED_MAX_PER_CELL;
  const int64_t cap = 2 * c->stage_cap;  // a staging record holds two of these
  T.rec_cap = (uint32_t)(cap < 0x7fffffff ? cap : 0x7fffffff);
  T.most_ctas = (uint32_t)c->num_sms * 8;
  const int64_t scratch = SECTOR * nseg + 4 * (ntiles + T.rec_cap / DEP_PART_MIN);
  if (T.max_n < T.min_n || A.cap < T.min_n || A.cap > 0x7fffffff || nseg > c->dep_segs || scratch > c->heavy_slots)
    return cudaSuccess;
  *done = true;
  T.ntiles = (uint32_t)ntiles;
  T.meta = c->dep_cnt;
  T.cnt = c->dep_cnt + SECTOR;
  T.cursor = c->sub_cnt;
  T.part = reinterpret_cast<uint4 *>(c->sub_cnt + SECTOR * nseg);
  DepRec *rec = static_cast<DepRec *>(c->stage);
  unsigned count_blocks = 0, blocks = 0;
  cudaError_t e = particle_grid(c, k_dep_count, A.cap, &count_blocks);
  if (e == cudaSuccess) e = particle_grid(c, k_dep_scatter, A.cap, &blocks);
  if (e != cudaSuccess) return e;
  k_dep_count<<<count_blocks, DEPOSIT_THREADS, 0, st>>>(A, T);
  k_dep_alloc<<<(unsigned)((nseg + ALLOC_THREADS - 1) / ALLOC_THREADS), ALLOC_THREADS, 0, st>>>(A, T);
  k_dep_scatter<<<blocks, DEPOSIT_THREADS, 0, st>>>(A, T, rec);
  // (four waves; a call without tiles waits for every CTA to leave: 24.7 us a call
  // of 1000 particles with 16 CTAs per SM, 28.3 with 32)
  const uint32_t most = (uint32_t)c->num_sms * 16, need = T.ntiles + T.rec_cap / DEP_PART_MIN;
  k_dep_tile<<<need < most ? need : most, TILE_THREADS, 0, st>>>(A, T, rec);
  c->launches += 4;
  return cudaGetLastError();
}

template <class Real>
cudaError_t launch_deposit(qed_ctx *c, const qed_species *s, const qed_yee *y, double weight_unit,
                           const int64_t *d_lim, cudaStream_t st) {
  DepArgs<Real> A;
  A.x = static_cast<const Real *>(s->x); A.y = static_cast<const Real *>(s->y);
  A.z = static_cast<const Real *>(s->z);
  A.px = static_cast<const Real *>(s->px); A.py = static_cast<const Real *>(s->py);
  A.pz = static_cast<const Real *>(s->pz); A.w = static_cast<const Real *>(s->w);
  A.d_n = s->d_n; A.d_lim = d_lim; A.cap = s->capacity;
  A.jx = y->jx; A.jy = y->jy; A.jz = y->jz;
  A.nx = y->nx; A.ny = y->ny; A.nz = y->nz;
  A.idx = (Real)(1.0 / y->dx); A.idy = (Real)(1.0 / y->dy); A.idz = (Real)(1.0 / y->dz);
  A.x0 = (Real)y->x0; A.y0 = (Real)y->y0; A.z0 = (Real)y->z0;
  A.scale = (Real)((double)s->q * weight_unit / (y->dx * y->dy * y->dz));
  A.half_dt = (Real)(0.5 * c->cfg.dt);
  A.cnt = c->d_counters;
  if constexpr (sizeof(Real) == 4) {
    bool done = false;
    const cudaError_t e = launch_deposit_tiled(c, A, y, &done, st);
    if (e != cudaSuccess || done) return e;
  }
  unsigned blocks = 0;
  const cudaError_t e = particle_grid(c, k_pic_deposit<Real>, s->capacity, &blocks);
  if (e != cudaSuccess) return e;
  k_pic_deposit<Real><<<blocks, DEPOSIT_THREADS, 0, st>>>(A);
  c->launches += 1;
  return cudaGetLastError();
}

__global__ void k_copy_counts(int64_t *dst, const int64_t *a, const int64_t *b) {
  dst[0] = *a;
  dst[1] = *b;
}

// a lepton species (an empty one of any charge is accepted: it deposits nothing)
bool lepton_ok(const qed_species *s) {
  if (!s || !s->d_n || s->capacity < 0) return false;
  if (s->capacity == 0) return true;
  return s->q != 0 && s->x && s->y && s->z && s->px && s->py && s->pz && s->w;
}

}  // namespace
}  // namespace qed

using namespace qed;

extern "C" int qed_pic_deposit(qed_ctx *c, const qed_species *s, const qed_yee *y,
                               double weight_unit, const int64_t *d_count, qed_stream_t stream) {
  if (!c || !lepton_ok(s) || !yee_ok(y) || !std::isfinite(weight_unit)) return QED_ERR_ARG;
  if (s->capacity == 0) return QED_OK;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = c->cfg.precision == QED_FP64
                      ? launch_deposit<double>(c, s, y, weight_unit, d_count, st)
                      : launch_deposit<float>(c, s, y, weight_unit, d_count, st);
  return cuda_fail(e, "qed_pic_deposit");
}

extern "C" int qed_pic_fields(qed_ctx *c, const qed_yee *y, int advance, qed_stream_t stream) {
  if (!c || !yee_ok(y) || (advance && !courant_ok(y, c->cfg.dt))) return QED_ERR_ARG;
  return cuda_fail(launch_fields(c, y, advance != 0, (cudaStream_t)stream), "qed_pic_fields");
}

extern "C" int qed_pic_step(qed_ctx *c, const qed_species *e, const qed_species *p,
                            const qed_species *g, const qed_yee *y, double weight_unit, int64_t step,
                            qed_stream_t stream) {
  if (!c || !yee_ok(y) || !courant_ok(y, c->cfg.dt) || !std::isfinite(weight_unit) ||
      !lepton_ok(e) || !lepton_ok(p))
    return QED_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  // lepton counts before the step: the leptons its pairs create are
  // deposited from the next step on
  k_copy_counts<<<1, 1, 0, st>>>(c->pic_n, e->d_n, p->d_n);
  c->launches += 1;
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return cuda_fail(err, "qed_pic_step");
  qed_fields f{};
  f.mode = QED_FIELDS_GRID;
  f.nx = y->nx; f.ny = y->ny; f.nz = y->nz;
  f.grid = y->nodes;
  f.dx = y->dx; f.dy = y->dy; f.dz = y->dz;
  f.x0 = y->x0; f.y0 = y->y0; f.z0 = y->z0;
  int rc = qed_step_fused(c, e, p, g, &f, step, stream);
  if (rc == QED_OK) rc = qed_pic_deposit(c, e, y, weight_unit, c->pic_n, stream);
  if (rc == QED_OK) rc = qed_pic_deposit(c, p, y, weight_unit, c->pic_n + 1, stream);
  if (rc == QED_OK) rc = qed_pic_fields(c, y, 1, stream);
  return rc;
}
