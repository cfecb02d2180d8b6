// qed_mlp.cu -- training and loading of the surrogate inverse CDF (the
// network is described in qed_mlp.cuh).
//
// Training (qed_mlp_train) runs entirely on the GPU with the project's own
// kernels:
//   k_mlp_grad   each CTA draws mini-batches of (ln chi, kappa) uniformly over
//                the network's domain (Philox), takes the target ln delta from
//                the FP64 inverse table (bicubic, FP64), and runs the forward
//                pass and the hand-written backward pass in FP32 as register-
//                tiled products (activations of one mini-batch in shared
//                memory); the CTA's gradient sum goes to its own row of a
//                partial-gradient array;
//   k_mlp_adam   sums the partial rows in a fixed order (deterministic), and
//                applies one bias-corrected Adam step to the FP32 weights;
//   k_mlp_pack   converts W2 and W3 to BF16 tensor-core fragments.
// The loss is the mean squared error of z (ln delta minus its asymptote).
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "qed_internal.h"
#include "qed_mlp.cuh"

namespace qed {

constexpr int GRAD_B = 128;            // samples per mini-batch
constexpr int GRAD_MATH = 256;         // threads of the matrix work: 8 samples x 4 units each
constexpr int GRAD_THREADS = GRAD_MATH + GRAD_B;  // and one thread per sample of the next mini-batch
constexpr int ALD = GRAD_B + 4;        // row length of the activation arrays [unit][sample]
constexpr int LOSS_ROWS = 8;           // optimiser steps whose losses are kept on the device

struct GradArgs {
  const float *w;        // FP32 weights
  float *partial;        // [gridDim.x][MLP_NP]
  double *loss_sum;      // [gridDim.x] sum of squared residuals
  // generated batches
  const double *Y64;     // FP64 inverse table (l rows, kappa columns)
  GridR<double> gl, gk;
  uint64_t seed;
  int64_t step;
  int batches_per_cta;
  // explicit batch (gradient checks): x [n][2], t [n]
  const float *x, *t;
  int64_t n;
  float scale;           // dL/dz = scale * (z - t)
};

// Shared memory of the gradient kernel.  Activations are kept unit-major, so
// that eight samples of a unit are two 16-byte loads; the weights twice, each
// with the four units u, u + 16, u + 32, u + 48 of a thread side by side:
// Wp[k][4 u' + q] = W[k][u' + 16 q] for the forward products and
// WT[k][4 u' + q] = W[u' + 16 q][k] for the backward ones.
struct GradSmem {
  float Wp[2][64 * 64], WT[2][64 * 64];
  float W1[128], b1[64], b2[64], b3[64], W4[64], b4[4];
  float X[2][2][GRAD_B], T[2][GRAD_B];  // inputs and targets (then dL/dz), two mini-batches
  float Zp[GRAD_B];                     // half-row output partials
  float H1[64 * ALD], H2[64 * ALD], D2[64 * ALD], D3[64 * ALD];
  double loss[GRAD_MATH / 32];
};

// C[8][4] += A[k][samples r0 .. r0+7] B[k][4 cg ..] over the 64 units k
__device__ __forceinline__ void gemm_8x4(const float *A, const float *B, int r0, int cg, float (&acc)[8][4]) {
#pragma unroll 4
  for (int k = 0; k < 64; ++k) {
    const float4 a0 = *reinterpret_cast<const float4 *>(A + k * ALD + r0);
    const float4 a1 = *reinterpret_cast<const float4 *>(A + k * ALD + r0 + 4);
    const float4 w = *reinterpret_cast<const float4 *>(B + k * 64 + 4 * cg);
    const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][q] = fmaf(av[i], wv[q], acc[i][q]);
  }
}

// G[i][q] += the sum over the mini-batch, in sample order, of
// H[jg + 16 i][s] D[kg + 16 q][s]
__device__ __forceinline__ void outer_4x4(const float *H, const float *D, int jg, int kg, float (&G)[4][4]) {
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[i][q] = 0.f;
#pragma unroll 2
  for (int r = 0; r < GRAD_B; r += 4) {
    float4 h[4], d[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      h[q] = *reinterpret_cast<const float4 *>(H + (jg + 16 * q) * ALD + r);
      d[q] = *reinterpret_cast<const float4 *>(D + (kg + 16 * q) * ALD + r);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        acc[i][q] = fmaf(h[i].w, d[q].w, fmaf(h[i].z, d[q].z, fmaf(h[i].y, d[q].y, fmaf(h[i].x, d[q].x, acc[i][q]))));
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) G[i][q] += acc[i][q];
}

// sum over the mini-batch, in sample order, of f[s] row[s] (f null: of row[s])
__device__ __forceinline__ float sample_sum(const float *row, const float *f) {
  float v = 0.f;
#pragma unroll 4
  for (int r = 0; r < GRAD_B; r += 4) {
    const float4 a = *reinterpret_cast<const float4 *>(row + r);
    const float4 b = f ? *reinterpret_cast<const float4 *>(f + r) : make_float4(1.f, 1.f, 1.f, 1.f);
    v = fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, v))));
  }
  return v;
}

__device__ __forceinline__ void put8(float *row, const float (&v)[8]) {
  *reinterpret_cast<float4 *>(row) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4 *>(row + 4) = make_float4(v[4], v[5], v[6], v[7]);
}

// SiLU and its derivative at a
__device__ __forceinline__ float silu_f(float a) { return a / (1.f + __expf(-a)); }
__device__ __forceinline__ float dsilu_f(float a) {
  const float s = 1.f / (1.f + __expf(-a));
  return s * (1.f + a * (1.f - s));
}

// the math threads' own barrier
__device__ __forceinline__ void math_sync() { asm volatile("bar.sync 1, %0;\n" ::"n"(GRAD_MATH) : "memory"); }

// all threads, reached from the two roles' own code
__device__ __forceinline__ void block_sync() { asm volatile("bar.sync 0, %0;\n" ::"n"(GRAD_THREADS) : "memory"); }

// Input and target of sample t of mini-batch bi.
__device__ __forceinline__ void grad_input(const GradArgs &A, GradSmem &S, int bi, int t) {
  const int64_t s = ((int64_t)bi * gridDim.x + blockIdx.x) * GRAD_B + t;
  float x0 = 0.f, x1 = 0.f, tt = 0.f;
  bool valid = true;
  if (A.x) {
    valid = s < A.n;
    if (valid) { x0 = A.x[2 * s]; x1 = A.x[2 * s + 1]; tt = A.t[s]; }
  } else {
    U4 r = philox4x32_10(U4{(uint32_t)s, (uint32_t)(s >> 32), (uint32_t)A.step, 0x4D4C5031u},
                         (uint32_t)A.seed, (uint32_t)(A.seed >> 32));
    const double ul = ((double)r.x + 0.5) * 0x1p-32, uk = ((double)r.y + 0.5) * 0x1p-32;
    // the training domain extends past the one the network serves, so
    // that its edges are not the edges of the fit
    const double l = (MLP_L_LO - MLP_TRAIN_DL) + (MLP_L_HI - MLP_L_LO + 2 * MLP_TRAIN_DL) * ul;
    const double k = (MLP_K_LO - MLP_TRAIN_DK) + (MLP_K_HI - MLP_K_LO + 2 * MLP_TRAIN_DK) * uk;
    const double Y = interp2(A.Y64, A.gl, l, A.gk, k);
    const double sp = k > 30.0 ? k : log1p(exp(k));
    x0 = (float)((l - MLP_LC) / MLP_LS);
    x1 = (float)((k - MLP_KC) / MLP_KS);
    tt = (float)(Y - (3.0 * k - 2.0 * sp));
  }
  S.X[bi & 1][0][t] = x0;
  S.X[bi & 1][1][t] = x1;
  S.T[bi & 1][t] = valid ? tt : NAN;  // NaN marks a padding row (no gradient)
}

// One CTA per SM.  The eight math warps run the six 64-wide matrix products of
// a mini-batch (two forward, two weight gradients, two backward) as register
// tiles: 8 samples x 4 units a thread, 32 FMAs per three 16-byte shared loads;
// the weight gradients stay in registers over the CTA's mini-batches.  The
// four auxiliary warps meanwhile make the next mini-batch's targets, whose
// FP64 arithmetic would otherwise stand alone, and the sums over samples of
// W1, W4 and the biases.  Every sum is taken in the order of the units or the
// samples, so the result does not depend on how the work is divided.
__global__ void __launch_bounds__(GRAD_THREADS, 1) k_mlp_grad(GradArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  GradSmem &S = *reinterpret_cast<GradSmem *>(smem_raw);
  const int tid = threadIdx.x;
  for (int k = tid; k < 64 * 64; k += GRAD_THREADS) {
    const int in = k >> 6, out = k & 63;
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      const float w = A.w[(l ? MLP_OFF_W3 : MLP_OFF_W2) + k];
      S.Wp[l][in * 64 + 4 * (out & 15) + (out >> 4)] = w;
      S.WT[l][out * 64 + 4 * (in & 15) + (in >> 4)] = w;
    }
  }
  if (tid < 128) S.W1[tid] = A.w[MLP_OFF_W1 + tid];
  if (tid < 64) {
    S.b1[tid] = A.w[MLP_OFF_B1 + tid];
    S.b2[tid] = A.w[MLP_OFF_B2 + tid];
    S.b3[tid] = A.w[MLP_OFF_B3 + tid];
    S.W4[tid] = A.w[MLP_OFF_W4 + tid];
  }
  if (tid == 0) S.b4[0] = A.w[MLP_OFF_B4];
  const int nb = A.x ? (int)((A.n + (int64_t)GRAD_B * gridDim.x - 1) / ((int64_t)GRAD_B * gridDim.x))
                     : A.batches_per_cta;
  float *P = A.partial + (size_t)blockIdx.x * MLP_NP;
  if (tid >= GRAD_MATH) {
    // ---- auxiliary warps: the block barriers match the math warps' below
    const int a = tid - GRAD_MATH, c = a & 63;
    const bool lo = a < 64;
    float gW4 = 0.f, gb4 = 0.f, gb3 = 0.f, gb2 = 0.f, gb1 = 0.f, gW1 = 0.f;
    grad_input(A, S, 0, a);
    block_sync();
    for (int bi = 0; bi < nb; ++bi) {
      const float *T = S.T[bi & 1], *X = S.X[bi & 1][lo ? 0 : 1];
      block_sync();  // (H2 free)
      block_sync();  // h3 in D3, dL/dz in T
      if (lo) gW4 += sample_sum(S.D3 + c * ALD, T);
      else if (a == 64) gb4 += sample_sum(T, nullptr);
      block_sync();  // (D3 free)
      block_sync();  // dA3 in D3
      if (!lo) gb3 += sample_sum(S.D3 + c * ALD, nullptr);
      if (bi + 1 < nb) grad_input(A, S, bi + 1, a);
      block_sync();  // dA2 in D2
      if (lo) gb2 += sample_sum(S.D2 + c * ALD, nullptr);
      block_sync();  // dA1 in H2, the next inputs in X and T
      if (lo) gb1 += sample_sum(S.H2 + c * ALD, nullptr);
      gW1 += sample_sum(S.H2 + c * ALD, X);
    }
    P[MLP_OFF_W1 + a] = gW1;
    if (lo) {
      P[MLP_OFF_W4 + c] = gW4;
      P[MLP_OFF_B2 + c] = gb2;
      P[MLP_OFF_B1 + c] = gb1;
    } else {
      P[MLP_OFF_B3 + c] = gb3;
      if (a == 64) P[MLP_OFF_B4] = gb4;
    }
    return;
  }
  // ---- math warps
  const int r0 = (tid >> 4) * 8, cg = tid & 15, jg = tid >> 4;  // samples, units; weight-gradient rows
  const int row = tid & (GRAD_B - 1), c0 = (tid / GRAD_B) * 32;  // output layer: sample, unit half
  float G2[4][4], G3[4][4];
  double loss = 0.0;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) G2[i][q] = G3[i][q] = 0.f;
  block_sync();
  for (int bi = 0; bi < nb; ++bi) {
    const float *X0 = S.X[bi & 1][0] + r0, *X1 = S.X[bi & 1][1] + r0;
    float *T = S.T[bi & 1];
    // ---- forward: layer 1 on two inputs
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = cg + 16 * q;
      float h[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) h[i] = silu_f(fmaf(X0[i], S.W1[c], fmaf(X1[i], S.W1[64 + c], S.b1[c])));
      put8(S.H1 + c * ALD + r0, h);
    }
    math_sync();
    float acc[8][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i][q] = S.b2[cg + 16 * q];
    gemm_8x4(S.H1, S.Wp[0], r0, cg, acc);
    block_sync();  // H2 free (the sums of dA1 of the mini-batch before)
#pragma unroll
    for (int q = 0; q < 4; ++q) {  // layer 2's output and derivative
      const int c = cg + 16 * q;
      float h[8], d[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        h[i] = silu_f(acc[i][q]);
        d[i] = dsilu_f(acc[i][q]);
      }
      put8(S.H2 + c * ALD + r0, h);
      put8(S.D2 + c * ALD + r0, d);
    }
    math_sync();
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i][q] = S.b3[cg + 16 * q];
    gemm_8x4(S.H2, S.Wp[1], r0, cg, acc);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float h[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) h[i] = silu_f(acc[i][q]);
      put8(S.D3 + (cg + 16 * q) * ALD + r0, h);
    }
    math_sync();
    // output and dL/dz (two threads per sample, unit halves)
    {
      float part = 0.f;
#pragma unroll 8
      for (int c = c0; c < c0 + 32; ++c) part = fmaf(S.D3[c * ALD + row], S.W4[c], part);
      if (c0) S.Zp[row] = part;
      math_sync();
      if (!c0) {
        const float z = part + S.Zp[row] + S.b4[0], t = T[row];
        float dz = 0.f;
        if (!isnan(t)) {
          const float r = z - t;
          loss += (double)r * r;
          dz = A.scale * r;
        }
        T[row] = dz;
      }
    }
    block_sync();  // h3 in D3, dL/dz in T
    // ---- backward: dA3 = dL/dz W4 silu'(a3)
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i][q] = T[r0 + i] * S.W4[cg + 16 * q] * dsilu_f(acc[i][q]);
    block_sync();  // D3 free
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float d[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) d[i] = acc[i][q];
      put8(S.D3 + (cg + 16 * q) * ALD + r0, d);
    }
    block_sync();  // dA3 in D3
    outer_4x4(S.H2, S.D3, jg, cg, G3);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i][q] = 0.f;
    gemm_8x4(S.D3, S.WT[1], r0, cg, acc);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float *own = S.D2 + (cg + 16 * q) * ALD + r0;  // this thread's elements
      float d[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) d[i] = acc[i][q] * own[i];
      put8(own, d);
    }
    block_sync();  // dA2 in D2
    outer_4x4(S.H1, S.D2, jg, cg, G2);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i][q] = 0.f;
    gemm_8x4(S.D2, S.WT[0], r0, cg, acc);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = cg + 16 * q;
      float d[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        d[i] = acc[i][q] * dsilu_f(fmaf(X0[i], S.W1[c], fmaf(X1[i], S.W1[64 + c], S.b1[c])));
      put8(S.H2 + c * ALD + r0, d);
    }
    block_sync();  // dA1 in H2
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int o = (jg + 16 * i) * 64 + cg + 16 * q;
      P[MLP_OFF_W2 + o] = G2[i][q];
      P[MLP_OFF_W3 + o] = G3[i][q];
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
  if ((tid & 31) == 0) S.loss[tid >> 5] = loss;
  math_sync();
  if (tid == 0) {
    double s = 0.0;
    for (int w = 0; w < GRAD_MATH / 32; ++w) s += S.loss[w];
    A.loss_sum[blockIdx.x] = s;
  }
}

struct AdamArgs {
  float *w, *m, *v;
  const float *partial;
  int nparts;
  float lr, b1, b2, eps, bc1, bc2;
  float *grad_out;  // optional: the summed gradient (gradient checks)
  int apply;
};

// One thread per parameter in CTAs of one warp, so that the rows' loads come
// from every SM; the rows are added in order, ADAM_BATCH loads in flight.
constexpr int ADAM_THREADS = 32, ADAM_BATCH = 16;
constexpr int ADAM_BLOCKS = (MLP_NP + ADAM_THREADS - 1) / ADAM_THREADS;
__global__ void __launch_bounds__(ADAM_THREADS) k_mlp_adam(AdamArgs A) {
  const int k = blockIdx.x * ADAM_THREADS + threadIdx.x;
  if (k >= MLP_NP) return;
  float g = 0.f;
#pragma unroll 2
  for (int p = 0; p < A.nparts; p += ADAM_BATCH) {
    float v[ADAM_BATCH];
#pragma unroll
    for (int q = 0; q < ADAM_BATCH; ++q) v[q] = p + q < A.nparts ? A.partial[(size_t)(p + q) * MLP_NP + k] : 0.f;
#pragma unroll
    for (int q = 0; q < ADAM_BATCH; ++q) g += v[q];
  }
  if (A.grad_out) A.grad_out[k] = g;
  if (!A.apply) return;
  const float m = A.b1 * A.m[k] + (1.f - A.b1) * g;
  const float v = A.b2 * A.v[k] + (1.f - A.b2) * g * g;
  A.m[k] = m;
  A.v[k] = v;
  A.w[k] -= A.lr * (m / A.bc1) / (sqrtf(v / A.bc2) + A.eps);
}

// BF16 B fragments of W2 and W3 for mma.sync m16n8k16 (B = W, K x N): the
// high parts, then the remainders W - hi (see qed_mlp.cuh).
__device__ __forceinline__ void pack_split(float a, float b, uint32_t &hi, uint32_t &lo) {
  split_bf16(a, b, hi, lo);
}

__global__ void k_mlp_pack(const float *w, uint32_t *frag) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;  // over [layer][kt][nt][lane]
  if (idx >= 2 * 4 * 8 * 32) return;
  const int lane = idx & 31, nt = (idx >> 5) & 7, kt = (idx >> 8) & 3, layer = idx >> 10;
  const float *W = w + (layer ? MLP_OFF_W3 : MLP_OFF_W2);
  const int g = lane >> 2, t = lane & 3, n = nt * 8 + g;
  const int k0 = kt * 16 + 2 * t;
  uint32_t *F = frag + layer * MLP_FRAG_LAYER;
  uint32_t *Fl = F + MLP_FRAG_LAYER / 2;
  const int o = 2 * (idx & 1023);
  pack_split(W[k0 * 64 + n], W[(k0 + 1) * 64 + n], F[o], Fl[o]);
  pack_split(W[(k0 + 8) * 64 + n], W[(k0 + 9) * 64 + n], F[o + 1], Fl[o + 1]);
}

static size_t grad_smem() { return sizeof(GradSmem); }

int mlp_alloc(qed_ctx *c) {
  c->mlp_parts = c->num_sms;
  size_t bytes = sizeof(float) * MLP_NP * 4 + sizeof(uint32_t) * MLP_FRAG_WORDS +
                 sizeof(float) * MLP_SMEM_FLOATS + sizeof(float) * (size_t)MLP_NP * c->mlp_parts +
                 sizeof(double) * LOSS_ROWS * c->mlp_parts;
  if (cudaMalloc(&c->mlp_mem, bytes) != cudaSuccess) return QED_ERR_NOMEM;
  float *f = static_cast<float *>(c->mlp_mem);
  c->mlp_w = f;
  c->mlp_m = f + MLP_NP;
  c->mlp_v = f + 2 * MLP_NP;
  c->mlp_g = f + 3 * MLP_NP;
  c->mlp_frag = reinterpret_cast<uint32_t *>(f + 4 * MLP_NP);
  c->mlp_fw = reinterpret_cast<float *>(c->mlp_frag + MLP_FRAG_WORDS);
  c->mlp_partial = c->mlp_fw + MLP_SMEM_FLOATS;
  c->mlp_loss = reinterpret_cast<double *>(c->mlp_partial + (size_t)MLP_NP * c->mlp_parts);
  if (cudaMemset(c->mlp_mem, 0, bytes) != cudaSuccess) return QED_ERR_CUDA;
  if (cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)grad_smem()) != cudaSuccess)
    return QED_ERR_CUDA;
  c->mlp_ready = 0;
  c->mlp_step = 0;
  // records of deferred learned-sampler emissions (single-pass lepton step of
  // an FP32 context with the learned sampler): 16 bytes (48 with grid
  // fields) per emission, at most one per lepton at step start.  Two species
  // of at most max_particles each fill 2 max_particles records of 16 bytes;
  // with grid fields two thirds of that, while a one-sub-step lepton emits
  // with probability <= 0.2 (a record past the end is counted as dropped).
  c->net_cap = 0;
  if (c->cfg.sampler != QED_SAMPLER_MLP || c->cfg.append_order != QED_APPEND_ANY ||
      c->cfg.precision != QED_FP32)
    return QED_OK;
  c->net_cap = 2 * (c->cfg.max_particles > 4096 ? c->cfg.max_particles : 4096);
  if (cudaMalloc(&c->net_rec, sizeof(float4) * (size_t)c->net_cap) != cudaSuccess ||
      cudaMalloc(&c->net_n, 2 * sizeof(unsigned long long)) != cudaSuccess)
    return QED_ERR_NOMEM;
  if (cudaMemset(c->net_n, 0, 2 * sizeof(unsigned long long)) != cudaSuccess) return QED_ERR_CUDA;
  return QED_OK;
}

// The FP32 small layers in the layout inference reads (as staged by mlp_stage).
__global__ void k_mlp_pack_fw(const float *w, float *fw) {
  for (int k = threadIdx.x; k < MLP_SMEM_FLOATS; k += blockDim.x) {
    float v = 0.f;
    if (k < 128) v = w[MLP_OFF_W1 + k];
    else if (k < 192) v = w[MLP_OFF_B1 + k - 128];
    else if (k < 256) v = w[MLP_OFF_B2 + k - 192];
    else if (k < 320) v = w[MLP_OFF_B3 + k - 256];
    else if (k < 384) v = w[MLP_OFF_W4 + k - 320];
    else if (k == 384) v = w[MLP_OFF_B4];
    fw[k] = v;
  }
}

static cudaError_t pack(qed_ctx *c, cudaStream_t st) {
  k_mlp_pack<<<(2 * 4 * 8 * 32 + 255) / 256, 256, 0, st>>>(c->mlp_w, c->mlp_frag);
  k_mlp_pack_fw<<<1, 128, 0, st>>>(c->mlp_w, c->mlp_fw);
  c->launches += 2;
  return cudaGetLastError();
}

static GradArgs grad_args(qed_ctx *c) {
  GradArgs g{};
  g.w = c->mlp_w;
  g.partial = c->mlp_partial;
  g.loss_sum = c->mlp_loss;
  g.Y64 = c->Y64;
  g.gl = to_r<double>(c->gl);
  g.gk = to_r<double>(c->gk);
  return g;
}

}  // namespace qed

using namespace qed;

static int fail(cudaError_t e, const char *what) {
  if (e == cudaSuccess) return QED_OK;
  fprintf(stderr, "libqed: %s: %s\n", what, cudaGetErrorString(e));
  return QED_ERR_CUDA;
}

extern "C" int qed_mlp_load(qed_ctx *c, const float *host_w, size_t n) {
  if (!c || !host_w || n != (size_t)MLP_NP) return QED_ERR_ARG;
  cudaError_t e = cudaMemcpy(c->mlp_w, host_w, sizeof(float) * MLP_NP, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(c->mlp_m, 0, sizeof(float) * 2 * MLP_NP);
  if (e == cudaSuccess) e = pack(c, 0);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return fail(e, "qed_mlp_load");
  c->mlp_ready = 1;
  c->mlp_step = 0;
  return QED_OK;
}

extern "C" int qed_mlp_get(qed_ctx *c, float *host_w, size_t n) {
  if (!c || !host_w || n != (size_t)MLP_NP) return QED_ERR_ARG;
  return fail(cudaMemcpy(host_w, c->mlp_w, sizeof(float) * MLP_NP, cudaMemcpyDeviceToHost),
              "qed_mlp_get");
}

extern "C" int qed_mlp_grad(qed_ctx *c, const float *x, const float *t, int64_t n, float *grad,
                            double *loss, qed_stream_t stream) {
  if (!c || !x || !t || !grad || n <= 0) return QED_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  GradArgs g = grad_args(c);
  g.x = x;
  g.t = t;
  g.n = n;
  g.scale = 2.f / (float)n;
  k_mlp_grad<<<c->mlp_parts, GRAD_THREADS, grad_smem(), st>>>(g);
  AdamArgs a{};
  a.w = c->mlp_w;
  a.partial = c->mlp_partial;
  a.nparts = c->mlp_parts;
  a.grad_out = grad;
  a.apply = 0;
  k_mlp_adam<<<ADAM_BLOCKS, ADAM_THREADS, 0, st>>>(a);
  c->launches += 2;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && loss) {
    double tmp[1024];
    int np = c->mlp_parts < 1024 ? c->mlp_parts : 1024;
    e = cudaMemcpyAsync(tmp, c->mlp_loss, sizeof(double) * np, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    double s = 0.0;
    for (int p = 0; p < np; ++p) s += tmp[p];
    *loss = s / (double)n;
  }
  return fail(e, "qed_mlp_grad");
}

extern "C" int qed_mlp_train(qed_ctx *c, int64_t n_samples, float lr, uint64_t seed,
                             double *final_loss, qed_stream_t stream) {
  if (!c || n_samples <= 0 || !(lr > 0.f)) return QED_ERR_ARG;
  if (!c->mlp_ready) return QED_ERR_ARG;  // initial weights must be loaded first
  cudaStream_t st = (cudaStream_t)stream;
  const int bpc = 2;  // mini-batches per CTA per optimizer step
  const int64_t per_step = (int64_t)GRAD_B * bpc * c->mlp_parts;
  const int64_t steps = (n_samples + per_step - 1) / per_step;
  GradArgs g = grad_args(c);
  g.seed = seed;
  g.batches_per_cta = bpc;
  g.scale = 2.f / (float)per_step;
  AdamArgs a{};
  a.w = c->mlp_w;
  a.m = c->mlp_m;
  a.v = c->mlp_v;
  a.partial = c->mlp_partial;
  a.nparts = c->mlp_parts;
  a.b1 = 0.9f;
  a.b2 = 0.999f;
  a.eps = 1e-8f;
  a.apply = 1;
  const float lr_min = lr * 0.01f;
  const int64_t tail = steps < LOSS_ROWS ? steps : LOSS_ROWS;  // steps whose mean loss is returned
  for (int64_t s = 0; s < steps; ++s) {
    g.step = c->mlp_step + s;
    g.loss_sum = c->mlp_loss + (s % LOSS_ROWS) * c->mlp_parts;
    k_mlp_grad<<<c->mlp_parts, GRAD_THREADS, grad_smem(), st>>>(g);
    const int64_t k = c->mlp_step + s + 1;  // Adam step count (from 1)
    a.lr = lr_min + 0.5f * (lr - lr_min) * (1.f + cosf(3.14159265f * (float)s / (float)steps));
    a.bc1 = 1.f - powf(a.b1, (float)k);
    a.bc2 = 1.f - powf(a.b2, (float)k);
    k_mlp_adam<<<ADAM_BLOCKS, ADAM_THREADS, 0, st>>>(a);
    c->launches += 2;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(e, "qed_mlp_train");
  }
  c->mlp_step += steps;
  double *rows = (double *)malloc(sizeof(double) * LOSS_ROWS * c->mlp_parts);
  if (!rows) return QED_ERR_NOMEM;
  cudaError_t e = pack(c, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(rows, c->mlp_loss, sizeof(double) * LOSS_ROWS * c->mlp_parts, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  double loss_tail = 0.0;
  for (int64_t s = steps - tail; s < steps; ++s) {
    double sum = 0.0;
    for (int p = 0; p < c->mlp_parts; ++p) sum += rows[(s % LOSS_ROWS) * c->mlp_parts + p];
    loss_tail += sum / (double)per_step;
  }
  free(rows);
  if (final_loss && e == cudaSuccess) *final_loss = loss_tail / (double)tail;
  return fail(e, "qed_mlp_train");
}
