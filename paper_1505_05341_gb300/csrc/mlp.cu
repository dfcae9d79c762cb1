// Learned aliasing / window correction (no counterpart in the paper's equations):
// a 5 -> 64 -> 64 -> 64 -> 3 network with GELU (erf form) on the hidden layers maps
// per-shell features of a coarse-mesh measurement to the residual against a fine
// mesh, (P_l^fine - P_l^coarse) / D with D = P_0 + S/I the coarse monopole before
// shot-noise subtraction.
//
// Weights are kept in bfloat16 for the forward and backward passes (FP32 master copy
// and Adam moments); activations and every accumulation are FP32.  A CTA walks tiles of
// MLP_ROWS rows with all weights and the tile's activations in shared memory; every
// 64 x 64 product of a tile is a register-blocked FP32 product (4 x 4 per thread), the
// activations' derivatives and the weight gradients stay in registers.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <new>
#include <string>
#include <vector>

#include "ys_internal.h"

namespace ys {
namespace {

constexpr int MLP_ROWS = 64;      // rows per tile
constexpr int MLP_THREADS = 256;  // 16 x 16 threads, a 4 x 4 block of every 64 x 64 product each
constexpr int RS = 68;            // row stride of the [feature][row] and weight buffers: a multiple of 4
                                  // floats, and 17 units of 16 bytes, so that 8 rows fall on distinct banks
constexpr int H = 64;
constexpr int IN = 5, OUT = 3;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + H * IN, OFF_W2 = OFF_B1 + H, OFF_B2 = OFF_W2 + H * H;
constexpr int OFF_W3 = OFF_B2 + H, OFF_B3 = OFF_W3 + H * H, OFF_W4 = OFF_B3 + H, OFF_B4 = OFF_W4 + OUT * H;
constexpr int NP = OFF_B4 + OUT;
static_assert(NP == YS_MLP_PARAMS, "parameter count");

// GELU (erf form) of x, and its derivative.
__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_both(float x, float& grad) {
  const float cdf = 0.5f * (1.f + erff(x * 0.70710678118654752f));
  grad = cdf + x * expf(-0.5f * x * x) * 0.39894228040143268f;
  return x * cdf;
}

struct MlpSmem {
  float w1[IN * H];       // [input][hidden]
  float w2[H * RS], w3[H * RS];
  float w4[OUT * RS];
  float b[3 * H + 4];     // biases of the hidden layers, then of the output
  float x[IN * RS];
  float y[OUT * RS];      // outputs, then their deltas
  float h[3][H * RS];     // post-activations; h[2] later holds the second layer's deltas
  float d[H * RS];        // deltas of the third, then of the first layer
};

__device__ __forceinline__ void load_weights(MlpSmem& s, const __nv_bfloat16* __restrict__ w16) {
  for (int k = threadIdx.x; k < H * H; k += MLP_THREADS) {
    const int o = k / H, i = k % H;
    s.w2[o * RS + i] = __bfloat162float(w16[OFF_W2 + k]);
    s.w3[o * RS + i] = __bfloat162float(w16[OFF_W3 + k]);
  }
  for (int k = threadIdx.x; k < H * IN; k += MLP_THREADS) s.w1[(k % IN) * H + k / IN] = __bfloat162float(w16[OFF_W1 + k]);
  if (threadIdx.x < OUT * H)
    s.w4[threadIdx.x / H * RS + threadIdx.x % H] = __bfloat162float(w16[OFF_W4 + threadIdx.x]);
  if (threadIdx.x < H) {
    s.b[threadIdx.x] = __bfloat162float(w16[OFF_B1 + threadIdx.x]);
    s.b[H + threadIdx.x] = __bfloat162float(w16[OFF_B2 + threadIdx.x]);
    s.b[2 * H + threadIdx.x] = __bfloat162float(w16[OFF_B3 + threadIdx.x]);
  }
  if (threadIdx.x < OUT) s.b[3 * H + threadIdx.x] = __bfloat162float(w16[OFF_B4 + threadIdx.x]);
}

// This thread's block of a layer's outputs: hidden units a + 16 k (k < 4) of rows
// 4 c .. 4 c + 3.
struct Block {
  int a, c;
  __device__ Block() {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    a = (lane & 7) + 8 * (warp & 1);
    c = (lane >> 3) + 4 * (warp >> 1);
  }
};

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void axpy4(float (&acc)[4], float w, const float4& v) {
  acc[0] = fmaf(w, v.x, acc[0]);
  acc[1] = fmaf(w, v.y, acc[1]);
  acc[2] = fmaf(w, v.z, acc[2]);
  acc[3] = fmaf(w, v.w, acc[3]);
}

// acc[k][.] = bias[a + 16 k] + sum_i W[a + 16 k][i] in[i][4 c ..]: 8 shared loads of 16
// bytes per 64 FMAs.
__device__ __forceinline__ void dense(const float* W, const float* bias, const float* in, const Block& t,
                                      float (&acc)[4][4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[k][r] = bias[t.a + 16 * k];
#pragma unroll 2
  for (int i = 0; i < H; i += 4) {
    float4 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = ld4(in + (i + j) * RS + 4 * t.c);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 w = ld4(W + (t.a + 16 * k) * RS + i);
      axpy4(acc[k], w.x, v[0]);
      axpy4(acc[k], w.y, v[1]);
      axpy4(acc[k], w.z, v[2]);
      axpy4(acc[k], w.w, v[3]);
    }
  }
}

// acc[k][.] = sum_o W[o][a + 16 k] D[o][4 c ..]
__device__ __forceinline__ void dense_t(const float* W, const float* D, const Block& t, float (&acc)[4][4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[k][r] = 0.f;
#pragma unroll 4
  for (int o = 0; o < H; ++o) {
    const float4 v = ld4(D + o * RS + 4 * t.c);
#pragma unroll
    for (int k = 0; k < 4; ++k) axpy4(acc[k], W[o * RS + t.a + 16 * k], v);
  }
}

// g[k][l] += sum_r D[a + 16 k][r] A[c + 16 l][r] over the tile's rows
__device__ __forceinline__ void outer(const float* D, const float* A, const Block& t, float (&g)[4][4]) {
#pragma unroll 2
  for (int r = 0; r < MLP_ROWS; r += 4) {
    float4 v[4];
#pragma unroll
    for (int l = 0; l < 4; ++l) v[l] = ld4(A + (t.c + 16 * l) * RS + r);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 d = ld4(D + (t.a + 16 * k) * RS + r);
#pragma unroll
      for (int l = 0; l < 4; ++l)
        g[k][l] = fmaf(d.x, v[l].x, fmaf(d.y, v[l].y, fmaf(d.z, v[l].z, fmaf(d.w, v[l].w, g[k][l]))));
    }
  }
}

// sum_r A[r] B[r] (B == nullptr: sum_r A[r]) over the tile's rows
__device__ __forceinline__ float row_dot(const float* A, const float* B) {
  float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
  for (int r = 0; r < MLP_ROWS; r += 4) {
    const float4 a = ld4(A + r), b = B ? ld4(B + r) : make_float4(1.f, 1.f, 1.f, 1.f);
    s[0] = fmaf(a.x, b.x, s[0]);
    s[1] = fmaf(a.y, b.y, s[1]);
    s[2] = fmaf(a.z, b.z, s[2]);
    s[3] = fmaf(a.w, b.w, s[3]);
  }
  return (s[0] + s[1]) + (s[2] + s[3]);
}

// Forward pass of the tile of nr rows from r0: outputs to s.y, post-activations in s.h and,
// with GRAD, the activations' derivatives of this thread's blocks in gp.  The caller has
// synchronised after the last use of s.x, s.h and s.y.
template <bool GRAD>
__device__ __forceinline__ void forward_tile(MlpSmem& s, const float* __restrict__ X, int64_t r0, int nr,
                                             const Block& t, float (&gp)[3][4][4]) {
  for (int k = threadIdx.x; k < IN * MLP_ROWS; k += MLP_THREADS) {
    // rows past the end repeat the last row: their deltas are zero, and activations that a
    // made-up input might overflow would turn zero deltas into NaN
    const int r = k / IN, f = k % IN;
    s.x[f * RS + r] = X[(r0 + min(r, nr - 1)) * IN + f];
  }
  __syncthreads();
  float acc[4][4];
#pragma unroll
  for (int layer = 0; layer < 3; ++layer) {
    if (layer == 0) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[k][r] = s.b[t.a + 16 * k];
#pragma unroll
      for (int i = 0; i < IN; ++i) {
        const float4 v = ld4(s.x + i * RS + 4 * t.c);
#pragma unroll
        for (int k = 0; k < 4; ++k) axpy4(acc[k], s.w1[i * H + t.a + 16 * k], v);
      }
    } else {
      dense(layer == 1 ? s.w2 : s.w3, s.b + layer * H, s.h[layer - 1], t, acc);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[k][r] = GRAD ? gelu_both(acc[k][r], gp[layer][k][r]) : gelu(acc[k][r]);
      st4(s.h[layer] + (t.a + 16 * k) * RS + 4 * t.c, acc[k]);
    }
    __syncthreads();
  }
  if (threadIdx.x < OUT * MLP_ROWS) {
    const int o = threadIdx.x / MLP_ROWS, r = threadIdx.x % MLP_ROWS;
    float y = s.b[3 * H + o];
#pragma unroll 16
    for (int i = 0; i < H; ++i) y = fmaf(s.w4[o * RS + i], s.h[2][i * RS + r], y);
    s.y[o * RS + r] = y;
  }
}

__global__ void __launch_bounds__(MLP_THREADS, 2) k_mlp_forward(const __nv_bfloat16* __restrict__ w16,
                                                                const float* __restrict__ X, int64_t rows,
                                                                float* __restrict__ Y) {
  extern __shared__ __align__(16) unsigned char raw[];
  MlpSmem& s = *reinterpret_cast<MlpSmem*>(raw);
  load_weights(s, w16);
  const Block t;
  const int64_t tiles = (rows + MLP_ROWS - 1) / MLP_ROWS;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t r0 = tile * MLP_ROWS;
    const int nr = rows - r0 < MLP_ROWS ? (int)(rows - r0) : MLP_ROWS;
    float gp[3][4][4];
    forward_tile<false>(s, X, r0, nr, t, gp);
    __syncthreads();
    for (int k = threadIdx.x; k < nr * OUT; k += MLP_THREADS) Y[r0 * OUT + k] = s.y[(k % OUT) * RS + k / OUT];
  }
}

// Gradient of loss = sum (y - t)^2 / (rows_total * 3): each CTA walks its tiles with the
// weight gradients in registers (a 4 x 4 block of each 64 x 64 layer per thread) and
// writes its sums to partial[blockIdx.x] (k_mlp_reduce adds them); the CTA's summed
// squared error goes to sse_part[blockIdx.x].
//
// What bounds it: FP32 FMA issue.  158 000 rows, 8.25 GFLOP: 2.00 ms with one row per
// thread of 64-thread CTAs (137 KB of shared memory, two warps per SM) and one atomic
// per weight and CTA, against 0.28 ms now
// (41 % of the FMA rate; erff and expf of the activations are a quarter of the instructions).
__global__ void __launch_bounds__(MLP_THREADS, 2) k_mlp_backward(const __nv_bfloat16* __restrict__ w16,
                                                                 const float* __restrict__ X,
                                                                 const float* __restrict__ T, int64_t rows,
                                                                 float* __restrict__ partial,
                                                                 double* __restrict__ sse_part) {
  extern __shared__ __align__(16) unsigned char raw[];
  MlpSmem& s = *reinterpret_cast<MlpSmem*>(raw);
  load_weights(s, w16);
  const Block t;
  const int tid = threadIdx.x;
  const float scale = 2.f / (float)(rows * OUT);
  float g2[4][4] = {}, g3[4][4] = {};   // layers 2 and 3
  float g1[2] = {}, g4 = 0.f;           // layer 1: weights tid and tid + 256; layer 4: weight tid
  float gb = 0.f;                       // biases: 64 per hidden layer, then the output's
  double e2 = 0.0;
  const int64_t tiles = (rows + MLP_ROWS - 1) / MLP_ROWS;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t r0 = tile * MLP_ROWS;
    const int nr = rows - r0 < MLP_ROWS ? (int)(rows - r0) : MLP_ROWS;
    float gp[3][4][4];
    forward_tile<true>(s, X, r0, nr, t, gp);
    // this thread wrote these outputs itself; rows past the end get zero deltas
    if (tid < OUT * MLP_ROWS) {
      const int o = tid / MLP_ROWS, r = tid % MLP_ROWS;
      float d = 0.f;
      if (r < nr) {
        const float diff = s.y[o * RS + r] - T[(r0 + r) * OUT + o];
        e2 += (double)diff * diff;
        d = scale * diff;
      }
      s.y[o * RS + r] = d;
    }
    __syncthreads();
    // layer 4, and the deltas of layer 3
    if (tid < OUT * H) g4 += row_dot(s.y + tid / H * RS, s.h[2] + tid % H * RS);
    if (tid >= 3 * H && tid < 3 * H + OUT) gb += row_dot(s.y + (tid - 3 * H) * RS, nullptr);
    float acc[4][4] = {};
#pragma unroll
    for (int o = 0; o < OUT; ++o) {
      const float4 v = ld4(s.y + o * RS + 4 * t.c);
#pragma unroll
      for (int k = 0; k < 4; ++k) axpy4(acc[k], s.w4[o * RS + t.a + 16 * k], v);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[k][r] *= gp[2][k][r];
      st4(s.d + (t.a + 16 * k) * RS + 4 * t.c, acc[k]);
    }
    __syncthreads();
    // layer 3, and the deltas of layer 2 (into h[2], which nothing reads any more)
    outer(s.d, s.h[1], t, g3);
    if (tid >= 2 * H && tid < 3 * H) gb += row_dot(s.d + (tid - 2 * H) * RS, nullptr);
    dense_t(s.w3, s.d, t, acc);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[k][r] *= gp[1][k][r];
      st4(s.h[2] + (t.a + 16 * k) * RS + 4 * t.c, acc[k]);
    }
    __syncthreads();
    // layer 2, and the deltas of layer 1
    outer(s.h[2], s.h[0], t, g2);
    if (tid >= H && tid < 2 * H) gb += row_dot(s.h[2] + (tid - H) * RS, nullptr);
    dense_t(s.w2, s.h[2], t, acc);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[k][r] *= gp[0][k][r];
      st4(s.d + (t.a + 16 * k) * RS + 4 * t.c, acc[k]);
    }
    __syncthreads();
    // layer 1
    if (tid < H) gb += row_dot(s.d + tid * RS, nullptr);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int k = tid + u * MLP_THREADS;
      if (k < H * IN) g1[u] += row_dot(s.d + k / IN * RS, s.x + k % IN * RS);
    }
    __syncthreads();
  }
  float* out = partial + (size_t)blockIdx.x * NP;
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int w = (t.a + 16 * k) * H + t.c + 16 * l;
      out[OFF_W2 + w] = g2[k][l];
      out[OFF_W3 + w] = g3[k][l];
    }
  for (int u = 0; u < 2; ++u)
    if (tid + u * MLP_THREADS < H * IN) out[OFF_W1 + tid + u * MLP_THREADS] = g1[u];
  if (tid < OUT * H) out[OFF_W4 + tid] = g4;
  if (tid < 3 * H + OUT) {
    const int layer = tid / H;
    out[(layer == 0 ? OFF_B1 : layer == 1 ? OFF_B2 : layer == 2 ? OFF_B3 : OFF_B4) + tid % H] = gb;
  }
  // squared error
  __shared__ double red[MLP_THREADS / 32];
  for (int o = 16; o > 0; o >>= 1) e2 += __shfl_xor_sync(0xffffffffu, e2, o);
  if ((tid & 31) == 0) red[tid >> 5] = e2;
  __syncthreads();
  if (tid == 0) {
    double v = 0;
    for (int k = 0; k < MLP_THREADS / 32; ++k) v += red[k];
    sse_part[blockIdx.x] = v;
  }
}

// grad[k] (and copy[k]) = sum over the n partial gradients, in one fixed order: 32
// parameters per CTA, 8 threads each.  The last CTA adds the squared errors.
__global__ void __launch_bounds__(256) k_mlp_reduce(const float* __restrict__ partial,
                                                    const double* __restrict__ sse_part, int n,
                                                    float* __restrict__ grad, float* __restrict__ copy,
                                                    double* __restrict__ sse, double* __restrict__ sse_copy) {
  if (blockIdx.x == gridDim.x - 1) {
    if (threadIdx.x < 32) {
      double v = 0.0;
      for (int q = threadIdx.x; q < n; q += 32) v += sse_part[q];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (threadIdx.x == 0) {
        *sse = v;
        if (sse_copy) *sse_copy = v;
      }
    }
    return;
  }
  __shared__ float part[8][32];
  const int p = threadIdx.x & 31, slice = threadIdx.x >> 5, k = blockIdx.x * 32 + p;
  float v = 0.f;
  if (k < NP) {
#pragma unroll 8
    for (int q = slice; q < n; q += 8) v += partial[(size_t)q * NP + k];
  }
  part[slice][p] = v;
  __syncthreads();
  if (slice == 0 && k < NP) {
    for (int q = 1; q < 8; ++q) v += part[q][p];
    grad[k] = v;
    if (copy) copy[k] = v;
  }
}

// Adam on the FP32 master weights, refresh of the bfloat16 copy.
__global__ void k_mlp_adam(float* __restrict__ w, __nv_bfloat16* __restrict__ w16, const float* __restrict__ grad,
                           float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2, float eps,
                           float c1, float c2) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= NP) return;
  const float g = grad[k];
  const float mk = b1 * m[k] + (1.f - b1) * g;
  const float vk = b2 * v[k] + (1.f - b2) * g * g;
  m[k] = mk;
  v[k] = vk;
  const float wk = w[k] - lr * (mk / c1) / (sqrtf(vk / c2) + eps);
  w[k] = wk;
  w16[k] = __float2bfloat16_rn(wk);
}

// Per-shell features of result rows (layout of ys_measure_multipoles_async) and,
// when fine rows are given, the targets.  A shell enters when it has modes, finite
// multipoles and D > 0.  Rows are appended in an order set by atomics; src[] maps
// each row back to (catalogue * n_bins + shell).
__global__ void k_mlp_features(const double* __restrict__ rows, const double* __restrict__ fine, int n_cat,
                               int64_t stride, int n_bins, double k_nyq, float* __restrict__ X,
                               float* __restrict__ T, int* __restrict__ src, int* __restrict__ count) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_cat * n_bins) return;
  const int c = idx / n_bins, b = idx % n_bins;
  const double* row = rows + (size_t)c * stride;
  const double nm = row[n_bins + b];
  const double p0 = row[2 * n_bins + b], p2 = row[3 * n_bins + b], p4 = row[4 * n_bins + b];
  const double psn = row[5 * n_bins + 2];
  const double D = p0 + psn;
  if (!(nm > 0) || !isfinite(p0) || !isfinite(p2) || !isfinite(p4) || !(psn > 0) || !(D > 0)) return;
  double t0 = 0, t2 = 0, t4 = 0;
  if (fine) {
    const double* fr = fine + (size_t)c * stride;
    const double f0 = fr[2 * n_bins + b], f2 = fr[3 * n_bins + b], f4 = fr[4 * n_bins + b];
    if (!isfinite(f0) || !isfinite(f2) || !isfinite(f4)) return;
    t0 = (f0 - p0) / D;
    t2 = (f2 - p2) / D;
    t4 = (f4 - p4) / D;
  }
  const int slot = atomicAdd(count, 1);
  float* x = X + (size_t)slot * IN;
  x[0] = (float)(row[b] / k_nyq);
  x[1] = (float)log(D / psn);
  x[2] = (float)(p2 / D);
  x[3] = (float)(p4 / D);
  x[4] = (float)(psn / D);
  if (T) {
    T[(size_t)slot * OUT + 0] = (float)t0;
    T[(size_t)slot * OUT + 1] = (float)t2;
    T[(size_t)slot * OUT + 2] = (float)t4;
  }
  src[slot] = idx;
}

// P_l <- P_l + D y_l for each featured shell (in place on out, which already holds
// a copy of rows).
__global__ void k_mlp_apply(const double* __restrict__ rows, int64_t stride, int n_bins, const float* __restrict__ Y,
                            const int* __restrict__ src, const int* __restrict__ count, double* __restrict__ out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= *count) return;
  const int idx = src[k];
  const int c = idx / n_bins, b = idx % n_bins;
  const double* row = rows + (size_t)c * stride;
  const double D = row[2 * n_bins + b] + row[5 * n_bins + 2];
  for (int l = 0; l < OUT; ++l)
    out[(size_t)c * stride + (2 + l) * n_bins + b] = row[(2 + l) * n_bins + b] + D * (double)Y[(size_t)k * OUT + l];
}

}  // namespace
}  // namespace ys

struct ys_mlp_s {
  unsigned char* slab = nullptr;  // one allocation; everything down to fcount but the features lies in it
  float* w = nullptr;            // FP32 master weights
  __nv_bfloat16* w16 = nullptr;  // bfloat16 copy used by the kernels
  float* grad = nullptr;
  float* m = nullptr;
  float* v = nullptr;
  double* sse = nullptr;
  float* partial = nullptr;      // [grid_max][NP] gradients of the CTAs
  double* sse_part = nullptr;    // [grid_max]
  int grid_max = 0;              // CTAs that are resident at once
  float* fx = nullptr;           // feature scratch for ys_mlp_correct
  float* fy = nullptr;
  int* fsrc = nullptr;
  int* fcount = nullptr;
  int64_t fcap = 0;
  int64_t t = 0;                 // Adam steps taken
};

namespace {

size_t smem_bytes() { return sizeof(ys::MlpSmem); }

ys_status fail(cudaError_t e) {
  ys::g_last_cuda_error = cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? YS_ERR_OOM : YS_ERR_CUDA;
}

void free_mlp(ys_mlp* m) {
  for (void* p : {(void*)m->slab, (void*)m->fx, (void*)m->fy, (void*)m->fsrc})
    if (p) cudaFree(p);
  delete m;
}

cudaError_t set_attrs() {
  cudaError_t e = cudaFuncSetAttribute(ys::k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes());
  if (!e) e = cudaFuncSetAttribute(ys::k_mlp_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes());
  return e;
}

// CTAs of the tile kernels: the tiles shared evenly among at most grid_max.
unsigned grid_for(const ys_mlp* m, int64_t rows) {
  const int64_t tiles = (rows + ys::MLP_ROWS - 1) / ys::MLP_ROWS;
  const int64_t per = (tiles + m->grid_max - 1) / m->grid_max;
  return (unsigned)((tiles + per - 1) / per);
}

}  // namespace

extern "C" {

ys_status ys_mlp_create(const float* h_params, ys_mlp** out) {
  if (!h_params || !out) return YS_ERR_ARG;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
    cudaGetLastError();
    ys::g_last_cuda_error = "no CUDA device";
    return YS_ERR_CUDA;
  }
  ys_mlp* m = new (std::nothrow) ys_mlp;
  if (!m) return YS_ERR_OOM;
  cudaError_t e;
  const size_t n = ys::NP;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) {
    free_mlp(m);
    return fail(e);
  }
  m->grid_max = 2 * sms;
  // one allocation for everything whose size is known
  size_t bytes = 0;
  auto part = [&](size_t size) {
    const size_t at = bytes;
    bytes += (size + 255) & ~size_t(255);
    return at;
  };
  const size_t at_w = part(n * 4), at_w16 = part(n * 2), at_grad = part(n * 4), at_m = part(n * 4), at_v = part(n * 4),
               at_sse = part(8), at_count = part(4), at_ssep = part((size_t)m->grid_max * 8),
               at_partial = part((size_t)m->grid_max * n * 4);
  if ((e = cudaMalloc(&m->slab, bytes))) {
    free_mlp(m);
    return fail(e);
  }
  m->w = reinterpret_cast<float*>(m->slab + at_w);
  m->w16 = reinterpret_cast<__nv_bfloat16*>(m->slab + at_w16);
  m->grad = reinterpret_cast<float*>(m->slab + at_grad);
  m->m = reinterpret_cast<float*>(m->slab + at_m);
  m->v = reinterpret_cast<float*>(m->slab + at_v);
  m->sse = reinterpret_cast<double*>(m->slab + at_sse);
  m->fcount = reinterpret_cast<int*>(m->slab + at_count);
  m->sse_part = reinterpret_cast<double*>(m->slab + at_ssep);
  m->partial = reinterpret_cast<float*>(m->slab + at_partial);
  std::vector<__nv_bfloat16> h16(n);
  for (size_t k = 0; k < n; ++k) h16[k] = __float2bfloat16_rn(h_params[k]);
  if ((e = cudaMemcpy(m->w, h_params, n * 4, cudaMemcpyHostToDevice)) ||
      (e = cudaMemcpy(m->w16, h16.data(), n * 2, cudaMemcpyHostToDevice)) || (e = cudaMemset(m->grad, 0, n * 4)) ||
      (e = cudaMemset(m->m, 0, n * 4)) || (e = cudaMemset(m->v, 0, n * 4)) || (e = set_attrs())) {
    free_mlp(m);
    return fail(e);
  }
  *out = m;
  return YS_OK;
}

ys_status ys_mlp_get_state(ys_mlp* m, float* h_params, float* h_m, float* h_v, int64_t* h_step) {
  if (!m) return YS_ERR_ARG;
  cudaError_t e = cudaDeviceSynchronize();
  if (!e && h_params) e = cudaMemcpy(h_params, m->w, ys::NP * 4, cudaMemcpyDeviceToHost);
  if (!e && h_m) e = cudaMemcpy(h_m, m->m, ys::NP * 4, cudaMemcpyDeviceToHost);
  if (!e && h_v) e = cudaMemcpy(h_v, m->v, ys::NP * 4, cudaMemcpyDeviceToHost);
  if (e) return fail(e);
  if (h_step) *h_step = m->t;
  return YS_OK;
}

ys_status ys_mlp_set_state(ys_mlp* m, const float* h_params, const float* h_m, const float* h_v, int64_t step) {
  if (!m || !h_params || step < 0) return YS_ERR_ARG;
  const size_t n = ys::NP;
  std::vector<__nv_bfloat16> h16(n);
  for (size_t k = 0; k < n; ++k) h16[k] = __float2bfloat16_rn(h_params[k]);
  cudaError_t e = cudaDeviceSynchronize();
  if (!e) e = cudaMemcpy(m->w, h_params, n * 4, cudaMemcpyHostToDevice);
  if (!e) e = cudaMemcpy(m->w16, h16.data(), n * 2, cudaMemcpyHostToDevice);
  if (!e) e = h_m ? cudaMemcpy(m->m, h_m, n * 4, cudaMemcpyHostToDevice) : cudaMemset(m->m, 0, n * 4);
  if (!e) e = h_v ? cudaMemcpy(m->v, h_v, n * 4, cudaMemcpyHostToDevice) : cudaMemset(m->v, 0, n * 4);
  if (e) return fail(e);
  m->t = step;
  return YS_OK;
}

ys_status ys_mlp_forward(ys_mlp* m, const float* d_x, int64_t rows, float* d_y, void* stream) {
  if (!m || rows < 0 || (rows > 0 && (!d_x || !d_y))) return YS_ERR_ARG;
  if (rows == 0) return YS_OK;
  ys::k_mlp_forward<<<grid_for(m, rows), ys::MLP_THREADS, smem_bytes(), static_cast<cudaStream_t>(stream)>>>(
      m->w16, d_x, rows, d_y);
  cudaError_t e = cudaGetLastError();
  return e ? fail(e) : YS_OK;
}

ys_status ys_mlp_gradient(ys_mlp* m, const float* d_x, const float* d_t, int64_t rows, float* d_grad,
                          double* d_loss, void* stream) {
  if (!m || rows <= 0 || !d_x || !d_t) return YS_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e;
  const unsigned grid = grid_for(m, rows);
  ys::k_mlp_backward<<<grid, ys::MLP_THREADS, smem_bytes(), st>>>(m->w16, d_x, d_t, rows, m->partial, m->sse_part);
  if ((e = cudaGetLastError())) return fail(e);
  ys::k_mlp_reduce<<<(ys::NP + 31) / 32 + 1, 256, 0, st>>>(m->partial, m->sse_part, (int)grid, m->grad, d_grad, m->sse,
                                                           d_loss);
  if ((e = cudaGetLastError())) return fail(e);
  return YS_OK;
}

ys_status ys_mlp_train_step(ys_mlp* m, const float* d_x, const float* d_t, int64_t rows, float lr, double* d_sse,
                            void* stream) {
  ys_status s = ys_mlp_gradient(m, d_x, d_t, rows, nullptr, d_sse, stream);
  if (s != YS_OK) return s;
  m->t += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)m->t), c2 = 1.f - powf(b2, (float)m->t);
  ys::k_mlp_adam<<<(ys::NP + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(m->w, m->w16, m->grad, m->m,
                                                                                       m->v, lr, b1, b2, 1e-8f, c1, c2);
  cudaError_t e = cudaGetLastError();
  return e ? fail(e) : YS_OK;
}

ys_status ys_mlp_features(const double* d_rows, const double* d_fine_rows, int32_t n_cat, int64_t stride,
                          int32_t n_bins, double k_nyq, float* d_x, float* d_t, int32_t* d_src, int32_t* d_count,
                          void* stream) {
  if (!d_rows || n_cat <= 0 || n_bins <= 0 || stride < 5 * (int64_t)n_bins + 5 || !(k_nyq > 0) || !d_x || !d_src ||
      !d_count || (d_fine_rows && !d_t))
    return YS_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemsetAsync(d_count, 0, 4, st);
  if (e) return fail(e);
  const int total = n_cat * n_bins;
  ys::k_mlp_features<<<(total + 255) / 256, 256, 0, st>>>(d_rows, d_fine_rows, n_cat, stride, n_bins, k_nyq, d_x,
                                                          d_fine_rows ? d_t : nullptr, d_src, d_count);
  e = cudaGetLastError();
  return e ? fail(e) : YS_OK;
}

ys_status ys_mlp_correct(ys_mlp* m, const double* d_rows, int32_t n_cat, int64_t stride, int32_t n_bins,
                         double k_nyq, double* d_out, void* stream) {
  if (!m || !d_rows || !d_out || n_cat <= 0 || n_bins <= 0 || stride < 5 * (int64_t)n_bins + 5) return YS_ERR_ARG;
  if (d_out != d_rows && d_out < d_rows + (size_t)n_cat * stride && d_rows < d_out + (size_t)n_cat * stride)
    return YS_ERR_ARG;  // partial overlap
  const int64_t need = (int64_t)n_cat * n_bins;
  cudaError_t e;
  if (need > m->fcap) {
    if (m->fx) cudaFree(m->fx);
    if (m->fy) cudaFree(m->fy);
    if (m->fsrc) cudaFree(m->fsrc);
    m->fx = nullptr;
    m->fy = nullptr;
    m->fsrc = nullptr;
    if ((e = cudaMalloc(&m->fx, need * 5 * 4)) || (e = cudaMalloc(&m->fy, need * 3 * 4)) ||
        (e = cudaMalloc(&m->fsrc, need * 4)))
      return fail(e);
    m->fcap = need;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  ys_status s = ys_mlp_features(d_rows, nullptr, n_cat, stride, n_bins, k_nyq, m->fx, nullptr, m->fsrc, m->fcount,
                                stream);
  if (s != YS_OK) return s;
  // all n_cat * n_bins slots are evaluated; slots past *count hold no row and are not used
  s = ys_mlp_forward(m, m->fx, need, m->fy, stream);
  if (s != YS_OK) return s;
  if (d_out != d_rows &&
      (e = cudaMemcpyAsync(d_out, d_rows, sizeof(double) * (size_t)(n_cat * stride), cudaMemcpyDeviceToDevice, st)))
    return fail(e);
  ys::k_mlp_apply<<<(unsigned)((need + 255) / 256), 256, 0, st>>>(d_rows, stride, n_bins, m->fy, m->fsrc, m->fcount,
                                                                 d_out);
  e = cudaGetLastError();
  return e ? fail(e) : YS_OK;
}

ys_status ys_mlp_destroy(ys_mlp* m) {
  if (!m) return YS_OK;
  cudaDeviceSynchronize();
  free_mlp(m);
  return YS_OK;
}

}  // extern "C"
