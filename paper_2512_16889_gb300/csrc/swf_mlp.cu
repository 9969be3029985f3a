// Surrogate network for scans of the pair probability: a multilayer perceptron
//   (E, omega, lambda, p_x, p_y, s) -> 4 x [256, GELU] -> (mu, log sigma^2)
// trained on solver outputs.  BF16 operands on the tensor cores with FP32 accumulation
// (mma.sync m16n8k16), FP32 master weights, Adam, Gaussian negative log-likelihood
//   L = mean_b [ (y_b - mu_b)^2 exp(-l_b) + l_b ] / 2.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "swf_internal.h"

namespace swf {
namespace mlp {

constexpr int NL = 5;                                // layers
constexpr int DIN[NL] = {6, 256, 256, 256, 256};
constexpr int DOUT[NL] = {256, 256, 256, 256, 2};

__host__ __device__ constexpr int n_params() {
  int n = 0;
  for (int l = 0; l < NL; ++l) n += DIN[l] * DOUT[l] + DOUT[l];
  return n;
}

// The normal distribution function Phi(x) = (1 + erf(x / sqrt 2)) / 2 and the density phi(x),
// with erf from Abramowitz and Stegun's formula 7.1.26 (Hastings' rational approximation):
// erf(z) = 1 - (a1 t + a2 t^2 + a3 t^3 + a4 t^4 + a5 t^5) e^{-z^2}, t = 1/(1 + p z), z >= 0,
// |error| <= 1.5e-7.  One reciprocal, one exponential and five fused multiply-adds; the GELU
// values it gives are rounded to bfloat16 (8 significand bits) before use, far coarser than it.
__device__ __forceinline__ void normal_cdf_pdf(float x, float& cdf, float& pdf) {
  const float z = fabsf(x) * 0.70710678118654752f;
  const float t = __fdividef(1.0f, fmaf(0.3275911f, z, 1.0f));
  const float poly = t * fmaf(t, fmaf(t, fmaf(t, fmaf(t, 1.061405429f, -1.453152027f), 1.421413741f),
                                      -0.284496736f), 0.254829592f);
  const float e = __expf(-0.5f * x * x);  // e^{-z^2}
  const float tail = 0.5f * poly * e;     // (1 - erf(z)) / 2
  cdf = x >= 0.0f ? 1.0f - tail : tail;
  pdf = 0.39894228040143268f * e;
}
__device__ __forceinline__ float gelu(float x) {
  float c, d;
  normal_cdf_pdf(x, c, d);
  return x * c;
}
__device__ __forceinline__ float gelu_grad(float x) {
  float c, d;
  normal_cdf_pdf(x, c, d);
  return fmaf(x, d, c);
}

// The activation and its derivative elementwise (the network's own GELU, for checks).
__global__ void k_gelu_eval(const float* __restrict__ x, int n, float* __restrict__ g, float* __restrict__ dg) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    g[i] = gelu(x[i]);
    dg[i] = gelu_grad(x[i]);
  }
}

// ---------------------------------------------------------------- training
// One step is three launches: k_train_rows takes 16 rows of the batch through the network and back
// (forward, dL/dz of every layer), k_train_dw forms the gradients and the loss, k_train_update applies
// Adam.  Operands are BF16 on the tensor cores (mma.sync m16n8k16, FP32
// accumulation in ascending k): a batch of 256 is 16 row blocks of 256 x 256 layers, far below what a
// tcgen05 tile needs to fill (M = 128), and what bounds it is the chain of layers and the launches, not
// the tensor rate.  A batch of 256 takes 33 us a step and one of 4096 101 us; as 25 kernels on 64 x 64
// tiles, each waiting on two-byte loads of its operands, they took 480 and 3170 us.  Every sum runs in
// the order it had there (ascending k and rows), and the expressions that a compiler may contract in more
// than one way (residual, loss, Adam's moments) have every rounding fixed below, so that the loss and its
// gradient share one r^2 w and no regrouping of the kernels changes a bit: one unit in the last place of
// an output bias grew to 1.6e-4 of the loss in eight steps.
namespace tr {

constexpr int ROWS = 16;         // rows per block of k_train_rows: one m16 tile
constexpr int THREADS = 512;     // 16 warps, warp w owns columns 16 w .. 16 w + 15 of every hidden layer
constexpr int AST = 264;         // bf16 row stride of an operand tile (528 bytes: odd in 16-byte units)
constexpr int TILE = 32;         // weight-gradient tile
constexpr int CHUNK = 64;        // rows per stage of its ring

// First weight of layer l in the parameter array, first bias after its weights.
__host__ __device__ constexpr int nweights(int l) { return l == 0 ? 6 * 256 : l < 4 ? 256 * 256 : 2 * 256; }
__host__ __device__ constexpr int woff(int l) { return l == 0 ? 0 : 7 * 256 + (l - 1) * 257 * 256; }
__host__ __device__ constexpr int boff(int l) { return woff(l) + nweights(l); }

// Weights of layers 1-3 in the order in which a lane of mma.m16n8k16 holds its B operand, for the
// forward pass (column n, reduction k) and the backward pass (column k, reduction n): per column tile
// of 8 and pair of k16 steps, 32 lanes of 8 bf16 (16 bytes).  col, red: column and reduction index.
__host__ __device__ __forceinline__ int frag_index(int col, int red) {
  const int nt = col >> 3, g = col & 7, ks = red >> 4, r = red & 15;
  const int t = (r & 7) >> 1, j = (r & 1) + ((r >> 3) << 1);
  return ((nt * 8 + (ks >> 1)) * 32 + g * 4 + t) * 8 + (ks & 1) * 4 + j;
}

__device__ __forceinline__ void mma(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm(uint32_t* r, const __nv_bfloat16* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void ldsm_t(uint32_t* r, const __nv_bfloat16* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// r = (y - y0) ys - mu, with the product and the subtraction in one rounding
__device__ __forceinline__ float residual(float y, float y0, float ys, float mu) {
  return __fmaf_rn(__fsub_rn(y, y0), ys, -mu);
}
// r^2 w, the product that the loss (r^2 w + l) / 2 and its derivative (1 - r^2 w) / 2 share
__device__ __forceinline__ float scaled_square(float r, float w) { return __fmul_rn(__fmul_rn(r, r), w); }
// b m + (1 - b) g and b v + (1 - b) g^2 of Adam: the new term in one rounding with the sum
__device__ __forceinline__ float moment1(float b, float m, float g) {
  return __fmaf_rn(__fsub_rn(1.0f, b), g, __fmul_rn(b, m));
}
__device__ __forceinline__ float moment2(float b, float v, float g) {
  return __fmaf_rn(__fmul_rn(__fsub_rn(1.0f, b), g), g, __fmul_rn(b, v));
}

// What the three kernels hand on, rows padded to ROWS with zero dL/dz.
struct Bufs {
  __nv_bfloat16* act[4];  // [rows][256]: outputs of hidden layers 0..3 (inputs of layers 1..4)
  __nv_bfloat16* dz[4];   // [rows][256]: dL/dz of hidden layers 0..3
  __nv_bfloat16* xin;     // [rows][8]: standardised inputs
  __nv_bfloat16* dzo;     // [rows][2]: dL/dz of the output layer
  float* dz32[4];         // the same before rounding (bias gradients)
  float* dzo32;
  float* zo;              // [rows][2]: the network's outputs
};

// B operands of one 256 x 256 layer for this warp's two column tiles: 16 loads of 16 bytes per lane,
// issued before the barrier that the previous layer's results need.
__device__ __forceinline__ void load_frags(uint4* b, const __nv_bfloat16* __restrict__ pack, int warp, int lane) {
  const uint4* p = reinterpret_cast<const uint4*>(pack) + (size_t)(2 * warp) * 8 * 32 + lane;
#pragma unroll
  for (int i = 0; i < 16; ++i) b[i] = __ldg(p + i * 32);
}
// acc (two column tiles) = A (16 rows in shared memory) times the loaded operands
__device__ __forceinline__ void layer_mma(float acc[2][4], const __nv_bfloat16* sa, const uint4* b, int lane) {
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[j][r] = 0.f;
  const __nv_bfloat16* p = sa + (lane & 15) * AST + (lane >> 4) * 8;
#pragma unroll
  for (int ks = 0; ks < 16; ++ks) {
    uint32_t a[4];
    ldsm(a, p + ks * 16);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint4 w = b[j * 8 + (ks >> 1)];
      if (ks & 1) mma(acc[j], a, w.z, w.w);
      else mma(acc[j], a, w.x, w.y);
    }
  }
}

// 16 rows: forward, Gaussian NLL on the standardised target y' = (y - y0) ys (loss: mean over the batch),
// backward.  Pre-activations stay in registers: the thread that holds columns 16 warp + 8 j + 2 t (+ 1)
// of rows g, g + 8 in the forward pass holds the same elements of dL/dz in the backward pass.
__global__ void __launch_bounds__(THREADS, 1)
k_train_rows(const float* __restrict__ x, const float* __restrict__ y, int B, const __nv_bfloat16* __restrict__ wbf,
             const __nv_bfloat16* __restrict__ fpack, const __nv_bfloat16* __restrict__ bpack,
             const float* __restrict__ params, const float* __restrict__ shift, const float* __restrict__ scale, float y0,
             float ys, Bufs W) {
  __shared__ __align__(16) __nv_bfloat16 sA[2][ROWS * AST];
  __shared__ uint32_t sDz[ROWS];   // (dmu, dl) of a row in bf16
  __shared__ float sBias[4][256];
  __shared__ uint32_t sX[ROWS][4];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int row0 = blockIdx.x * ROWS;
  const int col = 16 * warp + 2 * t;  // first column of tile j: col + 8 j
  uint4 b[16];
  load_frags(b, fpack, warp, lane);
  for (int i = tid; i < 4 * 256; i += THREADS) sBias[i >> 8][i & 255] = params[boff(i >> 8) + (i & 255)];
  if (tid < ROWS * 4) {  // standardised inputs x' = (x - shift) scale, features 6 and 7 zero
    const int r = tid >> 2, f = 2 * (tid & 3);
    float v[2] = {0.f, 0.f};
    if (row0 + r < B && f < 6)
      for (int u = 0; u < 2; ++u) v[u] = (x[(size_t)(row0 + r) * 6 + f + u] - shift[f + u]) * scale[f + u];
    const uint32_t w = pack2(v[0], v[1]);
    sX[r][tid & 3] = w;
    reinterpret_cast<uint32_t*>(W.xin)[(size_t)(row0 + r) * 4 + (tid & 3)] = w;
  }
  __syncthreads();
  float z[4][2][4];
  // hidden layer l's outputs from its pre-activations: to the next operand tile and to memory
  auto activate = [&](int l, int buf) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c = col + 8 * j;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        z[l][j][2 * h] += sBias[l][c];
        z[l][j][2 * h + 1] += sBias[l][c + 1];
        const uint32_t w = pack2(gelu(z[l][j][2 * h]), gelu(z[l][j][2 * h + 1]));
        *reinterpret_cast<uint32_t*>(&sA[buf][(g + 8 * h) * AST + c]) = w;
        *reinterpret_cast<uint32_t*>(W.act[l] + (size_t)(row0 + g + 8 * h) * 256 + c) = w;
      }
    }
  };
  {  // layer 0: one k16 step, features beyond 6 are zero
    uint32_t a[4] = {sX[g][t], sX[g + 8][t], 0u, 0u};
#pragma unroll
    for (int j = 0; j < 2; ++j) {
#pragma unroll
      for (int r = 0; r < 4; ++r) z[0][j][r] = 0.f;
      const int n = 16 * warp + 8 * j + g;
      const uint32_t b0 = t < 3 ? *reinterpret_cast<const uint32_t*>(wbf + woff(0) + n * 6 + 2 * t) : 0u;
      mma(z[0][j], a, b0, 0u);
    }
    activate(0, 0);
  }
  __syncthreads();
#pragma unroll
  for (int l = 1; l < 4; ++l) {
    layer_mma(z[l], sA[(l - 1) & 1], b, lane);
    if (l < 3) load_frags(b, fpack + (size_t)l * 65536, warp, lane);
    activate(l, l & 1);
    __syncthreads();
  }
  load_frags(b, bpack + (size_t)2 * 65536, warp, lane);  // layer 3's, for the backward pass
  if (warp == 0) {  // output layer and loss
    float o[4] = {0.f, 0.f, 0.f, 0.f};
    const __nv_bfloat16* p = sA[1] + (lane & 15) * AST + (lane >> 4) * 8;
    const uint32_t* w4 = reinterpret_cast<const uint32_t*>(wbf + woff(4) + g * 256);
#pragma unroll
    for (int ks = 0; ks < 16; ++ks) {
      uint32_t a[4];
      ldsm(a, p + ks * 16);
      mma(o, a, g < 2 ? w4[ks * 8 + t] : 0u, g < 2 ? w4[ks * 8 + t + 4] : 0u);
    }
    if (t == 0) {
      const float bm = params[boff(4)], bl = params[boff(4) + 1];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int b = row0 + g + 8 * h;
        float dmu = 0.f, dl = 0.f;
        if (b < B) {
          const float mu = o[2 * h] + bm, l = o[2 * h + 1] + bl;
          const float r = residual(y[b], y0, ys, mu), w = __expf(-l);
          dmu = -r * w / B;
          dl = 0.5f * __fsub_rn(1.0f, scaled_square(r, w)) / B;
          reinterpret_cast<float2*>(W.zo)[b] = make_float2(mu, l);
        }
        reinterpret_cast<float2*>(W.dzo32)[b] = make_float2(dmu, dl);
        const uint32_t d = pack2(dmu, dl);
        sDz[g + 8 * h] = d;
        reinterpret_cast<uint32_t*>(W.dzo)[b] = d;
      }
    }
  }
  __syncthreads();
  // dL/dz of hidden layer l from dL/d(its output) in d: to the next operand tile and to memory
  auto descend = [&](int l, float d[2][4], int buf) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c = col + 8 * j;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float d0 = d[j][2 * h] * gelu_grad(z[l][j][2 * h]), d1 = d[j][2 * h + 1] * gelu_grad(z[l][j][2 * h + 1]);
        const uint32_t w = pack2(d0, d1);
        const size_t e = (size_t)(row0 + g + 8 * h) * 256 + c;
        if (l > 0) *reinterpret_cast<uint32_t*>(&sA[buf][(g + 8 * h) * AST + c]) = w;
        *reinterpret_cast<uint32_t*>(W.dz[l] + e) = w;
        *reinterpret_cast<float2*>(W.dz32[l] + e) = make_float2(d0, d1);
      }
    }
  };
  float d[2][4];
  {  // through the output layer: two reduction terms, one k16 step
    uint32_t a[4] = {t == 0 ? sDz[g] : 0u, t == 0 ? sDz[g + 8] : 0u, 0u, 0u};
#pragma unroll
    for (int j = 0; j < 2; ++j) {
#pragma unroll
      for (int r = 0; r < 4; ++r) d[j][r] = 0.f;
      const int k = 16 * warp + 8 * j + g;
      uint32_t b0 = 0u;
      if (t == 0) {
        const __nv_bfloat162 v = __halves2bfloat162(wbf[woff(4) + k], wbf[woff(4) + 256 + k]);
        b0 = *reinterpret_cast<const uint32_t*>(&v);
      }
      mma(d[j], a, b0, 0u);
    }
    descend(3, d, 0);
  }
  __syncthreads();
#pragma unroll
  for (int l = 3; l > 0; --l) {
    layer_mma(d, sA[(3 - l) & 1], b, lane);
    if (l > 1) load_frags(b, bpack + (size_t)(l - 2) * 65536, warp, lane);
    descend(l - 1, d, (4 - l) & 1);
    if (l > 1) __syncthreads();
  }
}

// Gradients.  Blocks 0 .. 207: weight gradients dW(n, k) = sum_b dZ(b, n) X(b, k), one 32 x 32 tile of
// one layer each (64 tiles of layers 1-3, 8 of layers 0 and 4), accumulated over the whole batch in
// ascending rows; both operands come row by row through a ring of kStages chunks in shared memory
// (asynchronous copies) and are transposed by ldmatrix.  Blocks 208 .. 211: bias gradients of the hidden
// layers, one column per thread, in ascending rows; block 212: the loss and the output layer's biases.
constexpr int kTiles = 3 * 64 + 2 * 8;
constexpr int kStages = 4;

__device__ __forceinline__ void cp_async(void* dst, const void* src, int bytes, bool valid) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if (bytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}

__global__ void __launch_bounds__(128) k_train_dw(const float* __restrict__ y, int B, int rows, float y0, float ys, Bufs W,
                                                  float* __restrict__ grads, float* loss, float* loss_user) {
  __shared__ __align__(16) __nv_bfloat16 sD[kStages][CHUNK][TILE + 8], sX[kStages][CHUNK][TILE + 8];
  const int tid = threadIdx.x, blk = blockIdx.x;
  if (blk >= kTiles + 8) {  // the loss: 128 threads as the 256 strided partial sums, then halves
    __shared__ float red[256];
    for (int h = 0; h < 2; ++h) {
      float acc = 0.f;
      for (int b = tid + 128 * h; b < B; b += 256) {
        const float mu = W.zo[2 * b], l = W.zo[2 * b + 1];
        const float r = residual(y[b], y0, ys, mu), w = __expf(-l);
        acc = __fadd_rn(acc, 0.5f * __fadd_rn(scaled_square(r, w), l));
      }
      red[tid + 128 * h] = acc;
    }
    __syncthreads();
    for (int q = 128; q > 0; q >>= 1) {
      if (tid < q) red[tid] += red[tid + q];
      __syncthreads();
    }
    if (tid == 0) {
      *loss = red[0] / B;
      if (loss_user) *loss_user = red[0] / B;
    }
    if (tid < 2) {
      float s = 0.f;
#pragma unroll 32
      for (int b = 0; b < B; ++b) s += W.dzo32[2 * b + tid];
      grads[boff(4) + tid] = s;
    }
    return;
  }
  if (blk >= kTiles) {
    const int col = (blk - kTiles) * 128 + tid, l = col >> 8, n = col & 255;
    const float* d = W.dz32[l] + n;
    float s = 0.f;
#pragma unroll 32
    for (int b = 0; b < B; ++b) s += d[(size_t)b * 256];
    grads[boff(l) + n] = s;
    return;
  }
  // layer, tile origin (n0, k0)
  const int l = blk < 192 ? 1 + blk / 64 : (blk < 200 ? 0 : 4);
  const int n0 = blk < 192 ? (blk % 64 / 8) * TILE : (l == 0 ? (blk - 192) * TILE : 0);
  const int k0 = blk < 192 ? (blk % 8) * TILE : (l == 0 ? 0 : (blk - 200) * TILE);
  const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int wm = (warp >> 1) * 16, wn = (warp & 1) * 16;
  for (int i = tid; i < kStages * CHUNK * (TILE + 8) / 2; i += 128) {  // the columns that layers 0 and 4 lack
    reinterpret_cast<uint32_t*>(sD)[i] = 0u;
    reinterpret_cast<uint32_t*>(sX)[i] = 0u;
  }
  __syncthreads();
  const int nch = (rows + CHUNK - 1) / CHUNK;
  auto fetch = [&](int ch) {
    if (ch < nch) {
      const int st = ch % kStages, b0 = ch * CHUNK;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int e = tid + 128 * i, r = e >> 2, c = (e & 3) * 8;
        const bool in = b0 + r < rows;
        const size_t row = in ? b0 + r : 0;
        if (l < 4) cp_async(&sD[st][r][c], W.dz[l] + row * 256 + n0 + c, 16, in);
        if (l > 0) cp_async(&sX[st][r][c], W.act[l - 1] + row * 256 + k0 + c, 16, in);
      }
      if (tid < CHUNK) {
        const bool in = b0 + tid < rows;
        const size_t row = in ? b0 + tid : 0;
        if (l == 0) cp_async(&sX[st][tid][0], W.xin + row * 8, 16, in);
        if (l == 4) cp_async(&sD[st][tid][0], W.dzo + row * 2, 4, in);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[2][4];
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[j][r] = 0.f;
  for (int ch = 0; ch < kStages - 1; ++ch) fetch(ch);
  for (int ch = 0; ch < nch; ++ch) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();  // chunk ch has landed for all threads; chunk ch - 1's readers are done
    fetch(ch + kStages - 1);
    const int st = ch % kStages;
#pragma unroll
    for (int kk = 0; kk < CHUNK; kk += 16) {
      uint32_t a[4], b[4];
      // A, lanes 0-7, 8-15, 16-23, 24-31: rows k 0-7 at m, k 0-7 at m + 8, k 8-15 at m, k 8-15 at m + 8
      ldsm_t(a, &sD[st][kk + (lane & 7) + ((lane >> 4) << 3)][wm + ((lane >> 3) & 1) * 8]);
      // B: rows k 0-7 and k 8-15 at n, then both at n + 8
      ldsm_t(b, &sX[st][kk + (lane & 7) + ((lane >> 3) & 1) * 8][wn + (lane >> 4) * 8]);
      mma(acc[0], a, b[0], b[1]);
      mma(acc[1], a, b[2], b[3]);
    }
  }
  const int nk = l == 0 ? 6 : 256, nn = l == 4 ? 2 : 256;
  float* out = grads + woff(l);
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int n = n0 + wm + g + 8 * (r >> 1), k = k0 + wn + 8 * j + 2 * t + (r & 1);
      if (n < nn && k < nk) out[(size_t)n * nk + k] = acc[j][r];
    }
}

// BF16 copy of parameter i and, for the weights of layers 1-3, its places in the operand images.
__device__ __forceinline__ void store_bf16(int i, float v, __nv_bfloat16* wbf, __nv_bfloat16* fpack, __nv_bfloat16* bpack,
                                           __nv_bfloat16* wpack);

// Adam on the FP32 master parameters, then their BF16 copies.
__global__ void __launch_bounds__(256)
k_train_update(const float* __restrict__ grads, float lr, float c1, float c2, float b1, float b2, float eps, float* p,
               float* m, float* v, __nv_bfloat16* wbf, __nv_bfloat16* fpack, __nv_bfloat16* bpack, __nv_bfloat16* wpack) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_params(); i += gridDim.x * blockDim.x) {
    const float gi = grads[i];
    const float mi = moment1(b1, m[i], gi);
    const float vi = moment2(b2, v[i], gi);
    m[i] = mi;
    v[i] = vi;
    const float np = __fsub_rn(p[i], __fdiv_rn(__fmul_rn(lr, __fdiv_rn(mi, c1)), __fadd_rn(__fsqrt_rn(__fdiv_rn(vi, c2)), eps)));
    p[i] = np;
    store_bf16(i, np, wbf, fpack, bpack, wpack);
  }
}

// The BF16 copies of all parameters (after creation).
__global__ void k_refresh(const float* p, __nv_bfloat16* wbf, __nv_bfloat16* fpack, __nv_bfloat16* bpack,
                          __nv_bfloat16* wpack) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_params(); i += gridDim.x * blockDim.x)
    store_bf16(i, p[i], wbf, fpack, bpack, wpack);
}

}  // namespace tr

// ---------------------------------------------------------------- fused inference on tcgen05
// One CTA per SM, persistent over tiles of 128 rows, two tiles in flight.  Layer 0 (K = 6) and the
// output layer (N = 2) run on the CUDA cores; the three 256 x 256 layers are single-CTA tcgen05.mma
// (kind::f16, BF16 operands, M = 128, N = 128, K = 16 per instruction) from shared memory into an FP32
// accumulator of 256 tensor-memory columns per tile.  Operands use the K-major no-swizzle canonical
// layout, 8 x 8 core matrices of 128 contiguous bytes: element (r, k) of an activation tile is at byte
//     (r / 8) * 4096 + (k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2,
// i.e. K-adjacent core matrices 128 B apart (the descriptor's leading byte offset) and 8-row groups
// 4096 B apart (its stride byte offset); a layer's weights are cut into eight blocks of 128 rows and 64 k
// (16 KB), 8-row groups 1024 B apart, and kept in global memory in that image (packed after every
// update).
//
// What bounds it is the GELU: 1024 values a row, each about 12 multiply-adds (run as packed pairs), an
// exponential and a reciprocal: 16 k issue slots a tile and scheduler.  The matrix products (6.2k cycles
// a tile) and the weights' way from L2 (384 KB a tile) therefore have to hide behind it.  Two groups of
// eight warps each own a tile and its operand buffer; while one waits for a layer the other applies the
// activation.  A layer goes by halves of its columns: the products of the first column half with the
// first half of K start while the second half of the layer before is still being activated, and its
// activation starts while the second column half is being multiplied.  One thread issues all MMAs in a
// fixed order (layer by layer, group by group), another keeps a ring of four weight blocks filled in
// that order; both loops are unrolled over a layer's blocks, because the time that these two threads
// take between blocks is what a layer waits for.
// A million rows take 0.72 ms (0.41 ms of multiply-adds); with one tile in flight, whole layers and
// scalar GELUs they took 1.18 ms, and one tile alone 30 us instead of 27.  The halves gave the last 0.07 ms,
// unrolling those two threads' loops 0.03.
namespace tc {

constexpr int GROUP = 256;                        // threads of a tile
constexpr int THREADS = 2 * GROUP + 64;           // two groups, the weights' warp, the MMAs' warp
constexpr int TILE = 128;
constexpr int KB = 64;                            // k per weight block
constexpr int NBLK = 2 * 256 / KB;                // weight blocks of a layer: column half, then k
constexpr int RING = 4;                           // half a layer: a block's slot and parity follow from its place
constexpr uint32_t A_BYTES = TILE * 256 * 2;      // 64 KB
constexpr uint32_t W_BYTES = 128 * KB * 2;        // 16 KB
constexpr uint32_t OFF_A = 0;
constexpr uint32_t OFF_W = OFF_A + 2 * A_BYTES;
constexpr uint32_t OFF_W0 = OFF_W + RING * W_BYTES;   // float [128][16]: per column pair the weights
                                                      // (w_c0, w_d0, w_c1, ...), then the biases
constexpr uint32_t OFF_B = OFF_W0 + 128 * 16 * 4;     // float [3][256]: b1..b3
constexpr uint32_t OFF_W4 = OFF_B + 3 * 256 * 4;      // float [256][2]
constexpr uint32_t OFF_RED = OFF_W4 + 2 * 256 * 4;    // float [2][128][4]
constexpr uint32_t OFF_X = OFF_RED + 2 * TILE * 4 * 4;  // float [2][128][6]: inputs
constexpr uint32_t OFF_MISC = OFF_X + 2 * TILE * 6 * 4;
constexpr uint32_t SMEM = OFF_MISC + 256;
constexpr long long WAIT_CYCLES = 4000000000LL;   // about two seconds at the maximum clock

// instruction descriptor: D FP32, A and B BF16, both K-major, N = 128, M = 128
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ uint32_t act_offset(int r, int k) {
  return (uint32_t)((r >> 3) * 4096 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}
// element (n, k) of a layer's weights in its image, in bytes
__host__ __device__ __forceinline__ uint32_t weight_offset(int n, int k) {
  return (uint32_t)(((n >> 7) * (256 / KB) + k / KB) * (int)W_BYTES + ((n & 127) >> 3) * (KB / 8 * 128) +
                    ((k % KB) >> 3) * 128 + (n & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t stride) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(stride >> 4) << 32) |
         (1ull << 46);
}

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Waits for the phase with the given parity to complete; false after WAIT_CYCLES, or as soon as another
// thread has given up (*abort, where given), which it then says itself.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort) {
  auto done = [&] {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
  };
  if (done()) return true;
  const long long t0 = clock64();
  while (!done()) {
    if ((abort && *abort) || clock64() - t0 > WAIT_CYCLES) {
      if (abort) *abort = 1;
      return false;
    }
  }
  return true;
}

__device__ __forceinline__ void load_block(uint32_t dst, const void* src, uint32_t bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(W_BYTES) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(W_BYTES), "r"(bar)
               : "memory");
}

// D (+)= A W^T over one k16 step
__device__ __forceinline__ void mma_step(uint32_t tmem_d, uint64_t ad, uint64_t bd, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
          tmem_d),
      "l"(ad), "l"(bd), "r"(IDESC), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// 16 columns of this warp's 32 rows; complete after tmem_wait on the same registers
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])::"memory");
}

__device__ __forceinline__ float round_bf16(float a) { return __bfloat162float(__float2bfloat16(a)); }

// Two floats in one register pair: one instruction per operation on both, each rounded as alone.
using pair = unsigned long long;
__device__ __forceinline__ pair pack(float a, float b) {
  pair r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack(pair p, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p));
}
__device__ __forceinline__ pair both(float a) { return pack(a, a); }
__device__ __forceinline__ pair fma2(pair a, pair b, pair c) {
  pair r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ pair mul2(pair a, pair b) {
  pair r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ pair add2(pair a, pair b) {
  pair r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// gelu() of two values, the same operations and bits (below |x| = 13; beyond it a tail smaller than the
// smallest normal number is zero): factors 1/2 are folded into constants, which is exact, and the select
// between tail and 1 - tail is an addition, 0 + tail or 1 - tail.
__device__ __forceinline__ pair gelu2(pair x) {
  float x0, x1, y0, y1, t0, t1, e0, e1;
  unpack(x, x0, x1);
  unpack(fma2(both(0.3275911f), pack(fabsf(x0) * 0.70710678118654752f, fabsf(x1) * 0.70710678118654752f), both(1.0f)), y0, y1);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t0) : "f"(y0));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t1) : "f"(y1));
  const pair t = pack(t0, t1);
  pair h = fma2(t, both(0.5f * 1.061405429f), both(0.5f * -1.453152027f));
  h = fma2(t, h, both(0.5f * 1.421413741f));
  h = fma2(t, h, both(0.5f * -0.284496736f));
  h = fma2(t, h, both(0.5f * 0.254829592f));
  // e^{-x^2 / 2}: log2(e) as a float, halved
  unpack(mul2(mul2(x, x), both(-0.5f * 1.44269502f)), e0, e1);
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(e0));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(e1));
  unpack(mul2(mul2(t, h), pack(e0, e1)), t0, t1);  // the tail (1 - erf) / 2
  return mul2(x, add2(pack(copysignf(t0, -x0), copysignf(t1, -x1)), pack(x0 >= 0.0f ? 1.0f : 0.0f, x1 >= 0.0f ? 1.0f : 0.0f)));
}
__device__ __forceinline__ uint32_t pack_bf16(pair p) {
  float a, b;
  unpack(p, a, b);
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// x [B][6] fp32 features; wpack: layers 1-3 in the operand image; wbf: all parameters in BF16
// (W0 and W4 read from it); params: FP32 parameters (biases read from it).  Writes out [B][2]
// = (mu, log sigma^2) in the target's units.  *err is set to 1 if a wait timed out.
// Warp w of a group reads tensor-memory lanes 32 (w % 4) .. + 31 (its rows) and 64 columns of each half.
__global__ void __launch_bounds__(THREADS, 1)
k_mlp_forward(const float* __restrict__ x, int B, const __nv_bfloat16* __restrict__ wpack,
              const __nv_bfloat16* __restrict__ wbf, const float* __restrict__ params, const float* __restrict__ shift,
              const float* __restrict__ scale, float y0, float ys, float* __restrict__ out, int* err) {
  extern __shared__ __align__(1024) unsigned char sm[];
  float* sW0 = reinterpret_cast<float*>(sm + OFF_W0);
  float* sB = reinterpret_cast<float*>(sm + OFF_B);
  float* sW4 = reinterpret_cast<float*>(sm + OFF_W4);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + OFF_MISC);
  // per weight block: filled, free; per group: halves of the operand written (a), column halves
  // multiplied (d), first half of the operand no longer needed (k), partial outputs written (r)
  const uint32_t bar_full = saddr(bars), bar_free = saddr(bars + RING), bar_a = saddr(bars + 2 * RING);
  const uint32_t bar_d = bar_a + 32, bar_k = bar_a + 64, bar_r = bar_a + 80, bar_end = bar_a + 96;
  uint32_t* sTmem = reinterpret_cast<uint32_t*>(sm + OFF_MISC + 192);
  volatile int* sAbort = reinterpret_cast<volatile int*>(sm + OFF_MISC + 196);
  float* sB4 = reinterpret_cast<float*>(sm + OFF_MISC + 200);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ntiles = (B + TILE - 1) / TILE, step = 2 * gridDim.x;
  // tiles of group g: blockIdx.x + g gridDim.x, then every step-th
  const int n_own[2] = {(ntiles - (int)blockIdx.x + step - 1) / step,
                        max(0, (ntiles - (int)blockIdx.x - (int)gridDim.x + step - 1) / step)};

  // a tile's inputs (zero beyond the batch) into its group's buffer
  auto fetch_x = [&](int tile, int g) {
    for (int e = tid & (GROUP - 1); e < TILE * 6; e += GROUP) {
      const long i = (long)tile * (TILE * 6) + e;
      const bool in = i < (long)B * 6;
      tr::cp_async(sm + OFF_X + (g * TILE * 6 + e) * 4, x + (in ? i : 0), 4, in);
    }
  };
  if (tid < 2 * GROUP) fetch_x(blockIdx.x + (tid / GROUP) * gridDim.x, tid / GROUP);
  // small parameters (BF16 weights, FP32 biases)
  for (int i = tid; i < 256 * 6; i += THREADS) {
    const int c = i / 6, f = i - 6 * c;
    sW0[(c >> 1) * 16 + 2 * f + (c & 1)] = __bfloat162float(wbf[tr::woff(0) + i]);
  }
  for (int c = tid; c < 256; c += THREADS) {
    sW0[(c >> 1) * 16 + 12 + (c & 1)] = params[tr::boff(0) + c];
    for (int l = 1; l < 4; ++l) sB[(l - 1) * 256 + c] = params[tr::boff(l) + c];
    for (int u = 0; u < 2; ++u) sW4[2 * c + u] = __bfloat162float(wbf[tr::woff(4) + u * 256 + c]);
  }
  if (tid < 2) sB4[tid] = params[tr::boff(4) + tid];
  if (tid == 0) {
    *sAbort = 0;
    for (int i = 0; i < RING; ++i) {
      mbar_init(bar_full + 8 * i, 1);
      mbar_init(bar_free + 8 * i, 1);
    }
    for (int g = 0; g < 2; ++g) {
      for (int h = 0; h < 2; ++h) {
        mbar_init(bar_a + 16 * g + 8 * h, GROUP);
        mbar_init(bar_d + 16 * g + 8 * h, 1);
      }
      mbar_init(bar_k + 8 * g, 1);
      mbar_init(bar_r + 8 * g, GROUP / 2);
    }
    mbar_init(bar_end, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    const uint32_t dst = saddr(sTmem);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *sTmem;

  if (warp == 2 * GROUP / 32) {
    if (lane == 0) {  // the weights: per tile and layer its blocks in ascending k
      const uint32_t w_base = saddr(sm + OFF_W);
      bool ok = true;
      int used = 0;  // blocks fetched
      for (int i = 0; ok && i < n_own[0]; ++i)  // the order of the MMAs: tile pair, layer, group, block
        for (int l = 0; ok && l < 3; ++l)
          for (int g = 0; ok && g < 2 && i < n_own[g]; ++g) {
            const char* src = (const char*)wpack + (size_t)l * (NBLK * W_BYTES);
#pragma unroll
            for (int kb = 0; kb < NBLK; ++kb) {
              const int s = kb % RING;
              // the block before in this slot has been multiplied (nothing to wait for the first time)
              ok = ok && mbar_wait(bar_free + 8 * s, (kb / RING + 1) & 1, sAbort);
              if (ok) load_block(w_base + s * W_BYTES, src + kb * W_BYTES, bar_full + 8 * s), ++used;
            }
          }
      // given up: the last copy into each slot lands before the block ends
      for (int s = 0; !ok && s < RING && s < used; ++s)
        mbar_wait(bar_full + 8 * s, ((used - 1 - s) / RING) & 1, nullptr);
    }
  } else if (warp == 2 * GROUP / 32 + 1) {
    if (lane == 0) {
      const uint64_t a_desc = smem_desc(saddr(sm + OFF_A), 4096), w_desc = smem_desc(saddr(sm + OFF_W), KB / 8 * 128);
      bool ok = true;
      for (int i = 0; ok && i < n_own[0]; ++i)
        for (int l = 0; ok && l < 3; ++l)
          for (int g = 0; ok && g < 2 && i < n_own[g]; ++g) {
            const uint64_t ad = a_desc + g * (A_BYTES / 16);
            const uint32_t parity = (3 * i + l) & 1;
#pragma unroll
            for (int b = 0; b < NBLK; ++b) {
              const int s = b % RING, half = b / (NBLK / 2), kb = b % (NBLK / 2);
              // the first half of the operand is written and its accumulators are read; then the others
              if (b % (NBLK / 4) == 0 && b < NBLK / 2) {
                ok = ok && mbar_wait(bar_a + 16 * g + 8 * (b > 0), parity, sAbort);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              }
              ok = ok && mbar_wait(bar_full + 8 * s, (b / RING) & 1, sAbort);
              if (ok) {
#pragma unroll
                for (int kk = 0; kk < KB / 16; ++kk)  // 16 k are two core matrices, 256 bytes
                  mma_step(tmem + 256 * g + 128 * half, ad + kb * (KB / 8 * 128 / 16) + kk * 16,
                           w_desc + s * (W_BYTES / 16) + kk * 16, kb + kk > 0);
                mma_commit(bar_free + 8 * s);
                if (b == NBLK / 2 - 1 || b == NBLK - 1) mma_commit(bar_d + 16 * g + 8 * half);
                if (b == NBLK / 2 + NBLK / 4 - 1) mma_commit(bar_k + 8 * g);
              }
            }
          }
      mma_commit(bar_end);  // nothing of this thread is in flight when the tensor memory is given back
      mbar_wait(bar_end, 0, nullptr);
    }
  } else {
    const int g = warp >> 3, q = warp & 3, half = (warp >> 2) & 1;
    const int row_l = 32 * q + lane, c_first = 64 * half;  // and c_first + 128: a column quarter of each half
    unsigned char* sA = sm + OFF_A + g * A_BYTES;
    const uint32_t trow = tmem + 256 * g + c_first + ((uint32_t)(32 * q) << 16);
    float* sRed = reinterpret_cast<float*>(sm + OFF_RED) + (g * TILE + row_l) * 4;
    const uint32_t my_a = bar_a + 16 * g, my_d = bar_d + 16 * g, my_k = bar_k + 8 * g, my_r = bar_r + 8 * g;
    // layer 0: two rows a thread (a weight read from shared memory serves both), 32 columns of each half
    const int r0 = tid & 63, c0_first = 32 * ((tid >> 6) & 3);
    const float* sX = reinterpret_cast<const float*>(sm + OFF_X) + g * TILE * 6;
    int tile = blockIdx.x + g * gridDim.x;
    uint32_t ph = 0;  // layers done, for the parity
    bool ok = true;
    for (; ok && tile < ntiles; tile += step) {
      {
        pair xs[2][6];
#pragma unroll
        for (int f = 0; f < 6; ++f)
#pragma unroll
          for (int u = 0; u < 2; ++u)
            xs[u][f] = both(round_bf16((sX[(r0 + 64 * u) * 6 + f] - __ldg(shift + f)) * __ldg(scale + f)));
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
#pragma unroll 1
          for (int c0 = 128 * h + c0_first; c0 < 128 * h + c0_first + 32; c0 += 8) {
            uint32_t w[2][4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const ulonglong2* wr = reinterpret_cast<const ulonglong2*>(sW0 + (c0 / 2 + j) * 16);
              const ulonglong2 w01 = wr[0], w23 = wr[1], w45 = wr[2];
              const pair bias = *reinterpret_cast<const pair*>(wr + 3);
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                pair acc = fma2(xs[u][0], w01.x, both(0.0f));
                acc = fma2(xs[u][1], w01.y, acc);
                acc = fma2(xs[u][2], w23.x, acc);
                acc = fma2(xs[u][3], w23.y, acc);
                acc = fma2(xs[u][4], w45.x, acc);
                acc = fma2(xs[u][5], w45.y, acc);
                w[u][j] = pack_bf16(gelu2(add2(acc, bias)));
              }
            }
#pragma unroll
            for (int u = 0; u < 2; ++u)
              *reinterpret_cast<uint4*>(sA + act_offset(r0 + 64 * u, c0)) = make_uint4(w[u][0], w[u][1], w[u][2], w[u][3]);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          mbar_arrive(my_a + 8 * h);
        }
      }
      pair o[2] = {0, 0};  // (mu, log sigma^2) of this thread's two column quarters
      for (int l = 1; l <= 3; ++l, ++ph) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          // warp-uniform outcome: tcgen05.ld below is a warp-wide instruction
          ok = ok && __all_sync(0xffffffffu, mbar_wait(my_d + 8 * h, ph & 1, sAbort));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (l == 1 && h == 0) fetch_x(tile + step, g);  // everyone in the group is done with this tile's
          const int ch = c_first + 128 * h;
          const float* bias = sB + (l - 1) * 256 + ch;
          uint32_t r[2][16];
          tmem_ld16(trow + 128 * h, r[0]);
#pragma unroll 1
          for (int c0 = 0; c0 < 64; c0 += 32)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int c = c0 + 16 * u;
              tmem_wait(r[u]);
              if (c < 48) tmem_ld16(trow + 128 * h + c + 16, r[u ^ 1]);
              pair v[8];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(bias + c + 4 * i);
                v[2 * i] = gelu2(add2(pack(__uint_as_float(r[u][4 * i]), __uint_as_float(r[u][4 * i + 1])), b.x));
                v[2 * i + 1] = gelu2(add2(pack(__uint_as_float(r[u][4 * i + 2]), __uint_as_float(r[u][4 * i + 3])), b.y));
              }
              if (l < 3) {
                // the second column half's products with the first half of the operand are done
                if (h == 0 && c == 0) ok = __all_sync(0xffffffffu, mbar_wait(my_k, ph & 1, sAbort));
                if (ok) {
#pragma unroll
                  for (int i = 0; i < 2; ++i)
                    *reinterpret_cast<uint4*>(sA + act_offset(row_l, ch + c + 8 * i)) =
                        make_uint4(pack_bf16(v[4 * i]), pack_bf16(v[4 * i + 1]), pack_bf16(v[4 * i + 2]), pack_bf16(v[4 * i + 3]));
                }
              } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                  const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(sW4 + 2 * (ch + c + 2 * i));
                  const uint32_t a = pack_bf16(v[i]);  // rounded; a BF16 number is the upper half of its float
                  o[h] = fma2(both(__uint_as_float(a << 16)), w.x, o[h]);
                  o[h] = fma2(both(__uint_as_float(a & 0xffff0000u)), w.y, o[h]);
                }
              }
            }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          if (l < 3) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (l == 2) asm volatile("cp.async.wait_all;" ::: "memory");  // the next inputs: seen by all at layer 3
            mbar_arrive(my_a + 8 * h);
          }
        }
        if (!ok) break;
      }
      if (!ok) break;
      // the output: bias, then the four column quarters in order
      float q0, q1, q2, q3;
      unpack(o[0], q0, q1);
      unpack(o[1], q2, q3);
      if (half) {
        *reinterpret_cast<float4*>(sRed) = make_float4(q0, q1, q2, q3);
        mbar_arrive(my_r);
      } else {
        ok = __all_sync(0xffffffffu, mbar_wait(my_r, (ph / 3 + 1) & 1, sAbort));
        const long row = (long)tile * TILE + row_l;
        if (ok && row < B) {
          const float4 p = *reinterpret_cast<const float4*>(sRed);
          out[row * 2] = (sB4[0] + q0 + p.x + q2 + p.z) / ys + y0;
          out[row * 2 + 1] = (sB4[1] + q1 + p.y + q3 + p.w) - 2.0f * logf(ys);
        }
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*sAbort && tid == 0) atomicExch(err, 1);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

}  // namespace tc

namespace tr {
__device__ __forceinline__ void store_bf16(int i, float v, __nv_bfloat16* wbf, __nv_bfloat16* fpack, __nv_bfloat16* bpack,
                                           __nv_bfloat16* wpack) {
  const __nv_bfloat16 h = __float2bfloat16(v);
  wbf[i] = h;
  const int per = 256 * 256 + 256, r = i - woff(1);
  if (r < 0 || r >= 3 * per) return;
  const int l = r / per, e = r - l * per;
  if (e >= 65536) return;
  const int n = e >> 8, k = e & 255;
  fpack[(size_t)l * 65536 + frag_index(n, k)] = h;
  bpack[(size_t)l * 65536 + frag_index(k, n)] = h;
  wpack[(size_t)l * 65536 + tc::weight_offset(n, k) / 2] = h;
}
}  // namespace tr
}  // namespace mlp
}  // namespace swf

using namespace swf;
using namespace swf::mlp;

struct swf_mlp {
  int device;
  int max_batch;
  long step;
  float* params;             // FP32 master: per layer W [out][in] then b [out]
  float* grads;
  float* adam_m;
  float* adam_v;
  __nv_bfloat16* wbf;        // BF16 copy of all parameters (same layout)
  __nv_bfloat16* fpack;      // layers 1-3 in the training kernels' operand order, forward and backward
  __nv_bfloat16* bpack;
  __nv_bfloat16* wpack;      // layers 1-3 in the tensor-core operand image (inference kernel)
  tr::Bufs train;
  float* loss;
  float* in_shift;           // [6] feature standardisation
  float* in_scale;           // [6]
  float y0, ys;              // target standardisation
  int* err;                  // set by the inference kernel when a wait timed out
  int nsm;
  cudaStream_t last_stream;
  std::vector<void*> allocs;
};

namespace {
swf_status mlp_alloc(swf_mlp* m, void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    set_error("cudaMalloc failed for the surrogate network");
    return SWF_ENOMEM;
  }
  m->allocs.push_back(*p);
  return SWF_OK;
}

// One pass over a batch: the gradients into grads and the loss, then (update) an Adam step.
cudaError_t train_pass(swf_mlp* m, const float* x, const float* y, int B, bool update, float lr, float* grads, float* loss,
                       cudaStream_t st) {
  const int nblk = (B + tr::ROWS - 1) / tr::ROWS, rows = nblk * tr::ROWS;
  tr::k_train_rows<<<nblk, tr::THREADS, 0, st>>>(x, y, B, m->wbf, m->fpack, m->bpack, m->params, m->in_shift, m->in_scale,
                                                 m->y0, m->ys, m->train);
  tr::k_train_dw<<<tr::kTiles + 8 + 1, 128, 0, st>>>(y, B, rows, m->y0, m->ys, m->train, grads, m->loss, loss);
  if (update) {
    m->step += 1;
    const double b1 = 0.9, b2 = 0.999;
    tr::k_train_update<<<(n_params() + 511) / 512, 256, 0, st>>>(
        grads, lr, (float)(1.0 - std::pow(b1, (double)m->step)), (float)(1.0 - std::pow(b2, (double)m->step)), 0.9f, 0.999f,
        1e-8f, m->params, m->adam_m, m->adam_v, m->wbf, m->fpack, m->bpack, m->wpack);
  }
  return cudaGetLastError();
}
}  // namespace

extern "C" {

int swf_mlp_param_count(void) { return n_params(); }

swf_status swf_mlp_create(swf_mlp** out, int device, const float* init_params, int max_batch, const float* norm) {
  if (!out || !init_params || !norm || max_batch < 1) { set_error("swf_mlp_create: invalid arguments"); return SWF_EINVAL; }
  if (!(norm[13] > 0.f)) { set_error("swf_mlp_create: target scale must be positive"); return SWF_EINVAL; }
  *out = nullptr;
  cudaError_t e = cudaSetDevice(device);
  if (e != cudaSuccess) return cuda_status(e, "cudaSetDevice");
  swf_mlp* m = new swf_mlp();
  m->device = device;
  m->max_batch = max_batch;
  m->step = 0;
  const size_t np = n_params();
  swf_status s;
  auto fail = [&](swf_status st) {
    for (void* p : m->allocs) cudaFree(p);
    delete m;
    return st;
  };
  if ((s = mlp_alloc(m, (void**)&m->params, np * 4)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->grads, np * 4)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->adam_m, np * 4)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->adam_v, np * 4)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->wbf, np * 2)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->loss, 4)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->in_shift, 6 * 4)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->in_scale, 6 * 4)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->wpack, (size_t)3 * 256 * 256 * 2)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->err, sizeof(int))) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->fpack, (size_t)3 * 65536 * 2)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->bpack, (size_t)3 * 65536 * 2)) != SWF_OK) return fail(s);
  m->last_stream = 0;
  m->nsm = 0;
  e = cudaDeviceGetAttribute(&m->nsm, cudaDevAttrMultiProcessorCount, device);
  if (e != cudaSuccess || m->nsm < 1) return fail(cuda_status(e, "SM count"));
  e = cudaFuncSetAttribute(tc::k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::SMEM);
  if (e != cudaSuccess) return fail(cuda_status(e, "cudaFuncSetAttribute(k_mlp_forward)"));
  m->y0 = norm[12];
  m->ys = norm[13];
  const size_t nblk = ((size_t)max_batch + tr::ROWS - 1) / tr::ROWS, rows = nblk * tr::ROWS;
  for (int l = 0; l < 4; ++l) {
    if ((s = mlp_alloc(m, (void**)&m->train.act[l], rows * 512)) != SWF_OK) return fail(s);
    if ((s = mlp_alloc(m, (void**)&m->train.dz[l], rows * 512)) != SWF_OK) return fail(s);
  }
  if ((s = mlp_alloc(m, (void**)&m->train.xin, rows * 16)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->train.dzo, rows * 4)) != SWF_OK) return fail(s);
  for (int l = 0; l < 4; ++l)
    if ((s = mlp_alloc(m, (void**)&m->train.dz32[l], rows * 1024)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->train.dzo32, rows * 8)) != SWF_OK) return fail(s);
  if ((s = mlp_alloc(m, (void**)&m->train.zo, rows * 8)) != SWF_OK) return fail(s);
  e = cudaMemcpy(m->params, init_params, np * 4, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return fail(cuda_status(e, "upload parameters"));
  e = cudaMemcpy(m->in_shift, norm, 6 * 4, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return fail(cuda_status(e, "upload normalisation"));
  e = cudaMemcpy(m->in_scale, norm + 6, 6 * 4, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return fail(cuda_status(e, "upload normalisation"));
  cudaMemset(m->adam_m, 0, np * 4);
  cudaMemset(m->adam_v, 0, np * 4);
  cudaMemset(m->err, 0, sizeof(int));
  tr::k_refresh<<<256, 256>>>(m->params, m->wbf, m->fpack, m->bpack, m->wpack);
  e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return fail(cuda_status(e, "surrogate set-up"));
  *out = m;
  return SWF_OK;
}

swf_status swf_mlp_destroy(swf_mlp* m) {
  if (!m) return SWF_OK;
  cudaSetDevice(m->device);
  cudaDeviceSynchronize();
  for (void* p : m->allocs) cudaFree(p);
  delete m;
  return SWF_OK;
}

swf_status swf_mlp_forward(swf_mlp* m, const float* x_dev, int B, float* out_dev, void* stream) {
  if (!m || !x_dev || !out_dev || B < 1) { set_error("swf_mlp_forward: invalid arguments"); return SWF_EINVAL; }
  cudaSetDevice(m->device);
  cudaStream_t st = (cudaStream_t)stream;
  const int ntiles = (B + tc::TILE - 1) / tc::TILE;
  const int grid = ntiles < m->nsm ? ntiles : m->nsm;
  tc::k_mlp_forward<<<grid, tc::THREADS, tc::SMEM, st>>>(x_dev, B, m->wpack, m->wbf, m->params, m->in_shift,
                                                         m->in_scale, m->y0, m->ys, out_dev, m->err);
  m->last_stream = st;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "surrogate forward");
  return SWF_OK;
}

swf_status swf_mlp_status(swf_mlp* m) {
  if (!m) { set_error("swf_mlp_status: invalid arguments"); return SWF_EINVAL; }
  cudaSetDevice(m->device);
  cudaError_t e = cudaStreamSynchronize(m->last_stream);
  if (e != cudaSuccess) return cuda_status(e, "surrogate status");
  int flag = 0;
  e = cudaMemcpy(&flag, m->err, sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_status(e, "surrogate status");
  if (flag) {
    set_error("surrogate inference: a tensor-core wait timed out");
    return SWF_ETIMEOUT;
  }
  return SWF_OK;
}

swf_status swf_mlp_gradients(swf_mlp* m, const float* x_dev, const float* y_dev, int B, float* grad_dev,
                             float* loss_dev, void* stream) {
  if (!m || !x_dev || !y_dev || B < 1 || B > m->max_batch) {
    set_error("swf_mlp_gradients: invalid arguments (batch must be in [1, max_batch])");
    return SWF_EINVAL;
  }
  cudaSetDevice(m->device);
  const cudaError_t e = train_pass(m, x_dev, y_dev, B, false, 0.f, grad_dev ? grad_dev : m->grads, loss_dev, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_status(e, "surrogate gradients");
  return SWF_OK;
}

swf_status swf_mlp_train_step(swf_mlp* m, const float* x_dev, const float* y_dev, int B, float lr, float* loss_dev,
                              void* stream) {
  if (!m || !x_dev || !y_dev || B < 1 || B > m->max_batch) {
    set_error("swf_mlp_train_step: invalid arguments (batch must be in [1, max_batch])");
    return SWF_EINVAL;
  }
  cudaSetDevice(m->device);
  const cudaError_t e = train_pass(m, x_dev, y_dev, B, true, lr, m->grads, loss_dev, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_status(e, "surrogate update");
  return SWF_OK;
}

swf_status swf_mlp_activation(const float* x_dev, int n, float* gelu_dev, float* grad_dev, void* stream) {
  if (!x_dev || !gelu_dev || !grad_dev || n < 0) { set_error("swf_mlp_activation: invalid arguments"); return SWF_EINVAL; }
  if (n == 0) return SWF_OK;
  const int nb = (n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096;
  k_gelu_eval<<<nb, 256, 0, (cudaStream_t)stream>>>(x_dev, n, gelu_dev, grad_dev);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "swf_mlp_activation");
  return SWF_OK;
}

swf_status swf_mlp_get_params(swf_mlp* m, float* params_host) {
  if (!m || !params_host) { set_error("swf_mlp_get_params: invalid arguments"); return SWF_EINVAL; }
  cudaSetDevice(m->device);
  cudaError_t e = cudaMemcpy(params_host, m->params, (size_t)n_params() * 4, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_status(e, "download parameters");
  return SWF_OK;
}

}  // extern "C"
