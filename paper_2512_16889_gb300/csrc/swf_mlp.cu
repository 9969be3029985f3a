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
// the order it had there (ascending k and rows), so the results are the same bits.
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
          const float r = (y[b] - y0) * ys - mu, w = __expf(-l);
          dmu = -r * w / B;
          dl = 0.5f * (1.0f - r * r * w) / B;
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
        const float r = (y[b] - y0) * ys - mu, w = __expf(-l);
        acc += 0.5f * (r * r * w + l);
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
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float np = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
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
// One CTA (256 threads) per SM, persistent over tiles of 128 rows.  Layer 0 (K = 6) and the
// output layer (N = 2) run on the CUDA cores; the three 256 x 256 layers are single-CTA
// tcgen05.mma (kind::f16, BF16 operands, M = 128, N = 256, K = 16 per instruction) from shared
// memory into an FP32 accumulator of 256 tensor-memory columns.  Operands use the K-major
// no-swizzle canonical layout: element (r, k) of a 256-wide operand at byte
//     (r / 8) * 4096 + (k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2,
// i.e. 8 x 8 core matrices of 128 contiguous bytes, K-adjacent core matrices 128 B apart (the
// descriptor's leading byte offset) and 8-row groups 4096 B apart (its stride byte offset).
// The weights of layers 1-3 are kept in global memory in exactly that image (packed after every
// update) and brought in with one bulk asynchronous copy per layer, overlapping the previous
// layer's epilogue.  The epilogue adds the bias, applies GELU and writes the BF16 activation
// back into the operand buffer; after layer 3 it contracts with the output weights.
namespace tc {

constexpr int THREADS = 512;
constexpr int TILE = 128;
constexpr uint32_t OP_BYTES_A = TILE * 256 * 2;   // 64 KB
constexpr uint32_t OP_BYTES_W = 256 * 256 * 2;    // 128 KB
constexpr uint32_t OFF_A = 0;
constexpr uint32_t OFF_W = OFF_A + OP_BYTES_A;
constexpr uint32_t OFF_W0 = OFF_W + OP_BYTES_W;   // float [256][6]
constexpr uint32_t OFF_B = OFF_W0 + 256 * 6 * 4;  // float [4][256]: b0..b3
constexpr uint32_t OFF_W4 = OFF_B + 4 * 256 * 4;  // float [2][256]
constexpr uint32_t OFF_RED = OFF_W4 + 2 * 256 * 4;  // float [4][128][2]
constexpr uint32_t OFF_MISC = OFF_RED + 4 * TILE * 2 * 4;
constexpr uint32_t SMEM = OFF_MISC + 64;
constexpr long long WAIT_CYCLES = 4000000000LL;   // about two seconds at the maximum clock

// instruction descriptor: D FP32, A and B BF16, both K-major, N = 128 (one column half), M = 128
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

__host__ __device__ __forceinline__ uint32_t op_offset(int r, int k) {
  return (uint32_t)((r >> 3) * 4096 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(4096u >> 4) << 32) |
         (1ull << 46);
}

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

// Waits for the phase with the given parity to complete; false after WAIT_CYCLES.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  while (true) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > WAIT_CYCLES) return false;
  }
}

__device__ __forceinline__ void load_weights(uint32_t dst, const void* src, uint32_t bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(OP_BYTES_W) : "memory");
  for (uint32_t c = 0; c < OP_BYTES_W; c += 32768)
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst + c),
                 "l"((const char*)src + c), "r"(32768u), "r"(bar)
                 : "memory");
}

// D[:, 0:128) = A W_half^T over K = 256 (16 instructions); W_half = rows [128 h, 128 h + 128) of W
__device__ __forceinline__ void mma_half(uint32_t tmem_d, uint32_t a_base, uint32_t w_base) {
#pragma unroll
  for (int kk = 0; kk < 16; ++kk) {
    const uint64_t ad = smem_desc(a_base + kk * 256), bd = smem_desc(w_base + kk * 256);
    const uint32_t acc = kk > 0 ? 1u : 0u;
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
            tmem_d),
        "l"(ad), "l"(bd), "r"(IDESC), "r"(acc)
        : "memory");
  }
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ float round_bf16(float a) { return __bfloat162float(__float2bfloat16(a)); }

// x [B][6] fp32 features; wpack: layers 1-3 in the operand image; wbf: all parameters in BF16
// (W0 and W4 read from it); params: FP32 parameters (biases read from it).  Writes out [B][2]
// = (mu, log sigma^2) in the target's units.  *err is set to 1 if a wait timed out.
// 16 warps: warp w reads tensor-memory lanes 32 (w % 4) .. + 31 (its rows) and columns
// [64 (w / 4), + 64).  Each layer's MMAs run as two column halves with their own commits, so
// the warps of half 0 start their epilogue while half 1 is still multiplying; every warp holds
// its BF16 results in registers until both halves are done (all of A feeds both halves).
__global__ void __launch_bounds__(THREADS, 1)
k_mlp_forward(const float* __restrict__ x, int B, const __nv_bfloat16* __restrict__ wpack,
              const __nv_bfloat16* __restrict__ wbf, const float* __restrict__ params, const float* __restrict__ shift,
              const float* __restrict__ scale, float y0, float ys, float* __restrict__ out, int* err) {
  extern __shared__ __align__(1024) unsigned char sm[];
  float* sW0 = reinterpret_cast<float*>(sm + OFF_W0);
  float* sB = reinterpret_cast<float*>(sm + OFF_B);
  float* sW4 = reinterpret_cast<float*>(sm + OFF_W4);
  float* sRed = reinterpret_cast<float*>(sm + OFF_RED);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + OFF_MISC);  // [0] weights, [1] MMA half 0, [2] MMA half 1
  uint32_t* sTmem = reinterpret_cast<uint32_t*>(sm + OFF_MISC + 24);
  int* sAbort = reinterpret_cast<int*>(sm + OFF_MISC + 28);
  float* sB4 = reinterpret_cast<float*>(sm + OFF_MISC + 32);
  const int tid = threadIdx.x, warp = tid >> 5;
  const uint32_t a_base = saddr(sm + OFF_A), w_base = saddr(sm + OFF_W);
  const uint32_t barW = saddr(&bars[0]), barM0 = saddr(&bars[1]), barM1 = saddr(&bars[2]);
  const int ntiles = (B + TILE - 1) / TILE;

  // small parameters (BF16 weights as the GEMM path rounds them, FP32 biases)
  constexpr long W0OFF = 0, B0OFF = 6 * 256;
  for (int i = tid; i < 256 * 6; i += THREADS) sW0[i] = __bfloat162float(wbf[W0OFF + i]);
  for (int l = 0; l < 4; ++l) {
    const long bo = (l == 0) ? B0OFF : B0OFF + 256 + (long)(l - 1) * (256 * 256 + 256) + 256 * 256;
    for (int i = tid; i < 256; i += THREADS) sB[l * 256 + i] = params[bo + i];
  }
  const long w4off = B0OFF + 256 + 3L * (256 * 256 + 256);
  for (int i = tid; i < 2 * 256; i += THREADS) sW4[i] = __bfloat162float(wbf[w4off + i]);
  if (tid < 2) sB4[tid] = params[w4off + 2 * 256 + tid];
  if (tid == 0) {
    *sAbort = 0;
    mbar_init(barW, 1);
    mbar_init(barM0, 1);
    mbar_init(barM1, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    const uint32_t dst = saddr(sTmem);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(256u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *sTmem;
  uint32_t phW = 0, phM = 0;
  if (tid == 0 && blockIdx.x < ntiles) load_weights(w_base, wpack, barW);

  const int q = warp & 3, cq = warp >> 2;    // TMEM lane quarter and column quarter of this warp
  const int half = cq >> 1;                  // MMA column half whose commit this warp waits for
  const int erow = 32 * q + (tid & 31);      // epilogue row
  const uint32_t bar_mine = half ? barM1 : barM0;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const bool more = tile + (int)gridDim.x < ntiles;
    // layer 0 on the CUDA cores: row r, columns [64 h, 64 h + 64)
    {
      const int r = tid & (TILE - 1), h = tid >> 7;
      const long row = (long)tile * TILE + r;
      float xin[6];
#pragma unroll
      for (int f = 0; f < 6; ++f) xin[f] = row < B ? round_bf16((x[row * 6 + f] - shift[f]) * scale[f]) : 0.f;
      for (int c0 = 64 * h; c0 < 64 * h + 64; c0 += 8) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
          float z[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const float* wr = sW0 + (c0 + j + u) * 6;
            float acc = 0.f;
#pragma unroll
            for (int f = 0; f < 6; ++f) acc = fmaf(xin[f], wr[f], acc);
            z[u] = gelu(acc + sB[c0 + j + u]);
          }
          w[j >> 1] = pack_bf16(z[0], z[1]);
        }
        *reinterpret_cast<uint4*>(sm + OFF_A + op_offset(r, c0)) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    for (int l = 1; l <= 3; ++l) {
      if (tid == 0) {
        if (!mbar_wait(barW, phW)) {
          *sAbort = 1;
        } else {
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          mma_half(tmem, a_base, w_base);
          mma_commit(barM0);
          mma_half(tmem + 128, a_base, w_base + 65536);
          mma_commit(barM1);
        }
      }
      phW ^= 1;
      __syncthreads();
      if (*sAbort) break;
      // warp-uniform outcome: tcgen05.ld below is a warp-wide instruction
      bool ok = __all_sync(0xffffffffu, mbar_wait(bar_mine, phM));
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t trow = tmem + ((uint32_t)(32 * q) << 16);
      const float* bias = sB + l * 256;
      uint32_t packed[32];
      float o0 = 0.f, o1 = 0.f;
      if (ok) {
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          const int c0 = 64 * cq + 16 * cc;
          float v[16];
          tmem_ld16(trow + c0, v);
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = gelu(v[i] + bias[c0 + i]);
          if (l < 3) {
#pragma unroll
            for (int i = 0; i < 8; ++i) packed[8 * cc + i] = pack_bf16(v[2 * i], v[2 * i + 1]);
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float a = round_bf16(v[i]);
              o0 = fmaf(a, sW4[c0 + i], o0);
              o1 = fmaf(a, sW4[256 + c0 + i], o1);
            }
          }
        }
      }
      // every MMA of the layer is done before the operand buffers are overwritten; the weight
      // buffer is then free for the next layer's (or the next tile's first) weights
      if (half == 0 && l < 3) ok = __all_sync(0xffffffffu, ok && mbar_wait(barM1, phM));
      if (!ok) atomicExch(sAbort, 1);
      phM ^= 1;
      if (tid == 256 && ok && (l < 3 || more))
        load_weights(w_base, wpack + (size_t)(l < 3 ? l : 0) * 256 * 256, barW);
      if (ok && l < 3) {
#pragma unroll
        for (int cc = 0; cc < 8; ++cc) {
          const int c0 = 64 * cq + 8 * cc;
          *reinterpret_cast<uint4*>(sm + OFF_A + op_offset(erow, c0)) =
              make_uint4(packed[4 * cc], packed[4 * cc + 1], packed[4 * cc + 2], packed[4 * cc + 3]);
        }
      }
      if (l == 3) {
        sRed[(cq * TILE + erow) * 2] = o0;
        sRed[(cq * TILE + erow) * 2 + 1] = o1;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      if (*sAbort) break;
    }
    if (*sAbort) break;
    if (tid < TILE) {
      const long row = (long)tile * TILE + tid;
      if (row < B) {
        float z0 = sB4[0], z1 = sB4[1];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          z0 += sRed[(c * TILE + tid) * 2];
          z1 += sRed[(c * TILE + tid) * 2 + 1];
        }
        out[row * 2] = z0 / ys + y0;
        out[row * 2 + 1] = z1 - 2.0f * logf(ys);
      }
    }
  }
  if (*sAbort && tid == 0) atomicExch(err, 1);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u) : "memory");
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
  wpack[(size_t)l * 65536 + tc::op_offset(n, k) / 2] = h;
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
