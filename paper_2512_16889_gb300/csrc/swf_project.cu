// Projections at t_in (Sec. II, Eqs. 8-9) in FP64: grid transforms of the scattered waves,
// the C-spectrum (U_scat(m) | V_back(r, q)) over every grid positron, direct transforms at
// off-grid wave vectors, and grid norms.
#include <atomic>
#include <cstring>

#include "swf_pass.cuh"

namespace swf {

namespace {

constexpr int kT = 256;

// One axis of the forward transform of every component plane (F*4 planes of N points): lines along
// `axis` from `in` to `out` (in place when they are the same), nl of them per block (consecutive rows
// on the x axis, consecutive x columns otherwise), tpl threads per line.  scale: the last axis
// multiplies by it and, with sign, by the phase exp(-i kappa.x0) of a grid that starts at x0 = -L/2,
// which is (-1)^(j'x + j'y + j'z) exactly.  FP64 operations bound it (25 per point: radix-4 passes and
// their twiddles, a floor of 170 us per axis for 16 fields of 256^2; measured 231 us, 333 us with every
// pass in shared memory); the conversion of a complex64 input (28 us as a pass of its own) and the
// scale and sign (436 us with a sine and cosine per mode) ride along.
template <typename Rin>
__global__ void __launch_bounds__(kPassThreads, 1)
k_fft_axis(const cpx<Rin>* in, cpx<double>* out, GridDesc g, int axis, const __grid_constant__ RadixPlan pl,
           const cpx<double>* __restrict__ tw, int nl, int ld, int tpl, double scale, int sign) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2], na = pl.n;
  const size_t plane = (size_t)blockIdx.y * g.N;
  int l, b0, o = 0;    // line within the block, first butterfly, index on the other axis
  size_t base, stride;
  bool ok;
  if (axis == 0) {
    l = threadIdx.x / tpl;
    b0 = threadIdx.x - l * tpl;
    o = blockIdx.x * nl + l;  // row
    ok = l < nl && o < ny * nz;
    base = plane + (size_t)o * nx;
    stride = 1;
  } else {
    const int ntx = (nx + nl - 1) / nl, xt = blockIdx.x % ntx;
    o = blockIdx.x / ntx;  // z (axis 1) or y (axis 2)
    b0 = threadIdx.x / nl;
    l = threadIdx.x - b0 * nl;
    ok = b0 < tpl && xt * nl + l < nx;
    base = plane + (axis == 1 ? (size_t)o * nx * ny : (size_t)o * nx) + xt * nl + l;
    stride = axis == 1 ? (size_t)nx : (size_t)nx * ny;
  }
  cpx<double>* a = reinterpret_cast<cpx<double>*>(smem_raw);
  cpx<double>* b2 = a + nl * ld;
  if (ok)
    with_radix(end_radix(pl, true), [&](auto rc) {
      constexpr int R0 = decltype(rc)::value;
      const int nb = na / R0;
      for (int b = b0; b < nb; b += tpl) {
        cpx<double> v[R0];
#pragma unroll
        for (int q = 0; q < R0; ++q) v[q] = cvt<double>(in[base + (size_t)(b + q * nb) * stride]);
        first_butterfly<double, R0>(v, b, false, a + l * ld);
      }
    });
  __syncthreads();
  const cpx<double>* cur = middle_passes<double>(a, b2, ld, nl, pl, false, tw);
  if (!ok) return;
  int par = 0;  // parity of the other axes' mode numbers j'
  if (sign) {
    auto parity = [&](int j, int n) { return n > 1 ? (j < (n + 1) / 2 ? j : j - n) & 1 : 0; };
    if (axis == 0) par = 0;  // x is the last axis only where it is the only one
    else if (axis == 1) par = parity((int)((base - plane) % nx), nx) ^ parity(o, nz);
    else par = parity((int)((base - plane) % nx), nx) ^ parity(o, ny);
  }
  with_radix(end_radix(pl, false), [&](auto rc) {
    constexpr int RL = decltype(rc)::value;
    const int nm = na / RL;
    for (int b = b0; b < nm; b += tpl) {
      cpx<double> m[RL];
      last_butterfly<double, RL>(cur + l * ld, b, na, pl.npass < 2, false, tw, m);
#pragma unroll
      for (int q = 0; q < RL; ++q) {
        const int j = b + q * nm;
        double sc = scale;
        if (sign && (((j < (na + 1) / 2 ? j : j - na) ^ par) & 1)) sc = -scale;
        out[base + (size_t)j * stride] = sc * m[q];
      }
    }
  });
}

// C(m, (r, q)) = exp(i q0 t_in) sum_a conj(U~_a(-q)) v_{r,a}(q); the positron at mode j has
// q = -kappa_j (trivial axes: kappa = K of the electron wave).  A thread holds the two spinors of one
// mode, phase included, for fc fields (they depend on the mode and K alone; a field with another K has
// its own): the square roots and the sine and cosine in FP64 are about four times a field's products
// (16 fields of 256^2: 309 -> 108 us).
__global__ void __launch_bounds__(kT) k_c_spectrum(const cpx<double>* __restrict__ spec, const FieldDesc* fd, GridDesc g,
                                                   int F, int fc, double t_in, cpx<double>* c_out, double* prob) {
  const int f0 = blockIdx.y * fc, f1 = min(F, f0 + fc);
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= g.N) return;
  const int row = j / g.n[0];
  const int id[3] = {j - row * g.n[0], row % g.n[1], row / g.n[1]};
  double kap[3], v[2][8];
  for (int a = 0; a < 3; ++a) kap[a] = mode_kappa(id[a], g.n[a], g.L[a]);
  for (int f = f0; f < f1; ++f) {
    const double* K = fd[f].K;
    const bool same = f > f0 && K[0] == fd[f - 1].K[0] && K[1] == fd[f - 1].K[1] && K[2] == fd[f - 1].K[2];
    if (!same) {
      double q[3];
      for (int a = 0; a < 3; ++a) q[a] = -(g.n[a] > 1 ? kap[a] : K[a]);
      double sn = 0.0, cs = 1.0;
      if (c_out) sincos(energy3(q) * t_in, &sn, &cs);  // |C|^2 does not see it
#pragma unroll
      for (int ir = 0; ir < 2; ++ir) {
        double w[8];
        spinor_uv(q, ir == 0 ? 1 : -1, true, w);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          v[ir][2 * a] = cs * w[2 * a] - sn * w[2 * a + 1];
          v[ir][2 * a + 1] = cs * w[2 * a + 1] + sn * w[2 * a];
        }
      }
    }
    const cpx<double>* u = spec + (size_t)f * 4 * g.N + j;
    cpx<double> uc[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) uc[a] = u[(size_t)a * g.N];
#pragma unroll
    for (int ir = 0; ir < 2; ++ir) {
      cpx<double> acc = mk<double>(0, 0);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        acc.x = fma(uc[a].y, v[ir][2 * a + 1], fma(uc[a].x, v[ir][2 * a], acc.x));
        acc.y = fma(-uc[a].y, v[ir][2 * a], fma(uc[a].x, v[ir][2 * a + 1], acc.y));
      }
      const size_t e = ((size_t)f * 2 + ir) * g.N + j;
      if (c_out) c_out[e] = acc;
      if (prob) prob[e] = acc.x * acc.x + acc.y * acc.y;
    }
  }
}

template <typename Rin>
__device__ __forceinline__ cpx<double> ld_d(const void* p, size_t i) {
  return cvt<double>(reinterpret_cast<const cpx<Rin>*>(p)[i]);
}

// Entry f (field f % n_fields at kappa f): blocks' parts of sum_x psi_a(x) exp(-i kappa.x) for a = 0..3
// (deterministic order).
template <typename Rin>
__global__ void __launch_bounds__(kT) k_transform_at(const void* psi, GridDesc g, int n_fields, const double* kappa,
                                                     cpx<double>* part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<double>* ph = reinterpret_cast<cpx<double>*>(smem_raw);  // nx + ny + nz phases
  __shared__ cpx<double> red[kT / 32][4];
  const int f = blockIdx.y;
  const int nt = g.n[0] + g.n[1] + g.n[2];
  for (int i = threadIdx.x; i < nt; i += blockDim.x) {
    int axis = 0, j = i;
    while (j >= g.n[axis]) { j -= g.n[axis]; ++axis; }
    const double xc = g.n[axis] > 1 ? g.x0[axis] + j * g.dx[axis] : 0.0;
    const double k = g.n[axis] > 1 ? kappa[3 * f + axis] : 0.0;
    double sn, cs;
    sincos(-k * xc, &sn, &cs);
    ph[i] = mk<double>(cs, sn);
  }
  __syncthreads();
  cpx<double> acc[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) acc[a] = mk<double>(0, 0);
  const size_t fo = (size_t)(f % n_fields) * 4 * g.N;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < g.N; j += gridDim.x * blockDim.x) {
    const int ix = j % g.n[0];
    const int iy = (j / g.n[0]) % g.n[1];
    const int iz = j / (g.n[0] * g.n[1]);
    const cpx<double> e = ph[ix] * ph[g.n[0] + iy] * ph[g.n[0] + g.n[1] + iz];
#pragma unroll
    for (int a = 0; a < 4; ++a) acc[a] = acc[a] + ld_d<Rin>(psi, fo + (size_t)a * g.N + j) * e;
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      acc[a].x += __shfl_down_sync(0xffffffffu, acc[a].x, off);
      acc[a].y += __shfl_down_sync(0xffffffffu, acc[a].y, off);
    }
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
#pragma unroll
    for (int a = 0; a < 4; ++a) red[wid][a] = acc[a];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    cpx<double> s = mk<double>(0, 0);
    for (int w = 0; w < kT / 32; ++w) s = s + red[w][threadIdx.x];
    part[((size_t)f * gridDim.x + blockIdx.x) * 4 + threadIdx.x] = s;
  }
}

// out[f][q] = scale * sum_b part[f][b][q], the parts added in order of b (deterministic).
template <typename T>
__global__ void k_sum_parts(const T* __restrict__ part, int nb, int width, double scale, T* out) {
  const int f = blockIdx.x;
  for (int q = threadIdx.x; q < width; q += blockDim.x) {
    T s{};
    for (int b = 0; b < nb; ++b) s = s + part[((size_t)f * nb + b) * width + q];
    out[(size_t)f * width + q] = scale * s;
  }
}

// Streaming multiprocessors of the device.
int sms() {
  static int nsm = 0;
  if (nsm == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess || nsm <= 0)
      nsm = 152;
  }
  return nsm;
}

// Blocks per field of a grid reduction: about four waves of the GPU, at least 8 elements a thread.
int reduction_blocks(size_t elems, int n_f) {
  const size_t by_size = (elems + 8 * kT - 1) / (8 * kT);
  const size_t by_gpu = (4 * (size_t)sms() + n_f - 1) / n_f;
  size_t nb = by_size < by_gpu ? by_size : by_gpu;
  return nb < 1 ? 1 : (int)nb;
}

template <typename Rin>
__global__ void __launch_bounds__(kT) k_norms(const void* psi, GridDesc g, double* part) {
  __shared__ double red[kT / 32];
  const int f = blockIdx.y;
  const size_t fo = (size_t)f * 4 * g.N;
  double acc = 0.0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (size_t)4 * g.N; i += (size_t)gridDim.x * blockDim.x) {
    const cpx<double> v = ld_d<Rin>(psi, fo + i);
    acc += v.x * v.x + v.y * v.y;
  }
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < kT / 32; ++w) s += red[w];
    part[(size_t)f * gridDim.x + blockIdx.x] = s;
  }
}

constexpr size_t kFftSmem = 200 * 1024;

swf_status ensure_smem() {
  static std::atomic<bool> ready[64];
  const int dv = dev_slot();
  if (ready[dv].load(std::memory_order_acquire)) return SWF_OK;
  cudaError_t e = cudaFuncSetAttribute(k_fft_axis<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFftSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_fft_axis<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFftSmem);
  if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute(k_fft_axis)");
  ready[dv].store(true, std::memory_order_release);
  return SWF_OK;
}

}  // namespace

swf_status transform_fields(swf_ctx* ctx, const GridDesc& g, int n_f, swf_precision prec, const void* psi,
                            double2* spec, cudaStream_t st, bool raw) {
  swf_status s = ensure_smem();
  if (s != SWF_OK) return s;
  cpx<double>* d = reinterpret_cast<cpx<double>*>(spec);
  int axes[3], nax = 0;
  for (int a = 0; a < 3; ++a)
    if (g.n[a] > 1) axes[nax++] = a;
  if (nax == 0) axes[nax++] = 0;  // a single point: the conversion alone
  for (int k = 0; k < nax; ++k) {
    const int axis = axes[k], na = g.n[axis];
    RadixPlan pl;
    if (!make_pass_plan(na, &pl)) {
      set_error("grid size must factor into 2, 3 and 5");
      return SWF_EINVAL;
    }
    const void* tw = nullptr;
    if ((s = twiddles(ctx, na, 1, &tw)) != SWF_OK) return s;
    // lines per block: about 256 threads; eight neighbouring x columns (128 bytes) at most
    const int tpl = pass_threads(pl, 1);
    const int nrows = axis == 0 ? g.n[1] * g.n[2] : g.n[0];
    const int ld = padded_len<double>(na) | 1;
    int nl = std::max(1, std::min(std::min(axis == 0 ? 64 : 8, kT / tpl), nrows));
    while (nl > 1 && (size_t)2 * nl * ld * 16 > kFftSmem) --nl;
    const int blocks = axis == 0 ? (nrows + nl - 1) / nl : (nrows + nl - 1) / nl * (axis == 1 ? g.n[2] : g.n[1]);
    const dim3 grid(blocks, n_f * 4);
    const size_t smem = (size_t)2 * nl * ld * 16;
    const bool last = k + 1 == nax;
    const double scale = last && !raw ? g.dx[0] * g.dx[1] * g.dx[2] : 1.0;
    const int sign = last && !raw ? 1 : 0;
    ProfScope ps(ctx, "k_fft_axis", st);
    if (k == 0 && prec == SWF_C64)
      k_fft_axis<float><<<grid, nl * tpl, smem, st>>>((const cpx<float>*)psi, d, g, axis, pl, (const cpx<double>*)tw, nl,
                                                      ld, tpl, scale, sign);
    else
      k_fft_axis<double><<<grid, nl * tpl, smem, st>>>(k == 0 ? (const cpx<double>*)psi : d, d, g, axis, pl,
                                                       (const cpx<double>*)tw, nl, ld, tpl, scale, sign);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "transform kernels");
  return SWF_OK;
}

swf_status c_spectrum(swf_ctx* ctx, const GridDesc& g, int n_f, const FieldDesc* fd_host, double t_in,
                      const double2* spec, double2* c_out, double* prob, cudaStream_t st) {
  void* pfd = nullptr;
  swf_status s = ws_get(ctx, "proj.fd", sizeof(FieldDesc) * n_f, &pfd);
  if (s != SWF_OK) return s;
  cudaError_t e = cudaMemcpyAsync(pfd, fd_host, sizeof(FieldDesc) * n_f, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_status(e, "upload field descriptors");
  // fields per thread: as many as leave about two blocks per SM
  const int nb = (g.N + kT - 1) / kT;
  const int chunks = std::max(1, std::min(n_f, 2 * sms() / nb));
  const int fc = (n_f + chunks - 1) / chunks;
  ProfScope ps(ctx, "k_c_spectrum", st);
  k_c_spectrum<<<dim3(nb, (n_f + fc - 1) / fc), kT, 0, st>>>((const cpx<double>*)spec, (const FieldDesc*)pfd, g, n_f, fc,
                                                             t_in, (cpx<double>*)c_out, prob);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "c-spectrum kernel");
  return SWF_OK;
}

swf_status transform_at(swf_ctx* ctx, const GridDesc& g, int n_f, swf_precision prec, const void* psi,
                        const double* kappa_host, double2* out, cudaStream_t st, int n_fields) {
  if (n_fields < 1) n_fields = n_f;
  const size_t sm = (size_t)(g.n[0] + g.n[1] + g.n[2]) * sizeof(cpx<double>);
  const int nb = reduction_blocks(g.N, n_fields);
  // the parts of a chunk of entries, then its wave vectors: a chunk is a multiple of the fields
  const size_t parts = sizeof(cpx<double>) * 4 * (size_t)nb;
  int chunk;
  void* part = nullptr;
  swf_status s = ws_chunk(ctx, "proj.part", parts + 3 * sizeof(double), n_fields, n_f, &chunk, &part);
  if (s != SWF_OK) return s;
  double* pk = reinterpret_cast<double*>((unsigned char*)part + parts * chunk);
  cudaError_t e;
  for (int e0 = 0; e0 < n_f; e0 += chunk) {
    const int n = std::min(chunk, n_f - e0);
    e = cudaMemcpyAsync(pk, kappa_host + 3 * (size_t)e0, sizeof(double) * 3 * n, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return cuda_status(e, "upload wave vectors");
    {
      ProfScope ps(ctx, "k_transform_at", st);
      if (prec == SWF_C64) k_transform_at<float><<<dim3(nb, n), kT, sm, st>>>(psi, g, n_fields, pk, (cpx<double>*)part);
      else k_transform_at<double><<<dim3(nb, n), kT, sm, st>>>(psi, g, n_fields, pk, (cpx<double>*)part);
    }
    ProfScope ps(ctx, "k_sum_parts", st);
    k_sum_parts<cpx<double>><<<n, 32, 0, st>>>((const cpx<double>*)part, nb, 4, g.dx[0] * g.dx[1] * g.dx[2],
                                               (cpx<double>*)out + 4 * (size_t)e0);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "direct transform kernel");
  return SWF_OK;
}

swf_status field_norms(swf_ctx* ctx, const GridDesc& g, int n_f, swf_precision prec, const void* psi,
                       double* out, cudaStream_t st) {
  const int nb = reduction_blocks((size_t)4 * g.N, n_f);
  void* part = nullptr;
  swf_status s = ws_get(ctx, "proj.norm_part", sizeof(double) * (size_t)nb * n_f, &part);
  if (s != SWF_OK) return s;
  {
    ProfScope ps(ctx, "k_norms", st);
    if (prec == SWF_C64) k_norms<float><<<dim3(nb, n_f), kT, 0, st>>>(psi, g, (double*)part);
    else k_norms<double><<<dim3(nb, n_f), kT, 0, st>>>(psi, g, (double*)part);
  }
  {
    ProfScope ps(ctx, "k_sum_parts", st);
    k_sum_parts<double><<<n_f, 32, 0, st>>>((const double*)part, nb, 1, g.dx[0] * g.dx[1] * g.dx[2], (double*)out);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "norm kernel");
  return SWF_OK;
}

}  // namespace swf
