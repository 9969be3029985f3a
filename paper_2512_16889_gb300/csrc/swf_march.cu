// Time march of the scattered wave (Sec. II, Eq. 6; Sec. II.A) on the GPU.
//
// Right-hand side, per field f and stage value Y:
//     k = -i [ H0 Y + V(t, x) (Y + psi_b(t, x)) ]
// with H0 applied per Fourier mode (Eq. 10).  One evaluation is a chain of line passes over
// the planar state [f][4][z][y][x]:
//   x pass:             Y = y + h sum_j a_ij k_j (stage combine, Dormand-Prince), the local term
//                       Z = -i V (Y + psi_b) stashed in the output slot, forward x-FFT;
//   y and z passes:     forward FFT along the axis; on the last axis -i H0(kappa)/N and the
//                       inverse FFT;
//   the next x pass:    inverse x-FFT and k = (that) + Z, before its own evaluation's work.
// Complex64 lengths with line kernels (swf_line.cuh) transform in registers; complex128 and the other
// lengths run on the small-radix passes (k_xpass, k_mid).
// Gauge field and background are analytic and evaluated on the fly from per-field 1D tables
// (every field kind is a product of a time factor and one factor per axis).
#include <type_traits>
#include <atomic>
#include <algorithm>
#include <cmath>
#include <map>
#include <vector>
#include <cstdio>
#include <cstring>

#include "swf_line.cuh"
#include "swf_pass.cuh"

namespace swf {

// ---------------------------------------------------------------- Dormand-Prince 5(4) tableau
// Dormand & Prince (1980); first-same-as-last: the 7th stage value is the new state.
static const double DP_C[7] = {0.0, 1.0 / 5, 3.0 / 10, 4.0 / 5, 8.0 / 9, 1.0, 1.0};
static const double DP_A[7][6] = {
    {0, 0, 0, 0, 0, 0},
    {1.0 / 5, 0, 0, 0, 0, 0},
    {3.0 / 40, 9.0 / 40, 0, 0, 0, 0},
    {44.0 / 45, -56.0 / 15, 32.0 / 9, 0, 0, 0},
    {19372.0 / 6561, -25360.0 / 2187, 64448.0 / 6561, -212.0 / 729, 0, 0},
    {9017.0 / 3168, -355.0 / 33, 46732.0 / 5247, 49.0 / 176, -5103.0 / 18656, 0},
    {35.0 / 384, 0, 500.0 / 1113, 125.0 / 192, -2187.0 / 6784, 11.0 / 84}};

__global__ void k_clock_set(MarchClock* c, double t_out, double h) {
  c->t_out = t_out;
  c->h = h;
  c->step = 0;
  c->pad = 0;
}

__global__ void k_clock_advance(MarchClock* c, int by) {
  chain_wait();
  c->step += by;
}

// What a call's passes read, computed in FP64 and rounded once to the march precision: the fields' factors
// and background phases per axis, the mode momenta and, where the call knows its first evaluation's time
// (ft), that evaluation's time factors.  A single field comes with the launch (one; stored at fd), which
// saves an upload from pageable memory.  Chains of FP64 instructions bound it (an exponential, a sine), so
// every kind of entry has its own blocks.  A right-hand side on 64 x 64 takes 38 us; with the momenta as
// a second launch (6 us), an upload of the field and the time factors left to the x pass (which took 12
// instead of 10 us) it took 45.
constexpr int kTableThreads = 64;
template <typename R>
struct TableArgs {
  FieldDesc one;
  FieldDesc* fd;
  int single;
  GridDesc g;
  R* greal;
  cpx<R>* gcplx;
  R* kap;
  double t;
  R* ft;
  cpx<R>* tf;
  int nb, nfb;  // blocks per kind of entry, blocks of time factors (the phase has one more)
};
template <typename R>
__global__ void __launch_bounds__(kTableThreads) k_tables(const __grid_constant__ TableArgs<R> T) {
  chain_release();
  const GridDesc& g = T.g;
  const int f = blockIdx.y, nt = g.n[0] + g.n[1] + g.n[2];
  const FieldDesc& F = T.single ? T.one : T.fd[f];
  const int what = min((int)blockIdx.x / T.nb, 3), i = (blockIdx.x - what * T.nb) * kTableThreads + threadIdx.x;
  if (what == 3) {
    const int iy = i;
    if ((int)blockIdx.x < 3 * T.nb + T.nfb) {
      if (iy < (F.kind == SWF_FIELD_PULSE_GAUSS ? g.n[1] : 1))
        T.ft[(size_t)f * g.n[1] + iy] = (R)field_time_factor(F, T.t, g.n[1] > 1 ? g.x0[1] + iy * g.dx[1] : 0.0);
    } else if (threadIdx.x == 0) {
      double sn, cs;
      sincos(F.tsign * F.e0 * T.t, &sn, &cs);
      T.tf[f] = mk<R>((R)cs, (R)sn);
    }
    return;
  }
  if (i >= nt) {
    if (what == 1 && i < nt + 4)
      T.gcplx[(size_t)f * (nt + 4) + i] = mk<R>((R)F.w[2 * (i - nt)], (R)F.w[2 * (i - nt) + 1]);
    return;
  }
  int axis = 0, j = i;
  while (j >= g.n[axis]) { j -= g.n[axis]; ++axis; }
  const double xc = g.n[axis] > 1 ? g.x0[axis] + j * g.dx[axis] : 0.0;
  if (what == 0) {
    T.greal[(size_t)f * nt + i] = (R)axis_factor(F, axis, xc);
    if (T.single && i == 0) *T.fd = T.one;
  } else if (what == 1) {
    double sn, cs;
    sincos(F.pmom[axis] * xc, &sn, &cs);
    T.gcplx[(size_t)f * (nt + 4) + i] = mk<R>((R)cs, (R)sn);
  } else if (f == 0) {
    T.kap[i] = g.n[axis] > 1 ? (R)mode_kappa(j, g.n[axis], g.L[axis]) : (R)0;
  }
}
// The tables of F fields (descriptors in host memory: copied with the launch if there is one, else
// uploaded to A's) into A's buffers; t: the first evaluation's time, if its factors are wanted.
template <typename R>
static cudaError_t fill_tables(const StageArgs<R>& A, int F, const FieldDesc* fd_host, const double* t, cudaStream_t st) {
  TableArgs<R> T;
  T.one = fd_host[0];
  T.fd = const_cast<FieldDesc*>(A.fd);
  T.single = F == 1;
  T.g = A.g;
  T.greal = const_cast<R*>(A.greal);
  T.gcplx = const_cast<cpx<R>*>(A.gcplx);
  T.kap = const_cast<R*>(A.kap);
  T.t = t ? *t : 0.0;
  T.ft = t ? A.ft : nullptr;
  T.tf = A.tf;
  T.nb = (A.g.n[0] + A.g.n[1] + A.g.n[2] + 4 + kTableThreads - 1) / kTableThreads;
  T.nfb = T.ft ? (A.g.n[1] + kTableThreads - 1) / kTableThreads : 0;
  if (!T.single) {
    const cudaError_t e = cudaMemcpyAsync(T.fd, fd_host, sizeof(FieldDesc) * F, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
  }
  k_tables<R><<<dim3(3 * T.nb + (T.ft ? T.nfb + 1 : 0), F), kTableThreads, 0, st>>>(T);
  return cudaSuccess;  // a launch error stays for the caller's cudaGetLastError
}

// ---------------------------------------------------------------- pass kernels
static const size_t kPassSmemMax = 200 * 1024;  // the most shared memory that a pass may take

// Grids with x as the only non-trivial axis: the whole right-hand side of field blockIdx.y in one launch
// and block.  A thread takes all four components of its sites, so that their loads are in flight together,
// and what the sites share of the background is formed once: an evaluation of one field of 512 points
// takes 15 us in complex64 and 65 in complex128, 18 and 77 with a component a thread (and, in complex128,
// small radices for every length).
template <typename R>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 4 : 2) k_first(StageArgs<R> A, int ld) {
  if (A.ctl && A.ctl->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<R>* buf = reinterpret_cast<cpx<R>*>(smem_raw);
  cpx<R>* buf2 = buf + 4 * ld;
  __shared__ R s_ft;
  __shared__ cpx<R> s_tf;
  const int f = blockIdx.y, nx = A.g.n[0];
  const size_t N = A.g.N, fo = (size_t)f * 4 * N;
  row_factors(A, false, f, 0, 1, &s_ft, &s_tf);
  __syncthreads();
  const bool ff = sizeof(R) == 4 && A.ylo && A.write_y;
  const FieldDesc* F = A.fd + f;
  const int acomp = F->acomp, nt = nx + 2;
  const R* __restrict__ gx = A.greal + (size_t)f * nt;
  const cpx<R>* __restrict__ ex = A.gcplx + (size_t)f * (nt + 4);
  const R ar = s_ft * gx[nx] * gx[nx + 1];
  cpx<R> br[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) br[c] = ex[nt + c] * (s_tf * (ex[nx] * ex[nx + 1]));
  for (int x = threadIdx.x; x < nx; x += blockDim.x) {
    const cpx<R> e = ex[x];
    const R a = ar * gx[x];
    cpx<R> v[4];
    combine_sites<R, 4>(A, A.nterm, ff, fo + x, A.g.N, v);
    finish_sites<R, 4>(A, ff, fo + x, A.g.N, v);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      A.kout[fo + source_component(acomp, c) * N + x] = source_term<R>(v[c], br[c], e, a, source_rotation<R>(acomp, c));
      buf[c * ld + pad<R>(x)] = v[c];
    }
  }
  __syncthreads();
  cpx<R>* res = fft_pp<R>(buf, buf2, ld, 4, A.plan[0], false, A.tw[0]);
  const R kx0 = (R)F->K[0], ky = (R)F->K[1], kz = (R)F->K[2];
  for (int x = threadIdx.x; x < nx; x += blockDim.x) {
    cpx<R>* l = res + pad<R>(x);
    cpx<R> v[4] = {l[0], l[ld], l[2 * ld], l[3 * ld]};
    h0_mi<R>(v, nx > 1 ? A.kap[x] : kx0, ky, kz, A.inv_n);
#pragma unroll
    for (int c = 0; c < 4; ++c) l[c * ld] = v[c];
  }
  __syncthreads();
  res = fft_pp<R>(res, res == buf ? buf2 : buf, ld, 4, A.plan[0], true, A.tw[0]);
  for (int x = threadIdx.x; x < nx; x += blockDim.x) {
    cpx<R>* k = A.kout + fo + x;
    cpx<R> v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = k[c * N];
#pragma unroll
    for (int c = 0; c < 4; ++c) k[c * N] = v[c] + res[c * ld + pad<R>(x)];
  }
}

// ---- passes of small radices (2, 3, 4, 5), for every length and both precisions
// The same two kinds of passes as the register line kernels (swf_line.cuh), for complex128 and for
// lengths that have no line kernel: the first and the last butterfly of a transform work in the
// registers of the thread that loads, stores or uses the values, those between run in shared memory.
// FP64 decides the shape: the unit of an SM quarter takes 64 cycles per warp instruction, so a thread
// holds few values (one radix-4 butterfly) and a line is spread over n/4 threads, which loads all
// quarters of all SMs evenly even for a single 128 x 128 field.  The operations are those of 16 x 8
// butterflies within a few percent (22 per point).  One 128 x 128 complex128 field, per evaluation: 56
// us with 16 x 8 in shared memory, 50 us with 8 x 16 in registers (8 to 16 values a thread), 33 us here.
// x pass (k_xline's work; R0: the site side's radix), tpl threads per line.
template <typename R, int R0>
__global__ void __launch_bounds__(kPassThreads, 1)
k_xpass(const __grid_constant__ StageArgs<R> P, const __grid_constant__ StageArgs<R> A, int rows, int ld, int tpl,
        int flags) {
  chain_wait();
  chain_release();
  if (A.ctl && A.ctl->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ R s_ft[64];
  __shared__ cpx<R> s_tf;
  const RadixPlan& pl = A.plan[0];
  const int nx = pl.n, nb = nx / R0, rl = end_radix(pl, false);
  const size_t N = A.g.N;
  const int f = blockIdx.y, row0 = blockIdx.x * rows;
  const int line = threadIdx.x / tpl, g = threadIdx.x - line * tpl;
  const int c = line & 3, j = line >> 2, row = row0 + j;
  const bool ok = line < 4 * rows && row < A.nrows;
  const size_t gl = ((size_t)f * 4 + c) * N + (size_t)row * nx;  // the line
  cpx<R>* a = reinterpret_cast<cpx<R>*>(smem_raw);
  cpx<R>* b2 = a + 4 * rows * ld;
  const cpx<R>* __restrict__ tw = A.tw[0];
  const bool last = flags & XL_LAST, first = flags & XL_FIRST, one = pl.npass < 2;
  if (first) row_factors(A, flags & XL_FACTORS, f, row0, rows, s_ft, &s_tf);
  const bool ff = sizeof(R) == 4 && A.ylo && A.write_y;
  const int nold = A.nterm - ((flags & XL_REGK) ? 1 : 0);
  cpx<R> v[R0];
  if (first && ok && g < nb) combine_sites<R, R0>(A, nold, ff, gl + g, nb, v);  // overlaps the loads of T
  if (last) {
    if (ok)
      with_radix(rl, [&](auto rc) {
        constexpr int RL = decltype(rc)::value;
        const int nm = nx / RL;
        for (int b = g; b < nm; b += tpl) {
          cpx<R> m[RL];
#pragma unroll
          for (int q = 0; q < RL; ++q) m[q] = P.T[gl + b + q * nm];
          first_butterfly<R, RL>(m, b, true, a + line * ld);
        }
      });
    __syncthreads();
    cpx<R>* cur = middle_passes<R>(a, b2, ld, 4 * rows, pl, true, tw);
    if (cur != a) {
      b2 = a;
      a = cur;
    }
  } else {
    __syncthreads();  // the time factors
  }
  if (ok)
    for (int b = g; b < nb; b += tpl) {
      if (first && b != g) combine_sites<R, R0>(A, nold, ff, gl + b, nb, v);
      if (last) {
        cpx<R> r[R0];
        last_butterfly<R, R0>(a + line * ld, b, nx, one, true, tw, r);
        close_sites<R, R0>(P, gl + b, nb, r);
        if (first && (flags & XL_REGK)) {
          const R co = A.ctl ? (R)(A.coef[nold] * A.ctl->h) : A.coef_r[nold];
#pragma unroll
          for (int q = 0; q < R0; ++q) v[q] = v[q] + co * r[q];
        }
      }
      if (first) {
        open_sites<R, R0>(A, ff, gl + b, b, nb, f, c, row, s_ft[j], s_tf, v);
        first_butterfly<R, R0>(v, b, false, b2 + line * ld);
      }
    }
  if (!first) return;
  __syncthreads();
  const cpx<R>* cur = middle_passes<R>(b2, a, ld, 4 * rows, pl, false, tw);
  if (ok)
    with_radix(rl, [&](auto rc) {
      constexpr int RL = decltype(rc)::value;
      const int nm = nx / RL;
      for (int b = g; b < nm; b += tpl) {
        cpx<R> m[RL];
        last_butterfly<R, RL>(cur + line * ld, b, nx, one, false, tw, m);
#pragma unroll
        for (int q = 0; q < RL; ++q) A.T[gl + b + q * nm] = m[q];
      }
    });
}

// y or z pass (k_line's work): lines along `axis` of TX = 2^lgtx x columns, tpl threads per line, the
// four components of a mode in one warp.
template <typename R>
__global__ void __launch_bounds__(kPassThreads, 1)
k_mid(const __grid_constant__ StageArgs<R> A, int axis, int lgtx, int ld, int tpl, int flags) {
  chain_wait();
  chain_release();
  if (A.ctl && A.ctl->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nx = A.g.n[0], ny = A.g.n[1], nz = A.g.n[2];
  const int f = blockIdx.y;
  const int TX = 1 << lgtx, ntx = (nx + TX - 1) >> lgtx;
  const int other = axis == 1 ? nz : ny;
  if (blockIdx.x >= ntx * other) {
    coming_factors(A, f);
    return;
  }
  const RadixPlan& pl = A.plan[axis];
  const int na = pl.n, r0 = end_radix(pl, true), rl = end_radix(pl, false);
  const int xt = blockIdx.x % ntx, o = blockIdx.x / ntx;  // o: z index (axis 1) or y index (axis 2)
  const int t = threadIdx.x & (TX - 1), c = (threadIdx.x >> lgtx) & 3, g = threadIdx.x >> (lgtx + 2);
  const int x = xt * TX + t;
  const bool ok = x < nx && g < tpl;
  const size_t base = (axis == 1 ? (size_t)o * nx * ny : (size_t)o * nx) + ((size_t)f * 4 + c) * A.g.N + x;
  const size_t stride = axis == 1 ? (size_t)nx : (size_t)nx * ny;
  cpx<R>* a = reinterpret_cast<cpx<R>*>(smem_raw);
  cpx<R>* b2 = a + 4 * TX * ld;
  const int lo = (c * TX + t) * ld;
  const cpx<R>* __restrict__ tw = A.tw[axis];
  const bool one = pl.npass < 2;
  const bool fwd = flags & LN_FWD, h0 = flags & LN_H0, inv = flags & LN_INV;
  if (fwd) {
    if (ok)
      with_radix(r0, [&](auto rc) {
        constexpr int R0 = decltype(rc)::value;
        const int nb = na / R0;
        for (int b = g; b < nb; b += tpl) {
          cpx<R> v[R0];
#pragma unroll
          for (int q = 0; q < R0; ++q) v[q] = A.T[base + (size_t)(b + q * nb) * stride];
          first_butterfly<R, R0>(v, b, false, a + lo);
        }
      });
    __syncthreads();
    cpx<R>* cur = middle_passes<R>(a, b2, ld, 4 * TX, pl, false, tw);
    if (cur != a) {
      b2 = a;
      a = cur;
    }
  }
  with_radix(rl, [&](auto rc) {
    constexpr int RL = decltype(rc)::value;
    const int nm = na / RL, rounds = (nm + tpl - 1) / tpl;
    for (int k = 0; k < rounds; ++k) {
      const int b = g + k * tpl;
      const bool mode = ok && b < nm;
      cpx<R> m[RL];
#pragma unroll
      for (int q = 0; q < RL; ++q) m[q] = mk<R>(0, 0);
      if (mode) {
        if (fwd) {
          last_butterfly<R, RL>(a + lo, b, na, one, false, tw, m);
        } else {
#pragma unroll
          for (int q = 0; q < RL; ++q) m[q] = A.T[base + (size_t)(b + q * nm) * stride];
        }
        if (h0 && A.yspec) {
#pragma unroll
          for (int q = 0; q < RL; ++q) A.yspec[base + (size_t)(b + q * nm) * stride] = m[q];
        }
      }
      if (h0) h0_modes<R, RL>(A, axis, lgtx, f, c, x, o, b, nm, mode, m);
      if (mode) {
        if (inv) {
          first_butterfly<R, RL>(m, b, true, b2 + lo);
        } else {
#pragma unroll
          for (int q = 0; q < RL; ++q) A.T[base + (size_t)(b + q * nm) * stride] = m[q];
        }
      }
    }
  });
  if (!inv) return;
  __syncthreads();
  const cpx<R>* cur = middle_passes<R>(b2, a, ld, 4 * TX, pl, true, tw);
  if (ok)
    with_radix(r0, [&](auto rc) {
      constexpr int R0 = decltype(rc)::value;
      const int nb = na / R0;
      for (int b = g; b < nb; b += tpl) {
        cpx<R> v[R0];
        last_butterfly<R, R0>(cur + lo, b, na, one, true, tw, v);
#pragma unroll
        for (int q = 0; q < R0; ++q) A.T[base + (size_t)(b + q * nb) * stride] = v[q];
      }
    });
}

// ---------------------------------------------------------------- host side
template <typename R> struct Prec;
template <> struct Prec<float> { static constexpr int is_double = 0; };
template <> struct Prec<double> { static constexpr int is_double = 1; };

static const int kThreads = 256;

// Radix plan of the line FFTs that run as a whole in shared memory (fft_pp: one-axis grids, the
// partial-integration integrand): radix 16 first, then the composite radices 20 and 12, then 8, 4,
// 2, 3, 5 (every length of the form 2^a 3^b 5^c).
static bool make_march_plan(int n, RadixPlan* pl) {
  pl->n = n;
  pl->npass = 0;
  int m = n;
  const int order[8] = {16, 20, 12, 8, 4, 2, 3, 5};
  for (int r : order)
    while (m % r == 0 && pl->npass < 12) {
      pl->rad[pl->npass++] = r;
      m /= r;
    }
  return m == 1;
}

// The plan of an axis: small radices, and where x is the only axis the composite radices of whole-line
// transforms in complex64 and, in complex128, for lines long enough that their few butterflies still give
// every quarter of the SM a warp (one field of 512 points 13.0 against 13.6 ms for 40 steps, of 384 10.5
// against 11.0; of 256 points 9.1 against 7.3 ms with small radices, and of lengths without a factor 16
// the small ones are the faster ones as well).  The plan depends on the length alone: a field has the same
// bits among any number of others.
template <typename R>
static bool make_line_plan(const GridDesc& g, int axis, RadixPlan* pl) {
  const int n = g.n[axis];
  const bool whole = g.n[1] == 1 && g.n[2] == 1 && (sizeof(R) == 4 || (n >= 384 && n % 16 == 0));
  return whole ? make_march_plan(n, pl) : make_pass_plan(n, pl);
}

// Streaming multiprocessors of the current device (cached per device).
static int sm_count() {
  static int cache[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
  if (cache[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 152;
    cache[dev] = n;
  }
  return cache[dev];
}

// Keys of the tuned shapes: pass kind, element size and the sizes that decide the launch.
static std::string tune_key(char kind, int esz, int a, int b, int c, long d) {
  char buf[96];
  std::snprintf(buf, sizeof buf, "%c/%d/%d/%d/%d/%ld", kind, esz, a, b, c, d);
  return buf;
}

static int tune_lookup(swf_ctx* ctx, const std::string& key, int fallback) {
  if (!ctx || !ctx->tune.on) return fallback;
  auto it = ctx->tune.best.find(key);
  return it == ctx->tune.best.end() ? fallback : it->second;
}

template <typename R, int... R0>
static cudaError_t xpass_attrs(std::integer_sequence<int, R0...>) {
  cudaError_t e = cudaSuccess;
  ((e = e != cudaSuccess ? e : cudaFuncSetAttribute(k_xpass<R, R0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPassSmemMax)), ...);
  return e;
}
template <typename R>
static swf_status set_smem_attrs() {
  // per device; several host threads may arrive at once, and setting the attributes twice is harmless
  static std::atomic<bool> done[64];
  const int dv = dev_slot();
  if (done[dv].load(std::memory_order_acquire)) return SWF_OK;
  cudaError_t e = cudaFuncSetAttribute(k_first<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPassSmemMax);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mid<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPassSmemMax);
  if (e == cudaSuccess) e = xpass_attrs<R>(std::integer_sequence<int, 1, 2, 3, 4, 5>());
  if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute(pass kernels)");
  done[dv].store(true, std::memory_order_release);
  return SWF_OK;
}

// ---- register line kernels (swf_line.cuh): host side.  Complex64 only: a thread of theirs holds 8 to
// 32 values, which FP64's rate turns into long serial chains on few SM quarters (one 128 x 128 field in
// complex128: 50 us per evaluation, 33 us with the small-radix passes).
const LineEntry<float>* find_line0_float(int n);
const LineEntry<float>* find_line1_float(int n);
const LineEntry<float>* find_line2_float(int n);
const LineEntry<float>* find_line3_float(int n);
const LineEntry<float>* find_line4_float(int n);

// The line kernels of length n (null: the small-radix passes take it).
template <typename R>
static const LineEntry<R>* line_entry(int n) {
  if constexpr (sizeof(R) == 8) {
    return nullptr;
  } else {
    for (auto* find : {find_line0_float, find_line1_float, find_line2_float, find_line3_float, find_line4_float})
      if (const LineEntry<float>* e = find(n)) return e;
    return nullptr;
  }
}

// The line kernels of an axis of a grid: null on a trivial axis and where x is the only axis (one
// launch does the whole evaluation).
template <typename R>
static const LineEntry<R>* line_of(const GridDesc& g, int axis) {
  if (g.n[1] == 1 && g.n[2] == 1) return nullptr;
  return g.n[axis] > 1 ? line_entry<R>(g.n[axis]) : nullptr;
}

// Rows per block of k_xline and log2 columns of k_line: at most this many fit a block.
template <typename R>
static int xline_max_rows(const LineEntry<R>* e) {
  return std::max(1, kXLineThreads / (4 * line_threads(e->r1, e->r2)));
}
template <typename R>
static int line_max_lg(const LineEntry<R>* e, int nx) {
  int lg = 3;
  while (lg > 0 && ((1 << lg) > nx || line_block(e->r1, e->r2, lg) > line_max_threads((int)sizeof(cpx<R>))))
    --lg;
  return lg;
}
template <typename R>
static size_t xline_smem(const LineEntry<R>* e, int rows) {
  return (size_t)4 * rows * xline_stride(e->r1, e->r2) * sizeof(cpx<R>);
}
template <typename R>
static size_t line_smem(const LineEntry<R>* e, int lg) {
  return ((size_t)4 << lg) * line_stride(e->r1, e->r2) * sizeof(cpx<R>);
}

// Sets the shared-memory limits of an entry's kernels (once per device) before their first launch.
template <typename R>
static swf_status line_ready(const LineEntry<R>* e) {
  static std::atomic<bool> done[64][513];
  const int dv = dev_slot();
  if (done[dv][e->n].load(std::memory_order_acquire)) return SWF_OK;
  cudaError_t r = cudaFuncSetAttribute(e->x, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)xline_smem<R>(e, xline_max_rows<R>(e)));
  if (r == cudaSuccess)
    r = cudaFuncSetAttribute(e->line, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)line_smem<R>(e, line_max_lg<R>(e, 8)));
  if (r != cudaSuccess) return cuda_status(r, "cudaFuncSetAttribute(line kernels)");
  done[dv][e->n].store(true, std::memory_order_release);
  return SWF_OK;
}

// Launch shape of an x pass (v rows per block) or of a y or z pass (2^v columns per block) of either
// kind.  A small-radix y or z tile of more lines than have a thread per butterfly gives its threads several
// butterflies each: with a thread per butterfly, lines of 243 points and more came one column at a time (8
// bytes of every 32), and one field of 486 x 486 took 37 us a y pass in complex64 (29 in tiles of more
// columns), of 512 x 512 189 us in complex128 (174).  The fixed rule keeps to a thread per butterfly, which
// spreads small grids further; the timed shapes include both.
struct PassShape {
  int thr = 0, ld = 0, tpl = 0;
  size_t smem = 0;
  bool fits = false, shared = false;  // shared: a thread does several butterflies where one line has more threads
};
template <typename R>
static PassShape x_shape(const StageArgs<R>& A, int rows) {
  PassShape S;
  if (A.ltw[0]) {
    const LineEntry<R>* e = line_entry<R>(A.g.n[0]);
    S.thr = 4 * rows * line_threads(e->r1, e->r2);
    S.smem = xline_smem<R>(e, rows);
    S.fits = rows <= xline_max_rows<R>(e);
  } else {
    S.ld = padded_len<R>(A.g.n[0]);
    S.tpl = pass_threads(A.plan[0], 4);
    S.thr = 4 * rows * S.tpl;
    S.smem = (size_t)8 * rows * S.ld * sizeof(cpx<R>);
    S.fits = rows <= 64 && S.thr <= kPassThreads && S.smem <= kPassSmemMax;
  }
  return S;
}
template <typename R>
static PassShape mid_shape(const StageArgs<R>& A, int axis, int lg) {
  PassShape S;
  const int nx = A.g.n[0];
  if (A.ltw[axis]) {
    const LineEntry<R>* e = line_entry<R>(A.g.n[axis]);
    S.thr = line_block(e->r1, e->r2, lg);
    S.smem = line_smem<R>(e, lg);
    S.fits = lg <= line_max_lg<R>(e, nx);
  } else {
    S.ld = padded_len<R>(A.g.n[axis]) | 1;  // neighbouring threads hold neighbouring lines
    S.tpl = pass_threads(A.plan[axis], 4 << lg);
    S.shared = S.tpl < pass_threads(A.plan[axis], 4);
    S.thr = ((4 << lg) * S.tpl + 31) & ~31;  // whole warps: the shuffles of H0 name all 32 lanes
    S.smem = ((size_t)8 << lg) * S.ld * sizeof(cpx<R>);
    S.fits = lg <= 3 && (lg == 0 || (1 << lg) <= nx) && S.thr <= kPassThreads && S.smem <= kPassSmemMax;
  }
  return S;
}

// The fixed rule: as many rows (columns) as a block takes, fewer on small grids (about two blocks per
// SM; at least 32 bytes of contiguous x per line in the y and z passes).
template <typename R>
static int x_rule(const StageArgs<R>& A, int F) {
  int rows = 1;
  while (2 * rows <= A.nrows && x_shape<R>(A, 2 * rows).fits &&
         (long)F * ((A.nrows + 2 * rows - 1) / (2 * rows)) >= 2L * sm_count())
    rows *= 2;
  return rows;
}
template <typename R>
static int mid_rule(const StageArgs<R>& A, int axis, long tiles) {
  const int nx = A.g.n[0], min_lg = sizeof(cpx<R>) == 8 ? 2 : 1;
  int lg = 3;
  for (; lg > 0; --lg) {
    const PassShape S = mid_shape<R>(A, axis, lg);
    if (S.fits && !S.shared) break;
  }
  while (lg > min_lg && tiles * ((nx + (1 << lg) - 1) >> lg) < 2L * sm_count()) --lg;
  return lg;
}

// Whether a pass's blocks may be set up before the pass in front of it has ended.  It pays where the passes
// are short and launched one by one (a right-hand side on 64 x 64 took 46 us with it, 52 us without), and
// in complex64 also in the steps replayed from a graph (one field of 64 x 64 2.17 against 2.37 ms for 40
// steps).  Replayed complex128 passes are launched plainly: blocks set up early go to the SMs that happen
// to be free, and where a pass has a block or two per SM, FP64 issue then lies on some SMs twice and on
// others not at all (four fields of 243 x 45: 25.7 ms, 21.2 launched plainly; of 405 x 30 23.3 and 18.7; two of
// 128 x 128 13.0 and 11.3).  The smallest grids lose 2 to 6 % by it (one field of 64 x 64 6.12 and 6.40 ms).
template <typename R>
static bool may_chain(cudaStream_t st) {
  if (sizeof(R) == 4) return true;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(st, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone;
}

// Launches a kernel of a march's chain, with `chained` so that its blocks may be set up before the kernel
// in front of it on the stream has ended (it waits for that itself: chain_wait).
template <typename... P, typename... Q>
static void launch_chained(bool chained, void (*kernel)(P...), dim3 grid, int thr, size_t smem, cudaStream_t st,
                           Q... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(thr);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = chained ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, P(args)...);  // an error stays for the caller's cudaGetLastError
}

// Launches the x pass `rows` rows per block (flags as k_xline's).
template <typename R>
static void run_x(const StageArgs<R>& P, const StageArgs<R>& A, int rows, int flags, int F, cudaStream_t st) {
  const PassShape S = x_shape<R>(A, rows);
  const dim3 grid((A.nrows + rows - 1) / rows, F);
  if (A.ltw[0]) {
    launch_chained(may_chain<R>(st), line_entry<R>(A.g.n[0])->x, grid, S.thr, S.smem, st, P, A, rows, flags);
    return;
  }
  auto* kernel = k_xpass<R, 1>;
  switch (end_radix(A.plan[0], true)) {
    case 4: kernel = k_xpass<R, 4>; break;
    case 2: kernel = k_xpass<R, 2>; break;
    case 3: kernel = k_xpass<R, 3>; break;
    case 5: kernel = k_xpass<R, 5>; break;
    default: break;
  }
  launch_chained(may_chain<R>(st), kernel, grid, S.thr, S.smem, st, P, A, rows, S.ld, S.tpl, flags);
}

// Launches the y or z pass, 2^lg columns per block; factors: with the blocks that compute the coming
// evaluation's time factors.
template <typename R>
static void run_mid(const StageArgs<R>& A, int axis, int lg, int flags, bool factors, int F, cudaStream_t st) {
  const PassShape S = mid_shape<R>(A, axis, lg);
  const int tiles = ((A.g.n[0] + (1 << lg) - 1) >> lg) * (axis == 1 ? A.g.n[2] : A.g.n[1]);
  const dim3 grid(tiles + (factors ? 1 : 0), F);
  const bool chained = may_chain<R>(st);
  if (A.ltw[axis]) launch_chained(chained, line_entry<R>(A.g.n[axis])->line, grid, S.thr, S.smem, st, A, axis, lg, flags);
  else launch_chained(chained, k_mid<R>, grid, S.thr, S.smem, st, A, axis, lg, S.ld, S.tpl, flags);
}

// Grids with x as the only axis: k_first with `thr` threads a block.
template <typename R>
static void run_only_x(const StageArgs<R>& A, int thr, int F, cudaStream_t st) {
  const int ld = padded_len<R>(A.g.n[0]);
  k_first<R><<<dim3(1, F), thr, (size_t)8 * ld * sizeof(cpx<R>), st>>>(A, ld);
}

// One x pass: closes evaluation P (close) and/or opens evaluation A (open) on the same rows; factors:
// the pass before this one computed A's time factors.  Where x is the only axis the launch is the
// whole evaluation.
template <typename R>
static swf_status launch_x(swf_ctx* ctx, const StageArgs<R>& P, const StageArgs<R>& A, bool close, bool open,
                           bool factors, int F, cudaStream_t st) {
  constexpr int esz = (int)sizeof(cpx<R>);
  const int nx = A.g.n[0];
  ProfScope ps(ctx, close ? (open ? "k_last_first" : "k_last") : "k_first", st);
  if (A.g.n[1] == 1 && A.g.n[2] == 1) {
    run_only_x<R>(A, tune_lookup(ctx, tune_key('x', esz, nx, A.nrows, 0, F), kThreads), F, st);
    return SWF_OK;
  }
  const int rows = tune_lookup(ctx, tune_key('X', esz, nx, A.nrows, 0, F), x_rule<R>(A, F));
  const bool regk = close && open && A.nterm > 0 && A.kin[A.nterm - 1] == P.kout;
  run_x<R>(P, A, rows,
           (close ? XL_LAST : 0) | (open ? XL_FIRST : 0) | (regk ? XL_REGK : 0) | (factors ? XL_FACTORS : 0), F, st);
  return SWF_OK;
}

// One y or z pass; last: the last one of its evaluation (it computes the coming time factors).
template <typename R>
static void launch_mid(swf_ctx* ctx, const StageArgs<R>& A, int axis, int fwd, int h0, int inv, bool last, int F,
                       cudaStream_t st) {
  constexpr int esz = (int)sizeof(cpx<R>);
  const long tiles = (long)(axis == 1 ? A.g.n[2] : A.g.n[1]) * F;
  ProfScope ps(ctx, "k_mid", st);
  const int lg = tune_lookup(ctx, tune_key('M', esz, axis * 8 + fwd * 4 + h0 * 2 + inv, A.g.n[axis], A.g.n[0], tiles),
                             mid_rule<R>(A, axis, tiles));
  run_mid<R>(A, axis, lg, (fwd ? LN_FWD : 0) | (h0 ? LN_H0 : 0) | (inv ? LN_INV : 0), last && A.ft, F, st);
}

// The y and z passes of one evaluation.
template <typename R>
static void launch_mids(swf_ctx* ctx, const StageArgs<R>& A, int F, cudaStream_t st) {
  const bool y = A.g.n[1] > 1, z = A.g.n[2] > 1;
  if (y && z) {
    launch_mid<R>(ctx, A, 1, 1, 0, 0, false, F, st);
    launch_mid<R>(ctx, A, 2, 1, 1, 1, false, F, st);
    launch_mid<R>(ctx, A, 1, 0, 0, 1, true, F, st);
  } else if (y || z) {
    launch_mid<R>(ctx, A, y ? 1 : 2, 1, 1, 1, true, F, st);
  }
}

// Launches one right-hand-side evaluation for F fields (ctx may be null: no profiling).
template <typename R>
static swf_status launch_eval(swf_ctx* ctx, const StageArgs<R>& A, int F, cudaStream_t st, bool factors = false) {
  swf_status s = launch_x<R>(ctx, A, A, false, true, factors, F, st);
  if (s != SWF_OK || (A.g.n[1] == 1 && A.g.n[2] == 1)) return s;
  launch_mids<R>(ctx, A, F, st);
  return launch_x<R>(ctx, A, A, true, false, false, F, st);
}

// An evaluation whose inverse x pass is left for the next launch (march chains with at least one
// non-trivial axis besides x): the forward x pass and the y/z passes of A.
template <typename R>
static swf_status launch_eval_open(swf_ctx* ctx, const StageArgs<R>& A, int F, cudaStream_t st) {
  const swf_status s = launch_x<R>(ctx, A, A, false, true, false, F, st);
  if (s == SWF_OK) launch_mids<R>(ctx, A, F, st);
  return s;
}

// Closes the open evaluation P and runs evaluation Nx with it in one x pass, then Nx's y/z passes.
template <typename R>
static swf_status launch_eval_chain(swf_ctx* ctx, const StageArgs<R>& P, const StageArgs<R>& Nx, int F,
                                    cudaStream_t st) {
  const swf_status s = launch_x<R>(ctx, P, Nx, true, true, Nx.ft != nullptr, F, st);
  if (s == SWF_OK) launch_mids<R>(ctx, Nx, F, st);
  return s;
}

// Closes the open evaluation P (its inverse x pass).
template <typename R>
static swf_status launch_eval_close(swf_ctx* ctx, const StageArgs<R>& P, int F, cudaStream_t st) {
  return launch_x<R>(ctx, P, P, true, false, false, F, st);
}

// The node that follows stage i (1..6, or 0 for the march's first evaluation) of step ls: the time
// factors its last y/z pass computes.
template <typename R>
static void set_next_node(StageArgs<R>* A, int ls, int i) {
  A->nls = i == 6 ? ls + 1 : ls;
  A->nc = DP_C[i == 6 ? 1 : i + 1];
}

// Times the candidate launch shapes of one evaluation's pass kernels (rows per block or tile
// width; with x as the only axis also 256- or 128-thread blocks) and records the fastest in ctx->tune (once per shape key).  B must be harmless to run repeatedly: it may write only
// T and its output slot, and read y and its input slots (the march calls this before its first
// evaluation, when those hold nothing yet).  The shape decides only which lines a block
// transforms, never the arithmetic of a line, so results do not depend on the choice.
template <typename R>
static swf_status autotune_eval(swf_ctx* ctx, const StageArgs<R>& B, int F, cudaStream_t st) {
  if (!ctx || !ctx->tune.on) return SWF_OK;
  constexpr int esz = (int)sizeof(cpx<R>);
  const int nx = B.g.n[0], ny = B.g.n[1], nz = B.g.n[2];
  const bool only_x = (ny == 1 && nz == 1);
  cudaEvent_t ev[2];
  if (cudaEventCreate(&ev[0]) != cudaSuccess) return cuda_status(cudaGetLastError(), "tuning events");
  if (cudaEventCreate(&ev[1]) != cudaSuccess) {
    cudaEventDestroy(ev[0]);
    return cuda_status(cudaGetLastError(), "tuning events");
  }
  swf_status status = SWF_OK;
  // time `launch` (one warm-up, then four back to back); +inf on a launch error
  auto timed = [&](auto&& launch) -> float {
    launch();
    cudaEventRecord(ev[0], st);
    for (int r = 0; r < 4; ++r) launch();
    cudaEventRecord(ev[1], st);
    cudaError_t e = cudaEventSynchronize(ev[1]);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
      status = cuda_status(e, "tuning launches");
      return 3.4e38f;
    }
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ev[0], ev[1]);
    return ms;
  };
  if (only_x) {
    const std::string key = tune_key('x', esz, nx, B.nrows, 0, F);
    if (!ctx->tune.best.count(key)) {
      int best = kThreads;
      float tbest = 3.4e38f;
      for (int thr = kThreads; thr >= kThreads / 2 && status == SWF_OK; thr /= 2) {
        const float t = timed([&] { run_only_x<R>(B, thr, F, st); });
        if (t < tbest) { tbest = t; best = thr; }
      }
      if (status == SWF_OK) ctx->tune.best[key] = best;
    }
  } else {
    const std::string key = tune_key('X', esz, nx, B.nrows, 0, F);
    if (!ctx->tune.best.count(key)) {
      int best = 1;
      float tbest = 3.4e38f;
      for (int rows = 1; (rows == 1 || (rows <= B.nrows && x_shape<R>(B, rows).fits)) && status == SWF_OK; rows *= 2) {
        const float t = timed([&] { run_x<R>(B, B, rows, XL_LAST | XL_FIRST | (B.ft ? XL_FACTORS : 0), F, st); });
        if (t < tbest) { tbest = t; best = rows; }
      }
      if (status == SWF_OK) ctx->tune.best[key] = best;
    }
    const int one[1][4] = {{ny > 1 ? 1 : 2, 1, 1, 1}};
    const int three[3][4] = {{1, 1, 0, 0}, {2, 1, 1, 1}, {1, 0, 0, 1}};
    const bool both = ny > 1 && nz > 1;
    for (int ci = 0; ci < (both ? 3 : 1) && status == SWF_OK; ++ci) {
      const int* cb = both ? three[ci] : one[0];
      const int axis = cb[0];
      const std::string mkey = tune_key('M', esz, axis * 8 + cb[1] * 4 + cb[2] * 2 + cb[3], B.g.n[axis], nx,
                                        (long)(axis == 1 ? nz : ny) * F);
      if (ctx->tune.best.count(mkey)) continue;
      int best = 0;
      float tbest = 3.4e38f;
      for (int lg = 3; lg >= 0 && status == SWF_OK; --lg) {
        if (!mid_shape<R>(B, axis, lg).fits) continue;
        const float t = timed([&] {
          run_mid<R>(B, axis, lg, (cb[1] ? LN_FWD : 0) | (cb[2] ? LN_H0 : 0) | (cb[3] ? LN_INV : 0), false, F, st);
        });
        if (t < tbest) { tbest = t; best = lg; }
      }
      if (status == SWF_OK) ctx->tune.best[mkey] = best;
    }
  }
  cudaEventDestroy(ev[0]);
  cudaEventDestroy(ev[1]);
  return status;
}

template <typename R>
static swf_status prepare_args(swf_ctx* ctx, const GridDesc& g, int F, const FieldDesc* fd_host,
                               StageArgs<R>* A, const char* tag, cudaStream_t st, const double* t_first = nullptr) {
  swf_status s = set_smem_attrs<R>();
  if (s != SWF_OK) return s;
  std::memset(A, 0, sizeof(*A));
  A->g = g;
  A->nrows = g.n[1] * g.n[2];
  for (int a = 0; a < 3; ++a) {
    if (!make_line_plan<R>(g, a, &A->plan[a])) {
      set_error("grid size must factor into 2, 3 and 5");
      return SWF_EINVAL;
    }
    const void* tw = nullptr;
    s = twiddles(ctx, g.n[a], Prec<R>::is_double, &tw);
    if (s != SWF_OK) return s;
    A->tw[a] = reinterpret_cast<const cpx<R>*>(tw);
    if (const LineEntry<R>* le = line_of<R>(g, a)) {
      if ((s = line_ready<R>(le)) != SWF_OK) return s;
      if ((s = twiddles(ctx, g.n[a], Prec<R>::is_double, &tw, le->r2)) != SWF_OK) return s;
      A->ltw[a] = reinterpret_cast<const cpx<R>*>(tw);
    }
  }
  const int nt = g.n[0] + g.n[1] + g.n[2];
  if (g.n[1] > 1 || g.n[2] > 1) {  // the last y/z pass computes the x pass's time factors
    void *pft = nullptr, *ptf = nullptr;
    if ((s = ws_get(ctx, std::string(tag) + ".ft", sizeof(R) * F * g.n[1], &pft)) != SWF_OK) return s;
    if ((s = ws_get(ctx, std::string(tag) + ".tf", sizeof(cpx<R>) * F, &ptf)) != SWF_OK) return s;
    A->ft = (R*)pft;
    A->tf = (cpx<R>*)ptf;
  }
  void *pfd = nullptr, *pgr = nullptr, *pgc = nullptr;
  std::string t(tag);
  if ((s = ws_get(ctx, t + ".fd", sizeof(FieldDesc) * F, &pfd)) != SWF_OK) return s;
  if ((s = ws_get(ctx, t + ".greal", sizeof(R) * F * nt, &pgr)) != SWF_OK) return s;
  if ((s = ws_get(ctx, t + ".gcplx", sizeof(cpx<R>) * F * (nt + 4), &pgc)) != SWF_OK) return s;
  void* pkap = nullptr;
  if ((s = ws_get(ctx, t + ".kap", sizeof(R) * nt, &pkap)) != SWF_OK) return s;
  A->fd = (const FieldDesc*)pfd;
  A->greal = (const R*)pgr;
  A->gcplx = (const cpx<R>*)pgc;
  A->kap = (const R*)pkap;
  A->inv_n = (R)(1.0 / (double)g.N);
  ProfScope ps(ctx, "k_tables", st);
  const cudaError_t e = fill_tables<R>(*A, F, fd_host, t_first, st);
  if (e != cudaSuccess) return cuda_status(e, "upload field descriptors");
  return SWF_OK;
}

// `pairs` repetitions of two Dormand-Prince steps recorded by record(st) (launches only), each followed
// by advancing the march clock by two steps.  Unless kernel timing is on or st is the legacy default
// stream, the pair is captured once into a CUDA graph and replayed: one launch per two steps instead
// of one per kernel.  The slots rotate with period two, so the recorded pointers repeat; the stage
// times come from the device clock.  prepare() captures, launch() queues one repetition, finish()
// waits for the replays and releases the graph.
struct StepPairs {
  cudaStream_t st = nullptr;
  cudaGraphExec_t exec = nullptr;
  long long per_pair = 0;

  template <typename Rec>
  swf_status prepare(swf_ctx* ctx, cudaStream_t stream, MarchClock* clk, Rec&& record) {
    st = stream;
    if (ctx->prof.on || st == 0 || !ctx->use_graphs) return SWF_OK;
    const long long l0 = ctx->prof.launches;
    if (cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();
      return SWF_OK;
    }
    const swf_status s = record();
    k_clock_advance<<<1, 1, 0, st>>>(clk, 2);
    cudaGraph_t gr = nullptr;
    cudaError_t e = cudaStreamEndCapture(st, &gr);
    per_pair = ctx->prof.launches - l0 + 1;
    ctx->prof.launches = l0;
    if (s != SWF_OK) {
      if (gr) cudaGraphDestroy(gr);
      return s;
    }
    if (e != cudaSuccess) return cuda_status(e, "capture of the march steps");
    e = cudaGraphInstantiate(&exec, gr, 0);
    cudaGraphDestroy(gr);
    if (e != cudaSuccess) return cuda_status(e, "instantiate the march graph");
    return SWF_OK;
  }
  template <typename Rec>
  swf_status launch(swf_ctx* ctx, MarchClock* clk, Rec&& record) {
    if (exec) {
      const cudaError_t e = cudaGraphLaunch(exec, st);
      ctx->prof.launches += per_pair;
      return e == cudaSuccess ? SWF_OK : cuda_status(e, "launch the march graph");
    }
    const swf_status s = record();
    k_clock_advance<<<1, 1, 0, st>>>(clk, 2);
    ++ctx->prof.launches;
    return s;
  }
  // the executable graph is released once its launches have run
  swf_status finish() {
    if (!exec) return SWF_OK;
    const cudaError_t e = cudaStreamSynchronize(st);
    cudaGraphExecDestroy(exec);
    exec = nullptr;
    return e == cudaSuccess ? SWF_OK : cuda_status(e, "march graph");
  }
};

// complex64 fixed-step marches carry the state in float-float: a zeroed low part beside y.
template <typename R>
static swf_status state_low_part(swf_ctx* ctx, const std::string& name, size_t bytes, StageArgs<R>* A,
                                 cudaStream_t st) {
  A->ylo = nullptr;
  if (sizeof(R) != 4) return SWF_OK;
  void* p = nullptr;
  swf_status s = ws_get(ctx, name, bytes, &p);
  if (s != SWF_OK) return s;
  const cudaError_t e = cudaMemsetAsync(p, 0, bytes, st);
  if (e != cudaSuccess) return cuda_status(e, "memset state low part");
  A->ylo = (cpx<R>*)p;
  return SWF_OK;
}

template <typename R>
static swf_status march_impl(swf_ctx* ctx, const GridDesc& g, double t_in, double t_out, int n_steps, int F,
                             const FieldDesc* fd_host, void* psi_out, cudaStream_t st);

// ---------------------------------------------------------------- step-size control
// Fifth- minus fourth-order weights b_i - b*_i of the Dormand-Prince pair (1980).
static const double DP_DB[7] = {35.0 / 384 - 5179.0 / 57600, 0.0, 500.0 / 1113 - 7571.0 / 16695,
                                125.0 / 192 - 393.0 / 640, -2187.0 / 6784 + 92097.0 / 339200,
                                11.0 / 84 - 187.0 / 2100, -1.0 / 40};

struct ErrWeights {
  double db[7];
};

// part[f][b] = sum over block b's entries of field f of (|e| / (atol + rtol max(|y|, |y_new|)))^2,
// e = h sum_i (b_i - b*_i) k_i, in FP64 (fixed order inside the block).  FP64 operations bound it, so
// one square root serves both norms (of the larger square), the sums are chains of fused
// multiply-adds, and the blocks are small enough (four entries a thread) to load all SMs alike: six
// fields of 240 x 135 took 137 us with two roots and 16 entries a thread.
constexpr int kErrThreads = 256;
static int error_blocks(size_t per_field) { return (int)std::min<size_t>((per_field + 4 * kErrThreads - 1) / (4 * kErrThreads), 4096); }
template <typename R>
__global__ void __launch_bounds__(kErrThreads) k_step_error(const cpx<R>* __restrict__ y, const cpx<R>* __restrict__ ynew,
                                                            const cpx<R>* __restrict__ k0, const cpx<R>* __restrict__ k2,
                                                            const cpx<R>* __restrict__ k3, const cpx<R>* __restrict__ k4,
                                                            const cpx<R>* __restrict__ k5, const cpx<R>* __restrict__ k6,
                                                            ErrWeights W, const StepControl* ctl, size_t per_field,
                                                            double* part) {
  __shared__ double red[kErrThreads / 32];
  if (ctl->done) return;
  const int f = blockIdx.y;
  const double h = ctl->h, rtol = ctl->rtol, atol = ctl->atol;
  const cpx<R>* ks[6] = {k0, k2, k3, k4, k5, k6};  // the second weight is zero
  const double w[6] = {W.db[0], W.db[2], W.db[3], W.db[4], W.db[5], W.db[6]};
  double acc = 0.0;
  const size_t off = (size_t)f * per_field;
  for (size_t i = blockIdx.x * (size_t)kErrThreads + threadIdx.x; i < per_field; i += (size_t)gridDim.x * kErrThreads) {
    double ex = 0.0, ey = 0.0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const cpx<R> kv = ks[j][off + i];
      ex = fma(w[j], (double)kv.x, ex);
      ey = fma(w[j], (double)kv.y, ey);
    }
    const cpx<double> a = cvt<double>(y[off + i]), b = cvt<double>(ynew[off + i]);
    const double m = fmax(fma(a.x, a.x, a.y * a.y), fma(b.x, b.x, b.y * b.y));
    const double sc = fma(rtol, sqrt(m), atol);
    acc += fma(ex, ex, ey * ey) / (sc * sc);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w8 = 0; w8 < kErrThreads / 32; ++w8) sum += red[w8];
    part[(size_t)f * gridDim.x + blockIdx.x] = h * h * sum;
  }
}

// The larger of two error norms; NaN if either is (fmax would drop it, and a field gone bad would pass as
// one without error).
__device__ __forceinline__ double worse_error(double a, double b) { return a >= b ? a : (a == a ? b : a); }

// err = max over fields of the RMS scaled error (a warp per field in turn, lanes in a fixed order);
// accept when err <= 1 (and finite); next step h min(10, max(0.2, 0.9 err^(-1/5))), clamped so as not
// to pass t_in.  One block; one thread of it took 19 us to add 200 parts.
__global__ void __launch_bounds__(256) k_step_control(StepControl* ctl, const double* __restrict__ part, int nb, int F,
                                                      double count) {
  __shared__ double s_err[8];
  if (ctl->done) {
    if (threadIdx.x == 0) ctl->ok = 0;
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double err = 0.0;
  for (int f = warp; f < F; f += 8) {
    double sum = 0.0;
    for (int b = lane; b < nb; b += 32) sum += part[(size_t)f * nb + b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    err = worse_error(err, sqrt(sum / count));
  }
  if (lane == 0) s_err[warp] = err;
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 0; w < 8; ++w) err = worse_error(err, s_err[w]);
  if (!(err == err) || isinf(err)) {  // non-finite: stop
    ctl->ok = 0;
    ctl->failed = 1;
    ctl->done = 1;
    return;
  }
  const double fac = err == 0.0 ? 10.0 : fmin(10.0, fmax(0.2, 0.9 * pow(err, -0.2)));
  if (err <= 1.0) {
    ctl->t += ctl->h;
    ctl->ok = 1;
    ctl->accepted += 1;
  } else {
    ctl->ok = 0;
    ctl->rejected += 1;
  }
  double h = ctl->h * fac;
  const double rest = ctl->t_in - ctl->t;
  if (fabs(rest) <= 1e-12 * ctl->span) {
    ctl->done = 1;
  } else if (fabs(h) > fabs(rest)) {
    h = rest;
  }
  ctl->h = h;
  if (!ctl->done && ctl->accepted + ctl->rejected >= ctl->max_attempts) {
    ctl->failed = 1;
    ctl->done = 1;
  }
}

// After an accepted attempt: y <- y_new and k_1 <- k_7 (first same as last).
template <typename R>
__global__ void k_step_accept(const StepControl* ctl, cpx<R>* y, const cpx<R>* ynew, cpx<R>* k1, const cpx<R>* k7,
                              size_t n) {
  if (!ctl->ok) return;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    y[i] = ynew[i];
    k1[i] = k7[i];
  }
}

// Step-size-controlled march (Sec. II.A: Dopri5 with relative and absolute tolerances), from
// t_out with first step h0 toward t_in.  Every attempt (six evaluations, the error norm, the
// controller, the copy-in of an accepted step) is one CUDA graph replay; nothing is decided on
// the host: after t_in (or a failure) the remaining replays of a chunk do nothing.  The host
// reads the controller's state once per chunk of replays.
// Runs step attempts recorded by `attempt` (launches only, on st) until the controller in ctl
// reports t_in reached or a failure: chunks of 8, 16, .. 64 attempts as CUDA-graph replays
// (kernel by kernel when timing is on), the controller's state read once per chunk into *out.
// Condition of the device-side attempt loop: another attempt while the controller is not done
// (the controller itself stops at max_attempts; the bound is repeated here so that the loop ends
// whatever the state).
__global__ void k_attempt_condition(cudaGraphConditionalHandle h, const StepControl* ctl) {
  const bool more = !ctl->done && ctl->accepted + ctl->rejected < ctl->max_attempts;
  cudaGraphSetConditional(h, more ? 1u : 0u);
}

// The whole controlled march as one graph launch: a while node whose body is one attempt and
// k_attempt_condition, so that accepting, rejecting and stopping are decided on the device and
// the host reads the controller's state once, at the end.  *built = false (nothing launched) when
// the graph cannot be built here; the caller then runs its host loop.
template <typename Att>
static swf_status attempts_on_device(swf_ctx* ctx, cudaStream_t st, const StepControl* ctl, Att&& attempt,
                                     StepControl* out, bool* built) {
  *built = false;
  cudaGraph_t g = nullptr;
  cudaGraphExec_t exec = nullptr;
  if (cudaGraphCreate(&g, 0) != cudaSuccess) {
    cudaGetLastError();
    return SWF_OK;
  }
  swf_status s = SWF_OK;
  long long per_attempt = 0;
  cudaGraphConditionalHandle h;
  // the parameter union has no default constructor: zeroed storage
  alignas(cudaGraphNodeParams) unsigned char np_raw[sizeof(cudaGraphNodeParams)];
  std::memset(np_raw, 0, sizeof(np_raw));
  cudaGraphNodeParams& np = *reinterpret_cast<cudaGraphNodeParams*>(np_raw);
  cudaGraphNode_t node;
  bool ok = cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault) == cudaSuccess;
  if (ok) {
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = h;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    ok = cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &np) == cudaSuccess;
  }
  if (ok) ok = cudaStreamBeginCaptureToGraph(st, np.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                             cudaStreamCaptureModeThreadLocal) == cudaSuccess;
  if (ok) {
    const long long l0 = ctx->prof.launches;
    s = attempt();
    k_attempt_condition<<<1, 1, 0, st>>>(h, ctl);
    cudaGraph_t body = nullptr;
    const cudaError_t ec = cudaStreamEndCapture(st, &body);
    per_attempt = ctx->prof.launches - l0 + 1;
    ctx->prof.launches = l0;
    ok = s == SWF_OK && ec == cudaSuccess && cudaGraphInstantiate(&exec, g, 0) == cudaSuccess;
  }
  cudaGraphDestroy(g);
  if (s != SWF_OK) {
    if (exec) cudaGraphExecDestroy(exec);
    return s;
  }
  if (!ok) {
    if (exec) cudaGraphExecDestroy(exec);
    cudaGetLastError();  // an unsupported graph form is not an error of the march
    return SWF_OK;
  }
  *built = true;
  cudaError_t e = cudaGraphLaunch(exec, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(out, ctl, sizeof(StepControl), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaGraphExecDestroy(exec);
  if (e != cudaSuccess) return cuda_status(e, "step-size-controlled march (device loop)");
  ctx->prof.launches += per_attempt * (out->accepted + out->rejected);
  ctx->device_loop_marches += 1;
  return SWF_OK;
}

template <typename Att>
static swf_status run_attempts(swf_ctx* ctx, cudaStream_t st, int max_attempts, const StepControl* ctl,
                               Att&& attempt, StepControl* out) {
  swf_status s = SWF_OK;
  cudaError_t e = cudaSuccess;
  bool graph = !ctx->prof.on && st != 0 && ctx->use_graphs;
  cudaGraphExec_t exec = nullptr;
  long long per_attempt = 0;
  if (graph) {
    bool built = false;
    s = attempts_on_device(ctx, st, ctl, attempt, out, &built);
    if (s != SWF_OK || built) return s;
  }
  if (graph) {
    const long long l0 = ctx->prof.launches;
    if (cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();
      graph = false;
    } else {
      s = attempt();
      cudaGraph_t gr = nullptr;
      e = cudaStreamEndCapture(st, &gr);
      per_attempt = ctx->prof.launches - l0;
      ctx->prof.launches = l0;
      if (s != SWF_OK) {
        if (gr) cudaGraphDestroy(gr);
        return s;
      }
      if (e != cudaSuccess) return cuda_status(e, "capture of the step attempt");
      e = cudaGraphInstantiate(&exec, gr, 0);
      cudaGraphDestroy(gr);
      if (e != cudaSuccess) return cuda_status(e, "instantiate the step attempt");
    }
  }
  StepControl hc{};
  int chunk = 8, attempts = 0;
  while (true) {
    for (int a = 0; a < chunk; ++a) {
      if (graph) {
        e = cudaGraphLaunch(exec, st);
        ctx->prof.launches += per_attempt;
        if (e != cudaSuccess) break;
      } else if ((s = attempt()) != SWF_OK) {
        if (exec) cudaGraphExecDestroy(exec);
        return s;
      }
    }
    attempts += chunk;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hc, ctl, sizeof(StepControl), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess || hc.done) break;
    if (attempts > max_attempts + chunk) {  // the controller stops at max_attempts; this is a backstop
      hc.failed = 1;
      break;
    }
    chunk = std::min(chunk * 2, 64);
  }
  if (exec) cudaGraphExecDestroy(exec);
  if (e != cudaSuccess) return cuda_status(e, "step-size-controlled march");
  *out = hc;
  return SWF_OK;
}

template <typename R>
static swf_status march_adaptive_impl(swf_ctx* ctx, const GridDesc& g, double t_in, double t_out, double h0,
                                      int max_attempts, int F, const FieldDesc* fd_host, void* psi_out,
                                      cudaStream_t st) {
  StageArgs<R> A;
  swf_status s = prepare_args<R>(ctx, g, F, fd_host, &A, "march", st);
  if (s != SWF_OK) return s;
  const size_t per_field = (size_t)4 * g.N;
  const size_t state = (size_t)F * per_field * sizeof(cpx<R>);
  void *py = nullptr, *pyn = nullptr, *pT = nullptr, *pk[7], *pctl = nullptr, *ppart = nullptr;
  if ((s = ws_get(ctx, "march.y", state, &py)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "march.ynew", state, &pyn)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "march.T", state, &pT)) != SWF_OK) return s;
  for (int i = 0; i < 7; ++i) {
    char nm[32];
    std::snprintf(nm, sizeof nm, "march.k%d", i);
    if ((s = ws_get(ctx, nm, state, &pk[i])) != SWF_OK) return s;
  }
  const int nbe = error_blocks(per_field);
  if ((s = ws_get(ctx, "march.ctl", sizeof(StepControl), &pctl)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "march.err_part", sizeof(double) * (size_t)nbe * F, &ppart)) != SWF_OK) return s;
  cudaError_t e = cudaMemsetAsync(py, 0, state, st);
  if (e != cudaSuccess) return cuda_status(e, "memset state");
  StepControl c0{};
  c0.t = t_out;
  c0.h = (t_in < t_out) ? -std::fabs(h0) : std::fabs(h0);
  if (std::fabs(c0.h) > std::fabs(t_in - t_out)) c0.h = t_in - t_out;
  c0.t_in = t_in;
  c0.span = std::fabs(t_in - t_out);
  c0.rtol = ctx->rtol;
  c0.atol = ctx->atol;
  c0.max_attempts = max_attempts;
  StepControl* ctl = (StepControl*)pctl;
  e = cudaMemcpyAsync(ctl, &c0, sizeof(StepControl), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_status(e, "upload step control");
  A.y = (cpx<R>*)py;
  A.T = (cpx<R>*)pT;
  {
    StageArgs<R> B = A;  // shapes by timing, before the slots hold anything
    B.nterm = 6;
    for (int q = 0; q < 6; ++q) {
      B.kin[q] = (const cpx<R>*)pk[q + 1];
      B.coef[q] = 0.0;
      B.coef_r[q] = (R)0;
    }
    B.write_y = 0;
    B.ystage = nullptr;
    B.kout = (cpx<R>*)pk[0];
    B.t = t_out;
    if ((s = autotune_eval<R>(ctx, B, F, st)) != SWF_OK) return s;
  }
  // k_1 = f(t_out, 0)
  A.nterm = 0;
  A.write_y = 0;
  A.kout = (cpx<R>*)pk[0];
  A.t = t_out;
  if ((s = launch_eval<R>(ctx, A, F, st)) != SWF_OK) return s;
  A.ctl = ctl;
  A.ynew = (cpx<R>*)pyn;
  ErrWeights W;
  for (int j = 0; j < 7; ++j) W.db[j] = DP_DB[j];
  // an attempt's evaluations chain (one x pass closes one and opens the next); the attempt's last one is closed
  // before the error estimate reads k_7
  const bool chain = !(g.n[1] == 1 && g.n[2] == 1);
  auto attempt = [&]() -> swf_status {
    StageArgs<R> open = A;
    for (int i = 1; i < 7; ++i) {
      int nt = 0;
      for (int j = 0; j < i; ++j) {
        if (DP_A[i][j] == 0.0) continue;
        A.kin[nt] = (const cpx<R>*)pk[j];
        A.coef[nt] = DP_A[i][j];  // times the device-held h in k_first
        ++nt;
      }
      A.nterm = nt;
      A.write_y = (i == 6);
      A.kout = (cpx<R>*)pk[i];
      A.c = DP_C[i];
      set_next_node<R>(&A, 0, i);
      swf_status r = !chain ? launch_eval<R>(ctx, A, F, st)
                            : (i == 1 ? launch_eval_open<R>(ctx, A, F, st) : launch_eval_chain<R>(ctx, open, A, F, st));
      if (r != SWF_OK) return r;
      open = A;
    }
    if (chain) {
      swf_status r = launch_eval_close<R>(ctx, open, F, st);
      if (r != SWF_OK) return r;
    }
    {
      ProfScope ps(ctx, "k_step_error", st);
      k_step_error<R><<<dim3(nbe, F), kErrThreads, 0, st>>>(
          (const cpx<R>*)py, (const cpx<R>*)pyn, (const cpx<R>*)pk[0], (const cpx<R>*)pk[2], (const cpx<R>*)pk[3],
          (const cpx<R>*)pk[4], (const cpx<R>*)pk[5], (const cpx<R>*)pk[6], W, ctl, per_field, (double*)ppart);
    }
    {
      ProfScope ps(ctx, "k_step_control", st);
      k_step_control<<<1, 256, 0, st>>>(ctl, (const double*)ppart, nbe, F, (double)per_field);
    }
    {
      ProfScope ps(ctx, "k_step_accept", st);
      const size_t n = (size_t)F * per_field;
      k_step_accept<R><<<(unsigned)std::min<size_t>((n + 255) / 256, 4096), 256, 0, st>>>(
          ctl, (cpx<R>*)py, (const cpx<R>*)pyn, (cpx<R>*)pk[0], (const cpx<R>*)pk[6], n);
    }
    return SWF_OK;
  };
  StepControl hc{};
  if ((s = run_attempts(ctx, st, max_attempts, ctl, attempt, &hc)) != SWF_OK) return s;
  ctx->last_accepted = hc.accepted;
  ctx->last_rejected = hc.rejected;
  if (hc.failed) {
    set_error("step-size-controlled march: no convergence (too many attempts or a non-finite error)");
    return SWF_ENUMERIC;
  }
  e = cudaMemcpyAsync(psi_out, py, state, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return cuda_status(e, "copy psi(t_in)");
  return SWF_OK;
}

swf_status march_adaptive(swf_ctx* ctx, const GridDesc& g, double t_in, double t_out, double h0, int max_attempts,
                          int n_f, const FieldDesc* fd_host, swf_precision prec, void* psi_out, cudaStream_t st) {
  if (prec == SWF_C64)
    return march_adaptive_impl<float>(ctx, g, t_in, t_out, h0, max_attempts, n_f, fd_host, psi_out, st);
  return march_adaptive_impl<double>(ctx, g, t_in, t_out, h0, max_attempts, n_f, fd_host, psi_out, st);
}

// psi_out[f] = psi_u[rep[f]] with the components {1, 2} times sgn[f] (+1 or -1).
template <typename R>
__global__ void k_expand_fields(const cpx<R>* __restrict__ psi_u, const int* __restrict__ rep,
                                const int* __restrict__ sgn, size_t N, cpx<R>* __restrict__ psi_out) {
  const int f = blockIdx.y;
  const int c = blockIdx.z;
  const R s = (c == 1 || c == 2) ? (R)sgn[f] : (R)1;
  const cpx<R>* src = psi_u + ((size_t)rep[f] * 4 + c) * N;
  cpx<R>* dst = psi_out + ((size_t)f * 4 + c) * N;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = s * src[i];
}

static bool same_desc_but_spinor(const FieldDesc& a, const FieldDesc& b) {
  if (a.kind != b.kind || a.acomp != b.acomp || a.e0 != b.e0 || a.tsign != b.tsign) return false;
  for (int k = 0; k < 8; ++k)
    if (a.prm[k] != b.prm[k]) return false;
  for (int k = 0; k < 3; ++k)
    if (a.K[k] != b.K[k] || a.pmom[k] != b.pmom[k]) return false;
  return true;
}

// Fields whose march repeats another's: the same field, background momentum and energy, and a
// background spinor that is the same or (when the spin along z is conserved) the same with the
// components {1, 2} negated.  The second case is the other spin: R_- = diag(1, -1, -1, 1) R_+,
// and (1 +- p-slash), alpha^x, alpha^y, beta and A_0 never mix {0, 3} with {1, 2} when p_z = 0,
// the z axis is trivial and A_3 = 0, so the scattered wave of the other spin is the same wave
// with {1, 2} negated, exactly.  rep[f] indexes the unique list; sgn[f] is the sign of {1, 2}.
static int dedupe_fields(const GridDesc& g, int n_f, const FieldDesc* fd, std::vector<int>& rep,
                         std::vector<int>& sgn, std::vector<FieldDesc>& uniq) {
  rep.assign(n_f, 0);
  sgn.assign(n_f, 1);
  uniq.clear();
  std::vector<int> first;  // field index of each unique entry
  for (int f = 0; f < n_f; ++f) {
    const FieldDesc& a = fd[f];
    const bool zsym = g.n[2] == 1 && a.K[2] == 0.0 && a.acomp != 3;
    int found = -1, sign = 1;
    for (size_t u = 0; u < uniq.size() && found < 0; ++u) {
      const FieldDesc& b = uniq[u];
      if (!same_desc_but_spinor(a, b)) continue;
      bool eq = true, flip = zsym;
      for (int k = 0; k < 8; ++k) {
        const bool in_b = (k >> 1) == 1 || (k >> 1) == 2;  // components 1 and 2
        if (a.w[k] != b.w[k]) eq = false;
        if (a.w[k] != (in_b ? -b.w[k] : b.w[k])) flip = false;
      }
      if (eq) { found = (int)u; sign = 1; }
      else if (flip) { found = (int)u; sign = -1; }
    }
    if (found < 0) {
      found = (int)uniq.size();
      uniq.push_back(a);
      first.push_back(f);
    }
    rep[f] = found;
    sgn[f] = sign;
  }
  return (int)uniq.size();
}

// The buffers that prepare_args and march_impl take for F fields.
template <typename R>
static std::vector<std::pair<std::string, size_t>> march_buffers(const GridDesc& g, int F) {
  const size_t nt = g.n[0] + g.n[1] + g.n[2];
  const size_t state = (size_t)F * 4 * g.N * sizeof(cpx<R>);
  std::vector<std::pair<std::string, size_t>> b = {
      {"march.fd", sizeof(FieldDesc) * F}, {"march.greal", sizeof(R) * F * nt}, {"march.gcplx", sizeof(cpx<R>) * F * (nt + 4)},
      {"march.y", state}, {"march.T", state}};
  if (sizeof(R) == 4) b.push_back({"march.ylo", state});
  for (int i = 0; i < 7; ++i) b.push_back({"march.k" + std::to_string(i), state});
  b.push_back({"march.clock", sizeof(MarchClock)});
  b.push_back({"march.kap", sizeof(R) * nt});
  if (g.n[1] > 1 || g.n[2] > 1) {
    b.push_back({"march.ft", sizeof(R) * F * g.n[1]});
    b.push_back({"march.tf", sizeof(cpx<R>) * F});
  }
  return b;
}

bool march_held(swf_ctx* ctx, const GridDesc& g, int n_f, swf_precision prec) {
  for (const auto& b : prec == SWF_C64 ? march_buffers<float>(g, n_f) : march_buffers<double>(g, n_f))
    if (!ws_has(ctx, b.first, b.second)) return false;
  return true;
}

void march_release(swf_ctx* ctx, const GridDesc& g) {
  for (const auto& b : march_buffers<float>(g, 1)) ws_drop(ctx, b.first);  // single precision has them all
  ws_drop(ctx, "march.unique");
}

// Sizes the pass-kernel march's workspace for F fields without touching the device: growing a
// workspace buffer frees the old one, which waits for the whole device, so march_split does it before
// the fused kernel starts.
template <typename R>
static swf_status reserve_march(swf_ctx* ctx, const GridDesc& g, int F) {
  void* p = nullptr;
  swf_status s;
  for (const auto& b : march_buffers<R>(g, F))
    if ((s = ws_get(ctx, b.first, b.second, &p)) != SWF_OK) return s;
  for (int a = 0; a < 3; ++a) {
    const void* tw = nullptr;
    if ((s = twiddles(ctx, g.n[a], Prec<R>::is_double, &tw)) != SWF_OK) return s;
    const LineEntry<R>* le = line_of<R>(g, a);
    if (le && (s = line_ready<R>(le)) != SWF_OK) return s;
    if (le && (s = twiddles(ctx, g.n[a], Prec<R>::is_double, &tw, le->r2)) != SWF_OK) return s;
  }
  return SWF_OK;
}

// The fused kernel's 16-CTA clusters (one CTA per SM) fit once per GPC, so some SMs stay idle
// (on GB300: 7 clusters on 112 of 152 SMs).  Moving some fields to the pass kernels, run
// concurrently on those SMs, shortens the march when they finish within the fused kernel's
// time.  With R = ceil(2 n_f / ncl) rounds of sectors per cluster, removing r rounds leaves
// n_1 = floor((R - r) ncl / 2) fields to the clusters and n_2 = n_f - n_1 to the pass kernels,
// which take about alpha n_2 rounds' time on the free SMs.  alpha = 2.0 was measured with 40 free SMs
// on (2+1)D 256^2 complex64 marches of 1000 steps with small-radix passes in shared memory: 16 fields took
// 2.75 s on the free SMs while the fused launch took 32 rounds in 2.78 s; rounds of the pulled-transpose
// kernel are 1.46 times longer (alpha = 1.37).  With the register lines 16 fields take 1.45 s beside 32
// rounds in 2.46 s (alpha = 1.2), so the line lies on the safe side: the free SMs are done first.  Moving
// it has not been measured.  alpha scales with 40 / (free SMs).  The largest r with alpha n_2 <= R - r is
// taken.
int fused_split_count(int n_f, int ncl, int n_sm, int variant) {
  const int free_sm = n_sm - kFusedClusterCtas * ncl;
  if (ncl < 1 || free_sm < 16 || n_f < 16) return 0;
  const double alpha = (variant == 3 ? 2.0 : 1.37) * 40.0 / free_sm;
  const int R = (2 * n_f + ncl - 1) / ncl;
  int best = 0;
  for (int r = 1; r < R; ++r) {
    const int n1 = ((R - r) * ncl) / 2;
    const int n2 = n_f - n1;
    if (n2 <= 0) continue;
    if (alpha * n2 > (double)(R - r)) break;
    best = n2;
  }
  return best;
}

// The fused kernel on the first n_f - n2 fields (stream st) and, concurrently, the pass kernels
// on the last n2 fields (the context's auxiliary stream), which take the SMs that the fused
// kernel's clusters leave free.  The auxiliary stream starts after the work already queued on
// st and st continues after both.  complex64 only (the fused kernel's precision).
static swf_status march_split(swf_ctx* ctx, const GridDesc& g, double t_in, double t_out, int n_steps, int n_f,
                              int n2, const FieldDesc* fd_host, void* psi_out, cudaStream_t st) {
  cudaError_t e;
  if (!ctx->aux) {
    if ((e = cudaStreamCreateWithFlags(&ctx->aux, cudaStreamNonBlocking)) != cudaSuccess)
      return cuda_status(e, "auxiliary stream");
    for (int i = 0; i < 2; ++i)
      if ((e = cudaEventCreateWithFlags(&ctx->aux_ev[i], cudaEventDisableTiming)) != cudaSuccess)
        return cuda_status(e, "auxiliary stream events");
  }
  const int n1 = n_f - n2;
  swf_status s = reserve_march<float>(ctx, g, n2);
  if (s != SWF_OK) return s;
  if ((e = cudaEventRecord(ctx->aux_ev[0], st)) != cudaSuccess ||
      (e = cudaStreamWaitEvent(ctx->aux, ctx->aux_ev[0], 0)) != cudaSuccess)
    return cuda_status(e, "order the auxiliary stream");
  s = march_fused(ctx, g, t_in, t_out, n_steps, n1, fd_host, psi_out, st);
  if (s != SWF_OK) return s;
  cpx<float>* out2 = (cpx<float>*)psi_out + (size_t)n1 * 4 * g.N;
  s = march_impl<float>(ctx, g, t_in, t_out, n_steps, n2, fd_host + n1, out2, ctx->aux);
  if (s != SWF_OK) return s;
  if ((e = cudaEventRecord(ctx->aux_ev[1], ctx->aux)) != cudaSuccess ||
      (e = cudaStreamWaitEvent(st, ctx->aux_ev[1], 0)) != cudaSuccess)
    return cuda_status(e, "join the auxiliary stream");
  return SWF_OK;
}

static swf_status march_unique(swf_ctx* ctx, const GridDesc& g, double t_in, double t_out, int n_steps, int n_f,
                               const FieldDesc* fd_host, swf_precision prec, void* psi_out, cudaStream_t st,
                               int adaptive) {
  if (adaptive)  // first step (t_in - t_out)/n_steps, at most 100 n_steps + 100 attempts
    return march_adaptive(ctx, g, t_in, t_out, (t_in - t_out) / n_steps, 100 * n_steps + 100, n_f, fd_host, prec,
                          psi_out, st);
  if (ctx->use_fused && fused_applicable(g, n_f, fd_host, prec)) {
    const int n2 = (ctx->sm_split && ctx->fused_variant != 2)
                       ? fused_split_count(n_f, fused_resident_clusters(ctx), sm_count(), ctx->fused_variant)
                       : 0;
    if (n2 > 0) return march_split(ctx, g, t_in, t_out, n_steps, n_f, n2, fd_host, psi_out, st);
    swf_status s = march_fused(ctx, g, t_in, t_out, n_steps, n_f, fd_host, psi_out, st);
    if (s != SWF_EUNSUPPORTED) return s;
    ctx->use_fused = false;  // the cluster shape cannot be resident here: pass kernels from now on
  }
  if (prec == SWF_C64) return march_impl<float>(ctx, g, t_in, t_out, n_steps, n_f, fd_host, psi_out, st);
  return march_impl<double>(ctx, g, t_in, t_out, n_steps, n_f, fd_host, psi_out, st);
}

swf_status march_fields(swf_ctx* ctx, const GridDesc& g, double t_in, double t_out, int n_steps,
                        int n_f, const FieldDesc* fd_host, swf_precision prec, void* psi_out,
                        cudaStream_t st, int adaptive) {
  std::vector<int> rep, sgn;
  std::vector<FieldDesc> uniq;
  const int n_u = ctx->dedupe ? dedupe_fields(g, n_f, fd_host, rep, sgn, uniq) : n_f;
  ctx->fields_marched += n_u;
  if (n_u == n_f) return march_unique(ctx, g, t_in, t_out, n_steps, n_f, fd_host, prec, psi_out, st, adaptive);
  const size_t elem = prec == SWF_C64 ? 8 : 16;
  void *pu = nullptr, *ptab = nullptr;
  swf_status s = ws_get(ctx, "march.unique", (size_t)n_u * 4 * g.N * elem, &pu);
  if (s != SWF_OK) return s;
  if ((s = ws_get(ctx, "march.unique_map", sizeof(int) * 2 * (size_t)n_f, &ptab)) != SWF_OK) return s;
  if ((s = march_unique(ctx, g, t_in, t_out, n_steps, n_u, uniq.data(), prec, pu, st, adaptive)) != SWF_OK) return s;
  std::vector<int> tab(rep);
  tab.insert(tab.end(), sgn.begin(), sgn.end());
  cudaError_t e = cudaMemcpyAsync(ptab, tab.data(), sizeof(int) * 2 * (size_t)n_f, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_status(e, "upload field map");
  const dim3 grid((unsigned)std::min<size_t>((g.N + 255) / 256, 1024), n_f, 4);
  ProfScope ps(ctx, "k_expand_fields", st);
  if (prec == SWF_C64)
    k_expand_fields<float><<<grid, 256, 0, st>>>((const cpx<float>*)pu, (const int*)ptab, (const int*)ptab + n_f,
                                                 (size_t)g.N, (cpx<float>*)psi_out);
  else
    k_expand_fields<double><<<grid, 256, 0, st>>>((const cpx<double>*)pu, (const int*)ptab, (const int*)ptab + n_f,
                                                  (size_t)g.N, (cpx<double>*)psi_out);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "expand fields");
  // the host table must outlive its asynchronous upload
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_status(e, "expand fields");
  return SWF_OK;
}

template <typename R>
static swf_status rhs_impl(swf_ctx* ctx, const GridDesc& g, const FieldDesc& fd, double t,
                           const void* psi, void* out, cudaStream_t st) {
  StageArgs<R> A;
  swf_status s = prepare_args<R>(ctx, g, 1, &fd, &A, "rhs", st, &t);
  if (s != SWF_OK) return s;
  void* pT = nullptr;
  if ((s = ws_get(ctx, "rhs.T", (size_t)4 * g.N * sizeof(cpx<R>), &pT)) != SWF_OK) return s;
  A.y = const_cast<cpx<R>*>((const cpx<R>*)psi);  // read only: write_y = 0
  A.T = (cpx<R>*)pT;
  A.kout = (cpx<R>*)out;
  A.nterm = 0;
  A.write_y = 0;
  A.t = t;
  if ((s = launch_eval<R>(ctx, A, 1, st, A.ft != nullptr)) != SWF_OK) return s;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "rhs kernels");
  return SWF_OK;
}

swf_status rhs_eval(swf_ctx* ctx, const GridDesc& g, const FieldDesc& fd, swf_precision prec,
                    double t, const void* psi, void* out, cudaStream_t st) {
  if (prec == SWF_C64) return rhs_impl<float>(ctx, g, fd, t, psi, out, st);
  return rhs_impl<double>(ctx, g, fd, t, psi, out, st);
}

}  // namespace swf

// ---------------------------------------------------------------- right-hand side in caller scratch
namespace swf {

template <typename R>
__global__ void k_twiddles_into(cpx<R>* tw, int n, int r2) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const int m = r2 ? ((e / r2) * (e % r2)) % n : e;
    double s, c;
    sincospi(-2.0 * m / (double)n, &s, &c);
    tw[e] = mk<R>((R)c, (R)s);
  }
}

static size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

size_t rhs_scratch_bytes(const GridDesc& g, swf_precision prec) {
  const size_t e = prec == SWF_C64 ? 8 : 16, r = prec == SWF_C64 ? 4 : 8;
  const size_t nt = g.n[0] + g.n[1] + g.n[2];
  return align256(4 * (size_t)g.N * e) + align256(sizeof(FieldDesc)) + 2 * align256(nt * r) +
         align256((nt + 4) * e) + 3 * align256(512 * e);
}

// Same evaluation as rhs_eval, with every buffer (FFT workspace, field tables, twiddles, the
// field descriptor) carved out of `scratch` instead of the context's workspace; no device
// memory is allocated.
template <typename R>
static swf_status rhs_scratch_impl(const GridDesc& g, const FieldDesc& fd, double t, const void* psi, void* out,
                                   unsigned char* scratch, cudaStream_t st) {
  swf_status s = set_smem_attrs<R>();
  if (s != SWF_OK) return s;
  const int nt = g.n[0] + g.n[1] + g.n[2];
  unsigned char* p = scratch;
  cpx<R>* T = (cpx<R>*)p;
  p += align256((size_t)4 * g.N * sizeof(cpx<R>));
  FieldDesc* dfd = (FieldDesc*)p;
  p += align256(sizeof(FieldDesc));
  R* greal = (R*)p;
  p += align256((size_t)nt * sizeof(R));
  cpx<R>* gcplx = (cpx<R>*)p;
  p += align256((size_t)(nt + 4) * sizeof(cpx<R>));
  R* kap = (R*)p;
  p += align256((size_t)nt * sizeof(R));
  StageArgs<R> A;
  std::memset(&A, 0, sizeof(A));
  A.g = g;
  A.nrows = g.n[1] * g.n[2];
  for (int a = 0; a < 3; ++a) {
    if (!make_line_plan<R>(g, a, &A.plan[a])) {
      set_error("grid size must factor into 2, 3 and 5");
      return SWF_EINVAL;
    }
    const LineEntry<R>* le = line_of<R>(g, a);
    cpx<R>* tw = (cpx<R>*)p;
    p += align256(512 * sizeof(cpx<R>));
    k_twiddles_into<R><<<(g.n[a] + 127) / 128, 128, 0, st>>>(tw, g.n[a], le ? le->r2 : 0);
    (le ? A.ltw : A.tw)[a] = tw;
    if (le && (s = line_ready<R>(le)) != SWF_OK) return s;
  }
  A.kap = kap;
  A.inv_n = (R)(1.0 / (double)g.N);
  A.fd = dfd;
  A.greal = greal;
  A.gcplx = gcplx;
  fill_tables<R>(A, 1, &fd, nullptr, st);
  A.y = const_cast<cpx<R>*>((const cpx<R>*)psi);
  A.T = T;
  A.kout = (cpx<R>*)out;
  A.t = t;
  s = launch_eval<R>(nullptr, A, 1, st);
  if (s != SWF_OK) return s;
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "rhs kernels");
  return SWF_OK;
}

swf_status rhs_eval_scratch(const GridDesc& g, const FieldDesc& fd, swf_precision prec, double t, const void* psi,
                            void* out, void* scratch, cudaStream_t st) {
  if (prec == SWF_C64) return rhs_scratch_impl<float>(g, fd, t, psi, out, (unsigned char*)scratch, st);
  return rhs_scratch_impl<double>(g, fd, t, psi, out, (unsigned char*)scratch, st);
}

}  // namespace swf

// ---------------------------------------------------------------- Breit-Wheeler march (Sec. IV)
namespace swf {

// Dormand-Prince 5th-order weights b_i (the 7th is zero; FSAL)

// Photon plane-wave factor exp(i k.x) per axis for each instance (trivial axes: 1).
template <typename R>
__global__ void k_photon_tables(const double* photon, GridDesc g, int n_inst, cpx<R>* kph) {
  const int nt = g.n[0] + g.n[1] + g.n[2];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_inst * nt; i += gridDim.x * blockDim.x) {
    const int inst = i / nt;
    int j = i % nt, axis = 0;
    while (j >= g.n[axis]) { j -= g.n[axis]; ++axis; }
    const double xc = g.n[axis] > 1 ? g.x0[axis] + j * g.dx[axis] : 0.0;
    double s, c;
    sincos(photon[6 * inst + axis] * xc, &s, &c);
    kph[i] = mk<R>((R)c, (R)s);
  }
}

// Per instance, step and stage (Dormand-Prince nodes c_i) at t = t_out + (step + c_i) h, with the
// quadrature weight w_i = h b_{i+1} for i = 2..5 and h b_1 (of the next step) for the last stage,
// 0 elsewhere.  form 1: the background time phases of U and V and w_i dx^d e^{-i k0 t} (the
// integrand of Eq. 17 vanishes at the first stage, psi_s(t_out) = 0).  form 2 (Eqs. 30-33):
// w_i e^{-i(q0 - k0)t} and w_i e^{i(p0 - k0)t} for the direct transforms of the U and V waves
// and w_i e^{-i k0 t} for the mode sum; the first stage of the march carries h b_1 (the source
// term is not zero there).  FP64, computed once per march so that the integrand kernels need none.
__global__ void k_bw_phase_table(const FieldDesc* fd, const double* photon, int n_pi, int n_ph, int n_steps,
                                 double t_out, double h, double cell, int form, cpx<double>* tab) {
  const double DPc[7] = {0.0, 0.2, 0.3, 0.8, 8.0 / 9.0, 1.0, 1.0};
  const double DPb[7] = {35.0 / 384, 0.0, 500.0 / 1113, 125.0 / 192, -2187.0 / 6784, 11.0 / 84, 0.0};
  const long total = (long)n_pi * n_steps * 7;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total; e += (long)gridDim.x * blockDim.x) {
    const int pi = (int)(e / (7L * n_steps));  // photon-instance; its waves are those of instance pi / n_ph
    const int inst = pi / n_ph;
    const int step = (int)((e / 7) % n_steps), i = (int)(e % 7);
    const double t = t_out + (step + DPc[i]) * h;
    double w = (i >= 2 && i <= 5) ? h * DPb[i] : (i == 6 && step + 1 < n_steps ? h * DPb[0] : 0.0);
    if (form == 2 && i == 0 && step == 0) w = h * DPb[0];
    double sn, cs;
    const FieldDesc& FU = fd[2 * inst];
    const FieldDesc& FV = fd[2 * inst + 1];
    const double k0 = sqrt(photon[6 * pi] * photon[6 * pi] + photon[6 * pi + 1] * photon[6 * pi + 1] +
                           photon[6 * pi + 2] * photon[6 * pi + 2]);
    if (form == 2) {
      sincos(-(FV.e0 - k0) * t, &sn, &cs);
      tab[3 * e] = mk<double>(w * cs, w * sn);
      sincos((FU.e0 - k0) * t, &sn, &cs);
      tab[3 * e + 1] = mk<double>(w * cs, w * sn);
      sincos(-k0 * t, &sn, &cs);
      tab[3 * e + 2] = mk<double>(w * cs, w * sn);
      continue;
    }
    sincos(FU.tsign * FU.e0 * t, &sn, &cs);
    tab[3 * e] = mk<double>(cs, sn);
    sincos(FV.tsign * FV.e0 * t, &sn, &cs);
    tab[3 * e + 1] = mk<double>(cs, sn);
    sincos(-k0 * t, &sn, &cs);
    tab[3 * e + 2] = mk<double>(w * cell * cs, w * cell * sn);
  }
}

// Sum over the 32 lanes of a warp in the march precision (lane 0 holds it); the integrand kernels
// add the warps' sums of a block in FP64.  FP64 is scarce on GB300: a shuffle tree in FP64 per
// block and value cost more than the integrand itself.
template <typename R>
__device__ __forceinline__ cpx<R> warp_sum(cpx<R> v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    v.x += __shfl_down_sync(0xffffffffu, v.x, off);
    v.y += __shfl_down_sync(0xffffffffu, v.y, off);
  }
  return v;
}

// (alpha . e) v for a real vector e (Dirac representation).
template <typename R>
__device__ __forceinline__ void alpha_eps(const R* e, const cpx<R>* v, cpx<R>* o) {
  // sigma.e (u0, u1) = (ez u0 + ex u1 - i ey u1, ex u0 + i ey u0 - ez u1)
  o[0] = mk<R>(e[2] * v[2].x + e[0] * v[3].x + e[1] * v[3].y, e[2] * v[2].y + e[0] * v[3].y - e[1] * v[3].x);
  o[1] = mk<R>(e[0] * v[2].x - e[1] * v[2].y - e[2] * v[3].x, e[0] * v[2].y + e[1] * v[2].x - e[2] * v[3].y);
  o[2] = mk<R>(e[2] * v[0].x + e[0] * v[1].x + e[1] * v[1].y, e[2] * v[0].y + e[0] * v[1].y - e[1] * v[1].x);
  o[3] = mk<R>(e[0] * v[0].x - e[1] * v[0].y - e[2] * v[1].x, e[0] * v[0].y + e[1] * v[0].x - e[2] * v[1].y);
}

// J_a = x^+ alpha_a y for a = x, y, z (Dirac representation), every rounding fixed: the integrand of a
// photon is eps.J times its plane wave, so the products of the waves are formed once per site for all
// the photons of a block.
template <typename R>
__device__ __forceinline__ void current(const cpx<R>* x, const cpx<R>* y, cpx<R>* J) {
  const cpx<R> a = xcdot(x[0], y[3]), b = xcdot(x[1], y[2]), c = xcdot(x[2], y[1]), d = xcdot(x[3], y[0]);
  const cpx<R> ac = xadd(a, c), bd = xadd(b, d);
  J[0] = xadd(ac, bd);
  const cpx<R> m = mk<R>(rn_add(bd.x, -ac.x), rn_add(bd.y, -ac.y));
  J[1] = mul_i(m);
  const cpx<R> e = xadd(xcdot(x[0], y[2]), xcdot(x[2], y[0])), f = xadd(xcdot(x[1], y[3]), xcdot(x[3], y[1]));
  J[2] = mk<R>(rn_add(e.x, -f.x), rn_add(e.y, -f.y));
}
template <typename R>
__device__ __forceinline__ cpx<R> eps_dot(const R* e, const cpx<R>* J) {
  return mk<R>(rn_fma(e[2], J[2].x, rn_fma(e[1], J[1].x, rn_mul(e[0], J[0].x))),
               rn_fma(e[2], J[2].y, rn_fma(e[1], J[1].y, rn_mul(e[0], J[0].y))));
}
// s + a b
template <typename R>
__device__ __forceinline__ cpx<R> xmadd(cpx<R> s, cpx<R> a, cpx<R> b) {
  return mk<R>(rn_fma(-a.y, b.y, rn_fma(a.x, b.x, s.x)), rn_fma(a.y, b.x, rn_fma(a.x, b.y, s.y)));
}

// The three integrands of Eq. 17, dx^d sum_x U_a^+ (alpha.eps) V_b exp(-ikx), for (ss, bs, sb)
// at the stage values, integrated with weight w (= h b_i).  Block (b, by) sums the sites
// j = b*256 + threadIdx.x (stride gridDim.x*256) for NPH photons of one instance (several photons share
// one march; U and V are loaded and multiplied once per site) and adds w dx^d e^{-i k0 t} (from the
// phase table) times its sums to its own accumulators acc[photon-instance][b][3] (FP64; no other block
// touches them, so the march's sum is deterministic); k_mdot_final adds the accumulators in a fixed
// order.  64 photons on 192^2: 178 operations per site and photon became 57, and
// two blocks fit an SM (128 registers, polarisations in shared memory): 44 -> 22 us a stage.
template <typename R, int NPH>
__global__ void __launch_bounds__(256, sizeof(R) == 4 && NPH > 1 ? 2 : 1) k_mdot(const cpx<R>* __restrict__ ys, const cpx<R>* gcplx, const cpx<R>* kph,
                                              const double* photon, GridDesc g, const cpx<double>* __restrict__ ptab,
                                              const MarchClock* clk, int ls, int stage, int tab_stride,
                                              int n_ph, cpx<double>* acc) {
  chain_wait();
  chain_release();
  const long tab_row = (long)(clk->step + ls) * 7 + stage;
  __shared__ cpx<double> red[8][3 * NPH];
  // block row: instance inst, photons j0 .. j0 + nj - 1 (photon-instances pi0 + jj)
  const int nchunk = (n_ph + NPH - 1) / NPH;
  const int inst = blockIdx.y / nchunk;
  const int j0 = (blockIdx.y % nchunk) * NPH;
  const int nj = min(NPH, n_ph - j0);
  const int pi0 = inst * n_ph + j0;
  const int nx = g.n[0], ny = g.n[1], nt = nx + ny + g.n[2];
  const cpx<R>* tu = gcplx + (size_t)(2 * inst) * (nt + 4);
  const cpx<R>* tv = gcplx + (size_t)(2 * inst + 1) * (nt + 4);
  // the U and V time phases are the same in every photon's row of the phase table
  const cpx<double>* trow0 = ptab + 3 * (tab_row + (long)pi0 * tab_stride);
  const cpx<R> tfu = cvt<R>(trow0[0]), tfv = cvt<R>(trow0[1]);
  // the photons' polarisations and plane-wave tables (a partial last chunk repeats its last photon, which
  // is not stored)
  __shared__ R eps[NPH][4];
  if (threadIdx.x < 3 * NPH) {
    const int jj = threadIdx.x / 3, a = threadIdx.x % 3;
    eps[jj][a] = (R)photon[6 * (pi0 + min(jj, nj - 1)) + 3 + a];
  }
  const cpx<R>* kp0 = kph + (size_t)pi0 * nt;
  __syncthreads();
  const cpx<R>* U = ys + (size_t)(2 * inst) * 4 * g.N;
  const cpx<R>* V = ys + (size_t)(2 * inst + 1) * 4 * g.N;
  // per-thread sums in the march precision (a few sites each), the warp tree in it too, FP64 across warps
  cpx<R> tss[NPH], tbs[NPH], tsb[NPH];
#pragma unroll
  for (int jj = 0; jj < NPH; ++jj) tss[jj] = tbs[jj] = tsb[jj] = mk<R>(0, 0);
  const FastDiv fx((unsigned)nx), fy((unsigned)ny);
#pragma unroll(NPH == 1 ? 2 : 1)
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < g.N; j += gridDim.x * blockDim.x) {
    const int row = j < 8388608 ? (int)fx.div((unsigned)j) : j / nx;
    const int ix = j - row * nx;
    const int iz = row < 8388608 ? (int)fy.div((unsigned)row) : row / ny;
    const int iy = row - iz * ny;
    cpx<R> u[4], v[4], ub[4], vb[4], Jss[3], Jbs[3], Jsb[3];
    const cpx<R> phu = xmul(xmul(xmul(tfu, tu[ix]), tu[nx + iy]), tu[nx + ny + iz]);
    const cpx<R> phv = xmul(xmul(xmul(tfv, tv[ix]), tv[nx + iy]), tv[nx + ny + iz]);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      u[a] = U[(size_t)a * g.N + j];
      v[a] = V[(size_t)a * g.N + j];
      ub[a] = xmul(tu[nt + a], phu);
      vb[a] = xmul(tv[nt + a], phv);
    }
    current<R>(u, v, Jss);
    current<R>(ub, v, Jbs);
    current<R>(u, vb, Jsb);
#pragma unroll
    for (int jj = 0; jj < NPH; ++jj) {
      const cpx<R>* kp = kp0 + min(jj, nj - 1) * nt;
      const cpx<R> ph = xmul(xmul(kp[ix], kp[nx + iy]), kp[nx + ny + iz]);
      tss[jj] = xmadd(tss[jj], eps_dot<R>(eps[jj], Jss), ph);
      tbs[jj] = xmadd(tbs[jj], eps_dot<R>(eps[jj], Jbs), ph);
      tsb[jj] = xmadd(tsb[jj], eps_dot<R>(eps[jj], Jsb), ph);
    }
  }
#pragma unroll
  for (int jj = 0; jj < NPH; ++jj) {
    const cpx<R> ass = warp_sum<R>(tss[jj]), abs_ = warp_sum<R>(tbs[jj]), asb = warp_sum<R>(tsb[jj]);
    if ((threadIdx.x & 31) == 0) {
      red[threadIdx.x >> 5][3 * jj] = cvt<double>(ass);
      red[threadIdx.x >> 5][3 * jj + 1] = cvt<double>(abs_);
      red[threadIdx.x >> 5][3 * jj + 2] = cvt<double>(asb);
    }
  }
  __syncthreads();
  if (threadIdx.x < 3 * nj) {
    const int jj = threadIdx.x / 3, q = threadIdx.x % 3;
    cpx<double> sacc = mk<double>(0, 0);
    for (int wi = 0; wi < 8; ++wi) sacc = xadd(sacc, red[wi][threadIdx.x]);
    const cpx<double>* trow = ptab + 3 * (tab_row + (long)(pi0 + jj) * tab_stride);
    cpx<double>& a = acc[((size_t)(pi0 + jj) * gridDim.x + blockIdx.x) * 3 + q];
    a = xadd(a, xmul(trow[2], sacc));
  }
}

// macc[inst][q] = sum_b acc[inst][b][q]: warp q of block inst adds the accumulators
// b = lane, lane + 32, ... in order, then a fixed shuffle tree (deterministic).
__global__ void __launch_bounds__(96) k_mdot_final(const cpx<double>* __restrict__ acc, int nb, cpx<double>* macc) {
  const int inst = blockIdx.x;
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  cpx<double> sacc = mk<double>(0, 0);
  for (int b = lane; b < nb; b += 32) sacc = sacc + acc[((size_t)inst * nb + b) * 3 + q];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    sacc.x += __shfl_down_sync(0xffffffffu, sacc.x, off);
    sacc.y += __shfl_down_sync(0xffffffffu, sacc.y, off);
  }
  if (lane == 0) macc[3 * inst + q] = sacc;
}

// ---------------------------------------------------------------- partial-integration form (Sec. IV, Eqs. 28-33)
// The integrand of Eq. 33 and its analogues for (back, scat) and (scat, back), written with the grid
// transform psi~(kappa) and the energy projectors P_sigma of Eq. 23.  The time derivative of the split
// parts P_sigma psi~ e^{i sigma E t} is P_sigma F[Z] with Z = -i V (psi_s + psi_b) (Eq. 6), so per
// stage the march needs F[psi_s] and F[Z] of both waves on every grid mode (ss) and F[Z] at one
// off-grid momentum per wave (bs: V wave at p - k, sb: U wave at k - q).

// Per wave and axis: exp(-i kappa_a x_a) on the grid coordinates (trivial axes: 1), kappa = the wave's
// direct-transform momentum (3 doubles per wave).
template <typename R>
__global__ void k_f2_dtables(const double* wave_k, GridDesc g, int n_waves, cpx<R>* dph) {
  const int nt = g.n[0] + g.n[1] + g.n[2];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_waves * nt; i += gridDim.x * blockDim.x) {
    const int wv = i / nt;
    int j = i % nt, axis = 0;
    while (j >= g.n[axis]) { j -= g.n[axis]; ++axis; }
    const double xc = g.n[axis] > 1 ? g.x0[axis] + j * g.dx[axis] : 0.0;
    double sn, cs;
    sincos(-wave_k[3 * wv + axis] * xc, &sn, &cs);
    dph[i] = mk<R>((R)cs, (R)sn);
  }
}

// Parameters of one mode-sum table: the photon's mode shift per axis (0 <= shift < n), the fixed momenta
// of U and V along trivial axes, and k0.
struct F2Table {
  int shift[3];
  int pad;
  double Ku[3], Kv[3], k0;
};

// Per table and U grid mode j (V mode j - shift, periodic): 1 / Omega_{sigma sigma'} for
// (sigma, sigma') = (+,+), (+,-), (-,+), (-,-), Omega = sigma E_u - sigma' E_v - k0, in FP64 and
// rounded once.  (On the raw transforms the pair's grid-sum factor e^{i(kappa_v + k - kappa_u).x0}
// and the two origin phases combine into e^{i k.x0} for every pair, wrapped or not; the finalize
// kernel applies it.)
template <typename R>
__global__ void k_f2_omega_table(const F2Table* tabs, GridDesc g, int n_tab, R* omt) {
  const long total = (long)n_tab * g.N;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total; e += (long)gridDim.x * blockDim.x) {
    const F2Table& T = tabs[e / g.N];
    const int j = (int)(e % g.N);
    const int id[3] = {j % g.n[0], (j / g.n[0]) % g.n[1], j / (g.n[0] * g.n[1])};
    double ku[3], kv[3];
    for (int a = 0; a < 3; ++a) {
      const int jv = id[a] - T.shift[a] + (id[a] < T.shift[a] ? g.n[a] : 0);
      ku[a] = kappa_of(id[a], g.n[a], g.L[a], T.Ku[a]);
      kv[a] = kappa_of(jv, g.n[a], g.L[a], T.Kv[a]);
    }
    const double eu = energy3(ku), ev = energy3(kv);
    R* o = omt + 4 * e;
    o[0] = (R)(1.0 / (eu - ev - T.k0));
    o[1] = (R)(1.0 / (eu + ev - T.k0));
    o[2] = (R)(1.0 / (-eu - ev - T.k0));
    o[3] = (R)(1.0 / (-eu + ev - T.k0));
  }
}

// x pass of wave f = 2 inst + (0: U, 1: V) at a weighted stage (the shape of k_xpass, for lengths and
// precisions without line kernels; the others run k_f2_line): Z = -i V (Y + psi_b) of the stage value Y
// (from ys; the local term of the right-hand side) x-transformed into Zspec[f], and with do_y also Y into
// Yspec[f] (grids without a y or z pass; otherwise the right-hand side's pass writes the transform of Y);
// and the block's part of sum_x exp(-i kappa.x) Z(x) (the wave's direct transform), which trow[w] (w_i
// and its time phase) times adds to the block's own FP64 accumulators dpart[f][block][4] (no other block
// touches them: the sum is deterministic).  A thread that holds sites of Y's component c works on the
// component of Z that c feeds.  Rows per block are fixed, not tuned: they decide the order of the sum.
// Bound by FP64 issue; the threads' four or fewer values fill every quarter of every SM.  Three pairs
// on 160^2 in FP64: 80 us, where whole lines of one thread group took 106 us.
template <typename R, int R0>
__global__ void __launch_bounds__(kPassThreads, 1)
k_f2_x(const __grid_constant__ StageArgs<R> A, const cpx<R>* __restrict__ ys, cpx<R>* __restrict__ Yspec,
       cpx<R>* __restrict__ Zspec, int do_y, const cpx<R>* __restrict__ dph, const cpx<double>* __restrict__ ptab,
       int tab_stride, int stage, cpx<double>* dpart, int rows, int ld, int tpl) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ R s_ft[64];
  __shared__ cpx<R> s_tf;
  const RadixPlan& pl = A.plan[0];
  const int nx = pl.n, ny = A.g.n[1], nz = A.g.n[2], nb = nx / R0, rl = end_radix(pl, false);
  const size_t N = A.g.N;
  const int f = blockIdx.y, row0 = blockIdx.x * rows;
  const int line = threadIdx.x / tpl, g = threadIdx.x - line * tpl;
  const int c = line & 3, jr = line >> 2, row = row0 + jr;
  const bool ok = line < 4 * rows && row < A.nrows;
  cpx<R>* a = reinterpret_cast<cpx<R>*>(smem_raw);
  cpx<R>* b2 = a + 4 * rows * ld;
  const cpx<R>* __restrict__ tw = A.tw[0];
  const bool one = pl.npass < 2;
  row_factors(A, false, f, row0, rows, s_ft, &s_tf);
  __syncthreads();
  const int nt = nx + ny + nz;
  const R* __restrict__ gx = A.greal + (size_t)f * nt;
  const cpx<R>* __restrict__ ex = A.gcplx + (size_t)f * (nt + 4);
  const cpx<R>* __restrict__ dx = dph + (size_t)f * nt;
  const int acomp = A.fd[f].acomp;
  const int oc = source_component(acomp, c);
  const cpx<R> rot = source_rotation<R>(acomp, c);
  const size_t gl = ((size_t)f * 4 + c) * N + (size_t)row * nx;   // Y's line
  const size_t go = ((size_t)f * 4 + oc) * N + (size_t)row * nx;  // the line of Z
  const int iy = ok ? row % ny : 0, iz = ok ? row / ny : 0;
  const R ar = ok ? s_ft[jr] * gx[nx + iy] * gx[nx + ny + iz] : (R)0;
  const cpx<R> br = ex[nt + c] * (s_tf * (ex[nx + iy] * ex[nx + ny + iz]));
  cpx<R> dsum = mk<R>(0, 0);
  for (int part = do_y ? 0 : 1; part < 2; ++part) {
    const int sl = part ? 4 * jr + oc : line;  // the exchange line of what this thread transforms
    if (ok)
      for (int b = g; b < nb; b += tpl) {
        cpx<R> v[R0];
#pragma unroll
        for (int q = 0; q < R0; ++q) {
          const int x = b + q * nb;
          v[q] = ys[gl + x];
          if (part) {
            v[q] = source_term<R>(v[q], br, ex[x], ar * gx[x], rot);
            const cpx<R> e = dx[x];
            dsum = mk<R>(dsum.x + v[q].x * e.x - v[q].y * e.y, dsum.y + v[q].x * e.y + v[q].y * e.x);
          }
        }
        first_butterfly<R, R0>(v, b, false, a + sl * ld);
      }
    __syncthreads();
    const cpx<R>* cur = middle_passes<R>(a, b2, ld, 4 * rows, pl, false, tw);
    if (ok)
      with_radix(rl, [&](auto rc) {
        constexpr int RL = decltype(rc)::value;
        const int nm = nx / RL;
        cpx<R>* dst = part ? Zspec + go : Yspec + gl;
        for (int b = g; b < nm; b += tpl) {
          cpx<R> m[RL];
          last_butterfly<R, RL>(cur + sl * ld, b, nx, one, false, tw, m);
#pragma unroll
          for (int q = 0; q < RL; ++q) dst[b + q * nm] = m[q];
        }
      });
    __syncthreads();
  }
  // direct transform: the phases of the other axes, then the sum over the block's threads
  cpx<R>* red = a;
  if (line < 4 * rows) red[(oc * rows + jr) * tpl + g] = ok ? dsum * (dx[nx + iy] * dx[nx + ny + iz]) : mk<R>(0, 0);
  __syncthreads();
  direct_sums(A, red, rows * tpl, f, ptab, tab_stride, stage, dpart);
}

// o = P_+(kappa) x = (x + H0(kappa) x / E) / 2, the positive-energy part (evolves as e^{-iEt}); ke =
// kappa / (2 E), hp, hm = (1 +- 1/E) / 2.
template <typename R>
__device__ __forceinline__ void proj_plus(const R* ke, R hp, R hm, const cpx<R>* x, cpx<R>* o) {
  alpha_eps<R>(ke, x, o);
  o[0] = o[0] + hp * x[0];
  o[1] = o[1] + hp * x[1];
  o[2] = o[2] + hm * x[2];
  o[3] = o[3] + hm * x[3];
}
__device__ __forceinline__ float inv_root(float x) { return 1.0f / sqrtf(x); }
__device__ __forceinline__ double inv_root(double x) { return rsqrt(x); }

// s += sum_a conj(x_a) (a y_a + b z_a)
template <typename R>
__device__ __forceinline__ void form_add(cpx<R>& s, const cpx<R>* x, R a, const cpx<R>* y, R b, const cpx<R>* z) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const cpx<R> w = mk<R>(a * y[c].x + b * z[c].x, a * y[c].y + b * z[c].y);
    s.x = s.x + x[c].x * w.x + x[c].y * w.y;
    s.y = s.y + x[c].x * w.y - x[c].y * w.x;
  }
}

// The mode sum of the (scat, scat) integrand at one weighted stage, on the raw transforms Yspec, Zspec
// of the waves (no cell factor, no origin phase):
//   sum_j sum_{sigma,sigma'} 1/Omega [ (P_s Zu~)^+ (alpha.eps) P_s' Yv~ + (P_s Yu~)^+ (alpha.eps) P_s' Zv~ ]
// with U quantities at mode j and V quantities at mode j - shift.  Block (b, inst) adds trow[2]
// (w_i e^{-i k0 t}) times its part to its own accumulator sspart[inst][b].  In FP64 the instruction count
// is what bounds it: alpha.eps as additions of scaled components, both projections of a vector from one
// H0 x, both signs of sigma' summed before the contraction.  Three pairs on 160^2 in FP64: 70 us, where
// a projection and a contraction for every sign took 113 us.
// f2i per instance: shift[3], table index.
template <typename R>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 3 : 1) k_f2_ss(const cpx<R>* __restrict__ Yspec,
                                               const cpx<R>* __restrict__ Zspec, GridDesc g, const FieldDesc* fd,
                                               const double* photon, const int* __restrict__ f2i,
                                               const R* __restrict__ omt, const cpx<double>* __restrict__ ptab,
                                               const MarchClock* clk, int ls, int stage, int tab_stride,
                                               cpx<double>* sspart) {
  __shared__ cpx<double> red[8];
  const int inst = blockIdx.y;
  const int N = g.N;
  const int shift[3] = {f2i[4 * inst], f2i[4 * inst + 1], f2i[4 * inst + 2]};
  const R* om = omt + (size_t)f2i[4 * inst + 3] * 4 * N;
  const FieldDesc& FU = fd[2 * inst];
  const FieldDesc& FV = fd[2 * inst + 1];
  R eps[3];
  for (int a = 0; a < 3; ++a) eps[a] = (R)photon[6 * inst + 3 + a];
  const cpx<R>* Yu = Yspec + (size_t)(2 * inst) * 4 * N;
  const cpx<R>* Yv = Yu + (size_t)4 * N;
  const cpx<R>* Zu = Zspec + (size_t)(2 * inst) * 4 * N;
  const cpx<R>* Zv = Zu + (size_t)4 * N;
  // mode spacing 2 pi / L per axis (the mode index times it is kappa; trivial axes: fixed K)
  R du[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) du[a] = (R)(6.283185307179586476925286766559 / g.L[a]);
  cpx<R> tacc = mk<R>(0, 0);
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
    const int id[3] = {j % g.n[0], (j / g.n[0]) % g.n[1], j / (g.n[0] * g.n[1])};
    int jv[3];
    R ku[3], kv[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int n = g.n[a];
      jv[a] = id[a] - shift[a];  // 0 <= shift < n
      if (jv[a] < 0) jv[a] += n;
      const int fu = id[a] < (n + 1) / 2 ? id[a] : id[a] - n;
      const int fv = jv[a] < (n + 1) / 2 ? jv[a] : jv[a] - n;
      ku[a] = n > 1 ? du[a] * (R)fu : (R)FU.K[a];
      kv[a] = n > 1 ? du[a] * (R)fv : (R)FV.K[a];
    }
    const int j2 = (jv[2] * g.n[1] + jv[1]) * g.n[0] + jv[0];
    const R ieu = inv_root((R)1 + ku[0] * ku[0] + ku[1] * ku[1] + ku[2] * ku[2]);
    const R iev = inv_root((R)1 + kv[0] * kv[0] + kv[1] * kv[1] + kv[2] * kv[2]);
    const R hu = (R)0.5 * ieu, hv = (R)0.5 * iev;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      ku[a] *= hu;
      kv[a] *= hv;
    }
    // U side: the parts of Y and Z; V side: (alpha.eps) on the parts
    cpx<R> ym[4], yp[4], zm[4], zp[4], t[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      ym[c] = Yu[(size_t)c * N + j];
      zm[c] = Zu[(size_t)c * N + j];
    }
    proj_plus<R>(ku, (R)0.5 + hu, (R)0.5 - hu, ym, yp);
    proj_plus<R>(ku, (R)0.5 + hu, (R)0.5 - hu, zm, zp);
    cpx<R> y[4], z[4], ayp[4], aym[4], azp[4], azm[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      ym[c] = ym[c] - yp[c];
      zm[c] = zm[c] - zp[c];
      y[c] = Yv[(size_t)c * N + j2];
      z[c] = Zv[(size_t)c * N + j2];
    }
    proj_plus<R>(kv, (R)0.5 + hv, (R)0.5 - hv, y, t);
    alpha_eps<R>(eps, t, ayp);
#pragma unroll
    for (int c = 0; c < 4; ++c) t[c] = y[c] - t[c];
    alpha_eps<R>(eps, t, aym);
    proj_plus<R>(kv, (R)0.5 + hv, (R)0.5 - hv, z, t);
    alpha_eps<R>(eps, t, azp);
#pragma unroll
    for (int c = 0; c < 4; ++c) t[c] = z[c] - t[c];
    alpha_eps<R>(eps, t, azm);
    const R* o = om + 4 * (size_t)j;
    const R opp = o[0], opm = o[1], omp = o[2], omm = o[3];
    form_add<R>(tacc, zp, opp, ayp, opm, aym);
    form_add<R>(tacc, yp, opp, azp, opm, azm);
    form_add<R>(tacc, zm, omp, ayp, omm, aym);
    form_add<R>(tacc, ym, omp, azp, omm, azm);
  }
  const cpx<R> s = warp_sum<R>(tacc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = cvt<double>(s);
  __syncthreads();
  if (threadIdx.x == 0) {
    const long tab_row = (long)(clk->step + ls) * 7 + stage;
    const cpx<double> wt = ptab[3 * (tab_row + (long)inst * tab_stride) + 2];
    cpx<double> sacc = mk<double>(0, 0);
    for (int wi = 0; wi < (int)(blockDim.x >> 5); ++wi) sacc = sacc + red[wi];
    cpx<double>& a = sspart[(size_t)inst * gridDim.x + blockIdx.x];
    a = a + wt * sacc;
  }
}

// macc[inst] = (ss, D_U[4], D_V[4]): warp 0 sums the mode-sum accumulators of the instance, warps
// 1-4 the U wave's direct transform components, warps 5-8 the V wave's, each in a fixed order.
__global__ void __launch_bounds__(288) k_f2_final(const cpx<double>* __restrict__ sspart, int nbs,
                                                  const cpx<double>* __restrict__ dpart, int nbx,
                                                  cpx<double>* macc) {
  const int inst = blockIdx.x;
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  cpx<double> sacc = mk<double>(0, 0);
  if (q == 0) {
    for (int b = lane; b < nbs; b += 32) sacc = sacc + sspart[(size_t)inst * nbs + b];
  } else {
    const int wv = 2 * inst + (q - 1) / 4, c = (q - 1) % 4;
    for (int b = lane; b < nbx; b += 32) sacc = sacc + dpart[((size_t)wv * nbx + b) * 4 + c];
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    sacc.x += __shfl_down_sync(0xffffffffu, sacc.x, off);
    sacc.y += __shfl_down_sync(0xffffffffu, sacc.y, off);
  }
  if (lane == 0) macc[9 * inst + q] = sacc;
}

// Buffers and launch shapes of the partial-integration integrand.
template <typename R>
struct F2Plan {
  cpx<R>* Yspec = nullptr;   // [2 n_inst][4][N]: transforms of the stage values Y of both waves
  cpx<R>* Zspec = nullptr;   // [2 n_inst][4][N]: transforms of Z = -i V (Y + psi_b)
  int has_mid = 0;           // a y or z pass exists (it writes Yspec)
  cpx<R>* dph = nullptr;     // [2 n_inst][nx + ny + nz]: direct-transform phases per wave
  int* f2i = nullptr;        // [n_inst][4]: photon mode shift, table index
  R* omt = nullptr;          // [tables][N][4]: rho / Omega
  cpx<double>* dpart = nullptr;   // [2 n_inst][nbx][4]
  cpx<double>* sspart = nullptr;  // [n_inst][nbs]
  int n_inst = 0, nbx = 0, nbs = 0, rows = 0, ld = 0, tpl = 0;  // (k_f2_x: rows per block, threads per line)
  RadixPlan plan;
  const LineEntry<R>* entry = nullptr;  // the x axis's line kernels, if it has some
  size_t smem_x = 0;
};

template <typename R, int... R0>
static cudaError_t f2_attrs(std::integer_sequence<int, R0...>) {
  cudaError_t e = cudaSuccess;
  ((e = e != cudaSuccess ? e : cudaFuncSetAttribute(k_f2_x<R, R0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPassSmemMax)), ...);
  return e;
}

template <typename R>
static swf_status f2_prepare(swf_ctx* ctx, const GridDesc& g, int n_inst, const FieldDesc* fd_host,
                             const double* photon_host, const double* wave_k_host,
                             F2Plan<R>* p, cudaStream_t st) {
  cudaError_t e;
  {
    static std::atomic<bool> done[64];
    const int dv = dev_slot();
    if (!done[dv].load(std::memory_order_acquire)) {
      if ((e = f2_attrs<R>(std::integer_sequence<int, 1, 2, 3, 4, 5>())) != cudaSuccess)
        return cuda_status(e, "cudaFuncSetAttribute(k_f2_x)");
      done[dv].store(true, std::memory_order_release);
    }
  }
  const int nx = g.n[0];
  const int nrows = g.n[1] * g.n[2];
  const int nt = g.n[0] + g.n[1] + g.n[2];
  p->n_inst = n_inst;
  // a fixed shape (not the tuned one of the right-hand side's x passes): the block's rows decide the order
  // of the direct-transform sums, which must not depend on timing.  About 128 threads: as many rows as
  // that takes, at most 64.
  p->entry = line_of<R>(g, 0);
  if (p->entry) {
    p->tpl = line_threads(p->entry->r1, p->entry->r2);
    p->rows = std::max(1, std::min(128 / (4 * p->tpl), nrows));
    p->smem_x = xline_smem<R>(p->entry, p->rows);  // (at least as many values as threads)
  } else {
    make_pass_plan(nx, &p->plan);
    p->tpl = pass_threads(p->plan, 4);
    p->ld = padded_len<R>(nx);
    p->rows = std::max(1, std::min(std::min(128 / (4 * p->tpl), 64), nrows));
    p->smem_x = (size_t)8 * p->rows * p->ld * sizeof(cpx<R>);
  }
  p->nbx = (nrows + p->rows - 1) / p->rows;
  // one mode per thread where the grid allows (the gathers of the V modes are latency-bound)
  p->nbs = std::max(1, std::min((g.N + 255) / 256, (32 * sm_count() + n_inst - 1) / n_inst));
  // mode-sum tables, shared by instances with the same photon shift, trivial-axis momenta and k0
  std::vector<int> info(4 * (size_t)n_inst);
  std::vector<F2Table> tabs;
  std::map<std::vector<double>, int> seen;
  for (int i = 0; i < n_inst; ++i) {
    F2Table T;
    std::memset(&T, 0, sizeof T);
    const double* k = photon_host + 6 * i;
    for (int a = 0; a < 3; ++a) {
      // the modes are periodic and a photon's may lie any number of boxes out: 0 <= shift < n, so that the
      // mode sum reaches its partner with one wrap
      const long m = g.n[a] > 1 ? std::lround(k[a] * g.L[a] / 6.283185307179586476925286766559) : 0;
      T.shift[a] = (int)((m % g.n[a] + g.n[a]) % g.n[a]);
      T.Ku[a] = fd_host[2 * i].K[a];
      T.Kv[a] = fd_host[2 * i + 1].K[a];
    }
    T.k0 = std::sqrt(k[0] * k[0] + k[1] * k[1] + k[2] * k[2]);
    const std::vector<double> key = {(double)T.shift[0], (double)T.shift[1], (double)T.shift[2], T.Ku[0], T.Ku[1],
                                     T.Ku[2], T.Kv[0], T.Kv[1], T.Kv[2], T.k0};
    auto it = seen.find(key);
    int id;
    if (it == seen.end()) {
      id = (int)tabs.size();
      seen[key] = id;
      tabs.push_back(T);
    } else {
      id = it->second;
    }
    for (int a = 0; a < 3; ++a) info[4 * i + a] = T.shift[a];
    info[4 * i + 3] = id;
  }
  const int n_tab = (int)tabs.size();
  constexpr size_t esz = sizeof(cpx<R>);
  void *pY, *pZ, *pdph, *pinfo, *ptabs, *pomt, *pdp, *pss, *pwk;
  swf_status s;
  if ((s = ws_get(ctx, "bw2.yspec", (size_t)2 * n_inst * 4 * g.N * esz, &pY)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw2.zspec", (size_t)2 * n_inst * 4 * g.N * esz, &pZ)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw2.dph", (size_t)2 * n_inst * nt * esz, &pdph)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw2.wavek", sizeof(double) * 6 * (size_t)n_inst, &pwk)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw2.info", sizeof(int) * 4 * (size_t)n_inst, &pinfo)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw2.tabs", sizeof(F2Table) * (size_t)n_tab, &ptabs)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw2.omega", sizeof(R) * 4 * (size_t)n_tab * g.N, &pomt)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw2.dpart", sizeof(cpx<double>) * 4 * (size_t)2 * n_inst * p->nbx, &pdp)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw2.sspart", sizeof(cpx<double>) * (size_t)n_inst * p->nbs, &pss)) != SWF_OK) return s;
  p->Yspec = (cpx<R>*)pY;
  p->Zspec = (cpx<R>*)pZ;
  p->has_mid = (g.n[1] > 1 || g.n[2] > 1) ? 1 : 0;
  p->dph = (cpx<R>*)pdph;
  p->f2i = (int*)pinfo;
  p->omt = (R*)pomt;
  p->dpart = (cpx<double>*)pdp;
  p->sspart = (cpx<double>*)pss;
  if ((e = cudaMemcpyAsync(pwk, wave_k_host, sizeof(double) * 6 * n_inst, cudaMemcpyHostToDevice, st)) != cudaSuccess ||
      (e = cudaMemcpyAsync(pinfo, info.data(), sizeof(int) * info.size(), cudaMemcpyHostToDevice, st)) != cudaSuccess ||
      (e = cudaMemcpyAsync(ptabs, tabs.data(), sizeof(F2Table) * tabs.size(), cudaMemcpyHostToDevice, st)) != cudaSuccess)
    return cuda_status(e, "upload partial-integration tables");
  if ((e = cudaMemsetAsync(pdp, 0, sizeof(cpx<double>) * 4 * (size_t)2 * n_inst * p->nbx, st)) != cudaSuccess ||
      (e = cudaMemsetAsync(pss, 0, sizeof(cpx<double>) * (size_t)n_inst * p->nbs, st)) != cudaSuccess ||
      (e = cudaMemsetAsync(pY, 0, (size_t)2 * n_inst * 4 * g.N * esz, st)) != cudaSuccess)
    return cuda_status(e, "memset partial-integration accumulators");
  {
    ProfScope ps(ctx, "k_f2_dtables", st);
    k_f2_dtables<R><<<(2 * n_inst * nt + 127) / 128, 128, 0, st>>>((const double*)pwk, g, 2 * n_inst, p->dph);
  }
  {
    const long total = (long)n_tab * g.N;
    ProfScope ps(ctx, "k_f2_omega_table", st);
    k_f2_omega_table<R><<<(int)std::min((total + 255) / 256, 8192L), 256, 0, st>>>((const F2Table*)ptabs, g, n_tab,
                                                                                   p->omt);
  }
  // the host tables above are temporaries
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_status(e, "partial-integration tables");
  return SWF_OK;
}

// One evaluation of the partial-integration integrand at stage `stage` of step (clock step + ls), on
// the stage values ys of all waves: the x transform of Z (and of Y on grids without a y or z pass;
// otherwise the right-hand side's pass has written F[Y]) with the direct transforms, the forward y
// (and z) transforms of Z, then the mode sum.
template <typename R>
static swf_status f2_integrand(swf_ctx* ctx, const StageArgs<R>& A, const F2Plan<R>& p, const cpx<R>* ys,
                               const double* photon_dev, const cpx<double>* ptab, int tab_stride, int ls, int stage,
                               cudaStream_t st) {
  const GridDesc& g = A.g;
  const int G = p.n_inst;
  StageArgs<R> B = A;
  B.ls = ls;
  B.c = DP_C[stage];
  B.plan[0] = p.plan;
  {
    ProfScope ps(ctx, "k_f2_x", st);
    const dim3 grid(p.nbx, 2 * G);
    if (p.entry) {
      p.entry->f2<<<grid, 4 * p.rows * p.tpl, p.smem_x, st>>>(B, ys, p.Zspec, p.dph, ptab, tab_stride, stage, p.dpart,
                                                              p.rows);
    } else {
      auto* kernel = k_f2_x<R, 1>;
      switch (end_radix(p.plan, true)) {
        case 4: kernel = k_f2_x<R, 4>; break;
        case 2: kernel = k_f2_x<R, 2>; break;
        case 3: kernel = k_f2_x<R, 3>; break;
        case 5: kernel = k_f2_x<R, 5>; break;
        default: break;
      }
      kernel<<<grid, 4 * p.rows * p.tpl, p.smem_x, st>>>(B, ys, p.Yspec, p.Zspec, p.has_mid ? 0 : 1, p.dph, ptab,
                                                          tab_stride, stage, p.dpart, p.rows, p.ld, p.tpl);
    }
  }
  StageArgs<R> C = A;
  C.T = p.Zspec;
  C.yspec = nullptr;
  for (int axis = 1; axis <= 2; ++axis)
    if (g.n[axis] > 1) launch_mid<R>(ctx, C, axis, 1, 0, 0, false, 2 * G, st);
  {
    ProfScope ps(ctx, "k_f2_ss", st);
    k_f2_ss<R><<<dim3(p.nbs, G), kThreads, 0, st>>>(p.Yspec, p.Zspec, g, A.fd, photon_dev, p.f2i, p.omt, ptab, A.clk,
                                                    ls, stage, tab_stride, p.sspart);
  }
  return SWF_OK;
}

// One fixed-step march of F fields on one grid: plain (form 0), or U and V of F/2 Breit-Wheeler
// instances with the integrand of Eq. 17 (form 1; n_ph photons per instance) or of Eqs. 30-33 (form
// 2) integrated along.  setup() sizes the workspace and queues the tables, first() the evaluation
// k_1 = f(t_out, 0), step(ls) one step at clock offset ls (of a pair of steps), finish() what follows
// the last step.  All launches of one march go to one stream; several marches with workspaces of
// their own (tag) may run at once (march_multi).
template <typename R>
struct MarchPlan {
  swf_ctx* ctx = nullptr;
  cudaStream_t st = nullptr;
  GridDesc g;
  int n_steps = 0, F = 0, form = 0, n_inst = 0, n_ph = 1, NP = 0;
  int nph_blk = 1, nchunk = 1, nb = 1;
  double h = 0.0;
  StageArgs<R> A, open;
  bool chain = true;
  size_t state = 0;
  void *py = nullptr, *pk[7], *pys = nullptr, *pph = nullptr, *pkph = nullptr, *ptab = nullptr, *ppart = nullptr;
  int slot[7] = {0, 1, 2, 3, 4, 5, 6};
  MarchClock* clk = nullptr;
  F2Plan<R> p2;
  StepPairs pairs;

  swf_status buf(const std::string& name, size_t bytes, void** p) { return ws_get(ctx, name, bytes, p); }

  // tag: prefix of the workspace ("march" for a march that runs alone)
  swf_status setup(swf_ctx* c, const std::string& tag, const GridDesc& grid, double t_in, double t_out, int steps,
                   int n_f, const FieldDesc* fd_host, int form_, const double* photon_host, const double* wave_k_host,
                   int photons, cudaStream_t stream) {
    ctx = c;
    st = stream;
    g = grid;
    n_steps = steps;
    F = n_f;
    form = form_;
    n_ph = photons;
    n_inst = F / 2;
    NP = n_inst * n_ph;  // photon-instances: photon j of instance i is i n_ph + j
    h = (t_in - t_out) / n_steps;
    const bool alone = tag == "march";
    const std::string bt = alone ? "bw" : tag;  // prefix of the integrand's buffers
    // evaluations chain: each one's inverse x pass runs in one launch with the next one's forward x
    // pass, except on grids with x as the only non-trivial axis (one pass per evaluation).  The open
    // evaluation after every second step writes slot 0, as the first evaluation does, so a recorded
    // pair of steps replays unchanged.  (The integrands read only the stage value and the transforms
    // written by the forward passes, never T or the k slots.)
    chain = !(g.n[1] == 1 && g.n[2] == 1);
    swf_status s = prepare_args<R>(ctx, g, F, fd_host, &A, (form ? bt : tag).c_str(), st);
    if (s != SWF_OK) return s;
    state = (size_t)F * 4 * g.N * sizeof(cpx<R>);
    void *pT = nullptr, *pclk = nullptr;
    if ((s = buf(tag + ".y", state, &py)) != SWF_OK) return s;
    if ((s = buf(tag + ".T", state, &pT)) != SWF_OK) return s;
    for (int i = 0; i < 7; ++i)
      if ((s = buf(tag + ".k" + std::to_string(i), state, &pk[i])) != SWF_OK) return s;
    if ((s = buf(tag + ".clock", sizeof(MarchClock), &pclk)) != SWF_OK) return s;
    clk = (MarchClock*)pclk;
    cudaError_t e;
    if (form) {
      const int nt = g.n[0] + g.n[1] + g.n[2];
      if ((s = buf(bt + ".ystage", state, &pys)) != SWF_OK) return s;
      if ((s = buf(bt + ".photon", sizeof(double) * 6 * NP, &pph)) != SWF_OK) return s;
      if ((s = buf(bt + ".kph", sizeof(cpx<R>) * NP * nt, &pkph)) != SWF_OK) return s;
      // blocks per instance of the M-dot reduction: about four waves of the GPU in total, at least
      // 1024 sites per block (the same split for every photon count, so a photon of a scan sums
      // exactly as a solve of that photon alone); photons per block: 1, or 4 (8 in complex64) for
      // scans, which then read U and V once per site for the block's photons
      nph_blk = n_ph == 1 ? 1 : (sizeof(R) == 4 && n_ph > 4 ? 8 : 4);
      nchunk = (n_ph + nph_blk - 1) / nph_blk;
      nb = std::max(1, std::min((g.N + 1023) / 1024, (4 * sm_count() + n_inst - 1) / n_inst));
      if ((s = buf(bt + ".phase_table", sizeof(cpx<double>) * 3 * 7 * (size_t)n_steps * NP, &ptab)) != SWF_OK) return s;
      if ((s = buf(bt + ".mpart", sizeof(cpx<double>) * 3 * (size_t)nb * NP, &ppart)) != SWF_OK) return s;
      if ((e = cudaMemcpyAsync(pph, photon_host, sizeof(double) * 6 * NP, cudaMemcpyHostToDevice, st)) != cudaSuccess)
        return cuda_status(e, "upload photon table");
      {
        ProfScope ps(ctx, "k_photon_tables", st);
        k_photon_tables<R><<<(NP * nt + 127) / 128, 128, 0, st>>>((const double*)pph, g, NP, (cpx<R>*)pkph);
      }
      {
        const long total = (long)NP * n_steps * 7;
        ProfScope ps(ctx, "k_bw_phase_table", st);
        k_bw_phase_table<<<(int)std::min((total + 127) / 128, 4096L), 128, 0, st>>>(
            A.fd, (const double*)pph, NP, n_ph, n_steps, t_out, h, g.dx[0] * g.dx[1] * g.dx[2], form,
            (cpx<double>*)ptab);
      }
      if ((e = cudaMemsetAsync(ppart, 0, sizeof(cpx<double>) * 3 * (size_t)nb * NP, st)) != cudaSuccess)
        return cuda_status(e, "memset M accumulators");
    }
    if ((e = cudaMemsetAsync(py, 0, state, st)) != cudaSuccess) return cuda_status(e, "memset state");
    A.y = (cpx<R>*)py;
    A.T = (cpx<R>*)pT;
    if ((s = state_low_part<R>(ctx, tag + ".ylo", state, &A, st)) != SWF_OK) return s;
    {
      // shapes by timing, on the slots before they hold anything (the heaviest stage: six inputs)
      StageArgs<R> B = A;
      B.nterm = 6;
      for (int q = 0; q < 6; ++q) {
        B.kin[q] = (const cpx<R>*)pk[q + 1];
        B.coef[q] = 0.0;
        B.coef_r[q] = (R)0;
      }
      B.kout = (cpx<R>*)pk[0];
      B.t = t_out;
      if ((s = autotune_eval<R>(ctx, B, F, st)) != SWF_OK) return s;
    }
    if (form == 2 && (s = f2_prepare<R>(ctx, g, n_inst, fd_host, photon_host, wave_k_host, &p2, st)) != SWF_OK)
      return s;
    k_clock_set<<<1, 1, 0, st>>>(clk, t_out, h);
    A.clk = clk;
    return SWF_OK;
  }

  // k_1 = f(t_out, 0); the integrand of Eq. 17 vanishes at psi_s(t_out) = 0, the partial-integration
  // integrand does not (its source term is V psi_b): stage value y = 0
  swf_status first() {
    A.nterm = 0;
    A.write_y = 0;
    A.kout = (cpx<R>*)pk[slot[0]];
    A.ls = 0;
    A.c = 0.0;
    A.ystage = nullptr;
    set_next_node<R>(&A, 0, 0);
    swf_status s = chain ? launch_eval_open<R>(ctx, A, F, st) : launch_eval<R>(ctx, A, F, st);
    open = A;
    if (s == SWF_OK && form == 2)
      s = f2_integrand<R>(ctx, A, p2, (const cpx<R>*)py, (const double*)pph, (const cpx<double>*)ptab, 7 * n_steps, 0,
                          0, st);
    return s;
  }

  // One step at clock offset ls (stage times from the clock: tn = t_out + n h, t = tn + c_i h).  Stage
  // values with a quadrature weight: b_{i+1} for i = 2..5 and, for the new state (i = 6), b_1 of the
  // next step (the phase table holds 0 there on the last step, so every step launches the same kernels).
  swf_status step(int ls) {
    for (int i = 1; i < 7; ++i) {
      int nt = 0;
      for (int j = 0; j < i; ++j) {
        if (DP_A[i][j] == 0.0) continue;
        A.kin[nt] = (const cpx<R>*)pk[slot[j]];
        A.coef[nt] = h * DP_A[i][j];
        A.coef_r[nt] = (R)A.coef[nt];
        ++nt;
      }
      A.nterm = nt;
      A.write_y = (i == 6);
      A.kout = (cpx<R>*)pk[slot[i]];
      A.ls = ls;
      A.c = DP_C[i];
      set_next_node<R>(&A, ls, i);
      const bool weighted = form && i >= 2;
      A.ystage = weighted ? (cpx<R>*)pys : nullptr;
      A.yspec = (weighted && form == 2) ? p2.Yspec : nullptr;  // the y or z pass writes F[Y] (if there is one)
      swf_status r = chain ? launch_eval_chain<R>(ctx, open, A, F, st) : launch_eval<R>(ctx, A, F, st);
      if (r != SWF_OK) return r;
      open = A;
      if (!weighted) continue;
      if (form == 2) {
        if ((r = f2_integrand<R>(ctx, A, p2, (const cpx<R>*)pys, (const double*)pph, (const cpx<double>*)ptab,
                                 7 * n_steps, ls, i, st)) != SWF_OK)
          return r;
        continue;
      }
      ProfScope ps(ctx, "k_mdot", st);
      auto* kernel = nph_blk == 1 ? k_mdot<R, 1> : nph_blk == 4 ? k_mdot<R, 4> : k_mdot<R, sizeof(R) == 4 ? 8 : 4>;
      launch_chained(may_chain<R>(st), kernel, dim3(nb, n_inst * nchunk), 256, 0, st, (const cpx<R>*)pys, A.gcplx, (const cpx<R>*)pkph,
                     (const double*)pph, g, (const cpx<double>*)ptab, clk, ls, i, 7 * n_steps, n_ph, (cpx<double>*)ppart);
    }
    std::swap(slot[0], slot[6]);
    return SWF_OK;
  }

  swf_status pair() {
    const swf_status r = step(0);
    return r == SWF_OK ? step(1) : r;
  }
  swf_status prepare_pairs() {
    return n_steps > 1 ? pairs.prepare(ctx, st, clk, [&] { return pair(); }) : SWF_OK;
  }
  swf_status launch_pair() {
    return pairs.launch(ctx, clk, [&] { return pair(); });
  }

  // The odd step, the open evaluation's end, the integrals and the state.
  swf_status finish(void* psi_out, double2* macc) {
    swf_status s = pairs.finish();
    if (s != SWF_OK) return s;
    if (n_steps % 2 && (s = step(0)) != SWF_OK) return s;
    if (chain && (s = launch_eval_close<R>(ctx, open, F, st)) != SWF_OK) return s;
    if (form == 2) {
      ProfScope ps(ctx, "k_f2_final", st);
      k_f2_final<<<n_inst, 288, 0, st>>>(p2.sspart, p2.nbs, p2.dpart, p2.nbx, (cpx<double>*)macc);
    } else if (form == 1) {
      ProfScope ps(ctx, "k_mdot_final", st);
      k_mdot_final<<<NP, 96, 0, st>>>((const cpx<double>*)ppart, nb, (cpx<double>*)macc);
    }
    cudaError_t e = cudaMemcpyAsync(psi_out, py, state, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return cuda_status(e, "copy psi(t_in)");
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_status(e, "march kernels");
    return SWF_OK;
  }

  // A march that runs alone: everything in order.
  swf_status run(void* psi_out, double2* macc) {
    swf_status s = first();
    if (s == SWF_OK) s = prepare_pairs();
    for (int p = 0; p < n_steps / 2 && s == SWF_OK; ++p) s = launch_pair();
    if (s != SWF_OK) {
      pairs.finish();
      return s;
    }
    return finish(psi_out, macc);
  }
};

template <typename R>
static swf_status march_impl(swf_ctx* ctx, const GridDesc& g, double t_in, double t_out, int n_steps, int F,
                             const FieldDesc* fd_host, void* psi_out, cudaStream_t st) {
  MarchPlan<R> P;
  const swf_status s = P.setup(ctx, "march", g, t_in, t_out, n_steps, F, fd_host, 0, nullptr, nullptr, 1, st);
  return s == SWF_OK ? P.run(psi_out, nullptr) : s;
}

template <typename R>
static swf_status march_bw_impl(swf_ctx* ctx, const GridDesc& g, double t_in, double t_out, int n_steps, int n_inst,
                                const FieldDesc* fd_host, const double* photon_host, void* psi_out, double2* macc,
                                cudaStream_t st, int form, const double* wave_k_host, int n_ph) {
  MarchPlan<R> P;
  const swf_status s =
      P.setup(ctx, "march", g, t_in, t_out, n_steps, 2 * n_inst, fd_host, form, photon_host, wave_k_host, n_ph, st);
  return s == SWF_OK ? P.run(psi_out, macc) : s;
}

swf_status march_bw(swf_ctx* ctx, const GridDesc& g, double t_in, double t_out, int n_steps, int n_inst,
                    const FieldDesc* fd_host, const double* photon_host, swf_precision prec, void* psi_out,
                    double2* macc, cudaStream_t st, int form, const double* wave_k_host, int n_ph) {
  if (form == 2 && (!wave_k_host || n_ph != 1)) {
    set_error("march_bw: the partial-integration form needs the direct-transform momenta and one photon per instance");
    return SWF_EINVAL;
  }
  if (n_ph < 1) {
    set_error("march_bw: at least one photon per instance");
    return SWF_EINVAL;
  }
  if (prec == SWF_C64)
    return march_bw_impl<float>(ctx, g, t_in, t_out, n_steps, n_inst, fd_host, photon_host, psi_out, macc, st, form,
                                wave_k_host, n_ph);
  return march_bw_impl<double>(ctx, g, t_in, t_out, n_steps, n_inst, fd_host, photon_host, psi_out, macc, st, form,
                               wave_k_host, n_ph);
}

// ---------------------------------------------------------------- step-size-controlled Breit-Wheeler march
// Per attempt and photon-instance: the stage rows of the integrand's phase table from the
// controller's t and h (stage i at t + c_i h): the U and V background time phases and the
// quadrature factor h b_{i+1} dx^d e^{-i k0 t} (stage 0 is the accepted state y_n, stage 6 the
// new state, whose weight b_7 is zero).  rows [inst][7][3].
__global__ void k_bw_attempt_rows(const FieldDesc* fd, const double* photon, const StepControl* ctl, double cell,
                                  cpx<double>* rows) {
  const int inst = blockIdx.x, i = threadIdx.x;
  if (i >= 7 || ctl->done) return;
  const double DPc[7] = {0.0, 0.2, 0.3, 0.8, 8.0 / 9.0, 1.0, 1.0};
  const double DPb[7] = {35.0 / 384, 0.0, 500.0 / 1113, 125.0 / 192, -2187.0 / 6784, 11.0 / 84, 0.0};
  const double t = ctl->t + DPc[i] * ctl->h;
  const double w = ctl->h * DPb[i];
  const FieldDesc& FU = fd[2 * inst];
  const FieldDesc& FV = fd[2 * inst + 1];
  const double* k = photon + 6 * inst;
  const double k0 = sqrt(k[0] * k[0] + k[1] * k[1] + k[2] * k[2]);
  double sn, cs;
  cpx<double>* r = rows + 3 * (7 * (size_t)inst + i);
  sincos(FU.tsign * FU.e0 * t, &sn, &cs);
  r[0] = mk<double>(cs, sn);
  sincos(FV.tsign * FV.e0 * t, &sn, &cs);
  r[1] = mk<double>(cs, sn);
  sincos(-k0 * t, &sn, &cs);
  r[2] = mk<double>(w * cell * cs, w * cell * sn);
}

// After an accepted attempt: the attempt's integrand sums join the march's.
__global__ void k_mdot_commit(const StepControl* ctl, const cpx<double>* __restrict__ tryacc, cpx<double>* acc,
                              size_t n) {
  if (!ctl->ok) return;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    acc[i] = acc[i] + tryacc[i];
}

// The Breit-Wheeler march (U and V of every instance, the integrand of Eq. 17 appended) with
// step-size control: one controller for all 2 n_inst waves (the error norm is the largest of
// theirs), each attempt one graph replay as in march_adaptive_impl.  The integrand is summed per
// attempt and committed only when the step is accepted.  macc [n_inst][3] as march_bw's form 1.
template <typename R>
static swf_status march_bw_adaptive_impl(swf_ctx* ctx, const GridDesc& g, double t_in, double t_out, double h0,
                                         int max_attempts, int n_inst, const FieldDesc* fd_host,
                                         const double* photon_host, void* psi_out, double2* macc, cudaStream_t st) {
  const int F = 2 * n_inst;
  StageArgs<R> A;
  swf_status s = prepare_args<R>(ctx, g, F, fd_host, &A, "bw", st);
  if (s != SWF_OK) return s;
  const size_t per_field = (size_t)4 * g.N;
  const size_t state = (size_t)F * per_field * sizeof(cpx<R>);
  const int nt = g.n[0] + g.n[1] + g.n[2];
  void *py, *pyn, *pT, *pys, *pk[7], *pctl, *ppart, *pph, *pkph, *prow, *pacc, *ptry, *pclk;
  if ((s = ws_get(ctx, "march.y", state, &py)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "march.ynew", state, &pyn)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "march.T", state, &pT)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw.ystage", state, &pys)) != SWF_OK) return s;
  for (int i = 0; i < 7; ++i) {
    char nm[32];
    std::snprintf(nm, sizeof nm, "march.k%d", i);
    if ((s = ws_get(ctx, nm, state, &pk[i])) != SWF_OK) return s;
  }
  const int nbe = error_blocks(per_field);
  const int nb = std::max(1, std::min((g.N + 1023) / 1024, (4 * sm_count() + n_inst - 1) / n_inst));
  const size_t nacc = (size_t)3 * nb * n_inst;
  if ((s = ws_get(ctx, "march.ctl", sizeof(StepControl), &pctl)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "march.err_part", sizeof(double) * (size_t)nbe * F, &ppart)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw.photon", sizeof(double) * 6 * n_inst, &pph)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw.kph", sizeof(cpx<R>) * n_inst * nt, &pkph)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw.arows", sizeof(cpx<double>) * 3 * 7 * (size_t)n_inst, &prow)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw.mpart", sizeof(cpx<double>) * nacc, &pacc)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw.mtry", sizeof(cpx<double>) * nacc, &ptry)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "bw.aclock", sizeof(MarchClock), &pclk)) != SWF_OK) return s;
  cudaError_t e = cudaMemcpyAsync(pph, photon_host, sizeof(double) * 6 * n_inst, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_status(e, "upload photon table");
  {
    ProfScope ps(ctx, "k_photon_tables", st);
    k_photon_tables<R><<<(n_inst * nt + 127) / 128, 128, 0, st>>>((const double*)pph, g, n_inst, (cpx<R>*)pkph);
  }
  // k_mdot reads its phase row at (clock step + ls) * 7 + stage: a clock at step 0 and a row
  // stride of 7 select the attempt's rows
  MarchClock* clk = (MarchClock*)pclk;
  k_clock_set<<<1, 1, 0, st>>>(clk, t_out, 0.0);
  if ((e = cudaMemsetAsync(py, 0, state, st)) != cudaSuccess) return cuda_status(e, "memset state");
  if ((e = cudaMemsetAsync(pacc, 0, sizeof(cpx<double>) * nacc, st)) != cudaSuccess)
    return cuda_status(e, "memset M accumulators");
  StepControl c0{};
  c0.t = t_out;
  c0.h = (t_in < t_out) ? -std::fabs(h0) : std::fabs(h0);
  if (std::fabs(c0.h) > std::fabs(t_in - t_out)) c0.h = t_in - t_out;
  c0.t_in = t_in;
  c0.span = std::fabs(t_in - t_out);
  c0.rtol = ctx->rtol;
  c0.atol = ctx->atol;
  c0.max_attempts = max_attempts;
  StepControl* ctl = (StepControl*)pctl;
  e = cudaMemcpyAsync(ctl, &c0, sizeof(StepControl), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_status(e, "upload step control");
  A.y = (cpx<R>*)py;
  A.T = (cpx<R>*)pT;
  {
    StageArgs<R> B = A;  // shapes by timing, before the slots hold anything
    B.nterm = 6;
    for (int q = 0; q < 6; ++q) {
      B.kin[q] = (const cpx<R>*)pk[q + 1];
      B.coef[q] = 0.0;
      B.coef_r[q] = (R)0;
    }
    B.write_y = 0;
    B.ystage = nullptr;
    B.kout = (cpx<R>*)pk[0];
    B.t = t_out;
    if ((s = autotune_eval<R>(ctx, B, F, st)) != SWF_OK) return s;
  }
  // k_1 = f(t_out, 0)
  A.nterm = 0;
  A.write_y = 0;
  A.kout = (cpx<R>*)pk[0];
  A.t = t_out;
  if ((s = launch_eval<R>(ctx, A, F, st)) != SWF_OK) return s;
  A.ctl = ctl;
  A.ynew = (cpx<R>*)pyn;
  ErrWeights W;
  for (int j = 0; j < 7; ++j) W.db[j] = DP_DB[j];
  const double cell = g.dx[0] * g.dx[1] * g.dx[2];
  auto mdot = [&](const void* ys, int stage) {
    ProfScope ps(ctx, "k_mdot", st);
    k_mdot<R, 1><<<dim3(nb, n_inst), 256, 0, st>>>((const cpx<R>*)ys, A.gcplx, (const cpx<R>*)pkph,
                                                   (const double*)pph, g, (const cpx<double>*)prow, clk, 0, stage,
                                                   7, 1, (cpx<double>*)ptry);
  };
  // an attempt's evaluations chain through their x passes (the integrand reads only the stage
  // values); the attempt's last one is closed before the error estimate reads k_7
  const bool chain = !(g.n[1] == 1 && g.n[2] == 1);
  auto attempt = [&]() -> swf_status {
    cudaError_t e1 = cudaMemsetAsync(ptry, 0, sizeof(cpx<double>) * nacc, st);
    if (e1 != cudaSuccess) return cuda_status(e1, "memset attempt sums");
    {
      ProfScope ps(ctx, "k_bw_attempt_rows", st);
      k_bw_attempt_rows<<<n_inst, 32, 0, st>>>(A.fd, (const double*)pph, ctl, cell, (cpx<double>*)prow);
    }
    mdot(py, 0);  // stage 1 of the step: the accepted state
    StageArgs<R> open = A;
    for (int i = 1; i < 7; ++i) {
      int ntm = 0;
      for (int j = 0; j < i; ++j) {
        if (DP_A[i][j] == 0.0) continue;
        A.kin[ntm] = (const cpx<R>*)pk[j];
        A.coef[ntm] = DP_A[i][j];  // times the device-held h in k_first
        ++ntm;
      }
      A.nterm = ntm;
      A.write_y = (i == 6);
      A.kout = (cpx<R>*)pk[i];
      A.c = DP_C[i];
      set_next_node<R>(&A, 0, i);
      const bool weighted = i >= 2 && i <= 5;  // b_2 = b_7 = 0
      A.ystage = weighted ? (cpx<R>*)pys : nullptr;
      swf_status r = !chain ? launch_eval<R>(ctx, A, F, st)
                            : (i == 1 ? launch_eval_open<R>(ctx, A, F, st) : launch_eval_chain<R>(ctx, open, A, F, st));
      if (r != SWF_OK) return r;
      open = A;
      if (weighted) mdot(pys, i);
    }
    if (chain) {
      swf_status r = launch_eval_close<R>(ctx, open, F, st);
      if (r != SWF_OK) return r;
    }
    {
      ProfScope ps(ctx, "k_step_error", st);
      k_step_error<R><<<dim3(nbe, F), kErrThreads, 0, st>>>(
          (const cpx<R>*)py, (const cpx<R>*)pyn, (const cpx<R>*)pk[0], (const cpx<R>*)pk[2], (const cpx<R>*)pk[3],
          (const cpx<R>*)pk[4], (const cpx<R>*)pk[5], (const cpx<R>*)pk[6], W, ctl, per_field, (double*)ppart);
    }
    {
      ProfScope ps(ctx, "k_step_control", st);
      k_step_control<<<1, 256, 0, st>>>(ctl, (const double*)ppart, nbe, F, (double)per_field);
    }
    {
      ProfScope ps(ctx, "k_step_accept", st);
      const size_t n = (size_t)F * per_field;
      k_step_accept<R><<<(unsigned)std::min<size_t>((n + 255) / 256, 4096), 256, 0, st>>>(
          ctl, (cpx<R>*)py, (const cpx<R>*)pyn, (cpx<R>*)pk[0], (const cpx<R>*)pk[6], n);
    }
    {
      ProfScope ps(ctx, "k_mdot_commit", st);
      k_mdot_commit<<<(unsigned)std::min<size_t>((nacc + 255) / 256, 1024), 256, 0, st>>>(
          ctl, (const cpx<double>*)ptry, (cpx<double>*)pacc, nacc);
    }
    return SWF_OK;
  };
  StepControl hc{};
  if ((s = run_attempts(ctx, st, max_attempts, ctl, attempt, &hc)) != SWF_OK) return s;
  ctx->last_accepted = hc.accepted;
  ctx->last_rejected = hc.rejected;
  if (hc.failed) {
    set_error("step-size-controlled march: no convergence (too many attempts or a non-finite error)");
    return SWF_ENUMERIC;
  }
  {
    ProfScope ps(ctx, "k_mdot_final", st);
    k_mdot_final<<<n_inst, 96, 0, st>>>((const cpx<double>*)pacc, nb, (cpx<double>*)macc);
  }
  e = cudaMemcpyAsync(psi_out, py, state, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return cuda_status(e, "copy psi(t_in)");
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "Breit-Wheeler march kernels");
  return SWF_OK;
}

swf_status march_bw_adaptive(swf_ctx* ctx, const GridDesc& g, double t_in, double t_out, double h0, int max_attempts,
                             int n_inst, const FieldDesc* fd_host, const double* photon_host, swf_precision prec,
                             void* psi_out, double2* macc, cudaStream_t st) {
  if (prec == SWF_C64)
    return march_bw_adaptive_impl<float>(ctx, g, t_in, t_out, h0, max_attempts, n_inst, fd_host, photon_host,
                                         psi_out, macc, st);
  return march_bw_adaptive_impl<double>(ctx, g, t_in, t_out, h0, max_attempts, n_inst, fd_host, photon_host,
                                        psi_out, macc, st);
}

// ---------------------------------------------------------------- multi-grid march (batching of uneven grids)
// Groups of fields on different grids that share one time grid (t_out, t_in, steps) march side by
// side: each group is a MarchPlan with a workspace and a stream of its own, its step pair one CUDA
// graph, and the graphs of all groups are replayed in turn, so that small grids fill the SMs together.
// A group's kernels and shapes are those of marching it alone: bitwise the same result.

constexpr int kMaxMultiGroups = 8;

// Streams of the groups (kept with the context) and their fork and join events.
static swf_status multi_streams(swf_ctx* ctx, int n) {
  while ((int)ctx->multi_st.size() < n) {
    cudaStream_t s = nullptr;
    cudaEvent_t ev = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e == cudaSuccess && (e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming)) != cudaSuccess)
      cudaStreamDestroy(s);
    if (e != cudaSuccess) return cuda_status(e, "multi-grid streams");
    ctx->multi_st.push_back(s);
    ctx->multi_ev.push_back(ev);
  }
  return SWF_OK;
}

template <typename R>
static swf_status march_multi_impl(swf_ctx* ctx, const std::vector<MultiGroup>& G, double t_in, double t_out,
                                   int n_steps, int bw, cudaStream_t st) {
  const int ng = (int)G.size();
  swf_status s = multi_streams(ctx, ng + 1);
  if (s != SWF_OK) return s;
  std::vector<MarchPlan<R>> P(ng);
  // tables and tuned shapes on st, one group after another (the tuner times its launches alone)
  for (int gi = 0; gi < ng && s == SWF_OK; ++gi)
    s = P[gi].setup(ctx, "mg" + std::to_string(gi), G[gi].g, t_in, t_out, n_steps, G[gi].F, G[gi].fd, bw ? 1 : 0,
                    G[gi].photon, nullptr, 1, st);
  if (s != SWF_OK) return s;
  cudaError_t e = cudaEventRecord(ctx->multi_ev[ng], st);
  for (int gi = 0; gi < ng && e == cudaSuccess; ++gi) {
    P[gi].st = ctx->multi_st[gi];
    e = cudaStreamWaitEvent(P[gi].st, ctx->multi_ev[ng], 0);
  }
  if (e != cudaSuccess) return cuda_status(e, "fork the multi-grid streams");
  for (int gi = 0; gi < ng && s == SWF_OK; ++gi) s = P[gi].first();
  for (int gi = 0; gi < ng && s == SWF_OK; ++gi) s = P[gi].prepare_pairs();
  for (int p = 0; p < n_steps / 2 && s == SWF_OK; ++p)
    for (int gi = 0; gi < ng && s == SWF_OK; ++gi) s = P[gi].launch_pair();
  for (int gi = 0; gi < ng; ++gi) {
    if (s == SWF_OK) s = P[gi].finish(G[gi].psi_out, (double2*)G[gi].macc);
    else P[gi].pairs.finish();
  }
  for (int gi = 0; gi < ng; ++gi) {  // st continues after every group (also after an error)
    if (e == cudaSuccess) e = cudaEventRecord(ctx->multi_ev[gi], P[gi].st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ctx->multi_ev[gi], 0);
  }
  if (s != SWF_OK) return s;
  // the host tables of the set-up are the sources of asynchronous uploads
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_status(e, "multi-grid march");
  ctx->multi_marches += 1;
  return SWF_OK;
}

bool multi_compatible(const GridDesc& a, const GridDesc& b) {
  return (a.n[1] > 1) == (b.n[1] > 1) && (a.n[2] > 1) == (b.n[2] > 1);
}

swf_status march_multi(swf_ctx* ctx, const std::vector<MultiGroup>& groups, double t_in, double t_out, int n_steps,
                       swf_precision prec, int bw, cudaStream_t st) {
  if (groups.empty() || (int)groups.size() > kMaxMultiGroups) {
    set_error("multi-grid march: 1 to 8 groups");
    return SWF_EINVAL;
  }
  for (const MultiGroup& M : groups) {
    if (!multi_compatible(M.g, groups[0].g) || M.F < 1 || (bw && (M.F % 2 || !M.photon || !M.macc))) {
      set_error("multi-grid march: groups must share the non-trivial axes (and carry U, V pairs and photons)");
      return SWF_EINVAL;
    }
  }
  ctx->in_multi = true;  // its kernels are timed under names of their own
  const swf_status s = prec == SWF_C64 ? march_multi_impl<float>(ctx, groups, t_in, t_out, n_steps, bw, st)
                                       : march_multi_impl<double>(ctx, groups, t_in, t_out, n_steps, bw, st);
  ctx->in_multi = false;
  return s;
}

// Plain marches of several groups (the spin reuse of march_fields within each group).
swf_status march_fields_multi(swf_ctx* ctx, const std::vector<MultiGroup>& groups, double t_in, double t_out,
                              int n_steps, swf_precision prec, cudaStream_t st) {
  const int ng = (int)groups.size();
  std::vector<MultiGroup> todo(groups);
  std::vector<std::vector<int>> rep(ng), sgn(ng);
  std::vector<std::vector<FieldDesc>> uniq(ng);
  const size_t elem = prec == SWF_C64 ? 8 : 16;
  swf_status s;
  for (int gi = 0; gi < ng; ++gi) {
    const MultiGroup& M = groups[gi];
    const int n_u = ctx->dedupe ? dedupe_fields(M.g, M.F, M.fd, rep[gi], sgn[gi], uniq[gi]) : M.F;
    ctx->fields_marched += n_u;
    if (n_u == M.F) {
      rep[gi].clear();
      continue;
    }
    void* pu = nullptr;
    if ((s = ws_get(ctx, "mg.unique" + std::to_string(gi), (size_t)n_u * 4 * M.g.N * elem, &pu)) != SWF_OK) return s;
    todo[gi].F = n_u;
    todo[gi].fd = uniq[gi].data();
    todo[gi].psi_out = pu;
  }
  if ((s = march_multi(ctx, todo, t_in, t_out, n_steps, prec, 0, st)) != SWF_OK) return s;
  for (int gi = 0; gi < ng; ++gi) {
    if (rep[gi].empty()) continue;
    const MultiGroup& M = groups[gi];
    void* ptab = nullptr;
    if ((s = ws_get(ctx, "mg.unique_map" + std::to_string(gi), sizeof(int) * 2 * (size_t)M.F, &ptab)) != SWF_OK)
      return s;
    std::vector<int> tabv(rep[gi]);
    tabv.insert(tabv.end(), sgn[gi].begin(), sgn[gi].end());
    cudaError_t e = cudaMemcpyAsync(ptab, tabv.data(), sizeof(int) * 2 * (size_t)M.F, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return cuda_status(e, "upload field map");
    const dim3 grid((unsigned)std::min<size_t>((M.g.N + 255) / 256, 1024), M.F, 4);
    ProfScope ps(ctx, "k_expand_fields", st);
    if (prec == SWF_C64)
      k_expand_fields<float><<<grid, 256, 0, st>>>((const cpx<float>*)todo[gi].psi_out, (const int*)ptab,
                                                   (const int*)ptab + M.F, (size_t)M.g.N, (cpx<float>*)M.psi_out);
    else
      k_expand_fields<double><<<grid, 256, 0, st>>>((const cpx<double>*)todo[gi].psi_out, (const int*)ptab,
                                                    (const int*)ptab + M.F, (size_t)M.g.N, (cpx<double>*)M.psi_out);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e, "expand fields");
    e = cudaStreamSynchronize(st);  // the host table must outlive its upload
    if (e != cudaSuccess) return cuda_status(e, "expand fields");
  }
  return SWF_OK;
}

}  // namespace swf
