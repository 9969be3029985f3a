// Line passes of the march whose transforms live in registers: a line of n = R1 R2 points is
// transformed by max(R1, R2) threads with one exchange through shared memory per direction.
//
// With x = i + R2 q (i < R2, q < R1) and k = k1 + R1 k2 (k1 < R1, k2 < R2), thread i of a line owns
// the R1 points x of one i (the "site side") and thread k1 the R2 modes k of one k1 (the "mode
// side"): forward is a DFT over q, the twiddle exp(-2 pi i i k1/n), the exchange and a DFT over i;
// inverse runs the same steps backwards.  Whatever happens on the sites between an inverse and the
// next forward transform (k_i, the stage combine, the local term) or on the modes between a forward
// and an inverse (H0) happens in the registers of the thread that owns them.  An evaluation's line
// therefore passes through shared memory twice (Stockham passes: six times, with a barrier each), and
// global memory is read into and written from the same registers: n/R2 = R1 independent loads per thread
// and array, R2 (or R1) neighbouring points per load instruction.
//
// What bounds them, and what they measured against the Stockham passes they replaced (complex64, per
// launch): on 256^3 the x pass moves 8.8 arrays on average, 53 in the six launches of a step, at 5.8 TB/s,
// 0.86 of the measured copy rate (1276 -> 816 us), and the y and z passes two each at 4.7 TB/s (489 ->
// 227 us); 16 fields of 256^2 beside the fused kernel, on 40 SMs: x pass 302 ->
// 177 us, y pass 147 -> 69 us (before: six barriers and six trips through shared memory per line, 20 %
// of the issue slots used).  The x pass takes 128 registers (the older stage terms are summed before
// the exchange, so that their loads overlap those of T); the y and z passes 64 where R1, R2 <= 16, for
// 32 warps per SM.
#pragma once

#include "swf_stage.cuh"

namespace swf {

// What an x pass does (the flags of k_xline).
enum : int {
  XL_LAST = 1,     // close evaluation P: inverse x-FFT, k = (that) + Z
  XL_FIRST = 2,    // open evaluation A: stage combine, local term, forward x-FFT
  XL_REGK = 4,     // the newest term of A's stage combine is P's output (still in registers)
  XL_FACTORS = 8,  // A's time factors were computed by a launch before this one (y or z pass, k_tables)
};
// What a y or z pass does (the flags of k_line).
enum : int { LN_FWD = 1, LN_H0 = 2, LN_INV = 4 };

template <typename R> using XLineKernel = void (*)(StageArgs<R>, StageArgs<R>, int, int);
template <typename R> using LineKernel = void (*)(StageArgs<R>, int, int, int);
template <typename R>
using F2LineKernel = void (*)(StageArgs<R>, const cpx<R>*, cpx<R>*, const cpx<R>*, const cpx<double>*, int, int,
                              cpx<double>*, int);

// One length n = r1 r2 and its kernels.
template <typename R>
struct LineEntry {
  int n, r1, r2;
  XLineKernel<R> x;
  LineKernel<R> line;
  F2LineKernel<R> f2;
};

// Threads per line and shared-memory complex values per line of the two kernels.  x pass: rows of R2
// values at an odd stride, so that threads k1 writing row k1 and threads i reading column i both
// fall on distinct banks; y/z pass: neighbouring threads hold neighbouring lines, so only the line
// stride has to be odd.
__host__ __device__ constexpr int line_threads(int r1, int r2) { return r1 > r2 ? r1 : r2; }
__host__ __device__ constexpr int xline_stride(int r1, int r2) { return r1 * (r2 | 1); }
__host__ __device__ constexpr int line_stride(int r1, int r2) { return (r1 * r2) | 1; }
constexpr int kXLineThreads = 256;                                                // at most, per block
// k_line's block: whole warps (the shuffles of H0 name all 32 lanes)
__host__ __device__ constexpr int line_block(int r1, int r2, int lg) { return ((4 << lg) * line_threads(r1, r2) + 31) & ~31; }
constexpr int line_max_threads(int esz) { return esz == 8 ? 512 : 256; }          // y/z pass, by sizeof(cpx<R>)

#ifdef __CUDACC__
// ---- what happens on the sites, NV points gs + q stride (q < NV) of one line and component

// The older terms of A's stage combine: v = [y +] sum of its first nold terms (ff: without y, which
// joins in float-float when the sum is complete).
template <typename R, int NV>
__device__ __forceinline__ void combine_sites(const StageArgs<R>& A, int nold, bool ff, size_t gs, int stride, cpx<R>* v) {
  if (ff) {
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = mk<R>(0, 0);
  } else {
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = A.y[gs + q * stride];
  }
#pragma unroll
  for (int t = 0; t < 6; ++t)
    if (t < nold) {
      const R co = A.ctl ? (R)(A.coef[t] * A.ctl->h) : A.coef_r[t];  // a_ij, times h here under control
      const cpx<R>* __restrict__ kt = A.kin[t] + gs;
#pragma unroll
      for (int q = 0; q < NV; ++q) v[q] = v[q] + co * kt[q * stride];
    }
}

// k = Z + (the inverse transform r) of evaluation P, also left in r.
template <typename R, int NV>
__device__ __forceinline__ void close_sites(const StageArgs<R>& P, size_t gs, int stride, cpx<R>* r) {
  cpx<R>* ko = P.kout + gs;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    r[q] = ko[q * stride] + r[q];
    ko[q * stride] = r[q];
  }
}

// The local term Z = -i V (Y + psi_b): V has one non-zero component, so every component of Z comes from
// one component of Y + psi_b.  Component c feeds component source_component (A_1, A_2: the mirrored one,
// A_3: two away): -i V phi = rot a phi with rot = -i, times i (-i) for A_2's even (odd) components, times
// -1 for A_3's odd ones; 0 without a field.
__device__ __forceinline__ int source_component(int acomp, int c) {
  return acomp == 1 || acomp == 2 ? 3 - c : acomp == 3 ? (c ^ 2) : c;
}
template <typename R>
__device__ __forceinline__ cpx<R> source_rotation(int acomp, int c) {
  return acomp < 0 ? mk<R>(0, 0)
         : acomp == 2 ? ((c & 1) ? mk<R>(-1, 0) : mk<R>(1, 0))
         : acomp == 3 && (c & 1) ? mk<R>(0, 1)
                                 : mk<R>(0, -1);
}
// rot a (y + br e), rot = +-1 or +-i (or 0)
template <typename R>
__device__ __forceinline__ cpx<R> source_term(cpx<R> y, cpx<R> br, cpx<R> e, R a, cpx<R> rot) {
  const cpx<R> phi = mk<R>(a * ((y.x + br.x * e.x) - br.y * e.y), a * ((y.y + br.x * e.y) + br.y * e.x));
  return rot.x != (R)0 ? rot.x * phi : mk<R>(-rot.y * phi.y, rot.y * phi.x);
}

// The stage combine's end: v becomes the stage value Y, which is stored where A asks for it.
template <typename R, int NV>
__device__ __forceinline__ void finish_sites(const StageArgs<R>& A, bool ff, size_t gs, int stride, cpx<R>* v) {
  if (ff) {
    // the new state: (y, ylo) += the step's increment in float-float, so that the single-precision
    // rounding of y does not accumulate over steps
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      const cpx<R> yh = A.y[gs + q * stride];
      const cpx<R> lo = A.ylo[gs + q * stride];
      float sx = (float)v[q].x, sy = (float)v[q].y, lx = (float)lo.x, ly = (float)lo.y;
      ff_accumulate((float)yh.x, lx, sx);
      ff_accumulate((float)yh.y, ly, sy);
      v[q] = mk<R>((R)sx, (R)sy);
      A.ylo[gs + q * stride] = mk<R>((R)lx, (R)ly);
    }
  }
  if (A.write_y) {
    cpx<R>* yo = (A.ynew ? A.ynew : A.y) + gs;
#pragma unroll
    for (int q = 0; q < NV; ++q) yo[q * stride] = v[q];
  }
  if (A.ystage) {
#pragma unroll
    for (int q = 0; q < NV; ++q) A.ystage[gs + q * stride] = v[q];
  }
}

// The same, then the local term: Z goes to the output slot (of the component this thread's one feeds)
// until the evaluation is closed.  x = x0 + q stride are the sites' x indices, f, c, row the line, ftr and
// tf its time factors.
template <typename R, int NV>
__device__ __forceinline__ void open_sites(const StageArgs<R>& A, bool ff, size_t gs, int x0, int stride, int f, int c,
                                           int row, R ftr, cpx<R> tf, cpx<R>* v) {
  finish_sites<R, NV>(A, ff, gs, stride, v);
  const int nx = A.g.n[0], ny = A.g.n[1], nz = A.g.n[2], nt = nx + ny + nz;
  const size_t N = A.g.N;
  const R* __restrict__ gx = A.greal + (size_t)f * nt;
  const cpx<R>* __restrict__ ex = A.gcplx + (size_t)f * (nt + 4);
  const int iy = row % ny, iz = row / ny;
  const R ar = ftr * gx[nx + iy] * gx[nx + ny + iz];                       // A_mu = ar gx
  const cpx<R> br = ex[nt + c] * (tf * (ex[nx + iy] * ex[nx + ny + iz]));  // psi_b = br ex
  const int acomp = A.fd[f].acomp;
  const int oc = source_component(acomp, c);
  const cpx<R> rot = source_rotation<R>(acomp, c);
  cpx<R>* zo = A.kout + ((size_t)f * 4 + oc) * N + (size_t)row * nx + x0;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    zo[q * stride] = source_term<R>(v[q], br, ex[x0 + q * stride], ar * gx[x0 + q * stride], rot);
  }
}

// The time factors of A's stage for the block's rows row0 .. row0 + rows - 1 of field f: read from what
// the pass before left (pre), or evaluated here in FP64 (the caller synchronises).
template <typename R>
__device__ __forceinline__ void row_factors(const StageArgs<R>& A, bool pre, int f, int row0, int rows, R* s_ft,
                                            cpx<R>* s_tf) {
  const FieldDesc* F = A.fd + f;
  const int ny = A.g.n[1];
  const double tst = pre ? 0.0 : stage_time(A);
  for (int j = threadIdx.x; j < rows; j += blockDim.x) {
    const int iy = (row0 + j) % ny;
    s_ft[j] = pre ? A.ft[(size_t)f * ny + (F->kind == SWF_FIELD_PULSE_GAUSS ? iy : 0)]
                  : (R)field_time_factor(*F, tst, ny > 1 ? A.g.x0[1] + iy * A.g.dx[1] : 0.0);
  }
  if (threadIdx.x == 0) {
    if (pre) {
      *s_tf = A.tf[f];
    } else {
      double sn, cs;
      sincos(F->tsign * F->e0 * tst, &sn, &cs);
      *s_tf = mk<R>((R)cs, (R)sn);
    }
  }
}

// The block past the tiles of the last y or z pass: field f's time factors of the coming evaluation,
// in FP64, off the path of the x pass that needs them.
template <typename R>
__device__ __forceinline__ void coming_factors(const StageArgs<R>& A, int f) {
  const FieldDesc* F = A.fd + f;
  const int ny = A.g.n[1];
  const double t = node_time(A, A.nls, A.nc);
  const int rows = F->kind == SWF_FIELD_PULSE_GAUSS ? ny : 1;
  for (int iy = threadIdx.x; iy < rows; iy += blockDim.x)
    A.ft[(size_t)f * ny + iy] = (R)field_time_factor(*F, t, ny > 1 ? A.g.x0[1] + iy * A.g.dx[1] : 0.0);
  if (threadIdx.x == blockDim.x - 1) {
    double sn, cs;
    sincos(F->tsign * F->e0 * t, &sn, &cs);
    A.tf[f] = mk<R>((R)cs, (R)sn);
  }
}

template <typename R>
__device__ __forceinline__ cpx<R> shfl_xor(cpx<R> a, int mask) {
  return mk<R>(__shfl_xor_sync(0xffffffffu, a.x, mask), __shfl_xor_sync(0xffffffffu, a.y, mask));
}

// -i H0/N on the NV modes m0 + q mstep of one line along `axis` whose four components sit in the lanes
// lane ^ (1, 2, 3) << lgtx: component c takes s3 kz times component c ^ 2 and (s kx - i s3 ky) times
// component 3 - c, s3 = +s for even and -s for odd components, and +-s itself, s = 1/N.  o: the index
// on the other axis.  Every lane of the warp calls it (lanes without modes: ok = false).
template <typename R, int NV>
__device__ __forceinline__ void h0_modes(const StageArgs<R>& A, int axis, int lgtx, int f, int c, int x, int o, int m0,
                                         int mstep, bool ok, cpx<R>* m) {
  const int nx = A.g.n[0], ny = A.g.n[1], nz = A.g.n[2];
  const FieldDesc* F = A.fd + f;
  const R s = A.inv_n, s3 = (c & 1) ? -s : s, sb = c < 2 ? s : -s;
  const R kx = s * (nx > 1 ? A.kap[x < nx ? x : 0] : (R)F->K[0]);
  const R k_o = axis == 1 ? (nz > 1 ? A.kap[nx + ny + o] : (R)F->K[2]) : (ny > 1 ? A.kap[nx + o] : (R)F->K[1]);
  const R* __restrict__ ka = A.kap + (axis == 1 ? nx : nx + ny);
  const bool flat = axis == 1 && nz == 1 && k_o == (R)0;  // uniform in the block
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const R k_a = ok ? ka[m0 + q * mstep] : (R)0;
    const R ky = s3 * (axis == 1 ? k_a : k_o), kz = s3 * (axis == 1 ? k_o : k_a);
    const cpx<R> b = shfl_xor(m[q], 3 << lgtx);
    cpx<R> h = mk<R>(sb * m[q].x + kx * b.x + ky * b.y, sb * m[q].y + kx * b.y - ky * b.x);
    if (!flat) {
      const cpx<R> d = shfl_xor(m[q], 2 << lgtx);
      h = mk<R>(h.x + kz * d.x, h.y + kz * d.y);
    }
    m[q] = mk<R>(h.y, -h.x);
  }
}

template <typename R, int R1, int R2>
__global__ void __launch_bounds__(kXLineThreads, sizeof(R) == 4 ? 2 : 1)
k_xline(const __grid_constant__ StageArgs<R> P, const __grid_constant__ StageArgs<R> A, int rows, int flags) {
  constexpr int TPL = line_threads(R1, R2);
  constexpr int S = R2 | 1, LS = xline_stride(R1, R2);
  chain_wait();
  chain_release();
  if (A.ctl && A.ctl->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ R s_ft[16];
  __shared__ cpx<R> s_tf;
  const int f = blockIdx.y;
  const int row0 = blockIdx.x * rows;
  const int nx = R1 * R2;
  const size_t N = A.g.N;
  // site side: thread g of line (row j, component c); mode side: the same lines in blocks of R1
  // threads, so that the threads left over when R1 < R2 are whole warps
  const int line = threadIdx.x / TPL, g = threadIdx.x - line * TPL;
  const int c = line & 3, j = line >> 2, row = row0 + j;
  const int mline = threadIdx.x / R1, gm = threadIdx.x - mline * R1;
  const bool site = row < A.nrows && g < R2;
  const bool mode = mline < 4 * rows && row0 + (mline >> 2) < A.nrows;
  const size_t gs = ((size_t)f * 4 + c) * N + (size_t)row * nx + g;  // this thread's first site (stride R2)
  const size_t gt = ((size_t)f * 4 + (mline & 3)) * N + (size_t)(row0 + (mline >> 2)) * nx + gm;  // mode (stride R1)
  cpx<R>* sl = reinterpret_cast<cpx<R>*>(smem_raw) + line * LS;
  cpx<R>* sm = reinterpret_cast<cpx<R>*>(smem_raw) + mline * LS + gm * S;
  const cpx<R>* __restrict__ tw = A.ltw[0];
  const bool last = flags & XL_LAST, first = flags & XL_FIRST;

  cpx<R> m[R2];
  if (last && mode) {
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) m[k2] = P.T[gt + k2 * R1];
  }
  if (first) row_factors(A, flags & XL_FACTORS, f, row0, rows, s_ft, &s_tf);
  // the older terms of the stage combine (their loads overlap those of T)
  const bool ff = sizeof(R) == 4 && A.ylo && A.write_y;
  const int nold = A.nterm - ((flags & XL_REGK) ? 1 : 0);
  cpx<R> v[R1];
  if (first && site) combine_sites<R, R1>(A, nold, ff, gs, R2, v);
  if (last) {
    if (mode) {
      Dft<R, R2>::run(m, true);
#pragma unroll
      for (int i = 0; i < R2; ++i) sm[i] = m[i];
    }
    __syncthreads();
    if (site) {
      cpx<R> r[R1];
      r[0] = sl[g];
#pragma unroll
      for (int k1 = 1; k1 < R1; ++k1) r[k1] = sl[k1 * S + g] * cconj(tw[k1 * R2 + g]);
      Dft<R, R1>::run(r, true);
      close_sites<R, R1>(P, gs, R2, r);
      if (first && (flags & XL_REGK)) {
        const R co = A.ctl ? (R)(A.coef[nold] * A.ctl->h) : A.coef_r[nold];
#pragma unroll
        for (int q = 0; q < R1; ++q) v[q] = v[q] + co * r[q];
      }
    }
  } else {
    __syncthreads();  // the time factors
  }
  if (!first) return;
  if (site) {
    open_sites<R, R1>(A, ff, gs, g, R2, f, c, row, s_ft[j], s_tf, v);
    // forward x-FFT: this thread overwrites the column of the exchange that only it has read
    Dft<R, R1>::run(v, false);
    sl[g] = v[0];
#pragma unroll
    for (int k1 = 1; k1 < R1; ++k1) sl[k1 * S + g] = v[k1] * tw[k1 * R2 + g];
  }
  __syncthreads();
  if (mode) {
#pragma unroll
    for (int i = 0; i < R2; ++i) m[i] = sm[i];
    Dft<R, R2>::run(m, false);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) A.T[gt + k2 * R1] = m[k2];
  }
}

// Lines along axis 1 (y) or 2 (z) of TX = 2^lgtx consecutive x columns (TX <= 8): forward FFT, -i H0/N
// and inverse FFT, as selected.  Thread ((g, c), t): butterfly g of component c of column t, so that
// the four components of a mode sit in one warp and H0 takes its partners by shuffles.  Blocks past
// the tiles (one per field, when A.ft is given) compute the time factors of the coming evaluation in
// FP64, off the path of the x pass that needs them.
template <typename R, int R1, int R2>
__global__ void __launch_bounds__(line_max_threads((int)sizeof(cpx<R>)), sizeof(R) == 4 && R1 <= 16 && R2 <= 16 ? 2 : 1)
k_line(const __grid_constant__ StageArgs<R> A, int axis, int lgtx, int flags) {
  constexpr int LS = line_stride(R1, R2);
  chain_wait();
  chain_release();
  if (A.ctl && A.ctl->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nx = A.g.n[0], ny = A.g.n[1], nz = A.g.n[2];
  const int f = blockIdx.y;
  const int TX = 1 << lgtx;
  const int ntx = (nx + TX - 1) >> lgtx;
  const int other = axis == 1 ? nz : ny;
  if (blockIdx.x >= ntx * other) {
    coming_factors(A, f);
    return;
  }
  const int xt = blockIdx.x % ntx, o = blockIdx.x / ntx;  // o: z index (axis 1) or y index (axis 2)
  const int t = threadIdx.x & (TX - 1), c = (threadIdx.x >> lgtx) & 3, g = threadIdx.x >> (lgtx + 2);
  const int x = xt * TX + t;
  const bool site = x < nx && g < R2, mode = x < nx && g < R1;
  const size_t base = (axis == 1 ? (size_t)o * nx * ny : (size_t)o * nx) + ((size_t)f * 4 + c) * A.g.N + x;
  const size_t stride = axis == 1 ? (size_t)nx : (size_t)nx * ny;
  cpx<R>* sl = reinterpret_cast<cpx<R>*>(smem_raw) + (c * TX + t) * LS;
  const cpx<R>* __restrict__ tw = A.ltw[axis];
  cpx<R> m[R2];
  if (flags & LN_FWD) {
    if (site) {
      cpx<R> v[R1];
#pragma unroll
      for (int q = 0; q < R1; ++q) v[q] = A.T[base + (size_t)(g + q * R2) * stride];
      Dft<R, R1>::run(v, false);
      sl[g] = v[0];
#pragma unroll
      for (int k1 = 1; k1 < R1; ++k1) sl[k1 * R2 + g] = v[k1] * tw[k1 * R2 + g];
    }
    __syncthreads();
    if (mode) {
#pragma unroll
      for (int i = 0; i < R2; ++i) m[i] = sl[g * R2 + i];
      Dft<R, R2>::run(m, false);
    }
  } else if (mode) {
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) m[k2] = A.T[base + (size_t)(g + k2 * R1) * stride];
  }
  if (!mode) {
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) m[k2] = mk<R>(0, 0);
  }
  if ((flags & LN_H0) && A.yspec && mode) {
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) A.yspec[base + (size_t)(g + k2 * R1) * stride] = m[k2];
  }
  if (flags & LN_H0) h0_modes<R, R2>(A, axis, lgtx, f, c, x, o, g, R1, mode, m);
  if (flags & LN_INV) {
    if (mode) {
      Dft<R, R2>::run(m, true);
#pragma unroll
      for (int i = 0; i < R2; ++i) sl[g * R2 + i] = m[i];
    }
    __syncthreads();
    if (site) {
      cpx<R> v[R1];
      v[0] = sl[g];
#pragma unroll
      for (int k1 = 1; k1 < R1; ++k1) v[k1] = sl[k1 * R2 + g] * cconj(tw[k1 * R2 + g]);
      Dft<R, R1>::run(v, true);
#pragma unroll
      for (int q = 0; q < R1; ++q) A.T[base + (size_t)(g + q * R2) * stride] = v[q];
    }
  } else if (mode) {
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) A.T[base + (size_t)(g + k2 * R1) * stride] = m[k2];
  }
}

// s + e += b + be, e the rounding errors of s (Knuth's two-sum); double: s alone.
__device__ __forceinline__ void add_exact(float& s, float& e, float b, float be) {
  const float t = __fadd_rn(s, b), bp = __fsub_rn(t, s);
  e = __fadd_rn(e, __fadd_rn(be, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(b, bp))));
  s = t;
}
__device__ __forceinline__ void add_exact(double& s, double&, double b, double) { s += b; }

// The direct-transform sums of a block of wave f: red[component][row][thread] holds the threads' sums (in
// the march precision; the caller has synchronised), eight lanes of the first warp per component (one in
// a block of less than a warp) add them in a fixed order, and trow[w] (the stage's weight and time phase)
// times adds them to the block's own FP64 accumulators dpart[f][block][4].  Single-precision sums carry
// their rounding errors, which makes the block's as good as one in FP64: additions in FP64 itself hold an
// SM quarter for 64 cycles each (16 pairs on 384^2, 21 launches of k_f2_line: 4.0 ms with them and a warp
// per component, 3.25 ms so; 3.4 ms with rounded sums by a warp per component).
template <typename R>
__device__ __forceinline__ void direct_sums(const StageArgs<R>& A, const cpx<R>* red, int per, int f,
                                            const cpx<double>* __restrict__ ptab, int tab_stride, int stage,
                                            cpx<double>* dpart) {
  const int g = blockDim.x >= 32 ? 8 : 1;
  if (threadIdx.x >= 4 * g) return;
  const int k = threadIdx.x / g, l = threadIdx.x - k * g;
  cpx<R> s = mk<R>(0, 0), err = mk<R>(0, 0);
  for (int e = l; e < per; e += g) {
    const cpx<R> v = red[k * per + e];
    add_exact(s.x, err.x, v.x, 0);
    add_exact(s.y, err.y, v.y, 0);
  }
  if (g > 1) {
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
      const cpx<R> v = shfl_xor(s, off), ve = shfl_xor(err, off);
      add_exact(s.x, err.x, v.x, ve.x);
      add_exact(s.y, err.y, v.y, ve.y);
    }
  }
  if (l == 0) {
    const long tab_row = (long)(A.clk->step + A.ls) * 7 + stage;
    const cpx<double> wt = ptab[3 * (tab_row + (long)(f >> 1) * tab_stride) + (f & 1)];
    cpx<double>& d = dpart[((size_t)f * gridDim.x + blockIdx.x) * 4 + k];
    d = d + wt * mk<double>((double)s.x + (double)err.x, (double)s.y + (double)err.y);
  }
}

// The x pass of the partial-integration integrand (see k_f2_x in swf_march.cu) on the register lines: Z =
// -i V (Y + psi_b) of the stage value in ys, its forward x-FFT into Zspec and its direct transform.  Its
// traffic is one read and one write of the waves; with the new mode sum it took four steps of 16 pairs on
// 384^2 from 29.5 to 21.2 ms (33.7 ms with small-radix passes here).
template <typename R, int R1, int R2>
__global__ void __launch_bounds__(kXLineThreads, 2)
k_f2_line(const __grid_constant__ StageArgs<R> A, const cpx<R>* __restrict__ ys, cpx<R>* __restrict__ Zspec,
          const cpx<R>* __restrict__ dph, const cpx<double>* __restrict__ ptab, int tab_stride, int stage,
          cpx<double>* dpart, int rows) {
  constexpr int TPL = line_threads(R1, R2);
  constexpr int S = R2 | 1, LS = xline_stride(R1, R2);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ R s_ft[16];
  __shared__ cpx<R> s_tf;
  cpx<R>* sm = reinterpret_cast<cpx<R>*>(smem_raw);
  const int nx = R1 * R2, ny = A.g.n[1], nz = A.g.n[2], nt = nx + ny + nz;
  const size_t N = A.g.N;
  const int f = blockIdx.y, row0 = blockIdx.x * rows;
  const int line = threadIdx.x / TPL, g = threadIdx.x - line * TPL;
  const int c = line & 3, j = line >> 2, row = row0 + j;
  const int mline = threadIdx.x / R1, gm = threadIdx.x - mline * R1;
  const bool ok = row < A.nrows, site = ok && g < R2;
  const bool mode = mline < 4 * rows && row0 + (mline >> 2) < A.nrows;
  const cpx<R>* __restrict__ tw = A.ltw[0];
  const int acomp = A.fd[f].acomp, oc = source_component(acomp, c);
  const size_t gs = ((size_t)f * 4 + c) * N + (size_t)row * nx + g;
  cpx<R> v[R1];
  if (site) {
#pragma unroll
    for (int q = 0; q < R1; ++q) v[q] = ys[gs + q * R2];
  }
  row_factors(A, false, f, row0, rows, s_ft, &s_tf);
  __syncthreads();
  cpx<R> dsum = mk<R>(0, 0);
  if (site) {
    const R* __restrict__ gx = A.greal + (size_t)f * nt;
    const cpx<R>* __restrict__ ex = A.gcplx + (size_t)f * (nt + 4);
    const cpx<R>* __restrict__ dx = dph + (size_t)f * nt;
    const int iy = row % ny, iz = row / ny;
    const R ar = s_ft[j] * gx[nx + iy] * gx[nx + ny + iz];
    const cpx<R> br = ex[nt + c] * (s_tf * (ex[nx + iy] * ex[nx + ny + iz]));
    const cpx<R> rot = source_rotation<R>(acomp, c);
#pragma unroll
    for (int q = 0; q < R1; ++q) {
      const int x = g + q * R2;
      v[q] = source_term<R>(v[q], br, ex[x], ar * gx[x], rot);
      const cpx<R> e = dx[x];
      dsum = mk<R>(dsum.x + v[q].x * e.x - v[q].y * e.y, dsum.y + v[q].x * e.y + v[q].y * e.x);
    }
    dsum = dsum * (dx[nx + iy] * dx[nx + ny + iz]);
    Dft<R, R1>::run(v, false);
    cpx<R>* sl = sm + (4 * j + oc) * LS + g;
    sl[0] = v[0];
#pragma unroll
    for (int k1 = 1; k1 < R1; ++k1) sl[k1 * S] = v[k1] * tw[k1 * R2 + g];
  }
  __syncthreads();
  if (mode) {
    const size_t gt = ((size_t)f * 4 + (mline & 3)) * N + (size_t)(row0 + (mline >> 2)) * nx + gm;
    const cpx<R>* sl = sm + mline * LS + gm * S;
    cpx<R> m[R2];
#pragma unroll
    for (int i = 0; i < R2; ++i) m[i] = sl[i];
    Dft<R, R2>::run(m, false);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) Zspec[gt + k2 * R1] = m[k2];
  }
  __syncthreads();
  sm[(oc * rows + j) * TPL + g] = dsum;
  __syncthreads();
  direct_sums(A, sm, rows * TPL, f, ptab, tab_stride, stage, dpart);
}
#endif

}  // namespace swf
