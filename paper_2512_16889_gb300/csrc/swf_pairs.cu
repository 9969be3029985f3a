// Full pair numbers N(m, n) of Eq. 8 for every electron m of one list and positron n of another,
// all in one field, grid and time window (Sec. II, Eqs. 8-9; Sec. II.A: scans over momenta).
//
// Instead of one U and one V march per pair, every electron is marched once (U waves) and every
// positron once (V waves), and the four overlaps of Eq. 8 are formed in FP64:
//   C(m, n) = e^{i q0 t} sum_c conj(U~_m(-q_n))_c v_n,c       (a plane wave: a direct transform)
//   A(m, n) = e^{i p0 t} sum_c conj(u_m,c) V~_n(p_m)_c
//   B(m, n) = L^-d sum_j (P_+(k_j) U~_m(j))^+ V~_n(j)         (grid modes, P_+- energy projectors)
//   D(m, n) = L^-d sum_j (P_-(k_j) U~_m(j))^+ V~_n(j)
// with U~, V~ the continuum-normalised transforms at t = t_in.  The sums over s' and the grid modes Q
// of Eq. 8 are the projectors (sum_s' u u^+ = P_+, sum_s' v v^+ = P_-), as in the single-pair path.
// N = |C + D|^2 = |A + B|^2.
//
// A plane wave is a product of one factor per axis, so the direct transforms of one wave at all n
// momenta of the other list need one pass over the grid per distinct momentum along some of the axes
// (a scan along one axis: one) and a small product after it, instead of 4 N products per pair.  In an
// orthonormal eigenbasis of every mode's H0 the projectors are a choice of two of the four
// amplitudes, so B and D are matrix products over 2 N amplitudes each.  Together 4 N FP64 products per
// pair instead of 16 N.
#include <algorithm>
#include <array>
#include <cmath>
#include <map>
#include <string>
#include <vector>

#include "swf_internal.h"

namespace swf {
namespace pairs {

constexpr int TK = 16;      // k step of the product kernel
constexpr int kTile = 32;   // output tile of a block: at most 32 x 32, one output per thread
constexpr int DB = 4;       // momenta per block of the first contraction

// Phase tables exp(-i sum_a kappa_a x_a) over the sites of the axes in `axes` (bit a: axis a; trivial
// axes carry no phase): tab[d][site], d < n.
__global__ void k_phases(const double* __restrict__ kappa, int n, GridDesc g, int axes, int len, cpx<double>* tab) {
  const int d = blockIdx.y;
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < len; r += gridDim.x * blockDim.x) {
    int rest = r;
    double ph = 0.0;
    for (int a = 0; a < 3; ++a) {
      if (!(axes >> a & 1)) continue;
      const int j = rest % g.n[a];
      rest /= g.n[a];
      if (g.n[a] > 1) ph -= kappa[3 * d + a] * (g.x0[a] + j * g.dx[a]);
    }
    double sn, cs;
    sincos(ph, &sn, &cs);
    tab[(size_t)d * len + r] = mk<double>(cs, sn);
  }
}

// First contraction over rows (y, z): G[line][d][x] = sum_r psi[line][r][x] tab[d][r], line = (field,
// component), DB values of d per block.  32 x columns by 8 row groups per block, the groups added in
// order.
template <typename R>
__global__ void __launch_bounds__(256) k_contract_rows(const cpx<R>* __restrict__ psi, const cpx<double>* __restrict__ tab,
                                                       int nrows, int nx, int D, cpx<double>* G) {
  __shared__ cpx<double> red[8][DB][32];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const int x = blockIdx.x * 32 + lane, d0 = blockIdx.z * DB;
  const size_t line = blockIdx.y;
  cpx<double> acc[DB];
#pragma unroll
  for (int k = 0; k < DB; ++k) acc[k] = mk<double>(0, 0);
  if (x < nx) {
    const cpx<R>* p = psi + line * (size_t)nrows * nx + x;
    for (int r = grp; r < nrows; r += 8) {
      const cpx<double> v = cvt<double>(p[(size_t)r * nx]);
#pragma unroll
      for (int k = 0; k < DB; ++k)
        if (d0 + k < D) {
          const cpx<double> w = tab[(size_t)(d0 + k) * nrows + r];
          acc[k] = mk<double>(acc[k].x + v.x * w.x - v.y * w.y, acc[k].y + v.x * w.y + v.y * w.x);
        }
    }
  }
#pragma unroll
  for (int k = 0; k < DB; ++k) red[grp][k][lane] = acc[k];
  __syncthreads();
  if (grp < DB && x < nx && d0 + grp < D) {
    cpx<double> s = red[0][grp][lane];
    for (int q = 1; q < 8; ++q) s = s + red[q][grp][lane];
    G[(line * D + d0 + grp) * nx + x] = s;
  }
}

// First contraction over x: G[line][d][r] = sum_x psi[line][r][x] tab[d][x]; a warp per row.
template <typename R>
__global__ void __launch_bounds__(256) k_contract_x(const cpx<R>* __restrict__ psi, const cpx<double>* __restrict__ tab,
                                                    int nrows, int nx, int D, cpx<double>* G) {
  const int lane = threadIdx.x & 31, r = blockIdx.x * 8 + (threadIdx.x >> 5), d0 = blockIdx.z * DB;
  if (r >= nrows) return;
  const size_t line = blockIdx.y;
  const cpx<R>* p = psi + (line * nrows + r) * (size_t)nx;
  cpx<double> acc[DB];
#pragma unroll
  for (int k = 0; k < DB; ++k) acc[k] = mk<double>(0, 0);
  for (int x = lane; x < nx; x += 32) {
    const cpx<double> v = cvt<double>(p[x]);
#pragma unroll
    for (int k = 0; k < DB; ++k)
      if (d0 + k < D) {
        const cpx<double> w = tab[(size_t)(d0 + k) * nx + x];
        acc[k] = mk<double>(acc[k].x + v.x * w.x - v.y * w.y, acc[k].y + v.x * w.y + v.y * w.x);
      }
  }
#pragma unroll
  for (int k = 0; k < DB; ++k) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      acc[k].x += __shfl_down_sync(0xffffffffu, acc[k].x, off);
      acc[k].y += __shfl_down_sync(0xffffffffu, acc[k].y, off);
    }
    if (lane == 0 && d0 + k < D) G[(line * D + d0 + k) * nrows + r] = acc[k];
  }
}

// Last contraction: out[line / 4][k][line % 4] = scale sum_i G[line][map[k]][i] tab[k][i]; a warp per
// (line, k).
__global__ void __launch_bounds__(256) k_contract_last(const cpx<double>* __restrict__ G,
                                                       const cpx<double>* __restrict__ tab, const int* __restrict__ map,
                                                       int len, int D, int n_k, double scale, cpx<double>* out) {
  const int lane = threadIdx.x & 31, k = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (k >= n_k) return;
  const size_t line = blockIdx.y;
  const cpx<double>* p = G + (line * D + map[k]) * len;
  const cpx<double>* w = tab + (size_t)k * len;
  cpx<double> s = mk<double>(0, 0);
  for (int i = lane; i < len; i += 32) s = s + p[i] * w[i];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    s.x += __shfl_down_sync(0xffffffffu, s.x, off);
    s.y += __shfl_down_sync(0xffffffffu, s.y, off);
  }
  if (lane == 0) out[((line >> 2) * n_k + k) * 4 + (line & 3)] = scale * s;
}

// Every mode's four components (in place) to its amplitudes in an orthonormal eigenbasis of H0(kappa)
// (Dirac representation, w = kappa/(E + 1), c^2 = (E + 1)/(2E)): c (1, 0, wz, wx + i wy), c (0, 1, wx -
// i wy, -wz) of energy +E, c (-wz, -wx - i wy, 1, 0), c (-wx + i wy, wz, 0, 1) of energy -E.
__global__ void __launch_bounds__(256) k_energy_amps(cpx<double>* spec, GridDesc g, const double* __restrict__ Ku, int n_f,
                                                     int fc) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= g.N) return;
  const int row = j / g.n[0];
  const int id[3] = {j - row * g.n[0], row % g.n[1], row / g.n[1]};
  double k[3];
  for (int a = 0; a < 3; ++a) k[a] = g.n[a] > 1 ? mode_kappa(id[a], g.n[a], g.L[a]) : Ku[a];
  const double E = sqrt(1.0 + k[0] * k[0] + k[1] * k[1] + k[2] * k[2]);
  const double c = sqrt((E + 1.0) / (2.0 * E)), ie = c / (E + 1.0);
  const double wx = k[0] * ie, wy = k[1] * ie, wz = k[2] * ie;  // times c
  const int f1 = min(n_f, (int)(blockIdx.y + 1) * fc);
  for (int f = blockIdx.y * fc; f < f1; ++f) {
    cpx<double>* u = spec + (size_t)f * 4 * g.N + j;
    const size_t N = g.N;
    const cpx<double> a = u[0], b = u[N], p = u[2 * N], q = u[3 * N];
    // (wx - i wy) z = (wx z.x + wy z.y, wx z.y - wy z.x); (wx + i wy) z = (wx z.x - wy z.y, wx z.y + wy z.x)
    u[0] = mk<double>(c * a.x + wz * p.x + wx * q.x + wy * q.y, c * a.y + wz * p.y + wx * q.y - wy * q.x);
    u[N] = mk<double>(c * b.x + wx * p.x - wy * p.y - wz * q.x, c * b.y + wx * p.y + wy * p.x - wz * q.y);
    u[2 * N] = mk<double>(c * p.x - wz * a.x - wx * b.x - wy * b.y, c * p.y - wz * a.y - wx * b.y + wy * b.x);
    u[3 * N] = mk<double>(c * q.x - wx * a.x + wy * a.y + wz * b.x, c * q.y - wx * a.y - wy * a.x + wz * b.y);
  }
}

// part[sign][s][m][n] = sum over k in split s of conj(X[m][sign K + k]) Y[n][sign K + k], rows of `ld`
// values.  One output per thread: FP64 issues an instruction in 64 cycles per SM quarter, so the two
// shared-memory reads of a product are hidden without a register tile, and tiles of exactly TM x TN
// outputs (100 x 100 pairs: 16 tiles of 25 x 25, 625 of 640 threads) leave few lanes idle.  The next
// k step's operands are on their way while the present one is used.  100 x 100 pairs on 256 x 128: 9.3
// ms (107 ms with 2 x 2 outputs a thread, 32 x 32 tiles and four times the products; 8.3 ms at the FP64
// unit's full rate).
__global__ void __launch_bounds__(kTile* kTile, 1)
k_pair_products(const cpx<double>* __restrict__ X, const cpx<double>* __restrict__ Y, int M, int Nn, long K, long ld,
                long kchunk, int S, int TM, int TN, cpx<double>* part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lx = TM | 1, ly = TN | 1;
  cpx<double>* xs = reinterpret_cast<cpx<double>*>(smem_raw);  // [2][TK][lx], then [2][TK][ly]
  cpx<double>* ys = xs + 2 * TK * lx;
  const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
  const int sign = blockIdx.z / S, sp = blockIdx.z - sign * S;
  const long k0 = sp * kchunk, k1 = min(K, k0 + kchunk), off = sign * K;
  const int m = threadIdx.x / TN, n = threadIdx.x - m * TN;
  const bool live = m < TM;
  const int total = (TM + TN) * TK;
  // element e of a step: row e / TK of X's TM rows, then Y's TN rows; column e % TK
  auto fetch = [&](long kb, int e) {
    const int r = e / TK;
    const long k = kb + e % TK;
    if (k >= k1) return mk<double>(0, 0);
    if (r < TM) return m0 + r < M ? X[(size_t)(m0 + r) * ld + off + k] : mk<double>(0, 0);
    return n0 + r - TM < Nn ? Y[(size_t)(n0 + r - TM) * ld + off + k] : mk<double>(0, 0);
  };
  auto store = [&](int buf, int e, cpx<double> v) {
    const int r = e / TK, c = e % TK;
    if (r < TM) xs[(buf * TK + c) * lx + r] = v;
    else ys[(buf * TK + c) * ly + r - TM] = v;
  };
  for (int e = threadIdx.x; e < total; e += blockDim.x) store(0, e, fetch(k0, e));
  __syncthreads();
  cpx<double> acc = mk<double>(0, 0);
  int buf = 0;
  for (long kb = k0; kb < k1; kb += TK, buf ^= 1) {
    const bool more = kb + TK < k1;
    const int e0 = threadIdx.x;
    cpx<double> nxt = mk<double>(0, 0);
    if (more && e0 < total) nxt = fetch(kb + TK, e0);
    if (live) {
      const cpx<double>* xp = xs + buf * TK * lx + m;
      const cpx<double>* yp = ys + buf * TK * ly + n;
#pragma unroll
      for (int c = 0; c < TK; ++c) {
        const cpx<double> x = xp[c * lx], y = yp[c * ly];
        acc.x = fma(x.y, y.y, fma(x.x, y.x, acc.x));
        acc.y = fma(-x.y, y.x, fma(x.x, y.y, acc.y));
      }
    }
    if (more) {
      if (e0 < total) store(buf ^ 1, e0, nxt);
      for (int e = e0 + blockDim.x; e < total; e += blockDim.x) store(buf ^ 1, e, fetch(kb + TK, e));
    }
    __syncthreads();
  }
  if (live && m0 + m < M && n0 + n < Nn) part[((size_t)blockIdx.z * M + m0 + m) * Nn + n0 + n] = acc;
}

// results[m][n]: C and A from the direct transforms (TU[m][n][4] = U~_m(-q_n), TV[n][m][4] = V~_n(p_m))
// and the backgrounds' spinors with their time phases, B and D from the products' parts (splits in
// order, times sBD).
__global__ void k_pair_results(const cpx<double>* __restrict__ TU, const cpx<double>* __restrict__ TV,
                               const cpx<double>* __restrict__ wU, const cpx<double>* __restrict__ wV,
                               const cpx<double>* __restrict__ part, int S, double sBD, const double* normU,
                               const double* normV, int n_e, int n_p, swf_result* res) {
  const long MN = (long)n_e * n_p;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < MN; i += (long)gridDim.x * blockDim.x) {
    const long m = i / n_p, n = i % n_p;
    cpx<double> C = mk<double>(0, 0), A = mk<double>(0, 0), B = mk<double>(0, 0), D = mk<double>(0, 0);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      C = C + cdot(TU[4 * i + c], wV[4 * n + c]);
      A = A + cdot(wU[4 * m + c], TV[4 * (n * n_e + m) + c]);
    }
    for (int s = 0; s < S; ++s) {
      B = B + part[s * MN + i];
      D = D + part[(S + s) * MN + i];
    }
    B = sBD * B;
    D = sBD * D;
    swf_result o;
    o.amp[0] = C.x; o.amp[1] = C.y;
    o.amp[2] = D.x; o.amp[3] = D.y;
    o.amp[4] = A.x; o.amp[5] = A.y;
    o.amp[6] = B.x; o.amp[7] = B.y;
    const cpx<double> CD = C + D, AB = A + B;
    o.prob[0] = CD.x * CD.x + CD.y * CD.y;
    o.prob[1] = AB.x * AB.x + AB.y * AB.y;
    o.diag[0] = normU[m];
    o.diag[1] = normV[n];
    res[i] = o;
  }
}

int sms() {
  int dev = 0, n = 152;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    n = 152;
  return n;
}

// out[f][k][4] = dx^d sum_x psi_f(x) exp(-i kappa_k.x) for every field f and wave vector k.  One of two
// orders: rows (y, z) first and then x, or x first and then the rows; the first contraction runs once
// per distinct momentum of its axes, over the whole grid, so the order with fewer of those is taken
// (the second is smaller by the length it leaves).  Fields go in chunks that keep the intermediate
// below 256 MB, one at a time where a single field's is larger (3D with many momenta along x: 419 MB for
// 100 of them on 256^3, a fraction 1/n_x of a hundred waves).
swf_status transform_many(swf_ctx* ctx, const GridDesc& g, int n_f, swf_precision prec, const void* psi,
                          const std::vector<double>& kappa, const std::string& tag, cpx<double>* out, cudaStream_t st) {
  const int n_k = (int)(kappa.size() / 3);
  const int nx = g.n[0], nrows = g.n[1] * g.n[2];
  // distinct momenta along the axes of `mask`, and every wave vector's index among them
  auto distinct = [&](int mask, std::vector<double>& vals, std::vector<int>& map) {
    std::map<std::array<double, 3>, int> seen;
    map.resize(n_k);
    for (int k = 0; k < n_k; ++k) {
      std::array<double, 3> key = {0, 0, 0};
      for (int a = 0; a < 3; ++a)
        if ((mask >> a & 1) && g.n[a] > 1) key[a] = kappa[3 * k + a];
      auto it = seen.find(key);
      if (it == seen.end()) {
        it = seen.emplace(key, (int)seen.size()).first;
        vals.insert(vals.end(), key.begin(), key.end());
      }
      map[k] = it->second;
    }
    return (int)seen.size();
  };
  std::vector<double> vx, vr;
  std::vector<int> mx, mr;
  const int Dx = distinct(1, vx, mx), Dr = distinct(6, vr, mr);
  const double cost_rows = 4.0 * g.N * Dr + 4.0 * nx * n_k, cost_x = 4.0 * g.N * Dx + 4.0 * nrows * n_k;
  const bool rows_first = cost_rows <= cost_x;
  const int D = rows_first ? Dr : Dx, len1 = rows_first ? nrows : nx, len2 = rows_first ? nx : nrows;
  const std::vector<double>& v1 = rows_first ? vr : vx;
  const std::vector<int>& m1 = rows_first ? mr : mx;
  const size_t per = (size_t)4 * D * len2 * 16;
  const int fc = (int)std::max<size_t>(1, std::min<size_t>(n_f, ((size_t)256 << 20) / per));
  void *pk, *pv, *pm, *t1, *t2, *G;
  swf_status s;
  if ((s = ws_get(ctx, tag + ".kappa", sizeof(double) * kappa.size(), &pk)) != SWF_OK) return s;
  if ((s = ws_get(ctx, tag + ".distinct", sizeof(double) * v1.size(), &pv)) != SWF_OK) return s;
  if ((s = ws_get(ctx, tag + ".map", sizeof(int) * n_k, &pm)) != SWF_OK) return s;
  if ((s = ws_get(ctx, tag + ".phase1", (size_t)D * len1 * 16, &t1)) != SWF_OK) return s;
  if ((s = ws_get(ctx, tag + ".phase2", (size_t)n_k * len2 * 16, &t2)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "pairs.G", per * fc, &G)) != SWF_OK) return s;
  cudaError_t e = cudaMemcpyAsync(pk, kappa.data(), sizeof(double) * kappa.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(pv, v1.data(), sizeof(double) * v1.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(pm, m1.data(), sizeof(int) * n_k, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_status(e, "upload pair momenta");
  const int ax1 = rows_first ? 6 : 1, ax2 = 7 - ax1;
  {
    ProfScope ps(ctx, "k_phases", st);
    k_phases<<<dim3((len1 + 127) / 128, D), 128, 0, st>>>((const double*)pv, D, g, ax1, len1, (cpx<double>*)t1);
    k_phases<<<dim3((len2 + 127) / 128, n_k), 128, 0, st>>>((const double*)pk, n_k, g, ax2, len2, (cpx<double>*)t2);
  }
  const double cell = g.dx[0] * g.dx[1] * g.dx[2];
  const size_t elem = prec == SWF_C64 ? 8 : 16;
  for (int f0 = 0; f0 < n_f; f0 += fc) {
    const int nf = std::min(fc, n_f - f0);
    const void* src = (const unsigned char*)psi + (size_t)f0 * 4 * g.N * elem;
    {
      ProfScope ps(ctx, "k_contract", st);
      const dim3 grid(rows_first ? (nx + 31) / 32 : (nrows + 7) / 8, 4 * nf, (D + DB - 1) / DB);
      const cpx<double>* tab = (const cpx<double>*)t1;
      if (rows_first && prec == SWF_C64)
        k_contract_rows<float><<<grid, 256, 0, st>>>((const cpx<float>*)src, tab, nrows, nx, D, (cpx<double>*)G);
      else if (rows_first)
        k_contract_rows<double><<<grid, 256, 0, st>>>((const cpx<double>*)src, tab, nrows, nx, D, (cpx<double>*)G);
      else if (prec == SWF_C64)
        k_contract_x<float><<<grid, 256, 0, st>>>((const cpx<float>*)src, tab, nrows, nx, D, (cpx<double>*)G);
      else
        k_contract_x<double><<<grid, 256, 0, st>>>((const cpx<double>*)src, tab, nrows, nx, D, (cpx<double>*)G);
    }
    ProfScope ps(ctx, "k_contract_last", st);
    k_contract_last<<<dim3((n_k + 7) / 8, 4 * nf), 256, 0, st>>>((const cpx<double>*)G, (const cpx<double>*)t2,
                                                                 (const int*)pm, len2, D, n_k, cell,
                                                                 out + (size_t)f0 * n_k * 4);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "pair transforms");
  // the tables above are the sources of asynchronous uploads
  e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? SWF_OK : cuda_status(e, "pair transforms");
}

bool same_grid(const swf_grid& a, const swf_grid& b) {
  for (int k = 0; k < 3; ++k) {
    if (a.n[k] != b.n[k]) return false;
    if (a.n[k] > 1 && a.L[k] != b.L[k]) return false;
  }
  return a.t_in == b.t_in && a.t_out == b.t_out && a.n_steps == b.n_steps;
}

bool same_field(const swf_field& a, const swf_field& b) {
  if (a.kind != b.kind) return false;
  for (int k = 0; k < 8; ++k)
    if (a.prm[k] != b.prm[k]) return false;
  return true;
}

}  // namespace pairs
}  // namespace swf

using namespace swf;

extern "C" swf_status swf_pair_matrix(swf_ctx* ctx, int n_e, const swf_instance* electrons, int n_p,
                                      const swf_instance* positrons, swf_precision prec, swf_result* results) {
  if (!ctx) { set_error("ctx is NULL"); return SWF_EINVAL; }
  if (n_e < 1 || n_p < 1 || !electrons || !positrons || !results) {
    set_error("swf_pair_matrix: need n_e >= 1, n_p >= 1 and non-NULL arrays");
    return SWF_EINVAL;
  }
  swf_status s = validate_instances(n_e, electrons, prec);
  if (s != SWF_OK) return s;
  if ((s = validate_instances(n_p, positrons, prec)) != SWF_OK) return s;
  const swf_instance& i0 = electrons[0];
  for (int k = 0; k < n_e + n_p; ++k) {
    const swf_instance& in = k < n_e ? electrons[k] : positrons[k - n_e];
    if (!pairs::same_grid(in.grid, i0.grid) || !pairs::same_field(in.field, i0.field) ||
        ((in.flags ^ i0.flags) & SWF_ADAPTIVE)) {
      set_error("swf_pair_matrix: every electron and positron must share the field, grid, time window and step control");
      return SWF_EINVAL;
    }
    for (int a = 0; a < 3; ++a) {
      if (i0.grid.n[a] != 1) continue;
      const bool ok = k < n_e ? in.p[a] == i0.p[a] : in.q[a] == -i0.p[a];
      if (!ok) {
        set_error("swf_pair_matrix: along a trivial axis every p must be equal and every q = -p");
        return SWF_EINVAL;
      }
    }
  }
  cudaSetDevice(ctx->device);
  cudaStream_t st = ctx->stream;
  const GridDesc g = make_grid(i0.grid);
  const long K = 4L * g.N;
  const size_t elem = prec == SWF_C64 ? 8 : 16;
  const double t_in = i0.grid.t_in;
  // spinors with their background's time phase at t_in (e^{i p0 t} of conj(U_back), e^{i q0 t} of V_back),
  // and the wave vectors of the direct transforms
  std::vector<FieldDesc> fdU(n_e), fdV(n_p);
  std::vector<double> wU(8 * (size_t)n_e), wV(8 * (size_t)n_p), kU(3 * (size_t)n_p), kV(3 * (size_t)n_e);
  auto wave = [&](const double* mom, int spin, bool positron, double* w) {
    double sp[8];
    spinor_uv(mom, spin, positron, sp);
    const double ph = (positron ? 1.0 : -1.0) * energy3(mom) * t_in, cs = std::cos(ph), sn = std::sin(ph);
    for (int c = 0; c < 4; ++c) {
      w[2 * c] = cs * sp[2 * c] - sn * sp[2 * c + 1];
      w[2 * c + 1] = cs * sp[2 * c + 1] + sn * sp[2 * c];
    }
  };
  for (int m = 0; m < n_e; ++m) {
    fdU[m] = make_field_desc(electrons[m], 0);
    wave(electrons[m].p, electrons[m].s, false, &wU[8 * (size_t)m]);
    for (int a = 0; a < 3; ++a) kV[3 * (size_t)m + a] = electrons[m].p[a];
  }
  for (int n = 0; n < n_p; ++n) {
    fdV[n] = make_field_desc(positrons[n], 1);
    wave(positrons[n].q, positrons[n].r, true, &wV[8 * (size_t)n]);
    for (int a = 0; a < 3; ++a) kU[3 * (size_t)n + a] = -positrons[n].q[a];
  }
  void *psiU, *psiV, *specU, *specV, *TU, *TV, *pwU, *pwV, *normU, *normV, *pku, *pres;
  if ((s = ws_get(ctx, "pairs.psiU", (size_t)n_e * K * elem, &psiU)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "pairs.psiV", (size_t)n_p * K * elem, &psiV)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "pairs.specU", (size_t)n_e * K * 16, &specU)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "pairs.specV", (size_t)n_p * K * 16, &specV)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "pairs.TU", (size_t)n_e * n_p * 64, &TU)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "pairs.TV", (size_t)n_e * n_p * 64, &TV)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "pairs.wU", (size_t)n_e * 64, &pwU)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "pairs.wV", (size_t)n_p * 64, &pwV)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "pairs.normU", (size_t)n_e * 8, &normU)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "pairs.normV", (size_t)n_p * 8, &normV)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "pairs.Ku", 3 * sizeof(double), &pku)) != SWF_OK) return s;
  if ((s = ws_get(ctx, "pairs.results", sizeof(swf_result) * (size_t)n_e * n_p, &pres)) != SWF_OK) return s;
  // one march per electron (U waves) and per positron (V waves), then their FP64 transforms
  const int adaptive = (i0.flags & SWF_ADAPTIVE) ? 1 : 0;
  if ((s = march_fields(ctx, g, t_in, i0.grid.t_out, i0.grid.n_steps, n_e, fdU.data(), prec, psiU, st, adaptive)) != SWF_OK)
    return s;
  if ((s = march_fields(ctx, g, t_in, i0.grid.t_out, i0.grid.n_steps, n_p, fdV.data(), prec, psiV, st, adaptive)) != SWF_OK)
    return s;
  if ((s = transform_fields(ctx, g, n_e, prec, psiU, (double2*)specU, st, true)) != SWF_OK) return s;
  if ((s = transform_fields(ctx, g, n_p, prec, psiV, (double2*)specV, st, true)) != SWF_OK) return s;
  if ((s = field_norms(ctx, g, n_e, prec, psiU, (double*)normU, st)) != SWF_OK) return s;
  if ((s = field_norms(ctx, g, n_p, prec, psiV, (double*)normV, st)) != SWF_OK) return s;
  if ((s = pairs::transform_many(ctx, g, n_e, prec, psiU, kU, "pairs.U", (cpx<double>*)TU, st)) != SWF_OK) return s;
  if ((s = pairs::transform_many(ctx, g, n_p, prec, psiV, kV, "pairs.V", (cpx<double>*)TV, st)) != SWF_OK) return s;
  cudaError_t e = cudaMemcpyAsync(pwU, wU.data(), (size_t)n_e * 64, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(pwV, wV.data(), (size_t)n_p * 64, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(pku, fdU[0].K, 3 * sizeof(double), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_status(e, "upload pair tables");
  {
    ProfScope ps(ctx, "k_energy_amps", st);
    const int nb = (g.N + 255) / 256;
    const int fc = std::max(1, 8 * nb / (4 * pairs::sms()));  // fields per thread: enough blocks to fill the SMs
    for (int k = 0; k < 2; ++k) {
      const int n = k ? n_p : n_e;
      const int f = std::min(n, std::max(fc, (n + 65534) / 65535));
      pairs::k_energy_amps<<<dim3(nb, (n + f - 1) / f), 256, 0, st>>>((cpx<double>*)(k ? specV : specU), g,
                                                                       (const double*)pku, n, f);
    }
  }
  // tiles as even as they come, k split so that the blocks fill the SMs
  const int TM = (n_e + (n_e + pairs::kTile - 1) / pairs::kTile - 1) / ((n_e + pairs::kTile - 1) / pairs::kTile);
  const int TN = (n_p + (n_p + pairs::kTile - 1) / pairs::kTile - 1) / ((n_p + pairs::kTile - 1) / pairs::kTile);
  const int tx = (n_p + TN - 1) / TN, ty = (n_e + TM - 1) / TM;
  const int thr = (TM * TN + 31) & ~31;
  const size_t smem = (size_t)2 * pairs::TK * ((TM | 1) + (TN | 1)) * 16;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pairs::k_pair_products, thr, smem) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  const long Ks = 2L * g.N;
  // the split whose blocks fill whole waves best (at least 256 values of k each; fewer splits on a tie)
  const long slots = (long)per_sm * pairs::sms(), tiles = 2L * tx * ty;
  long S = 1;
  double best = 0.0;
  for (long c = 1; c <= std::min(64L, std::max(1L, Ks / 256)); ++c) {
    const double fill = (double)(tiles * c) / (double)((tiles * c + slots - 1) / slots * slots);
    if (fill > best + 0.01) {
      best = fill;
      S = c;
    }
  }
  const long kchunk = ((Ks + S - 1) / S + pairs::TK - 1) / pairs::TK * pairs::TK;
  S = (Ks + kchunk - 1) / kchunk;
  void* part = nullptr;
  if ((s = ws_get(ctx, "pairs.part", (size_t)2 * S * n_e * n_p * 16, &part)) != SWF_OK) return s;
  {
    ProfScope ps(ctx, "k_pair_products", st);
    pairs::k_pair_products<<<dim3(tx, ty, (unsigned)(2 * S)), thr, smem, st>>>(
        (const cpx<double>*)specU, (const cpx<double>*)specV, n_e, n_p, Ks, K, kchunk, (int)S, TM, TN, (cpx<double>*)part);
  }
  double vol = 1.0;
  for (int a = 0; a < 3; ++a)
    if (g.n[a] > 1) vol *= g.L[a];
  const double cell = g.dx[0] * g.dx[1] * g.dx[2];
  {
    ProfScope ps(ctx, "k_pair_results", st);
    const long MN = (long)n_e * n_p;
    pairs::k_pair_results<<<(unsigned)std::min((MN + 127) / 128, 65535L), 128, 0, st>>>(
        (const cpx<double>*)TU, (const cpx<double>*)TV, (const cpx<double>*)pwU, (const cpx<double>*)pwV,
        (const cpx<double>*)part, (int)S, cell * cell / vol, (const double*)normU, (const double*)normV, n_e, n_p,
        (swf_result*)pres);
  }
  e = cudaGetLastError();
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(results, pres, sizeof(swf_result) * (size_t)n_e * n_p, cudaMemcpyDeviceToHost, st);
  if (e != cudaSuccess) return cuda_status(e, "download pair results");
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_status(e, "pair matrix");
  return SWF_OK;
}
