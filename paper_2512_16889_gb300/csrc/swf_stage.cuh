// Device code shared by the march's kernels (Sec. II, Eq. 6; Sec. II.A): the arguments of one
// right-hand-side evaluation, the stage clock, the analytic gauge fields, V and the composite DFTs.
#pragma once

#include "swf_internal.h"

namespace swf {

template <typename R>
struct StageArgs {
  cpx<R>* y;
  const cpx<R>* kin[6];
  double coef[6];
  R coef_r[6];          // the same, rounded once (used without ctl)
  int nterm;
  int write_y;
  cpx<R>* kout;
  cpx<R>* T;
  const FieldDesc* fd;
  const R* greal;       // per field: gx[nx] gy[ny] gz[nz]
  const cpx<R>* gcplx;  // per field: ex[nx] ey[ny] ez[nz] w[4]
  const cpx<R>* tw[3];
  const R* kap;         // mode momenta kappa_j = 2 pi j'/L_a of the axes with n_a > 1, rounded once
                        // from FP64, at offsets 0, nx, nx + ny (FP64 is scarce on this GPU)
  R inv_n;              // 1/N rounded once
  RadixPlan plan[3];
  GridDesc g;
  int nrows;            // ny * nz
  double t;             // stage time when clk is null
  cpx<R>* ystage;       // optional: receives the stage value Y (Breit-Wheeler integrand)
  const struct MarchClock* clk;  // march clock (graph replays), or null
  int ls;               // step within the replayed pair of steps (0 or 1)
  double c;             // Dormand-Prince node c_i of the stage
  const struct StepControl* ctl;  // step-size-controlled march, or null (see march_adaptive)
  cpx<R>* ynew;         // with ctl: the last stage writes the step's result here, not into y
  cpx<R>* yspec;        // optional: receives the grid transform of the stage value (written by the
                        // y or z pass that applies H0, before it does)
  const cpx<R>* ltw[3]; // twiddles of the register line FFTs (swf_line.cuh) per axis, or null
  R* ft;                // optional: field time factors of the coming evaluation, [F][ny] (entry 0 of a
                        // field whose factor does not depend on y), and its background time phases
  cpx<R>* tf;           // [F]: written by the last y or z pass, read by the next x pass
  int nls;              // step (within the pair) and node of that coming evaluation
  double nc;
  cpx<R>* ylo;          // optional (complex64 fixed-step marches): the rounding error of y, so that
                        // y + ylo carries the state in float-float (Knuth's two-sum per step)
};

// (hi, lo) += s in float-float arithmetic (Knuth's two-sum, then a fast renormalisation): on
// return s holds the new rounded state and lo its rounding error.
__device__ __forceinline__ void ff_accumulate(float hi, float& lo, float& s) {
  const float t = __fadd_rn(hi, s);
  const float bp = __fsub_rn(t, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bp)), __fsub_rn(s, bp));
  const float l = __fadd_rn(lo, e);
  const float nh = __fadd_rn(t, l);
  lo = __fsub_rn(l, __fsub_rn(nh, t));
  s = nh;
}

// State of a step-size-controlled march, in device memory: the accepted time t and the step h
// of the current attempt (the stage times are t + c_i h and the stage coefficients h a_ij), the
// tolerances, counters and flags.  One thread of k_step_control updates it after every attempt.
struct StepControl {
  double t, h, t_in, span, rtol, atol;
  int done;        // t_in reached, or the march failed: later attempts do nothing
  int ok;          // the last attempt was accepted (its result and k_7 are copied in)
  int failed;      // too many attempts or a non-finite error
  int accepted, rejected, max_attempts;
};

// Device clock of a march whose steps are replayed from a CUDA graph: the stage time is
// (t_out + (step + ls) h) + c_i h, the host loop's arithmetic, with `step` advanced on the device
// after each replay.
struct MarchClock {
  double t_out, h;
  int step;
  int pad;
};

// Programmatic dependent launch (the kernels of a march's steps, see launch_chained): the next kernel of
// the chain is set up while this one runs.  chain_wait() returns when the kernels before this one have
// ended and their results are visible: nothing of theirs is read or overwritten before it.
// chain_release() lets the next kernel's blocks come in as this one's leave.  Without the launch
// attribute both do nothing.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename R>
__device__ __forceinline__ double node_time(const StageArgs<R>& A, int ls, double c) {
  if (A.ctl) return A.ctl->t + c * A.ctl->h;
  if (!A.clk) return A.t;
  const double tn = A.clk->t_out + (A.clk->step + ls) * A.clk->h;
  return tn + c * A.clk->h;
}
template <typename R>
__device__ __forceinline__ double stage_time(const StageArgs<R>& A) {
  return node_time(A, A.ls, A.c);
}

// ---------------------------------------------------------------- field and background
__device__ __forceinline__ double field_time_factor(const FieldDesc& F, double t, double y) {
  switch (F.kind) {
    case SWF_FIELD_SAUTER_GAUSS: {
      const double c = cosh(F.prm[1] * t);
      return (F.prm[0] / F.prm[1]) / (c * c);
    }
    case SWF_FIELD_PULSE_GAUSS: {
      const double u = t - y;
      return F.prm[0] * sin(F.prm[1] * u) * exp(-u * u / (F.prm[2] * F.prm[2]));
    }
    case SWF_FIELD_SINGLE_E:
    case SWF_FIELD_DOUBLE_E: {
      const double a = F.prm[1] * t;
      return exp(-a * a);
    }
    default:
      return 0.0;
  }
}

__device__ __forceinline__ double single_e_x(const FieldDesc& F, double x) {
  const double kx = F.prm[2];
  return -(F.prm[0] / kx) * sin(kx * x) * exp(-(kx * x) * (kx * x));
}

__device__ inline double axis_factor(const FieldDesc& F, int axis, double xc) {
  switch (F.kind) {
    case SWF_FIELD_SAUTER_GAUSS: {
      const double lam = F.prm[2];
      return lam > 0.0 ? exp(-xc * xc / (lam * lam)) : 1.0;
    }
    case SWF_FIELD_PULSE_GAUSS:
      if (axis == 0) return exp(-xc * xc / (F.prm[3] * F.prm[3]));
      if (axis == 1) return F.prm[4] > 0.0 ? exp(-xc * xc / (F.prm[4] * F.prm[4])) : 1.0;
      return 1.0;
    case SWF_FIELD_SINGLE_E:
    case SWF_FIELD_DOUBLE_E: {
      if (axis == 0) {
        if (F.kind == SWF_FIELD_SINGLE_E) return single_e_x(F, xc);
        return single_e_x(F, xc + F.prm[5]) + single_e_x(F, xc - F.prm[5]);
      }
      const double k = F.prm[2 + axis];
      return exp(-(k * xc) * (k * xc));
    }
    default:
      return 0.0;
  }
}

// v <- -i s (alpha.kappa + beta) v  (Dirac representation, sigma.kappa blocks).
template <typename R>
__device__ __forceinline__ void h0_mi(cpx<R>* v, R kx, R ky, R kz, R s) {
  const cpx<R> a = v[0], b = v[1], c = v[2], d = v[3];
  // sigma.k (u0, u1) = (kz u0 + (kx - i ky) u1, (kx + i ky) u0 - kz u1)
  const cpx<R> sl0 = kz * c + kx * d + ky * mul_mi(d);
  const cpx<R> sl1 = kx * c + ky * mul_i(c) - kz * d;
  const cpx<R> su0 = kz * a + kx * b + ky * mul_mi(b);
  const cpx<R> su1 = kx * a + ky * mul_i(a) - kz * b;
  v[0] = s * mul_mi(a + sl0);
  v[1] = s * mul_mi(b + sl1);
  v[2] = s * mul_mi(su0 - c);
  v[3] = s * mul_mi(su1 - d);
}

__device__ __forceinline__ double kappa_of(int j, int n, double L, double K) {
  return n > 1 ? mode_kappa(j, n, L) : K;
}


// ---------------------------------------------------------------- composite DFTs in registers
// cos and sin of 2 pi e / N for the composite radices (written out to 25 digits; indices and N are
// compile-time constants after unrolling, so every call folds to a literal).
__host__ __device__ constexpr double tw_const(int N, int e, bool want_cos) {
  switch (N) {
    case 6: {
      const double c[6] = {1.0, 0.5, -0.5, -1.0, -0.5, 0.5};
      const double s[6] = {0.0, 0.8660254037844386467637232, 0.8660254037844386467637232, 0.0,
          -0.8660254037844386467637232, -0.8660254037844386467637232};
      return want_cos ? c[e] : s[e];
    }
    case 8: {
      const double c[8] = {1.0, 0.7071067811865475244008444, 0.0, -0.7071067811865475244008444, -1.0,
          -0.7071067811865475244008444, 0.0, 0.7071067811865475244008444};
      const double s[8] = {0.0, 0.7071067811865475244008444, 1.0, 0.7071067811865475244008444, 0.0,
          -0.7071067811865475244008444, -1.0, -0.7071067811865475244008444};
      return want_cos ? c[e] : s[e];
    }
    case 9: {
      const double c[9] = {1.0, 0.7660444431189780352023927, 0.1736481776669303488517166, -0.5,
          -0.9396926207859083840541093, -0.9396926207859083840541093, -0.5, 0.1736481776669303488517166,
          0.7660444431189780352023927};
      const double s[9] = {0.0, 0.6427876096865393263226434, 0.984807753012208059366743, 0.8660254037844386467637232,
          0.3420201433256687330440996, -0.3420201433256687330440996, -0.8660254037844386467637232,
          -0.984807753012208059366743, -0.6427876096865393263226434};
      return want_cos ? c[e] : s[e];
    }
    case 10: {
      const double c[10] = {1.0, 0.8090169943749474241022934, 0.3090169943749474241022934,
          -0.3090169943749474241022934, -0.8090169943749474241022934, -1.0, -0.8090169943749474241022934,
          -0.3090169943749474241022934, 0.3090169943749474241022934, 0.8090169943749474241022934};
      const double s[10] = {0.0, 0.587785252292473129168706, 0.9510565162951535721164393,
          0.9510565162951535721164393, 0.587785252292473129168706, 0.0, -0.587785252292473129168706,
          -0.9510565162951535721164393, -0.9510565162951535721164393, -0.587785252292473129168706};
      return want_cos ? c[e] : s[e];
    }
    case 12: {
      const double c[12] = {1.0, 0.8660254037844386467637232, 0.5, 0.0, -0.5, -0.8660254037844386467637232, -1.0,
          -0.8660254037844386467637232, -0.5, 0.0, 0.5, 0.8660254037844386467637232};
      const double s[12] = {0.0, 0.5, 0.8660254037844386467637232, 1.0, 0.8660254037844386467637232, 0.5, 0.0, -0.5,
          -0.8660254037844386467637232, -1.0, -0.8660254037844386467637232, -0.5};
      return want_cos ? c[e] : s[e];
    }
    case 15: {
      const double c[15] = {1.0, 0.9135454576426008955021276, 0.6691306063588582138262733,
          0.3090169943749474241022934, -0.1045284632676534713998342, -0.5, -0.8090169943749474241022934,
          -0.9781476007338056379285667, -0.9781476007338056379285667, -0.8090169943749474241022934, -0.5,
          -0.1045284632676534713998342, 0.3090169943749474241022934, 0.6691306063588582138262733,
          0.9135454576426008955021276};
      const double s[15] = {0.0, 0.406736643075800207753986, 0.743144825477394235014697, 0.9510565162951535721164393,
          0.9945218953682733369226919, 0.8660254037844386467637232, 0.587785252292473129168706,
          0.2079116908177593371017423, -0.2079116908177593371017423, -0.587785252292473129168706,
          -0.8660254037844386467637232, -0.9945218953682733369226919, -0.9510565162951535721164393,
          -0.743144825477394235014697, -0.406736643075800207753986};
      return want_cos ? c[e] : s[e];
    }
    case 16: {
      const double c[16] = {1.0, 0.9238795325112867561281832, 0.7071067811865475244008444, 0.38268343236508977172846,
          0.0, -0.38268343236508977172846, -0.7071067811865475244008444, -0.9238795325112867561281832, -1.0,
          -0.9238795325112867561281832, -0.7071067811865475244008444, -0.38268343236508977172846, 0.0,
          0.38268343236508977172846, 0.7071067811865475244008444, 0.9238795325112867561281832};
      const double s[16] = {0.0, 0.38268343236508977172846, 0.7071067811865475244008444, 0.9238795325112867561281832,
          1.0, 0.9238795325112867561281832, 0.7071067811865475244008444, 0.38268343236508977172846, 0.0,
          -0.38268343236508977172846, -0.7071067811865475244008444, -0.9238795325112867561281832, -1.0,
          -0.9238795325112867561281832, -0.7071067811865475244008444, -0.38268343236508977172846};
      return want_cos ? c[e] : s[e];
    }
    case 18: {
      const double c[18] = {1.0, 0.9396926207859083840541093, 0.7660444431189780352023927, 0.5,
          0.1736481776669303488517166, -0.1736481776669303488517166, -0.5, -0.7660444431189780352023927,
          -0.9396926207859083840541093, -1.0, -0.9396926207859083840541093, -0.7660444431189780352023927, -0.5,
          -0.1736481776669303488517166, 0.1736481776669303488517166, 0.5, 0.7660444431189780352023927,
          0.9396926207859083840541093};
      const double s[18] = {0.0, 0.3420201433256687330440996, 0.6427876096865393263226434,
          0.8660254037844386467637232, 0.984807753012208059366743, 0.984807753012208059366743,
          0.8660254037844386467637232, 0.6427876096865393263226434, 0.3420201433256687330440996, 0.0,
          -0.3420201433256687330440996, -0.6427876096865393263226434, -0.8660254037844386467637232,
          -0.984807753012208059366743, -0.984807753012208059366743, -0.8660254037844386467637232,
          -0.6427876096865393263226434, -0.3420201433256687330440996};
      return want_cos ? c[e] : s[e];
    }
    case 20: {
      const double c[20] = {1.0, 0.9510565162951535721164393, 0.8090169943749474241022934,
          0.587785252292473129168706, 0.3090169943749474241022934, 0.0, -0.3090169943749474241022934,
          -0.587785252292473129168706, -0.8090169943749474241022934, -0.9510565162951535721164393, -1.0,
          -0.9510565162951535721164393, -0.8090169943749474241022934, -0.587785252292473129168706,
          -0.3090169943749474241022934, 0.0, 0.3090169943749474241022934, 0.587785252292473129168706,
          0.8090169943749474241022934, 0.9510565162951535721164393};
      const double s[20] = {0.0, 0.3090169943749474241022934, 0.587785252292473129168706,
          0.8090169943749474241022934, 0.9510565162951535721164393, 1.0, 0.9510565162951535721164393,
          0.8090169943749474241022934, 0.587785252292473129168706, 0.3090169943749474241022934, 0.0,
          -0.3090169943749474241022934, -0.587785252292473129168706, -0.8090169943749474241022934,
          -0.9510565162951535721164393, -1.0, -0.9510565162951535721164393, -0.8090169943749474241022934,
          -0.587785252292473129168706, -0.3090169943749474241022934};
      return want_cos ? c[e] : s[e];
    }
    case 24: {
      const double c[24] = {1.0, 0.9659258262890682867497432, 0.8660254037844386467637232,
          0.7071067811865475244008444, 0.5, 0.2588190451025207623488988, 0.0, -0.2588190451025207623488988, -0.5,
          -0.7071067811865475244008444, -0.8660254037844386467637232, -0.9659258262890682867497432, -1.0,
          -0.9659258262890682867497432, -0.8660254037844386467637232, -0.7071067811865475244008444, -0.5,
          -0.2588190451025207623488988, 0.0, 0.2588190451025207623488988, 0.5, 0.7071067811865475244008444,
          0.8660254037844386467637232, 0.9659258262890682867497432};
      const double s[24] = {0.0, 0.2588190451025207623488988, 0.5, 0.7071067811865475244008444,
          0.8660254037844386467637232, 0.9659258262890682867497432, 1.0, 0.9659258262890682867497432,
          0.8660254037844386467637232, 0.7071067811865475244008444, 0.5, 0.2588190451025207623488988, 0.0,
          -0.2588190451025207623488988, -0.5, -0.7071067811865475244008444, -0.8660254037844386467637232,
          -0.9659258262890682867497432, -1.0, -0.9659258262890682867497432, -0.8660254037844386467637232,
          -0.7071067811865475244008444, -0.5, -0.2588190451025207623488988};
      return want_cos ? c[e] : s[e];
    }
    case 25: {
      const double c[25] = {1.0, 0.9685831611286311194901684, 0.8763066800438635873081159,
          0.7289686274214115231467303, 0.5358267949789966182713088, 0.3090169943749474241022934,
          0.06279051952931337607617822, -0.1873813145857246305425507, -0.4257792915650726488625024,
          -0.6374239897486897101767128, -0.8090169943749474241022934, -0.9297764858882514036609426,
          -0.992114701314477831049793, -0.992114701314477831049793, -0.9297764858882514036609426,
          -0.8090169943749474241022934, -0.6374239897486897101767128, -0.4257792915650726488625024,
          -0.1873813145857246305425507, 0.06279051952931337607617822, 0.3090169943749474241022934,
          0.5358267949789966182713088, 0.7289686274214115231467303, 0.8763066800438635873081159,
          0.9685831611286311194901684};
      const double s[25] = {0.0, 0.2486898871648547882422837, 0.4817536741017152749871915,
          0.6845471059286886737322834, 0.8443279255020150785485581, 0.9510565162951535721164393,
          0.9980267284282715619523368, 0.9822872507286886810856417, 0.9048270524660195277136686,
          0.7705132427757892308030096, 0.587785252292473129168706, 0.3681245526846779591569471,
          0.1253332335643042453731188, -0.1253332335643042453731188, -0.3681245526846779591569471,
          -0.587785252292473129168706, -0.7705132427757892308030096, -0.9048270524660195277136686,
          -0.9822872507286886810856417, -0.9980267284282715619523368, -0.9510565162951535721164393,
          -0.8443279255020150785485581, -0.6845471059286886737322834, -0.4817536741017152749871915,
          -0.2486898871648547882422837};
      return want_cos ? c[e] : s[e];
    }
    case 32: {
      const double c[32] = {1.0, 0.9807852804032304491261822, 0.9238795325112867561281832,
          0.8314696123025452370787884, 0.7071067811865475244008444, 0.5555702330196022247428308,
          0.38268343236508977172846, 0.1950903220161282678482849, 0.0, -0.1950903220161282678482849,
          -0.38268343236508977172846, -0.5555702330196022247428308, -0.7071067811865475244008444,
          -0.8314696123025452370787884, -0.9238795325112867561281832, -0.9807852804032304491261822, -1.0,
          -0.9807852804032304491261822, -0.9238795325112867561281832, -0.8314696123025452370787884,
          -0.7071067811865475244008444, -0.5555702330196022247428308, -0.38268343236508977172846,
          -0.1950903220161282678482849, 0.0, 0.1950903220161282678482849, 0.38268343236508977172846,
          0.5555702330196022247428308, 0.7071067811865475244008444, 0.8314696123025452370787884,
          0.9238795325112867561281832, 0.9807852804032304491261822};
      const double s[32] = {0.0, 0.1950903220161282678482849, 0.38268343236508977172846, 0.5555702330196022247428308,
          0.7071067811865475244008444, 0.8314696123025452370787884, 0.9238795325112867561281832,
          0.9807852804032304491261822, 1.0, 0.9807852804032304491261822, 0.9238795325112867561281832,
          0.8314696123025452370787884, 0.7071067811865475244008444, 0.5555702330196022247428308,
          0.38268343236508977172846, 0.1950903220161282678482849, 0.0, -0.1950903220161282678482849,
          -0.38268343236508977172846, -0.5555702330196022247428308, -0.7071067811865475244008444,
          -0.8314696123025452370787884, -0.9238795325112867561281832, -0.9807852804032304491261822, -1.0,
          -0.9807852804032304491261822, -0.9238795325112867561281832, -0.8314696123025452370787884,
          -0.7071067811865475244008444, -0.5555702330196022247428308, -0.38268343236508977172846,
          -0.1950903220161282678482849};
      return want_cos ? c[e] : s[e];
    }
    default:
      return 0.0;
  }
}

// v * W_N^e (forward, W = exp(-2 pi i / N)) or v * conj(W_N^e) (inverse); quarter turns exact.
template <typename R>
__device__ __forceinline__ cpx<R> twiddle_const(cpx<R> v, int N, int e, bool inv) {
  if (e == 0) return v;
  if ((4 * e) % N == 0) {
    const int q = (4 * e / N) & 3;
    if (q == 2) return mk<R>(-v.x, -v.y);
    if ((q == 1) != inv) return mul_mi(v);
    return mul_i(v);
  }
  const R c = (R)tw_const(N, e, true), s = (R)tw_const(N, e, false);
  return v * mk<R>(c, inv ? s : -s);
}

// DFT of length A*B in registers (Cooley-Tukey): index n = B n1 + n2 in, k = k1 + A k2 out.
template <typename R, int A, int B>
struct DftCT {
  __device__ __forceinline__ static void run(cpx<R>* a, bool inv) {
    constexpr int N = A * B;
    cpx<R> y[N];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) {
      cpx<R> t[A];
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) t[n1] = a[B * n1 + n2];
      Dft<R, A>::run(t, inv);
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1) y[n2 * A + k1] = twiddle_const<R>(t[k1], N, n2 * k1, inv);
    }
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
      cpx<R> t[B];
#pragma unroll
      for (int n2 = 0; n2 < B; ++n2) t[n2] = y[n2 * A + k1];
      Dft<R, B>::run(t, inv);
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) a[k1 + A * k2] = t[k2];
    }
  }
};
template <typename R> struct Dft<R, 6> : DftCT<R, 2, 3> {};
template <typename R> struct Dft<R, 8> : DftCT<R, 4, 2> {};
template <typename R> struct Dft<R, 9> : DftCT<R, 3, 3> {};
template <typename R> struct Dft<R, 10> : DftCT<R, 2, 5> {};
template <typename R> struct Dft<R, 12> : DftCT<R, 4, 3> {};
template <typename R> struct Dft<R, 15> : DftCT<R, 3, 5> {};
template <typename R> struct Dft<R, 16> : DftCT<R, 4, 4> {};
template <typename R> struct Dft<R, 18> : DftCT<R, 2, 9> {};
template <typename R> struct Dft<R, 20> : DftCT<R, 4, 5> {};
template <typename R> struct Dft<R, 24> : DftCT<R, 4, 6> {};
template <typename R> struct Dft<R, 25> : DftCT<R, 5, 5> {};
template <typename R> struct Dft<R, 32> : DftCT<R, 4, 8> {};

}  // namespace swf
