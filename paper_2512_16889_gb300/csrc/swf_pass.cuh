// Line FFTs in shared memory: whole lines (fft_pp), and the pieces of transforms whose first and last
// butterflies work in the registers of the thread that loads, stores or uses the values.
#pragma once

#include <algorithm>
#include <type_traits>

#include "swf_stage.cuh"

namespace swf {

// ---------------------------------------------------------------- out-of-place line FFT
// Element e of a line sits at e + e/16 (complex64) or e + e/8 (complex128): a gap every 128 bytes
// spreads the strided stores of the early passes over the shared-memory banks.
template <typename R>
__host__ __device__ __forceinline__ int pad(int e) { return e + (e >> (sizeof(R) == 4 ? 4 : 3)); }
template <typename R>
static inline int padded_len(int n) { return pad<R>(n - 1) + 1; }

// One self-sorting (Stockham) radix-RAD pass from `src` to `dst` over `nlines` lines of length
// n (stride ld, padded positions): butterfly (line, i < n/RAD) reads elements i + q n/RAD,
// multiplies by exp(-+ 2 pi i q k/(p RAD)) (k = i mod p, p = product of the radices so far),
// applies the RAD-point DFT and writes elements (i - k) RAD + k + q p.  Out of place, so each
// butterfly finishes before the next starts (one barrier per pass).
template <typename R, int RAD>
__device__ __forceinline__ void pp_pass(const cpx<R>* __restrict__ src, cpx<R>* __restrict__ dst, int ld,
                                        int nlines, int n, int p, bool inv, const cpx<R>* __restrict__ tw) {
  const int m = n / RAD;
  const int nb = nlines * m;
  const int twstep = n / (p * RAD);
  const FastDiv fm((unsigned)m), fp((unsigned)p);
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const int line = (int)fm.div((unsigned)b);
    const int i = b - line * m;
    const int k = i - p * (int)fp.div((unsigned)i);
    const cpx<R>* s = src + line * ld;
    cpx<R>* d = dst + line * ld;
    cpx<R> v[RAD];
#pragma unroll
    for (int q = 0; q < RAD; ++q) v[q] = s[pad<R>(i + q * m)];
    if (k != 0) {
      const int ks = k * twstep;
      if (RAD <= 5) {
#pragma unroll
        for (int q = 1; q < RAD; ++q) {
          cpx<R> w = tw[q * ks];
          if (inv) w.y = -w.y;
          v[q] = v[q] * w;
        }
      } else {
        // w^q for q < RAD from the table entries at the powers of two (at most three products
        // per factor: a few units in the last place)
        cpx<R> w[RAD];
#pragma unroll
        for (int q = 1; q < RAD; ++q) {
          if ((q & (q - 1)) == 0) {
            w[q] = tw[q * ks];
            if (inv) w[q].y = -w[q].y;
          } else {
            const int lo = q & (-q);  // lowest set bit: w^q = w^lo w^(q - lo)
            w[q] = w[lo] * w[q - lo];
          }
          v[q] = v[q] * w[q];
        }
      }
    }
    Dft<R, RAD>::run(v, inv);
    const int o = (i - k) * RAD + k;
#pragma unroll
    for (int q = 0; q < RAD; ++q) d[pad<R>(o + q * p)] = v[q];
  }
  __syncthreads();
}

// Full FFT of `nlines` lines held in `a` (padded layout; the caller has synchronised after
// writing them), using `b` as the second buffer.  Returns the buffer holding the result.
template <typename R>
__device__ cpx<R>* fft_pp(cpx<R>* a, cpx<R>* b, int ld, int nlines, const RadixPlan& pl, bool inv,
                          const cpx<R>* __restrict__ tw) {
  int p = 1;
  for (int ps = 0; ps < pl.npass; ++ps) {
    const int r = pl.rad[ps];
    switch (r) {
      case 16: pp_pass<R, 16>(a, b, ld, nlines, pl.n, p, inv, tw); break;
      case 20: pp_pass<R, 20>(a, b, ld, nlines, pl.n, p, inv, tw); break;
      case 12: pp_pass<R, 12>(a, b, ld, nlines, pl.n, p, inv, tw); break;
      case 8: pp_pass<R, 8>(a, b, ld, nlines, pl.n, p, inv, tw); break;
      case 4: pp_pass<R, 4>(a, b, ld, nlines, pl.n, p, inv, tw); break;
      case 2: pp_pass<R, 2>(a, b, ld, nlines, pl.n, p, inv, tw); break;
      case 3: pp_pass<R, 3>(a, b, ld, nlines, pl.n, p, inv, tw); break;
      default: pp_pass<R, 5>(a, b, ld, nlines, pl.n, p, inv, tw); break;
    }
    cpx<R>* t = a;
    a = b;
    b = t;
    p *= r;
  }
  return a;
}

// ---------------------------------------------------------------- passes of small radices
// Radix plan of the small-radix passes : fours, then fives, threes and a two; the two
// largest go to the ends.
static inline bool make_pass_plan(int n, RadixPlan* pl) {
  pl->n = n;
  pl->npass = 0;
  int m = n;
  const int order[4] = {4, 5, 3, 2};
  for (int r : order)
    while (m % r == 0 && pl->npass < 12) {
      pl->rad[pl->npass++] = r;
      m /= r;
    }
  if (pl->npass > 2) std::rotate(pl->rad + 1, pl->rad + 2, pl->rad + pl->npass);  // the second largest to the end
  return m == 1;
}

constexpr int kPassThreads = 512;  // at most, per block

// The march's plan for these passes: fours at both ends where the length has two, else the largest
// radices outside; sites side first.
__host__ __device__ inline int end_radix(const RadixPlan& pl, bool site) {
  return pl.npass == 0 ? 1 : pl.rad[site ? 0 : pl.npass - 1];
}
// Threads per line: one butterfly of the site side each, or several where `per` lines of that many
// threads would not fit a block.
static inline int pass_threads(const RadixPlan& pl, int per) {
  const int nb = pl.n / end_radix(pl, true);
  const int rounds = (nb * per + kPassThreads - 1) / kPassThreads;
  return (nb + rounds - 1) / rounds;
}

// The passes between the first and the last of a forward or inverse transform; a holds the first
// one's results (synchronised).  Returns the buffer with the last one's operands.
template <typename R>
__device__ __forceinline__ cpx<R>* middle_passes(cpx<R>* a, cpx<R>* b, int ld, int nlines, const RadixPlan& pl, bool inv,
                                                 const cpx<R>* __restrict__ tw) {
  int p = end_radix(pl, !inv);
  for (int s = 1; s < pl.npass - 1; ++s) {
    const int r = pl.rad[inv ? pl.npass - 1 - s : s];
    switch (r) {
      case 4: pp_pass<R, 4>(a, b, ld, nlines, pl.n, p, inv, tw); break;
      case 2: pp_pass<R, 2>(a, b, ld, nlines, pl.n, p, inv, tw); break;
      case 3: pp_pass<R, 3>(a, b, ld, nlines, pl.n, p, inv, tw); break;
      default: pp_pass<R, 5>(a, b, ld, nlines, pl.n, p, inv, tw); break;
    }
    cpx<R>* t = a;
    a = b;
    b = t;
    p *= r;
  }
  return a;
}

template <typename R> struct Dft<R, 1> {
  __device__ __forceinline__ static void run(cpx<R>*, bool) {}
};

// First butterfly b of a transform: DFT of v to positions b RAD .. of a line.
template <typename R, int RAD>
__device__ __forceinline__ void first_butterfly(cpx<R>* v, int b, bool inv, cpx<R>* line) {
  Dft<R, RAD>::run(v, inv);
#pragma unroll
  for (int q = 0; q < RAD; ++q) line[pad<R>(b * RAD + q)] = v[q];
}
// Last butterfly b of a transform of n points: the values b + q n/RAD (a transform of one pass has
// left them ready).
template <typename R, int RAD>
__device__ __forceinline__ void last_butterfly(const cpx<R>* line, int b, int n, bool one_pass, bool inv,
                                               const cpx<R>* __restrict__ tw, cpx<R>* v) {
  const int m = n / RAD;
#pragma unroll
  for (int q = 0; q < RAD; ++q) v[q] = line[pad<R>(b + q * m)];
  if (one_pass) return;
#pragma unroll
  for (int q = 1; q < RAD; ++q) {
    cpx<R> w = tw[q * b];
    if (inv) w.y = -w.y;
    v[q] = v[q] * w;
  }
  Dft<R, RAD>::run(v, inv);
}

// body(std::integral_constant<int, radix>) for the runtime radix of a plan's end.
template <typename Body>
__device__ __forceinline__ void with_radix(int r, Body&& body) {
  switch (r) {
    case 4: body(std::integral_constant<int, 4>()); break;
    case 2: body(std::integral_constant<int, 2>()); break;
    case 3: body(std::integral_constant<int, 3>()); break;
    case 5: body(std::integral_constant<int, 5>()); break;
    default: body(std::integral_constant<int, 1>()); break;
  }
}

}  // namespace swf
