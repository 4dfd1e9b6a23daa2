// window.cuh -- FP64 cells in windowed fixed point, on the integer pipes.
//
// The values that meet in a stencil cell usually lie within a few binades of
// each other.  While all values a warp holds have exponents within a window
// [eref, eref + k] (biased; k at most 7), a value is the integer X * 2^(eref -
// 1075), X = significand << (exponent - eref) < 2^60, converted once and used
// by every cell that reads it.  A plan's weights are integers too: W =
// significand << (exponent - emin), emin the smallest weight's exponent.  A
// cell's exact sum is then sum X * W, with no per-term alignment (compare
// stencil_exact_n() in common.cuh, which aligns every product of every cell):
// X is split at bit 32 (a1:a0), W at bit 29 (b1:b0), and the partial products
// of each weight of 2^0, 2^29, 2^61 add up in 64-bit accumulators that cannot
// overflow (b0s = 8 * b0 gives a1 * b0 the weight of a0 * b1):
//   S0 = sum a0 b0 < 5 * 2^61, S1 = S0 >> 29 + sum (a0 b1 + a1 b0s),
//   S2 = S1 >> 32 + sum a1 b1.
// S1 is bounded by the plan's own weights (window_weights()): of random normalised
// weights it stays below 2^64 for every set of an exponent spread h up to 6 and one in five
// of h = 7 (nine terms, below: up to 4, and one set in four of h = 5).  k = 7 for
// h <= 4, else 3, so k + h <= 11 = kExactGuard, so every windowed cell satisfies the
// integer path's contract and its correctly rounded sum is the result stencil_exact()
// gives: bit for bit the same, at about 50 instructions per cell instead of 166 (350
// against 150 Gcells/s measured alone at 1.99 GHz, register operands).
//
// The FMA chain's first product and its first FMA are evaluated the same way
// (window_mul, window_mul_fma: each rounded once, as the FP64 pipe rounds them),
// which leaves the FP64 pipe three of the chain's five operations.  That pipe
// takes 64 clocks for a warp's operation, about 40 integer instructions' worth
// of issue per SM quarter: alone, the chain runs at 100 Gcells/s, 125 with one
// and 164 with two operations moved; half windowed exact cells and half
// chains at 198, 244 and 309.
#pragma once

#include <cstring>

#include "common.cuh"

namespace j2d {

// The nine-term box cell works the same way with W split at bit 28 (J below), so
// that nine products still fit the columns.  A quarter of random nine-weight sets have
// no window (most for S1), four in a hundred five-weight ones.

// Weights in fixed point, in the cell's term order: xm, xp, ym, c, yp (NT = 5), or
// the box's chain order (NT = 9).
template <int NT> struct WindowWeightsN {
  static constexpr int J = NT == 5 ? 29 : 28;
  uint32_t b0[NT], b0s[NT], b1[NT];
  int emin;      // biased exponent of the smallest weight
  uint32_t lim;  // (k + 1) << 20: a value is in the window when (high word - (eref << 20)) < lim; 0: not applicable
};

using WindowWeights = WindowWeightsN<5>;

template <int NT> inline WindowWeightsN<NT> window_weights(const double (&w)[NT]) {
  constexpr int J = WindowWeightsN<NT>::J;
  WindowWeightsN<NT> r{};
  uint64_t m[NT];
  int e[NT], emin = 2047, emax = 0;
  for (int i = 0; i < NT; ++i) {
    uint64_t b;
    memcpy(&b, &w[i], 8);
    e[i] = (int)(b >> 52);  // with the sign: a negative weight fails the test below
    if (e[i] < 1 || e[i] > 2046) return r;
    m[i] = (b & ((1ull << 52) - 1)) | (1ull << 52);
    emin = e[i] < emin ? e[i] : emin;
    emax = e[i] > emax ? e[i] : emax;
  }
  const int h = emax - emin;
  if (h > 8) return r;
  uint64_t sum1 = 0, sum0s = 0;
  for (int i = 0; i < NT; ++i) {
    const uint64_t W = m[i] << (e[i] - emin);
    r.b0[i] = (uint32_t)(W & ((1u << J) - 1));
    r.b0s[i] = r.b0[i] << (32 - J);
    r.b1[i] = (uint32_t)(W >> J);
    sum1 += W >> J;
    sum0s += r.b0s[i];
  }
  r.emin = emin;
  for (int k : {7, 3})  // the wider window whose S1 < 2^32 sum b1 + 2^(21 + k) sum b0s + 2^36 stays below 2^64
    if (h + k <= kExactGuard && sum1 + (sum0s >> (11 - k)) + 17 <= 0xFFFFFFFFull) {
      r.lim = (uint32_t)(k + 1) << 20;
      break;
    }
  return r;
}

// A windowed value X = a1:a0.
struct Fx {
  uint32_t a0, a1;
};

__device__ __forceinline__ Fx shfl_up_fx(Fx v) {
  return {__shfl_up_sync(0xffffffffu, v.a0, 1), __shfl_up_sync(0xffffffffu, v.a1, 1)};
}
__device__ __forceinline__ Fx shfl_down_fx(Fx v) {
  return {__shfl_down_sync(0xffffffffu, v.a0, 1), __shfl_down_sync(0xffffffffu, v.a1, 1)};
}

// The window of a warp: cref = eref << 20, cb = (eref + emin - 1035) << 20 (NT = 9: - 1036).
struct Window {
  uint32_t cref, cb;
};

// A window whose top binade is the one above the biased exponent emax (of four
// binades only: that of emax); false when some result could be subnormal or too large.
template <int NT> __device__ __forceinline__ bool window_set(Window &q, const WindowWeightsN<NT> &w, int emax) {
  const int n = (int)(w.lim >> 20), eref = emax - n + (n == 8 ? 2 : 1);
  q.cref = (uint32_t)eref << 20;
  q.cb = (uint32_t)(eref + w.emin - 1064 + WindowWeightsN<NT>::J) << 20;
  return eref >= 1 && eref <= 1900 && eref + w.emin >= 1036 && eref + w.emin <= 3000;
}
// A value inside every window of that reference (padding outside the grid).
__device__ __forceinline__ double window_dummy(const Window &q) { return __hiloint2double((int)(q.cref + (2u << 20)), 0); }

// v in fixed point; dor collects the high words' distances from the window's
// start: the value is in the window when its distance is below WindowWeights::lim
// (a power of two, so the OR of several is below it only when each is; zeros,
// negative values, infinities and NaNs are not).
__device__ __forceinline__ Fx window_conv(double v, const Window &q, uint32_t &dor) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const uint32_t d = hi - q.cref;
  dor |= d;
  const uint32_t s = d >> 20;
  return {lo << (s & 31), __funnelshift_l(lo, (hi & 0xFFFFFu) | 0x100000u, s)};
}

__device__ __forceinline__ uint64_t mad_wide(uint32_t a, uint32_t b, uint64_t c) { return (uint64_t)a * b + c; }

// Round T = S2 * 2^(32 + J) + (S1 mod 2^32) * 2^J + S0 mod 2^J to 53 bits, to nearest
// even: hi:lo >> 10 is the rounded significand (2^52 .. 2^53, the leading bit moved
// to bit 62 of hi:lo); returns the leading bit's place p in S2's high word (11 .. 26).
template <int J> __device__ __forceinline__ uint32_t window_round(uint64_t S0, uint64_t S1, uint64_t S2, uint32_t &hi, uint32_t &lo) {
  const uint32_t s2h = (uint32_t)(S2 >> 32), s2l = (uint32_t)S2, s1l = (uint32_t)S1;
  uint32_t p;
  asm("bfind.u32 %0, %1;" : "=r"(p) : "r"(s2h));
  const uint32_t z = 30u - p;
  hi = __funnelshift_l(s2l, s2h, z);
  lo = __funnelshift_l(s1l, s2l, z);
  lo |= min(__funnelshift_l(0u, s1l, z) | ((uint32_t)S0 & ((1u << J) - 1)), 1u);  // sticky
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(lo), "+r"(hi) : "r"(0x1FFu + ((lo >> 10) & 1u)));
  return p;
}
__device__ __forceinline__ double window_compose(uint32_t p, uint32_t hi, uint32_t lo, const Window &q) {
  return __hiloint2double((int)((hi >> 10) + (p * 0x100000u + q.cb)), (int)__funnelshift_r(lo, hi, 10));
}

// The correctly rounded sum of the NT products.
template <int NT>
__device__ __forceinline__ double window_sum(const WindowWeightsN<NT> &w, const Window &q, const Fx (&x)[NT]) {
  constexpr int J = WindowWeightsN<NT>::J;
  uint64_t S0 = 0;
#pragma unroll
  for (int i = 0; i < NT; ++i) S0 = mad_wide(x[i].a0, w.b0[i], S0);
  uint64_t S1 = S0 >> J;
#pragma unroll
  for (int i = 0; i < NT; ++i) S1 = mad_wide(x[i].a1, w.b0s[i], mad_wide(x[i].a0, w.b1[i], S1));
  uint64_t S2 = S1 >> 32;
#pragma unroll
  for (int i = 0; i < NT; ++i) S2 = mad_wide(x[i].a1, w.b1[i], S2);
  uint32_t hi, lo;
  const uint32_t p = window_round<J>(S0, S1, S2, hi, lo);
  return window_compose(p, hi, lo, q);
}
__device__ __forceinline__ double window_exact(const WindowWeights &w, const Window &q, Fx xm, Fx xp, Fx ym, Fx c,
                                               Fx yp) {
  return window_sum<5>(w, q, {xm, xp, ym, c, yp});
}

// A cell of the integer path with a value outside the window, out of line (few
// cells take it).
static __device__ __noinline__ double general_exact_cell(double W, double E, double S, double C, double N, double xm,
                                                         double xp, double ym, double c, double yp) {
  const Links<double> l{W, E, S, C, N};
  return stencil_cell(l, exact_weights(l), true, xm, xp, ym, c, yp);
}

static __device__ __noinline__ double general_box_cell(Box9<double> b, double m0, double m1, double m2, double c0,
                                                       double c1, double c2, double p0, double p1, double p2) {
  return stencil_box_cell(b, box_exact_weights(b), true, m0, m1, m2, c0, c1, c2, p0, p1, p2);
}

// The first NI operations of the FMA chain, RN(.. RN(W[t1] x1 + RN(W[t0] x0))), each
// rounded once; t: the terms' indices in xm, xp, ym, c, yp order.
template <int NI, int NT>
__device__ __forceinline__ double window_head(const WindowWeightsN<NT> &w, const Window &q, const int (&t)[NI],
                                              const Fx (&x)[NI]) {
  constexpr int J = WindowWeightsN<NT>::J;
  uint32_t hi = 0, lo = 0, w0 = 0, w1 = 0, w2 = 0, p = 0;
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    if (i > 0) {
      // the rounded sum so far back at its place in the frame: bit 62 of hi:lo
      // belongs at bit 64 + J + p of T, i.e. hi:lo << (p + 2) in units of 2^J
      lo &= ~0x3FFu;
      const uint32_t r = p + 2;
      w0 = __funnelshift_l(0u, lo, r);
      w1 = __funnelshift_l(lo, hi, r);
      w2 = __funnelshift_l(hi, 0u, r);
    }
    const uint64_t S0 = mad_wide(x[i].a0, w.b0[t[i]], 0);
    const uint64_t S1 = mad_wide(x[i].a1, w.b0s[t[i]], mad_wide(x[i].a0, w.b1[t[i]], (S0 >> J) + w0));
    const uint64_t S2 = mad_wide(x[i].a1, w.b1[t[i]], (((uint64_t)w2 << 32) | w1) + (S1 >> 32));
    p = window_round<J>(S0, S1, S2, hi, lo);
  }
  return window_compose(p, hi, lo, q);
}

}  // namespace j2d
