#pragma once

// Fixed-point arithmetic of the Lindblad sweeps: FP64-grade products on the
// integer pipe.
//
// This GPU issues one FP64 warp instruction per 67 cycles and SM
// sub-partition (multiply-add; 78 for an add, 70 latency), but one 32 x 32
// -> 64 bit multiply-add (IMAD.WIDE) per 2 cycles with a latency of 2.6
// through the accumulator, and a 64-bit add in 2 (measured).  A state entry is therefore
// held as a 64-bit integer X = x 2^sc with one power of two per state, kept
// so that the largest entry stays near 2^58, and multiplied by coefficients
// with 62 fraction bits through their 31-bit halves: three IMAD.WIDE per real
// product, 6 cycles against 67.  The absolute rounding of an entry is then
// 2^-60 of the state's largest entry, against 2^-54 of each entry in FP64:
// over a whole state (its 2-norm) that is the smaller error, and sums are
// exact and independent of their order.  Against 80-bit references the sweeps
// are 20 to 40 times closer than FP64 (qubit and CNOT gradients).

#include <cstdint>

#include <cuda_runtime.h>

namespace lbk {

namespace {

// value h 2^31 + l; l in [0, 2^31) for entries, [-2^30, 2^30) for coefficients
struct Fx {
  int h, l;
};
struct Cx {
  long long x, y;
};
// a sum of products: hi 2^62 + mid 2^31 (the low x low products, below one
// unit of the result, are left out; `mid` starts from 2^30 plus their mean,
// so that the result is rounded and unbiased)
struct FxAcc {
  long long hi, mid;
};

__host__ __device__ __forceinline__ Fx fx_split(long long X) {
  Fx r;
  r.h = (int)(X >> 31);
  r.l = (int)((unsigned)X & 0x7fffffffu);
  return r;
}
// a coefficient: signed low half, so that negation is the halves' negation
// and the low products have zero mean over the entries' low halves' centre
__host__ __device__ __forceinline__ Fx fx_coef(long long A) {
  Fx r;
  r.l = (int)((unsigned)A & 0x7fffffffu);
  long long h = A >> 31;
  if (r.l >= 0x40000000) {
    r.l = (int)((unsigned)r.l - 0x80000000u);
    ++h;
  }
  r.h = (int)h;
  return r;
}
__host__ __device__ __forceinline__ Fx fx_neg(Fx a) {
  Fx r;
  r.h = -a.h;
  r.l = -a.l;
  return r;
}
// s + a b, as one IMAD.WIDE.  (Written in C++ the compiler sees that a low half
// is never negative, extends it without sign and then finds no mixed-sign wide
// product: it emits full 64-bit ones, 4 instructions each.)
__host__ __device__ __forceinline__ long long fx_madw(int a, int b, long long s) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(s));
  return r;
#else
  return s + (long long)a * (long long)b;
#endif
}
__host__ __device__ __forceinline__ void fx_mac(FxAcc& s, Fx a, Fx x) {
  s.hi = fx_madw(a.h, x.h, s.hi);
  s.mid = fx_madw(a.h, x.l, s.mid);
  s.mid = fx_madw(a.l, x.h, s.mid);
}
__host__ __device__ __forceinline__ long long fx_val(const FxAcc& s) { return s.hi + (s.mid >> 31); }
// the start of `mid` for the coefficients with low halves summing to l
__host__ __device__ __forceinline__ FxAcc fx_acc(int l) {
  FxAcc s;
  s.hi = 0;
  s.mid = (1LL << 30) + (long long)(l >> 1);
  return s;
}
// (ax + i ay) t, 62 fraction bits in the coefficient; |ax|, |ay| <= 1/2 and
// |t| <= 2^61 keep every partial sum inside 64 bits
__host__ __device__ __forceinline__ Cx fx_cmul(Fx ax, Fx ay, Cx t) {
  const Fx tx = fx_split(t.x), ty = fx_split(t.y);
  FxAcc re = fx_acc(ax.l - ay.l), im = fx_acc(ax.l + ay.l);
  fx_mac(re, ax, tx);
  fx_mac(re, fx_neg(ay), ty);
  fx_mac(im, ax, ty);
  fx_mac(im, ay, tx);
  Cx r;
  r.x = fx_val(re);
  r.y = fx_val(im);
  return r;
}
// magnitude's high word, and the magnitude saturated to 32 bits
__host__ __device__ __forceinline__ unsigned fx_hi_abs(long long X) {
  const int h = (int)(X >> 32);
  return (unsigned)(h ^ (h >> 31));
}
__host__ __device__ __forceinline__ unsigned fx_abs_sat(long long X) {
  const unsigned long long a = X < 0 ? 0ull - (unsigned long long)X : (unsigned long long)X;
  return (a >> 32) ? 0xffffffffu : (unsigned)a;
}
// X 2^-s (s < 0: X 2^|s|)
__host__ __device__ __forceinline__ long long fx_shift(long long X, int s) {
  if (s > 61 || s < -61) return 0;  // (to the left: X is zero there)
  return s >= 0 ? (X + ((1LL << s) >> 1)) >> s : (long long)((unsigned long long)X << -s);
}

// (I - dt/2 D)^-1 - 1 = (dt/2 D)/(1 - dt/2 D), 62 fraction bits
__device__ __forceinline__ int4 fx_dinv1(double2 D, double hh) {
  const double nr = hh * D.x, ni = hh * D.y, ar = 1.0 - nr, ai = -ni, den = ar * ar + ai * ai;
  const Fx x = fx_coef(__double2ll_rn(scalbn((nr * ar + ni * ai) / den, 62)));
  const Fx y = fx_coef(__double2ll_rn(scalbn((ni * ar - nr * ai) / den, 62)));
  return make_int4(x.h, x.l, y.h, y.l);
}
// the element's frame factor per step, half of the unit-modulus part of
// g = (1 + dt/2 D)/(1 - dt/2 D), 62 fraction bits; unit modulus to 2^-60
__device__ __forceinline__ Cx fx_frame(double2 D, double hh) {
  const double nr = hh * D.x, ni = hh * D.y, ar = 1.0 - nr, ai = -ni, den = ar * ar + ai * ai;
  const double gr = ((1.0 + nr) * ar + ni * ai) / den, gi = (ni * ar - (1.0 + nr) * ai) / den;
  const double r = hypot(gr, gi);
  Cx u;
  u.x = 1LL << 61;
  u.y = 0;
  if (!(r > 1e-3)) return u;
  const double ur = gr / r, ui = gi / r;
  const double e = 0.5 * (fma(-ur, ur, 1.0) - ui * ui);  // 1 - |u| to first order
  u.x = __double2ll_rn(scalbn(ur, 61)) + __double2ll_rn(scalbn(ur * e, 61));
  u.y = __double2ll_rn(scalbn(ui, 61)) + __double2ll_rn(scalbn(ui * e, 61));
  return u;
}

// dt/2 D, 62 fraction bits (magnitude below 1/2 where it is used)
__device__ __forceinline__ int4 fx_halfd(double2 D, double hh) {
  const Fx x = fx_coef(__double2ll_rn(scalbn(hh * D.x, 62))), y = fx_coef(__double2ll_rn(scalbn(hh * D.y, 62)));
  return make_int4(x.h, x.l, y.h, y.l);
}

// headroom of a state's scale: the largest entry is set to [2^59, 2^60) at the
// start and the scale moved by 2 when it has left [2^58.5, 2^60)
constexpr int kFxTop = 59;
constexpr unsigned kFxHigh = 1u << (60 - 32), kFxLow = 94906266u;  // 2^26.5

}  // namespace
}  // namespace lbk
