#pragma once

// Fixed-point arithmetic of the Lindblad sweeps: FP64-grade products on the
// integer pipe.
//
// This GPU issues one FP64 warp instruction per 67 cycles and SM
// sub-partition (multiply-add; 78 for an add, 70 latency), but one 32 x 32
// -> 64 bit multiply-add (IMAD.WIDE) per 2 cycles with a latency of 2.6
// through the accumulator, a 32-bit add in 1, and a shift or a logical
// operation in 2 (measured).  A state entry is therefore held as a 64-bit
// integer X = x 2^sc with one power of two per state, kept so that the largest
// entry stays near 2^59, and multiplied by coefficients with 64 fraction
// bits through their signed 32-bit halves: three IMAD.WIDE per real
// product, 6 cycles against 67.  The absolute rounding of an entry is then
// 2^-60 of the state's largest entry, against 2^-53 of each entry in FP64:
// over a whole state (its 2-norm) that is the smaller error while the largest
// entry is below some 128 times the root mean square (kGridCrest, lb_internal.h:
// any state of N^2 <= 2^14, spread states of any size), but the small entries of
// a peaked state have fewer bits than in FP64, and those below 2^-60 are zero.
// Sums are exact and independent of their order.  Gradients against 80-bit
// references (largest error over the largest entry, fixed point and FP64): qubit,
// 1000 steps, eight seeds 0.8e-14 to 8.6e-14 and 8.7e-14 to 2.7e-13; CNOT, 1000
// steps, five seeds 0.9e-14 to 3.4e-14 and 4.2e-14 to 9.1e-14; four 4-level
// qudits, 30 steps, 1.4e-13 and 1.5e-13; six qutrits, 12 steps, 1.1e-13 and
// 1.1e-13 (there the solver's tolerance decides).

#include <cstdint>

#include <cuda_runtime.h>

namespace lbk {

namespace {

// value h 2^32 + l, l in [-2^31, 2^31): the low half is the integer's own low
// word, the high half its rounded high word (an add and a carry, where an
// unsigned low half of 31 bits takes a shift and a mask), and the left-out
// low x low products have zero mean
struct Fx {
  int h, l;
};
struct Cx {
  long long x, y;
};
// a sum of products: hi 2^64 + mid 2^32 (the low x low products, below one
// unit of the result, are left out)
struct FxAcc {
  long long hi, mid;
};

__host__ __device__ __forceinline__ Fx fx_split(long long X) {
  Fx r;
  r.l = (int)(unsigned)(unsigned long long)X;
  r.h = (int)((X + 0x80000000LL) >> 32);
  return r;
}
// a coefficient (magnitude below 1/2) with 64 fraction bits
__host__ __device__ __forceinline__ Fx fx_coef(long long A) { return fx_split(A); }
__host__ __device__ __forceinline__ Fx fx_neg(Fx a) {
  Fx r;
  r.h = -a.h;
  r.l = -a.l;
  return r;
}
// s + a b, as one IMAD.WIDE.  (Left to itself the compiler finds out the signs of
// the halves, extends them differently and then emits full 64-bit products,
// 4 instructions each.)
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
// the sum: rounded when `mid` started at 2^31 (fx_acc), else truncated
__host__ __device__ __forceinline__ long long fx_val(const FxAcc& s) { return fx_madw((int)(s.mid >> 32), 1, s.hi); }
__host__ __device__ __forceinline__ FxAcc fx_acc() {
  FxAcc s;
  s.hi = 0;
  s.mid = 0x80000000LL;
  return s;
}
// high half of a 32 x 32 bit product
__host__ __device__ __forceinline__ int fx_mulhi(int a, int b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int)(((long long)a * (long long)b) >> 32);
#endif
}
// A sum of products of two states' entries, hi 2^32 + lo in units of 2^32: each
// product whole but for its last 32 bits.  A gradient sum adds the products of
// all entries, and with one large entry among many small ones those small
// products are the gradient: cut at 2^64 (fx_val) they would carry an error of
// 2^-56 of the two states' largest entries each.
struct FxSum {
  long long hi;
  unsigned lo;
};
__host__ __device__ __forceinline__ void fx_sum_mac(FxSum& s, Fx a, Fx x) {
  long long mid = fx_madw(a.h, x.l, (long long)fx_mulhi(a.l, x.l));
  mid = fx_madw(a.l, x.h, mid);
  const unsigned long long lo = (unsigned long long)s.lo + (unsigned)mid;
  s.lo = (unsigned)lo;
  s.hi = fx_madw(a.h, x.h, s.hi) + (mid >> 32) + (long long)(lo >> 32);
}
__host__ __device__ __forceinline__ long long fx_join(Fx a) {
  return (long long)((unsigned long long)(unsigned)a.h << 32) + (long long)a.l;
}
// (ax + i ay) t, 64 fraction bits in the coefficient; |ax + i ay| < 0.48 and
// |t| <= 2^61 keep every partial sum inside 64 bits
__host__ __device__ __forceinline__ Cx fx_cmul(Fx ax, Fx ay, Cx t) {
  const Fx tx = fx_split(t.x), ty = fx_split(t.y);
  FxAcc re = fx_acc(), im = fx_acc();
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
  const int l = (int)(unsigned)(unsigned long long)X, h = (int)(X >> 32);
  const unsigned a = l < 0 ? 0u - (unsigned)l : (unsigned)l;
  return h == (l >> 31) ? a : 0xffffffffu;
}
// leading zero bits of h != 0
__host__ __device__ __forceinline__ int fx_clz(unsigned h) {
#ifdef __CUDA_ARCH__
  return __clz((int)h);
#else
  return __builtin_clz(h);
#endif
}
// X 2^-s (s < 0: X 2^|s|)
__host__ __device__ __forceinline__ long long fx_shift(long long X, int s) {
  if (s > 61 || s < -61) return 0;  // (to the left: X is zero there)
  return s >= 0 ? (X + ((1LL << s) >> 1)) >> s : (long long)((unsigned long long)X << -s);
}

// integer extrapolation weights (-1)^(k+1) C(n, k) of the predictors
__constant__ int kExtrapI[11][10] = {
    {0, 0, 0, 0, 0, 0, 0, 0, 0, 0},
    {1, 0, 0, 0, 0, 0, 0, 0, 0, 0},
    {2, -1, 0, 0, 0, 0, 0, 0, 0, 0},
    {3, -3, 1, 0, 0, 0, 0, 0, 0, 0},
    {4, -6, 4, -1, 0, 0, 0, 0, 0, 0},
    {5, -10, 10, -5, 1, 0, 0, 0, 0, 0},
    {6, -15, 20, -15, 6, -1, 0, 0, 0, 0},
    {7, -21, 35, -35, 21, -7, 1, 0, 0, 0},
    {8, -28, 56, -70, 56, -28, 8, -1, 0, 0},
    {9, -36, 84, -126, 126, -84, 36, -9, 1, 0},
    {10, -45, 120, -210, 252, -210, 120, -45, 10, -1}};

// a phase of one as the predictors' frames hold it: a quarter, 64 fraction bits
constexpr long long kFxPhase1 = 1LL << 62;
// (I - dt/2 D)^-1 - 1 = (dt/2 D)/(1 - dt/2 D), 64 fraction bits
__device__ __forceinline__ int4 fx_dinv1(double2 D, double hh) {
  const double nr = hh * D.x, ni = hh * D.y, ar = 1.0 - nr, ai = -ni, den = ar * ar + ai * ai;
  const Fx x = fx_coef(__double2ll_rn(scalbn((nr * ar + ni * ai) / den, 64)));
  const Fx y = fx_coef(__double2ll_rn(scalbn((ni * ar - nr * ai) / den, 64)));
  return make_int4(x.h, x.l, y.h, y.l);
}
// the element's frame factor per step, a quarter of the unit-modulus part of
// g = (1 + dt/2 D)/(1 - dt/2 D), 64 fraction bits; unit modulus to 2^-60
__device__ __forceinline__ Cx fx_frame(double2 D, double hh) {
  const double nr = hh * D.x, ni = hh * D.y, ar = 1.0 - nr, ai = -ni, den = ar * ar + ai * ai;
  const double gr = ((1.0 + nr) * ar + ni * ai) / den, gi = (ni * ar - (1.0 + nr) * ai) / den;
  const double r = hypot(gr, gi);
  Cx u;
  u.x = kFxPhase1;
  u.y = 0;
  if (!(r > 1e-3)) return u;
  const double ur = gr / r, ui = gi / r;
  const double e = 0.5 * (fma(-ur, ur, 1.0) - ui * ui);  // 1 - |u| to first order
  u.x = __double2ll_rn(scalbn(ur, 62)) + __double2ll_rn(scalbn(ur * e, 62));
  u.y = __double2ll_rn(scalbn(ui, 62)) + __double2ll_rn(scalbn(ui * e, 62));
  return u;
}

// dt/2 D, 64 fraction bits (magnitude below 1/2 where it is used)
__device__ __forceinline__ int4 fx_halfd(double2 D, double hh) {
  const Fx x = fx_coef(__double2ll_rn(scalbn(hh * D.x, 64))), y = fx_coef(__double2ll_rn(scalbn(hh * D.y, 64)));
  return make_int4(x.h, x.l, y.h, y.l);
}

// x 2^sc rounded, for |x| 2^sc < 2^62, on the integer pipe (subnormal x: zero)
__device__ __forceinline__ long long fx_from_bits(double x, int sc) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff, s = e - 1075 + sc;
  long long m = (long long)((b & 0xfffffffffffffull) | 0x10000000000000ull);
  if (s >= 0)
    m <<= s & 63;
  else
    m = s > -55 ? (m + ((1LL << (-s & 63)) >> 1)) >> (-s & 63) : 0;
  if (e == 0) m = 0;
  return (long long)b < 0 ? -m : m;
}

// headroom of a state's scale: the largest entry is set to [2^59, 2^60) at the
// start and the scale moved when it has left [2^58.5, 2^60)
constexpr int kFxTop = 59;
constexpr unsigned kFxHigh = 1u << (60 - 32), kFxLow = 94906266u;  // 2^26.5

// Largest change of an iterate that ends a solve: fac (rtol times the step's
// factor) of the right-hand side's largest entry (its high word), in units of
// the state; never below one unit, so that a state of zeros and an iterate
// that a tolerance below the format's resolution asks for are accepted.
__device__ __forceinline__ unsigned fx_stop(float fac, unsigned qtop) {
  const float t = fac * (float)qtop * 4294967296.0f;
  return t >= 4294967040.0f ? 0xffffff00u : (t >= 1.0f ? (unsigned)t : 1u);
}

// The shift that brings a state's largest entry back to [2^59, 2^60) from its
// high word (by more than one bit at once: a decay may halve a state and more
// each step); 0 while it lies in [2^58.5, 2^60) and for a state of zeros.
__host__ __device__ __forceinline__ int fx_rescale_shift(unsigned qtop) {
  return qtop < kFxHigh && (qtop >= kFxLow || qtop == 0) ? 0 : 4 - fx_clz(qtop);
}

// The shift that gives a quarter of a state its scale, from the quarter's
// largest high word: back to the state as it is when that lies in [2^58.5,
// 2^60), else to a largest entry in [2^59, 2^60).
__host__ __device__ __forceinline__ int fx_quarter_shift(unsigned top) {
  if (top == 0 || (top < kFxHigh / 4 && top >= kFxLow / 4)) return -2;
  return 4 - fx_clz(top);  // the top bit of the high word to bit 27
}

}  // namespace
}  // namespace lbk
