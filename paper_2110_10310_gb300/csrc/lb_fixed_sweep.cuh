#pragma once

// One-CTA-per-state sweeps in fixed point (lb_fixed.cuh): the device code
// their forward, backward and propagation kernels share.
//
// The Jacobi sweeps of small and medium states (N^2 <= 4096) with every step's
// iteration matrix bounded by kFixedRho (lb_api.cu decides; larger controls, the
// Neumann iteration and GMRES keep the FP64 sweeps).  One CTA owns a state,
// its iterate in shared memory as split 64-bit integers, and runs the whole
// time loop; a step whose predicted first iterate is within the tolerance
// costs one operator product and two CTA barriers.
//
// Two neighbouring lanes share an element, one per real component: the real
// ladder and decay coefficients act on each component alone, so a lane needs
// its own component of the neighbours only, and the two meet in one exchange
// per product for the complex control factors.  That halves each lane's
// chain and registers and doubles the warps, which is what the single warp per
// sub-partition of a small state lacks (one lane per element: 4 cycles per
// instruction, all of them dependent-issue waits).
//
// What bounds it: the issue of integer multiply-adds (IMAD.WIDE, one warp
// instruction per 2 cycles and SM sub-partition) for large states, the
// dependent chain of a step for small ones.  In FP64 the element takes 18
// instructions of 67 cycles per subsystem and product.
//
// E: elements per lane pair.  QT > 0 (E = 1, up to 256 elements): the
// element's neighbour offsets and coefficients for QT units (subsystems and
// Jaynes-Cummings pairs) and the predictor's difference table in registers.
// QT == 0: coefficients from small shared-memory tables, the predictor's ring
// in the workspace.

#include "lb_device.cuh"
#include "lb_fixed.cuh"

namespace lbk {

namespace {

constexpr int kFxPlanThreads = 512;  // largest CTA of the register plan (128 registers per thread)
constexpr int kFxTabThreads = 1024;  // ... of the table path (64 registers)
// ... of its smaller CTAs with one element per lane pair: 80 registers and next
// to no spills (300 elements, 9 states: forward 4.33 us per step against 4.70
// in 64 registers).  More elements in one pair instead of more threads
// is slower (406 elements, 28 states: 11.8 us with two in 416 threads, 8.3 in 832).
constexpr int kFxTabFew = 768;
constexpr int kFxWarps = 32;
constexpr int kFxOrder = 8;          // highest extrapolation order of the register difference table
template <int QT>
constexpr int fx_max_threads() {
  return QT > 0 ? kFxPlanThreads : kFxTabThreads;
}

// one subsystem, for the table path: levels n, index stride s, bit position of
// its digit, whether it decays, and the offsets of its ladder and decay factors
struct FxSub {
  int n_sh;  // n | digit shift << 8 | decay << 16
  int s;
  int co, jo;
};

struct FxSmem {
  Hdr* hdr;
  FxSub* sub;       // [Q]
  int4* ck;         // [ncoef] (cu, cd): sqrt(n+1) 2^-kc of the subsystem (0 at the top level), sqrt(n) 2^-kc
  int4* cl;         // [ncoef] (-cd, -cu)
  Fx* jf;           // [njcoef] decay factors
  Fx* ja;
  uint32_t* dig;    // [N]
  uint16_t* hmap;   // [Vh] vec index of element u (Hermitian symmetry)
  uint16_t* hmir;   // [Vh] its mirror, 0xffff on the diagonal
  unsigned* slots;  // [2][2][32]: per step parity the warps' max |rhs|, per iteration parity their max change
  int4* ctl;        // [2][cq + 1] control factors of the step (a, b split), last the stopping factor
  int* gred;        // [2][Q][4][kFxWarps][3] limbs of the warps' gradient sums, by step parity
  unsigned long long* mx;  // [kFxWarps] fx_cta_max's
  int4* dsm;        // [nel] (I - dt/2 D)^-1 - 1 (QT == 0)
  Fx* zb0;          // [V][2] iterate, split, component by component
  Fx* zb1;
  unsigned char* base;
  __device__ __forceinline__ int off(const void* p) const {
    return (int)(reinterpret_cast<const unsigned char*>(p) - base);
  }
};

__host__ __device__ inline size_t fx_smem_bytes(int ncoef, int njcoef, int N, int V, int Q, int cq, int nel, int QT) {
  size_t b = align16(sizeof(Hdr)) + sizeof(FxSub) * LB_MAXQ;
  b += 2 * sizeof(int4) * ncoef + 2 * align16(sizeof(Fx) * njcoef);
  b += align16(sizeof(uint32_t) * N);
  b += 2 * align16(sizeof(uint16_t) * (size_t)N * (N + 1) / 2);
  b += sizeof(unsigned) * 128;
  b += sizeof(int4) * 2 * (cq + 1);
  b += align16(sizeof(int) * 2 * 4 * Q * kFxWarps * 3);
  b += sizeof(unsigned long long) * kFxWarps;
  // the table path reads up to V/2 + N/2 entries before and after a buffer
  const size_t pad = sizeof(Fx) * (size_t)(V + N);
  if (QT == 0 && b < pad) b = align16(pad);
  b += sizeof(Fx) * 4 * (size_t)V;
  if (QT == 0) b += sizeof(int4) * (size_t)nel > pad ? sizeof(int4) * (size_t)nel : pad;
  return b;
}

__device__ __forceinline__ FxSmem fx_carve(unsigned char* base, const ProbDev& P, int nel, int QT) {
  FxSmem S;
  S.base = base;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    unsigned char* p = base + o;
    o += align16(bytes);
    return p;
  };
  S.hdr = reinterpret_cast<Hdr*>(take(sizeof(Hdr)));
  S.sub = reinterpret_cast<FxSub*>(take(sizeof(FxSub) * LB_MAXQ));
  S.ck = reinterpret_cast<int4*>(take(sizeof(int4) * P.ncoef));
  S.cl = reinterpret_cast<int4*>(take(sizeof(int4) * P.ncoef));
  S.jf = reinterpret_cast<Fx*>(take(sizeof(Fx) * P.njcoef));
  S.ja = reinterpret_cast<Fx*>(take(sizeof(Fx) * P.njcoef));
  S.dig = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * P.N));
  S.hmap = reinterpret_cast<uint16_t*>(take(sizeof(uint16_t) * (size_t)P.N * (P.N + 1) / 2));
  S.hmir = reinterpret_cast<uint16_t*>(take(sizeof(uint16_t) * (size_t)P.N * (P.N + 1) / 2));
  S.slots = reinterpret_cast<unsigned*>(take(sizeof(unsigned) * 128));
  S.ctl = reinterpret_cast<int4*>(take(sizeof(int4) * 2 * (P.cq + 1)));
  S.gred = reinterpret_cast<int*>(take(sizeof(int) * 2 * 4 * P.Q * kFxWarps * 3));
  S.mx = reinterpret_cast<unsigned long long*>(take(sizeof(unsigned long long) * kFxWarps));
  const size_t pad = sizeof(Fx) * (size_t)(P.V + P.N);
  if (QT == 0 && o < pad) o = align16(pad);
  S.zb0 = reinterpret_cast<Fx*>(take(sizeof(Fx) * 2 * (size_t)P.V));
  S.zb1 = reinterpret_cast<Fx*>(take(sizeof(Fx) * 2 * (size_t)P.V));
  S.dsm = reinterpret_cast<int4*>(QT == 0 ? take(sizeof(int4) * (size_t)nel) : nullptr);
  return S;
}

__device__ __forceinline__ long long fx_from(double x, int sc) { return __double2ll_rn(scalbn(x, sc)); }
__device__ __forceinline__ double fx_to(long long X, int sc) { return scalbn((double)X, -sc); }
__device__ __forceinline__ long long fx_other(long long x) { return __shfl_xor_sync(kFull, x, 1); }
__device__ __forceinline__ void fx_setup(const FxSmem& S, const ProbDev& P, int herm) {
  if (threadIdx.x == 0) {
    load_hdr(*S.hdr, P);
    S.hdr->herm = herm;
  }
  if ((int)threadIdx.x < P.Q) {
    const int q = threadIdx.x;
    FxSub b;
    b.n_sh = P.levels[q] | (P.dbits * q) << 8 | (P.jump[q] != 0.0 ? 1 << 16 : 0);
    b.s = P.stride[q];
    b.co = P.coff[q];
    b.jo = P.joff[q];
    S.sub[q] = b;
  }
  if (herm)
    for (int i = threadIdx.x; i < P.N * (P.N + 1) / 2; i += blockDim.x) {
      const uint32_t t = P.hkl[i];
      const int k = (int)(t & 0xffffu), l = (int)(t >> 16);
      S.hmap[i] = (uint16_t)(k + P.N * l);
      S.hmir[i] = k != l ? (uint16_t)(l + P.N * k) : (uint16_t)0xffffu;
    }
  for (int i = threadIdx.x; i < P.ncoef; i += blockDim.x) {
    int q = 0;
    while (q + 1 < P.Q && P.coff[q + 1] <= i) ++q;
    const Fx u = fx_coef(__double2ll_rn(scalbn(P.cu[i], 64 - P.kc[q])));
    const Fx d = fx_coef(__double2ll_rn(scalbn(P.cd[i], 64 - P.kc[q])));
    S.ck[i] = make_int4(u.h, u.l, d.h, d.l);
    S.cl[i] = make_int4(-d.h, -d.l, -u.h, -u.l);
  }
  for (int i = threadIdx.x; i < P.njcoef; i += blockDim.x) {
    S.jf[i] = fx_coef(__double2ll_rn(scalbn(P.jf[i], 64)));
    S.ja[i] = fx_coef(__double2ll_rn(scalbn(P.ja[i], 64)));
  }
  for (int i = threadIdx.x; i < P.N; i += blockDim.x) S.dig[i] = P.digits[i];
  for (int i = threadIdx.x; i < 128; i += blockDim.x) S.slots[i] = 0u;
  __syncthreads();
}

// max of the warps' values over the CTA (w: the warps' slots, 32 entries, unused ones 0)
__device__ __forceinline__ unsigned fx_slots_max(const unsigned* w, int nwarps) {
  if (nwarps > 8) return __reduce_max_sync(kFull, w[threadIdx.x & 31]);
  const uint4 a = *reinterpret_cast<const uint4*>(w);
  unsigned m = max(max(a.x, a.y), max(a.z, a.w));
  if (nwarps > 4) {
    const uint4 b = *reinterpret_cast<const uint4*>(w + 4);
    m = max(m, max(max(b.x, b.y), max(b.z, b.w)));
  }
  return m;
}

// CTA maximum of a double's magnitude bits
__device__ __forceinline__ unsigned long long fx_cta_max(const FxSmem& S, unsigned long long m) {
  unsigned long long* w = S.mx;
  m = warp_max_u64(m);
  if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = m;
  __syncthreads();
  m = 0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) m = umax64(m, w[i]);
  __syncthreads();
  return m;
}
// scale exponent sc with max 2^sc in [2^59, 2^60) (max: FP64 bits, finite)
__device__ __forceinline__ int fx_scale(unsigned long long maxbits) {
  const int e = (int)(maxbits >> 52);
  return maxbits ? kFxTop - (e ? e - 1023 : -1022) : kFxTop;
}

// ---------------------------------------------------------------------------
// elements and operator product

// QT > 0: the lane's neighbours (byte offsets into an iterate buffer, its
// component included) and real coefficients for every unit, a subsystem's
// control terms or (past the subsystems) a Jaynes-Cummings pair's:
//   P = c0 x[o0] + c1 x[o1], R = c2 x[o2] + c3 x[o3]   (c1, c3 negated)
// with, for a subsystem, P = sqrt(nk+1) x[k+s,l] - sqrt(nl) x[k,l-s] and
// R = sqrt(nk) x[k-s,l] - sqrt(nl+1) x[k,l+s], times 2^-kc.
template <int QT>
struct FxPlan {
  int o[QT][4];
  Fx c[QT][4];
  int oj[QT][2];  // decay neighbour of M ([k+s,l+s]) and of M^+ ([k-s,l-s])
  Fx cj[QT][2];
  int nu;         // units
  int nq;         // subsystems
  unsigned jon;   // bit q: subsystem q decays
};
template <>
struct FxPlan<0> {};

template <int QT>
__device__ __forceinline__ void fx_plan(FxPlan<QT>& pl, const FxSmem& S, const ProbDev& P, int v) {
  const Hdr& H = *S.hdr;
  const bool ok = v < H.V;
  const Fx zero{0, 0};
  const uint32_t kd = ok ? S.dig[v % H.N] : 0u, ld = ok ? S.dig[v / H.N] : 0u;
  pl.nu = H.Q + H.npair;
  pl.nq = H.Q;
  pl.jon = H.jon;
  auto at = [&](int w) { return (2 * w + (int)(threadIdx.x & 1)) * (int)sizeof(Fx); };
#pragma unroll
  for (int u = 0; u < QT; ++u) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      pl.o[u][i] = 0;
      pl.c[u][i] = zero;
    }
    pl.oj[u][0] = pl.oj[u][1] = 0;
    pl.cj[u][0] = pl.cj[u][1] = zero;
    if (!ok || u >= pl.nu) continue;
    if (u < H.Q) {
      const int q = u, n = H.lev[q], s = H.stride[q], co = H.coff[q], sN = s * H.N;
      const int nk = (kd >> (H.db * q)) & H.dm, nl = (ld >> (H.db * q)) & H.dm;
      const int jo = H.joff[q] + nk * n + nl;
      pl.o[u][0] = at(v + (nk + 1 < n ? s : 0));
      pl.o[u][1] = at(v - (nl > 0 ? sN : 0));
      pl.o[u][2] = at(v - (nk > 0 ? s : 0));
      pl.o[u][3] = at(v + (nl + 1 < n ? sN : 0));
      const int4 ck = S.ck[co + nk], cl = S.cl[co + nl];
      pl.c[u][0] = Fx{ck.x, ck.y};
      pl.c[u][1] = Fx{cl.x, cl.y};
      pl.c[u][2] = Fx{ck.z, ck.w};
      pl.c[u][3] = Fx{cl.z, cl.w};
      pl.oj[u][0] = at(v + ((nk + 1 < n && nl + 1 < n) ? s + sN : 0));
      pl.oj[u][1] = at(v - ((nk > 0 && nl > 0) ? s + sN : 0));
      pl.cj[u][0] = S.jf[jo];
      pl.cj[u][1] = S.ja[jo];
    } else {
      // U like P with the factor G, W like R with its conjugate (offdiag_acc)
      const int kp = u - H.Q, p = H.jp[kp], q = H.jq[kp];
      const int np = H.lev[p], nq = H.lev[q], d = H.stride[q] - H.stride[p], cp = H.coff[p], cq = H.coff[q];
      const int pk = (kd >> (H.db * p)) & H.dm, qk = (kd >> (H.db * q)) & H.dm;
      const int pL = (ld >> (H.db * p)) & H.dm, qL = (ld >> (H.db * q)) & H.dm;
      auto cf = [&](double a, double b) { return fx_coef(__double2ll_rn(scalbn(a * b, 64 - P.kc[u]))); };
      pl.o[u][0] = at(v + ((pk > 0 && qk + 1 < nq) ? d : 0));
      pl.o[u][1] = at(v - ((qL > 0 && pL + 1 < np) ? d * H.N : 0));
      pl.o[u][2] = at(v - ((qk > 0 && pk + 1 < np) ? d : 0));
      pl.o[u][3] = at(v + ((pL > 0 && qL + 1 < nq) ? d * H.N : 0));
      pl.c[u][0] = cf(P.cd[cp + pk], P.cu[cq + qk]);
      pl.c[u][1] = cf(-P.cu[cp + pL], P.cd[cq + qL]);
      pl.c[u][2] = cf(P.cu[cp + pk], P.cd[cq + qk]);
      pl.c[u][3] = cf(-P.cd[cp + pL], P.cu[cq + qL]);
    }
  }
}

// P and R of one unit, this lane's component (2^-kc times the neighbour combinations)
struct FxPR {
  long long p, r;
};
__device__ __forceinline__ FxPR fx_pr(Fx x1, Fx x2, Fx x3, Fx x4, Fx c1, Fx c2, Fx c3, Fx c4) {
  FxAcc p{0, 0}, r{0, 0};
  fx_mac(p, c1, x1);
  fx_mac(p, c2, x2);
  fx_mac(r, c3, x3);
  fx_mac(r, c4, x4);
  return FxPR{fx_val(p), fx_val(r)};
}
// This lane's shares of a unit with factors (a, b), a + i b = (dt/2) d:
//   b (P - R) - i a (P + R) = (b W.x + a U.y) + i (b W.y - a U.x)
// of its component W, U: own += b W (+ the decay term), cross += a U.
__device__ __forceinline__ void fx_unit(long long& own, long long& cross, const FxPR& p, int4 t, bool decay, Fx cj,
                                        Fx x5) {
  const Fx a{t.x, t.y}, b{t.z, t.w};
  const Fx u = fx_split(p.p + p.r), w = fx_split(p.p - p.r);
  FxAcc o = fx_acc(), x = fx_acc();
  fx_mac(o, b, w);
  fx_mac(x, a, u);
  if (decay) fx_mac(o, cj, x5);
  own += fx_val(o);
  cross += fx_val(x);
}
// ... for the adjoint (its Hamiltonian part is minus that of M)
__device__ __forceinline__ void fx_unit_adj(long long& own, long long& cross, const FxPR& p, int4 t, bool decay, Fx cj,
                                            Fx x5) {
  const Fx a{t.x, t.y}, b{t.z, t.w};
  const Fx u = fx_split(p.p + p.r), w = fx_split(p.r - p.p);
  FxAcc o = fx_acc(), x = fx_acc();
  fx_mac(o, b, w);
  fx_mac(x, a, u);
  if (decay) fx_mac(o, cj, x5);
  own += fx_val(o);
  cross -= fx_val(x);
}

__device__ __forceinline__ Fx ldb(const Fx* z, int byte_off) {
  return *reinterpret_cast<const Fx*>(reinterpret_cast<const char*>(z) + byte_off);
}

// (dt/2) O z at the lane's element: the lane's shares `own` and `cross`
// (fx_unit); the element's component c is own_c + (c ? -1 : 1) cross_{1-c}
template <int QT, bool ADJ>
__device__ __forceinline__ void fx_apply_plan(long long& own, long long& cross, const Fx* __restrict__ z,
                                              const FxPlan<QT>& pl, const int4* __restrict__ ctl) {
#pragma unroll
  for (int u = 0; u < QT; ++u)
    if (u < pl.nu) {
      const FxPR p = fx_pr(ldb(z, pl.o[u][0]), ldb(z, pl.o[u][1]), ldb(z, pl.o[u][2]), ldb(z, pl.o[u][3]),
                           pl.c[u][0], pl.c[u][1], pl.c[u][2], pl.c[u][3]);
      const bool dec = (pl.jon >> u) & 1u;
      const Fx x5 = dec ? ldb(z, pl.oj[u][ADJ]) : Fx{0, 0};
      if (ADJ)
        fx_unit_adj(own, cross, p, ctl[u], dec, pl.cj[u][ADJ], x5);
      else
        fx_unit(own, cross, p, ctl[u], dec, pl.cj[u][ADJ], x5);
    }
}

// Neighbour combinations of a subsystem for an element of the table path, z at
// the element and the lane's component, s and sN the strides in entries.  A
// neighbour outside the range has the factor 0 and is read wherever it lies:
// fx_carve leaves room for it on both sides of the iterate buffers.
__device__ __forceinline__ FxPR fx_pr_tab(const Fx* __restrict__ z, int4 ck, int4 cl, int s, int sN) {
  return fx_pr(z[2 * s], z[-2 * sN], z[-2 * s], z[2 * sN], Fx{ck.x, ck.y}, Fx{cl.x, cl.y}, Fx{ck.z, ck.w},
               Fx{cl.z, cl.w});
}
// (not inlined: the element loops call it once per element.  Everything it
// needs comes in registers, shared memory as offsets from its start: of a
// pointer the callee could not tell that it is shared memory.)
template <bool ADJ>
__device__ __noinline__ Cx fx_apply_tab(int zo, int subo, int cko, int clo, int cjo, int ctlo, int QN, uint32_t kd,
                                        uint32_t ld) {
  extern __shared__ __align__(16) unsigned char smem[];
  const Fx* const z = reinterpret_cast<const Fx*>(smem + zo);
  // QN: Q | N << 8 | bits of a digit << 24
  const int Q = QN & 0xff, N = (QN >> 8) & 0xffff, dm = (1 << (QN >> 24)) - 1;
  Cx r{0, 0};
#pragma unroll 1
  for (int q = 0; q < Q; ++q) {
    const FxSub b = *reinterpret_cast<const FxSub*>(smem + subo + q * sizeof(FxSub));
    const int sh = (b.n_sh >> 8) & 0xff, s = b.s, sN = s * N;
    const int nk = (kd >> sh) & dm, nl = (ld >> sh) & dm;
    const int4 ck = *reinterpret_cast<const int4*>(smem + cko + (b.co + nk) * sizeof(int4));
    const int4 cl = *reinterpret_cast<const int4*>(smem + clo + (b.co + nl) * sizeof(int4));
    const int4 t = *reinterpret_cast<const int4*>(smem + ctlo + q * sizeof(int4));
    const FxPR p = fx_pr_tab(z, ck, cl, s, sN);
    const bool dec = b.n_sh >> 16;
    Fx c5{0, 0}, x5{0, 0};
    if (dec) {
      c5 = *reinterpret_cast<const Fx*>(smem + cjo + (b.jo + nk * (b.n_sh & 0xff) + nl) * sizeof(Fx));
      x5 = z[ADJ ? -2 * (s + sN) : 2 * (s + sN)];
    }
    if (ADJ)
      fx_unit_adj(r.x, r.y, p, t, dec, c5, x5);
    else
      fx_unit(r.x, r.y, p, t, dec, c5, x5);
  }
  return r;
}

// ax own + s oth
__device__ __forceinline__ long long fx_cmuls(Fx ax, Fx s, long long own, long long oth) {
  FxAcc a = fx_acc();
  fx_mac(a, ax, fx_split(own));
  fx_mac(a, s, fx_split(oth));
  return fx_val(a);
}
// component c of (ax + i ay) t for t_c = own, t_{1-c} = oth; ADJ: the conjugate factor
template <bool ADJ>
__device__ __forceinline__ long long fx_cmulc(Fx ax, Fx ay, long long own, long long oth, bool im) {
  // real: ax x - ay y, imaginary: ax y + ay x
  return fx_cmuls(ax, im != ADJ ? ay : fx_neg(ay), own, oth);
}

// ---------------------------------------------------------------------------
// a state being swept: a lane's elements, scale and predictor
//
// Predictor (as in lb_device.cuh): the corrections of the previous steps in
// the frame that turns with each element's free evolution, c~_j = conj(p_j)
// c_j with p_j = u^m, u the unit-modulus part of g, are extrapolated by the
// polynomial through the last n of them.  |u| = 1 to 2^-60, so the frame never
// needs a new anchor.  Integer sums make the extrapolation exact.

template <int QT>
struct FxPred {
  long long d[kFxOrder];  // backward differences of the corrections (in the frame)
  long long s;            // their sum over the valid ones: the prediction in the frame
  Cx p, u;
};
template <>
struct FxPred<0> {
  long long* ring;  // [kRingOrder] slots of this state's V entries (two components each), `stride` apart
  Cx* ph;           // [V] p
  Cx* fu;           // [V] u
  size_t stride;
};

template <int E, int QT>
struct FxState {
  int v[1], m[1];          // QT > 0: vec index (V: none) and mirror (-1: none)
  uint32_t kd[E], ld[E];   // QT == 0: packed digits
  FxPlan<QT> pl;
  Fx dx, dy;               // QT > 0: (I - dt/2 D)^-1 - 1, its imaginary part negated in the real lane
  bool im;                 // the lane's component
  long long q[E];          // right-hand side of the step (q^j, or the adjoint's qhat^{j+1}), its component
  int sc;                  // its scale: X = x 2^sc
  FxPred<QT> pr;
  int n, slot, cap;        // corrections recorded, ring position, highest order
  bool frame;              // turn the frame (else the phases are too small to matter)
};

template <int E, int QT>
__device__ __forceinline__ int fx_u(int e) {
  return (int)(threadIdx.x >> 1) + e * (int)(blockDim.x >> 1);
}
template <int E, int QT>
__device__ __forceinline__ int fx_v(const FxState<E, QT>& st, const FxSmem& S, const Hdr& H, int e) {
  if constexpr (QT > 0) {
    return st.v[0];
  } else {
    const int u = fx_u<E, QT>(e);
    if (!H.herm) return u;
    return u < H.Vh ? (int)S.hmap[u] : H.V;
  }
}
template <int E, int QT>
__device__ __forceinline__ int fx_m(const FxState<E, QT>& st, const FxSmem& S, const Hdr& H, int e) {
  if constexpr (QT > 0) {
    return st.m[0];
  } else {
    const int u = fx_u<E, QT>(e);
    if (!H.herm || u >= H.Vh) return -1;
    const int mm = S.hmir[u];
    return mm == 0xffff ? -1 : mm;
  }
}

// write the lane's component of an iterate entry and, under the Hermitian
// symmetry, of its mirror's conjugate
__device__ __forceinline__ void fx_put(Fx* z, int v, int m, bool im, long long x) {
  z[2 * v + im] = fx_split(x);
  if (m >= 0) z[2 * m + im] = fx_split(im ? -x : x);
}
// the same for a state in FP64 (scale sc)
__device__ __forceinline__ void fx_put_d(double2* a, int v, int m, bool im, long long x, int sc) {
  double* d = reinterpret_cast<double*>(a);
  const double y = fx_to(x, sc);
  d[2 * (size_t)v + im] = y;
  if (m >= 0) d[2 * (size_t)m + im] = im ? -y : y;
}

template <int E, int QT>
__device__ __forceinline__ void fx_init(FxState<E, QT>& st, const FxSmem& S, const ProbDev& P) {
  const Hdr& H = *S.hdr;
  const double hh = 0.5 * H.h;
  st.cap = QT > 0 ? min(P.pred_order, kFxOrder) : P.pred_order;
  st.n = st.slot = 0;
  st.frame = P.fxframe != 0;
  st.im = threadIdx.x & 1;
  if constexpr (QT > 0) {
    const int u = fx_u<E, QT>(0);
    const int v = H.herm ? (u < H.Vh ? (int)S.hmap[u] : H.V) : u;
    st.v[0] = v < H.V ? v : H.V;
    const int mm = H.herm && u < H.Vh ? (int)S.hmir[u] : 0xffff;
    st.m[0] = mm == 0xffff ? -1 : mm;
    fx_plan<QT>(st.pl, S, P, st.v[0]);
    const int4 d = v < H.V ? fx_dinv1(P.D[v], hh) : make_int4(0, 0, 0, 0);
    st.dx = Fx{d.x, d.y};
    st.dy = st.im ? Fx{d.z, d.w} : fx_neg(Fx{d.z, d.w});
    st.pr.u = v < H.V ? fx_frame(P.D[v], hh) : Cx{kFxPhase1, 0};
    st.pr.p = Cx{kFxPhase1, 0};
    st.pr.s = 0;
#pragma unroll
    for (int k = 0; k < kFxOrder; ++k) st.pr.d[k] = 0;
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int v = fx_v(st, S, H, e);
      st.kd[e] = v < H.V ? S.dig[v % H.N] : 0u;
      st.ld[e] = v < H.V ? S.dig[v / H.N] : 0u;
      if (v < H.V && !st.im) S.dsm[fx_u<E, QT>(e)] = fx_dinv1(P.D[v], hh);
    }
    __syncthreads();
  }
}
// the predictor's ring of this launch (QT == 0) in `ring`, `ph`, `fu` of the workspace
template <int E, int QT>
__device__ __forceinline__ void fx_ring(FxState<E, QT>& st, const FxSmem& S, const ProbDev& P, double2* ring, double2* ph, double2* fu,
                        size_t base) {
  if constexpr (QT == 0) {
    st.pr.ring = reinterpret_cast<long long*>(ring + base);
    st.pr.ph = reinterpret_cast<Cx*>(ph + base);
    st.pr.fu = reinterpret_cast<Cx*>(fu + base);
    st.pr.stride = 2 * (size_t)P.M * P.V;
    const Hdr& H = *S.hdr;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int v = fx_v(st, S, H, e);
      if (v < H.V && !st.im) st.pr.fu[v] = fx_frame(P.D[v], 0.5 * H.h);
    }
    __syncthreads();
  }
}

// Load this state's elements from FP64 values, setting the scale; returns
// false on NaN or Inf.
template <int E, int QT, class F>
__device__ __forceinline__ bool fx_load(FxState<E, QT>& st, const FxSmem& S, F&& val) {
  const Hdr& H = *S.hdr;
  unsigned long long mx = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int v = fx_v(st, S, H, e);
    if (v < H.V) {
      const double2 x = val(v);
      mx = umax64(mx, umax64(abs_bits(x.x), abs_bits(x.y)));
    }
  }
  mx = fx_cta_max(S, mx);
  if (mx >= kInfBits) return false;
  st.sc = fx_scale(mx);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int v = fx_v(st, S, H, e);
    st.q[e] = 0;
    if (v < H.V) {
      const double2 x = val(v);
      st.q[e] = fx_from(st.im ? x.y : x.x, st.sc);
    }
  }
  return true;
}

// Load this state's elements from a chunk boundary (fixed point, with its scale).
template <int E, int QT>
__device__ __forceinline__ void fx_load_fixed(FxState<E, QT>& st, const FxSmem& S, const longlong2* x, int sc) {
  const Hdr& H = *S.hdr;
  st.sc = sc;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int v = fx_v(st, S, H, e);
    st.q[e] = v < H.V ? reinterpret_cast<const long long*>(x)[2 * v + st.im] : 0;
  }
}
// a step that did not converge: the first error of the sweep, or of a chunk
// (chunks run at the same time: the earliest step counts)
__device__ __forceinline__ void fx_fail(DevStatus* st, int j, bool chunked) {
  if (threadIdx.x) return;
  if (chunked)
    atomicMax(&st->late, 0x7fffffff - j);
  else
    record_error(st, LB_ENOTCONV, j);
}

// an adjoint state that a source before step j made infinite; chunks run at the
// same time: the latest step, which a step-by-step sweep meets first, counts
__device__ __forceinline__ void fx_overflow(DevStatus* st, int j, bool chunked) {
  if (threadIdx.x) return;
  if (!chunked)
    record_error(st, LB_ENAN, j);
  else if (const int c = atomicCAS(&st->code, 0, LB_ENAN); c == 0 || c == LB_ENAN)
    atomicMax(&st->step, j);
}

// steps of a launch so far (they select buffers)
struct FxCount {
  unsigned step = 0;
};

// the control row of step j into the step's buffer (all threads; visible after the next barrier)
__device__ __forceinline__ void fx_ctl(const FxSmem& S, const ProbDev& P, int cq, int j, unsigned step) {
  if ((int)threadIdx.x <= cq) S.ctl[(step & 1) * (cq + 1) + threadIdx.x] = P.ctabx[(size_t)j * (cq + 1) + threadIdx.x];
}

// the prediction in the frame from the n newest entries of a ring (QT == 0), one component
__device__ __noinline__ long long fx_ring_sum(const long long* __restrict__ ring, size_t stride, int slot, int n) {
  // sums of the weights times the entries' halves (|w| <= 252: no overflow)
  long long hi = 0, lo = 0;
  int sl = slot - 1;
  auto term = [&](int i) {
    if (sl < 0) sl += kRingOrder;
    const Fx c = fx_split(ring[(size_t)sl * stride]);
    const int w = kExtrapI[n][i];
    hi = fx_madw(w, c.h, hi);
    lo = fx_madw(w, c.l, lo);
    --sl;
  };
  if (n == kDefaultRingOrder) {
#pragma unroll
    for (int i = 0; i < kDefaultRingOrder; ++i) term(i);
  } else {
    for (int i = 0; i < n; ++i) term(i);
  }
  return (long long)((unsigned long long)hi << 32) + lo;
}

// One implicit-midpoint solve (I - dt/2 M) z = q (ADJ: M^+) of the CTA's
// state, with the predicted first iterate when `pred`.  Returns the
// iteration count, or -1 (max_iter, or a control factor out of this
// arithmetic's range: the caller changed the controls of a captured launch); z
// is left in the iterate buffer `cur` and, per lane, in zr (QT > 0), the last
// iteration's correction in cr (QT > 0) or the predictor's ring, and the
// state's largest magnitude (high word) in qtop.
// The first iterate goes to the buffer the solve before did not leave its z
// in, so that threads may still read that z until the next barrier.
// jnext: the step after this one (< 0: none), whose control row is fetched.
template <int E, int QT, bool ADJ>
__device__ __forceinline__ int fx_solve(FxState<E, QT>& st, const FxSmem& S, const ProbDev& P, int jnext, bool pred, FxCount& cnt,
                        int& cur, unsigned& qtop, long long& zr, long long& cr) {
  const Hdr& H = *S.hdr;
  const int V = H.V, cq = H.cq, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int4* ctl = S.ctl + (cnt.step & 1) * (cq + 1);
  unsigned* qs = S.slots + 64 * (cnt.step & 1);
  ++cnt.step;
  if (jnext >= 0) fx_ctl(S, P, cq, jnext, cnt.step);
  const int maxit = H.max_iter, qn = H.Q | H.N << 8 | H.db << 24;
  const bool im = st.im;
  unsigned qm = 0;
  if constexpr (QT > 0) {
    const long long q = st.q[0];
    qm = st.v[0] < V ? fx_hi_abs(q) : 0u;
    long long t = q;
    if (pred) {
      if (st.n == 0) {
        st.pr.p = Cx{kFxPhase1, 0};
        st.pr.s = 0;
      } else if (st.frame) {
        t += fx_cmulc<ADJ>(fx_coef(st.pr.p.x), fx_coef(st.pr.p.y), st.pr.s, fx_other(st.pr.s), im) << 2;
      } else {
        t += st.pr.s;
      }
    }
    zr = t + fx_cmuls(st.dx, ADJ ? fx_neg(st.dy) : st.dy, t, fx_other(t));
    if (st.v[0] < V) fx_put(cur ? S.zb0 : S.zb1, st.v[0], st.m[0], im, zr);
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int v = fx_v(st, S, H, e);
      // both lanes of a pair have an element or neither has
      const bool ok = v < V;
      long long t = st.q[e];
      int4 d = make_int4(0, 0, 0, 0);
      long long s = 0;
      Cx p{0, 0};
      if (ok) {
        qm = max(qm, fx_hi_abs(t));
        d = S.dsm[fx_u<E, QT>(e)];
        if (pred) {
          if (st.n == 0) {
            if (!im) st.pr.ph[v] = Cx{kFxPhase1, 0};
          } else {
            s = fx_ring_sum(st.pr.ring + 2 * v + im, st.pr.stride, st.slot, st.n);
            if (st.frame) p = st.pr.ph[v];
          }
        }
      }
      if (pred && st.frame && st.n > 0)
        s = fx_cmulc<ADJ>(fx_coef(p.x), fx_coef(p.y), s, fx_other(s), im) << 2;
      t += s;
      t += fx_cmulc<ADJ>(Fx{d.x, d.y}, Fx{d.z, d.w}, t, fx_other(t), im);
      if (ok) fx_put(cur ? S.zb0 : S.zb1, v, fx_m(st, S, H, e), im, t);
    }
  }
  cur ^= 1;
  qm = __reduce_max_sync(kFull, qm);
  if (lane == 0) qs[warp] = qm;
  __syncthreads();
  qtop = fx_slots_max(qs, nwarps);
  const int4 last = ctl[cq];
  if (last.y != 0) return -1;
  const unsigned thr = fx_stop(__int_as_float(last.x), qtop);
  for (int it = 0; it < maxit; ++it) {
    const Fx* __restrict__ zc = cur ? S.zb1 : S.zb0;
    Fx* __restrict__ zn = cur ? S.zb0 : S.zb1;
    const int zo = S.off(zc), ctlo = S.off(ctl);
    unsigned* ds = S.slots + 64 * (it & 1) + 32;
    unsigned dm = 0;
    if constexpr (QT > 0) {
      long long own = 0, cross = 0;
      fx_apply_plan<QT, ADJ>(own, cross, zc, st.pl, ctl);
      // both components of q + c in both lanes, from one exchange
      const long long t0 = st.q[0] + own, to = fx_other(t0), xo = fx_other(cross);
      const long long t = im ? t0 - xo : t0 + xo, o = im ? to + cross : to - cross;
      cr = t - st.q[0];
      const long long z = t + fx_cmuls(st.dx, ADJ ? fx_neg(st.dy) : st.dy, t, o);
      if (st.v[0] < V) {
        fx_put(zn, st.v[0], st.m[0], im, z);
        dm = fx_abs_sat(z - zr);
      }
      zr = z;
    } else {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int v = fx_v(st, S, H, e);
        const bool ok = v < V;
        Cx r{0, 0};
        int4 d = make_int4(0, 0, 0, 0);
        Cx p{0, 0};
        if (ok) {
          r = fx_apply_tab<ADJ>(zo + (2 * v + im) * (int)sizeof(Fx), S.off(S.sub), S.off(S.ck), S.off(S.cl),
                                S.off(ADJ ? S.ja : S.jf), ctlo, qn, st.kd[e], st.ld[e]);
          d = S.dsm[fx_u<E, QT>(e)];
          if (pred && st.frame) p = st.pr.ph[v];
        }
        const long long t0 = st.q[e] + r.x, to = fx_other(t0), xo = fx_other(r.y);
        const long long t = im ? t0 - xo : t0 + xo, o = im ? to + r.y : to - r.y;
        const long long z = t + fx_cmulc<ADJ>(Fx{d.x, d.y}, Fx{d.z, d.w}, t, o, im);
        if (pred) {
          // the correction in the frame, to the ring slot of this step
          long long c = t - st.q[e];
          if (st.frame) c = fx_cmulc<!ADJ>(fx_coef(p.x), fx_coef(p.y), c << 2, fx_other(c) << 2, im);
          if (ok) st.pr.ring[(size_t)st.slot * st.pr.stride + 2 * v + im] = c;
        }
        if (ok) {
          dm = max(dm, fx_abs_sat(z - fx_join(zc[2 * v + im])));
          fx_put(zn, v, fx_m(st, S, H, e), im, z);
        }
      }
    }
    dm = __reduce_max_sync(kFull, dm);
    if (lane == 0) ds[warp] = dm;
    __syncthreads();
    dm = fx_slots_max(ds, nwarps);
    cur ^= 1;
    if (dm <= thr) return it + 1;
  }
  return -1;
}

// After a converged step: record its correction (cr, QT > 0), turn the frame
// one step on.
template <int E, int QT, bool ADJ>
__device__ __forceinline__ void fx_commit(FxState<E, QT>& st, const FxSmem& S, long long cr) {
  const Hdr& H = *S.hdr;
  if constexpr (QT > 0) {
    long long c = cr;
    if (st.frame) {
      c = fx_cmulc<!ADJ>(fx_coef(st.pr.p.x), fx_coef(st.pr.p.y), cr << 2, fx_other(cr) << 2, st.im);
      // p <- p u (both quarters: the product is a sixteenth)
      const Cx w = fx_cmul(fx_coef(st.pr.u.x), fx_coef(st.pr.u.y), st.pr.p);
      st.pr.p = Cx{w.x << 2, w.y << 2};
    }
    // the newest difference of order n is the prediction's error; the lower
    // ones follow by adding it up
    long long a = c - st.pr.s, s = 0;
    const int n = st.n;
    if (n == kFxOrder) {
#pragma unroll
      for (int k = kFxOrder - 1; k >= 0; --k) {
        a += st.pr.d[k];
        st.pr.d[k] = a;
        s += a;
      }
    } else {
      const long long top = a;
#pragma unroll
      for (int k = kFxOrder - 1; k >= 0; --k) {
        if (k < n) {
          a += st.pr.d[k];
          st.pr.d[k] = a;
          s += a;
        } else if (k == n && n < st.cap) {
          st.pr.d[k] = top;
          s += top;
        }
      }
    }
    st.pr.s = s;
  } else if (st.frame) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int v = fx_v(st, S, H, e);
      if (v < H.V && !st.im) {
        const Cx u = st.pr.fu[v];
        const Cx w = fx_cmul(fx_coef(u.x), fx_coef(u.y), st.pr.ph[v]);
        st.pr.ph[v] = Cx{w.x << 2, w.y << 2};
      }
    }
    __syncwarp();
  }
  st.n = st.n < st.cap ? st.n + 1 : st.cap;
  st.slot = st.slot + 1 < kRingOrder ? st.slot + 1 : 0;
}

// scale the state (and its predictor) by 2^-s
template <int E, int QT>
__device__ __forceinline__ void fx_scale_by(FxState<E, QT>& st, const FxSmem& S, int s, bool pred) {
  const Hdr& H = *S.hdr;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    st.q[e] = fx_shift(st.q[e], s);
    if constexpr (QT == 0) {
      const int v = fx_v(st, S, H, e);
      if (pred && v < H.V) {
        int sl = st.slot - 1;
        for (int i = 0; i < st.n; ++i) {
          if (sl < 0) sl += kRingOrder;
          long long* c = st.pr.ring + (size_t)sl * st.pr.stride + 2 * v + st.im;
          *c = fx_shift(*c, s);
          --sl;
        }
      }
    }
  }
  if constexpr (QT > 0) {
    long long sum = 0;
#pragma unroll
    for (int k = 0; k < kFxOrder; ++k)
      if (k < st.n) {
        st.pr.d[k] = fx_shift(st.pr.d[k], s);
        sum += st.pr.d[k];
      }
    st.pr.s = sum;
  }
  st.sc -= s;
}
// Keep the state's largest entry in [2^58.5, 2^60): called between steps with
// the last right-hand side's largest magnitude (uniform over the CTA).
template <int E, int QT>
__device__ __forceinline__ void fx_rescale(FxState<E, QT>& st, const FxSmem& S, unsigned qtop, bool pred) {
  const int s = fx_rescale_shift(qtop);
  if (s) fx_scale_by(st, S, s, pred);
}
// q += src (FP64, each lane's component): the scale first follows the largest
// of state, source and sum, which a source may raise by any factor in one step
// (of the sum alone it would shift a state that the source cancels past 64
// bits) (all threads).  False when state or source is not finite.
template <int E, int QT>
__device__ __forceinline__ bool fx_add_source(FxState<E, QT>& st, const FxSmem& S, const double (&src)[E], bool pred) {
  unsigned long long mx = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const double x = fx_to(st.q[e], st.sc);
    mx = umax64(mx, umax64(abs_bits(x + src[e]), umax64(abs_bits(x), abs_bits(src[e]))));
  }
  mx = fx_cta_max(S, mx);
  if (mx >= kInfBits) return false;
  const int sc = fx_scale(mx);
  if (mx && (sc < st.sc || sc > st.sc + 1)) fx_scale_by(st, S, st.sc - sc, pred);
#pragma unroll
  for (int e = 0; e < E; ++e) st.q[e] += fx_from(src[e], st.sc);
  return true;
}

// q <- 2 z - q for the lane's elements, z from the solve (zr for QT > 0); the
// stage vector's component also to tp[2 v + component] when given
template <int E, int QT>
__device__ __forceinline__ void fx_update(FxState<E, QT>& st, const FxSmem& S, const Fx* z, long long zr,
                                          long long* tp) {
  const Hdr& H = *S.hdr;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int v = fx_v(st, S, H, e);
    if (v < H.V) {
      const long long x = QT > 0 ? zr : fx_join(z[2 * v + st.im]);
      if (tp) tp[2 * v + st.im] = x;
      st.q[e] = 2 * x - st.q[e];
    }
  }
}

// deterministic CTA sum of one double per thread, to every thread
__device__ __forceinline__ double fx_cta_sum(const FxSmem& S, double x) {
  double* w = reinterpret_cast<double*>(S.mx);
  x = warp_sum(x);
  if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = x;
  __syncthreads();
  double t = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += w[i];
  __syncthreads();
  return t;
}

// one component's share of the merit summand
__device__ __forceinline__ double fx_merit(int kind, double q, double t) {
  if (kind == LB_J_FROB) return (q - t) * (q - t);
  return t * q;
}

}  // namespace
}  // namespace lbk
