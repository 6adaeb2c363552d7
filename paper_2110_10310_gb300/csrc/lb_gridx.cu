// Grid-wide cooperative sweeps in fixed point (lb_fixed.cuh), and their
// launchers: the large states of lb_grid.cu with the operator product, the
// step and the predictor on the integer pipe.
//
// The FP64 sweeps are bound by the FP64 pipe: one operator product of six
// subsystems takes 114 FP64 instructions of 67 cycles per warp.  Here the
// same product takes 36 (42 with decay) IMAD.WIDE of 2 cycles per subsystem,
// and what remains is the memory traffic of the step: the predictor's ring,
// the iterates and the neighbours.  Every state buffer holds 64-bit integers
// with one power of two per state; the iterates and the ring hold them split
// (lb_fixed.cuh) so that neighbours and ring entries are multiplied as loaded.
//
// A step: one pass that commits the step before (q <- 2 z - q, the recorded
// correction turned into the predictor's frame) and forms the next first
// iterate, a grid barrier, then one pass and barrier per inner iteration.  The
// correction is not stored by the iteration: c = (I - dt/2 D) z - q recovers it
// to the rounding of z.

#include <algorithm>
#include <type_traits>

#include "lb_grid.cuh"
#include "lb_fixed.cuh"

namespace lbk {

namespace {

static_assert(kRingOrder == 10, "kExtrapI is written for order 10");
constexpr int kGxWarps = kGridThreads / 32;
constexpr int kGxBlocks = 2;  // blocks per SM
constexpr int kApplyBlocks = 3;  // ... of the product alone, and of its launch (12 per SM: their table set-ups took 3%)

// kernel parameter: what the element loops need of the system, in the
// constant bank (the subsystem loop is unrolled for QN > 0)
struct GxSub {
  int n, s, sh, co, jo, decay;
  int t1, t2;  // s (s + 1)/2, s (s - 1)/2
};
struct GxParams {
  GxSub sub[LB_MAXQ];
  int Q, dm;
};

struct GxSmem {
  GridHdr* g;
  int4* cc;       // [ncoef] ladder factors (cu, cd), 2^-kc
  Fx* jf;         // [njcoef]
  Fx* ja;
  int4* ctl;      // [LB_MAXQ] this solve's control factors (a, b), negated for the adjoint
  unsigned* red;  // [4][kGxWarps]
  longlong2* gs;  // [kGxQP][4][kGxWarps] the warps' gradient sums
  int* flag;      // [0] decision, [1] stopping factor (float bits)
  int* sc;        // [M] scale of each state
  int* sh;        // [M] the commit's change of it
  unsigned long long* due;  // arrivals that end the last barrier
  int* passed;              // ... and whether it did
};

__host__ __device__ inline size_t gx_smem_bytes(int ncoef, int njcoef, int M) {
  return align16(sizeof(GridHdr)) + sizeof(int4) * ncoef + 2 * align16(sizeof(Fx) * njcoef) + sizeof(int4) * LB_MAXQ +
         align16(sizeof(unsigned) * 4 * kGxWarps) + sizeof(longlong2) * 12 * kGxWarps + 32 + 2 * align16(sizeof(int) * M);
}

// M: the states whose scales it keeps (none in the product alone)
__device__ GxSmem gx_setup(unsigned char* base, const ProbDev& P, int nstates, int herm, int M) {
  GxSmem S;
  size_t o = 0;
  auto take = [&](size_t b) {
    unsigned char* p = base + o;
    o += align16(b);
    return p;
  };
  S.g = reinterpret_cast<GridHdr*>(take(sizeof(GridHdr)));
  S.cc = reinterpret_cast<int4*>(take(sizeof(int4) * P.ncoef));
  S.jf = reinterpret_cast<Fx*>(take(sizeof(Fx) * P.njcoef));
  S.ja = reinterpret_cast<Fx*>(take(sizeof(Fx) * P.njcoef));
  S.ctl = reinterpret_cast<int4*>(take(sizeof(int4) * LB_MAXQ));
  S.red = reinterpret_cast<unsigned*>(take(sizeof(unsigned) * 4 * kGxWarps));
  S.gs = reinterpret_cast<longlong2*>(take(sizeof(longlong2) * 12 * kGxWarps));
  S.flag = reinterpret_cast<int*>(take(16));
  S.due = reinterpret_cast<unsigned long long*>(take(16));
  S.passed = reinterpret_cast<int*>(S.due + 1);
  S.sc = reinterpret_cast<int*>(take(sizeof(int) * M));
  S.sh = reinterpret_cast<int*>(take(sizeof(int) * M));
  if (threadIdx.x == 0) {
    *S.due = 0;
    load_hdr(S.g->h, P);
    S.g->M = nstates;
    S.g->herm = herm;
    S.g->Vh = herm ? P.N * (P.N + 1) / 2 : P.V;
    S.g->total = (long long)nstates * S.g->Vh;
    const long long per = (S.g->total + gridDim.x - 1) / gridDim.x;
    S.g->chunk = (per + 31) / 32 * 32;  // whole warps
  }
  for (int i = threadIdx.x; i < P.ncoef; i += blockDim.x) {
    int q = 0;
    while (q + 1 < P.Q && P.coff[q + 1] <= i) ++q;
    const Fx u = fx_coef(__double2ll_rn(scalbn(P.cu[i], 64 - P.kc[q])));
    const Fx d = fx_coef(__double2ll_rn(scalbn(P.cd[i], 64 - P.kc[q])));
    S.cc[i] = make_int4(u.h, u.l, d.h, d.l);
  }
  // (the product alone scales its own decay factors)
  for (int i = threadIdx.x; M && i < P.njcoef; i += blockDim.x) {
    S.jf[i] = fx_coef(__double2ll_rn(scalbn(P.jf[i], 64)));
    S.ja[i] = fx_coef(__double2ll_rn(scalbn(P.ja[i], 64)));
  }
  for (int i = threadIdx.x; i < M; i += blockDim.x) S.sc[i] = S.sh[i] = 0;
  __syncthreads();
  return S;
}

// Grid barrier with a bounded wait, as grid_sync (lb_grid.cuh) in fewer round
// trips to L2: one counter that only grows (zeroed before the launch), so an
// arrival is one atomic whose value already ends the wait of the last block,
// and a poll is one load with nothing between two of them.  (grid_sync reads the
// generation, resets the count, reads the error word beside every poll and
// sleeps: one state of 3240 elements, 1000 steps forward and back, 36.0 ms with it,
// 30.5 with this one; three states of vec 65536, 400 steps, 35.3 and 31.0 ms.)
// The top bit is set by a wait that gave up; the counter is short of the
// barrier's arrivals then, so no block that looks later passes it.
constexpr unsigned long long kGxGaveUp = 1ull << 63;
__device__ __forceinline__ bool gx_sync(const GxSmem& S, GridBar* bar, long long limit) {
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long due = *S.due + gridDim.x;
    *S.due = due;
    __threadfence();
    unsigned long long v = atomicAdd(&bar->arrived, 1ull) + 1;
    long long spins = 0;
    while (v < due) {
      if (++spins > limit) v = atomicOr(&bar->arrived, kGxGaveUp) | kGxGaveUp;
      else v = *(volatile unsigned long long*)&bar->arrived;
    }
    __threadfence();
    *S.passed = v < kGxGaveUp;
  }
  __syncthreads();
  return *S.passed != 0;
}

__device__ __forceinline__ int4 gx_pack(Cx z) {
  const Fx a = fx_split(z.x), b = fx_split(z.y);
  return make_int4(a.h, a.l, b.h, b.l);
}
__device__ __forceinline__ Cx gx_join(int4 p) {
  return Cx{fx_join(Fx{p.x, p.y}), fx_join(Fx{p.z, p.w})};
}
__device__ __forceinline__ Cx gx_ld(const double2* p) {
  const longlong2 a = *reinterpret_cast<const longlong2*>(p);
  return Cx{a.x, a.y};
}
__device__ __forceinline__ void gx_st(double2* p, Cx x) { *reinterpret_cast<longlong2*>(p) = make_longlong2(x.x, x.y); }
__device__ __forceinline__ Fx gx_re(int4 a) { return Fx{a.x, a.y}; }
__device__ __forceinline__ Fx gx_im(int4 a) { return Fx{a.z, a.w}; }

// Per-state maxima over a block's chunk, of 32-bit magnitudes (as StateMax of
// lb_grid.cu): in registers when the chunk covers at most 4 states.
struct GxMax {
  int sb0, ns, bcur;
  bool local;
  unsigned m[4], mcur;
  __device__ void init(long long e0, long long e1, int V) {
    sb0 = (int)(e0 / V);
    const int sb1 = e1 > e0 ? (int)((e1 - 1) / V) : sb0;
    ns = sb1 - sb0 + 1;
    local = ns <= 4;
    m[0] = m[1] = m[2] = m[3] = 0;
    bcur = -1;
    mcur = 0;
  }
  __device__ __forceinline__ void add(int b, unsigned x, unsigned* slots) {
    if (local) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k == b - sb0) m[k] = max(m[k], x);
    } else {
      if (b != bcur) {
        if (bcur >= 0 && mcur) atomicMax(slots + bcur, mcur);
        bcur = b;
        mcur = 0;
      }
      mcur = max(mcur, x);
    }
  }
  __device__ void push(unsigned* slots, unsigned* red) {
    if (local) {
      const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k < ns) {
          const unsigned v = __reduce_max_sync(kFull, m[k]);
          if (lane == 0) red[k * kGxWarps + warp] = v;
        }
      __syncthreads();
      if ((int)threadIdx.x < ns) {
        unsigned r = 0;
        for (int w = 0; w < kGxWarps; ++w) r = max(r, red[threadIdx.x * kGxWarps + w]);
        if (r) atomicMax(slots + sb0 + threadIdx.x, r);
      }
      __syncthreads();
    } else if (bcur >= 0 && mcur) {
      atomicMax(slots + bcur, mcur);
    }
  }
};

// Neighbours of element (k, l) for one subsystem, as offsets into the state's
// slab.  Packed (k <= l): the row neighbour above and the column neighbour
// before can lie below the diagonal, both exactly when l - k < s; they are read
// at their mirrors and conjugated (mir).
struct GxNb {
  int o1, o2, o3, o4;
  bool mir;
};
template <bool PK>
__device__ __forceinline__ GxNb gx_nb(const GxSub& b, int i, int k, int l, int N, int nk, int nl) {
  GxNb r;
  if constexpr (PK) {
    const int sl = b.s * l;
    r.mir = l - k < b.s;
    r.o1 = r.mir ? (((k + b.s) * (k + b.s + 1)) >> 1) + l : i + b.s;
    r.o2 = r.mir ? ((k * (k + 1)) >> 1) + l - b.s : i - sl + b.t2;
    r.o3 = i - b.s;
    r.o4 = i + sl + b.t1;
  } else {
    r.mir = false;
    r.o1 = i + b.s;
    r.o2 = i - b.s * N;
    r.o3 = i - b.s;
    r.o4 = i + b.s * N;
  }
  // outside the range (factor 0): the element itself
  if (nk + 1 >= b.n) r.o1 = i;
  if (nl == 0) r.o2 = i;
  if (nk == 0) r.o3 = i;
  if (nl + 1 >= b.n) r.o4 = i;
  return r;
}
struct GxPR {
  long long pr, pi, rr, ri;
};
template <bool PK>
__device__ __forceinline__ GxPR gx_pr(const int4* __restrict__ z, const GxSub& b, const int4* __restrict__ cc, int i,
                                      int k, int l, int N, int nk, int nl) {
  const GxNb n = gx_nb<PK>(b, i, k, l, N, nk, nl);
  const int4 x1 = z[n.o1], x2 = z[n.o2], x3 = z[n.o3], x4 = z[n.o4];
  const int4 ck = cc[b.co + nk], cl = cc[b.co + nl];
  const Fx c1{ck.x, ck.y}, c2 = fx_neg(Fx{cl.z, cl.w}), c3{ck.z, ck.w}, c4 = fx_neg(Fx{cl.x, cl.y});
  const Fx c1i = PK && n.mir ? fx_neg(c1) : c1, c2i = PK && n.mir ? fx_neg(c2) : c2;
  FxAcc pr{0, 0}, pi{0, 0}, rr{0, 0}, ri{0, 0};
  fx_mac(pr, c1, gx_re(x1));
  fx_mac(pr, c2, gx_re(x2));
  fx_mac(pi, c1i, gx_im(x1));
  fx_mac(pi, c2i, gx_im(x2));
  fx_mac(rr, c3, gx_re(x3));
  fx_mac(rr, c4, gx_re(x4));
  fx_mac(ri, c3, gx_im(x3));
  fx_mac(ri, c4, gx_im(x4));
  return GxPR{fx_val(pr), fx_val(pi), fx_val(rr), fx_val(ri)};
}

// (dt/2) O z at an element (the sums of offdiag_acc): b (P - R) - i a (P + R)
// per subsystem, plus the decay sandwich
template <bool ADJ, bool PK, int QN>
__device__ __forceinline__ Cx gx_apply(const int4* __restrict__ z, const GxParams& gp, const GxSmem& S, int i, int k,
                                       int l, int N, uint32_t kd, uint32_t ld) {
  Cx r{0, 0};
  auto sub = [&](int q) {
    const GxSub& b = gp.sub[q];
    const int nk = (kd >> b.sh) & gp.dm, nl = (ld >> b.sh) & gp.dm;
    const GxPR p = gx_pr<PK>(z, b, S.cc, i, k, l, N, nk, nl);
    const int4 t = S.ctl[q];
    const Fx a{t.x, t.y}, bb{t.z, t.w};
    const Fx ux = fx_split(p.pr + p.rr), uy = fx_split(p.pi + p.ri);
    const Fx wx = fx_split(p.pr - p.rr), wy = fx_split(p.pi - p.ri);
    Fx cj{0, 0};
    int4 x5 = make_int4(0, 0, 0, 0);
    if (b.decay) {
      const int jo = b.jo + nk * b.n + nl;
      int o;
      if (!ADJ) {
        cj = S.jf[jo];
        o = PK ? i + b.s * l + b.t1 + b.s : i + b.s + b.s * N;
        if (nk + 1 >= b.n || nl + 1 >= b.n) o = i;
      } else {
        cj = S.ja[jo];
        o = PK ? i - b.s * l + b.t2 - b.s : i - b.s - b.s * N;
        if (nk == 0 || nl == 0) o = i;
      }
      x5 = z[o];
    }
    FxAcc cr = fx_acc(), ci = fx_acc();
    fx_mac(cr, bb, wx);
    fx_mac(cr, a, uy);
    fx_mac(ci, bb, wy);
    fx_mac(ci, fx_neg(a), ux);
    if (b.decay) {
      fx_mac(cr, cj, gx_re(x5));
      fx_mac(ci, cj, gx_im(x5));
    }
    r.x += fx_val(cr);
    r.y += fx_val(ci);
  };
  if constexpr (QN > 0) {
#pragma unroll
    for (int q = 0; q < QN; ++q) sub(q);
  } else {
    for (int q = 0; q < gp.Q; ++q) sub(q);
  }
  return r;
}

// t + A t, A = (I - dt/2 D)^-1 - 1 (ADJ: its conjugate)
template <bool ADJ>
__device__ __forceinline__ Cx gx_dinv(int4 d, Cx t) {
  const Fx ay{d.z, d.w};
  const Cx a = fx_cmul(Fx{d.x, d.y}, ADJ ? fx_neg(ay) : ay, t);
  return Cx{t.x + a.x, t.y + a.y};
}

// the sweep's position: predictor ring and iterate buffers
struct GxHist {
  int4* ring = nullptr;   // [kRingOrder][M Vh]
  double2* ph = nullptr;  // [M Vh] p
  int n = 0, slot = 0, cap = kRingOrder;
  __device__ void advance() {
    n = n < cap ? n + 1 : cap;
    slot = slot + 1 < kRingOrder ? slot + 1 : 0;
  }
};

// one inner iteration over a block's chunk: zn from zc, the per-state maxima of the change
template <bool ADJ, bool PK, int QN>
__device__ __forceinline__ void gx_pass(const ProbDev& P, const GxParams& gp, const GxSmem& S, long long e0,
                                        long long e1, const double2* __restrict__ rhs, const int4* __restrict__ zc,
                                        int4* __restrict__ zn, unsigned* bank) {
  const GridHdr& G = *S.g;
  const int N = G.h.N;
  GxMax sm;
  sm.init(e0, e1, G.Vh);
  for (GIter it_(G, e0 + threadIdx.x); it_.e < e1; it_.next(G, blockDim.x)) {
    const GEl g = gel_at(G, P.hkl, it_.b, it_.i);
    const size_t base = (size_t)g.b * G.Vh, o = base + g.i;
    const uint32_t kd = __ldg(P.digits + g.k), ld = __ldg(P.digits + g.l);
    const Cx c = gx_apply<ADJ, PK, QN>(zc + base, gp, S, g.i, g.k, g.l, N, kd, ld);
    const Cx q = gx_ld(rhs + o);
    const Cx zo = gx_join(zc[o]);
    const Cx z = gx_dinv<ADJ>(__ldg(P.fxd + g.v), Cx{q.x + c.x, q.y + c.y});
    zn[o] = gx_pack(z);
    sm.add(g.b, max(fx_abs_sat(z.x - zo.x), fx_abs_sat(z.y - zo.y)), bank);
  }
  sm.push(bank, S.red);
}

// The first pass of a solve for one element: z_0 = (I - dt/2 D)^-1 (q + the
// predicted correction), |q| into the solve's maxima.  s: the ring's sum in
// the frame, p: the frame's phase there.
template <bool ADJ>
__device__ __forceinline__ void gx_first(const ProbDev& P, const GEl& g, size_t o, Cx q, bool pred, bool frame, Cx s,
                                         Cx p, GxMax& sm, unsigned* qbank) {
  Cx t = q;
  if (pred) {
    if (frame) {
      s = fx_cmul(fx_coef(p.x), fx_coef(ADJ ? -p.y : p.y), s);
      s.x <<= 2;
      s.y <<= 2;
    }
    t.x += s.x;
    t.y += s.y;
  }
  reinterpret_cast<int4*>(P.zA)[o] = gx_pack(gx_dinv<ADJ>(__ldg(P.fxd + g.v), t));
  sm.add(g.b, max(fx_hi_abs(q.x), fx_hi_abs(q.y)), qbank);
}

// the weighted sum of the n newest ring entries of element o, the newest given (newest = the entry in `slot - 1`)
__device__ __forceinline__ Cx gx_ring_sum(const int4* __restrict__ ring, size_t stride, int slot, int n, int4 newest) {
  long long xh = 0, xl = 0, yh = 0, yl = 0;
  auto term = [&](int w, int4 c) {
    xh = fx_madw(w, c.x, xh);
    xl = fx_madw(w, c.y, xl);
    yh = fx_madw(w, c.z, yh);
    yl = fx_madw(w, c.w, yl);
  };
  if (n == 8 || n == 9) {
    // the orders in use: every load issued before the sums
    int4 c[9];
    c[0] = newest;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      int sl = slot - 1 - i;
      if (sl < 0) sl += kRingOrder;
      c[i] = i < n ? ring[(size_t)sl * stride] : make_int4(0, 0, 0, 0);
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) term(kExtrapI[n][i], c[i]);
  } else {
    term(kExtrapI[n][0], newest);
    for (int i = 1; i < n; ++i) {
      int sl = slot - 1 - i;
      if (sl < 0) sl += kRingOrder;
      term(kExtrapI[n][i], ring[(size_t)sl * stride]);
    }
  }
  return Cx{(long long)((unsigned long long)xh << 32) + xl, (long long)((unsigned long long)yh << 32) + yl};
}

// Commit of a converged step at one element: q <- 2 z - q and, with the
// predictor, the step's correction c = (I - dt/2 D) z - q into the ring in
// its frame, the frame turned; scaled by the state's change of scale sh.
// Returns the new q; s, p are what the next first pass needs (h: the ring
// before advance(), hn: after, possibly restarted).
template <bool ADJ>
__device__ __forceinline__ Cx gx_commit(const ProbDev& P, const GEl& g, size_t o, size_t stride, Cx z, Cx q, bool pred,
                                        bool frame, const GxHist& h, const GxHist& hn, int sh, Cx& s, Cx& p) {
  Cx qn{2 * z.x - q.x, 2 * z.y - q.y};
  if (sh) qn = Cx{fx_shift(qn.x, sh), fx_shift(qn.y, sh)};
  if (!pred) return qn;
  const int4 hd = __ldg(P.fxh + g.v);
  const Fx hy{hd.z, hd.w};
  const Cx w = fx_cmul(Fx{hd.x, hd.y}, ADJ ? fx_neg(hy) : hy, z);
  Cx c{z.x - w.x - q.x, z.y - w.y - q.y};
  if (frame) {
    p = gx_ld(h.ph + o);
    if (h.n == 0) p = Cx{kFxPhase1, 0};  // a fresh frame
    c = fx_cmul(fx_coef(p.x), fx_coef(ADJ ? p.y : -p.y), Cx{c.x << 2, c.y << 2});
    const longlong2 u = __ldg(P.fxu + g.v);
    const Cx pn = fx_cmul(fx_coef(u.x), fx_coef(u.y), p);
    p = Cx{pn.x << 2, pn.y << 2};
    gx_st(h.ph + o, p);
  }
  if (sh) {
    c = Cx{fx_shift(c.x, sh), fx_shift(c.y, sh)};
    int sl = h.slot;
    for (int i = 0; i < h.n; ++i) {
      sl = sl > 0 ? sl - 1 : kRingOrder - 1;
      int4* e = h.ring + (size_t)sl * stride + o;
      const Cx x = gx_join(*e);
      *e = gx_pack(Cx{fx_shift(x.x, sh), fx_shift(x.y, sh)});
    }
  }
  const int4 cp = gx_pack(c);
  h.ring[(size_t)h.slot * stride + o] = cp;
  if (hn.n > 0) s = gx_ring_sum(h.ring + o, stride, hn.slot, hn.n, cp);
  return qn;
}

// this solve's control row (all threads; visible after the next block barrier)
template <bool ADJ>
__device__ __forceinline__ void gx_ctl(const GxSmem& S, const ProbDev& P, int Q, int cq, int j) {
  if ((int)threadIdx.x < Q) {
    int4 t = P.ctabx[(size_t)j * (cq + 1) + threadIdx.x];
    if (ADJ) t = make_int4(-t.x, -t.y, -t.z, -t.w);
    S.ctl[threadIdx.x] = t;
  } else if ((int)threadIdx.x == Q) {
    const int4 t = P.ctabx[(size_t)j * (cq + 1) + cq];
    S.flag[1] = t.x;
    S.flag[2] = t.y;
  }
}

// The inner iterations of a solve whose first pass is done (zA holds the first
// iterate): returns the iteration count, -1 (max_iter or a control factor
// out of range) or -3 (a barrier wait gave up); on success z in *zout, and the
// states' changes of scale in S.sh (already taken into S.sc).
template <bool ADJ, int QN>
__device__ int gx_solve(const ProbDev& P, const GxParams& gp, const GxSmem& S, const double2* __restrict__ rhs, int j,
                        long long& it_global, long long& solve, int4** zout) {
  const GridHdr& G = *S.g;
  const int M = G.M;
  const long long e0 = (long long)blockIdx.x * G.chunk, e1 = min(G.total, e0 + G.chunk);
  unsigned* slots = reinterpret_cast<unsigned*>(P.gslots);  // [3][M] changes, [2][M] |q|
  unsigned* qslots = slots + 3 * M;
  unsigned* qbank = qslots + (solve & 1) * M;
  const long long limit = P.spin_limit > 0 ? P.spin_limit : kSpinLimit;
  gx_ctl<ADJ>(S, P, G.h.Q, G.h.cq, j);
  if (!gx_sync(S, P.bar, limit)) return -3;
  if (S.flag[2]) return -1;
  // the previous solve's |q| bank is free again: clear it for the next solve
  if (blockIdx.x == 0)
    for (int b = threadIdx.x; b < M; b += blockDim.x) qslots[((solve + 1) & 1) * M + b] = 0;
  ++solve;
  int4* zc = reinterpret_cast<int4*>(P.zA);
  int4* zn = reinterpret_cast<int4*>(P.zB);
  for (int it = 0; it < G.h.max_iter; ++it, ++it_global) {
    unsigned* bank = slots + (it_global % 3) * M;
    if (G.herm)
      gx_pass<ADJ, true, QN>(P, gp, S, e0, e1, rhs, zc, zn, bank);
    else
      gx_pass<ADJ, false, QN>(P, gp, S, e0, e1, rhs, zc, zn, bank);
    if (!gx_sync(S, P.bar, limit)) return -3;
    // bank of iteration it_global + 2 is no longer read by anyone: clear it
    if (blockIdx.x == 0)
      for (int b = threadIdx.x; b < M; b += blockDim.x) slots[((it_global + 2) % 3) * M + b] = 0;
    // every block takes the same decision from the same slots
    if (threadIdx.x < 32) {
      bool open = false;
      const float fac = __int_as_float(S.flag[1]);
      for (int b = threadIdx.x; b < M; b += 32) {
        const unsigned q = __ldcg(qbank + b), d = __ldcg(bank + b);
        if (d > fx_stop(fac, q)) open = true;
      }
      open = __any_sync(kFull, open);
      if (!open)
        for (int b = threadIdx.x; b < M; b += 32) {
          const int s = fx_rescale_shift(__ldcg(qbank + b));
          S.sh[b] = s;
          S.sc[b] -= s;
        }
      if (threadIdx.x == 0) S.flag[0] = open;
    }
    __syncthreads();
    const bool open = S.flag[0] != 0;
    __syncthreads();
    int4* t = zc;
    zc = zn;
    zn = t;
    if (!open) {
      ++it_global;
      *zout = zc;
      return it + 1;
    }
  }
  return -1;
}

constexpr int kGxZeroScale = 1 << 13;  // larger than any scale of a state that is not zero

__device__ __forceinline__ double gx_to(long long X, int sc) { return scalbn((double)X, -sc); }
__device__ __forceinline__ long long gx_from(double x, int sc) { return __double2ll_rn(scalbn(x, sc)); }

// Load the states from FP64 values val(g) into q (fixed point), setting every
// state's scale from its largest entry; returns 1, 0 (NaN or Inf) or -3 (a
// barrier wait gave up).  Uses the iteration's maxima slots, cleared again.
template <class F>
__device__ int gx_load(const ProbDev& P, const GxSmem& S, double2* q, F&& val) {
  const GridHdr& G = *S.g;
  const int M = G.M;
  const long long e0 = (long long)blockIdx.x * G.chunk, e1 = min(G.total, e0 + G.chunk);
  const long long limit = P.spin_limit > 0 ? P.spin_limit : kSpinLimit;
  unsigned* slots = reinterpret_cast<unsigned*>(P.gslots) + 5 * M;  // [M]
  GxMax sm;
  sm.init(e0, e1, G.Vh);
  for (GIter it_(G, e0 + threadIdx.x); it_.e < e1; it_.next(G, blockDim.x)) {
    const GEl g = gel_at(G, P.hkl, it_.b, it_.i);
    const double2 x = val(g);
    // high words of the magnitudes order them; a nonzero value below the smallest high word counts as one unit of it
    const unsigned long long a = abs_bits(x.x), b = abs_bits(x.y), m = umax64(a, b);
    sm.add(g.b, m ? max((unsigned)(m >> 32), 1u) : 0u, slots);
  }
  sm.push(slots, S.red);
  if (!gx_sync(S, P.bar, limit)) return -3;
  bool bad = false;
  if (threadIdx.x < 32) {
    for (int b = threadIdx.x; b < M; b += 32) {
      const unsigned h = __ldcg(slots + b);
      if (h >= 0x7ff00000u) bad = true;
      const int e = (int)(h >> 20);
      // a state of zeros: above every other's, to which it is to say nothing
      S.sc[b] = h ? kFxTop - (e ? e - 1023 : -1022) : kGxZeroScale;
    }
    bad = __any_sync(kFull, bad);
    if (threadIdx.x == 0) S.flag[0] = bad;
  }
  __syncthreads();
  bad = S.flag[0] != 0;
  // every block has read the slots before block 0 clears them for the next load
  if (!gx_sync(S, P.bar, limit)) return -3;
  if (blockIdx.x == 0)
    for (int b = threadIdx.x; b < M; b += blockDim.x) slots[b] = 0;
  if (bad) return 0;
  for (GIter it_(G, e0 + threadIdx.x); it_.e < e1; it_.next(G, blockDim.x)) {
    const GEl g = gel_at(G, P.hkl, it_.b, it_.i);
    const double2 x = val(g);
    gx_st(q + gslab(G, g, g.b), Cx{gx_from(x.x, S.sc[g.b]), gx_from(x.y, S.sc[g.b])});
  }
  return 1;
}

__device__ void gx_fail(const ProbDev& P, int code, int step) {
  // a wait may give up in one block while the others pass the launch's last barrier
  if (threadIdx.x == 0 && (blockIdx.x == 0 || code == -3))
    record_error(P.status, code == -3 ? LB_ECUDA : (code == 0 ? LB_ENAN : LB_ENOTCONV), step);
}

// first pass of a solve on its own (not fused with a commit)
template <bool ADJ>
__device__ void gx_first_pass(const ProbDev& P, const GxSmem& S, const double2* __restrict__ q, const GxHist& h,
                              bool pred, bool frame, long long solve) {
  const GridHdr& G = *S.g;
  const long long e0 = (long long)blockIdx.x * G.chunk, e1 = min(G.total, e0 + G.chunk);
  unsigned* qbank = reinterpret_cast<unsigned*>(P.gslots) + 3 * G.M + (solve & 1) * G.M;
  const size_t stride = (size_t)G.M * G.Vh;
  GxMax sm;
  sm.init(e0, e1, G.Vh);
  for (GIter it_(G, e0 + threadIdx.x); it_.e < e1; it_.next(G, blockDim.x)) {
    const GEl g = gel_at(G, P.hkl, it_.b, it_.i);
    const size_t o = gslab(G, g, g.b);
    Cx s{0, 0}, p{0, 0};
    const bool pr = pred && h.n > 0;
    if (pr) {
      int sl = h.slot - 1;
      if (sl < 0) sl += kRingOrder;
      s = gx_ring_sum(h.ring + o, stride, h.slot, h.n, h.ring[(size_t)sl * stride + o]);
      if (frame) p = gx_ld(h.ph + o);
    }
    gx_first<ADJ>(P, g, o, gx_ld(q + o), pr, frame, s, p, sm, qbank);
  }
  sm.push(qbank, S.red);
}

// mode 0: forward sweep of the system's states (checkpoints or stage tape if
// tape); mode 1 (ADJ: 2): steps j0..j1-1 in place on the vectors x
template <bool ADJ, int QN>
__global__ void __launch_bounds__(kGridThreads, kGxBlocks)
    k_sweep_gx(const ProbDev* __restrict__ pp, const __grid_constant__ GxParams gp, int mode, int tape, int j0, int j1,
               double2* __restrict__ x, int nstates) {
  extern __shared__ __align__(16) unsigned char smem[];
  const ProbDev& P = *pp;
  const GxSmem S = gx_setup(smem, P, nstates, mode == 0 ? P.herm : 0, P.M);
  const GridHdr& G = *S.g;
  const Hdr& H = G.h;
  const int V = H.V;
  double2* q = P.qf;
  const long long e0 = (long long)blockIdx.x * G.chunk, e1 = min(G.total, e0 + G.chunk);
  const double2* src = mode == 0 ? P.q0 : x;
  const int ld = gx_load(P, S, q, [&](const GEl& g) { return src[(size_t)g.b * V + g.v]; });
  if (ld <= 0) {
    gx_fail(P, ld, ADJ ? j1 - 1 : j0);
    return;
  }
  int* const fxs = P.fxs;  // [M][2 NT] scales of the stage vectors, then of the checkpoints
  long long itg = 0, nsolve = 0;
  unsigned long long iters = 0, steps = 0;
  int maxit = 0;
  const int R = mode == 0 ? P.pred_restart : 0;
  const bool pred = R >= 0, frame = P.fxframe != 0;
  GxHist hist;
  hist.ring = reinterpret_cast<int4*>(P.hist);
  hist.ph = P.hgp;
  hist.cap = P.pred_order;
  const size_t stride = (size_t)G.M * G.Vh;
  bool failed = false, prepped = false;
  const int nst = j1 - j0;
  // Stage vectors kept: all of them, or with checkpoints those of the last
  // segment, which the backward sweep starts with: it recomputes the others
  // only (six qutrits, 32 states, 100 steps in one segment: gradient 648 ms with
  // the recompute, 447 without, side by side).
  const int jkeep = mode != 0 || !tape ? INT32_MAX : H.K > 0 ? (H.NT - 1) / H.K * H.K : 0;
  unsigned long long iters_kept = 0, steps_kept = 0;
  for (int jj = 0; jj < nst; ++jj) {
    const int j = ADJ ? j1 - 1 - jj : j0 + jj;
    if (!prepped) {
      if (mode == 0 && tape && H.K > 0 && j % H.K == 0) {
        for (GIter it_(G, e0 + threadIdx.x); it_.e < e1; it_.next(G, blockDim.x)) {
          const GEl g = gel_at(G, P.hkl, it_.b, it_.i);
          P.ckpt[gslab(G, g, (size_t)g.b * H.n_ckpt + j / H.K)] = q[gslab(G, g, g.b)];
        }
        if (blockIdx.x == 0)
          for (int b = threadIdx.x; b < G.M; b += blockDim.x) fxs[(size_t)b * 2 * H.NT + H.NT + j / H.K] = S.sc[b];
      }
      gx_first_pass<ADJ>(P, S, q, hist, pred, frame, nsolve);
    }
    int4* z = nullptr;
    if (j >= jkeep && blockIdx.x == 0)
      for (int b = threadIdx.x; b < G.M; b += blockDim.x) fxs[(size_t)b * 2 * H.NT + j] = S.sc[b];
    const int it = gx_solve<ADJ, QN>(P, gp, S, q, j, itg, nsolve, &z);
    if (it < 0) {
      gx_fail(P, it, j);
      failed = true;
      break;
    }
    iters += (unsigned long long)it * G.M;
    steps += G.M;
    if (H.K > 0 && j >= jkeep) {
      iters_kept += (unsigned long long)it * G.M;
      steps_kept += G.M;
    }
    maxit = max(maxit, it);
    // the commit of step j in one pass with the first pass of the next step
    const bool next = jj + 1 < nst;
    const int jn = ADJ ? j - 1 : j + 1;
    GxHist hn = hist;
    if (pred) {
      hn.advance();
      if (next && R > 0 && jn % R == 0) hn.n = 0;
    }
    const bool ckn = next && mode == 0 && tape && H.K > 0 && jn % H.K == 0;
    unsigned* qbn = reinterpret_cast<unsigned*>(P.gslots) + 3 * G.M + (nsolve & 1) * G.M;
    GxMax smn;
    smn.init(e0, e1, G.Vh);
    for (GIter it_(G, e0 + threadIdx.x); it_.e < e1; it_.next(G, blockDim.x)) {
      const GEl g = gel_at(G, P.hkl, it_.b, it_.i);
      const size_t o = gslab(G, g, g.b);
      const Cx zz = gx_join(z[o]), qq = gx_ld(q + o);
      if (j >= jkeep)
        gx_st(H.K > 0 ? P.seg + gslab(G, g, (size_t)g.b * H.K + (j - jkeep))
                      : P.ckpt + gslab(G, g, (size_t)g.b * H.NT + j), zz);
      Cx s{0, 0}, p{0, 0};
      const Cx qn = gx_commit<ADJ>(P, g, o, stride, zz, qq, pred, frame, hist, hn, S.sh[g.b], s, p);
      gx_st(q + o, qn);
      if (next) {
        if (ckn) gx_st(P.ckpt + gslab(G, g, (size_t)g.b * H.n_ckpt + jn / H.K), qn);
        gx_first<ADJ>(P, g, o, qn, pred && hn.n > 0, frame, s, p, smn, qbn);
      }
    }
    if (ckn && blockIdx.x == 0)
      for (int b = threadIdx.x; b < G.M; b += blockDim.x) fxs[(size_t)b * 2 * H.NT + H.NT + jn / H.K] = S.sc[b];
    if (next) smn.push(qbn, S.red);
    hist = hn;
    prepped = next;
  }
  // the final states, in the vec layout with their mirrors
  if (!failed)
    for (GIter it_(G, e0 + threadIdx.x); it_.e < e1; it_.next(G, blockDim.x)) {
      const GEl g = gel_at(G, P.hkl, it_.b, it_.i);
      const Cx a = gx_ld(q + gslab(G, g, g.b));
      gput(mode == 0 ? P.qT : x, g, V, make_double2(gx_to(a.x, S.sc[g.b]), gx_to(a.y, S.sc[g.b])));
    }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const int phase = ADJ ? 2 : 0;
    atomicAdd(&P.status->iters[phase], iters);
    atomicAdd(&P.status->steps[phase], steps);
    if (steps_kept) {
      atomicAdd(&P.status->iters[1], iters_kept);
      atomicAdd(&P.status->steps[1], steps_kept);
    }
    atomicMax(&P.status->max_iter_seen, maxit);
  }
}

// Gradient pieces of one step over a block's chunk (eq. reducedgradient),
// kGxQP subsystems from q0 per pass: per subsystem A = sum Z conj(R), B = sum
// Z conj(P) of zhat, scaled by 2^-kc and both states' scales.  Everything is
// summed in 128-bit integers -- each product to 32 bits below its cut at 2^64
// (FxSum, lb_fixed.cuh), every state's sums brought to the smallest scale eref -- and
// added over the blocks by 64-bit integer atomics: exact, whatever their order.
// (Summed in FP64 and over the blocks by block 0, these sums took 55 us of
// an adjoint step of three states of vec 65536, the elements' products 12.)
constexpr int kGxQP = 3;
template <bool PK>
__device__ __forceinline__ void gx_grad(const ProbDev& P, const GxParams& gp, const GxSmem& S, long long e0,
                                        long long e1, const int4* __restrict__ zh, const double2* __restrict__ tape,
                                        size_t tslabs, int trow, const int* __restrict__ zsc, int eref, int q0,
                                        unsigned long long* acc) {
  const GridHdr& G = *S.g;
  const int N = G.h.N;
  constexpr int NS = PK ? 2 : 4;  // sums per subsystem
  // the current state's sums and, at the scale eref, those of the states before
  __int128 cs[kGxQP][NS], ts[kGxQP][NS];
#pragma unroll
  for (int u = 0; u < kGxQP; ++u)
#pragma unroll
    for (int c = 0; c < NS; ++c) cs[u][c] = ts[u][c] = 0;
  auto leave = [&](int b) {
    const int s = min(zsc[(size_t)b * 2 * G.h.NT] + S.sc[b] - eref, 120);
#pragma unroll
    for (int u = 0; u < kGxQP; ++u)
#pragma unroll
      for (int c = 0; c < NS; ++c) {
        ts[u][c] += s ? (cs[u][c] + (((__int128)1 << s) >> 1)) >> s : cs[u][c];
        cs[u][c] = 0;
      }
  };
  int bcur = -1;
  for (GIter it_(G, e0 + threadIdx.x); it_.e < e1; it_.next(G, blockDim.x)) {
    const GEl g = gel_at(G, P.hkl, it_.b, it_.i);
    if (g.b != bcur) {
      if (bcur >= 0) leave(bcur);
      bcur = g.b;
    }
    const size_t base = (size_t)g.b * G.Vh;
    const uint32_t kd = __ldg(P.digits + g.k), ld = __ldg(P.digits + g.l);
    const Cx Z = gx_ld(tape + ((size_t)g.b * tslabs + trow) * G.Vh + g.i);
    const Fx zx = fx_split(Z.x), zy = fx_split(Z.y), nzx = fx_split(-Z.x);
    auto add = [&](__int128& t, Fx a, long long x, Fx b, long long y) {
      FxSum v{0, 0u};
      fx_sum_mac(v, a, fx_split(x));
      fx_sum_mac(v, b, fx_split(y));
      t += ((__int128)v.hi << 32) | v.lo;
    };
#pragma unroll
    for (int u = 0; u < kGxQP; ++u)
      if (q0 + u < gp.Q) {
        const GxSub& b = gp.sub[q0 + u];
        const GxPR p = gx_pr<PK>(zh + base, b, S.cc, g.i, g.k, g.l, N, (kd >> b.sh) & gp.dm, (ld >> b.sh) & gp.dm);
        if constexpr (!PK) {
          add(cs[u][0], zx, p.rr, zy, p.ri);
          add(cs[u][1], zy, p.rr, nzx, p.ri);
          add(cs[u][2], zx, p.pr, zy, p.pi);
          add(cs[u][3], zy, p.pr, nzx, p.pi);
        } else {
          // Hermitian Z and zhat: an off-diagonal element and its mirror add
          // A - conj(B) to the g_a sum, a diagonal one A
          const bool od = g.vm >= 0;
          add(cs[u][0], zx, od ? p.rr - p.pr : p.rr, zy, od ? p.ri - p.pi : p.ri);
          add(cs[u][1], zy, od ? p.rr + p.pr : p.rr, nzx, od ? p.ri + p.pi : p.ri);
        }
      }
  }
  if (bcur >= 0) leave(bcur);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();  // the sums of the pass before are taken
#pragma unroll
  for (int u = 0; u < kGxQP; ++u)
#pragma unroll
    for (int c = 0; c < NS; ++c) {
      // in limbs of 27, 27, 27 and the rest of the bits: exact in 32-bit warp sums
      const unsigned long long l = (unsigned long long)ts[u][c];
      const long long h = (long long)(ts[u][c] >> 64);
      const unsigned r0 = __reduce_add_sync(kFull, (unsigned)l & 0x7ffffffu);
      const unsigned r1 = __reduce_add_sync(kFull, (unsigned)(l >> 27) & 0x7ffffffu);
      const unsigned r2 = __reduce_add_sync(kFull, (unsigned)(l >> 54 | (unsigned long long)h << 10) & 0x7ffffffu);
      const int r3 = __reduce_add_sync(kFull, (int)(h >> 17));
      if (lane == 0) {
        // value = r0 + r1 2^27 + (r2 + r3 2^27) 2^54
        S.gs[(u * 4 + c) * kGxWarps + warp] = make_longlong2((long long)r0 + ((long long)r1 << 27),
                                                             (long long)r2 + (long long)r3 * (1LL << 27));
      }
    }
  __syncthreads();
  if (threadIdx.x < kGxQP * 4) {
    const int u = threadIdx.x >> 2, c = threadIdx.x & 3;
    if (c < NS && q0 + u < gp.Q) {
      long long a = 0, b = 0;
      for (int w = 0; w < kGxWarps; ++w) {
        const longlong2 v = S.gs[(u * 4 + c) * kGxWarps + w];
        a += v.x;
        b += v.y;
      }
      // 54 bits in the low part: the low parts of up to 512 blocks add up without overflow
      b += a >> 54;
      a &= (1LL << 54) - 1;
      atomicAdd(acc + ((q0 + u) * 4 + c) * 2, (unsigned long long)a);
      atomicAdd(acc + ((q0 + u) * 4 + c) * 2 + 1, (unsigned long long)b);
    }
  }
}

// Backward sweep over all states: recompute each checkpoint segment, then the
// adjoint steps with the gradient pieces.  The gradient pass and the adjoint's
// commit fused with its next first pass are separate passes: the gradient
// reads zhat's neighbours in the buffer the solve left it in, which the first
// pass may write: a barrier separates the two.
template <int QN>
__global__ void __launch_bounds__(kGridThreads, kGxBlocks)
    k_backward_gx(const ProbDev* __restrict__ pp, const __grid_constant__ GxParams gp) {
  extern __shared__ __align__(16) unsigned char smem[];
  const ProbDev& P = *pp;
  const GxSmem S = gx_setup(smem, P, P.M, P.herm, P.M);
  const GridHdr& G = *S.g;
  const Hdr& H = G.h;
  const int V = H.V;
  const long long e0 = (long long)blockIdx.x * G.chunk, e1 = min(G.total, e0 + G.chunk);
  const long long limit = P.spin_limit > 0 ? P.spin_limit : kSpinLimit;
  if (blockIdx.x == 0)
    for (int t = threadIdx.x; t < 3 * LB_MAXQ * 8; t += blockDim.x)
      reinterpret_cast<unsigned long long*>(P.partials)[t] = 0ull;
  // terminal condition qhat^{N_T} = beta_i/M g_i (Appendix B)
  const int ld = gx_load(P, S, P.lam, [&](const GEl& g) {
    const size_t o = (size_t)g.b * V + g.v;
    const double w = P.wgt[g.b];
    const double2 t = P.tar[o];
    if (H.kind == LB_J_FROB) {
      const double2 qq = P.qT[o];
      return make_double2(w * (qq.x - t.x), w * (qq.y - t.y));
    }
    const double wt = linear_sign(P.kind) * w;
    return make_double2(wt * t.x, wt * t.y);
  });
  if (ld <= 0) {
    gx_fail(P, ld, H.NT - 1);
    return;
  }
  int* const fxs = P.fxs;
  long long itg = 0, nsolve = 0;
  unsigned long long it_rec = 0, st_rec = 0, it_adj = 0, st_adj = 0;
  int maxit = 0;
  const int nseg = H.K > 0 ? (H.NT + H.K - 1) / H.K : 1;
  bool failed = false;
  const bool frame = P.fxframe != 0;
  GxHist ahist;
  ahist.ring = reinterpret_cast<int4*>(P.hist);
  ahist.ph = P.hgp;
  ahist.cap = P.pred_order;
  const int R = P.pred_restart;
  const bool fpred = H.K > 0 && R > 0;
  GxHist fhist;
  fhist.ring = reinterpret_cast<int4*>(P.histf);
  fhist.ph = P.fgp;
  fhist.cap = P.pred_order;
  const size_t stride = (size_t)G.M * G.Vh;
  int* const asc = S.sc;
  // the pieces' sums of a step, [3][LB_MAXQ][4][2] by step: added to by every
  // block, read and cleared by block 0 after the step's barrier
  unsigned long long* const gacc = reinterpret_cast<unsigned long long*>(P.partials);
  constexpr int kAcc = LB_MAXQ * 8;
  unsigned gstep = 0;
  for (int sg = nseg - 1; sg >= 0 && !failed; --sg) {
    const int j0 = H.K > 0 ? sg * H.K : 0, j1 = H.K > 0 ? min(H.NT, j0 + H.K) : H.NT;
    if (H.K > 0 && sg < nseg - 1) {
      // the stage vectors of the segment recomputed (the last segment's are
      // still there from the forward sweep);
      // the adjoint's scales set aside (block 0's global copy), the checkpoint's taken
      if (blockIdx.x == 0)
        for (int b = threadIdx.x; b < G.M; b += blockDim.x) P.gsc[b] = asc[b];
      __syncthreads();
      for (int b = threadIdx.x; b < G.M; b += blockDim.x) S.sc[b] = fxs[(size_t)b * 2 * H.NT + H.NT + sg];
      __syncthreads();
      for (GIter it_(G, e0 + threadIdx.x); it_.e < e1; it_.next(G, blockDim.x)) {
        const GEl g = gel_at(G, P.hkl, it_.b, it_.i);
        P.qf[gslab(G, g, g.b)] = P.ckpt[gslab(G, g, (size_t)g.b * H.n_ckpt + sg)];
      }
      fhist.n = fhist.slot = 0;
      bool prepped = false;
      for (int j = j0; j < j1; ++j) {
        if (!prepped) gx_first_pass<false>(P, S, P.qf, fhist, fpred, frame, nsolve);
        if (blockIdx.x == 0)
          for (int b = threadIdx.x; b < G.M; b += blockDim.x) fxs[(size_t)b * 2 * H.NT + j] = S.sc[b];
        int4* z = nullptr;
        const int it = gx_solve<false, QN>(P, gp, S, P.qf, j, itg, nsolve, &z);
        if (it < 0) {
          gx_fail(P, it, j);
          failed = true;
          break;
        }
        it_rec += (unsigned long long)it * G.M;
        st_rec += G.M;
        maxit = max(maxit, it);
        const bool next = j + 1 < j1;
        GxHist hn = fhist;
        if (fpred) {
          hn.advance();
          if (next && (j + 1) % R == 0) hn.n = 0;
        }
        unsigned* qbn = reinterpret_cast<unsigned*>(P.gslots) + 3 * G.M + (nsolve & 1) * G.M;
        GxMax smn;
        smn.init(e0, e1, G.Vh);
        for (GIter it_(G, e0 + threadIdx.x); it_.e < e1; it_.next(G, blockDim.x)) {
          const GEl g = gel_at(G, P.hkl, it_.b, it_.i);
          const size_t o = gslab(G, g, g.b);
          const Cx zz = gx_join(z[o]), qq = gx_ld(P.qf + o);
          gx_st(P.seg + gslab(G, g, (size_t)g.b * H.K + (j - j0)), zz);  // read back at the same element only
          Cx s{0, 0}, p{0, 0};
          const Cx qn = gx_commit<false>(P, g, o, stride, zz, qq, fpred, frame, fhist, hn, S.sh[g.b], s, p);
          gx_st(P.qf + o, qn);
          if (next) gx_first<false>(P, g, o, qn, fpred && hn.n > 0, frame, s, p, smn, qbn);
        }
        if (next) smn.push(qbn, S.red);
        fhist = hn;
        prepped = next;
      }
      if (failed) break;
      // every block reads the adjoint's scales and the segment's stage scales block 0 wrote
      if (!gx_sync(S, P.bar, limit)) {
        gx_fail(P, -3, j0);
        failed = true;
        break;
      }
      for (int b = threadIdx.x; b < G.M; b += blockDim.x) asc[b] = __ldcg(P.gsc + b);
      __syncthreads();
    }
    bool prepped = false;
    for (int j = j1 - 1; j >= j0; --j) {
      if (!prepped) gx_first_pass<true>(P, S, P.lam, ahist, true, frame, nsolve);
      int4* zh = nullptr;
      const int it = gx_solve<true, QN>(P, gp, S, P.lam, j, itg, nsolve, &zh);
      if (it < 0) {
        gx_fail(P, it, j);
        failed = true;
        break;
      }
      it_adj += (unsigned long long)it * G.M;
      st_adj += G.M;
      maxit = max(maxit, it);
      // S.sc already holds the next step's scales: the pieces use this step's;
      // eref: the smallest sum of both scales
      __syncthreads();
      if (threadIdx.x < 32) {
        int m = INT32_MAX;
        for (int b = threadIdx.x; b < G.M; b += 32) {
          S.sc[b] += S.sh[b];
          m = min(m, fxs[(size_t)b * 2 * H.NT + j] + S.sc[b]);
        }
        m = __reduce_min_sync(kFull, m);
        if (threadIdx.x == 0) S.flag[3] = m;
      }
      __syncthreads();
      const int eref = S.flag[3];
      unsigned long long* const acc = gacc + (gstep % 3) * kAcc;
      const double2* tp = H.K > 0 ? P.seg : P.ckpt;
      const size_t slabs = H.K > 0 ? H.K : H.NT;
      for (int q0 = 0; q0 < H.Q; q0 += kGxQP) {
        if (G.herm)
          gx_grad<true>(P, gp, S, e0, e1, zh, tp, slabs, j - j0, fxs + j, eref, q0, acc);
        else
          gx_grad<false>(P, gp, S, e0, e1, zh, tp, slabs, j - j0, fxs + j, eref, q0, acc);
      }
      __syncthreads();
      for (int b = threadIdx.x; b < G.M; b += blockDim.x) S.sc[b] -= S.sh[b];
      // the first pass below writes zA, whose neighbours other blocks may still be reading
      if (!gx_sync(S, P.bar, limit)) {
        gx_fail(P, -3, j);
        failed = true;
        break;
      }
      // block 0: the step's sums, multiplied by -i: g = (S.im, -S.re)
      ++gstep;
      if (blockIdx.x == 0 && threadIdx.x < 4 * H.Q) {
        const int q = threadIdx.x >> 2;
        int c = threadIdx.x & 3;
        // Hermitian Z and zhat: the g_ad sum is minus the conjugate of the g_a sum
        const bool flip = G.herm && c == 2;
        if (G.herm) c &= 1;
        long long lo = (long long)__ldcg(acc + (q * 4 + c) * 2), hi = (long long)__ldcg(acc + (q * 4 + c) * 2 + 1);
        hi += lo >> 54;
        lo &= (1LL << 54) - 1;
        double t = scalbn(fma((double)hi, 18014398509481984.0, (double)lo), 32 - eref + P.kc[q]);
        if (flip) t = -t;
        double* gg = reinterpret_cast<double*>(P.gproj + ((size_t)j * H.Q + q) * 2);
        const int d = threadIdx.x & 3;
        if (d == 0) gg[1] = -t;
        if (d == 1) gg[0] = t;
        if (d == 2) gg[3] = -t;
        if (d == 3) gg[2] = t;
        __syncwarp(__activemask());
        if (!G.herm || d < 2) acc[(q * 4 + c) * 2] = acc[(q * 4 + c) * 2 + 1] = 0ull;
      }
      const bool next = j > j0;
      GxHist hn = ahist;
      hn.advance();
      unsigned* qbn = reinterpret_cast<unsigned*>(P.gslots) + 3 * G.M + (nsolve & 1) * G.M;
      GxMax smn;
      smn.init(e0, e1, G.Vh);
      for (GIter it_(G, e0 + threadIdx.x); it_.e < e1; it_.next(G, blockDim.x)) {
        const GEl g = gel_at(G, P.hkl, it_.b, it_.i);
        const size_t o = gslab(G, g, g.b);
        const Cx zz = gx_join(zh[o]), ll = gx_ld(P.lam + o);
        Cx s{0, 0}, p{0, 0};
        const Cx ln = gx_commit<true>(P, g, o, stride, zz, ll, true, frame, ahist, hn, S.sh[g.b], s, p);
        gx_st(P.lam + o, ln);
        if (next) gx_first<true>(P, g, o, ln, true, frame, s, p, smn, qbn);
      }
      if (next) smn.push(qbn, S.red);
      ahist = hn;
      prepped = next;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    atomicAdd(&P.status->iters[1], it_rec);
    atomicAdd(&P.status->steps[1], st_rec);
    atomicAdd(&P.status->iters[2], it_adj);
    atomicAdd(&P.status->steps[2], st_adj);
    atomicMax(&P.status->max_iter_seen, maxit);
  }
}

// ---------------------------------------------------------------------------
// y = M x on many elements (lb_apply): the off-diagonal part on the integer pipe.
// The vectors are split once (k_apply_split, scaled by each one's largest entry)
// into a buffer of the product's own; the control factors are scaled up by a
// common 2^ka so that the small sums keep 2^-60 of the largest entry times
// 2^-ka.  The diagonal and the result are FP64.

// scale with the largest entry in [2^59, 2^60) from its magnitude's high word
__device__ __forceinline__ int gx_scale_of(unsigned h) {
  const int e = (int)(h >> 20);
  return h ? kFxTop - (e ? e - 1023 : -1022) : kFxTop;
}
// A vector's largest entry and the sum of its squares: the high word of the
// largest magnitude and the sum over the squares of the entries in units of
// 2^(its exponent).  Joined in a fixed order, so that a call's route repeats.
struct GxCrest {
  unsigned h;
  float s;
};
__device__ __forceinline__ GxCrest gx_join_crest(GxCrest a, GxCrest b) {
  const unsigned h = max(a.h, b.h);
  const int e = (int)(h >> 20);
  return GxCrest{h, ldexpf(a.s, 2 * ((int)(a.h >> 20) - e)) + ldexpf(b.s, 2 * ((int)(b.h >> 20) - e))};
}
__device__ GxCrest gx_block_crest(GxCrest c) {
  __shared__ GxCrest w[kGxWarps];
  for (int o = 16; o; o >>= 1) c = gx_join_crest(c, GxCrest{__shfl_xor_sync(kFull, c.h, o), __shfl_xor_sync(kFull, c.s, o)});
  if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = c;
  __syncthreads();
  c = w[0];
  for (int i = 1; i < kGxWarps; ++i) c = gx_join_crest(c, w[i]);
  return c;
}
// ... of each block's share of a vector, part[vector][block]
__global__ void __launch_bounds__(kGridThreads) k_crest(const double2* __restrict__ x, int V, GxCrest* __restrict__ part) {
  const double2* xv = x + (size_t)blockIdx.y * V;
  GxCrest c{0u, 0.0f};
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x) {
    const double2 a = xv[v];
    const unsigned long long b = umax64(abs_bits(a.x), abs_bits(a.y));
    // (a nonzero value below the smallest high word counts as one unit of it)
    const unsigned h = b ? max((unsigned)(b >> 32), 1u) : 0u;
    float s = 0.0f;
    if (h && h < 0x7ff00000u) {
      const int sc = gx_scale_of(h);
      const float fx = (float)(int)(fx_from_bits(a.x, sc) >> 32), fy = (float)(int)(fx_from_bits(a.y, sc) >> 32);
      s = (fx * fx + fy * fy) * (1.0f / 18014398509481984.0f);  // 2^-54: units of 2^27 = 2^(59 - 32)
    }
    c = gx_join_crest(c, GxCrest{h, s});
  }
  c = gx_block_crest(c);
  if (threadIdx.x == 0) part[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = c;
}
// slots[vector] = the high word of its largest entry, or kGxNotFixed for a
// vector that holds NaN or Inf or whose entries are not spread (kGridCrest)
constexpr unsigned kGxNotFixed = 0x7ff00000u;
__global__ void __launch_bounds__(kGridThreads) k_crest_vectors(const GxCrest* __restrict__ part, int n, int V,
                                                               unsigned* __restrict__ slots) {
  GxCrest c{0u, 0.0f};
  for (int i = threadIdx.x; i < n; i += blockDim.x) c = gx_join_crest(c, part[(size_t)blockIdx.x * n + i]);
  c = gx_block_crest(c);
  if (threadIdx.x) return;
  // the largest entry in [1, 2)
  const float m = 1.0f + (float)(c.h & 0xfffffu) * (1.0f / 1048576.0f);
  const bool spread = c.h == 0 || (float)V * m * m <= (float)(kGridCrest * kGridCrest) * c.s;
  slots[blockIdx.x] = c.h < kGxNotFixed && spread ? c.h : kGxNotFixed;
}
__global__ void k_apply_split(const double2* __restrict__ x, int V, const unsigned* __restrict__ slots,
                              int4* __restrict__ z) {
  const unsigned h = slots[blockIdx.y];
  if (h >= kGxNotFixed) return;  // k_apply_gx computes this vector in FP64
  const int sc = gx_scale_of(h);
  const size_t base = (size_t)blockIdx.y * V;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x) {
    const double2 a = x[base + v];
    z[base + v] = gx_pack(Cx{fx_from_bits(a.x, sc), fx_from_bits(a.y, sc)});
  }
}
template <bool ADJ, int QN>
__global__ void __launch_bounds__(kGridThreads, kApplyBlocks)
    k_apply_gx(const ProbDev* __restrict__ pp, const __grid_constant__ GxParams gp, int step,
               const double2* __restrict__ x, const int4* __restrict__ z, const unsigned* __restrict__ slots,
               double2* __restrict__ y, int n_vec) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_ka;
  __shared__ unsigned long long s_d[kGxWarps];
  const ProbDev& P = *pp;
  const GxSmem S = gx_setup(smem, P, n_vec, 0, 0);
  const Hdr& H = S.g->h;
  const int V = H.V, N = H.N;
  const double2* ct = P.ctab + (size_t)step * H.cq;
  // the largest power of two that keeps every factor below 0.45, and those
  // that one sum of gx_apply takes (both control factors and a decay factor)
  // below 0.75 together: its middle part adds each factor's high half times a
  // low half of 2^31 and each one's low half times a high half of 2^28
  double d = 0.0;
  for (int i = threadIdx.x; i < P.njcoef; i += blockDim.x) d = fmax(d, fmax(P.jf[i], P.ja[i]));
  const unsigned long long dm = warp_max_u64(abs_bits(d));
  if ((threadIdx.x & 31) == 0) s_d[threadIdx.x >> 5] = dm;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = 0.0, c = 0.0;
    for (int q = 0; q < gp.Q; ++q) {
      m = fmax(m, scalbn(fmax(fabs(ct[q].x), fabs(ct[q].y)), P.kc[q]));
      c = fmax(c, scalbn(fabs(ct[q].x) + fabs(ct[q].y), P.kc[q]));
    }
    for (int w = 0; w < kGxWarps; ++w) d = fmax(d, __longlong_as_double((long long)s_d[w]));
    m = fmax(fmax(m, d), 0.6 * (c + d));
    s_ka = m > 0.0 ? min(20, ilogb(0.45 / m)) : 20;
  }
  __syncthreads();
  const int ka = s_ka;
  if ((int)threadIdx.x < gp.Q) {
    const int q = threadIdx.x;
    const double sg = ADJ ? -1.0 : 1.0;
    const Fx a = fx_coef(__double2ll_rn(scalbn(sg * ct[q].x, 64 + P.kc[q] + ka)));
    const Fx b = fx_coef(__double2ll_rn(scalbn(sg * ct[q].y, 64 + P.kc[q] + ka)));
    S.ctl[q] = make_int4(a.h, a.l, b.h, b.l);
  }
  for (int i = threadIdx.x; i < P.njcoef; i += blockDim.x) {
    S.jf[i] = fx_coef(__double2ll_rn(scalbn(P.jf[i], 64 + ka)));
    S.ja[i] = fx_coef(__double2ll_rn(scalbn(P.ja[i], 64 + ka)));
  }
  __syncthreads();
  const double inv = 2.0 / H.h;
  const long long n = (long long)n_vec * V;
  const int nt = gridDim.x * blockDim.x;
  for (GIter it_(*S.g, (long long)blockIdx.x * blockDim.x + threadIdx.x); it_.e < n; it_.next(*S.g, nt)) {
    const long long e = it_.e;
    const int b = it_.b, v = it_.i, l = (int)((unsigned)v / (unsigned)N), k = v - l * N;
    const uint32_t kd = __ldg(P.digits + k), ld = __ldg(P.digits + l);
    const unsigned h = __ldg(slots + b);
    double cr = 0.0, ci = 0.0;
    if (h < kGxNotFixed) {
      const Cx c = gx_apply<ADJ, false, QN>(z + (size_t)b * V, gp, S, v, k, l, N, kd, ld);
      const double f = scalbn(inv, -gx_scale_of(h) - ka);
      cr = f * (double)c.x;
      ci = f * (double)c.y;
    } else {
      const Tabs T{P.cu, P.cd, P.jf, P.ja};
      offdiag_acc<ADJ>(cr, ci, x + (size_t)b * V, v, kd, ld, H, T, ct);
      cr *= inv;
      ci *= inv;
    }
    const double2 D = __ldg(P.D + v), xx = x[e];
    const double di = ADJ ? -D.y : D.y;
    y[e] = make_double2(fma(D.x, xx.x, -di * xx.y) + cr, fma(D.x, xx.y, di * xx.x) + ci);
  }
}

GxParams gx_params(const ProbDev& h) {
  GxParams p{};
  p.Q = h.Q;
  p.dm = (1 << h.dbits) - 1;
  for (int q = 0; q < h.Q; ++q) {
    GxSub& b = p.sub[q];
    b.n = h.levels[q];
    b.s = h.stride[q];
    b.sh = h.dbits * q;
    b.co = h.coff[q];
    b.jo = h.joff[q];
    b.decay = h.jump[q] != 0.0;
    b.t1 = b.s * (b.s + 1) / 2;
    b.t2 = b.s * (b.s - 1) / 2;
  }
  return p;
}

// the kernels' instantiation for Q subsystems
template <bool ADJ>
const void* sweep_kernel(int Q) {
  switch (Q) {
    case 3: return (const void*)k_sweep_gx<ADJ, 3>;
    case 4: return (const void*)k_sweep_gx<ADJ, 4>;
    case 6: return (const void*)k_sweep_gx<ADJ, 6>;
    default: return (const void*)k_sweep_gx<ADJ, 0>;
  }
}
const void* backward_kernel(int Q) {
  switch (Q) {
    case 3: return (const void*)k_backward_gx<3>;
    case 4: return (const void*)k_backward_gx<4>;
    case 6: return (const void*)k_backward_gx<6>;
    default: return (const void*)k_backward_gx<0>;
  }
}

// Blocks of a launch: all the device holds at once, but no more than give each
// kGxMinElems elements (a barrier costs with every block that arrives: gradients
// of 2 x 2 x 20 levels, 300 steps, 9.7 ms at 32 and 64, 9.8 at 128, 10.2 at 256,
// 13.3 at 512; four qutrits, 8 states, 200 steps, 9.25, 9.26, 9.03, 12.3).
constexpr int kGxMinElems = 64;
constexpr int kGxMaxBlocks = 512;  // gx_grad's sums over the blocks
cudaError_t gx_launch(const void* k, long long elements, size_t smem, void** args, cudaStream_t s) {
  int dev = 0, nsm = 0, per = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, kGridThreads, smem);
  if (e != cudaSuccess) return e;
  long long n = (long long)nsm * per;
  const long long few = (elements + kGxMinElems - 1) / kGxMinElems;
  if (n > few) n = few;
  if (n > kGxMaxBlocks) n = kGxMaxBlocks;
  return cudaLaunchCooperativeKernel(k, dim3((unsigned)n), dim3(kGridThreads), args, smem, s);
}

template <bool ADJ, int QN>
cudaError_t run_apply(unsigned blocks, size_t smem, cudaStream_t s, const ProbDev* p, const GxParams& gp, int step,
                      const double2* x, const int4* z, const unsigned* slots, double2* y, int n_vec) {
  // (above 48 KB for one mode of some 55 levels and more)
  cudaError_t e =
      cudaFuncSetAttribute(k_apply_gx<ADJ, QN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_apply_gx<ADJ, QN><<<blocks, kGridThreads, smem, s>>>(p, gp, step, x, z, slots, y, n_vec);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_crest(const ProbDev& h, const double2* x, int n_vec, cudaStream_t s) {
  GxCrest* part = reinterpret_cast<GxCrest*>(h.apx);
  const int n = std::min((h.V + 8 * kGridThreads - 1) / (8 * kGridThreads), 512);
  k_crest<<<dim3((unsigned)n, n_vec), kGridThreads, 0, s>>>(x, h.V, part);
  k_crest_vectors<<<n_vec, kGridThreads, 0, s>>>(part, n, h.V, h.apm);
  return cudaGetLastError();
}

cudaError_t launch_apply_gx(const ProbDev* d_prob, const ProbDev& h, int adjoint, int64_t step, const double2* x,
                            double2* y, int n_vec, cudaStream_t s) {
  const GxParams gp = gx_params(h);
  const unsigned* slots = h.apm;
  int4* z = h.apx;
  cudaError_t e = launch_crest(h, x, n_vec, s);
  if (e != cudaSuccess) return e;
  const unsigned bx = (unsigned)((h.V + 8 * 256 - 1) / (8 * 256));
  k_apply_split<<<dim3(bx, n_vec), 256, 0, s>>>(x, h.V, slots, z);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const long long nb = ((long long)n_vec * h.V + kGridThreads - 1) / kGridThreads;
  // the blocks the device holds at once: the tables are set up once per block
  int dev = 0, nsm = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (unsigned)std::min<long long>(nb, (long long)nsm * kApplyBlocks);
  const size_t smem = gx_smem_bytes(h.ncoef, h.njcoef, 0);
  auto run = [&](auto adj) {
    constexpr bool ADJ = decltype(adj)::value;
    switch (h.Q) {
      case 4: return run_apply<ADJ, 4>(blocks, smem, s, d_prob, gp, (int)step, x, z, slots, y, n_vec);
      case 6: return run_apply<ADJ, 6>(blocks, smem, s, d_prob, gp, (int)step, x, z, slots, y, n_vec);
      default: return run_apply<ADJ, 0>(blocks, smem, s, d_prob, gp, (int)step, x, z, slots, y, n_vec);
    }
  };
  return adjoint ? run(std::true_type{}) : run(std::false_type{});
}

cudaError_t launch_sweep_gx(const ProbDev* d_prob, const ProbDev& h, int mode, int tape, int64_t j0, int64_t j1,
                            double2* x, int nstates, cudaStream_t s) {
  GxParams gp = gx_params(h);
  int m = mode, tp = tape, a = (int)j0, b = (int)j1, ns = nstates;
  const ProbDev* p = d_prob;
  void* args[] = {(void*)&p, (void*)&gp, (void*)&m, (void*)&tp, (void*)&a, (void*)&b, (void*)&x, (void*)&ns};
  const long long vh = mode == 0 && h.herm ? (long long)h.N * (h.N + 1) / 2 : h.V;
  return gx_launch(mode == 2 ? sweep_kernel<true>(h.Q) : sweep_kernel<false>(h.Q), vh * nstates,
                   gx_smem_bytes(h.ncoef, h.njcoef, h.M), args, s);
}

cudaError_t launch_backward_gx(const ProbDev* d_prob, const ProbDev& h, cudaStream_t s) {
  GxParams gp = gx_params(h);
  const ProbDev* p = d_prob;
  void* args[] = {(void*)&p, (void*)&gp};
  const long long vh = h.herm ? (long long)h.N * (h.N + 1) / 2 : h.V;
  return gx_launch(backward_kernel(h.Q), vh * h.M, gx_smem_bytes(h.ncoef, h.njcoef, h.M), args, s);
}

}  // namespace lbk
