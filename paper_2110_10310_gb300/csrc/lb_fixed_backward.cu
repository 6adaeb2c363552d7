// Recompute and adjoint sweep in fixed point, one CTA per state, with the
// gradient pieces of eq. reducedgradient.

#include "lb_fixed_sweep.cuh"

namespace lbk {

namespace {

// sum over the warp of v without its last 16 bits, in three limbs of 27 bits (the
// sums unsigned, unsigned and signed), to every lane.  (All 32 bits take a
// fourth reduction per sum: CNOT gradient, 10000 steps, 5.90 ms against 5.79.
// 2^-16 of the cut over 4096 products stays 2^-6 below what one entry's rounding adds.)
__device__ __forceinline__ int3 fx_warp_sum(const FxSum& v) {
  const unsigned h0 = (unsigned)v.hi;
  int3 r;
  r.x = (int)__reduce_add_sync(kFull, (v.lo >> 16 | h0 << 16) & 0x7ffffffu);
  r.y = (int)__reduce_add_sync(kFull, (unsigned)(v.hi >> 11) & 0x7ffffffu);
  r.z = __reduce_add_sync(kFull, (int)(v.hi >> 38));
  return r;
}

// a lane's share of the gradient pieces of one subsystem and element, from
// its component Zc of Z, the other component Zo and its component of P and R
// of zhat (R: a lane of component c adds Z_c R_c to Re A = sum Re(Z conj(R)) and
// +-Z_{1-c} R_c to Im A; the same with P for B).  herm: 0, or under the
// Hermitian symmetry 1 off and 2 on the diagonal.
struct FxG {
  FxSum ar, ai, br, bi;
};
__device__ __forceinline__ void fx_prod(FxSum& s, long long a, long long b) { fx_sum_mac(s, fx_split(a), fx_split(b)); }
__device__ __forceinline__ void fx_grad_acc(FxG& g, const FxPR& p, long long Zc, long long Zo, bool im, int herm) {
  // Im A = Zy Rx - Zx Ry
  const long long Zs = im ? -Zo : Zo;
  if (herm == 0) {
    fx_prod(g.ar, Zc, p.r);
    fx_prod(g.ai, Zs, p.r);
    fx_prod(g.br, Zc, p.p);
    fx_prod(g.bi, Zs, p.p);
  } else if (herm == 1) {
    // the element and its mirror add A - conj(B) to the g_a sum
    fx_prod(g.ar, Zc, p.r - p.p);
    fx_prod(g.ai, Zs, p.r + p.p);
  } else {
    fx_prod(g.ar, Zc, p.r);
    fx_prod(g.ai, Zs, p.r);
  }
}

// Gradient pieces of one step (eq. reducedgradient): per subsystem A = sum Z
// conj(R) and B = sum Z conj(P) of zhat (scaled 2^-kc and by both scales).
// The warps' sums go to shared memory; fx_grad_store adds them after
// the next barrier.  Z0: the lane's element of the stage vector (QT > 0).
template <int E, int QT>
__device__ __forceinline__ void fx_grad(const FxState<E, QT>& st, const FxSmem& S, const Fx* __restrict__ zh,
                                        const Cx* __restrict__ Zt, Cx Z0, unsigned step) {
  const Hdr& H = *S.hdr;
  const int V = H.V, Q = H.Q, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool im = st.im;
  int* const gr = S.gred + (step & 1) * (4 * Q * kFxWarps * 3) + warp * 3;
  auto put = [&](int q, const FxG& g) {
    const int3 a = fx_warp_sum(g.ar), b = fx_warp_sum(g.ai);
    int* o = gr + q * (4 * kFxWarps * 3);
    if (lane < 3) o[lane] = lane == 0 ? a.x : (lane == 1 ? a.y : a.z);
    else if (lane < 6) o[kFxWarps * 3 + lane - 3] = lane == 3 ? b.x : (lane == 4 ? b.y : b.z);
    if (!H.herm) {
      const int3 c = fx_warp_sum(g.br), d = fx_warp_sum(g.bi);
      o += 2 * kFxWarps * 3;
      if (lane < 3) o[lane] = lane == 0 ? c.x : (lane == 1 ? c.y : c.z);
      else if (lane < 6) o[kFxWarps * 3 + lane - 3] = lane == 3 ? d.x : (lane == 4 ? d.y : d.z);
    }
  };
  if constexpr (QT > 0) {
    const int hm = H.herm ? (st.m[0] >= 0 ? 1 : 2) : 0;
    const long long Zc = im ? Z0.y : Z0.x, Zo = im ? Z0.x : Z0.y;
#pragma unroll
    for (int q = 0; q < QT; ++q)
      if (q < st.pl.nq) {
        FxG g{};
        if (st.v[0] < V) {
          const FxPR p = fx_pr(ldb(zh, st.pl.o[q][0]), ldb(zh, st.pl.o[q][1]), ldb(zh, st.pl.o[q][2]),
                               ldb(zh, st.pl.o[q][3]), st.pl.c[q][0], st.pl.c[q][1], st.pl.c[q][2], st.pl.c[q][3]);
          fx_grad_acc(g, p, Zc, Zo, im, hm);
        }
        put(q, g);
      }
  } else {
    for (int q = 0; q < Q; ++q) {
      FxG g{};
      const FxSub b = S.sub[q];
      const int sh = (b.n_sh >> 8) & 0xff, s = b.s, sN = s * H.N, dm = H.dm;
      const int4 *ck = S.ck + b.co, *cl = S.cl + b.co;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int v = fx_v(st, S, H, e);
        if (v < V) {
          const Cx Z = Zt[v];
          const FxPR p = fx_pr_tab(zh + 2 * v + im, ck[(st.kd[e] >> sh) & dm], cl[(st.ld[e] >> sh) & dm], s, sN);
          fx_grad_acc(g, p, im ? Z.y : Z.x, im ? Z.x : Z.y, im, H.herm ? (fx_m(st, S, H, e) >= 0 ? 1 : 2) : 0);
        }
      }
      put(q, g);
    }
  }
}
// the CTA's sums of the step's pieces, times -i and 2^-ssum, to g[q][2] (threads < 4 Q)
__device__ __forceinline__ void fx_grad_store(const FxSmem& S, const ProbDev& P, double2* g, int ssum, unsigned step) {
  const Hdr& H = *S.hdr;
  const int Q = H.Q, nwarps = blockDim.x >> 5;
  if ((int)threadIdx.x >= 4 * Q) return;
  const int q = threadIdx.x >> 2;
  int c = threadIdx.x & 3;
  // Hermitian Z and zhat: the g_ad sum is minus the conjugate of the g_a sum
  const bool flip = H.herm && c == 2;
  if (H.herm) c &= 1;
  const int* w = S.gred + (step & 1) * (4 * Q * kFxWarps * 3) + (q * 4 + c) * (kFxWarps * 3);
  unsigned long long a = 0, b = 0;
  long long hi = 0;
  for (int i = 0; i < nwarps; ++i) {
    a += (unsigned)w[3 * i];
    b += (unsigned)w[3 * i + 1];
    hi += w[3 * i + 2];
  }
  // the sum is hi 2^54 + b 2^27 + a in units of 2^-16
  b += a >> 27;
  hi += (long long)(b >> 27);
  const unsigned long long lo = (b & 0x7ffffffull) << 27 | (a & 0x7ffffffull);
  double t = scalbn(fma((double)hi, 18014398509481984.0, (double)lo), P.kc[q] - ssum - 16);
  if (flip) t = -t;
  double* o = reinterpret_cast<double*>(g + q * 2);
  const int d = threadIdx.x & 3;
  if (d == 0) o[1] = -t;
  if (d == 1) o[0] = t;
  if (d == 2) o[3] = -t;
  if (d == 3) o[2] = t;
}

// QT > 0: the adjoint's own values set aside in the workspace (PUT), and taken
// back, around a segment's recompute: the right-hand side, the difference
// table and the frame, in the slots of the ring this predictor does not use.
// They would otherwise stay in registers through the recompute's loop.
template <int E, int QT, bool PUT>
__device__ __forceinline__ void fx_aside(FxState<E, QT>& st, const FxSmem& S, const ProbDev& P, size_t base) {
  const Hdr& H = *S.hdr;
  const size_t stride = 2 * (size_t)P.M * P.V;
  auto mv = [&](long long& x, long long* p) {
    if constexpr (PUT) *p = x;
    else x = *p;
  };
  if constexpr (QT > 0) {
    const int v = st.v[0];
    if (v >= H.V) return;
    long long* a = reinterpret_cast<long long*>(P.hist + base) + 2 * v + st.im;
#pragma unroll
    for (int k = 0; k < kFxOrder; ++k) mv(st.pr.d[k], a + (size_t)k * stride);
    static_assert(kFxOrder + 2 <= kRingOrder, "the ring's slots hold the table, the sum and the right-hand side");
    mv(st.pr.s, a + (size_t)kFxOrder * stride);
    mv(st.q[0], a + (size_t)(kFxOrder + 1) * stride);
    // each lane its own copy of p (both components)
    Cx* f = reinterpret_cast<Cx*>((st.im ? P.hgm : P.hgp) + base) + v;
    mv(st.pr.p.x, &f->x);
    mv(st.pr.p.y, &f->y);
  }
}

template <int E, int QT, int T>
__global__ void __launch_bounds__(T)
    k_backward_fx(const ProbDev* __restrict__ probs, const WorkItem* __restrict__ items, int mode) {
  extern __shared__ __align__(16) unsigned char smem[];
  // items == null: one CTA per (chunk, state) of the first problem (full
  // stage tape); mode 1: no gradient, only the chunk's adjoint state that its
  // running penalty's sources alone leave (zero at the chunk's end)
  const bool chunked = QT > 0 && items == nullptr;
  const ProbDev& P = probs[chunked ? 0 : items[blockIdx.x].prob];
  const int i = chunked ? (int)blockIdx.x % P.M : items[blockIdx.x].state;
  const int ch = chunked ? (int)blockIdx.x / P.M : 0;
  const FxSmem S = fx_carve(smem, P, E * (blockDim.x / 2), QT);
  fx_setup(S, P, P.herm);
  const Hdr& H = *S.hdr;
  const int V = H.V, NT = H.NT, K = H.K, Q = H.Q;
  FxState<E, QT> st;
  fx_init(st, S, P);
  const size_t base = (size_t)i * V;
  const double w = P.wgt[i], wt = linear_sign(P.kind) * w;
  const bool penal = H.gamma1 != 0.0;
  const int cl = chunked ? P.chunkL : NT;
  const int ja = ch * cl, jb = min(NT, ja + cl);  // this CTA's steps
  // running penalty: q^j is rebuilt backwards, q^j = 2 z^j - q^{j+1}, from the
  // state at the end of the CTA's steps (a register for QT > 0, else in qb)
  double qbr = 0.0;
  if (penal) {
    if constexpr (QT > 0) {
      const int v = st.v[0];
      if (v < V) {
        const size_t b = (size_t)(ch + 1) * P.M + i;
        qbr = jb < NT ? fx_to(reinterpret_cast<const long long*>(P.bst + b * V)[2 * v + st.im], P.bsc[b])
                      : reinterpret_cast<const double*>(P.qT + base)[2 * v + st.im];
      }
    } else {
      for (int v = threadIdx.x; v < V; v += blockDim.x) P.qb[base + v] = P.qT[base + v];
    }
  }
  CtaStats stats;
  // terminal condition qhat^{N_T} = beta_i/M g_i (Appendix B), or the chunk's
  bool zero = chunked && mode == 1;  // nothing but zeros so far
  if (chunked) {
    const size_t C1 = P.chunkC + 1, b = (C1 + ch + 1) * P.M + i;
    if (zero)
      st.q[0] = 0, st.sc = kFxTop;
    else
      fx_load_fixed(st, S, P.bst + b * V, P.bsc[b]);
  } else if (!fx_load(st, S, [&](int v) {
               const double2 t = P.tar[base + v];
               if (H.kind != LB_J_FROB) return make_double2(wt * t.x, wt * t.y);
               const double2 qq = P.qT[base + v];
               return make_double2(w * (qq.x - t.x), w * (qq.y - t.y));
             })) {
    if (threadIdx.x == 0) record_error(P.status, LB_ENAN, NT - 1);
    return;
  }
  int* const scz = P.fxs + (size_t)i * 2 * NT;
  const int nseg = K > 0 ? (NT + K - 1) / K : 1;
  const int R = P.pred_restart;
  const bool fpred = K > 0 && R > 0 && P.fxfwd;
  FxCount cnt;
  int cur = 0;
  // the pieces of the step before, stored after the next barrier
  int jprev = -1, sprev = 0;
  unsigned gstep = 0;
  for (int sg = nseg - 1; sg >= 0; --sg) {
    const int j0 = K > 0 ? sg * K : ja, j1 = K > 0 ? min(NT, j0 + K) : jb;
    if (K > 0 && sg < nseg - 1) {
      // recompute the stage vectors of this segment from its checkpoint (the
      // last segment's are still there from the forward sweep)
      __syncthreads();
      if (jprev >= 0) fx_grad_store(S, P, P.gproj + (((size_t)i * NT + jprev) * Q) * 2, sprev, gstep - 1);
      jprev = -1;
      const int an = st.n, aslot = st.slot, asc = st.sc;
      long long lam[E];
      if constexpr (QT > 0) {
        fx_aside<E, QT, true>(st, S, P, base);
      } else {
#pragma unroll
        for (int e = 0; e < E; ++e) lam[e] = st.q[e];
      }
      if (fpred) fx_ring(st, S, P, P.histf, P.fgp, P.fgm, base);
      st.n = st.slot = 0;
      const long long* ck = reinterpret_cast<const long long*>(P.ckpt + ((size_t)i * H.n_ckpt + sg) * V) + st.im;
      st.sc = scz[NT + sg];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int v = fx_v(st, S, H, e);
        st.q[e] = v < V ? ck[2 * v] : 0;
      }
      fx_ctl(S, P, H.cq, j0, cnt.step);
      for (int j = j0; j < j1; ++j) {
        if (fpred && j % R == 0) st.n = 0;
        unsigned qtop;
        long long z = 0, c = 0;
        const int it = fx_solve<E, QT, false>(st, S, P, j + 1 < j1 ? j + 1 : -1, fpred, cnt, cur, qtop, z, c);
        if (it < 0) {
          fx_fail(P.status, j, false);
          stats.flush(P.status);
          return;
        }
        stats.add(1, it);
        if (fpred) fx_commit<E, QT, false>(st, S, c);
        if (threadIdx.x == 0) scz[j] = st.sc;
        fx_update(st, S, cur ? S.zb1 : S.zb0, z, reinterpret_cast<long long*>(P.seg + ((size_t)i * K + (j - j0)) * V));
        fx_rescale(st, S, qtop, fpred);
      }
      if constexpr (QT > 0) {
        fx_aside<E, QT, false>(st, S, P, base);
      } else {
#pragma unroll
        for (int e = 0; e < E; ++e) st.q[e] = lam[e];
        st.pr.ring = reinterpret_cast<long long*>(P.hist + base);
        st.pr.ph = reinterpret_cast<Cx*>(P.hgp + base);
        st.pr.fu = reinterpret_cast<Cx*>(P.hgm + base);
      }
      st.n = an;
      st.slot = aslot;
      st.sc = asc;
      __syncthreads();  // the segment's stage vectors and scales are complete
    }
    fx_ctl(S, P, H.cq, j1 - 1, cnt.step);
    if (sg == nseg - 1) fx_ring(st, S, P, P.hist, P.hgp, P.hgm, base);
    const Cx* tape = reinterpret_cast<const Cx*>(K > 0 ? P.seg + (size_t)i * K * V : P.ckpt + ((size_t)i * NT + ja) * V);
    // QT > 0: the lane's element of the stage vector, loaded one step ahead
    Cx Zn{0, 0};
    int scn = scz[j1 - 1];
    if constexpr (QT > 0)
      if (st.v[0] < V) Zn = tape[(size_t)(j1 - 1 - j0) * V + st.v[0]];
    for (int j = j1 - 1; j >= j0; --j) {
      const Cx Z = Zn;
      const int sz = scn;
      const Cx* Zt = tape + (size_t)(j - j0) * V;
      if (j > j0) {
        scn = scz[j - 1];
        if constexpr (QT > 0)
          if (st.v[0] < V) Zn = tape[(size_t)(j - 1 - j0) * V + st.v[0]];
      }
      // the running penalty's source gamma1 beta_i/M dt beta(t_j) g(q^j) at the
      // lane's element e (Appendix B), rebuilding q^j
      const double pw = penal ? H.gamma1 * w * P.pen[j] : 0.0;
      auto source = [&](int e) {
        const int v = fx_v(st, S, H, e);
        const Cx Ze = QT > 0 ? Z : Zt[v];
        double* qb = QT > 0 ? &qbr : reinterpret_cast<double*>(P.qb + base) + 2 * v + st.im;
        const double t = (reinterpret_cast<const double*>(P.tar + base))[2 * v + st.im];
        const double qj = fma(2.0, fx_to(st.im ? Ze.y : Ze.x, sz), -*qb);
        *qb = qj;
        return pw * (H.kind == LB_J_FROB ? qj - t : linear_sign(H.kind) * t);
      };
      if (QT > 0 && zero) {
        // a zero adjoint state stays zero: start from the first nonzero source
        const double sr = st.v[0] < V ? source(0) : 0.0;
        const unsigned long long mx = fx_cta_max(S, abs_bits(sr));
        if (j > j0) fx_ctl(S, P, H.cq, j - 1, cnt.step);
        if (mx >= kInfBits && j > 0) {
          fx_overflow(P.status, j - 1, chunked);
          return;
        }
        if (mx == 0 || mx >= kInfBits) continue;
        st.sc = fx_scale(mx);
        st.q[0] = fx_from(sr, st.sc);
        zero = false;
        continue;
      }
      unsigned qtop;
      long long z = 0, c = 0;
      // (I - dt/2 (M^{j+1/2})^+) zhat^j = qhat^{j+1}   (eq. linsystem_adjoint)
      const int it = fx_solve<E, QT, true>(st, S, P, j > j0 ? j - 1 : -1, true, cnt, cur, qtop, z, c);
      if (it < 0) {
        fx_fail(P.status, j, chunked);
        stats.flush(P.status);
        return;
      }
      if (QT == 0 || mode == 0) stats.add(2, it);
      if (jprev >= 0) fx_grad_store(S, P, P.gproj + (((size_t)i * NT + jprev) * Q) * 2, sprev, gstep - 1);
      fx_commit<E, QT, true>(st, S, c);
      const Fx* zh = cur ? S.zb1 : S.zb0;
      if (QT == 0 || mode == 0) {
        fx_grad(st, S, zh, Zt, Z, gstep);
        jprev = j;
        sprev = sz + st.sc - 64;
        ++gstep;
      }
      // qhat^j = 2 zhat - qhat^{j+1}, plus the penalty's source
      fx_update(st, S, zh, z, nullptr);
      if (penal) {
        double src[E];
#pragma unroll
        for (int e = 0; e < E; ++e) src[e] = fx_v(st, S, H, e) < V ? source(e) : 0.0;
        // (the state before step 0 is not used)
        if (!fx_add_source(st, S, src, true) && j > 0) {
          fx_overflow(P.status, j - 1, chunked);
          stats.flush(P.status);
          return;
        }
      } else {
        fx_rescale(st, S, qtop, true);
      }
    }
  }
  __syncthreads();
  if (jprev >= 0) fx_grad_store(S, P, P.gproj + (((size_t)i * NT + jprev) * Q) * 2, sprev, gstep - 1);
  if constexpr (QT > 0)
    if (mode == 1) {
      const size_t C1 = P.chunkC + 1, b = (2 * C1 + ch) * P.M + i;
      if (st.v[0] < V) reinterpret_cast<long long*>(P.bst + b * V)[2 * st.v[0] + st.im] = st.q[0];
      if (threadIdx.x == 0) P.bsc[b] = st.sc;
    }
  stats.flush(P.status);
}

}  // namespace

template <int E, int QT, int T = fx_max_threads<QT>()>
static cudaError_t run(const FixedConfig& fc, int n, cudaStream_t s, const ProbDev* p, const WorkItem* it, int mode = 0) {
  cudaError_t e = cudaFuncSetAttribute(k_backward_fx<E, QT, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fc.smem);
  if (e != cudaSuccess) return e;
  k_backward_fx<E, QT, T><<<n, fc.threads, fc.smem, s>>>(p, it, mode);
  return cudaGetLastError();
}

cudaError_t launch_backward_fixed_chunked(const ProbDev* d_prob, int n_ctas, int mode, const FixedConfig& fc,
                                          cudaStream_t s) {
  switch (fc.QT) {
    case 2: return run<1, 2>(fc, n_ctas, s, d_prob, nullptr, mode);
    case 3: return run<1, 3>(fc, n_ctas, s, d_prob, nullptr, mode);
    case 4: return run<1, 4>(fc, n_ctas, s, d_prob, nullptr, mode);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_backward_fixed(const ProbDev* d_probs, const WorkItem* d_items, int n_items, const FixedConfig& fc,
                                  cudaStream_t s) {
  switch (fc.QT) {
    case 2: return run<1, 2>(fc, n_items, s, d_probs, d_items);
    case 3: return run<1, 3>(fc, n_items, s, d_probs, d_items);
    case 4: return run<1, 4>(fc, n_items, s, d_probs, d_items);
    default: break;
  }
  switch (fc.E) {
    case 1:
      return fc.threads <= kFxTabFew ? run<1, 0, kFxTabFew>(fc, n_items, s, d_probs, d_items)
                                     : run<1, 0>(fc, n_items, s, d_probs, d_items);
    case 2: return run<2, 0>(fc, n_items, s, d_probs, d_items);
    case 3: return run<3, 0>(fc, n_items, s, d_probs, d_items);
    case 5: return run<5, 0>(fc, n_items, s, d_probs, d_items);
    case 8: return run<8, 0>(fc, n_items, s, d_probs, d_items);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lbk
