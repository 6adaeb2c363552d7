// Forward sweep in fixed point, one CTA per state.

#include "lb_fixed_sweep.cuh"

namespace lbk {

namespace {

template <int E, int QT, int T>
__global__ void __launch_bounds__(T)
    k_forward_fx(const ProbDev* __restrict__ probs, const WorkItem* __restrict__ items, int tape) {
  extern __shared__ __align__(16) unsigned char smem[];
  // items == null: one CTA per (chunk, state) of the first problem
  const bool chunked = QT > 0 && items == nullptr;
  const ProbDev& P = probs[chunked ? 0 : items[blockIdx.x].prob];
  const int i = chunked ? (int)blockIdx.x % P.M : items[blockIdx.x].state;
  const int ch = chunked ? (int)blockIdx.x / P.M : 0;
  const FxSmem S = fx_carve(smem, P, E * (blockDim.x / 2), QT);
  fx_setup(S, P, P.herm);
  const Hdr& H = *S.hdr;
  const int V = H.V, NT = H.NT, K = H.K;
  FxState<E, QT> st;
  fx_init(st, S, P);
  const size_t base = (size_t)i * V;
  fx_ring(st, S, P, P.hist, P.hgp, P.hgm, base);
  CtaStats stats;
  const int ja = chunked ? ch * P.chunkL : 0, jb = chunked ? min(NT, ja + P.chunkL) : NT;
  if (chunked) {
    const size_t b = (size_t)ch * P.M + i;
    fx_load_fixed(st, S, P.bst + b * V, P.bsc[b]);
  } else if (!fx_load(st, S, [&](int v) { return P.q0[base + v]; })) {
    if (threadIdx.x == 0) record_error(P.status, LB_ENAN, 0);
    return;
  }
  const int R = P.pred_restart;
  const bool pred = R >= 0 && P.fxfwd, penal = H.gamma1 != 0.0;
  int* const scz = P.fxs + (size_t)i * 2 * NT;  // scale of each step's stage vector, then of each checkpoint
  // Stage vectors kept: all of them, or with checkpoints those of the last
  // segment, which the backward sweep starts with: it recomputes the others only.
  // phase 1's counters take the kept steps with the iterations they took here.
  const int jkeep = !tape ? NT : K > 0 ? (NT - 1) / K * K : 0;
  const double* const tar = reinterpret_cast<const double*>(P.tar + base) + st.im;
  double jpen = 0.0, psum = 0.0;
  FxCount cnt;
  int cur = 0;
  unsigned itkeep = 0;  // iterations before step jkeep
  fx_ctl(S, P, H.cq, ja, 0);
  for (int j = ja; j < jb; ++j) {
    if (j == jkeep) itkeep = (unsigned)stats.iters[0];
    if (penal) {
      const double pj = P.pen[j];
      psum += pj;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int v = fx_v(st, S, H, e);
        if (v < V)
          jpen = fma(pj * (fx_m(st, S, H, e) >= 0 ? 2.0 : 1.0), fx_merit(H.kind, fx_to(st.q[e], st.sc), tar[2 * v]), jpen);
      }
    }
    if (tape && K > 0 && j % K == 0) {
      long long* ck = reinterpret_cast<long long*>(P.ckpt + ((size_t)i * H.n_ckpt + j / K) * V) + st.im;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int v = fx_v(st, S, H, e);
        if (v < V) ck[2 * v] = st.q[e];
      }
      if (threadIdx.x == 0) scz[NT + j / K] = st.sc;
    }
    if (pred && R > 0 && j % R == 0) st.n = 0;
    unsigned qtop;
    long long z = 0, c = 0;
    const int it = fx_solve<E, QT, false>(st, S, P, j + 1 < jb ? j + 1 : -1, pred, cnt, cur, qtop, z, c);
    if (it < 0) {
      fx_fail(P.status, j, chunked);
      stats.flush(P.status);
      return;
    }
    stats.add(0, it);
    if (pred) fx_commit<E, QT, false>(st, S, c);
    long long* tp = nullptr;
    if (j >= jkeep)
      tp = reinterpret_cast<long long*>(K > 0 ? P.seg + ((size_t)i * K + (j - jkeep)) * V
                                              : P.ckpt + ((size_t)i * NT + j) * V);
    if (tp && threadIdx.x == 0) scz[j] = st.sc;
    fx_update(st, S, cur ? S.zb1 : S.zb0, z, tp);
    fx_rescale(st, S, qtop, pred);
  }
  if (chunked && penal) {
    const double u = fx_cta_sum(S, jpen);
    if (threadIdx.x == 0) P.jpart[(size_t)i * P.chunkC + ch] = make_double2(u, psum);
  }
  if (jb < NT) {
    stats.flush(P.status);
    return;
  }
  if (K > 0 && tape) {
    stats.iters[1] = (unsigned)stats.iters[0] - itkeep;
    stats.steps[1] = NT - jkeep;
  }
  // final state and merit functional (Sec. III)
  double acc = 0.0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int v = fx_v(st, S, H, e);
    if (v < V) {
      const int m = fx_m(st, S, H, e);
      fx_put_d(P.qT + base, v, m, st.im, st.q[e], st.sc);
      acc = fma(m >= 0 ? 2.0 : 1.0, fx_merit(H.kind, fx_to(st.q[e], st.sc), tar[2 * v]), acc);
    }
  }
  double J = merit_value(H.kind, fx_cta_sum(S, acc));
  if (penal && !chunked) {
    // sum_j pen_j merit(s_j) = merit(sum_j pen_j s_j) + merit(0) (sum_j pen_j - 1), merit affine
    const double u = fx_cta_sum(S, jpen);
    J += H.gamma1 * (merit_value(H.kind, u) + merit_value(H.kind, 0.0) * (psum - 1.0));
  }
  if (threadIdx.x == 0) P.J[i] = J;
  stats.flush(P.status);
}

}  // namespace

template <int E, int QT, int T = fx_max_threads<QT>()>
static cudaError_t run(const FixedConfig& fc, int n, cudaStream_t s, const ProbDev* p, const WorkItem* it, int tape) {
  cudaError_t e = cudaFuncSetAttribute(k_forward_fx<E, QT, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fc.smem);
  if (e != cudaSuccess) return e;
  k_forward_fx<E, QT, T><<<n, fc.threads, fc.smem, s>>>(p, it, tape);
  return cudaGetLastError();
}

FixedConfig fixed_config(int nel, int V, int Q, int units, int ncoef, int njcoef, int N, int cq) {
  FixedConfig fc{};
  if (2 * nel <= kFxPlanThreads && units <= 4) {
    fc.E = 1;
    fc.QT = units < 2 ? 2 : units;
    fc.threads = (2 * nel + 31) / 32 * 32;
  } else {
    static const int kE[] = {1, 2, 3, 5, 8};
    for (int E : kE)
      if ((long long)E * (kFxTabThreads / 2) >= nel) {
        fc.E = E;
        break;
      }
    if (!fc.E) return FixedConfig{};
    fc.QT = 0;
    fc.threads = ((2 * nel + fc.E - 1) / fc.E + 31) / 32 * 32;
    if (fc.threads < 64) fc.threads = 64;  // the first 4 Q and cq + 1 threads have work of their own
  }
  fc.smem = fx_smem_bytes(ncoef, njcoef, N, V, Q, cq, fc.E * (fc.threads / 2), fc.QT);
  // (one mode of 59 levels and more, 63 under the Hermitian symmetry: its decay
  // tables take up to 64 KB beside the state's 128; the FP64 sweep ends at 58)
  return fc.smem <= kFxMaxSmem ? fc : FixedConfig{};
}

cudaError_t launch_forward_fixed_chunked(const ProbDev* d_prob, int n_ctas, int tape, const FixedConfig& fc,
                                         cudaStream_t s) {
  switch (fc.QT) {
    case 2: return run<1, 2>(fc, n_ctas, s, d_prob, nullptr, tape);
    case 3: return run<1, 3>(fc, n_ctas, s, d_prob, nullptr, tape);
    case 4: return run<1, 4>(fc, n_ctas, s, d_prob, nullptr, tape);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_forward_fixed(const ProbDev* d_probs, const WorkItem* d_items, int n_items, int tape,
                                 const FixedConfig& fc, cudaStream_t s) {
  switch (fc.QT) {
    case 2: return run<1, 2>(fc, n_items, s, d_probs, d_items, tape);
    case 3: return run<1, 3>(fc, n_items, s, d_probs, d_items, tape);
    case 4: return run<1, 4>(fc, n_items, s, d_probs, d_items, tape);
    default: break;
  }
  switch (fc.E) {
    case 1:
      return fc.threads <= kFxTabFew ? run<1, 0, kFxTabFew>(fc, n_items, s, d_probs, d_items, tape)
                                     : run<1, 0>(fc, n_items, s, d_probs, d_items, tape);
    case 2: return run<2, 0>(fc, n_items, s, d_probs, d_items, tape);
    case 3: return run<3, 0>(fc, n_items, s, d_probs, d_items, tape);
    case 5: return run<5, 0>(fc, n_items, s, d_probs, d_items, tape);
    case 8: return run<8, 0>(fc, n_items, s, d_probs, d_items, tape);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lbk
