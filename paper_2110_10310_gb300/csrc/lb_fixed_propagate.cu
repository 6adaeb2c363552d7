// Steps on given vectors in fixed point (lb_propagate), one CTA per vector.

#include "lb_fixed_sweep.cuh"

namespace lbk {

namespace {

template <int E, int QT, int T, bool ADJ>
__global__ void __launch_bounds__(T)
    k_propagate_fx(const ProbDev* __restrict__ pp, int j0, int j1, double2* __restrict__ x) {
  extern __shared__ __align__(16) unsigned char smem[];
  const ProbDev& P = *pp;
  const FxSmem S = fx_carve(smem, P, E * (blockDim.x / 2), QT);
  fx_setup(S, P, 0);  // vectors given to lb_propagate may be anything
  const Hdr& H = *S.hdr;
  const int V = H.V;
  FxState<E, QT> st;
  fx_init(st, S, P);
  double2* xv = x + (size_t)blockIdx.x * V;
  CtaStats stats;
  if (!fx_load(st, S, [&](int v) { return xv[v]; })) {
    if (threadIdx.x == 0) record_error(P.status, LB_ENAN, ADJ ? j1 - 1 : j0);
    return;
  }
  // the ring (QT == 0) lives in the system's own M states' workspace: more
  // vectors than states go without the predictor
  const bool pred = QT > 0 || (int)blockIdx.x < P.M;
  if (pred) fx_ring(st, S, P, P.hist, P.hgp, P.hgm, (size_t)blockIdx.x * V);
  FxCount cnt;
  int cur = 0;
  fx_ctl(S, P, H.cq, ADJ ? j1 - 1 : j0, 0);
  for (int jj = 0; jj < j1 - j0; ++jj) {
    const int j = ADJ ? j1 - 1 - jj : j0 + jj;
    const int jn = jj + 1 < j1 - j0 ? (ADJ ? j - 1 : j + 1) : -1;
    unsigned qtop;
    long long z = 0, c = 0;
    const int it = fx_solve<E, QT, ADJ>(st, S, P, jn, pred, cnt, cur, qtop, z, c);
    if (it < 0) {
      if (threadIdx.x == 0) record_error(P.status, LB_ENOTCONV, j);
      stats.flush(P.status);
      return;
    }
    stats.add(ADJ ? 2 : 0, it);
    if (pred) fx_commit<E, QT, ADJ>(st, S, c);
    fx_update(st, S, cur ? S.zb1 : S.zb0, z, nullptr);
    fx_rescale(st, S, qtop, pred);
  }
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int v = fx_v(st, S, H, e);
    if (v < V) fx_put_d(xv, v, -1, st.im, st.q[e], st.sc);
  }
  stats.flush(P.status);
}

}  // namespace

template <int E, int QT, int T = fx_max_threads<QT>()>
static cudaError_t run(const FixedConfig& fc, int n, cudaStream_t s, const ProbDev* p, int adj, int j0, int j1,
                       double2* x) {
  auto k = adj ? k_propagate_fx<E, QT, T, true> : k_propagate_fx<E, QT, T, false>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fc.smem);
  if (e != cudaSuccess) return e;
  k<<<n, fc.threads, fc.smem, s>>>(p, j0, j1, x);
  return cudaGetLastError();
}

cudaError_t launch_propagate_fixed(const ProbDev* d_prob, int adjoint, int64_t j0, int64_t j1, double2* x, int n_vec,
                                   const FixedConfig& fc, cudaStream_t s) {
  const int a = (int)j0, b = (int)j1;
  switch (fc.QT) {
    case 2: return run<1, 2>(fc, n_vec, s, d_prob, adjoint, a, b, x);
    case 3: return run<1, 3>(fc, n_vec, s, d_prob, adjoint, a, b, x);
    case 4: return run<1, 4>(fc, n_vec, s, d_prob, adjoint, a, b, x);
    default: break;
  }
  switch (fc.E) {
    case 1:
      return fc.threads <= kFxTabFew ? run<1, 0, kFxTabFew>(fc, n_vec, s, d_prob, adjoint, a, b, x)
                                     : run<1, 0>(fc, n_vec, s, d_prob, adjoint, a, b, x);
    case 2: return run<2, 0>(fc, n_vec, s, d_prob, adjoint, a, b, x);
    case 3: return run<3, 0>(fc, n_vec, s, d_prob, adjoint, a, b, x);
    case 5: return run<5, 0>(fc, n_vec, s, d_prob, adjoint, a, b, x);
    case 8: return run<8, 0>(fc, n_vec, s, d_prob, adjoint, a, b, x);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lbk
