// Small states over many steps: chunks of steps advanced at the same time.
//
// One CTA per state leaves a small problem bound by the dependent chain of its
// steps: a two-transmon gradient keeps 10 of 152 SMs busy, each waiting 3300
// cycles per step on latency.  A step is linear in the state, so the steps
// are cut into C chunks of L, and
//   1. every chunk's propagator is found by running its L steps from the
//      unit matrices |k><l|, k <= l (the step commutes with the conjugate
//      transpose), all chunks and columns at once;
//   2. the states at the chunk boundaries follow by C products, one CTA per
//      state (C short steps instead of N_T);
//   3. every (chunk, state) pair runs its L steps from its boundary state at
//      the same time, writing the stage tape;
//   4. the adjoint states at the boundaries follow by C products with the
//      same propagators' conjugate transposes (plus, with the running
//      penalty, each chunk's response to its own sources), and
//   5. every (chunk, state) pair runs its adjoint steps and gradient pieces.
// The results are those of the sequential sweep up to rounding.  The work
// grows by N (N + 1) / 2 columns against the M states of the problem, which
// the idle SMs and the overlap of many CTAs per SM pay for while N^2 <= 128.

#include "lb_fixed_sweep.cuh"

namespace lbk {

namespace {

constexpr int kPShift = 62;  // the propagators' entries (at most 1 in magnitude, up to the step error) as coefficients: a quarter

// columns of the chunks' propagators: CTA (chunk, column)
template <int QT>
__global__ void __launch_bounds__(2 * kFxChunkV, 3) k_columns_fx(const ProbDev* __restrict__ pp) {
  extern __shared__ __align__(16) unsigned char smem[];
  const ProbDev& P = *pp;
  const int Vc = P.N * (P.N + 1) / 2, ch = blockIdx.x / Vc, col = blockIdx.x % Vc;
  const FxSmem S = fx_carve(smem, P, blockDim.x / 2, QT);
  fx_setup(S, P, 0);
  const Hdr& H = *S.hdr;
  const int V = H.V, ja = ch * P.chunkL, jb = min(H.NT, ja + P.chunkL);
  FxState<1, QT> st;
  fx_init(st, S, P);
  const uint32_t kl = P.hkl[col];
  st.sc = kFxTop;
  st.q[0] = st.v[0] == (int)(kl & 0xffffu) + H.N * (int)(kl >> 16) && !st.im ? 1LL << kFxTop : 0;
  const int R = P.pred_restart;
  const bool pred = R >= 0;
  FxCount cnt;
  int cur = 0;
  fx_ctl(S, P, H.cq, ja, 0);
  for (int j = ja; j < jb; ++j) {
    if (pred && R > 0 && j % R == 0) st.n = 0;
    unsigned qtop;
    long long z = 0, c = 0;
    if (fx_solve<1, QT, false>(st, S, P, j + 1 < jb ? j + 1 : -1, pred, cnt, cur, qtop, z, c) < 0) {
      fx_fail(P.status, j, true);
      break;
    }
    if (pred) fx_commit<1, QT, false>(st, S, c);
    fx_update(st, S, nullptr, z, nullptr);
    fx_rescale(st, S, qtop, pred);
  }
  if (st.v[0] < V) {
    Fx* o = reinterpret_cast<Fx*>(P.pmat + ((size_t)ch * Vc + col) * V + st.v[0]);
    o[st.im] = fx_coef(fx_shift(st.q[0], st.sc - kPShift));
  }
}

// Boundary products.  One CTA per state multiplies it by the chunks' propagators
// one after another; a chunk's matrix is fetched into shared memory while the
// one before is used (two buffers; read from global memory when they do not fit),
// and every thread sums a share of a column (forward) or row (adjoint) group.
struct FxCombine {
  longlong2* part;  // [G][V] partial sums
  int4* x;          // [V] the state, split
  int* vkl;         // [Vc] vec index of column e's |k><l|
  int* vlk;         // [Vc] ... of |l><k| (-1 on the diagonal)
  unsigned long long* mx;  // [32]
  int4* mat;        // [2][Vc * V], or null
};
__host__ __device__ inline size_t fx_combine_bytes(int V, int Vc, int G, bool stage) {
  return align16(sizeof(longlong2) * (size_t)G * V) + sizeof(int4) * V + align16(sizeof(int) * Vc) * 2 +
         sizeof(unsigned long long) * 32 + (stage ? sizeof(int4) * 2 * (size_t)Vc * V : 0);
}
__device__ FxCombine fx_combine_carve(unsigned char* base, const ProbDev& P, int G, bool stage) {
  FxCombine S;
  const int V = P.V, Vc = P.N * (P.N + 1) / 2;
  size_t o = 0;
  S.part = reinterpret_cast<longlong2*>(base + o);
  o += align16(sizeof(longlong2) * (size_t)G * V);
  S.x = reinterpret_cast<int4*>(base + o);
  o += sizeof(int4) * V;
  S.vkl = reinterpret_cast<int*>(base + o);
  o += align16(sizeof(int) * Vc);
  S.vlk = reinterpret_cast<int*>(base + o);
  o += align16(sizeof(int) * Vc);
  S.mx = reinterpret_cast<unsigned long long*>(base + o);
  o += sizeof(unsigned long long) * 32;
  S.mat = stage ? reinterpret_cast<int4*>(base + o) : nullptr;
  for (int e = threadIdx.x; e < Vc; e += blockDim.x) {
    const uint32_t t = P.hkl[e];
    const int k = (int)(t & 0xffffu), l = (int)(t >> 16);
    S.vkl[e] = k + P.N * l;
    S.vlk[e] = k != l ? l + P.N * k : -1;
  }
  __syncthreads();
  return S;
}
// chunk c's matrix on its way to buffer c & 1 (c < 0 or >= C: nothing)
__device__ __forceinline__ void fx_fetch(const FxCombine& S, const ProbDev& P, int c) {
  if (!S.mat) return;
  if (c >= 0 && c < P.chunkC) {
    const int n = P.N * (P.N + 1) / 2 * P.V;
    const int4* src = P.pmat + (size_t)c * n;
    int4* dst = S.mat + (size_t)(c & 1) * n;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(dst + i));
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(src + i) : "memory");
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// wait for every matrix but the newest fetched; the matrix of chunk c
__device__ __forceinline__ const int4* fx_fetched(const FxCombine& S, const ProbDev& P, int c) {
  const size_t n = (size_t)(P.N * (P.N + 1) / 2) * P.V;
  if (!S.mat) return P.pmat + c * n;
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  __syncthreads();
  return S.mat + (c & 1) * n;
}
__device__ unsigned long long fx_block_max(unsigned long long* w, unsigned long long m) {
  m = warp_max_u64(m);
  if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = m;
  __syncthreads();
  m = 0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) m = umax64(m, w[i]);
  __syncthreads();
  return m;
}
// a += A x / 4 (conj: A^* x / 4) for split A and x, folded into 64-bit sums
// that may wrap before the last
template <bool CONJ>
__device__ __forceinline__ void fx_cmac(long long& re, long long& im, int4 A, int4 x) {
  const Fx ax{A.x, A.y}, ay{A.z, A.w}, xr{x.x, x.y}, xi{x.z, x.w};
  FxAcc r = fx_acc(), i = fx_acc();
  fx_mac(r, ax, xr);
  fx_mac(r, CONJ ? ay : fx_neg(ay), xi);
  fx_mac(i, ax, xi);
  fx_mac(i, CONJ ? fx_neg(ay) : ay, xr);
  re += fx_val(r);
  im += fx_val(i);
}
__device__ __forceinline__ int4 fx_split2(Cx q) {
  const Fx a = fx_split(q.x), b = fx_split(q.y);
  return make_int4(a.h, a.l, b.h, b.l);
}

// Take the value of entry threadIdx.x (< V, else ignored) of the next boundary
// state, at the scale sc, plus `add` (ADD): set its scale by its largest entry,
// keep it split in S.x and store it.
template <bool ADD>
__device__ void fx_boundary(const FxCombine& S, const ProbDev& P, Cx q, double2 add, int& sc, int V, size_t b) {
  const int t = threadIdx.x;
  int s = 0;
  if (ADD) {
    // the largest of state, addend and sum: the two may cancel
    unsigned long long m = 0;
    if (t < V) {
      const double2 x = make_double2(fx_to(q.x, sc), fx_to(q.y, sc));
      m = umax64(umax64(abs_bits(x.x), abs_bits(x.y)), umax64(abs_bits(add.x), abs_bits(add.y)));
      m = umax64(m, umax64(abs_bits(x.x + add.x), abs_bits(x.y + add.y)));
    }
    const unsigned long long mx = fx_block_max(S.mx, m);
    if (mx && mx < kInfBits) s = sc - fx_scale(mx);
  } else {
    unsigned* w = reinterpret_cast<unsigned*>(S.mx);
    const unsigned m = __reduce_max_sync(kFull, t < V ? max(fx_hi_abs(q.x), fx_hi_abs(q.y)) : 0u);
    if ((t & 31) == 0) w[t >> 5] = m;
    __syncthreads();
    const unsigned top = __reduce_max_sync(kFull, (t & 31) < (int)(blockDim.x >> 5) ? w[t & 31] : 0u);
    s = fx_quarter_shift(top);
  }
  sc -= s;
  if (t < V) {
    q.x = fx_shift(q.x, s);
    q.y = fx_shift(q.y, s);
    if (ADD) {
      q.x += fx_from(add.x, sc);
      q.y += fx_from(add.y, sc);
    }
    S.x[t] = fx_split2(q);
    P.bst[b * V + t] = make_longlong2(q.x, q.y);
  }
  if (t == 0) P.bsc[b] = sc;
  __syncthreads();
}
// entry threadIdx.x of the product from the G partial sums: a quarter of it.
// A chunk can raise the largest entry (a uniform superposition turned into a
// basis state: up to N times), so the sum stays a quarter, its scale 2 less,
// until fx_boundary has seen its size.
__device__ __forceinline__ Cx fx_take(const FxCombine& S, int G, int V) {
  Cx q{0, 0};
  if ((int)threadIdx.x < V) {
    for (int k = 0; k < G; ++k) {
      const longlong2 p = S.part[k * V + threadIdx.x];
      q.x += p.x;
      q.y += p.y;
    }
  }
  return q;
}

// boundary states: thread (g, v) sums entry v over the columns e = g, g + G, ...
__global__ void __launch_bounds__(1024) k_boundary_fx(const ProbDev* __restrict__ pp, int G, int stage) {
  extern __shared__ __align__(16) unsigned char smem[];
  const ProbDev& P = *pp;
  const int V = P.V, N = P.N, Vc = N * (N + 1) / 2, M = P.M, i = blockIdx.x, t = threadIdx.x;
  const FxCombine S = fx_combine_carve(smem, P, G, stage);
  fx_fetch(S, P, 0);
  const double2 q0 = t < V ? P.q0[(size_t)i * V + t] : make_double2(0.0, 0.0);
  const unsigned long long mx = fx_block_max(S.mx, umax64(abs_bits(q0.x), abs_bits(q0.y)));
  const bool bad = mx >= kInfBits;
  if (bad && t == 0) record_error(P.status, LB_ENAN, 0);
  int sc = kFxTop;
  fx_boundary<true>(S, P, Cx{0, 0}, bad ? make_double2(0.0, 0.0) : q0, sc, V, i);
  const int g = t / V, v = t - g * V, vt = v / N + N * (v % N);
  for (int c = 0; c < P.chunkC; ++c) {
    fx_fetch(S, P, c + 1);
    const int4* A = fx_fetched(S, P, c);
    if (g < G) {
      long long re = 0, im = 0;
#pragma unroll 4
      for (int e = g; e < Vc; e += G) {
        const int lk = S.vlk[e];
        const int4 a = A[(size_t)e * V + v], at = A[(size_t)e * V + vt];
        fx_cmac<false>(re, im, a, S.x[S.vkl[e]]);
        if (lk >= 0) fx_cmac<true>(re, im, at, S.x[lk]);
      }
      S.part[g * V + v] = make_longlong2(re, im);
    }
    __syncthreads();
    sc -= 2;
    fx_boundary<false>(S, P, fx_take(S, G, V), make_double2(0.0, 0.0), sc, V, (size_t)(c + 1) * M + i);
  }
}

// adjoint states at the boundaries: thread (e, g) sums the products with
// columns |k><l| and |l><k| of pair e over the entries v = g, g + G, ...
__global__ void __launch_bounds__(1024) k_boundary_adj_fx(const ProbDev* __restrict__ pp, int G, int stage) {
  extern __shared__ __align__(16) unsigned char smem[];
  const ProbDev& P = *pp;
  const int V = P.V, N = P.N, Vc = N * (N + 1) / 2, M = P.M, i = blockIdx.x, t = threadIdx.x;
  const FxCombine S = fx_combine_carve(smem, P, G, stage);
  const size_t base = (size_t)i * V, C1 = P.chunkC + 1;
  fx_fetch(S, P, P.chunkC - 1);
  // terminal condition qhat^{N_T} = beta_i/M g_i (Appendix B)
  double2 lam = make_double2(0.0, 0.0);
  if (t < V) {
    const double w = P.wgt[i];
    const double2 tar = P.tar[base + t];
    if (P.kind == LB_J_FROB) {
      const double2 qq = P.qT[base + t];
      lam = make_double2(w * (qq.x - tar.x), w * (qq.y - tar.y));
    } else {
      const double wt = linear_sign(P.kind) * w;
      lam = make_double2(wt * tar.x, wt * tar.y);
    }
  }
  const unsigned long long mx = fx_block_max(S.mx, umax64(abs_bits(lam.x), abs_bits(lam.y)));
  const bool bad = mx >= kInfBits;
  if (bad && t == 0) record_error(P.status, LB_ENAN, P.NT - 1);
  int sc = kFxTop;
  fx_boundary<true>(S, P, Cx{0, 0}, bad ? make_double2(0.0, 0.0) : lam, sc, V, (C1 + P.chunkC) * M + i);
  const int e = t / G, g = t - e * G;
  for (int c = P.chunkC - 1; c >= 0; --c) {
    fx_fetch(S, P, c - 1);
    const int4* A = fx_fetched(S, P, c);
    if (e < Vc) {
      // <P(|k><l|), lam> and <P(|l><k|), lam>
      long long ar = 0, ai = 0, br = 0, bi = 0;
#pragma unroll 3
      for (int v = g; v < V; v += G) {
        const int4 a = A[(size_t)e * V + v];
        fx_cmac<true>(ar, ai, a, S.x[v]);
        fx_cmac<false>(br, bi, a, S.x[v / N + N * (v % N)]);
      }
      S.part[g * V + S.vkl[e]] = make_longlong2(ar, ai);
      if (S.vlk[e] >= 0) S.part[g * V + S.vlk[e]] = make_longlong2(br, bi);
    }
    __syncthreads();
    const Cx q = fx_take(S, G, V);
    sc -= 2;
    if (P.gamma1 != 0.0) {
      // the chunk's response to its own penalty sources
      double2 add = make_double2(0.0, 0.0);
      if (t < V) {
        const size_t b = (2 * C1 + c) * M + i;
        const longlong2 r = P.bst[b * V + t];
        add = make_double2(fx_to(r.x, P.bsc[b]), fx_to(r.y, P.bsc[b]));
      }
      fx_boundary<true>(S, P, q, add, sc, V, (C1 + c) * M + i);
    } else {
      fx_boundary<false>(S, P, q, make_double2(0.0, 0.0), sc, V, (C1 + c) * M + i);
    }
  }
}

// J_i with the running penalty's sums of all chunks (in chunk order)
__global__ void k_penalty_fx(const ProbDev* __restrict__ pp) {
  const ProbDev& P = *pp;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P.M) return;
  double u = 0.0, ps = 0.0;
  for (int c = 0; c < P.chunkC; ++c) {
    const double2 p = P.jpart[(size_t)i * P.chunkC + c];
    u += p.x;
    ps += p.y;
  }
  P.J[i] += P.gamma1 * (merit_value(P.kind, u) + merit_value(P.kind, 0.0) * (ps - 1.0));
}

template <int QT>
cudaError_t run_columns(const ProbDev* p, int n, const FixedConfig& fc, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k_columns_fx<QT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fc.smem);
  if (e != cudaSuccess) return e;
  k_columns_fx<QT><<<n, fc.threads, fc.smem, s>>>(p);
  return cudaGetLastError();
}

// thread groups of a boundary product: 1024 threads over the V entries
// (forward), or up to 16 per pair of columns (adjoint)
int boundary_groups(int V, int Vc) {
  const int g = 1024 / V;
  return g < 1 ? 1 : (g < Vc ? g : Vc);
}
int boundary_groups_adj(int V, int Vc) {
  int g = 1024 / Vc;
  if (g > 16) g = 16;
  return g < V ? g : V;
}
// whether two matrices fit shared memory with G groups' sums, and the bytes
template <class K>
cudaError_t boundary_shape(K kern, int V, int Vc, int G, int* stage, size_t* smem) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  *stage = fx_combine_bytes(V, Vc, G, true) <= (size_t)optin;
  *smem = fx_combine_bytes(V, Vc, G, *stage);
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*smem);
}

}  // namespace

cudaError_t launch_forward_chunks(const ProbDev* d_prob, const ProbDev& h, int tape, const FixedConfig& fc,
                                  cudaStream_t s) {
  const int Vc = h.N * (h.N + 1) / 2, n = h.chunkC * Vc;
  cudaError_t e;
  switch (fc.QT) {
    case 2: e = run_columns<2>(d_prob, n, fc, s); break;
    case 3: e = run_columns<3>(d_prob, n, fc, s); break;
    case 4: e = run_columns<4>(d_prob, n, fc, s); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  const int G = boundary_groups(h.V, Vc);
  int stage = 0;
  size_t smem = 0;
  e = boundary_shape(k_boundary_fx, h.V, Vc, G, &stage, &smem);
  if (e != cudaSuccess) return e;
  k_boundary_fx<<<h.M, (G * h.V + 31) / 32 * 32, smem, s>>>(d_prob, G, stage);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = launch_forward_fixed_chunked(d_prob, h.M * h.chunkC, tape, fc, s);
  if (e != cudaSuccess || h.gamma1 == 0.0) return e;
  k_penalty_fx<<<(h.M + 31) / 32, 32, 0, s>>>(d_prob);
  return cudaGetLastError();
}

cudaError_t launch_backward_chunks(const ProbDev* d_prob, const ProbDev& h, const FixedConfig& fc, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  if (h.gamma1 != 0.0) e = launch_backward_fixed_chunked(d_prob, h.M * h.chunkC, 1, fc, s);
  if (e != cudaSuccess) return e;
  const int Vc = h.N * (h.N + 1) / 2;
  const int G = boundary_groups_adj(h.V, Vc);
  int stage = 0;
  size_t smem = 0;
  e = boundary_shape(k_boundary_adj_fx, h.V, Vc, G, &stage, &smem);
  if (e != cudaSuccess) return e;
  k_boundary_adj_fx<<<h.M, (G * Vc + 31) / 32 * 32, smem, s>>>(d_prob, G, stage);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_backward_fixed_chunked(d_prob, h.M * h.chunkC, 0, fc, s);
}

}  // namespace lbk
