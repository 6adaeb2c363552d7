#pragma once

// What the grid-wide cooperative sweeps share (FP64 and fixed point): the grid
// barrier and the walk over the elements of all states.

#include "lb_device.cuh"

namespace lbk {

namespace {

// ---------------------------------------------------------------------------
// grid-wide persistent sweeps (states too large for one CTA's shared memory)
//
// One cooperative launch keeps every SM busy on all M states at once.  Block
// b owns a contiguous chunk of the flattened [M][V] element range; each inner
// iteration reads the previous iterate of every element (neighbours through
// L1, see kNbL2) and ends with a grid barrier.  Per-state maxima of
// |z_new - z| and |q| are combined with atomicMax on the integer bit patterns
// (order independent), so every block takes the same stopping decision and a
// recompute is bit-identical.

constexpr long long kSpinLimit = 1LL << 26;  // ~seconds of polling before a barrier gives up

// Neighbour reads of the iterates go through L1 (kNbL2 = false): each value
// is read by up to 1 + 5Q elements, most of them in the same block's chunk.
// The iterates are rewritten by other blocks between iterations; every such
// read follows a grid_sync, whose fence after the wait (acquire, GPU scope)
// makes the writes of the previous iteration visible to ordinary loads (the
// ordering cooperative groups' grid sync provides with the same pattern).
constexpr bool kNbL2 = false;

// Grid barrier with a bounded wait: at most `limit` polls (kSpinLimit unless
// the handle set another bound, lb_set_wait_limit).  Returns false on every
// block once a wait has given up (the kernel then returns).
__device__ bool grid_sync(GridBar* bar, unsigned nblocks, long long limit) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* vgen = &bar->gen;
    volatile int* verr = &bar->err;
    const unsigned g = *vgen;
    __threadfence();
    const unsigned arrived = atomicAdd(&bar->count, 1u);
    int ok = 1;
    if (arrived == nblocks - 1) {
      atomicExch(&bar->count, 0u);
      __threadfence();
      atomicAdd(&bar->gen, 1u);
    } else {
      long long spins = 0;
      while (*vgen == g) {
        if (*verr) {
          ok = 0;
          break;
        }
        __nanosleep(64);
        if (++spins > limit) {
          atomicExch(&bar->err, 1);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
    if (*verr) ok = 0;
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

struct GridHdr {
  Hdr h;
  int M;
  int herm;         // Hermitian symmetry: only elements k <= l are iterated and stored
  int Vh;           // elements per state in the loops and in the sweep's own buffers: V, or N (N + 1) / 2
  long long total;  // M * Vh
  long long chunk;  // elements per block
};

// Element e of a grid sweep's loops: state b, vec index v = k + N l, and i,
// its place in the state's slab of the sweep's own buffers (iterates,
// adjoint, recomputed state, checkpoints, segment tape, predictor rings).
// Without the symmetry the slab is the vec layout (i = v).  With it the loops
// visit k <= l only ((k, l) from the table hkl) and the slabs hold those entries
// packed, column by column (i = l (l + 1)/2 + k); vm is then the mirror index
// l + N k of an off-diagonal element in the vec layout of the inputs and
// outputs (q0, targets, final states), whose value is the conjugate (-1 for
// diagonal elements and without the symmetry).
struct GEl {
  int b, v, vm, i, k, l;
};
// element i of state b's slab
__device__ __forceinline__ GEl gel_at(const GridHdr& G, const uint32_t* __restrict__ hkl, int b, int i) {
  GEl r;
  const int N = G.h.N;
  r.b = b;
  r.i = i;
  if (!G.herm) {
    r.v = i;
    r.vm = -1;
    r.k = i % N;
    r.l = i / N;
    return r;
  }
  const uint32_t t = __ldg(hkl + i);
  r.k = (int)(t & 0xffffu);
  r.l = (int)(t >> 16);
  r.v = r.k + N * r.l;
  r.vm = r.k != r.l ? r.l + N * r.k : -1;
  return r;
}

// A thread's walk over its elements e = e0 + threadIdx.x, + blockDim.x, ...
// of a block's chunk [e0, e1) of the flattened [M][Vh] range, keeping the
// state b and slab index i of e (one division at the start).
struct GIter {
  long long e;
  int b, i;
  __device__ GIter(const GridHdr& G, long long e_start) : e(e_start) {
    b = (int)(e / G.Vh);
    i = (int)(e - (long long)b * G.Vh);
  }
  __device__ __forceinline__ void next(const GridHdr& G, int step) {
    e += step;
    i += step;
    while (i >= G.Vh) {
      i -= G.Vh;
      ++b;
    }
  }
};

// offset of element g in slab `slab` (state b's, or a checkpoint's) of a sweep buffer
__device__ __forceinline__ size_t gslab(const GridHdr& G, const GEl& g, size_t slab) {
  return slab * (size_t)G.Vh + g.i;
}
// store x at element g of an input/output array in the vec layout (and its mirror)
__device__ __forceinline__ void gput(double2* a, const GEl& g, int V, double2 x) {
  a[(size_t)g.b * V + g.v] = x;
  if (g.vm >= 0) a[(size_t)g.b * V + g.vm] = make_double2(x.x, -x.y);
}

}  // namespace
}  // namespace lbk
