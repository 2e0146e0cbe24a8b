// D2Q9 two-pass form with the node's streamed populations staged in shared
// memory (variants 6 and 7).  Every thread issues the asynchronous copies of
// all its pulled populations (9 L of them; the pull addresses already hold
// the periodic wrap and the bounce-back rule; reservoir ghosts are computed
// and stored directly), waits once, and works from shared memory.
#pragma once

#include "lbm_march2d.cuh"

namespace lbm {

// populations per node
template <int M, bool EN>
constexpr int n_pops2() {
  return (M + 1 + (EN ? 1 : 0)) * 9;
}

// Stages the pulled populations of node (x, y) into col[(l*9 + i) * stride].
template <class R, int M, bool EN>
__device__ __forceinline__ void stage_node(const Params<R>& p, const InletTables<R>& it, const R* __restrict__ src,
                                           const Site<R, 2>& st, const Ghost<R, 2>& gh, R* col, int stride) {
  constexpr int Q = 9, L = M + 1 + (EN ? 1 : 0);
  const unsigned N = (unsigned)p.N;
  const bool ghost = st.has_ghost();
  const int out = ghost ? (gh.side == 0 ? 1 : -1) : 0;   // c_x of the missing directions
#pragma unroll 1
  for (int cy = -1; cy <= 1; ++cy) {
#pragma unroll
    for (int cx = -1; cx <= 1; ++cx) {
      if (cx != 0 && cx == out) continue;
      const int i = (cx + 1) + 3 * (cy + 1);
      const int h = st.source(cx, cy, 0);
      const int node = h >= 0 ? h : -1 - h;          // bounce-back: the node's own opposite population
      const R* q = src + (size_t)(unsigned)(h >= 0 ? i : Q - 1 - i) * N + node;
      R* c = col + i * stride;
#pragma unroll
      for (int l = 0; l < L; ++l) cp_async_ca<sizeof(R)>(c + l * Q * stride, q + (size_t)(unsigned)(l * Q) * N);
    }
  }
  if (ghost) {
    ghost_face<R, 2, M, EN>(p, it, gh, [&](int l, int cy, int, const R& v) {
      col[(l * Q + (out + 1) + 3 * (cy + 1)) * stride] = v;
    });
  }
  cp_async_commit();
  cp_async_wait<0>();
}

// Moments, state and gradient inputs of a staged node.
template <class R, int M, bool EN>
__device__ __forceinline__ void staged_state(const Params<R>& p, const StepArgs<R>& a, const SmemPull<R, 2>& pf,
                                             int n, int x, int y, Moments<R, 2, M, EN, true>& mo,
                                             State<R, 2, M>& s, Grad<R, 2, M, EN>& gr) {
  moments_gen<R, 2, M, EN, true>(pf, mo);
  s.template from_moments<EN, true>(p, mo, a.phi[n], EN ? R(0) : a.Tfix[n]);
  const R* __restrict__ mac = a.mac;
  const int N = p.N;
  gr.compute(p, x, y, [&](int k, int nb) { return mac[(size_t)k * N + nb]; });
}

// Macro fields of node n (u, Pi_alpha, Y_a for the neighbours' gradients)
// from its populations staged in col[(l*9 + i) * stride].
template <class R, int M, bool EN>
__device__ __forceinline__ void macro_staged_node(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a,
                                                  int n, R* col, int stride) {
  int x, y, z;
  node_xyz<R, 2>(p, n, x, y, z);
  Site<R, 2> st;
  st.init(p, x, y, z);
  Ghost<R, 2> gh;
  gh.side = -1;
  if (st.has_ghost()) ghost_velocity<R, 2, M>(p, a.src, a.phi, x, y, z, gh);
  stage_node<R, M, EN>(p, it, a.src, st, gh, col, stride);
  SmemPull<R, 2> pf{col, stride};
  Moments<R, 2, M, EN, false> mo;
  moments_gen<R, 2, M, EN, false>(pf, mo);
  State<R, 2, M> s;
  s.template from_moments<EN, false>(p, mo, a.phi[n], EN ? R(0) : a.Tfix[n]);
  const size_t N = p.N;
  macro_fields<R, 2, M, EN>(s, [&](int k, const R& v) { a.mac[(size_t)k * N + n] = v; });
}

// Node update of node n from its staged populations.
template <class R, int M, bool EN>
__device__ __forceinline__ void collide_staged_node(const Params<R>& p, const InletTables<R>& it,
                                                    const StepArgs<R>& a, int n, R* col, int stride) {
  int x, y, z;
  node_xyz<R, 2>(p, n, x, y, z);
  Site<R, 2> st;
  st.init(p, x, y, z);
  Ghost<R, 2> gh;
  gh.side = -1;
  if (st.has_ghost()) ghost_velocity<R, 2, M>(p, a.src, a.phi, x, y, z, gh);
  stage_node<R, M, EN>(p, it, a.src, st, gh, col, stride);
  SmemPull<R, 2> pf{col, stride};
  Moments<R, 2, M, EN, true> mo;
  State<R, 2, M> s;
  Grad<R, 2, M, EN> gr;
  staged_state<R, M, EN>(p, a, pf, n, x, y, mo, s, gr);
  collide_gen<R, 2, M, EN>(p, pf, n, mo, s, gr, a.dst, a.status);
}

// Macro-field pass from staged populations.
template <class R, int M, bool EN, int TB>
__global__ void __launch_bounds__(TB) k_macro_staged(Params<R> p, InletTables<R> it, StepArgs<R> a) {
  extern __shared__ unsigned char smem_raw[];
  const int n = blockIdx.x * TB + threadIdx.x;
  if (n >= p.N) return;
  macro_staged_node<R, M, EN>(p, it, a, n, reinterpret_cast<R*>(smem_raw) + threadIdx.x, TB);
}

template <class R, int M, bool EN, int TB>
__global__ void __launch_bounds__(TB) k_collide_staged(Params<R> p, InletTables<R> it, StepArgs<R> a) {
  extern __shared__ unsigned char smem_raw[];
  const int n = blockIdx.x * TB + threadIdx.x;
  if (n >= p.N) return;
  collide_staged_node<R, M, EN>(p, it, a, n, reinterpret_cast<R*>(smem_raw) + threadIdx.x, TB);
}

}  // namespace lbm
