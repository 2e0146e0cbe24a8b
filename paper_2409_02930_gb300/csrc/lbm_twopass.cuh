// Two-pass form of the step, and the macroscopic fields for lbm_moments.
//
// 2-D nodes hold their 5 x 9 (or fewer) streamed populations in registers
// (pull_node: every load independent and in flight at once).  D3Q27 steps run
// split by lattice (lbm_split3d.cuh); here they only take their moments.
#pragma once

#include "lbm_compact.cuh"

namespace lbm {

// Macro fields that the neighbours' gradients need -- u, Pi_alpha of Eq. 45
// and Y_a (Eq. 59): put(field, value), fields u [D], Pi [D], Y [M].
template <class R, int D, int M, bool EN, class Put>
LBM_HD void macro_fields(const State<R, D, M>& s, Put&& put) {
#pragma unroll
  for (int b = 0; b < D; ++b) {
    put(b, s.u(b));
    put(D + b, s.Pi(b));
  }
  if (EN) {
#pragma unroll
    for (int k = 0; k < M; ++k) put(2 * D + k, s.Y[k]);
  }
}

// Pass 1: macro fields of node n to global memory.
template <class R, int D, int M, bool EN>
LBM_HD void macro_node(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, int n) {
  int x, y, z;
  node_xyz<R, D>(p, n, x, y, z);
  R P[(M + 1 + (EN ? 1 : 0)) * Lat<D>::Q];
  pull_node<R, D, M, EN>(p, it, a.src, a.phi, x, y, z, P);
  Moments<R, D, M, EN, false> mo;
  moments_gen<R, D, M, EN, false>(ArrayPull<R, D>{P}, mo);
  State<R, D, M> s;
  s.template from_moments<EN, false>(p, mo, a.phi[n], EN ? R(0) : a.Tfix[n]);
  macro_fields<R, D, M, EN>(s, [&](int k, const R& v) { a.mac[(size_t)k * p.N + n] = v; });
}

template <class R, int D, int M, bool EN>
__global__ void __launch_bounds__(256) k_macro(Params<R> p, InletTables<R> it, StepArgs<R> a) {
  after_previous();
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n < p.N) macro_node<R, D, M, EN>(p, it, a, n);
}

// Pass 2: full node update reading the neighbours' macro fields from global
// memory.
template <class R, int D, int M, bool EN>
LBM_HD void collide_node(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, int n) {
  int x, y, z;
  node_xyz<R, D>(p, n, x, y, z);
  R P[(M + 1 + (EN ? 1 : 0)) * Lat<D>::Q];
  pull_node<R, D, M, EN>(p, it, a.src, a.phi, x, y, z, P);
  ArrayPull<R, D> pf{P};
  Moments<R, D, M, EN, true> mo;
  moments_gen<R, D, M, EN, true>(pf, mo);
  State<R, D, M> s;
  s.template from_moments<EN, true>(p, mo, a.phi[n], EN ? R(0) : a.Tfix[n]);
  Grad<R, D, M, EN> gr;
  const R* __restrict__ mac = a.mac;
  const int N = p.N;
  gr.compute(p, x, y, [&](int k, int nb) { return mac[(size_t)k * N + nb]; });
  collide_gen<R, D, M, EN>(p, pf, n, mo, s, gr, a.dst, a.status);
}

template <class R, int D, int M, bool EN>
__global__ void __launch_bounds__(256) k_collide(Params<R> p, InletTables<R> it, StepArgs<R> a) {
  after_previous();
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n < p.N) collide_node<R, D, M, EN>(p, it, a, n);
}

// ---------------------------------------------------------------------------
// Macroscopic fields of the current state for lbm_moments.
// ---------------------------------------------------------------------------
template <class R, int D, int M, bool EN>
__global__ void __launch_bounds__(256) k_moments(Params<R> p, InletTables<R> it, StepArgs<R> a, int which,
                                                double cvel, double* __restrict__ out) {
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= p.N) return;
  const int N = p.N;
  int x, y, z;
  node_xyz<R, D>(p, n, x, y, z);
  R P[(M + 1 + (EN ? 1 : 0)) * Lat<D>::Q];
  pull_node<R, D, M, EN>(p, it, a.src, a.phi, x, y, z, P);
  Moments<R, D, M, EN, true> mo;
  moments_gen<R, D, M, EN, true>(ArrayPull<R, D>{P}, mo);
  State<R, D, M> s;
  s.template from_moments<EN, true>(p, mo, a.phi[n], EN ? R(0) : a.Tfix[n]);
  const R inv_phi = R(1) / s.phi;
  switch (which) {
    case 0:
      for (int k = 0; k < M; ++k) out[(size_t)k * N + n] = (double)(s.sa[k] * inv_phi);
      break;
    case 1:
      for (int k = 0; k < M; ++k)
        for (int b = 0; b < D; ++b) out[((size_t)k * D + b) * N + n] = (double)mo.ja[k][b];
      break;
    case 2: out[n] = (double)(s.sf * inv_phi); break;
    case 3:
      for (int b = 0; b < D; ++b) out[(size_t)b * N + n] = (double)s.u(b);
      break;
    case 4: out[n] = (double)s.T; break;
    case 5: out[n] = (double)(s.sf * inv_phi * (s.Rg * s.T)) * cvel * cvel; break;      // Eq. 3
    case 6:
    case 7: {
      Transport<R, D, M> tr;
      tr.compute(p, s, inv_phi, &mo.ja[0][0], mo.sabs);
      for (int k = 0; k < M; ++k)
        for (int b = 0; b < D; ++b) {
          double v = (double)(s.phi * tr.v[k][b]);
          if (which == 7) v = (double)(s.sa[k] * inv_phi) * ((double)s.u(b) + v) * cvel / (double)p.m[k];
          out[((size_t)k * D + b) * N + n] = v;
        }
      break;
    }
    case 9: out[n] = (double)(s.ss * inv_phi); break;
    default: break;
  }
}

}  // namespace lbm
