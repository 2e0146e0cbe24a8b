// Arguments of the step kernels, the gradient stencil and the initial
// populations.
#pragma once

#include "lbm_launch.h"
#include "lbm_node.cuh"

namespace lbm {

// Arguments shared by the step kernels (device pointers).
template <class R>
struct StepArgs {
  const R* src;                  // post-collision populations of the previous step
  R* dst;                        // new post-collision populations
  const R* __restrict__ phi;     // porosity [N]
  const R* __restrict__ Tfix;    // fixed temperature [N] (isothermal lattices)
  R* mac;                        // macro fields for the gradients [2D+M][N]
  int* status;                   // bit 0: non-finite / non-positive density, bit 1: FP64 solve used,
                                 // bit 2: surface Newton not converged, bit 3: a bounded wait gave up
};

constexpr int kStatusTimeout = 8;   // status bit 3: a bounded device wait gave up

LBM_HD void flag(int* status, int bit) {
#ifdef __CUDA_ARCH__
  atomicOr(status, bit);
#else
  *status |= bit;
#endif
}

template <class R, int D>
LBM_HD void node_xyz(const Params<R>& p, int n, int& x, int& y, int& z) {
  x = n % p.nx;
  int r = n / p.nx;
  y = r % p.ny;
  z = (D == 3) ? r / p.ny : 0;
}

// Gradient inputs of a node; compute() takes them from the neighbours' macro
// fields on a D2Q9 lattice (isotropic stencil; zero-gradient copy across
// non-periodic x faces).  D3Q27 differentiates in lbm_split3d.cuh.
template <class R, int D, int M, bool EN>
struct Grad {
  R divu, dPi[D], dY[M][D];
  template <class Fetch>
  LBM_HD void compute(const Params<R>& p, int x, int y, Fetch&& fetch) {
    static_assert(D == 2, "the gather stencil is a 2-D form");
    divu = R(0);
#pragma unroll
    for (int b = 0; b < D; ++b) {
      dPi[b] = R(0);
#pragma unroll
      for (int k = 0; k < M; ++k) dY[k][b] = R(0);
    }
    Unroll<0, 9>::run([&](auto ic) {
      constexpr int I = decltype(ic)::value;
      if (csq_of<D>(I) == 0) return;
      const R w = grad_w<R, D>(I);
      int sx = x + c_of<D>(I, 0);
      if (sx < 0) sx = (p.bc_lo == BC_PERIODIC) ? sx + p.nx : 0;
      if (sx >= p.nx) sx = (p.bc_hi == BC_PERIODIC) ? sx - p.nx : p.nx - 1;
      const int nb = sx + p.nx * wrapi(y + c_of<D>(I, 1), p.ny);
#pragma unroll
      for (int b = 0; b < D; ++b) {
        const int cb = c_of<D>(I, b);
        if (cb == 0) continue;
        const R wc = w * R(cb);
        divu += wc * fetch(b, nb);
        dPi[b] += wc * fetch(D + b, nb);
        if (EN) {
#pragma unroll
          for (int k = 0; k < M; ++k) dY[k][b] += wc * fetch(2 * D + k, nb);
        }
      }
    });
  }
};

// ---------------------------------------------------------------------------
// Initial populations: equilibria of the initial fields (Eq. 15, Eq. 44
// without extension, Eq. 51).
// ---------------------------------------------------------------------------
// Initial populations of node n: equilibria of the initial fields (Eq. 15,
// Eq. 44 without extension, Eq. 51).  R is the computing type, PR the
// parameter type; store(l, i, value).
template <class R, int D, int M, bool EN, class PR, class Store>
LBM_HD void init_node(const PR& p, const double* __restrict__ X, const double* __restrict__ T0,
                      const double* __restrict__ P0, const double* __restrict__ U0v, double cvel, double RU_si,
                      int n, int N, R phi, Store&& store) {
  constexpr int Q = Lat<D>::Q;
  R T = (R)T0[n];
  R rho_a[M], rho = R(0), inv_m = R(0);
#pragma unroll
  for (int a = 0; a < M; ++a) {
    // rho_a = P X_a m_a / (R_U T)  (Dalton and the ideal-gas law, Sec. 2.1)
    rho_a[a] = (R)(P0[n] * X[(size_t)a * N + n] * (double)p.m[a] / (RU_si * T0[n]));
    rho += rho_a[a];
  }
#pragma unroll
  for (int a = 0; a < M; ++a) inv_m += (rho_a[a] / rho) / R(p.m[a]);
  R Rg = R(p.RU) * inv_m;
  R u[D], w[D];
#pragma unroll
  for (int b = 0; b < D; ++b) {
    u[b] = U0v ? (R)(U0v[(size_t)b * N + n] / cvel) : R(0);
    w[b] = u[b] / phi;
  }
#pragma unroll
  for (int a = 0; a < M; ++a) {
    R F[D][3];
#pragma unroll
    for (int b = 0; b < D; ++b) psi3<R>(w[b], w[b] * w[b] + R(p.Ra[a]) * T, F[b]);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      R v = phi * rho_a[a];
#pragma unroll
      for (int b = 0; b < D; ++b) v *= F[b][c_of<D>(i, b) + 1];
      store(a, i, v);
    }
  }
  {
    R F[D][3];
#pragma unroll
    for (int b = 0; b < D; ++b) psi3<R>(w[b], w[b] * w[b] + Rg * T, F[b]);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      R v = phi * rho;
#pragma unroll
      for (int b = 0; b < D; ++b) v *= F[b][c_of<D>(i, b) + 1];
      store(M, i, v);
    }
  }
  if (EN) {
    R U = R(0);
#pragma unroll
    for (int a = 0; a < M; ++a) U += (rho_a[a] / rho) * (R(p.U0[a]) + R(p.cvR[a]) * (T - R(p.T_thermo)));
    GeqFactors<R, D> G;
    G.init(phi, rho, u, Rg * T, U);
    Unroll<0, Q>::run([&](auto ic) {
      constexpr int I = decltype(ic)::value;
      store(M + 1, I, G.template value<I>());
    });
  }
}

template <class R, int D, int M, bool EN>
__global__ void __launch_bounds__(256) k_init(Params<R> p, const double* __restrict__ X, const double* __restrict__ T0,
                                             const double* __restrict__ P0, const double* __restrict__ U0v,
                                             double cvel, double RU_si, R* __restrict__ dst,
                                             const R* __restrict__ phiA) {
  constexpr int Q = Lat<D>::Q;
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= p.N) return;
  const int N = p.N;
  init_node<R, D, M, EN>(p, X, T0, P0, U0v, cvel, RU_si, n, N, phiA[n],
                         [&](int l, int i, R v) { dst[(size_t)(l * Q + i) * N + n] = v; });
}

}  // namespace lbm
