// Fused single-kernel D2Q9 time step (variant 5).
//
// A block owns TX columns and marches over SEG rows.  For every row it first
// recomputes, from the streamed populations, the macroscopic fields that the
// isotropic gradients need (u, Pi_alpha of Eq. 45, Y_a) on the row plus a
// one-node halo, into a rolling shared-memory ring of three rows; then it
// collides the nodes of the previous row, whose stencil now lies entirely in
// the ring.  No macro field goes through global memory, so the populations are
// read from HBM about once per step (the halo re-reads hit L2) and written
// once.
#pragma once

#include "lbm_tile2d.cuh"

namespace lbm {

// macro fields of a node that its neighbours' gradients need
template <int M, bool EN>
LBM_HD constexpr int n_macro2() { return 4 + (EN ? M : 0); }

template <class R, int M, bool EN, int TX>
constexpr size_t fused_smem_bytes() {
  return sizeof(R) * 3 * n_macro2<M, EN>() * (TX + 2);
}

template <class R, int M, bool EN, int TX, int SEG>
__global__ void __launch_bounds__(TX) k_fused(Params<R> p, InletTables<R> it, StepArgs<R> a) {
  constexpr int PX = TX + 2;
  constexpr int NF = n_macro2<M, EN>();
  constexpr int LQ = (M + 1 + (EN ? 1 : 0)) * 9;
  extern __shared__ unsigned char smem_raw[];
  R* ring = reinterpret_cast<R*>(smem_raw);           // [3][NF][PX]

  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * SEG;
  const int yend = min(y0 + SEG, p.ny);
  const int tx = threadIdx.x;

  // macro fields of one extended row into a ring slot
  auto compute_row = [&](int row, int slot) {
    const int y = modp(row, p.ny);
    R* dstp = ring + (size_t)slot * NF * PX;
    for (int e = tx; e < PX; e += TX) {
      int x = x0 - 1 + e;
      if (x < 0 || x >= p.nx) {
        const int bc = x < 0 ? p.bc_lo : p.bc_hi;
        x = (bc == BC_PERIODIC) ? modp(x, p.nx) : (x < 0 ? 0 : p.nx - 1);   // zero-gradient ghost
      }
      const int n = x + p.nx * y;
      R P[LQ];
      pull_node<R, 2, M, EN>(p, it, a.src, a.phi, x, y, 0, P);
      Moments<R, 2, M, EN, false> mo;
      moments_gen<R, 2, M, EN, false>(ArrayPull<R, 2>{P}, mo);
      State<R, 2, M> s;
      s.template from_moments<EN, false>(p, mo, a.phi[n], EN ? R(0) : a.Tfix[n]);
      macro_fields<R, 2, M, EN>(s, [&](int k, const R& v) { dstp[k * PX + e] = v; });
    }
  };
  auto slot_of = [](int r) { return (r + 1) % 3; };    // r = y - y0 in [-1, SEG]

  const int x = x0 + tx;
  const bool active = x < p.nx;

  compute_row(y0 - 1, slot_of(-1));
  compute_row(y0, slot_of(0));
  for (int r = 0; r < yend - y0; ++r) {
    compute_row(y0 + r + 1, slot_of(r + 1));
    __syncthreads();
    if (active) {
      const int y = y0 + r, n = x + p.nx * y;
      R P[LQ];
      pull_node<R, 2, M, EN>(p, it, a.src, a.phi, x, y, 0, P);
      ArrayPull<R, 2> pf{P};
      Moments<R, 2, M, EN, true> mo;
      moments_gen<R, 2, M, EN, true>(pf, mo);
      State<R, 2, M> s;
      s.template from_moments<EN, true>(p, mo, a.phi[n], EN ? R(0) : a.Tfix[n]);
      // gradient inputs from the ring (isotropic stencil, weights 3 w_i)
      Grad<R, 2, M, EN> gr;
      gr.divu = R(0);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        gr.dPi[b] = R(0);
#pragma unroll
        for (int k = 0; k < M; ++k) gr.dY[k][b] = R(0);
      }
      Unroll<0, 9>::run([&](auto ic) {
        constexpr int I = decltype(ic)::value;
        constexpr int cx = c_of<2>(I, 0), cy = c_of<2>(I, 1);
        if (csq_of<2>(I) == 0) return;
        const R w = R(3) * (cx == 0 ? R(2) / R(3) : R(1) / R(6)) * (cy == 0 ? R(2) / R(3) : R(1) / R(6));
        const int e = tx + 1 + cx;
        const R* src_row = ring + (size_t)slot_of(r + cy) * NF * PX;
        const int cc[2] = {cx, cy};
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          if (cc[b] == 0) continue;
          const R wc = w * R(cc[b]);
          gr.divu += wc * src_row[b * PX + e];
          gr.dPi[b] += wc * src_row[(2 + b) * PX + e];
          if (EN) {
#pragma unroll
            for (int k = 0; k < M; ++k) gr.dY[k][b] += wc * src_row[(4 + k) * PX + e];
          }
        }
      });
      collide_gen<R, 2, M, EN>(p, pf, n, mo, s, gr, a.dst, a.status);
    }
    __syncthreads();
  }
}

}  // namespace lbm
