// Single-launch D2Q9 step on tiles, populations in registers.
//
// A block owns TX x TY nodes, one per thread.  A thread pulls the streamed
// populations of its node once (all loads independent, straight to
// registers), forms the macro fields that the gradients need into a shared
// tile, and the block's threads then evaluate the one-node halo around the
// tile (the zeroth and first moments only); after one barrier every thread
// takes its gradients from the tile and collides from its registers.  Nothing
// goes through global memory between pull and store, there is one launch per
// step, and any row length, wall or reservoir runs the same code (reservoir
// columns overwrite the missing populations after the loads).  Where one tile
// spans all rows (ny <= TY: capillaries, lines) the rows wrap inside the tile
// and only the two columns beside it are evaluated.
//
// What bounds it: on large lattices the L2 and DRAM traffic and the part of
// the arithmetic that the other resident blocks do not hide (512 x 512 FP32:
// a bare copy of the state 14.0 us, pulls and halo without arithmetic 20.7 us,
// the step 30.4 us at 12 warps per SM; 128 registers and 16 warps, 256-node
// blocks, and two nodes per thread in packed FP32 arithmetic were no faster);
// in FP64 the FP64 pipe.  Against the form that served each size before, us per
// step of long runs: 512 x 384 FP32 with reservoirs 148 -> 21.9, 701 x 523 with
// walls 65 -> 41, 512 x 512 FP64 974 -> 533.  Lattices of a few thousand nodes are
// bound by one block's latency and run split by lattice (lbm_split2d.cuh).
#pragma once

#include "lbm_twopass.cuh"

namespace lbm {

LBM_HD int modp(int v, int n) {
  int r = v % n;
  return r < 0 ? r + n : r;
}

template <class R, int M, bool EN, int TX, int TY>
struct TileShape {
  static constexpr int NF = 4 + (EN ? M : 0), PX = TX + 2, PY = TY + 2, PN = PX * PY;
  static constexpr int NL = M + 1 + (EN ? 1 : 0);
};

// One tile at (x0, y0); mac is the block's shared [NF][PN].
template <class R, int M, bool EN, int TX, int TY>
__device__ __forceinline__ void tile2d_step(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, int x0,
                                            int y0, R* __restrict__ mac) {
  using T = TileShape<R, M, EN, TX, TY>;
  constexpr int PX = T::PX, PN = T::PN, NT = TX * TY;
  const int t = threadIdx.x, tx = t % TX, ty = t / TX;
  const bool wrap = p.ny <= TY;                       // all rows in this tile
  // lattice node of a tile cell: periodic wrap, or the zero-gradient copy of
  // the boundary node across an open face
  auto place = [&](int ex, int ey, int& x, int& y) {
    x = x0 + ex;
    if (x < 0 || x >= p.nx) {
      const int bc = x < 0 ? p.bc_lo : p.bc_hi;
      x = (bc == BC_PERIODIC) ? modp(x, p.nx) : (x < 0 ? 0 : p.nx - 1);
    }
    y = modp(y0 + ey, p.ny);
  };
  int x, y;
  place(tx, ty, x, y);
  const int n = x + p.nx * y;
  R P[T::NL * 9];
  pull_node<R, 2, M, EN>(p, it, a.src, a.phi, x, y, 0, P);
  const R phi = a.phi[n], Tf = EN ? R(0) : a.Tfix[n];
  // ---- halo: rows above and below (unless they wrap), columns beside --------
  const int rows = wrap ? 0 : 2 * PX;
  const int cells = rows + 2 * (wrap ? p.ny : TY);
#pragma unroll 1
  for (int e = t; e < cells; e += NT) {
    int ex, ey;
    if (e < rows) {
      ex = e % PX - 1;
      ey = e < PX ? -1 : TY;
    } else {
      ex = ((e - rows) & 1) ? TX : -1;
      ey = (e - rows) >> 1;
    }
    if (x0 + ex > p.nx || y0 + ey > p.ny) continue;   // beyond the last needed cell of a ragged tile
    int hx, hy;
    place(ex, ey, hx, hy);
    R H[T::NL * 9];
    pull_node<R, 2, M, EN>(p, it, a.src, a.phi, hx, hy, 0, H);
    Moments<R, 2, M, EN, false> mo;
    moments_gen<R, 2, M, EN, false>(ArrayPull<R, 2>{H}, mo);
    State<R, 2, M> s;
    const int hn = hx + p.nx * hy;
    s.template from_moments<EN, false>(p, mo, a.phi[hn], EN ? R(0) : a.Tfix[hn]);
    R* m = mac + (ey + 1) * PX + ex + 1;
    macro_fields<R, 2, M, EN>(s, [&](int k, const R& v) { m[k * PN] = v; });
  }
  // ---- own node ------------------------------------------------------------------
  ArrayPull<R, 2> pf{P};
  Moments<R, 2, M, EN, true> mo;
  moments_gen<R, 2, M, EN, true>(pf, mo);
  State<R, 2, M> s;
  s.template from_moments<EN, true>(p, mo, phi, Tf);
  const int row = (ty + 1) * PX + tx + 1;
  macro_fields<R, 2, M, EN>(s, [&](int k, const R& v) { mac[k * PN + row] = v; });
  __syncthreads();
  if (x0 + tx >= p.nx || y0 + ty >= p.ny) return;
  // tile rows of the neighbours
  int up = row + PX, dn = row - PX;
  if (wrap) {
    if (ty == p.ny - 1) up = row - ty * PX;
    if (ty == 0) dn = row + (p.ny - 1) * PX;
  }
  Grad<R, 2, M, EN> gr;
  // central differences (1/2), smoothed (1/6, 2/3, 1/6) along the other axis:
  // weights 1/3 on the axis and 1/12 on the corners
  const R wa = R(1) / R(3), wc = R(1) / R(12);
  auto ddx = [&](int k) {
    const R* m = mac + k * PN;
    return wa * (m[row + 1] - m[row - 1]) + wc * ((m[up + 1] - m[up - 1]) + (m[dn + 1] - m[dn - 1]));
  };
  auto ddy = [&](int k) {
    const R* m = mac + k * PN;
    return wa * (m[up] - m[dn]) + wc * ((m[up + 1] - m[dn + 1]) + (m[up - 1] - m[dn - 1]));
  };
  gr.divu = ddx(0) + ddy(1);
  gr.dPi[0] = ddx(2);
  gr.dPi[1] = ddy(3);
#pragma unroll
  for (int k = 0; k < M; ++k) {
    gr.dY[k][0] = EN ? ddx(4 + k) : R(0);
    gr.dY[k][1] = EN ? ddy(4 + k) : R(0);
  }
  collide_gen<R, 2, M, EN>(p, pf, n, mo, s, gr, a.dst, a.status);
}

template <class R, int M, bool EN, int TX, int TY, int MINB>
__global__ void __launch_bounds__(TX * TY, MINB) k_tile2d(Params<R> p, InletTables<R> it, StepArgs<R> a) {
  using T = TileShape<R, M, EN, TX, TY>;
  __shared__ R mac[T::NF * T::PN];
  after_previous();
  tile2d_step<R, M, EN, TX, TY>(p, it, a, blockIdx.x * TX, blockIdx.y * TY, mac);
}

}  // namespace lbm
