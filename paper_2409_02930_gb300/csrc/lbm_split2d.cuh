// D2Q9 step of small lattices, lattice by lattice: a block owns a tile of
// 8 x 4 nodes and has one warp per lattice and one for the halo, so the 32
// nodes' update runs as several short instruction streams side by side.
//
// What bounds it: one block's latency.  A lattice of a few thousand nodes has
// fewer tiles than the GPU has SMs; with one warp per tile (lbm_tile2d.cuh) the
// step is that warp's single stream of instructions, 2,000 in FP32 at four
// cycles each and 4,250 in FP64 at thirteen (dependent FP64 operations leave
// the SM's FP64 pipe 81 % idle).  Here
//   - the lattices' warps pull and sum nine populations each while the halo
//     warp forms the macro fields around the tile;
//   - the last lattice's warp forms the state of the 32 nodes and their macro
//     fields; the halo warp takes the gradients from the tile, the species'
//     warps solve the diffusion system together (Gauss-Jordan, one row each,
//     the pivot row through shared memory), and the last warp forms the mixture
//     coefficients meanwhile;
//   - every warp relaxes its own lattice.
// Where the tiles fill the SMs the repeated set-up costs more than the shorter
// streams give (figures at default_variant).
#pragma once

#include "lbm_split3d.cuh"
#include "lbm_tile2d.cuh"

namespace lbm {

// Fields of the tile's nodes in shared memory, [field][32].
template <int M, bool EN>
struct Split2dFields {
  // sums: per species sa, j, sum |f|; momentum sf, j, Pt (3); energy sg, q
  static constexpr int kSp = 4, kMo = kSp * M, kEn = kMo + 6, kSums = kEn + (EN ? 3 : 0);
  // state: w, T, sum of sa, sqrt(T)/phi, Y_b C/2; row sums and margins of the
  // diffusion system; v_a; pivot rows
  static constexpr int kW = kSums, kT = kW + 2, kSS = kT + 1, kKT = kSS + 1, kHY = kKT + 1, kCond = kHY + M,
                       kV = kCond + 2 * M, kPv = kV + 2 * M;
  // gradients: div u, d_b Pi_b, d_b Y_a; momentum axes, relaxation; difference moments
  static constexpr int kG = kPv + M * (M + 2), kF = kG + 3 + (EN ? 2 * M : 0), kOm = kF + 4, kD = kOm + 1,
                       kAll = kD + 8 * M;
};

// Streamed populations of lattice l at node (x, y).
template <class R, int M, bool EN>
__device__ __forceinline__ void pull_lattice2(const Params<R>& p, const InletTables<R>& it, const R* __restrict__ src,
                                              const R* __restrict__ phiA, int x, int y, int l, R (&f)[9]) {
  Site<R, 2> st;
  st.init(p, x, y, 0);
  const unsigned N = (unsigned)p.N;
  const R* __restrict__ fl = src + (size_t)(unsigned)(l * 9) * N;
  Unroll<0, 9>::run([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    int s = st.source(c_of<2>(i, 0), c_of<2>(i, 1), 0);
    unsigned k = i;
    if (c_of<2>(i, 0) != 0 && s < 0) {
      if (s != SRC_GHOST) k = 8 - i;
      s = st.n;
    }
    f[i] = fl[(size_t)k * N + s];
  });
  if (st.has_ghost()) {
    Ghost<R, 2> gh;
    ghost_velocity<R, 2, M>(p, src, phiA, x, y, 0, gh);
    const bool lo = gh.side == 0;
    ghost_lattice<R, 2, M, EN>(p, it, gh, l, [&](int cy, int, const R& v) {
      const int row = 1 + 3 * (cy + 1);
      if (lo) f[row + 1] = v;
      else f[row - 1] = v;
    });
  }
}

// Row l of the FP64 diffusion solve of one node (FP32 lattices above the
// condition bound): the whole system from the sums in shared memory.
template <class R, int M, bool EN>
__device__ __noinline__ void solve_row2_fp64(const Params<R>& p, const R* S, R phi, int l, R (&v)[2]) {
  using F = Split2dFields<M, EN>;
  typename Transport<float, 2, M>::Fp64System y;
  y.phi = phi; y.sf = S[F::kMo * 32]; y.T = S[F::kT * 32]; y.Kc = p.Kc;
  const R ss = S[F::kSS * 32];
  for (int a = 0; a < M; ++a) {
    const R sa = S[F::kSp * a * 32];
    y.sa[a] = sa;
    y.Y[a] = sa / ss;
    y.knc[a] = p.knudsen ? p.knc[a] : R(0);
    y.tiny[a] = Transport<R, 2, M>::unresolved(sa, ss, S[(F::kSp * a + 3) * 32]);
    for (int b = 0; b < M; ++b) y.D_[a][b] = p.invDmm[a][b];
    for (int b = 0; b < 2; ++b) y.ja[a][b] = S[(F::kSp * a + 1 + b) * 32];
  }
  for (int b = 0; b < 2; ++b) y.w[b] = S[(F::kW + b) * 32];
  Transport<float, 2, M>::solve_system(y);
  for (int b = 0; b < 2; ++b) v[b] = y.v[l][b];
}

template <class R, int M, bool EN>
__global__ void __launch_bounds__(32 * (M + 2 + (EN ? 1 : 0))) k_split2d(Params<R> p, InletTables<R> it, StepArgs<R> a) {
  constexpr int TX = 8, TY = 4, L = M + 1 + (EN ? 1 : 0);
  using T = TileShape<R, M, EN, TX, TY>;
  using F = Split2dFields<M, EN>;
  constexpr int PX = T::PX, PN = T::PN;
  // barriers: 1 sums ready (all lattices), 2 state ready (last to the species),
  // 3 own macro fields ready (last to halo), 4 gradients ready (halo to last),
  // 5 pivot rows and difference moments (species), 6 v ready (species to
  // last), 7 mixture ready (last to momentum)
  __shared__ R mac[T::NF * PN];
  __shared__ R sh[F::kAll * 32];
  after_previous();
  const int lane = threadIdx.x & 31, l = __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0);
  R* S = sh + lane;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  const int tx = lane % TX, ty = lane / TX;
  const bool wrap = p.ny <= TY;                       // all rows in this tile
  auto place = [&](int ex, int ey, int& x, int& y) {   // as in tile2d_step
    x = x0 + ex;
    if (x < 0 || x >= p.nx) {
      const int bc = x < 0 ? p.bc_lo : p.bc_hi;
      x = (bc == BC_PERIODIC) ? modp(x, p.nx) : (x < 0 ? 0 : p.nx - 1);
    }
    y = modp(y0 + ey, p.ny);
  };
  const int row = (ty + 1) * PX + tx + 1;
  if (l == L) {
    // ---- halo warp: macro fields around the tile, then the gradients ----------------
    const int rows = wrap ? 0 : 2 * PX, cells = rows + 2 * (wrap ? p.ny : TY);
    static_assert(2 * PX + 2 * TY <= 32, "one halo cell per lane");
    if (lane < cells) {
      int ex, ey;
      if (lane < rows) {
        ex = lane % PX - 1;
        ey = lane < PX ? -1 : TY;
      } else {
        ex = ((lane - rows) & 1) ? TX : -1;
        ey = (lane - rows) >> 1;
      }
      if (x0 + ex <= p.nx && y0 + ey <= p.ny) {       // up to the last needed cell of a ragged tile
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
    }
    bar_sync(3, 64);
    // neighbours' rows inside the tile; cells beyond a ragged edge are computed
    // from whatever the tile holds and never stored
    int up = row + PX, dn = row - PX;
    if (wrap) {
      if (ty == p.ny - 1) up = row - ty * PX;
      if (ty == 0) dn = row + (p.ny - 1) * PX;
    }
    const R wa = R(1) / R(3), wc = R(1) / R(12);
    auto ddx = [&](int k) {
      const R* m = mac + k * PN;
      return wa * (m[row + 1] - m[row - 1]) + wc * ((m[up + 1] - m[up - 1]) + (m[dn + 1] - m[dn - 1]));
    };
    auto ddy = [&](int k) {
      const R* m = mac + k * PN;
      return wa * (m[up] - m[dn]) + wc * ((m[up + 1] - m[dn + 1]) + (m[up - 1] - m[dn - 1]));
    };
    S[F::kG * 32] = ddx(0) + ddy(1);
    S[(F::kG + 1) * 32] = ddx(2);
    S[(F::kG + 2) * 32] = ddy(3);
    if (EN) {
#pragma unroll
      for (int k = 0; k < M; ++k) {
        S[(F::kG + 3 + 2 * k) * 32] = ddx(4 + k);
        S[(F::kG + 4 + 2 * k) * 32] = ddy(4 + k);
      }
    }
    bar_arrive(4, 64);
    return;
  }
  int x, y;
  place(tx, ty, x, y);
  const int n = x + p.nx * y;
  const bool live = x0 + tx < p.nx && y0 + ty < p.ny;
  const unsigned N = (unsigned)p.N;
  R f[9], s0, j0[2], sabs = R(0);
  pull_lattice2<R, M, EN>(p, it, a.src, a.phi, x, y, l, f);
  const R phi = a.phi[n], Tf = EN ? R(0) : a.Tfix[n];
  auto get = [&](int i) { return f[i]; };
  {
    R Pt[2][2];
    lattice_sums<R, 2, 2>(get, s0, j0, Pt);
    const int k = l < M ? F::kSp * l : (l == M ? F::kMo : F::kEn);
    S[k * 32] = s0;
    S[(k + 1) * 32] = j0[0];
    S[(k + 2) * 32] = j0[1];
    if (l == M) {
      S[(k + 3) * 32] = Pt[0][0];
      S[(k + 4) * 32] = Pt[0][1];
      S[(k + 5) * 32] = Pt[1][1];
    }
    if (ScalarTraits<R>::single && l < M) {
      sabs = fabs(f[0]);
#pragma unroll
      for (int i = 1; i < 9; ++i) sabs += fabs(f[i]);
      S[(k + 3) * 32] = sabs;
    }
  }
  bar_sync(1, 32 * L);
  R* __restrict__ dl = a.dst + (size_t)(unsigned)(l * 9) * N + n;
  auto put = [&](int i, const R& v) {
    if (live) dl[(size_t)(unsigned)i * N] = v;
  };
  if (l < M) {
    // ---- species l: its row of the diffusion system (Eq. 23, 24, 22, 26, 29) ------
    bar_sync(2, 32 * (M + 1));
    R w[2], v[2], rw[M];
#pragma unroll
    for (int b = 0; b < 2; ++b) w[b] = S[(F::kW + b) * 32];
    R h = R(0), hYl = R(0);
#pragma unroll
    for (int b = 0; b < M; ++b) {
      const R hY = S[(F::kHY + b) * 32], t = hY * p.invDmm[l][b];      // zero on the diagonal
      if (b == l) hYl = hY;
      rw[b] = -t;
      h += t;
    }
    const R itk = p.knc[l] * S[F::kKT * 32], q = R(1) / (R(1) + h), beta = h * q;
    const R hk = R(0.5) * itk, margin = R(1) + hk;
    const bool tiny = Transport<R, 2, M>::unresolved(s0, S[F::kSS * 32], sabs);
    const R isa = R(1) / s0;
#pragma unroll
    for (int b = 0; b < 2; ++b) v[b] = (tiny ? R(0) : j0[b] * isa - w[b]) - hk * w[b];
    if (ScalarTraits<R>::single) {
      R rs = fabs(margin + h);
#pragma unroll
      for (int b = 0; b < M; ++b) rs += fabs(rw[b]);
      S[(F::kCond + l) * 32] = rs;
      S[(F::kCond + M + l) * 32] = margin;
    }
#pragma unroll
    for (int b = 0; b < M; ++b)
      if (b == l) rw[b] = margin + h;
    bool fp64 = false;
#pragma unroll
    for (int k = 0; k < M; ++k) {
      R* pv = S + (F::kPv + k * (M + 2)) * 32;
      if (l == k) {
        const R inv = R(1) / rw[k];
#pragma unroll
        for (int c = k + 1; c < M; ++c) {
          rw[c] *= inv;
          pv[c * 32] = rw[c];
        }
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          v[b] *= inv;
          pv[(M + b) * 32] = v[b];
        }
      }
      bar_sync(5, 32 * M);
      if (l != k) {
        const R g = rw[k];
#pragma unroll
        for (int c = k + 1; c < M; ++c) rw[c] -= g * pv[c * 32];
#pragma unroll
        for (int b = 0; b < 2; ++b) v[b] -= g * pv[(M + b) * 32];
      }
      if (ScalarTraits<R>::single && k == 0) {
        // condition bound (R12): above it the system is solved in double
        R amax = R(0), dmin = R(1e30);
#pragma unroll
        for (int b = 0; b < M; ++b) {
          const R rs = S[(F::kCond + b) * 32], d = S[(F::kCond + M + b) * 32];
          amax = rs > amax ? rs : amax;
          dmin = d < dmin ? d : dmin;
        }
        fp64 = amax > p.kappa_thr * dmin;
      }
    }
    if constexpr (ScalarTraits<R>::single) {
      if (fp64) solve_row2_fp64<R, M, EN>(p, S, phi, l, v);
      if (live && l == 0 && fp64) flag(a.status, 2);
    }
#pragma unroll
    for (int b = 0; b < 2; ++b) S[(F::kV + 2 * l + b) * 32] = v[b];
    bar_arrive(6, 32 * (M + 1));
    // ---- its difference moments and relaxation (Eq. 21, Eq. 25) --------------------
    SpeciesTarget<R, 2> t;
    const R gd = q * itk, qY = R(2) * q * hYl;         // (1 - beta) Y_l C
    t.th = R(0.5) * p.Ra[l] * S[F::kT * 32];
    t.gE = gd * s0;
    t.cE = R(2) * beta * s0;
    SpeciesAxes<R, 2> ax;
    ax.set(w, v, s0, t.th);
    R m[9];
    ax.template delta<0>(m);
#pragma unroll
    for (int e = 1; e < 9; ++e) S[(F::kD + 8 * l + e - 1) * 32] = m[e];
#pragma unroll
    for (int e = 1; e < 9; ++e) m[e] = t.template entry<0>(ax, w, e % 3, e / 3);
    bar_sync(5, 32 * M);
#pragma unroll
    for (int b = 0; b < M; ++b) {
      const R X = (b == l) ? -gd : qY * p.invDmm[l][b];
#pragma unroll
      for (int e = 1; e < 9; ++e) m[e] += X * S[(F::kD + 8 * b + e - 1) * 32];
    }
    put(4, s0 - relax_dirs<R, 2, false>(get, 0, R(1) - R(2) * beta, m, nullptr, put));
    return;
  }
  R m[1][9], ex[2] = {R(0), R(0)}, total, keep;
  if (l == L - 1) {
    // ---- last lattice: state, then mixture (and the energy lattice) -----------------
    Moments<R, 2, M, EN, true> mo;
#pragma unroll
    for (int k = 0; k < M; ++k) mo.sa[k] = S[F::kSp * k * 32];
    mo.sf = S[F::kMo * 32];
#pragma unroll
    for (int b = 0; b < 2; ++b) mo.jf[b] = S[(F::kMo + 1 + b) * 32];
    if (EN) mo.sg = s0;
    State<R, 2, M> s;
    s.template from_moments<EN, true>(p, mo, phi, Tf);
    const R inv_phi = R(1) / s.phi;
    const R kT = s.T * rsqrt_<R>(s.T) * inv_phi, hC = R(0.5) * p.Kc * s.sf * kT;      // as in Transport
#pragma unroll
    for (int b = 0; b < 2; ++b) S[(F::kW + b) * 32] = s.w[b];
    S[F::kT * 32] = s.T;
    S[F::kSS * 32] = s.ss;
    S[F::kKT * 32] = p.knudsen ? kT : R(0);
#pragma unroll
    for (int k = 0; k < M; ++k) S[(F::kHY + k) * 32] = hC * s.Y[k];
    bar_arrive(2, 32 * (M + 1));
    macro_fields<R, 2, M, EN>(s, [&](int k, const R& v) { mac[k * PN + row] = v; });
    bar_arrive(3, 64);
    if (live && bad_state(s, inv_phi)) flag(a.status, 1);
    R itk[M];
#pragma unroll
    for (int k = 0; k < M; ++k) itk[k] = p.knudsen ? p.knc[k] * kT : R(0);
    bar_sync(4, 64);
    Grad<R, 2, M, EN> gr;
    gr.divu = S[F::kG * 32];
#pragma unroll
    for (int b = 0; b < 2; ++b) gr.dPi[b] = S[(F::kG + 1 + b) * 32];
    Mixture<R, 2> mix;
    mix.template scalars<M, EN>(p, s, inv_phi, gr.divu);
    bar_sync(6, 32 * (M + 1));
    R v[M][2], vbar[2];
#pragma unroll
    for (int k = 0; k < M; ++k)
#pragma unroll
      for (int b = 0; b < 2; ++b) v[k][b] = S[(F::kV + 2 * k + b) * 32];
    mix.template force<M>(s, itk, v, vbar);
    Axis<R> F2[2];
#pragma unroll
    for (int b = 0; b < 2; ++b) mix.momentum_axis(s.w[b], s.inv_sf, b, gr.dPi[b], F2[b]);
    keep = R(1) - mix.omega;
    if constexpr (EN) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        S[(F::kF + 2 * b) * 32] = F2[b].m[1];
        S[(F::kF + 2 * b + 1) * 32] = F2[b].m[2];
      }
      S[F::kOm * 32] = mix.omega;
      bar_arrive(7, 64);
      // ---- energy (Eq. 43, Eq. 51, Eq. 54) ----------------------------------------
      mo.Pt[0][0] = S[(F::kMo + 3) * 32];
      mo.Pt[0][1] = mo.Pt[1][0] = S[(F::kMo + 4) * 32];
      mo.Pt[1][1] = S[(F::kMo + 5) * 32];
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        mo.q[b] = j0[b];
#pragma unroll
        for (int k = 0; k < M; ++k) gr.dY[k][b] = S[(F::kG + 3 + 2 * k + b) * 32];
      }
      mix.template heat<M, EN>(p, mo, s, v, vbar, gr);
#pragma unroll
      for (int b = 0; b < 2; ++b) ex[b] = mix.Dq[b];
      energy_moments<R, 2>(mix.omega * s.sf * mix.U, mix.omega * s.sf, mix.RT, s.w, m);
    } else {
      product_moments<R, 2>(mix.omega * s.sf, F2, m);
    }
    total = s0;
  } else {
    // ---- momentum (Eq. 42, Eq. 44) ---------------------------------------------------
    bar_sync(7, 64);
    Axis<R> F2[2];
#pragma unroll
    for (int b = 0; b < 2; ++b) F2[b].set(R(1), S[(F::kF + 2 * b) * 32], S[(F::kF + 2 * b + 1) * 32]);
    const R om = S[F::kOm * 32];
    product_moments<R, 2>(om * s0, F2, m);
    total = s0;
    keep = R(1) - om;
  }
  put(4, total - relax_dirs<R, 2, true>(get, 0, keep, m[0], ex, put));
}

}  // namespace lbm
