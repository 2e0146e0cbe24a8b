// Node code of the step: the pull with its boundary rules, the moments, the
// gradient inputs and the collision, from any source of streamed populations.
//
// The collision works in the moments of the product forms.  Every
// distribution of the step (Eq. 15, Eq. 16, Eq. 18, Eq. 44, Eq. 51) is a
// product over the axes of Psi_c with Psi_{+-1} = (P +- xi)/2, Psi_0 = 1 - P,
// so along one axis it is given by the three moments (1, xi, P) and the
// moments over D axes are products of those.  Relaxation is linear, so the
// target T_a of Eq. 21 (equilibrium, the quasi-equilibrium couplings of
// Eq. 25 and the Knudsen term) is combined in moments and transformed to
// populations once per lattice: 16 additions in D2Q9 and 78 in D3Q27 instead
// of evaluating 2 M + 1 distributions direction by direction.  The
// differences of equilibria that Eq. 25 takes, E - S and E - K, are formed in
// closed form (they vanish with v_a and w), and the zeroth moment is not
// needed, since the rest population is the remainder that conserves it.
// Moments carry a factor 1/2 per axis in which they are not the zeroth (exact
// in binary), which makes the transform pure additions.
//
// Measured against the same step written per direction with the divisions of
// the equations: 512 x 512 slab FP64 1.01 -> 0.72 ms per step, FP32 two-pass
// 512 x 384 with reservoirs 0.158 -> 0.041 ms, 64 x 40 0.029 -> 0.0095 ms; the
// FP32 error against double precision fell by 30 to 50 % (closed-form
// differences, fewer roundings).
#pragma once

#include "lbm_kernels.cuh"

namespace lbm {

// Source of the streamed population i at node (x, y, z) (pull with the
// boundary rules).  Returns the source node index, or -1 - n for bounce-back
// at this node, or SRC_GHOST for a reservoir ghost.
template <class R, int D>
struct Site {
  int x, y, z, n;
  int nx, ny, nz, bc_lo, bc_hi;
  LBM_HD void init(const Params<R>& p, int x_, int y_, int z_) {
    x = x_; y = y_; z = z_;
    nx = p.nx; ny = p.ny; nz = p.nz; bc_lo = p.bc_lo; bc_hi = p.bc_hi;
    n = x + nx * (y + ny * z);
  }
  LBM_HD int source(int cx, int cy, int cz) const {
    int sy = wrapi(y - cy, ny);
    int sz = (D == 3) ? wrapi(z - cz, nz) : 0;
    int sx = x - cx;
    if (sx < 0 || sx >= nx) {
      int bc = sx < 0 ? bc_lo : bc_hi;
      if (bc == BC_PERIODIC) sx = wrapi(sx, nx);
      else if (bc == BC_BOUNCEBACK) return -1 - n;
      else return SRC_GHOST;
    }
    return sx + nx * (sy + ny * sz);
  }
  LBM_HD bool has_ghost() const {
    return (x == 0 && bc_lo == BC_INLET) || (x == nx - 1 && bc_hi == BC_INLET);
  }
};

// velocity of the node adjacent to a reservoir face (all its sources inside)
template <class R, int D, int M>
LBM_HD void ghost_velocity(const Params<R>& p, const R* __restrict__ src, const R* __restrict__ phiA, int x, int y,
                           int z, Ghost<R, D>& gh) {
  constexpr int Q = Lat<D>::Q;
  gh.side = (x == 0 && p.bc_lo == BC_INLET) ? 0 : 1;
  const int xa = gh.side == 0 ? 1 : p.nx - 2;
  Site<R, D> sa;
  sa.init(p, xa, y, z);
  R s0 = R(0), j[D];
#pragma unroll
  for (int b = 0; b < D; ++b) j[b] = R(0);
  Unroll<0, Q>::run([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    const R f = src[(size_t)(M * Q + i) * p.N + sa.source(c_of<D>(i, 0), c_of<D>(i, 1), c_of<D>(i, 2))];
    s0 += f;
#pragma unroll
    for (int b = 0; b < D; ++b) {
      if (c_of<D>(i, b) > 0) j[b] += f;
      if (c_of<D>(i, b) < 0) j[b] -= f;
    }
  });
  R rho_f = s0 / phiA[sa.n];
#pragma unroll
  for (int b = 0; b < D; ++b) gh.u[b] = j[b] / rho_f;
  gh.phi = phiA[x + p.nx * (y + p.ny * z)];
}

// Missing populations of a reservoir face in lattice l: the equilibria
// (Eq. 15, Eq. 44, Eq. 51) at the reservoir state, moving with gh.u, of the
// 3^(D-1) directions that enter through the face (c_x = +1 at side 0, -1 at
// side 1).  put(cy, cz, value).
template <class R, int D, int M, bool EN, class Put>
LBM_HD void ghost_lattice(const Params<R>& p, const InletTables<R>& it, const Ghost<R, D>& gh, int l, Put&& put) {
  const int sd = gh.side;
  const R phi = gh.phi, T = it.T[sd];
  constexpr int zlo = (D == 3) ? 0 : 1, zhi = (D == 3) ? 2 : 1;
  if (!EN || l <= M) {
    R w[D];
#pragma unroll
    for (int b = 0; b < D; ++b) w[b] = gh.u[b] / phi;
    const R xi = sd == 0 ? w[0] : -w[0];
    const R RT = (l < M) ? p.Ra[l] * T : it.Rmix[sd] * T;
    const R rho = (l < M) ? it.rho[sd][l] : it.rho_sum[sd];
    const R vx = phi * rho * (R(0.5) * (xi + w[0] * w[0] + RT));
    R F[D][3];
#pragma unroll
    for (int b = 1; b < D; ++b) psi3<R>(w[b], w[b] * w[b] + RT, F[b]);
#pragma unroll
    for (int kz = zlo; kz <= zhi; ++kz) {
      R vz = vx;
      if (D == 3) vz *= F[D - 1][kz];
#pragma unroll
      for (int ky = 0; ky < 3; ++ky) put(ky - 1, kz - 1, vz * F[1][ky]);
    }
    return;
  }
  GeqFactors<R, D> G;
  G.init(phi, it.rho_sum[sd], gh.u, it.Rmix[sd] * T, it.Umix[sd]);
  const R p1 = sd == 0 ? G.P1[0][2] : G.P1[0][0], p2 = sd == 0 ? G.P2[0][2] : G.P2[0][0];
  const R a1 = G.pref_U * p1 + G.pref * p2, a2 = G.pref * p1;
#pragma unroll
  for (int kz = zlo; kz <= zhi; ++kz)
#pragma unroll
    for (int ky = 0; ky < 3; ++ky) {
      R v = a1 * G.P1[1][ky] + a2 * G.P2[1][ky];
      if (D == 3) v = v * G.P1[D - 1][kz] + a2 * G.P1[1][ky] * G.P2[D - 1][kz];
      put(ky - 1, kz - 1, v);
    }
}

// The same for every lattice: put(l, cy, cz, value).
template <class R, int D, int M, bool EN, class Put>
LBM_HD void ghost_face(const Params<R>& p, const InletTables<R>& it, const Ghost<R, D>& gh, Put&& put) {
#pragma unroll
  for (int l = 0; l < M + 1 + (EN ? 1 : 0); ++l)
    ghost_lattice<R, D, M, EN>(p, it, gh, l, [&](int cy, int cz, const R& v) { put(l, cy, cz, v); });
}

// Streamed populations of node (x, y, z) into P[l*Q + i], all loads
// independent and addressed by compile-time directions (2-D: they stay in
// registers).  Bounce-back only changes an address; reservoir columns load
// their own node there and overwrite it with the face's equilibria.
template <class R, int D, int M, bool EN>
LBM_HD void pull_node(const Params<R>& p, const InletTables<R>& it, const R* __restrict__ src,
                      const R* __restrict__ phiA, int x, int y, int z, R (&P)[(M + 1 + (EN ? 1 : 0)) * Lat<D>::Q]) {
  constexpr int Q = Lat<D>::Q, L = M + 1 + (EN ? 1 : 0);
  Site<R, D> st;
  st.init(p, x, y, z);
  const unsigned N = (unsigned)p.N;
  Unroll<0, Q>::run([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    constexpr int cx = c_of<D>(i, 0), cy = c_of<D>(i, 1), cz = c_of<D>(i, 2);
    unsigned isrc = i;
    int s = st.source(cx, cy, cz);
    if (cx != 0 && s < 0) {
      if (s != SRC_GHOST) isrc = Q - 1 - i;
      s = st.n;
    }
    const R* q = src + (size_t)isrc * N + s;
#pragma unroll
    for (int l = 0; l < L; ++l) P[l * Q + i] = q[(size_t)(unsigned)(l * Q) * N];
  });
  if (st.has_ghost()) {
    Ghost<R, D> gh;
    ghost_velocity<R, D, M>(p, src, phiA, x, y, z, gh);
    const bool lo = gh.side == 0;
    ghost_face<R, D, M, EN>(p, it, gh, [&](int l, int cy, int cz, const R& v) {
      const int row = 1 + 3 * (cy + 1) + ((D == 3) ? 9 * (cz + 1) : 0);
      if (lo) P[l * Q + row + 1] = v;
      else P[l * Q + row - 1] = v;
    });
  }
}

// Puller over such an array.
template <class R, int D>
struct ArrayPull {
  const R* P;
  LBM_HD R get(int l, int i) const { return P[l * Lat<D>::Q + i]; }
};

// Sums of one lattice, axis by axis: s = sum f; with NEED >= 1 the first
// moments j, with NEED >= 2 the second moments Pt (symmetric).
template <class R, int D, int NEED, class Get>
LBM_HD void lattice_sums(Get&& f, R& s, R* j, R (*Pt)[D]) {
  constexpr int NZ = (D == 3) ? 3 : 1;
  R m0[NZ], jx[NZ], jy[NZ], xx[NZ], xy[NZ], yy[NZ];
#pragma unroll
  for (int k = 0; k < NZ; ++k) {
    R r0[3], r1[3], r2[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int i = 3 * c + ((D == 3) ? 9 * k : 0);
      const R a = f(i), b = f(i + 1), d = f(i + 2);
      const R e = a + d;
      r0[c] = e + b;
      if (NEED >= 1) r1[c] = d - a;
      if (NEED >= 2) r2[c] = e;
    }
    const R e = r0[0] + r0[2];
    m0[k] = e + r0[1];
    if (NEED >= 1) {
      jy[k] = r0[2] - r0[0];
      jx[k] = r1[0] + r1[2] + r1[1];
    }
    if (NEED >= 2) {
      yy[k] = e;
      xy[k] = r1[2] - r1[0];
      xx[k] = r2[0] + r2[2] + r2[1];
    }
  }
  if constexpr (D == 2) {
    s = m0[0];
    if (NEED >= 1) {
      j[0] = jx[0];
      j[1] = jy[0];
    }
    if (NEED >= 2) {
      Pt[0][0] = xx[0];
      Pt[1][1] = yy[0];
      Pt[0][1] = Pt[1][0] = xy[0];
    }
  } else {
    const R e = m0[0] + m0[2];
    s = e + m0[1];
    if (NEED >= 1) {
      j[0] = jx[0] + jx[2] + jx[1];
      j[1] = jy[0] + jy[2] + jy[1];
      j[2] = m0[2] - m0[0];
    }
    if (NEED >= 2) {
      Pt[0][0] = xx[0] + xx[2] + xx[1];
      Pt[1][1] = yy[0] + yy[2] + yy[1];
      Pt[2][2] = e;
      Pt[0][1] = Pt[1][0] = xy[0] + xy[2] + xy[1];
      Pt[0][2] = Pt[2][0] = jx[2] - jx[0];
      Pt[1][2] = Pt[2][1] = jy[2] - jy[0];
    }
  }
}

// Moments of the streamed populations from any puller: FULL for the
// collision, else those that the macro fields need.
template <class R, int D, int M, bool EN, bool FULL, class PullF>
LBM_HD void moments_gen(const PullF& pf, Moments<R, D, M, EN, FULL>& mo) {
#pragma unroll
  for (int a = 0; a < M; ++a) {
    lattice_sums<R, D, FULL ? 1 : 0>([&](int i) { return pf.get(a, i); }, mo.sa[a], mo.ja[a], mo.Pt);
    if (FULL && ScalarTraits<R>::single) {
      R s = fabs(pf.get(a, 0));
#pragma unroll
      for (int i = 1; i < Lat<D>::Q; ++i) s += fabs(pf.get(a, i));
      mo.sabs[a] = s;
    }
  }
  lattice_sums<R, D, (FULL && EN) ? 2 : 1>([&](int i) { return pf.get(M, i); }, mo.sf, mo.jf, mo.Pt);
  if (EN) lattice_sums<R, D, FULL ? 1 : 0>([&](int i) { return pf.get(M + 1, i); }, mo.sg, mo.q, mo.Pt);
}

// Moments of one axis with the factor 1/2 folded in: (1, xi/2, P/2), or a
// general zeroth moment.
template <class R>
struct Axis {
  R m[3];
  LBM_HD void set(R a, R b, R c) {
    m[0] = a; m[1] = b; m[2] = c;
  }
};

// Populations of one xy slice from its 9 scaled moments m[i + 3 j]:
// put(cx, cy, value); without ALL the centre (0, 0) is left out and m[0] is
// not read.
template <class R, bool ALL, class Put>
LBM_HD void slice_pops(const R (&m)[9], Put&& put) {
  R t0[3], tp[3], tm[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (ALL || i > 0) t0[i] = m[i] - R(2) * m[i + 6];
    tp[i] = m[i + 6] + m[i + 3];
    tm[i] = m[i + 6] - m[i + 3];
  }
  auto row = [&](const R (&t)[3], int cy, bool centre) {
    put(-1, cy, t[2] - t[1]);
    if (centre) put(0, cy, t[0] - R(2) * t[2]);
    put(1, cy, t[2] + t[1]);
  };
  row(tm, -1, true);
  row(t0, 0, ALL);
  row(tp, 1, true);
}

// Relaxes the populations of one slice cz of a lattice: stores
// keep * f + T (+- the extra first-order part ex on the axis directions)
// and returns the sum of what it stored.  get(i), put(i, value).
template <class R, int D, bool EXTRA, class Get, class Put>
LBM_HD R relax_dirs(Get&& get, int cz, R keep, const R (&m)[9], const R* ex, Put&& put) {
  R acc = R(0);
  auto one = [&](int cx, int cy, const R& T) {
    const int i = (cx + 1) + 3 * (cy + 1) + ((D == 3) ? 9 * (cz + 1) : 0);
    R o = keep * get(i) + T;
    if (EXTRA && cx * cx + cy * cy + cz * cz == 1) {
      if (cx > 0) o += ex[0];
      if (cx < 0) o -= ex[0];
      if (cy > 0) o += ex[1];
      if (cy < 0) o -= ex[1];
      if (D == 3 && cz > 0) o += ex[D - 1];
      if (D == 3 && cz < 0) o -= ex[D - 1];
    }
    acc += o;
    put(i, o);
  };
  if (D == 3 && cz != 0) slice_pops<R, true>(m, one);
  else slice_pops<R, false>(m, one);
  return acc;
}

// The same for lattice l of a D2Q9 node: put(l, i, value).
template <class R, int D, bool EXTRA, class PullF, class Put>
LBM_HD R relax_slice(const PullF& pf, int l, R keep, const R (&m)[9], const R* ex, Put&& put) {
  return relax_dirs<R, D, EXTRA>([&](int i) { return pf.get(l, i); }, 0, keep, m, ex,
                                 [&](int i, const R& v) { put(l, i, v); });
}

// Axis moments of one species: E (moving with w), S (moving with w + v) and
// the scaled difference d = sa (S - E) per axis.
template <class R, int D>
struct SpeciesAxes {
  Axis<R> E[D], S[D], d[D];
  LBM_HD void set(const R* w, const R* v, R sa, R th /* R_a T / 2 */) {
#pragma unroll
    for (int b = 0; b < D; ++b) {
      const R hw = R(0.5) * w[b], hv = R(0.5) * v[b];
      const R d2 = hv * (R(2) * w[b] + v[b]);
      E[b].set(R(1), hw, hw * w[b] + th);
      S[b].set(R(1), hw + hv, E[b].m[2] + d2);
      d[b].set(R(0), sa * hv, sa * d2);
    }
  }
  // scaled moments of sa (S - E) at z order k, m[i + 3 j] (m[0] unused at k = 0)
  template <int k>
  LBM_HD void delta(R (&m)[9]) const {
    constexpr bool Z = (D == 3) && k > 0;
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        R v, S2;
        if (j == 0) {
          v = d[0].m[i];
          S2 = S[0].m[i];
        } else if (i == 0) {
          v = d[1].m[j];
          S2 = S[1].m[j];
        } else {
          v = d[0].m[i] * E[1].m[j] + S[0].m[i] * d[1].m[j];
          if (Z) S2 = S[0].m[i] * S[1].m[j];
        }
        if (Z) {
          if (i == 0 && j == 0) v = d[D - 1].m[k];
          else v = v * E[D - 1].m[k] + S2 * d[D - 1].m[k];
        }
        if (i + j > 0 || Z) m[i + 3 * j] = v;
      }
  }
};

// Relaxation target of species a in scaled moments at z order k (Eq. 21, Eq. 25):
//   T_a = cE E_a - gE (E_a - K_a) + sum_b X_ab d_b,  X_ab = qY invDmm_ab, X_aa = -gd
// with d_b = sa_b (S_b - E_b), gd = (1 - beta_a)/tau^k_a, gE = gd sa_a,
// qY = (1 - beta_a) Y_a C and cE = 2 beta_a sa_a (+ the source of Eq. 89).
template <class R, int D>
struct SpeciesTarget {
  R cE, gE, th;
  // the part without the coupling
  template <int k>
  LBM_HD R entry(const SpeciesAxes<R, D>& ax, const R* w, int i, int j) const {
    constexpr bool Z = (D == 3) && k > 0;
    R Em = ax.E[0].m[i];
    if (j > 0) Em = (i > 0) ? Em * ax.E[1].m[j] : ax.E[1].m[j];
    if (Z) Em = (i + j > 0) ? Em * ax.E[D - 1].m[k] : ax.E[D - 1].m[k];
    R t;
    if (i == 1 || j == 1 || k == 1) {
      t = (cE - gE) * Em;                             // K rests: no odd moment
    } else {
      // E - K, formed from the powers of w
      R ek = R(0), kk = R(1);
      if (i > 0) {
        ek = R(0.5) * w[0] * w[0];
        kk = th;
      }
      if (j > 0) {
        const R h = R(0.5) * w[1] * w[1];
        ek = (i > 0) ? ek * ax.E[1].m[2] + kk * h : h;
        kk = (i > 0) ? kk * th : th;
      }
      if (Z) {
        const R h = R(0.5) * w[D - 1] * w[D - 1];
        ek = (i + j > 0) ? ek * ax.E[D - 1].m[2] + kk * h : h;
      }
      t = cE * Em - gE * ek;
    }
    return t;
  }
};

// Mixture quantities of one node that the momentum and energy lattices need.
template <class R, int D>
struct Mixture {
  R RT, inv_om, omega, omega1, muP, bdu;
  R Fk[D];                   // net Knudsen force (Eq. 48)
  R Dq[D];                   // half of (omega - omega1)(q* - q^eq) (Eq. 54, Eq. 55)
  R U, hw2;                  // specific internal energy, w^2/2

  // what does not depend on the diffusion velocities
  template <int M, bool EN>
  LBM_HD void scalars(const Params<R>& p, const State<R, D, M>& s, R inv_phi, R divu) {
    // Eq. 65, Eq. 67: 1/omega = 1/2 + mu/P, P of Eq. 3
    RT = s.Rg * s.T;
    R mu = R(0);
#pragma unroll
    for (int a = 0; a < M; ++a) mu += s.Y[a] * p.mum[a];
    mu *= pow_<R>(s.T * p.inv_T_ref, p.mu_exp) / s.inv_m;
    muP = mu / (s.sf * inv_phi * RT);
    inv_om = R(0.5) + muP;
    omega = R(1) / inv_om;
    omega1 = R(1) / (R(0.5) + muP * p.inv_Pr);
    bdu = mu * (R(2) / R(D) - p.bulk_ratio - (EN ? s.Rg * s.inv_cv : R(0))) * divu;
  }

  // Knudsen force (part of the momentum lattice) and the mass average of v
  template <int M>
  LBM_HD void force(const State<R, D, M>& s, const R* inv_tauk, const R (*v)[D], R* vbar) {
    // component velocity u* + (V_a - Vbar): diffusion velocities taken
    // relative to the species' mass average, the mixture velocity at the
    // middle of the step (trapezoidal drag of the mixture; reading R8)
    R ks[M], kdrag = R(0);
#pragma unroll
    for (int a = 0; a < M; ++a) {
      ks[a] = s.sa[a] * inv_tauk[a];
      kdrag += ks[a];
    }
    const R drag = R(1) / (R(1) + R(0.5) * kdrag * s.inv_sf);
#pragma unroll
    for (int b = 0; b < D; ++b) {
      vbar[b] = R(0);
#pragma unroll
      for (int a = 0; a < M; ++a) vbar[b] += s.Y[a] * v[a][b];
      R f = kdrag * (s.w[b] - vbar[b]);
#pragma unroll
      for (int a = 0; a < M; ++a) f += ks[a] * v[a][b];
      Fk[b] = -drag * f;
    }
  }

  // first-order part of the energy lattice (Eq. 54, Eq. 55)
  template <int M, bool EN>
  LBM_HD void heat(const Params<R>& p, const Moments<R, D, M, EN, true>& mo, const State<R, D, M>& s, const R (*v)[D],
                   const R* vbar, const Grad<R, D, M, EN>& gr) {
    U = R(0);
    hw2 = R(0);
    if (EN) {
#pragma unroll
      for (int b = 0; b < D; ++b) hw2 += s.w[b] * s.w[b];
      hw2 *= R(0.5);
      U = s.E - hw2;                                  // Eq. 40
      const R dom = omega - omega1, sRT = s.sf * RT;
      R Ha[M], HY[M], HYs = R(0);
#pragma unroll
      for (int a = 0; a < M; ++a) {
        Ha[a] = p.U0[a] + p.cvR[a] * (s.T - p.T_thermo) + p.Ra[a] * s.T;
        HY[a] = Ha[a] * s.Y[a];
        HYs += HY[a];
      }
#pragma unroll
      for (int b = 0; b < D; ++b) {
        R uP = R(0);
#pragma unroll
        for (int c = 0; c < D; ++c)
          uP += s.w[c] * (mo.Pt[b][c] - (b == c ? s.jf[b] * s.w[c] + sRT : s.jf[b] * s.w[c]));
        R sV = -HYs * vbar[b], sdY = R(0);
#pragma unroll
        for (int a = 0; a < M; ++a) {
          sV += HY[a] * v[a][b];
          sdY += Ha[a] * gr.dY[a][b];
        }
        const R d = dom * (mo.q[b] - uP - (s.E + RT) * s.jf[b]) + omega1 * s.sf * sV +
                    (R(1) - R(0.5) * omega1) * sRT * sdY + s.w[b] * (omega * bdu - R(0.5) * dom * gr.dPi[b]);
        Dq[b] = R(0.5) * d;
      }
    }
  }

  template <int M, bool EN>
  LBM_HD void compute(const Params<R>& p, const Moments<R, D, M, EN, true>& mo, const State<R, D, M>& s, R inv_phi,
                      const Transport<R, D, M>& tr, const Grad<R, D, M, EN>& gr) {
    R vbar[D];
    scalars<M, EN>(p, s, inv_phi, gr.divu);
    force<M>(s, tr.inv_tauk, tr.v, vbar);
    heat<M, EN>(p, mo, s, tr.v, vbar, gr);
  }

  // axis moments of the extended equilibrium (Eq. 44, Eq. 45; reading of u^ex)
  LBM_HD void momentum_axis(R w, R inv_sf, int b, R dPi, Axis<R>& F) const {
    const R xi = w + Fk[b] * inv_om * inv_sf;
    const R Pex = RT + w * w + inv_sf * (bdu + muP * dPi);
    F.set(R(1), R(0.5) * xi, R(0.5) * Pex);
  }
};

// Scaled moments of c times the product of the axes.
template <class R, int D>
LBM_HD void product_moments(R c, const Axis<R> (&F)[D], R (&m)[(D == 3) ? 3 : 1][9]) {
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      R v = (i > 0) ? c * F[0].m[i] : c;
      if (j > 0) v *= F[1].m[j];
      m[0][i + 3 * j] = v;
      if constexpr (D == 3) {
        m[1][i + 3 * j] = v * F[D - 1].m[1];
        m[2][i + 3 * j] = v * F[D - 1].m[2];
      }
    }
}

// Scaled moments of the energy equilibrium (Eq. 51) on the generating
// function U + sum_b w_b^2/2: cU multiplies the product of the axis moments
// (1, w, RT + w^2), c2 the products with one axis replaced by
// (w^2/2, RT w + w^3/2, RT^2 + 5/2 RT w^2 + w^4/2).
template <class R, int D>
LBM_HD void energy_moments(R cU, R c2, R RT, const R* w, R (&m)[(D == 3) ? 3 : 1][9]) {
  Axis<R> F1[D], F2[D];
#pragma unroll
  for (int b = 0; b < D; ++b) {
    const R w2 = w[b] * w[b], h = R(0.5) * w2;
    F1[b].set(R(1), R(0.5) * w[b], R(0.5) * (RT + w2));
    F2[b].set(c2 * h, c2 * R(0.5) * (w[b] * (RT + h)), c2 * R(0.5) * (RT * (RT + R(2.5) * w2) + h * w2));
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const R pi = cU * F1[0].m[i] + F2[0].m[i];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const R v = pi * F1[1].m[j] + F1[0].m[i] * F2[1].m[j];
      if constexpr (D == 3) {
        const R ab = F1[0].m[i] * F1[1].m[j];
#pragma unroll
        for (int k = 0; k < 3; ++k) m[k][i + 3 * j] = v * F1[D - 1].m[k] + ab * F2[D - 1].m[k];
      } else {
        m[0][i + 3 * j] = v;
      }
    }
  }
}

// non-finite or non-positive density, or a non-finite temperature
template <class R, int D, int M>
LBM_HD bool bad_state(const State<R, D, M>& s, R inv_phi) {
  return !(s.ss * inv_phi > R(0)) || !(s.sf * inv_phi > R(0)) || !finite_<R>(s.T);
}

// Collision and store of one D2Q9 node given its streamed populations
// (through the puller), its moments, state and gradient inputs (a4-a9).
template <class R, int D, int M, bool EN, class PullF>
LBM_HD void collide_gen(const Params<R>& p, const PullF& pf, int n, const Moments<R, D, M, EN, true>& mo,
                        const State<R, D, M>& s, const Grad<R, D, M, EN>& gr, R* __restrict__ dst, int* status) {
  static_assert(D == 2, "D3Q27 nodes collide lattice by lattice (lbm_split3d.cuh)");
  constexpr int Q = Lat<D>::Q;
  constexpr int REST = (Q - 1) / 2;
  const unsigned N = (unsigned)p.N;
  R* __restrict__ dn = dst + n;
  auto put = [&](int l, int i, const R& v) { dn[(size_t)(unsigned)(l * Q + i) * N] = v; };
  const R inv_phi = R(1) / s.phi;
  if (bad_state(s, inv_phi)) flag(status, 1);

  Transport<R, D, M> tr;
  tr.compute(p, s, inv_phi, &mo.ja[0][0], mo.sabs);
  if (tr.used_fp64) flag(status, 2);
  Mixture<R, D> mix;
  mix.template compute<M, EN>(p, mo, s, inv_phi, tr, gr);

  // ---- species (Eq. 21, Eq. 25) --------------------------------------------
  {
    SpeciesAxes<R, D> ax[M];
    R dl[M][9];
#pragma unroll
    for (int a = 0; a < M; ++a) {
      ax[a].set(s.w, tr.v[a], s.sa[a], R(0.5) * p.Ra[a] * s.T);
      ax[a].template delta<0>(dl[a]);
    }
#pragma unroll
    for (int a = 0; a < M; ++a) {
      SpeciesTarget<R, D> t;
      const R gd = tr.q[a] * tr.inv_tauk[a], qY = tr.q[a] * s.Y[a] * tr.C;
      t.cE = R(2) * tr.beta[a] * s.sa[a];
      t.gE = gd * s.sa[a];
      t.th = R(0.5) * p.Ra[a] * s.T;
      R X[M], T[9];
#pragma unroll
      for (int b = 0; b < M; ++b) X[b] = (b == a) ? -gd : qY * p.invDmm[a][b];
#pragma unroll
      for (int e = 1; e < 9; ++e) {
        T[e] = t.template entry<0>(ax[a], s.w, e % 3, e / 3);
#pragma unroll
        for (int b = 0; b < M; ++b) T[e] += X[b] * dl[b][e];
      }
      const R acc = relax_slice<R, D, false>(pf, a, R(1) - R(2) * tr.beta[a], T, nullptr, put);
      put(a, REST, mo.sa[a] - acc);
    }
  }
  const R keep = R(1) - mix.omega;
  // ---- momentum (Eq. 42, Eq. 44) ----------------------------------------------
  {
    Axis<R> F[D];
#pragma unroll
    for (int b = 0; b < D; ++b) mix.momentum_axis(s.w[b], s.inv_sf, b, gr.dPi[b], F[b]);
    R m[1][9];
    product_moments<R, D>(mix.omega * s.sf, F, m);
    const R acc = relax_slice<R, D, false>(pf, M, keep, m[0], nullptr, put);
    put(M, REST, mo.sf - acc);
  }
  // ---- energy (Eq. 43, Eq. 51, Eq. 54) ------------------------------------------
  if (EN) {
    R m[1][9];
    energy_moments<R, D>(mix.omega * s.sf * mix.U, mix.omega * s.sf, mix.RT, s.w, m);
    const R acc = relax_slice<R, D, true>(pf, M + 1, keep, m[0], mix.Dq, put);
    put(M + 1, REST, mo.sg - acc);
  }
}

}  // namespace lbm
