// Reverse mode of the D2Q9 node update, written out: given the adjoint lam of
// a node's post-collision populations, the adjoints of its streamed
// populations' moments, of its gradient inputs, of the porosity and of the
// Knudsen scale, in one backward pass over the forward quantities of
// collide_gen (same names, same order reversed; x_ is the adjoint of x).
// One pass costs about three node updates; evaluating the node code in
// forward-mode dual numbers took 15 two-lane evaluations (30 derivative
// directions).
#pragma once

#include "lbm_compact.cuh"

namespace lbm {

// Adjoints of the moments a node update reads.
template <class R, int M>
struct MomentBar {
  R sa[M], ja[M][2], sf, jf[2], Pt[2][2], sg, q[2];
};

// Adjoints of the state's derived fields.
template <class R, int M>
struct StateBar {
  R sa[M], Y[M], inv_m, Rg, sf, inv_sf, jf[2], w[2], E, T, inv_cv;
  LBM_HD void zero() {
#pragma unroll
    for (int a = 0; a < M; ++a) sa[a] = Y[a] = R(0);
    inv_m = Rg = sf = inv_sf = E = T = inv_cv = R(0);
#pragma unroll
    for (int b = 0; b < 2; ++b) jf[b] = w[b] = R(0);
  }
};

// State::from_moments backwards: adjoints of sa, sf, jf, sg from those of the state.
template <class R, int M, bool EN>
LBM_HD void state_reverse(const Params<R>& p, const State<R, 2, M>& s, R sg, StateBar<R, M>& b_, R (&sa_)[M], R& sf_,
                          R (&jf_)[2], R& sg_) {
  sg_ = R(0);
  if (EN) {
    // T = T_thermo + (E - w^2/2 - U0m) / cv
    b_.E += b_.T * s.inv_cv;
    const R u0_ = -b_.T * s.inv_cv;
    b_.inv_cv += b_.T * (s.T - p.T_thermo) / s.inv_cv;
    const R cv_ = -s.inv_cv * s.inv_cv * b_.inv_cv;
#pragma unroll
    for (int a = 0; a < M; ++a) b_.Y[a] += cv_ * p.cvR[a] + u0_ * p.U0[a];
#pragma unroll
    for (int b = 0; b < 2; ++b) b_.w[b] += u0_ * s.w[b];
    sg_ = b_.E * s.inv_sf;
    b_.inv_sf += b_.E * sg;
  }
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    jf_[b] = b_.jf[b] + b_.w[b] * s.inv_sf;
    b_.inv_sf += b_.w[b] * s.jf[b];
  }
  sf_ = b_.sf - s.inv_sf * s.inv_sf * b_.inv_sf;
  const R im_ = b_.inv_m + p.RU * b_.Rg;
  const R inv_ss = R(1) / s.ss;
  R iss_ = R(0);
#pragma unroll
  for (int a = 0; a < M; ++a) {
    b_.Y[a] += im_ * p.inv_m[a];
    iss_ += b_.Y[a] * s.sa[a];
  }
  const R ss_ = -inv_ss * inv_ss * iss_;
#pragma unroll
  for (int a = 0; a < M; ++a) sa_[a] = b_.sa[a] + b_.Y[a] * inv_ss + ss_;
}

// Transpose of slice_pops without its centre: adjoints of the scaled moments
// (m_[0] stays 0) from those of the eight moving populations.
template <class R>
LBM_HD void slice_transpose(const R (&mu)[9], R (&m_)[9]) {
  R t0[3], tp[3], tm[3];
  auto row = [&](R (&t)[3], int c, bool centre) {
    const R a = mu[3 * c], z = mu[3 * c + 1], b = mu[3 * c + 2];
    t[1] = b - a;
    t[2] = a + b;
    if (centre) t[2] -= R(2) * z;
    t[0] = centre ? z : R(0);
  };
  row(tm, 0, true);
  row(t0, 1, false);
  row(tp, 2, true);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    m_[i] = t0[i];
    m_[i + 3] = tp[i] - tm[i];
    m_[i + 6] = tp[i] + tm[i] - R(2) * t0[i];
  }
  m_[0] = R(0);
}

// lam(l, i): adjoint of the post-collision populations; f(l, i): streamed
// populations.  keep[l]: coefficient of a population's own relaxation.
// Returns in mb the moments' adjoints, in gb those of the gradient inputs, in
// phi_ and k_ those of the porosity and of the Knudsen scale.
template <class R, int M, bool EN, class Lam, class Pop>
LBM_HD void collide_reverse(const Params<R>& p, const Moments<R, 2, M, EN, true>& mo, const State<R, 2, M>& s,
                            const Grad<R, 2, M, EN>& gr, Lam&& lam, Pop&& f, MomentBar<R, M>& mb,
                            Grad<R, 2, M, EN>& gb, R& phi_, R& k_, R (&keep)[M + 1 + (EN ? 1 : 0)]) {
  constexpr int REST = 4;
  // ---- forward quantities ---------------------------------------------------
  const R inv_phi = R(1) / s.phi;
  const R sqT = s.T * rsqrt_<R>(s.T);
  const R C = p.Kc * (s.sf * inv_phi) * sqT, hC = R(0.5) * C, kT = sqT * inv_phi;
  R A[M][M], h[M], q[M], beta[M], itk[M], isa[M], v[M][2], piv[M];
  bool tiny[M];
#pragma unroll
  for (int a = 0; a < M; ++a) {
    itk[a] = p.knudsen ? p.knc[a] * kT : R(0);
    h[a] = R(0);
#pragma unroll
    for (int b = 0; b < M; ++b)
      if (b != a) {
        const R t = hC * s.Y[b] * p.invDmm[a][b];
        A[a][b] = -t;
        h[a] += t;
      }
    q[a] = R(1) / (R(1) + h[a]);
    beta[a] = h[a] * q[a];
    const R hk = R(0.5) * itk[a];
    A[a][a] = R(1) + hk + h[a];
    tiny[a] = Transport<R, 2, M>::unresolved(s, mo.sabs, a);
    isa[a] = R(1) / s.sa[a];
#pragma unroll
    for (int b = 0; b < 2; ++b)
      v[a][b] = (tiny[a] ? R(0) : (mo.ja[a][b] * isa[a] - s.w[b])) - hk * s.w[b];
  }
  // LU of A in place (unit lower part below the diagonal), v = A^-1 B
#pragma unroll
  for (int k = 0; k < M; ++k) {
    piv[k] = R(1) / A[k][k];
#pragma unroll
    for (int r = k + 1; r < M; ++r) {
      A[r][k] *= piv[k];
#pragma unroll
      for (int c = k + 1; c < M; ++c) A[r][c] -= A[r][k] * A[k][c];
#pragma unroll
      for (int b = 0; b < 2; ++b) v[r][b] -= A[r][k] * v[k][b];
    }
  }
#pragma unroll
  for (int k = M - 1; k >= 0; --k)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      R t = v[k][b];
#pragma unroll
      for (int j = k + 1; j < M; ++j) t -= A[k][j] * v[j][b];
      v[k][b] = t * piv[k];
    }
  const R RT = s.Rg * s.T, mm = R(1) / s.inv_m;
  R ms = R(0);
#pragma unroll
  for (int a = 0; a < M; ++a) ms += s.Y[a] * p.mum[a];
  const R pw = pow_<R>(s.T * p.inv_T_ref, p.mu_exp);
  const R mu = ms * pw * mm, inv_P = s.phi * s.inv_sf / RT, muP = mu * inv_P;
  const R inv_om = R(0.5) + muP, om = R(1) / inv_om, om1 = R(1) / (R(0.5) + muP * p.inv_Pr);
  const R kb = R(1) - p.bulk_ratio - (EN ? s.Rg * s.inv_cv : R(0));
  const R bdu = mu * kb * gr.divu;
  R ks[M], kd = R(0), vbar[2], g[2], Fk[2];
#pragma unroll
  for (int a = 0; a < M; ++a) {
    ks[a] = s.sa[a] * itk[a];
    kd += ks[a];
  }
  const R drag = R(1) / (R(1) + R(0.5) * kd * s.inv_sf);
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    vbar[b] = R(0);
#pragma unroll
    for (int a = 0; a < M; ++a) vbar[b] += s.Y[a] * v[a][b];
    g[b] = kd * (s.w[b] - vbar[b]);
#pragma unroll
    for (int a = 0; a < M; ++a) g[b] += ks[a] * v[a][b];
    Fk[b] = -drag * g[b];
  }
  // ---- adjoints -------------------------------------------------------------------
  StateBar<R, M> S_;
  S_.zero();
  R om_ = R(0), om1_ = R(0), RT_ = R(0), bdu_ = R(0), muP_ = R(0), iom_ = R(0), kd_ = R(0);
  R Fk_[2] = {R(0), R(0)}, vbar_[2] = {R(0), R(0)}, v_[M][2];
#pragma unroll
  for (int a = 0; a < M; ++a) v_[a][0] = v_[a][1] = R(0);
  R rest[M + 2];
  gb.dPi[0] = gb.dPi[1] = R(0);

  auto load = [&](int l, R (&mu9)[9], R& keep_) {
    rest[l] = lam(l, REST);
    keep_ = R(0);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      mu9[i] = R(0);
      if (i == REST) continue;
      mu9[i] = lam(l, i) - rest[l];
      keep_ += mu9[i] * f(l, i);
    }
  };
  // energy lattice
  rest[M + 1] = R(0);
#pragma unroll
  for (int b = 0; b < 2; ++b) mb.q[b] = R(0);
#pragma unroll
  for (int b = 0; b < 2; ++b)
#pragma unroll
    for (int c = 0; c < 2; ++c) mb.Pt[b][c] = R(0);
  if constexpr (EN) {
    R m9[9], m_[9], keep_;
    load(M + 1, m9, keep_);
    om_ -= keep_;
    slice_transpose(m9, m_);
    const R Dq_[2] = {m9[5] - m9[3], m9[7] - m9[1]};
    R hw2 = R(0.5) * (s.w[0] * s.w[0] + s.w[1] * s.w[1]);
    const R U = s.E - hw2, cU = om * s.sf * U, c2 = om * s.sf;
    R U_ = R(0), cU_ = R(0), c2_ = R(0);
    {
      R a1[2][3], a2[2][3], e2[2][3];           // axis moments; those of w^2/2 with and without c2
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const R w = s.w[b], w2 = w * w, hh = R(0.5) * w2;
        a1[b][0] = R(1); a1[b][1] = R(0.5) * w; a1[b][2] = R(0.5) * (RT + w2);
        e2[b][0] = hh; e2[b][1] = R(0.5) * (w * (RT + hh)); e2[b][2] = R(0.5) * (RT * (RT + R(2.5) * w2) + hh * w2);
#pragma unroll
        for (int i = 0; i < 3; ++i) a2[b][i] = c2 * e2[b][i];
      }
      R A1_[2][3], A2_[2][3], pi[3], pi_[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        pi[i] = cU * a1[0][i] + a2[0][i];
        pi_[i] = R(0);
        R t = R(0);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          pi_[i] += m_[i + 3 * j] * a1[1][j];
          t += m_[i + 3 * j] * a2[1][j];
        }
        A1_[0][i] = t + cU * pi_[i];
        A2_[0][i] = pi_[i];
        cU_ += pi_[i] * a1[0][i];
      }
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        A1_[1][j] = R(0);
        A2_[1][j] = R(0);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          A1_[1][j] += m_[i + 3 * j] * pi[i];
          A2_[1][j] += m_[i + 3 * j] * a1[0][i];
        }
      }
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const R w = s.w[b], w2 = w * w, hh = R(0.5) * w2;
        S_.w[b] += R(0.5) * A1_[b][1] + A1_[b][2] * w +
                   c2 * (A2_[b][0] * w + R(0.5) * A2_[b][1] * (RT + R(3) * hh) +
                         R(0.5) * A2_[b][2] * (R(5) * RT * w + R(2) * w * w2));
        RT_ += R(0.5) * A1_[b][2] + c2 * R(0.5) * (A2_[b][1] * w + A2_[b][2] * (R(2) * RT + R(2.5) * w2));
#pragma unroll
        for (int i = 0; i < 3; ++i) c2_ += A2_[b][i] * e2[b][i];
      }
    }
    om_ += cU_ * s.sf * U + c2_ * s.sf;
    S_.sf += om * (cU_ * U + c2_);
    U_ += cU_ * om * s.sf;
    // first-order part (Eq. 55)
    const R dom = om - om1, sRT = s.sf * RT;
    R Ha[M], HY[M], HYs = R(0), Ha_[M], HY_[M], HYs_ = R(0), dom_ = R(0), sRT_ = R(0);
#pragma unroll
    for (int a = 0; a < M; ++a) {
      Ha[a] = p.U0[a] + p.cvR[a] * (s.T - p.T_thermo) + p.Ra[a] * s.T;
      HY[a] = Ha[a] * s.Y[a];
      HYs += HY[a];
      Ha_[a] = HY_[a] = R(0);
    }
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const R d_ = R(0.5) * Dq_[b];
      R uP = R(0), sV = -HYs * vbar[b], sdY = R(0);
#pragma unroll
      for (int c = 0; c < 2; ++c) uP += s.w[c] * (mo.Pt[b][c] - (b == c ? s.jf[b] * s.w[c] + sRT : s.jf[b] * s.w[c]));
#pragma unroll
      for (int a = 0; a < M; ++a) {
        sV += HY[a] * v[a][b];
        sdY += Ha[a] * gr.dY[a][b];
      }
      const R X = mo.q[b] - uP - (s.E + RT) * s.jf[b], wdPi = s.w[b] * gr.dPi[b];
      dom_ += d_ * (X - R(0.5) * wdPi);
      const R X_ = dom * d_;
      om1_ += d_ * (s.sf * sV - R(0.5) * sRT * sdY);
      S_.sf += d_ * om1 * sV;
      const R sV_ = d_ * om1 * s.sf;
      sRT_ += d_ * (R(1) - R(0.5) * om1) * sdY;
      const R sdY_ = d_ * (R(1) - R(0.5) * om1) * sRT;
      S_.w[b] += d_ * (om * bdu - R(0.5) * dom * gr.dPi[b]);
      om_ += d_ * s.w[b] * bdu;
      bdu_ += d_ * s.w[b] * om;
      gb.dPi[b] -= R(0.5) * d_ * s.w[b] * dom;
      mb.q[b] += X_;
      S_.E -= X_ * s.jf[b];
      RT_ -= X_ * s.jf[b];
      S_.jf[b] -= X_ * (s.E + RT);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        // uP_ = -X_
        S_.w[c] -= X_ * (mo.Pt[b][c] - (b == c ? s.jf[b] * s.w[c] + sRT : s.jf[b] * s.w[c]));
        mb.Pt[b][c] -= X_ * s.w[c];
        S_.jf[b] += X_ * s.w[c] * s.w[c];
        S_.w[c] += X_ * s.w[c] * s.jf[b];
        if (b == c) sRT_ += X_ * s.w[b];
      }
      HYs_ -= sV_ * vbar[b];
      vbar_[b] -= sV_ * HYs;
#pragma unroll
      for (int a = 0; a < M; ++a) {
        HY_[a] += sV_ * v[a][b];
        v_[a][b] += sV_ * HY[a];
        Ha_[a] += sdY_ * gr.dY[a][b];
        gb.dY[a][b] = sdY_ * Ha[a];
      }
    }
#pragma unroll
    for (int a = 0; a < M; ++a) {
      HY_[a] += HYs_;
      Ha_[a] += HY_[a] * s.Y[a];
      S_.Y[a] += HY_[a] * Ha[a];
      S_.T += Ha_[a] * (p.cvR[a] + p.Ra[a]);
    }
    S_.sf += sRT_ * RT;
    RT_ += sRT_ * s.sf;
    om_ += dom_;
    om1_ -= dom_;
    S_.E += U_;
#pragma unroll
    for (int b = 0; b < 2; ++b) S_.w[b] -= U_ * s.w[b];
    keep[M + 1] = R(1) - om;
  } else {
#pragma unroll
    for (int a = 0; a < M; ++a) gb.dY[a][0] = gb.dY[a][1] = R(0);
  }
  // momentum lattice
  {
    R m9[9], m_[9], keep_;
    load(M, m9, keep_);
    om_ -= keep_;
    slice_transpose(m9, m_);
    const R c = om * s.sf;
    R F[2][3], F_[2][3], c_ = R(0);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      F[b][0] = R(1);
      F[b][1] = R(0.5) * (s.w[b] + Fk[b] * inv_om * s.inv_sf);
      F[b][2] = R(0.5) * (RT + s.w[b] * s.w[b] + s.inv_sf * (bdu + muP * gr.dPi[b]));
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      R t = R(0);
#pragma unroll
      for (int j = 0; j < 3; ++j) t += m_[i + 3 * j] * F[1][j];
      F_[0][i] = c * t;
      c_ += t * F[0][i];
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      F_[1][j] = R(0);
#pragma unroll
      for (int i = 0; i < 3; ++i) F_[1][j] += m_[i + 3 * j] * F[0][i];
      F_[1][j] *= c;
    }
    om_ += c_ * s.sf;
    S_.sf += c_ * om;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const R xi_ = R(0.5) * F_[b][1], P_ = R(0.5) * F_[b][2];
      S_.w[b] += xi_ + R(2) * s.w[b] * P_;
      Fk_[b] = xi_ * inv_om * s.inv_sf;
      iom_ += xi_ * Fk[b] * s.inv_sf;
      S_.inv_sf += xi_ * Fk[b] * inv_om + P_ * (bdu + muP * gr.dPi[b]);
      RT_ += P_;
      bdu_ += P_ * s.inv_sf;
      muP_ += P_ * s.inv_sf * gr.dPi[b];
      gb.dPi[b] += P_ * s.inv_sf * muP;
    }
    keep[M] = R(1) - om;
  }
  // species lattices
  R C_ = R(0), beta_[M], q_[M], itk_[M];
  {
    R dl[M][9], dl_[M][9], th[M], th_[M], E_[M][2][3];
#pragma unroll
    for (int a = 0; a < M; ++a) {
      th[a] = R(0.5) * p.Ra[a] * s.T;
      th_[a] = R(0);
      SpeciesAxes<R, 2> ax;
      ax.set(s.w, v[a], s.sa[a], th[a]);
      ax.template delta<0>(dl[a]);
#pragma unroll
      for (int e = 1; e < 9; ++e) dl_[a][e] = R(0);
    }
#pragma unroll
    for (int a = 0; a < M; ++a) {
      R m9[9], m_[9], keep_;
      load(a, m9, keep_);
      slice_transpose(m9, m_);
      const R cE = R(2) * beta[a] * s.sa[a], gd = q[a] * itk[a], gE = gd * s.sa[a], qY = q[a] * s.Y[a] * C;
      const R hx = R(0.5) * s.w[0] * s.w[0], hy = R(0.5) * s.w[1] * s.w[1];
      const R Ex[3] = {R(1), R(0.5) * s.w[0], hx + th[a]}, Ey[3] = {R(1), R(0.5) * s.w[1], hy + th[a]};
      R cE_ = R(0), gE_ = R(0), gd_ = R(0), qY_ = R(0), hx_ = R(0), hy_ = R(0);
      R Ex_[3] = {R(0), R(0), R(0)}, Ey_[3] = {R(0), R(0), R(0)};
#pragma unroll
      for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const int e = i + 3 * j;
          if (e == 0) continue;
          const R m = m_[e], Em = Ex[i] * Ey[j];
          R sum = R(0);
#pragma unroll
          for (int b = 0; b < M; ++b)
            if (b != a) {
              sum += p.invDmm[a][b] * dl[b][e];
              dl_[b][e] += qY * p.invDmm[a][b] * m;
            }
          gd_ -= m * dl[a][e];
          dl_[a][e] -= gd * m;
          qY_ += m * sum;
          cE_ += m * Em;
          R Em_;
          if (i == 1 || j == 1) {
            gE_ -= m * Em;
            Em_ = (cE - gE) * m;
          } else {
            const R ek_ = -gE * m;
            Em_ = cE * m;
            if (j == 0) {
              gE_ -= m * hx;
              hx_ += ek_;
            } else if (i == 0) {
              gE_ -= m * hy;
              hy_ += ek_;
            } else {
              gE_ -= m * (hx * Ey[2] + th[a] * hy);
              hx_ += ek_ * Ey[2];
              Ey_[2] += ek_ * hx;
              th_[a] += ek_ * hy;
              hy_ += ek_ * th[a];
            }
          }
          if (i > 0) Ex_[i] += Em_ * Ey[j];
          if (j > 0) Ey_[j] += Em_ * Ex[i];
        }
      S_.w[0] += hx_ * s.w[0];
      S_.w[1] += hy_ * s.w[1];
      gd_ += gE_ * s.sa[a];
      S_.sa[a] += R(2) * beta[a] * cE_ + gE_ * gd;
      beta_[a] = R(2) * s.sa[a] * cE_ - R(2) * keep_;
      q_[a] = gd_ * itk[a] + qY_ * s.Y[a] * C;
      itk_[a] = gd_ * q[a];
      S_.Y[a] += qY_ * q[a] * C;
      C_ += qY_ * q[a] * s.Y[a];
      keep[a] = R(1) - R(2) * beta[a];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        E_[a][0][i] = Ex_[i];
        E_[a][1][i] = Ey_[i];
      }
    }
    // the difference moments and the axes
#pragma unroll
    for (int a = 0; a < M; ++a) {
      SpeciesAxes<R, 2> ax;
      ax.set(s.w, v[a], s.sa[a], th[a]);
      R d_[2][3], S0_[3] = {R(0), R(0), R(0)};
#pragma unroll
      for (int i = 1; i < 3; ++i) {
        d_[0][i] = dl_[a][i];
        d_[1][i] = dl_[a][3 * i];
      }
#pragma unroll
      for (int j = 1; j < 3; ++j)
#pragma unroll
        for (int i = 1; i < 3; ++i) {
          const R t = dl_[a][i + 3 * j];
          d_[0][i] += t * ax.E[1].m[j];
          E_[a][1][j] += t * ax.d[0].m[i];
          S0_[i] += t * ax.d[1].m[j];
          d_[1][j] += t * ax.S[0].m[i];
        }
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const R w = s.w[b], vv = v[a][b], hv = R(0.5) * vv, wv = R(2) * w + vv, d2 = hv * wv;
        const R s1 = b == 0 ? S0_[1] : R(0), s2 = b == 0 ? S0_[2] : R(0);
        const R E2_ = E_[a][b][2] + s2;
        S_.sa[a] += d_[b][1] * hv + d_[b][2] * d2;
        const R d2_ = d_[b][2] * s.sa[a] + s2;
        const R hv_ = d_[b][1] * s.sa[a] + s1 + d2_ * wv;
        S_.w[b] += R(0.5) * (s1 + E_[a][b][1]) + E2_ * w + R(2) * d2_ * hv;
        v_[a][b] += d2_ * hv + R(0.5) * hv_;
        th_[a] += E2_;
      }
      S_.T += R(0.5) * p.Ra[a] * th_[a];
    }
  }
  // mixture scalars
  {
    R drag_ = R(0), ks_[M];
#pragma unroll
    for (int a = 0; a < M; ++a) ks_[a] = R(0);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      drag_ -= Fk_[b] * g[b];
      const R g_ = -drag * Fk_[b];
      kd_ += g_ * (s.w[b] - vbar[b]);
      S_.w[b] += g_ * kd;
      vbar_[b] -= g_ * kd;
#pragma unroll
      for (int a = 0; a < M; ++a) {
        ks_[a] += g_ * v[a][b];
        v_[a][b] += g_ * ks[a] + vbar_[b] * s.Y[a];
        S_.Y[a] += vbar_[b] * v[a][b];
      }
    }
    const R x_ = -drag * drag * drag_;
    kd_ += R(0.5) * x_ * s.inv_sf;
    S_.inv_sf += R(0.5) * x_ * kd;
#pragma unroll
    for (int a = 0; a < M; ++a) {
      ks_[a] += kd_;
      S_.sa[a] += ks_[a] * itk[a];
      itk_[a] += ks_[a] * s.sa[a];
    }
  }
  R iphi_ = R(0), mu_;
  {
    mu_ = bdu_ * kb * gr.divu;
    gb.divu = bdu_ * mu * kb;
    if (EN) {
      const R kb_ = bdu_ * mu * gr.divu;
      S_.Rg -= kb_ * s.inv_cv;
      S_.inv_cv -= kb_ * s.Rg;
    }
    iom_ -= om * om * om_;
    muP_ += iom_ - om1 * om1 * om1_ * p.inv_Pr;
    // muP = mu phi / (sf RT)
    mu_ += muP_ * inv_P;
    const R r = muP_ * muP;
    S_.sf -= r * s.inv_sf;
    iphi_ -= r * s.phi;
    RT_ -= r / RT;
    const R ms_ = mu_ * pw * mm;
#pragma unroll
    for (int a = 0; a < M; ++a) S_.Y[a] += ms_ * p.mum[a];
    const R mm_ = mu_ * mu;
    S_.T += mm_ * p.mu_exp / s.T;
    S_.inv_m -= mm_ * mm;
    S_.Rg += RT_ * s.T;
    S_.T += RT_ * s.Rg;
  }
  // transport: A^T B_ = v_, A_ = -B_ v^T
  {
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      // U^T y = v_, then L^T B_ = y
#pragma unroll
      for (int k = 0; k < M; ++k) {
#pragma unroll
        for (int j = 0; j < k; ++j) v_[k][b] -= A[j][k] * v_[j][b];
        v_[k][b] *= piv[k];
      }
#pragma unroll
      for (int k = M - 1; k >= 0; --k)
#pragma unroll
        for (int j = k + 1; j < M; ++j) v_[k][b] -= A[j][k] * v_[j][b];
    }
    R hC_ = R(0), kT_ = R(0);
    k_ = R(0);
#pragma unroll
    for (int a = 0; a < M; ++a) {
      const R hk = R(0.5) * itk[a];
      R Aaa = R(0), hk_ = R(0);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const R B_ = v_[a][b];
        Aaa -= B_ * v[a][b];
        hk_ -= B_ * s.w[b];
        S_.w[b] -= B_ * (tiny[a] ? hk : R(1) + hk);
        mb.ja[a][b] = tiny[a] ? R(0) : B_ * isa[a];
        if (!tiny[a]) S_.sa[a] -= mb.ja[a][b] * mo.ja[a][b] * isa[a];
      }
      hk_ += Aaa;
      // beta = h q, q = 1/(1 + h)
      const R qq_ = q_[a] + beta_[a] * h[a];
      const R h_ = Aaa + beta_[a] * q[a] - q[a] * q[a] * qq_;
#pragma unroll
      for (int c = 0; c < M; ++c)
        if (c != a) {
          // A_ac = -t: A_ac_ = -B_a . v_c
          R t_ = h_;
#pragma unroll
          for (int b = 0; b < 2; ++b) t_ += v_[a][b] * v[c][b];
          hC_ += t_ * s.Y[c] * p.invDmm[a][c];
          S_.Y[c] += t_ * hC * p.invDmm[a][c];
        }
      itk_[a] += R(0.5) * hk_;
      k_ += itk_[a] * itk[a];
      if (p.knudsen) kT_ += itk_[a] * p.knc[a];
    }
    C_ += R(0.5) * hC_;
    const R r = C_ * C;
    S_.sf += r * s.inv_sf;
    iphi_ += r * s.phi + kT_ * sqT;
    const R sqT_ = r / sqT + kT_ * inv_phi;
    S_.T += R(0.5) * sqT_ / sqT;
  }
  phi_ = -inv_phi * inv_phi * iphi_;
  if (!EN) S_.T = R(0);                                // fixed temperature
  state_reverse<R, M, EN>(p, s, mo.sg, S_, mb.sa, mb.sf, mb.jf, mb.sg);
#pragma unroll
  for (int a = 0; a < M; ++a) mb.sa[a] += rest[a];
  mb.sf += rest[M];
  if (EN) mb.sg += rest[M + 1];
}

}  // namespace lbm
