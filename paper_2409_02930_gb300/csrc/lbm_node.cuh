// Per-node building blocks, shared by every kernel form: reservoir data, the
// moments of the streamed populations, the state and the transport
// coefficients with the diffusion-velocity solve.
//
// Arithmetic.  The FP64 step is bound by the FP64 pipe (two fused
// multiply-adds per clock and SM) and the FP32 step by instruction issue, and
// an IEEE division costs about ten operations, so the node code is written on
// the porosity-weighted fields that the populations sum to.  With sa_a =
// phi rho_a, sf = phi rho and w = u / phi (the velocity in which every
// equilibrium is written) the porosity drops out of composition, velocity,
// temperature, energy and the momentum flux: w = j / sf, E = sum g / sf,
// rho u = j.  The diffusion system is solved for v_a = V_a / phi.  What is
// left is 1/phi (pressure, Knudsen rates) and one reciprocal each of sf, the
// summed densities, C_v, m, the three relaxation denominators and, per
// species, its density, its rate and its pivot: 5 + 3 M divisions and one
// reciprocal square root per node update where the equations written out
// take about 20 + 10 M divisions and a dozen square roots.
#pragma once

#include <type_traits>

#include "lbm_device.cuh"

namespace lbm {

constexpr int BC_PERIODIC = 0;
constexpr int BC_INLET = 1;
constexpr int BC_BOUNCEBACK = 2;
constexpr int SRC_GHOST = -0x7fffffff;

// Ghost state of a reservoir face: reservoir density, temperature and
// composition from the configuration, velocity of the adjacent interior node
// of the same step (reading of the "simplified flux" condition of Sec. 5.1,
// replacing only the missing populations).
template <class R, int D>
struct Ghost {
  int side;        // 0: x = 0 face, 1: x = nx-1 face
  R phi;
  R u[D];
};

template <class R>
struct InletTables {
  R rho[2][MMAX];   // species densities of the reservoirs
  R rho_sum[2];
  R Rmix[2];        // mixture gas constant
  R Umix[2];        // mixture specific internal energy at T_in
  R T[2];
};

// Moments of the streamed populations (Eq. 4, Eq. 5,
// Eq. 37, Eq. 38, Eq. 39, q, P).
template <class R, int D, int M, bool EN, bool FULL>
struct Moments {
  R sa[M], ja[M][D];
  R sabs[M];              // sum_i |f_ai| (FP32 full moments only): resolution of rho_a
  R sf, jf[D];
  R Pt[D][D];
  R sg, q[D];
};

// Composition, velocity, temperature and pressure of one node.
template <class R, int D, int M>
struct State {
  R phi;
  R sa[M], ss;               // phi rho_a and their sum
  R Y[M], inv_m, Rg;         // mass fractions, 1/m, R = R_U/m (Sec. 2.1)
  R sf, inv_sf, jf[D], w[D]; // phi rho (Eq. 37), j (Eq. 38), w = u / phi
  R E, T, inv_cv;

  template <bool EN, bool FULL>
  LBM_HD void from_moments(const Params<R>& p, const Moments<R, D, M, EN, FULL>& mo, R phi_, R Tfixed) {
    phi = phi_;
    ss = mo.sa[0];
#pragma unroll
    for (int a = 1; a < M; ++a) ss += mo.sa[a];            // Eq. 4, Eq. 1
    const R inv_ss = R(1) / ss;
    inv_m = R(0);
#pragma unroll
    for (int a = 0; a < M; ++a) {
      sa[a] = mo.sa[a];
      Y[a] = sa[a] * inv_ss;
      inv_m += Y[a] * p.inv_m[a];
    }
    Rg = p.RU * inv_m;
    sf = mo.sf;
    inv_sf = R(1) / sf;
#pragma unroll
    for (int b = 0; b < D; ++b) {
      jf[b] = mo.jf[b];
      w[b] = jf[b] * inv_sf;
    }
    if (EN) {
      // Eq. 41 with constant C_v and u^2/(2 phi^2)
      R cv = R(0), U0m = R(0), w2 = R(0);
#pragma unroll
      for (int a = 0; a < M; ++a) {
        cv += Y[a] * p.cvR[a];
        U0m += Y[a] * p.U0[a];
      }
#pragma unroll
      for (int b = 0; b < D; ++b) w2 += w[b] * w[b];
      inv_cv = R(1) / cv;
      E = mo.sg * inv_sf;
      T = p.T_thermo + (E - R(0.5) * w2 - U0m) * inv_cv;
    } else {
      E = R(0);
      inv_cv = R(0);
      T = Tfixed;
    }
  }

  LBM_HD R u(int b) const { return phi * w[b]; }
  // Pi_alpha = rho u_alpha (1 - 3RT) - rho u_alpha^3 / phi^2 (Eq. 45)
  LBM_HD R Pi(int b) const { return jf[b] * (R(1) - R(3) * (Rg * T) - w[b] * w[b]); }
};

// Transport coefficients (Eq. 23, Eq. 24, Eq. 22, Eq. 26) and the
// diffusion-velocity solve (Eq. 29).
template <class R, int D, int M>
struct Transport {
  R C;                       // 1/tau_ab = C invDmm_ab
  R beta[M], q[M];           // beta_a = dt/(2 tau_a + dt) with dt = 1, and 1 - beta_a
  R inv_tauk[M];
  R v[M][D];                 // V_a / phi
  int used_fp64;

  LBM_HD void compute(const Params<R>& p, const State<R, D, M>& s, R inv_phi,
                      const R* ja /* [M][D] */, const R* sabs /* [M] */) {
    // D_ab = D_ref (T/T_ref)^1.5 (P_ref/P) and 1/tau_ab = m R_U T / (D_ab m_a m_b)
    // with m P = (sf/phi) R_U T (Eq. 3) leave C ~ rho sqrt(T)
    const R sqT = s.T * rsqrt_<R>(s.T);
    C = p.Kc * (s.sf * inv_phi) * sqT;
    const R kT = sqT * inv_phi;
    const R hC = R(0.5) * C;
    // A v = j_a/sa_a - w - w/(2tau^k_a), A_aa = 1 + 1/(2tau_a) + 1/(2tau^k_a),
    // A_ab = -Y_b/(2 tau_ab): the trapezoidal rule on the Knudsen relaxation
    // toward the resting f^k acts on the component velocity u + V_a, which
    // adds -u/(2tau^k_a) to the right-hand side (reading R27)
    R A[M][M], B[M][D], hY[M];
    R amax = R(0), dmin = R(1e30);
#pragma unroll
    for (int b = 0; b < M; ++b) hY[b] = hC * s.Y[b];
#pragma unroll
    for (int a = 0; a < M; ++a) {
      inv_tauk[a] = p.knudsen ? p.knc[a] * kT : R(0);
      R h = R(0), rs = R(0);                          // h = 1/(2 tau_a)
#pragma unroll
      for (int b = 0; b < M; ++b)
        if (b != a) {
          const R t = hY[b] * p.invDmm[a][b];
          A[a][b] = -t;
          h += t;
          if (ScalarTraits<R>::single) rs += fabs(t);
        }
      q[a] = R(1) / (R(1) + h);
      beta[a] = h * q[a];
      const R hk = R(0.5) * inv_tauk[a];
      const R d = R(1) + hk;
      A[a][a] = d + h;
      if (ScalarTraits<R>::single) {
        rs += fabs(A[a][a]);
        amax = rs > amax ? rs : amax;
        dmin = d < dmin ? d : dmin;
      }
      const bool tiny = unresolved(s, sabs, a);
      const R isa = R(1) / s.sa[a];
#pragma unroll
      for (int b = 0; b < D; ++b)
        B[a][b] = (tiny ? R(0) : ja[a * D + b] * isa - s.w[b]) - hk * s.w[b];
    }
    used_fp64 = 0;
    if constexpr (std::is_same<R, float>::value) {
      if (amax > p.kappa_thr * dmin) {
        solve_fp64(p, s, ja, sabs);
        used_fp64 = 1;
        return;
      }
    }
    gauss<R>(A, B);
#pragma unroll
    for (int a = 0; a < M; ++a)
#pragma unroll
      for (int b = 0; b < D; ++b) v[a][b] = B[a][b];
  }

  // Trace species move with the mixture: below 1e-14 of the mixture density
  // (the oracle's bound) and, in FP32, where the species density is not
  // resolved by its populations.  Where the streamed populations of a species
  // cancel (sum |f_ai| > 1e4 rho_a: a trace tail crossed by weakly relaxed
  // non-equilibrium populations), FP32 leaves j_a / rho_a to rounding noise,
  // which the quasi-equilibrium then amplifies.
  LBM_HD static bool unresolved(const State<R, D, M>& s, const R* sabs, int a) {
    return unresolved(s.sa[a], s.ss, sabs[a]);
  }
  LBM_HD static bool unresolved(R sa, R ss, R sabs) {
    bool tiny = sa < R(1e-14) * ss;
    if (ScalarTraits<R>::single) tiny = tiny || !(sabs <= R(1e4) * sa);
    return tiny;
  }

  // FP32, condition bound above the threshold: assembled and solved in double
  // from the single-precision moments (the relaxation rates and the
  // right-hand side's differences of velocities formed in double).  Rarely
  // taken and kept out of line: inlined, its double matrices cost the FP32
  // kernels registers on every node.
  struct Fp64System {
    float phi, sf, T, Kc, w[D], Y[M], sa[M], knc[M], D_[M][M], ja[M][D], v[M][D];
    bool tiny[M];
  };
  static __host__ __device__ __noinline__ void solve_system(Fp64System& s) {
    double Ad[M][M], Bd[M][D];
    const double sq = ::sqrt((double)s.T), ip = 1.0 / (double)s.phi;
    const double hC = 0.5 * (double)s.Kc * (double)s.sf * ip * sq;
    for (int a = 0; a < M; ++a) {
      const double hk = 0.5 * (double)s.knc[a] * sq * ip;
      double h = 0.0;
      for (int b = 0; b < M; ++b)
        if (b != a) {
          Ad[a][b] = -hC * (double)s.Y[b] * (double)s.D_[a][b];
          h -= Ad[a][b];
        }
      Ad[a][a] = 1.0 + h + hk;
      for (int b = 0; b < D; ++b)
        Bd[a][b] = (s.tiny[a] ? 0.0 : ((double)s.ja[a][b] / (double)s.sa[a] - (double)s.w[b])) - hk * (double)s.w[b];
    }
    gauss<double>(Ad, Bd);
    for (int a = 0; a < M; ++a)
      for (int b = 0; b < D; ++b) s.v[a][b] = (float)Bd[a][b];
  }
  LBM_HD void solve_fp64(const Params<R>& p, const State<R, D, M>& s, const R* ja, const R* sabs) {
    Fp64System y;
    y.phi = s.phi; y.sf = s.sf; y.T = s.T; y.Kc = p.Kc;
#pragma unroll
    for (int a = 0; a < M; ++a) {
      y.Y[a] = s.Y[a]; y.sa[a] = s.sa[a]; y.knc[a] = p.knudsen ? p.knc[a] : 0.f; y.tiny[a] = unresolved(s, sabs, a);
#pragma unroll
      for (int b = 0; b < M; ++b) y.D_[a][b] = p.invDmm[a][b];
#pragma unroll
      for (int b = 0; b < D; ++b) y.ja[a][b] = ja[a * D + b];
    }
#pragma unroll
    for (int b = 0; b < D; ++b) y.w[b] = s.w[b];
    solve_system(y);
#pragma unroll
    for (int a = 0; a < M; ++a)
#pragma unroll
      for (int b = 0; b < D; ++b) v[a][b] = y.v[a][b];
  }

  // Gaussian elimination without pivoting: the matrix is strictly row
  // diagonally dominant (margin 1 + dt/2tau^k), so no pivoting is needed.
  template <class T>
  LBM_HD static void gauss(T (&A)[M][M], T (&B)[M][D]) {
    T piv[M];
#pragma unroll
    for (int k = 0; k < M; ++k) {
      piv[k] = T(1) / A[k][k];
#pragma unroll
      for (int r = k + 1; r < M; ++r) {
        T f = A[r][k] * piv[k];
#pragma unroll
        for (int c = k + 1; c < M; ++c) A[r][c] -= f * A[k][c];
#pragma unroll
        for (int c = 0; c < D; ++c) B[r][c] -= f * B[k][c];
      }
    }
#pragma unroll
    for (int k = M - 1; k >= 0; --k) {
#pragma unroll
      for (int c = 0; c < D; ++c) {
        T s = B[k][c];
#pragma unroll
        for (int j = k + 1; j < M; ++j) s -= A[k][j] * B[j][c];
        B[k][c] = s * piv[k];
      }
    }
  }
};

// Isotropic gradient weights 3 w_i (c_s^2 = 1/3) of the standard lattice.
template <class R, int D>
LBM_HD constexpr R grad_w(int i) {
  return R(3) * ((c_of<D>(i, 0) == 0 ? R(2) / R(3) : R(1) / R(6)) * (c_of<D>(i, 1) == 0 ? R(2) / R(3) : R(1) / R(6)) *
                 (D == 3 ? (c_of<D>(i, 2) == 0 ? R(2) / R(3) : R(1) / R(6)) : R(1)));
}

}  // namespace lbm
