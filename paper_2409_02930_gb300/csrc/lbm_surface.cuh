// Heterogeneous surface source on the GPU (Sec. 4, Sec. 4.2) and the
// reactive two-pass step that applies it.
//
// Per node and step: mass-action rates with Arrhenius constants, backward
// Euler in the reaction extents over the physical time step solved by
// Newton's method (analytic sparse Jacobian, Gaussian elimination with
// partial pivoting, steps shortened so that no concentration crosses zero).
// Rates, residual and extents are FP64 whatever the population precision;
// the Jacobian is FP64 on the FP64 path and FP32 on the FP32 path, and is
// reused across iterations (iterative refinement to the same FP64 root).  Then the gas mass production
// (Eq. 68, Eq. 69), the new coverages
// (Eq. 70, Eq. 71 with the TPB edge
// steps), the volumetric current (Eq. 74) and the change of the
// fluid internal energy: the unified internal energy of fluid and adsorbed
// phases (Eq. 80, Eq. 85) gains the ohmic heat
// and loses the electric power of the current (Sec. 4.2).
#pragma once

#include "lbm_twopass.cuh"

namespace lbm {

constexpr double R_UNIV_DEV = 8.314462618;    // J/(mol K)

// Mechanism and unit data of a reactive context (device memory, read-only).
// Species are indexed 0..M-1 (gas, mol/m^3 of fluid) then M..M+S-1 (surface,
// mol/m^2); reactant lists hold the integer mass-action orders.
struct MechDev {
  int M, S, R;
  int npart[RMAX];                   // species taking part in each step (nonzero stoichiometry)
  int pidx[RMAX][8];
  double pnu[RMAX][8];
  int nsr[MMAX + SMAX];               // steps in which each species takes part
  int sr_k[MMAX + SMAX][RMAX];
  double sr_nud[MMAX + SMAX][RMAX];
  // nu = A B of rank r (A: the columns of r basis species, B: every species'
  // change by theirs): entries of A per step, of B per species
  int r, bas[MMAX + SMAX];
  int na[RMAX], ai[RMAX][8];
  double av[RMAX][8];
  float avf[RMAX][8];
  int nb[MMAX + SMAX], bi[MMAX + SMAX][MMAX + SMAX];
  double bv[MMAX + SMAX][MMAX + SMAX];
  float bvf[MMAX + SMAX][MMAX + SMAX];
  int nre[RMAX];                     // reactants of each step
  int ridx[RMAX][4];
  int rord[RMAX][4];
  double A[RMAX], Ea[RMAX];
  double gamma, a_s;
  double cvs[SMAX], Us0[SMAX];       // molar C_v / R_U and molar U at T_thermo of the adsorbates
  double m[MMAX];                    // gas molar masses
  double T_thermo;
  double dt;                         // physical time step [s]
  double cvel2;                      // (dx/dt)^2 [m^2/s^2]
  // electrochemistry: TPB (edge) steps run as surface steps whose extent is
  // counted per unit surface (the per-length extent times l_tpb/a_s), so
  // their constants carry the factor l_tpb/a_s and the potential factor
  int edge[RMAX];
  double nel[RMAX];                  // electrons released per step
  double l_tpb, beta_ct, resist, dphi, dx;
  const double* dphi_field;          // per-node potential difference [N] (null: dphi everywhere)
};

constexpr double FARADAY_DEV = 96485.33212;   // C/mol

// q-th entry of A of step k and of B of species j, in the Jacobian's precision
template <class RK> __device__ __forceinline__ RK a_of(const MechDev& mc, int k, int q);
template <> __device__ __forceinline__ float a_of<float>(const MechDev& mc, int k, int q) { return mc.avf[k][q]; }
template <> __device__ __forceinline__ double a_of<double>(const MechDev& mc, int k, int q) { return mc.av[k][q]; }
template <class RK> __device__ __forceinline__ RK b_of(const MechDev& mc, int j, int q);
template <> __device__ __forceinline__ float b_of<float>(const MechDev& mc, int j, int q) { return mc.bvf[j][q]; }
template <> __device__ __forceinline__ double b_of<double>(const MechDev& mc, int j, int q) { return mc.bv[j][q]; }

__device__ __forceinline__ double ipow(double x, int n) {
  double r = 1.0;
  for (int k = 0; k < n; ++k) r *= x;
  return r;
}

// Surface source of one node.  rho_a in kg/m^3 of fluid, T in K; returns
// rhodot[a] (kg/m^3 of porous medium per step), the new coverages and dU
// (fluid internal energy change per unit volume, lattice units).
//
// Mixed precision (iterative refinement): concentrations, rates, the
// residual F = xi - dt r(xi) and the extents are FP64; the Newton systems are
// solved in FP32 (RK = float) or FP64 (RK = double) in the space of the r
// independent species changes (Woodbury identity, r x r instead of R x R: 9
// for the 20 steps and 14 species of the anode mechanism), whose factors are
// reused across iterations (simplified Newton) until the
// contraction of the steps slows down or a step is shortened, when they are
// rebuilt at the current iterate.  The FP64 residual fixes the root, so every variant
// converges to the same FP64 solution.
//
// What bounds it: the FP64 pipe and the latency of the per-thread work arrays
// in local memory.  FP64 divisions are kept out of the loops (one 1/(R_U T)
// per node; the rates' derivatives are products without the factor they are
// taken by, so no rate is divided by a concentration), the concentrations
// follow the extents by increments, and the tests that only steer the
// iteration compare high words as integers.  The factorisation is unrolled
// over the pivots with the pivot row in registers and the triangular solves
// over both indices with the right-hand side in registers, so each multiply-
// add touches local memory once (twice while factorising) instead of twice
// (three times).  Solving in the r independent changes instead of all species'
// (9 for 14 in the anode mechanism: 243 multiply-adds per factorisation for 915,
// 0.3 KB of factors for 0.8) took the 128 x 64 x 64 FP32 reactive step from 4.42
// to 3.55 ms; on the warp form, bound by its chain of steps, it changed nothing.
template <int M, class RK>
__device__ void surface_source_dev(const MechDev& mc, double T, const double* rho_a, double phi, const double* Xs0,
                                   double* rhodot, double* Xs1, double& dU, double& current, double dphi,
                                   int* status) {
  const int S = mc.S, Rn = mc.R, NS = M + mc.S;
  constexpr int NSX = MMAX + SMAX;
  double c0[NSX], d[NSX], kr[RMAX], xi[RMAX];
  const double inv_RT = 1.0 / (R_UNIV_DEV * T);
  for (int a = 0; a < M; ++a) c0[a] = rho_a[a] / mc.m[a];
  for (int s = 0; s < S; ++s) c0[M + s] = mc.gamma * Xs0[s];
  for (int i = 0; i < NS; ++i) d[i] = 0.0;
  for (int k = 0; k < Rn; ++k) {
    double v = mc.A[k] * exp(-mc.Ea[k] * inv_RT);
    // TPB step: rate per unit TPB length, extent counted per unit surface
    if (mc.edge[k]) v *= (mc.l_tpb / mc.a_s) * exp(mc.beta_ct * mc.nel[k] * FARADAY_DEV * dphi * inv_RT);
    kr[k] = v;
    xi[k] = 0.0;
  }
  const double scale = mc.a_s / phi;     // gas concentration change per extent
  const RK rscale = RK(scale);
  // J = I - U diag(scale) B^T A^T with U = dt dr/dc (R x NS, the reactants of
  // each step); by the Woodbury identity J^-1 b = b + U z, z = diag(scale) B^T y,
  // K y = A^T b with K = I - A^T U diag(scale) B^T (r x r, the determinant of J),
  // whose LU factors and U are kept while the iteration reuses them.
  const int r_ = mc.r;
  RK LU[NSX][NSX];
  RK uk[RMAX][4];
  int perm[NSX];
  bool refresh = true, converged = false;
  double prev = 0.0;
  for (int it = 0; it < 40; ++it) {
    double c[NSX], pos[NSX];
    RK b[RMAX], w[NSX];
    for (int i = 0; i < NS; ++i) {
      c[i] = c0[i] + (i < M ? scale : 1.0) * d[i];
      pos[i] = fmax(c[i], 0.0);
    }
    for (int i = 0; i < r_; ++i) w[i] = RK(0);
    if (refresh)
      for (int i = 0; i < r_; ++i)
        for (int j = 0; j < r_; ++j) LU[i][j] = (i == j) ? RK(1) : RK(0);
    for (int k = 0; k < Rn; ++k) {
      // rate r = k prod c^o; where the Jacobian is rebuilt also its derivatives
      // u_j = dt k o_j c_j^(o_j - 1) prod of the others (zero where c_j <= 0)
      const int nre = mc.nre[k];
      double f[4], g[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        f[j] = g[j] = 1.0;
        if (j < nre) {
          const double v = pos[mc.ridx[k][j]];
          const int o = mc.rord[k][j];
          if (o > 1) g[j] = ipow(v, o - 1);
          f[j] = o > 1 ? g[j] * v : v;
        }
      }
      double r = kr[k] * f[0];
      if (nre > 1) r *= f[1];
      if (nre > 2) r *= f[2] * f[3];
      const RK bk = RK(-(xi[k] - mc.dt * r));
      b[k] = bk;
      const int na = mc.na[k];
      for (int q = 0; q < na; ++q) w[mc.ai[k][q]] += a_of<RK>(mc, k, q) * bk;
      if (refresh) {
        const double dk = mc.dt * kr[k];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (j >= nre) continue;
          const int jj = mc.ridx[k][j];
          double u = dk * g[j];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (e != j && e < nre) u *= f[e];
          const RK ur = c[jj] > 0.0 ? RK(u * mc.rord[k][j]) : RK(0);
          const RK us = jj < M ? rscale * ur : ur;
          uk[k][j] = us;
          const int nb = mc.nb[jj];
          for (int e = 0; e < nb; ++e) {
            const RK t = us * b_of<RK>(mc, jj, e);
            const int i2 = mc.bi[jj][e];
            for (int q = 0; q < na; ++q) LU[mc.ai[k][q]][i2] -= a_of<RK>(mc, k, q) * t;
          }
        }
      }
    }
    if (refresh) {
      // LU factors of K with partial pivoting (row order recorded in perm)
      for (int i = 0; i < r_; ++i) perm[i] = i;
#pragma unroll
      for (int cc = 0; cc < NSX; ++cc) {
        if (cc >= r_) break;
        int pv = cc;
        RK best = fabs(LU[cc][cc]);
        for (int k = cc + 1; k < r_; ++k) {
          const RK v = fabs(LU[k][cc]);
          if (v > best) {
            best = v;
            pv = k;
          }
        }
        RK prow[NSX];
        const int pp = perm[pv];
        perm[pv] = perm[cc];
        perm[cc] = pp;
#pragma unroll
        for (int l = 0; l < NSX; ++l) {
          if (l >= r_) break;
          const RK t = LU[cc][l];
          prow[l] = LU[pv][l];
          if (pv != cc) {
            LU[pv][l] = t;
            LU[cc][l] = prow[l];
          }
        }
        const RK inv = RK(1) / prow[cc];
        for (int k = cc + 1; k < r_; ++k) {
          const RK f = LU[k][cc] * inv;
          LU[k][cc] = f;
#pragma unroll
          for (int l = cc + 1; l < NSX; ++l) {
            if (l >= r_) break;
            LU[k][l] -= f * prow[l];
          }
        }
        LU[cc][cc] = inv;                              // the solves multiply by the pivot's reciprocal
      }
      refresh = false;
    }
    // solve J dxi = -F:  w = A^T b, K y = w, z = B^T y (U holds the scale), dxi = b + U z
    RK z[NSX];
    {
      RK y[NSX];
#pragma unroll
      for (int k = 0; k < NSX; ++k) {
        if (k >= r_) break;
        y[k] = w[perm[k]];
#pragma unroll
        for (int l = 0; l < k; ++l) y[k] -= LU[k][l] * y[l];
      }
#pragma unroll
      for (int k = NSX - 1; k >= 0; --k) {
        if (k >= r_) continue;
#pragma unroll
        for (int l = k + 1; l < NSX; ++l) {
          if (l >= r_) break;
          y[k] -= LU[k][l] * y[l];
        }
        y[k] *= LU[k][k];
        w[k] = y[k];
      }
    }
    for (int i = 0; i < NS; ++i) {
      RK t = RK(0);
      const int nb = mc.nb[i];
      for (int e = 0; e < nb; ++e) t += b_of<RK>(mc, i, e) * w[mc.bi[i][e]];
      z[i] = t;
    }
    double dd[NSX], dxi[RMAX];
    for (int i = 0; i < NS; ++i) dd[i] = 0.0;
    for (int k = 0; k < Rn; ++k) {
      RK x = b[k];
      for (int j = 0; j < mc.nre[k]; ++j) x += uk[k][j] * z[mc.ridx[k][j]];
      dxi[k] = (double)x;
      for (int j = 0; j < mc.npart[k]; ++j) dd[mc.pidx[k][j]] += mc.pnu[k][j] * dxi[k];
    }
    // steps that would take a non-negative concentration below zero are shortened
    double alpha = 1.0;
    for (int i = 0; i < NS; ++i) {
      const double di = dd[i] * (i < M ? scale : 1.0);
      if (c[i] >= 0.0 && c[i] + di < 0.0) alpha = fmin(alpha, 0.9 * c[i] / (-di));
    }
    // largest step and extent, by the high words (20 mantissa bits: they only
    // decide when to stop and when to rebuild)
    int dtop = 0, xtop = 0;
    for (int k = 0; k < Rn; ++k) {
      const double st = alpha * dxi[k];
      xi[k] += st;
      dtop = max(dtop, __double2hiint(st) & 0x7fffffff);
      xtop = max(xtop, __double2hiint(xi[k]) & 0x7fffffff);
    }
    for (int i = 0; i < NS; ++i) d[i] += alpha * dd[i];
    const double dmax = __hiloint2double(dtop, 0), xmax = __hiloint2double(xtop, 0);
    if (alpha == 1.0 && dmax <= 1e-14 * (xmax + 1e-300)) {
      converged = true;
      break;
    }
    // rebuild the Jacobian when a step was shortened or the steps stop contracting fast
    refresh = (alpha < 1.0) || (it > 0 && dmax > 0.25 * prev);
    prev = dmax;
  }
  if (!converged) flag(status, 4);
  // moles produced per unit surface, nu^T xi, over the few species of each step
  double dn_all[MMAX + SMAX];
  for (int i = 0; i < NS; ++i) dn_all[i] = 0.0;
  for (int k = 0; k < Rn; ++k)
    for (int j = 0; j < mc.npart[k]; ++j) dn_all[mc.pidx[k][j]] += mc.pnu[k][j] * xi[k];
  for (int a = 0; a < M; ++a) rhodot[a] = mc.a_s * mc.m[a] * dn_all[a];
  double dUs = 0.0;
  for (int s = 0; s < S; ++s) {
    const double dn = dn_all[M + s];
    Xs1[s] = Xs0[s] + dn / mc.gamma;
    const double Us = mc.Us0[s] + mc.cvs[s] * R_UNIV_DEV * (T - mc.T_thermo);
    dUs += mc.a_s * dn * Us;
  }
  // volumetric current: F a_s (electrons per unit surface) per second, the
  // same as F l_tpb (electrons per TPB length) per second
  double ne = 0.0;
  for (int k = 0; k < Rn; ++k)
    if (mc.edge[k]) ne += mc.nel[k] * xi[k];
  current = FARADAY_DEV * mc.a_s * ne / mc.dt;
  // ohmic heat stays in the fluid, electric power leaves (Sec. 4.2)
  double Usrc = 0.0;
  if (mc.l_tpb > 0.0)
    Usrc = ((mc.a_s / mc.l_tpb) * current * current * mc.resist * mc.dx - fabs(dphi) * current) * mc.dt;
  dU = (-dUs + Usrc) / mc.cvel2;
}

// Arguments of the reactive passes.
struct ReactArgs {
  const MechDev* mech;
  const double* Xs_in;     // [S][N]
  double* Xs_out;          // [S][N]
  double* src;             // [M + 2][N]: rhodot_a, then dU, then the volumetric current
};

// Surface source of every node, from the species sums and temperatures that
// the macro-field pass left in aux ([M + 1][N]).
template <class R, int M, int MINB>
__global__ void __launch_bounds__(128, MINB) k_source(int N, const R* aux, const R* __restrict__ phi,
                                                int* status, ReactArgs ra) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const MechDev& mc = *ra.mech;
  double rho[MMAX], Xs0[SMAX], Xs1[SMAX], rd[MMAX], dU = 0.0, cur = 0.0;
  const R ph = phi[n];
  for (int k = 0; k < M; ++k) rho[k] = (double)(aux[(size_t)k * N + n] / ph);
  for (int k = 0; k < mc.S; ++k) Xs0[k] = ra.Xs_in[(size_t)k * N + n];
  const double dphi_n = mc.dphi_field ? mc.dphi_field[n] : mc.dphi;
  surface_source_dev<M, R>(mc, (double)aux[(size_t)M * N + n], rho, (double)ph, Xs0, rd, Xs1, dU, cur, dphi_n, status);
  for (int k = 0; k < M; ++k) ra.src[(size_t)k * N + n] = rd[k];
  ra.src[(size_t)M * N + n] = dU;
  ra.src[(size_t)(M + 1) * N + n] = cur;
  for (int k = 0; k < mc.S; ++k) ra.Xs_out[(size_t)k * N + n] = Xs1[k];
}

// Which form a lattice of N nodes takes; us per reactive step of a D3Q27 anode.
// A warp per node up to 48 (FP32) or 32 (FP64) nodes per SM: its time grows with
// the nodes, a thread per node takes one node's latency until the threads fill
// the GPU (warp / thread: FP32 2,048 nodes 126 / 278, 4,096 181 / 283, 7,168 241 /
// 287, 7,680 281 / 289, 8,192 287 / 287; FP64 48 nodes 101 / 294, 2,048 197 / 367,
// 4,864 350 / 413, 6,144 493 / 442).  Above it a thread per node: without a
// register limit up to two blocks of 128 threads per SM, then limited to 48 (FP32)
// or 64 (FP64) registers, so that more threads hide the latency of the work arrays
// (none / limited: FP32 16,384 nodes 303 / 326, 38,912 431 / 481, 65,536 763 / 648;
// FP64 616 / 642, 1,010 / 1,055, 1,663 / 1,530).
template <class R> constexpr int source_warp_nodes = 152 * (sizeof(R) == 4 ? 48 : 32);
constexpr int source_wide_nodes = 152 * 128 * 2;

// The same source with one warp per node, for lattices too small to fill the
// GPU with a thread per node: there the time is the latency of one node's
// Newton iteration, whose loops a warp runs side by side.  Lane k holds
// reaction k (rate, extent, Jacobian entries), lane i species i
// (concentration) and row i of K in registers; rows are eliminated in pivot
// order without being moved (the pivot lane's row is broadcast by shuffles),
// so no work array is indexed dynamically.  The iteration, its thresholds and
// the precision of every quantity are those of surface_source_dev; sums run
// over a species' steps in the same order, and the concentrations follow the
// extents by increments.  12 x 2 x 2 anode in FP64: see the figures above.
template <class RK, int M>
__global__ void __launch_bounds__(32) k_source_warp(int N, const RK* aux, const RK* __restrict__ phi,
                                                    int* status, ReactArgs ra) {
  constexpr int NSX = MMAX + SMAX;
  constexpr unsigned FULL = 0xffffffffu;
  __shared__ double s_nu[RMAX][NSX], s_c[32], s_x[32];
  __shared__ unsigned char s_k[RMAX][NSX];
  __shared__ RK s_b[32], s_u[RMAX][4], s_K[NSX][NSX + 1], s_y[32], s_bv[NSX][NSX];
  __shared__ unsigned char s_bi[NSX][NSX], s_nb[32];
  const int lane = threadIdx.x;
  const MechDev& mc = *ra.mech;
  const int S = mc.S, Rn = mc.R, NS = M + S, r_ = mc.r;
  const bool sp = lane < NS, re = lane < Rn;
  const int nq = sp ? mc.nsr[lane] : 0;
  for (int q = 0; q < nq; ++q) {
    s_k[q][lane] = (unsigned char)mc.sr_k[lane][q];
    s_nu[q][lane] = mc.sr_nud[lane][q];
  }
  // B of species `lane`, and the basis species of row `lane` of K
  const int nb = sp ? mc.nb[lane] : 0;
  for (int e = 0; e < nb; ++e) {
    s_bi[e][lane] = (unsigned char)mc.bi[lane][e];
    s_bv[e][lane] = b_of<RK>(mc, lane, e);
  }
  s_nb[lane] = (unsigned char)nb;
  const bool rowl = lane < r_;
  const int bs = rowl ? mc.bas[lane] : 0, nqb = rowl ? mc.nsr[bs] : 0;
  int nre = 0, ri[4], ro[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) ri[j] = ro[j] = 0;
  if (re) {
    nre = mc.nre[lane];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < nre) {
        ri[j] = mc.ridx[lane][j];
        ro[j] = mc.rord[lane][j];
      }
  }
  after_previous();                                         // the mechanism is constant, the fields are not
  const int n = blockIdx.x;
  const double ph = (double)phi[n], T = (double)aux[(size_t)M * N + n];
  const double dphi = mc.dphi_field ? mc.dphi_field[n] : mc.dphi;
  const double scale = lane < M ? mc.a_s / ph : 1.0;       // concentration change per extent of species `lane`
  const RK gscale = RK(mc.a_s / ph);
  double c0 = 0.0, Xs0 = 0.0;
  if (lane < M) c0 = (double)(aux[(size_t)lane * N + n] / phi[n]) / mc.m[lane];
  else if (sp) {
    Xs0 = ra.Xs_in[(size_t)(lane - M) * N + n];
    c0 = mc.gamma * Xs0;
  }
  double kr = 0.0;
  const bool edge = re && mc.edge[lane];
  if (re) {
    kr = mc.A[lane] * exp(-mc.Ea[lane] / (R_UNIV_DEV * T));
    if (edge) kr *= (mc.l_tpb / mc.a_s) * exp(mc.beta_ct * mc.nel[lane] * FARADAY_DEV * dphi / (R_UNIV_DEV * T));
  }
  double xi = 0.0, d = 0.0;
  RK row[NSX], inv[NSX], uk[4];
  int pl[NSX], mine = 0;                                    // pivot lanes, and the step in which this row pivots
#pragma unroll
  for (int j = 0; j < 4; ++j) uk[j] = RK(0);
  bool refresh = true, converged = false;
  double prev = 0.0;
  for (int it = 0; it < 40; ++it) {
    const double c = c0 + scale * d;
    s_c[lane] = c;
    __syncwarp();
    double r = kr;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < nre) r *= ipow(fmax(s_c[ri[j]], 0.0), ro[j]);
    const RK b = RK(-(xi - mc.dt * r));
    s_b[lane] = b;
    if (refresh) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (j < nre) {
          const double cj = s_c[ri[j]];
          uk[j] = cj > 0.0 ? RK(mc.dt * r * ro[j] / cj) * (ri[j] < M ? gscale : RK(1)) : RK(0);
        }
        s_u[lane][j] = uk[j];
      }
    }
    __syncwarp();
    if (refresh) {
      // row `lane` of K = I - A^T U diag(scale) B^T
      if (rowl) {
        for (int j = 0; j < r_; ++j) s_K[lane][j] = (j == lane) ? RK(1) : RK(0);
        for (int q = 0; q < nqb; ++q) {
          const int k = s_k[q][bs];
          const RK v = RK(s_nu[q][bs]);
          const int m = mc.nre[k];
          for (int j = 0; j < m; ++j) {
            const int jj = mc.ridx[k][j];
            const RK t = v * s_u[k][j];
            for (int e = 0; e < s_nb[jj]; ++e) s_K[lane][s_bi[e][jj]] -= t * s_bv[e][jj];
          }
        }
      }
#pragma unroll
      for (int j = 0; j < NSX; ++j) row[j] = (rowl && j < r_) ? s_K[lane][j] : RK(0);
      // LU with partial pivoting: the largest entry of the column among the
      // rows not yet taken (compared in single precision, lane in the low bits)
      bool taken = !rowl;
      mine = NSX;
#pragma unroll
      for (int cc = 0; cc < NSX; ++cc) {
        if (cc >= r_) break;
        const unsigned bits = (__float_as_uint((float)fabs(row[cc])) & ~31u) | 32u;
        const unsigned key = taken ? 0u : (bits | (unsigned)lane);
        pl[cc] = (int)(__reduce_max_sync(FULL, key) & 31u);
        if (lane == pl[cc]) {
          taken = true;
          mine = cc;
        }
        inv[cc] = RK(1) / __shfl_sync(FULL, row[cc], pl[cc]);
        const RK f = row[cc] * inv[cc];
#pragma unroll
        for (int j = cc + 1; j < NSX; ++j) {
          if (j >= r_) break;
          const RK pj = __shfl_sync(FULL, row[j], pl[cc]);
          if (!taken) row[j] -= f * pj;
        }
        if (!taken) row[cc] = f;
      }
      refresh = false;
    }
    // solve J dxi = -F:  w = A^T b, K y = w, z = B^T y (U holds the scale), dxi = b + U z
    RK w = RK(0);
    for (int q = 0; q < nqb; ++q) w += RK(s_nu[q][bs]) * s_b[s_k[q][bs]];
#pragma unroll
    for (int cc = 0; cc < NSX; ++cc) {
      if (cc >= r_) break;
      const RK wp = __shfl_sync(FULL, w, pl[cc]);
      if (rowl && mine > cc) w -= row[cc] * wp;
    }
    RK y = RK(0);
#pragma unroll
    for (int cc = NSX - 1; cc >= 0; --cc) {
      if (cc >= r_) continue;
      const RK xc = __shfl_sync(FULL, w, pl[cc]) * inv[cc];
      if (rowl && mine < cc) w -= row[cc] * xc;
      if (lane == cc) y = xc;
    }
    s_y[lane] = y;
    __syncwarp();
    RK z = RK(0);
    for (int e = 0; e < nb; ++e) z += s_bv[e][lane] * s_y[s_bi[e][lane]];
    double dxi = 0.0;
    {
      RK x = b;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const RK zj = __shfl_sync(FULL, z, ri[j]);
        if (j < nre) x += uk[j] * zj;
      }
      if (re) dxi = (double)x;
    }
    s_x[lane] = dxi;
    __syncwarp();
    // steps that would take a non-negative concentration below zero are shortened
    double dd = 0.0;
    for (int q = 0; q < nq; ++q) dd += s_nu[q][lane] * s_x[s_k[q][lane]];
    const double di = dd * scale;
    double alpha = (sp && c >= 0.0 && c + di < 0.0) ? fmin(1.0, 0.9 * c / (-di)) : 1.0;
    if (__any_sync(FULL, alpha < 1.0)) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) alpha = fmin(alpha, __shfl_xor_sync(FULL, alpha, o));
    } else {
      alpha = 1.0;
    }
    xi += alpha * dxi;
    d += alpha * dd;
    // largest step and extent, by the high words (20 mantissa bits: they only
    // decide when to stop and when to rebuild)
    auto top = [&](double v) {
      return __hiloint2double((int)__reduce_max_sync(FULL, (unsigned)__double2hiint(v) & 0x7fffffffu), 0);
    };
    const double dmax = top(alpha * dxi), xmax = top(xi);
    if (alpha == 1.0 && dmax <= 1e-14 * (xmax + 1e-300)) {
      converged = true;
      break;
    }
    refresh = (alpha < 1.0) || (it > 0 && dmax > 0.25 * prev);
    prev = dmax;
  }
  if (!converged && lane == 0) flag(status, 4);
  s_x[lane] = re ? xi : 0.0;
  __syncwarp();
  double dn = 0.0;                                          // moles produced per unit surface, nu^T xi
  for (int q = 0; q < nq; ++q) dn += s_nu[q][lane] * s_x[s_k[q][lane]];
  double dUs = 0.0, ne = edge ? mc.nel[lane] * xi : 0.0;
  if (lane < M) {
    ra.src[(size_t)lane * N + n] = mc.a_s * mc.m[lane] * dn;
  } else if (sp) {
    ra.Xs_out[(size_t)(lane - M) * N + n] = Xs0 + dn / mc.gamma;
    dUs = mc.a_s * dn * (mc.Us0[lane - M] + mc.cvs[lane - M] * R_UNIV_DEV * (T - mc.T_thermo));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    dUs += __shfl_xor_sync(FULL, dUs, o);
    ne += __shfl_xor_sync(FULL, ne, o);
  }
  if (lane == 0) {
    const double current = FARADAY_DEV * mc.a_s * ne / mc.dt;
    double Usrc = 0.0;
    if (mc.l_tpb > 0.0)
      Usrc = ((mc.a_s / mc.l_tpb) * current * current * mc.resist * mc.dx - fabs(dphi) * current) * mc.dt;
    ra.src[(size_t)M * N + n] = (-dUs + Usrc) / mc.cvel2;
    ra.src[(size_t)(M + 1) * N + n] = current;
  }
}

}  // namespace lbm
