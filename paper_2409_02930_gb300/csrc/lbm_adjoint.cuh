// Adjoint (reverse-mode) step kernels: given the adjoint lambda^{n+1} of
// the post-collision populations after step n, they return lambda^n and
// accumulate dJ/dphi (porosity field) and dJ/dlambda, where lambda scales
// every Knudsen coefficient 1/tau^k_a (pore radius and tortuosity enter the
// step only through tortuosity / pore radius, Eq. 26 with the Knudsen
// diffusivity of Sec. 5.1).
//
// The step f^{n+1} = C(S f^n) is differentiated in its own structure:
//   streamed populations P(x)   = pull of f^n with the boundary rules (a1)
//   macro fields     m(x)        = u, Pi, Y_a of P(x) and phi(x)       (a2, a3)
//   gradients        G(x)        = isotropic stencil of m              (a5)
//   node update      f^{n+1}(x)  = collide(P(x), phi(x), G(x), lambda) (a4, a6-a9)
// k_adj_fields forms the macro fields of f^n and keeps the sums they come
// from; k_adj_collide runs the node update backwards (lbm_reverse.cuh);
// k_adj_macro transposes the stencil, runs the macro fields backwards from
// the kept sums and scatters the streamed populations' adjoint to where each
// was pulled from (the transposed pull: every population has one reader);
// k_adj_ghost carries the reservoir ghosts' dependence on the adjacent node's
// velocity.  k_adj_init adds the dependence of the initial equilibria on the
// porosity.
//
// What bounds it: operations and registers (255 in the node update, whose blocks
// of 64 threads make two waves on 256 x 256).  20 steps of the 256 x 256 FP32 slab
// with checkpoints every 10 take 0.85 ms a step (forward, recomputed and reverse)
// with the node update in two-lane dual numbers (15 evaluations per node and
// step) and the pull transposed in a pass of its own, and 0.109 ms written out in
// reverse; 100 steps with checkpoints every 50 take 0.077 ms a step.
#pragma once

#include "lbm_dual.cuh"
#include "lbm_reverse.cuh"
#include "lbm_twopass.cuh"

namespace lbm {

template <int D, int M, bool EN>
LBM_HD constexpr int n_grad() { return 1 + D + (EN ? M * D : 0); }
template <int D, int M, bool EN>
LBM_HD constexpr int n_lat() { return M + 1 + (EN ? 1 : 0); }
// sums behind the macro fields: sa [M], sf, jf [2], sg
template <int M>
LBM_HD constexpr int n_sums() { return M + 4; }

template <class B>
struct AdjArgs {
  const B* f;         // f^n [L][Q][N]
  B* mac;             // macro fields of f^n [2D+M][N]
  B* sums;            // sums behind them [M + 4][N]
  const B* phi;       // [N]
  const B* Tfix;      // [N]
  const B* lam1;      // adjoint of f^{n+1} [L][Q][N]
  B* Pbar;            // adjoint of the streamed populations of step n [L][Q][N]
  B* Gbar;            // adjoint of the gradient inputs [NG][N]
  double* phibar;     // dJ/dphi accumulator [N]
  double* kbar;       // dJ/dlambda accumulator per node [N]
  B* lam0;            // adjoint of f^n [L][Q][N]
  int* status;
};

// Macro fields of f^n and the sums behind them.
template <class B, int M, bool EN>
__global__ void __launch_bounds__(128) k_adj_fields(Params<B> p, InletTables<B> it, AdjArgs<B> a) {
  after_previous();
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= p.N) return;
  const size_t N = p.N;
  int x, y, z;
  node_xyz<B, 2>(p, n, x, y, z);
  B P[n_lat<2, M, EN>() * 9];
  pull_node<B, 2, M, EN>(p, it, a.f, a.phi, x, y, z, P);
  Moments<B, 2, M, EN, false> mo;
  moments_gen<B, 2, M, EN, false>(ArrayPull<B, 2>{P}, mo);
  State<B, 2, M> s;
  s.template from_moments<EN, false>(p, mo, a.phi[n], EN ? B(0) : a.Tfix[n]);
  macro_fields<B, 2, M, EN>(s, [&](int k, const B& v) { a.mac[(size_t)k * N + n] = v; });
#pragma unroll
  for (int k = 0; k < M; ++k) a.sums[(size_t)k * N + n] = mo.sa[k];
  a.sums[(size_t)M * N + n] = mo.sf;
#pragma unroll
  for (int b = 0; b < 2; ++b) a.sums[(size_t)(M + 1 + b) * N + n] = mo.jf[b];
  if (EN) a.sums[(size_t)(M + 3) * N + n] = mo.sg;
}

// Node update backwards: adjoints of the gradient inputs and of the streamed
// populations (the moments' transpose plus the direct relaxation term).
template <class B, int M, bool EN>
__global__ void __launch_bounds__(64) k_adj_collide(Params<B> p, InletTables<B> it, AdjArgs<B> a) {
  constexpr int L = n_lat<2, M, EN>(), REST = 4;
  after_previous();
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= p.N) return;
  const int N = p.N;
  int x, y, z;
  node_xyz<B, 2>(p, n, x, y, z);
  B P[L * 9];
  pull_node<B, 2, M, EN>(p, it, a.f, a.phi, x, y, z, P);
  Moments<B, 2, M, EN, true> mo;
  moments_gen<B, 2, M, EN, true>(ArrayPull<B, 2>{P}, mo);
  State<B, 2, M> s;
  s.template from_moments<EN, true>(p, mo, a.phi[n], EN ? B(0) : a.Tfix[n]);
  Grad<B, 2, M, EN> gr, gb;
  const B* __restrict__ mac = a.mac;
  gr.compute(p, x, y, [&](int k, int nb) { return mac[(size_t)k * N + nb]; });
  const B* __restrict__ lam1 = a.lam1 + n;
  auto lam = [&](int l, int i) { return lam1[(size_t)(unsigned)(l * 9 + i) * (unsigned)N]; };
  MomentBar<B, M> mb;
  B phi_, k_, keep[L];
  collide_reverse<B, M, EN>(p, mo, s, gr, lam, [&](int l, int i) { return P[l * 9 + i]; }, mb, gb, phi_, k_, keep);
  if (bad_state(s, B(1) / s.phi)) flag(a.status, 1);
  a.Gbar[n] = gb.divu;
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    a.Gbar[(size_t)(1 + b) * N + n] = gb.dPi[b];
    if (EN) {
#pragma unroll
      for (int k = 0; k < M; ++k) a.Gbar[(size_t)(3 + 2 * k + b) * N + n] = gb.dY[k][b];
    }
  }
  const B pxy = mb.Pt[0][1] + mb.Pt[1][0];
#pragma unroll
  for (int l = 0; l < L; ++l) {
    const B rest = lam(l, REST);
    const B s0 = l < M ? mb.sa[l < M ? l : 0] : (l == M ? mb.sf : mb.sg);
    const B jx = l < M ? mb.ja[l < M ? l : 0][0] : (l == M ? mb.jf[0] : mb.q[0]);
    const B jy = l < M ? mb.ja[l < M ? l : 0][1] : (l == M ? mb.jf[1] : mb.q[1]);
    B* __restrict__ out = a.Pbar + n;
    Unroll<0, 9>::run([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      constexpr int cx = c_of<2>(i, 0), cy = c_of<2>(i, 1);
      B v = s0;
      if (cx > 0) v += jx;
      if (cx < 0) v -= jx;
      if (cy > 0) v += jy;
      if (cy < 0) v -= jy;
      if (EN && l == M) {
        if (cx != 0) v += mb.Pt[0][0];
        if (cy != 0) v += mb.Pt[1][1];
        if (cx * cy > 0) v += pxy;
        if (cx * cy < 0) v -= pxy;
      }
      if (i != REST) v += keep[l] * (lam(l, i) - rest);
      out[(size_t)(unsigned)(l * 9 + i) * (unsigned)N] = v;
    });
  }
  a.phibar[n] += (double)phi_;
  a.kbar[n] += (double)k_;
}

// With MACRO: adjoint of the macro fields at node n (every node whose stencil
// reads n, with the zero-gradient copy at open x faces), run backwards
// through the state and added to Pbar(n).  Then Pbar(n) is scattered to the
// populations it was pulled from: lam0.  Populations that leave through a
// reservoir have no reader (their adjoint is zero); the adjoint of a missing
// population stays in Pbar for k_adj_ghost.
template <class B, int M, bool EN, bool MACRO>
__global__ void __launch_bounds__(128) k_adj_macro(Params<B> p, AdjArgs<B> a) {
  after_previous();
  constexpr int L = n_lat<2, M, EN>();
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= p.N) return;
  const unsigned N = (unsigned)p.N;
  int x, y, z;
  node_xyz<B, 2>(p, n, x, y, z);
  Site<B, 2> st;
  st.init(p, x, y, 0);
  B sa_[M], sf_ = B(0), jf_[2] = {B(0), B(0)}, sg_ = B(0);
#pragma unroll
  for (int k = 0; k < M; ++k) sa_[k] = B(0);
  if constexpr (MACRO) {
    const bool open = p.bc_lo != BC_PERIODIC;
    B ub[2] = {B(0), B(0)}, Pb[2] = {B(0), B(0)}, Yb[M];
#pragma unroll
    for (int k = 0; k < M; ++k) Yb[k] = B(0);
    auto add = [&](int m, B w, int cx, int cy) {
      const B* __restrict__ G = a.Gbar + m;
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int cb = b == 0 ? cx : cy;
        if (cb == 0) continue;
        const B wc = w * B(cb);
        ub[b] += wc * G[0];
        Pb[b] += wc * G[(size_t)(unsigned)(1 + b) * N];
        if (EN) {
#pragma unroll
          for (int k = 0; k < M; ++k) Yb[k] += wc * G[(size_t)(unsigned)(3 + 2 * k + b) * N];
        }
      }
    };
    Unroll<0, 9>::run([&](auto ic) {
      constexpr int I = decltype(ic)::value;
      constexpr int cx = c_of<2>(I, 0), cy = c_of<2>(I, 1);
      if (I == 4) return;
      const B w = grad_w<B, 2>(I);
      const int my = p.nx * wrapi(y - cy, p.ny);
      int mx = x - cx;
      if (!open) add(wrapi(mx, p.nx) + my, w, cx, cy);
      else if (mx >= 0 && mx < p.nx) add(mx + my, w, cx, cy);
      // the copy across an open face: the face node's own stencil reads it again
      if (cx != 0 && open && x == (cx < 0 ? 0 : p.nx - 1)) add(x + my, w, cx, cy);
    });
    Moments<B, 2, M, EN, false> mo;
#pragma unroll
    for (int k = 0; k < M; ++k) mo.sa[k] = a.sums[(size_t)(unsigned)k * N + n];
    mo.sf = a.sums[(size_t)M * N + n];
#pragma unroll
    for (int b = 0; b < 2; ++b) mo.jf[b] = a.sums[(size_t)(M + 1 + b) * N + n];
    mo.sg = EN ? a.sums[(size_t)(M + 3) * N + n] : B(0);
    State<B, 2, M> s;
    s.template from_moments<EN, false>(p, mo, a.phi[n], EN ? B(0) : a.Tfix[n]);
    // u = phi w, Pi = j (1 - 3 R T - w^2), Y
    StateBar<B, M> S_;
    S_.zero();
    B phi_ = B(0), RT_ = B(0);
    const B RT = s.Rg * s.T;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      phi_ += ub[b] * s.w[b];
      S_.w[b] += ub[b] * s.phi - B(2) * Pb[b] * s.jf[b] * s.w[b];
      S_.jf[b] += Pb[b] * (B(1) - B(3) * RT - s.w[b] * s.w[b]);
      RT_ -= B(3) * Pb[b] * s.jf[b];
    }
    S_.Rg = RT_ * s.T;
    S_.T = EN ? RT_ * s.Rg : B(0);
#pragma unroll
    for (int k = 0; k < M; ++k) S_.Y[k] = Yb[k];
    state_reverse<B, M, EN>(p, s, mo.sg, S_, sa_, sf_, jf_, sg_);
    a.phibar[n] += (double)phi_;
  }
  // every load before the first store: the two arrays may alias for the
  // compiler, and load-store pairs in turn cost a round trip each
  B v[L * 9];
#pragma unroll
  for (int e = 0; e < L * 9; ++e) v[e] = a.Pbar[(size_t)(unsigned)e * N + n];
  Unroll<0, 9>::run([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    constexpr int cx = c_of<2>(i, 0), cy = c_of<2>(i, 1);
    const int h = st.source(cx, cy, 0);
    const unsigned isrc = (h >= 0 || h == SRC_GHOST) ? i : 8 - i;
    const int src = h >= 0 ? h : n;
    B jc = B(0);
    if (cx > 0) jc += jf_[0];
    if (cx < 0) jc -= jf_[0];
    if (cy > 0) jc += jf_[1];
    if (cy < 0) jc -= jf_[1];
#pragma unroll
    for (int l = 0; l < L; ++l) {
      const B t = v[l * 9 + i] + (l < M ? sa_[l < M ? l : 0] : (l == M ? sf_ + jc : sg_));
      if (h == SRC_GHOST) {
        a.Pbar[(size_t)(unsigned)(l * 9 + i) * N + n] = t;
        a.lam0[(size_t)(unsigned)(l * 9 + 8 - i) * N + n] = B(0);    // leaves through the face
      } else {
        a.lam0[(size_t)((unsigned)(l * 9) + isrc) * N + src] = t;
      }
    }
  });
}

// Reservoir ghosts: the missing populations of a face node are equilibria
// moving with u = j / (sum f / phi) of the adjacent node's streamed momentum
// populations.  One thread per row and side; the face's derivatives in u and
// in the node's own porosity come from three dual lanes, the chain to the
// adjacent node's sums is written out.  The sums' adjoint goes straight to
// the populations the adjacent node pulled (lam0).
template <class B, int M, bool EN>
__global__ void __launch_bounds__(32) k_adj_ghost(Params<B> p, InletTables<B> it, AdjArgs<B> a,
                                                  const __grid_constant__ Params<Dual<B, 3>> pd) {
  using T = Dual<B, 3>;
  after_previous();
  const int y = blockIdx.x * blockDim.x + threadIdx.x;
  if (y >= p.ny) return;
  const size_t N = p.N;
  // the two sides run side by side, or in turn where they share the adjacent
  // node (nx = 3)
  for (int side = blockIdx.y; side < 2; side += gridDim.y) {
    if ((side == 0 ? p.bc_lo : p.bc_hi) != BC_INLET) continue;
    const int nb = (side == 0 ? 0 : p.nx - 1) + p.nx * y, xa = side == 0 ? 1 : p.nx - 2, na = xa + p.nx * y;
    Site<B, 2> sa;
    sa.init(p, xa, y, 0);
    B s0 = B(0), j[2] = {B(0), B(0)}, lam[9];
    Unroll<0, 9>::run([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      const size_t at = (size_t)(M * 9 + i) * N + sa.source(c_of<2>(i, 0), c_of<2>(i, 1), 0);
      const B f = a.f[at];
      lam[i] = a.lam0[at];
      s0 += f;
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        if (c_of<2>(i, b) > 0) j[b] += f;
        if (c_of<2>(i, b) < 0) j[b] -= f;
      }
    });
    const B is0 = B(1) / s0, pa = a.phi[na];
    InletTables<T> itd;
#pragma unroll
    for (int k = 0; k < M; ++k) itd.rho[side][k] = T(it.rho[side][k]);
    itd.rho_sum[side] = T(it.rho_sum[side]);
    itd.Rmix[side] = T(it.Rmix[side]);
    itd.Umix[side] = T(it.Umix[side]);
    itd.T[side] = T(it.T[side]);
    Ghost<T, 2> gh;
    gh.side = side;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      gh.u[b] = T(j[b] * pa * is0);
      gh.u[b].d[b] = B(1);
    }
    gh.phi = T(a.phi[nb]);
    gh.phi.d[2] = B(1);
    B acc[3] = {B(0), B(0), B(0)};
    const int into = side == 0 ? 1 : -1;                 // c_x of the missing directions
    ghost_face<T, 2, M, EN>(pd, itd, gh, [&](int l, int cy, int, const T& g) {
      const B pb = a.Pbar[(size_t)(l * 9 + (into + 1) + 3 * (cy + 1)) * N + nb];
#pragma unroll
      for (int k = 0; k < 3; ++k) acc[k] += pb * g.d[k];
    });
    // u_b = j_b phi_a / s0
    const B s_ = -(acc[0] * gh.u[0].v + acc[1] * gh.u[1].v) * is0, r = pa * is0;
    Unroll<0, 9>::run([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      constexpr int cx = c_of<2>(i, 0), cy = c_of<2>(i, 1);
      a.lam0[(size_t)(M * 9 + i) * N + sa.source(cx, cy, 0)] = lam[i] + (s_ + r * (B(cx) * acc[0] + B(cy) * acc[1]));
    });
    a.phibar[na] += (double)((acc[0] * gh.u[0].v + acc[1] * gh.u[1].v) / pa);
    a.phibar[nb] += (double)acc[2];
  }
}

// Objective: J = w * sum over the nodes of plane x = xo of the species-a
// momentum along `axis` of the streamed populations (the flux moment j_a of
// the state); seeds Pbar with its gradient.
template <class B, int D, int M, bool EN>
__global__ void k_adj_seed_flux(Params<B> p, AdjArgs<B> a, int species, int axis, int xo, B w) {
  constexpr int Q = Lat<D>::Q, L = n_lat<D, M, EN>();
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= p.N) return;
  const int N = p.N;
  const bool on = (n % p.nx) == xo;
  for (int l = 0; l < L; ++l)
    for (int i = 0; i < Q; ++i)
      a.Pbar[(size_t)(l * Q + i) * N + n] = (on && l == species) ? w * B(c_of<D>(i, axis)) : B(0);
}

// Initial equilibria: phibar(x) += lambda^0(x)^T df^0(x)/dphi(x).
template <class B, int D, int M, bool EN>
__global__ void __launch_bounds__(128) k_adj_init(Params<B> p, const double* __restrict__ X,
                                                  const double* __restrict__ T0, const double* __restrict__ P0,
                                                  const double* __restrict__ U0v, double cvel, double RU_si,
                                                  AdjArgs<B> a) {
  using T = Dual<B, 1>;
  constexpr int Q = Lat<D>::Q;
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= p.N) return;
  const int N = p.N;
  T phid(a.phi[n]);
  phid.d[0] = B(1);
  double acc = 0.0;
  init_node<T, D, M, EN>(p, X, T0, P0, U0v, cvel, RU_si, n, N, phid, [&](int l, int i, const T& v) {
    acc += (double)a.lam0[(size_t)(l * Q + i) * N + n] * (double)v.d[0];
  });
  a.phibar[n] += acc;
}

// Launch table of the adjoint kernels for one (precision, D, M, energy).
template <class B>
struct AdjOps {
  int (*fields)(const Params<B>&, const InletTables<B>&, const AdjArgs<B>&, cudaStream_t);
  int (*collide)(const Params<B>&, const InletTables<B>&, const AdjArgs<B>&, cudaStream_t);
  // macro fields backwards and transposed pull; with `seed` only the pull
  int (*macro)(const Params<B>&, const AdjArgs<B>&, bool seed, cudaStream_t);
  int (*ghost)(const Params<B>&, const InletTables<B>&, const AdjArgs<B>&, cudaStream_t);
  void (*seed_flux)(const Params<B>&, const AdjArgs<B>&, int species, int axis, int xo, double w, cudaStream_t);
  void (*init)(const Params<B>&, const double*, const double*, const double*, const double*, double, double,
               const AdjArgs<B>&, cudaStream_t);
  int n_grad, n_sums;
};

bool get_adj_ops_f32(int D, int M, int energy, AdjOps<float>* out);
bool get_adj_ops_f64(int D, int M, int energy, AdjOps<double>* out);

}  // namespace lbm
