// D3Q27 step, lattice by lattice: a block owns NB consecutive nodes and has
// one group of NB threads per lattice (eight for six species with energy), so
// a thread holds the 27 streamed populations of one lattice of one node in
// registers instead of all 216 of the node in shared memory.
//
// What bounds it.  With a thread per node, 216 staged populations (55 KB of
// shared memory per 64 threads) and 255 registers left 8 warps per SM and
// straight-line code of 14,000 instructions per node: at 64 x 32 x 32 (FP32)
// the node update took 91.8 us at 32 % issue, its first pass 56.6 us at 21 %.
// Split by lattice a thread needs about 100 registers and the block's groups
// run the same short code for their own species.
//
// The first pass (k_macro3) sums every lattice and lets one group form the
// macro fields.  The node update (k_collide3) pulls again, takes its gradient
// inputs directly from the neighbours' macro fields (group a differentiates
// Y_a, the last two groups u and Pi; they hit L1/L2, which is cheaper than a
// pass that writes and re-reads 22 fields), forms state, transport and
// mixture quantities once per node in one group, shares the species'
// difference moments d_b (26 per species) through shared memory for the
// coupling sum of Eq. 25, and relaxes each lattice in its own group.
#pragma once

#include "lbm_surface.cuh"

namespace lbm {

// Fields of a node in shared memory, [field][NB].
template <int M, bool EN>
struct SplitFields {
  // sums: per species sa, j, sum |f|; momentum sf, j, Pt (6); energy sg, q
  static constexpr int kSp = 5, kMo = kSp * M, kEn = kMo + 10, kSums = kEn + (EN ? 4 : 0);
  // gradient inputs
  static constexpr int kDiv = kSums, kPi = kDiv + 1, kDY = kPi + 3, kGrad = kDY + (EN ? 3 * M : 0);
  // node quantities: per species v, sa, beta, gd, qY, source; then the mixture's
  static constexpr int kCo = kGrad, kCoN = 8, kMix = kCo + kCoN * M;
  static constexpr int kW = kMix, kT = kW + 3, kF = kT + 1 /* xi, Pex */, kOm = kF + 6, kCf = kOm + 1,
                       kRt = kCf + 1, kCu = kRt + 1, kC2 = kCu + 1, kDq = kC2 + 1, kTot = kDq + 3 /* sf, sg */,
                       kEnd = kTot + 2;
  // the species' difference moments (26 each) reuse the sums' and gradients' place
  static constexpr int kDelta = kEnd;
  static constexpr int kAll = kDelta + 26 * M;
};

template <class R, int M, bool EN>
constexpr size_t split_smem_bytes(int NB, bool collide) {
  using F = SplitFields<M, EN>;
  return sizeof(R) * (size_t)NB * (collide ? F::kAll : F::kSums);
}

// Pulls lattice l of node (x, y, z).
template <class R, int M, bool EN>
__device__ __forceinline__ void pull_lattice(const Params<R>& p, const InletTables<R>& it, const R* __restrict__ src,
                                             const R* __restrict__ phiA, int x, int y, int z, int l, R (&f)[27]) {
  const unsigned N = (unsigned)p.N;
  const R* __restrict__ fl = src + (size_t)(unsigned)(l * 27) * N;
  const int n = x + p.nx * (y + p.ny * z);
  // columns of the three x shifts; open faces read their own node (bounce-back
  // swaps the direction, reservoir values are overwritten below)
  int xs[3];
  bool open[3] = {false, false, false};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int s = x - (c - 1);
    xs[c] = s;
    if (s < 0 || s >= p.nx) {
      open[c] = (s < 0 ? p.bc_lo : p.bc_hi) != BC_PERIODIC;
      xs[c] = wrapi(s, p.nx);
    }
  }
  const int ys[3] = {wrapi(y + 1, p.ny), y, wrapi(y - 1, p.ny)}, zs[3] = {wrapi(z + 1, p.nz), z, wrapi(z - 1, p.nz)};
#pragma unroll
  for (int cz = 0; cz < 3; ++cz)
#pragma unroll
    for (int cy = 0; cy < 3; ++cy) {
      const int row = p.nx * (ys[cy] + p.ny * zs[cz]);
#pragma unroll
      for (int cx = 0; cx < 3; ++cx) {
        const int i = cx + 3 * cy + 9 * cz;
        int s = row + xs[cx];
        unsigned ii = i;
        if (cx != 1 && open[cx]) {
          s = n;
          ii = 26 - i;
        }
        f[i] = fl[(size_t)ii * N + s];
      }
    }
  const bool lo = x == 0 && p.bc_lo == BC_INLET, hi = x == p.nx - 1 && p.bc_hi == BC_INLET;
  if (lo || hi) {
    Ghost<R, 3> gh;
    ghost_velocity<R, 3, M>(p, src, phiA, x, y, z, gh);
    ghost_lattice<R, 3, M, EN>(p, it, gh, l, [&](int cy, int cz, const R& v) {
      const int row = 1 + 3 * (cy + 1) + 9 * (cz + 1);
      if (lo) f[row + 1] = v;
      else f[row - 1] = v;
    });
  }
}

// First pass: macro fields of NB nodes (u, Pi, Y_a), and with AUX the species
// sums and the temperature that the surface source reads.
template <class R, int M, bool EN, int NB, bool AUX>
__global__ void __launch_bounds__(NB * (M + 1 + (EN ? 1 : 0))) k_macro3(Params<R> p, InletTables<R> it, StepArgs<R> a,
                                                                       R* __restrict__ aux) {
  using F = SplitFields<M, EN>;
  extern __shared__ unsigned char smem_raw[];
  const int lane = threadIdx.x % NB, l = threadIdx.x / NB;
  R* S = reinterpret_cast<R*>(smem_raw) + lane;
  const int n = min((int)(blockIdx.x * NB) + lane, p.N - 1);
  int x, y, z;
  node_xyz<R, 3>(p, n, x, y, z);
  R f[27];
  pull_lattice<R, M, EN>(p, it, a.src, a.phi, x, y, z, l, f);
  auto get = [&](int i) { return f[i]; };
  R s, j[3], Pt[3][3];
  if (l == M) {
    lattice_sums<R, 3, 1>(get, s, j, Pt);
    S[F::kMo * NB] = s;
#pragma unroll
    for (int b = 0; b < 3; ++b) S[(F::kMo + 1 + b) * NB] = j[b];
  } else {
    lattice_sums<R, 3, 0>(get, s, j, Pt);
    S[(l < M ? F::kSp * l : F::kEn) * NB] = s;
  }
  __syncthreads();
  if (l != 0 || (int)(blockIdx.x * NB) + lane >= p.N) return;
  Moments<R, 3, M, EN, false> mo;
#pragma unroll
  for (int k = 0; k < M; ++k) mo.sa[k] = S[F::kSp * k * NB];
  mo.sf = S[F::kMo * NB];
#pragma unroll
  for (int b = 0; b < 3; ++b) mo.jf[b] = S[(F::kMo + 1 + b) * NB];
  if (EN) mo.sg = S[F::kEn * NB];
  State<R, 3, M> st;
  st.template from_moments<EN, false>(p, mo, a.phi[n], EN ? R(0) : a.Tfix[n]);
  macro_fields<R, 3, M, EN>(st, [&](int k, const R& v) { a.mac[(size_t)(unsigned)k * (unsigned)p.N + n] = v; });
  if (AUX) {
#pragma unroll
    for (int k = 0; k < M; ++k) aux[(size_t)(unsigned)k * (unsigned)p.N + n] = st.sa[k];
    aux[(size_t)(unsigned)M * (unsigned)p.N + n] = st.T;
  }
}

// Isotropic derivatives of one macro field at a node, from its 27-point
// neighbourhood (zero-gradient copy across open x faces): smoothing weights
// (1/6, 2/3, 1/6) along the other axes, central difference along the axis.
template <class R>
struct Stencil3 {
  unsigned row[3][3];
  int xs[3];
  __device__ __forceinline__ void init(const Params<R>& p, int x, int y, int z) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      int s = x + c - 1;
      if (s < 0) s = (p.bc_lo == BC_PERIODIC) ? s + p.nx : 0;
      if (s >= p.nx) s = (p.bc_hi == BC_PERIODIC) ? s - p.nx : p.nx - 1;
      xs[c] = s;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int b = 0; b < 3; ++b)
        row[c][b] = (unsigned)(p.nx * (wrapi(y + b - 1, p.ny) + p.ny * wrapi(z + c - 1, p.nz)));
  }
  template <bool DX, bool DY, bool DZ>
  __device__ __forceinline__ void grad(const R* __restrict__ g, R& gx, R& gy, R& gz) const {
    const R w0 = R(2) / R(3), w1 = R(1) / R(6);
    R sx[3][3], dx[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        if (!DX && ((!DY && c == 1) || (!DZ && b == 1))) continue;
        const R* q = g + row[c][b];
        const R lo = q[xs[0]], hi = q[xs[2]];
        if (DX) dx[c][b] = hi - lo;
        if (DY || DZ) sx[c][b] = w1 * (lo + hi) + w0 * q[xs[1]];
      }
    if (DX) {
      R t[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) t[c] = w1 * (dx[c][0] + dx[c][2]) + w0 * dx[c][1];
      gx = R(0.5) * (w1 * (t[0] + t[2]) + w0 * t[1]);
    }
    if (DY) {
      R t[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) t[c] = sx[c][2] - sx[c][0];
      gy = R(0.5) * (w1 * (t[0] + t[2]) + w0 * t[1]);
    }
    if (DZ) {
      R t[3];
#pragma unroll
      for (int b = 0; b < 3; ++b) t[b] = sx[2][b] - sx[0][b];
      gz = R(0.5) * (w1 * (t[0] + t[2]) + w0 * t[1]);
    }
  }
};

// Node update of NB nodes; with SRC the reaction sources are added: Eq. 89 to
// the species, Eq. 87 to the momentum and Eq. 88 to the energy lattice
// (src: [M + 2][N] in double, mass production per species, then the change of
// the fluid internal energy).
template <class R, int M, bool EN, int NB, bool SRC, int MINB>
__global__ void __launch_bounds__(NB * (M + 1 + (EN ? 1 : 0)), MINB)
    k_collide3(Params<R> p, InletTables<R> it, StepArgs<R> a, const double* __restrict__ srcv) {
  using F = SplitFields<M, EN>;
  constexpr int L = M + 1 + (EN ? 1 : 0);
  extern __shared__ unsigned char smem_raw[];
  const int lane = threadIdx.x % NB, l = threadIdx.x / NB;
  R* S = reinterpret_cast<R*>(smem_raw) + lane;
  const bool live = (int)(blockIdx.x * NB) + lane < p.N;
  const int n = live ? (int)(blockIdx.x * NB) + lane : p.N - 1;
  const unsigned N = (unsigned)p.N;
  R f[27];
  {
    int x, y, z;
    node_xyz<R, 3>(p, n, x, y, z);
    pull_lattice<R, M, EN>(p, it, a.src, a.phi, x, y, z, l, f);
    Stencil3<R> st;
    st.init(p, x, y, z);
    const R* __restrict__ mac = a.mac;
    if (EN && l < M) {
      R gx, gy, gz;
      st.template grad<true, true, true>(mac + (size_t)(unsigned)(6 + l) * N, gx, gy, gz);
      S[(F::kDY + 3 * l) * NB] = gx;
      S[(F::kDY + 3 * l + 1) * NB] = gy;
      S[(F::kDY + 3 * l + 2) * NB] = gz;
    }
    if (l == M) {
      R gx, gy, gz, u;
      st.template grad<true, false, false>(mac, gx, u, u);
      st.template grad<false, true, false>(mac + N, u, gy, u);
      st.template grad<false, false, true>(mac + (size_t)2 * N, u, u, gz);
      S[F::kDiv * NB] = gx + gy + gz;
    }
    if (l == L - 1) {
      R g, u;
      st.template grad<true, false, false>(mac + (size_t)3 * N, g, u, u);
      S[F::kPi * NB] = g;
      st.template grad<false, true, false>(mac + (size_t)4 * N, u, g, u);
      S[(F::kPi + 1) * NB] = g;
      st.template grad<false, false, true>(mac + (size_t)5 * N, u, u, g);
      S[(F::kPi + 2) * NB] = g;
    }
  }
  auto get = [&](int i) { return f[i]; };
  {
    R s, j[3], Pt[3][3];
    if (l == M) {
      lattice_sums<R, 3, EN ? 2 : 1>(get, s, j, Pt);
      S[F::kMo * NB] = s;
#pragma unroll
      for (int b = 0; b < 3; ++b) S[(F::kMo + 1 + b) * NB] = j[b];
      if (EN) {
        int k = F::kMo + 4;
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
          for (int c = b; c < 3; ++c) S[(k++) * NB] = Pt[b][c];
      }
    } else {
      lattice_sums<R, 3, 1>(get, s, j, Pt);
      const int k = l < M ? F::kSp * l : F::kEn;
      S[k * NB] = s;
#pragma unroll
      for (int b = 0; b < 3; ++b) S[(k + 1 + b) * NB] = j[b];
      if (ScalarTraits<R>::single && l < M) {
        R t = fabs(f[0]);
#pragma unroll
        for (int i = 1; i < 27; ++i) t += fabs(f[i]);
        S[(k + 4) * NB] = t;
      }
    }
  }
  __syncthreads();
  // ---- one group: state, transport, mixture -----------------------------------
  if (l == L - 1) {
    Moments<R, 3, M, EN, true> mo;
#pragma unroll
    for (int k = 0; k < M; ++k) {
      mo.sa[k] = S[F::kSp * k * NB];
#pragma unroll
      for (int b = 0; b < 3; ++b) mo.ja[k][b] = S[(F::kSp * k + 1 + b) * NB];
      if (ScalarTraits<R>::single) mo.sabs[k] = S[(F::kSp * k + 4) * NB];
    }
    mo.sf = S[F::kMo * NB];
#pragma unroll
    for (int b = 0; b < 3; ++b) mo.jf[b] = S[(F::kMo + 1 + b) * NB];
    Grad<R, 3, M, EN> gr;
    gr.divu = S[F::kDiv * NB];
#pragma unroll
    for (int b = 0; b < 3; ++b) gr.dPi[b] = S[(F::kPi + b) * NB];
    if (EN) {
      mo.sg = S[F::kEn * NB];
      int k = F::kMo + 4;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        mo.q[b] = S[(F::kEn + 1 + b) * NB];
#pragma unroll
        for (int c = b; c < 3; ++c) mo.Pt[b][c] = mo.Pt[c][b] = S[(k++) * NB];
#pragma unroll
        for (int q = 0; q < M; ++q) gr.dY[q][b] = S[(F::kDY + 3 * q + b) * NB];
      }
    }
    State<R, 3, M> s;
    s.template from_moments<EN, true>(p, mo, a.phi[n], EN ? R(0) : a.Tfix[n]);
    const R inv_phi = R(1) / s.phi;
    if (live && bad_state(s, inv_phi)) flag(a.status, 1);
    Transport<R, 3, M> tr;
    tr.compute(p, s, inv_phi, &mo.ja[0][0], mo.sabs);
    if (live && tr.used_fp64) flag(a.status, 2);
    R sum_rd = R(0);
#pragma unroll
    for (int k = 0; k < M; ++k) {
      R* c = S + (F::kCo + F::kCoN * k) * NB;
#pragma unroll
      for (int b = 0; b < 3; ++b) c[b * NB] = tr.v[k][b];
      c[3 * NB] = s.sa[k];
      c[4 * NB] = tr.beta[k];
      c[5 * NB] = tr.q[k] * tr.inv_tauk[k];
      c[6 * NB] = tr.q[k] * s.Y[k] * tr.C;
      if (SRC) {
        const R rd = (R)srcv[(size_t)(unsigned)k * N + n];
        c[7 * NB] = rd;
        sum_rd += rd;
      }
    }
    Mixture<R, 3> mix;
    mix.template compute<M, EN>(p, mo, s, inv_phi, tr, gr);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      Axis<R> ax;
      mix.momentum_axis(s.w[b], s.inv_sf, b, gr.dPi[b], ax);
      S[(F::kW + b) * NB] = s.w[b];
      S[(F::kF + 2 * b) * NB] = ax.m[1];
      S[(F::kF + 2 * b + 1) * NB] = ax.m[2];
    }
    S[F::kT * NB] = s.T;
    S[F::kOm * NB] = mix.omega;
    S[F::kCf * NB] = (SRC ? mix.omega + sum_rd * s.inv_sf : mix.omega) * s.sf;     // Eq. 42, Eq. 87
    S[F::kTot * NB] = s.sf + sum_rd;                                               // Eq. 78
    if (EN) {
      R cU = mix.omega * s.sf * mix.U, c2 = mix.omega * s.sf, tot = mo.sg;
      if (SRC) {
        // source distribution with the post-reaction density and internal
        // energy (Eq. 86): phi rho U gains dU, phi rho gains the sum of the sources
        const R dU = (R)srcv[(size_t)(unsigned)M * N + n];
        cU += dU;
        c2 += sum_rd;
        tot += dU + sum_rd * mix.hw2;
      }
      S[F::kRt * NB] = mix.RT;
      S[F::kCu * NB] = cU;
      S[F::kC2 * NB] = c2;
      S[(F::kTot + 1) * NB] = tot;
#pragma unroll
      for (int b = 0; b < 3; ++b) S[(F::kDq + b) * NB] = mix.Dq[b];
    }
  }
  __syncthreads();
  R* __restrict__ dn = a.dst + (size_t)(unsigned)(l * 27) * N + n;
  auto put = [&](int i, const R& v) {
    if (live) dn[(size_t)(unsigned)i * N] = v;
  };
  R w[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) w[b] = S[(F::kW + b) * NB];
  if (l < M) {
    // ---- species l (Eq. 21, Eq. 25) -----------------------------------------
    const R* c = S + (F::kCo + F::kCoN * l) * NB;
    const R sa = c[3 * NB], beta = c[4 * NB];
    SpeciesTarget<R, 3> t;
    t.th = R(0.5) * p.Ra[l] * S[F::kT * NB];
    t.gd = c[5 * NB];
    t.gE = t.gd * sa;
    t.qY = c[6 * NB];
    t.cE = R(2) * beta * sa;
    R total = sa;
    if (SRC) {
      t.cE += c[7 * NB];                              // R^r = fdot^r dt
      total += c[7 * NB];
    }
    const R v[3] = {c[0], c[NB], c[2 * NB]};
    SpeciesAxes<R, 3> ax;
    ax.set(w, v, sa, t.th);
    R* D0 = S + F::kDelta * NB;
    R own0[9], own1[9], own2[9];
    ax.template delta<0>(own0);
    ax.template delta<1>(own1);
    ax.template delta<2>(own2);
    {
      R* d = D0 + 26 * l * NB;
#pragma unroll
      for (int e = 1; e < 9; ++e) d[(e - 1) * NB] = own0[e];
#pragma unroll
      for (int e = 0; e < 9; ++e) d[(8 + e) * NB] = own1[e];
#pragma unroll
      for (int e = 0; e < 9; ++e) d[(17 + e) * NB] = own2[e];
    }
    asm volatile("bar.sync 1, %0;\n" ::"n"(NB * M) : "memory");     // the species' groups
    R D[M];
#pragma unroll
    for (int b = 0; b < M; ++b) D[b] = p.invDmm[l][b];              // zero on the diagonal
    auto couple = [&](int e) {
      R s = D[0] * D0[e * NB];
#pragma unroll
      for (int b = 1; b < M; ++b) s += D[b] * D0[(26 * b + e) * NB];
      return s;
    };
    const R keep = R(1) - R(2) * beta;
    R T2[9], T1[9], acc;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      T2[e] = t.template entry<2>(ax, w, e % 3, e / 3, own2[e], couple(17 + e));
      T1[e] = t.template entry<1>(ax, w, e % 3, e / 3, own1[e], couple(8 + e));
    }
    R m[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) m[e] = T2[e] - T1[e];
    acc = relax_dirs<R, 3, false>(get, -1, keep, m, nullptr, put);
#pragma unroll
    for (int e = 0; e < 9; ++e) m[e] = T2[e] + T1[e];
    acc += relax_dirs<R, 3, false>(get, 1, keep, m, nullptr, put);
#pragma unroll
    for (int e = 1; e < 9; ++e)
      m[e] = t.template entry<0>(ax, w, e % 3, e / 3, own0[e], couple(e - 1)) - R(2) * T2[e];
    acc += relax_dirs<R, 3, false>(get, 0, keep, m, nullptr, put);
    put(13, total - acc);
  } else {
    R m[3][9], ex[3] = {R(0), R(0), R(0)}, total;
    if (l == M) {
      // ---- momentum (Eq. 42, Eq. 44, Eq. 87) -----------------------------------
      Axis<R> ax[3];
#pragma unroll
      for (int b = 0; b < 3; ++b) ax[b].set(R(1), S[(F::kF + 2 * b) * NB], S[(F::kF + 2 * b + 1) * NB]);
      product_moments<R, 3>(S[F::kCf * NB], ax, m);
      total = S[F::kTot * NB];
    } else {
      // ---- energy (Eq. 43, Eq. 51, Eq. 54, Eq. 88) ------------------------------
      energy_moments<R, 3>(S[F::kCu * NB], S[F::kC2 * NB], S[F::kRt * NB], w, m);
#pragma unroll
      for (int b = 0; b < 3; ++b) ex[b] = S[(F::kDq + b) * NB];
      total = S[(F::kTot + 1) * NB];
    }
    const R keep = R(1) - S[F::kOm * NB];
    R t[9], acc;
#pragma unroll
    for (int e = 0; e < 9; ++e) t[e] = m[2][e] - m[1][e];
    acc = relax_dirs<R, 3, true>(get, -1, keep, t, ex, put);
#pragma unroll
    for (int e = 0; e < 9; ++e) t[e] = m[2][e] + m[1][e];
    acc += relax_dirs<R, 3, true>(get, 1, keep, t, ex, put);
#pragma unroll
    for (int e = 1; e < 9; ++e) t[e] = m[0][e] - R(2) * m[2][e];
    acc += relax_dirs<R, 3, true>(get, 0, keep, t, ex, put);
    put(13, total - acc);
  }
}

}  // namespace lbm
