// D3Q27 step, lattice by lattice: a block owns NB consecutive nodes and has
// one group of NB threads per lattice (eight for six species with energy), so
// a thread holds the 27 streamed populations of one lattice of one node in
// registers instead of all 216 of the node in shared memory.
//
// What bounds it.  With a thread per node, 216 staged populations (55 KB of
// shared memory per 64 threads) and 255 registers left 8 warps per SM and
// straight-line code of 14,000 instructions per node: 5.6 ms per step of the
// 256 x 128 x 128 FP32 anode.  Split by lattice the block's groups run the same
// short code for their own species.  Whatever one group did alone for the
// whole block then set its pace (instructions that one warp runs once are
// fetched at about eight cycles each: state and transport of the 32 nodes in
// the last group 5,700 cycles, six derivatives in the momentum group 7,600, of
// 14,000 in all), so the species' groups now share that work too.
//
// The first pass (k_macro3) sums every lattice and lets one group form the
// macro fields.  In the node update (k_collide3)
//   - every species' group pulls, sums, differentiates its Y_a and one of u and
//     Pi straight from the neighbours' macro fields (they hit L1/L2; a pass of
//     its own wrote and re-read 22 fields);
//   - the last group forms the state; the species' groups set up their row of
//     the diffusion system and solve it together (Gauss-Jordan, the pivot row
//     through shared memory; the matrix is row diagonally dominant);
//   - the species share their difference moments d_b (26 each) through shared
//     memory for the coupling sum of Eq. 25, read 16 bytes at a time and summed
//     two at a time (packed FP32 multiply-add), while the last group forms the
//     mixture quantities; every group relaxes its own lattice.
#pragma once

#include "lbm_surface.cuh"

namespace lbm {

// Fields of a node in shared memory, [field][NB], then the species'
// difference moments [M][NB][kStride]: z order 0 at kO0 (8 entries, without
// the zeroth moment), 1 at kO1 and 2 at kO2 (9 each).  The stride is an odd
// number of 16-byte units, so 16-byte accesses of consecutive nodes touch
// every bank once.
template <class R, int M, bool EN>
struct SplitFields {
  // sums: per species sa, j, sum |f|; momentum sf, j, Pt (6); energy sg, q
  static constexpr int kSp = 5, kMo = kSp * M, kEn = kMo + 10, kSums = kEn + (EN ? 4 : 0);
  // gradient inputs: d_b u_b, d_b Pi_b, d_b Y_a
  static constexpr int kU = kSums, kDY = kU + 6, kGrad = kDY + (EN ? 3 * M : 0);
  // state: w, T, sum of sa, sqrt(T)/phi, Y_b C/2; row sums and margins of the
  // diffusion system; v_a; sources
  static constexpr int kW = kGrad, kT = kW + 3, kSS = kT + 1, kKT = kSS + 1, kHY = kKT + 1, kCond = kHY + M,
                       kV = kCond + 2 * M, kRd = kV + 3 * M;
  // momentum axes, relaxation, prefactor, total; pivot rows
  static constexpr int kF = kRd + M, kOm = kF + 6, kCf = kOm + 1, kTot = kCf + 1, kPv = kTot + 1,
                       kAll = kPv + M * (M + 3);
  static constexpr int kStride = sizeof(R) == 4 ? 36 : 30, kO0 = 0, kO1 = 8, kO2 = sizeof(R) == 4 ? 20 : 18;
};

// With PARK the populations wait in shared memory, not in registers, between
// their sums and their relaxation.
template <class R, int M, bool EN>
constexpr size_t split_smem_bytes(int NB, bool collide, bool park) {
  using F = SplitFields<R, M, EN>;
  return sizeof(R) * (size_t)NB *
         (collide ? F::kAll + M * F::kStride + (park ? 27 * (M + 1 + (EN ? 1 : 0)) : 0) : F::kSums);
}

// FP64 lattices up to these many nodes take blocks of 8 and of 16 nodes.  An
// FP64 instruction of a warp holds its SM's only FP64 pipe for 16 cycles, so a
// small lattice is bound by the pipes of the few SMs that its blocks reach:
// 48 nodes in blocks of 32 ran 16 warps on two SMs, in blocks of 8 four warps on
// each of six.  Larger lattices lose, since more warps carry the same nodes.
// us per step with 32 / 16 / 8 nodes in a block: 12 x 2 x 2 88 / 63 / 56, 512
// nodes 85 / 61 / 54, 1,024 85 / 61 / 74, 4,096 152 / 123 / 137, 4,864 153 / 126,
// 5,120 153 / 162, 8,192 153 / 201 / 238; reactive 12 x 2 x 2 141 / 115 / 107.  FP32 gains nothing (12 x 2 x 2 9.5 /
// 10.1 / 9.4, 4,096 nodes 12.9 / 13.4 / 16.8).
constexpr int split3d_nodes8 = 152 * 4, split3d_nodes16 = 152 * 32;

// Threads of a block of NB nodes: the species' groups of NB threads first,
// rounded up to whole warps, then the momentum and the energy group in warps of
// their own.  With NB < 32 a warp holds several species, and threads beyond the
// last species or node repeat another thread's work (same values to the same
// places).
template <int NB, int M, bool EN>
struct SplitThreads {
  static constexpr int kSp = (M * NB + 31) / 32 * 32, kOne = NB < 32 ? 32 : NB, kAll = kSp + kOne * (EN ? 2 : 1);
};

// lattice of this thread; where a warp holds one lattice, known to the compiler
// as one value per warp (addresses of its planes then come from uniform registers)
template <int NB, int M, bool EN>
__device__ __forceinline__ int group_of() {
  using B = SplitThreads<NB, M, EN>;
  const int t = (int)threadIdx.x;
  if (NB % 32 == 0) return __shfl_sync(0xffffffffu, t / NB, 0);
  return t < B::kSp ? min(t / NB, M - 1) : M + (t - B::kSp) / B::kOne;
}

// Named barriers among `n` threads of the block, whole warps.  A warp may come
// here from branches that only some of its lanes took (reservoir and wall
// columns, the FP64 solve, a flag), so it reconverges first, and the forms are
// those that do not ask for a converged warp (bar.* is the aligned form, which
// a warp that arrives in parts would be counted at more than once).
__device__ __forceinline__ void bar_sync(int id, int n) {
  __syncwarp();
  asm volatile("barrier.cta.sync %0, %1;\n" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int n) {
  __syncwarp();
  asm volatile("barrier.cta.arrive %0, %1;\n" ::"r"(id), "r"(n) : "memory");
}

// two values as one register pair: FP32 pairs use the packed multiply-add
template <class R> struct Pair;
template <> struct Pair<float> {
  unsigned long long v;
  __device__ __forceinline__ static Pair make(float a, float b) {
    Pair p;
    asm("mov.b64 %0, {%1, %2};" : "=l"(p.v) : "f"(a), "f"(b));
    return p;
  }
  __device__ __forceinline__ void fma(const Pair& a, const Pair& b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(v) : "l"(a.v), "l"(b.v));
  }
  __device__ __forceinline__ void get(float& a, float& b) const { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
};
template <> struct Pair<double> {
  double a, b;
  __device__ __forceinline__ static Pair make(double x, double y) { return Pair{x, y}; }
  __device__ __forceinline__ void fma(const Pair& x, const Pair& y) {
    a += x.a * y.a;
    b += x.b * y.b;
  }
  __device__ __forceinline__ void get(double& x, double& y) const {
    x = a;
    y = b;
  }
};
// 16 bytes of shared memory as pairs
__device__ __forceinline__ void load16(const float* s, Pair<float>* o) {
  const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(s);
  o[0].v = t.x;
  o[1].v = t.y;
}
__device__ __forceinline__ void load16(const double* s, Pair<double>* o) {
  const double2 t = *reinterpret_cast<const double2*>(s);
  o[0] = Pair<double>{t.x, t.y};
}

// CNT values to shared memory, 16 bytes at a time (the last unit padded)
template <int CNT>
__device__ __forceinline__ void store16(float* s, const float* m) {
#pragma unroll
  for (int q = 0; q < CNT; q += 4)
    *reinterpret_cast<float4*>(s + q) = make_float4(m[q], q + 1 < CNT ? m[q + 1] : 0.f, q + 2 < CNT ? m[q + 2] : 0.f,
                                                    q + 3 < CNT ? m[q + 3] : 0.f);
}
template <int CNT>
__device__ __forceinline__ void store16(double* s, const double* m) {
#pragma unroll
  for (int q = 0; q < CNT; q += 2)
    *reinterpret_cast<double2*>(s + q) = make_double2(m[q], q + 1 < CNT ? m[q + 1] : 0.0);
}

// sum_b X[b] d_b of CNT difference moments at offset OFF: 16 bytes per read
template <class R, int M, int STRIDE, int NB, int CNT>
__device__ __forceinline__ void couple(const R* __restrict__ d, const R (&X)[M], R (&out)[9]) {
  constexpr int PER = 16 / (int)sizeof(R), NV = (CNT + PER - 1) / PER, NP = NV * PER / 2;
  Pair<R> acc[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) acc[q] = Pair<R>::make(R(0), R(0));
#pragma unroll
  for (int b = 0; b < M; ++b) {
    const Pair<R> x = Pair<R>::make(X[b], X[b]);
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      Pair<R> v[PER / 2];
      load16(d + b * NB * STRIDE + q * PER, v);
#pragma unroll
      for (int k = 0; k < PER / 2; ++k) acc[q * (PER / 2) + k].fma(x, v[k]);
    }
  }
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    R a, b;
    acc[q].get(a, b);
    if (2 * q < CNT) out[2 * q] = a;
    if (2 * q + 1 < CNT) out[2 * q + 1] = b;
  }
}

// Row offsets (elements) of the 3 x 3 neighbouring rows of node (x, y, z) and
// the x offsets of its neighbours (wrapped, or clamped to the boundary node
// with CLAMP at open faces).
template <class R>
struct Rows3 {
  int row[3][3];          // [z + cz][y + cy] rows, at column x
  int dx[3];
  template <bool CLAMP>
  __device__ __forceinline__ void init(const Params<R>& p, int x, int y, int z) {
    const int ys[3] = {wrapi(y - 1, p.ny), y, wrapi(y + 1, p.ny)}, zs[3] = {wrapi(z - 1, p.nz), z, wrapi(z + 1, p.nz)};
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int b = 0; b < 3; ++b) row[c][b] = x + p.nx * (ys[b] + p.ny * zs[c]);
    dx[0] = x > 0 ? -1 : ((CLAMP && p.bc_lo != BC_PERIODIC) ? 0 : p.nx - 1);
    dx[1] = 0;
    dx[2] = x < p.nx - 1 ? 1 : ((CLAMP && p.bc_hi != BC_PERIODIC) ? 0 : 1 - p.nx);
  }
};

// Velocity of the reservoir ghost beside face node (x, y, z) (the adjacent
// node's, all of whose sources are inside); rolled loops, few nodes take it.
template <class R, int M>
__device__ __forceinline__ void ghost_velocity3(const Params<R>& p, const R* __restrict__ src,
                                                const R* __restrict__ phiA, int x, int y, int z, Ghost<R, 3>& gh) {
  gh.side = x == 0 ? 0 : 1;
  const int xa = gh.side == 0 ? 1 : p.nx - 2;
  R s0 = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll 1
  for (int cz = -1; cz <= 1; ++cz)
#pragma unroll 1
    for (int cy = -1; cy <= 1; ++cy) {
      const R* q = src + (size_t)(unsigned)(M * 27 + 3 * (cy + 1) + 9 * (cz + 1)) * (unsigned)p.N +
                   (xa + p.nx * (wrapi(y - cy, p.ny) + p.ny * wrapi(z - cz, p.nz)));
      const R a = q[1], b = q[(size_t)(unsigned)p.N], c = q[(size_t)2 * (unsigned)p.N - 1];
      const R r = a + c + b;
      s0 += r;
      jx += c - a;
      jy += R(cy) * r;
      jz += R(cz) * r;
    }
  const R rho_f = s0 / phiA[xa + p.nx * (y + p.ny * z)];
  gh.u[0] = jx / rho_f;
  gh.u[1] = jy / rho_f;
  gh.u[2] = jz / rho_f;
  gh.phi = phiA[x + p.nx * (y + p.ny * z)];
}

// Pulls lattice l of node (x, y, z).  Every address is a row pointer plus the
// direction's plane (one wide multiply-add each); the planes' byte stride fits
// 32 bits because a D3Q27 state that fits the card has fewer than 2^29 nodes.
// Open faces load their wrapped column first and are patched below.
template <class R, int M, bool EN>
__device__ __forceinline__ void pull_lattice(const Params<R>& p, const InletTables<R>& it, const R* __restrict__ src,
                                             const R* __restrict__ phiA, int x, int y, int z, int l, R (&f)[27]) {
  const unsigned plane = (unsigned)p.N * (unsigned)sizeof(R);
  const char* fl = reinterpret_cast<const char*>(src) + (size_t)(unsigned)(l * 27) * plane;
  Rows3<R> r;
  r.template init<false>(p, x, y, z);
#pragma unroll
  for (int cz = 0; cz < 3; ++cz)
#pragma unroll
    for (int cy = 0; cy < 3; ++cy)
#pragma unroll
      for (int cx = 0; cx < 3; ++cx) {
        const int i = cx + 3 * cy + 9 * cz;
        const R* q = reinterpret_cast<const R*>(fl + (size_t)(unsigned)i * plane);
        f[i] = q[r.row[2 - cz][2 - cy] + r.dx[2 - cx]];
      }
  const bool flo = x == 0 && p.bc_lo != BC_PERIODIC, fhi = x == p.nx - 1 && p.bc_hi != BC_PERIODIC;
  if (flo || fhi) {
    const int n = r.row[1][1];
    if ((flo ? p.bc_lo : p.bc_hi) == BC_BOUNCEBACK) {
#pragma unroll
      for (int i = 0; i < 27; i += 3) {
        const R v = reinterpret_cast<const R*>(fl + (size_t)(unsigned)(flo ? 24 - i : 26 - i) * plane)[n];
        if (flo) f[i + 2] = v;
        else f[i] = v;
      }
    } else {
      Ghost<R, 3> gh;
      ghost_velocity3<R, M>(p, src, phiA, x, y, z, gh);
      ghost_lattice<R, 3, M, EN>(p, it, gh, l, [&](int cy, int cz, const R& v) {
        const int row = 1 + 3 * (cy + 1) + 9 * (cz + 1);
        if (flo) f[row + 1] = v;
        else f[row - 1] = v;
      });
    }
  }
}

// First pass: macro fields of NB nodes (u, Pi, Y_a), and with AUX the species
// sums and the temperature that the surface source reads.
template <class R, int M, bool EN, int NB, bool AUX>
__global__ void __launch_bounds__(SplitThreads<NB, M, EN>::kAll) k_macro3(Params<R> p, InletTables<R> it, StepArgs<R> a,
                                                                          R* aux) {
  using F = SplitFields<R, M, EN>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  after_previous();
  const int lane = threadIdx.x % NB, l = group_of<NB, M, EN>();
  R* S = reinterpret_cast<R*>(smem_raw) + lane;
  const int n = min((int)(blockIdx.x * NB) + lane, p.N - 1);
  {
    int x, y, z;
    node_xyz<R, 3>(p, n, x, y, z);
    R f[27];
    pull_lattice<R, M, EN>(p, it, a.src, a.phi, x, y, z, l, f);
    // every group takes the first moments: one code path for all lattices
    R s, j[3], Pt[3][3];
    lattice_sums<R, 3, 1>([&](int i) { return f[i]; }, s, j, Pt);
    S[(l < M ? F::kSp * l : (l == M ? F::kMo : F::kEn)) * NB] = s;
    if (l == M) {
#pragma unroll
      for (int b = 0; b < 3; ++b) S[(F::kMo + 1 + b) * NB] = j[b];
    }
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

// Isotropic derivatives of macro field g at a node from its 27-point
// neighbourhood: smoothing weights (1/6, 2/3, 1/6) along the other axes,
// central difference along the axis.
template <class R>
__device__ __forceinline__ void grad3(const Rows3<R>& r, const R* __restrict__ g, R (&o)[3]) {
  const R w0 = R(2) / R(3), w1 = R(1) / R(6);
  R sx[3][3], t[3];
  o[0] = R(0);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const R* q = g + r.row[c][b];
      const R lo = q[r.dx[0]], hi = q[r.dx[2]];
      const R w = R(0.5) * (b == 1 ? w0 : w1) * (c == 1 ? w0 : w1);
      o[0] += w * (hi - lo);
      sx[c][b] = w1 * (lo + hi) + w0 * q[0];
    }
    t[c] = sx[c][2] - sx[c][0];
  }
  o[1] = R(0.5) * (w1 * (t[0] + t[2]) + w0 * t[1]);
#pragma unroll
  for (int b = 0; b < 3; ++b) t[b] = sx[2][b] - sx[0][b];
  o[2] = R(0.5) * (w1 * (t[0] + t[2]) + w0 * t[1]);
}

// Derivative of field g along `axis` (0 x, 1 y, 2 z) only.
template <class R>
__device__ __forceinline__ R grad_axis3(const Rows3<R>& r, const R* __restrict__ g, int axis) {
  const R w0 = R(2) / R(3), w1 = R(1) / R(6);
  R s = R(0);
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      // c, b run over the other two axes; the pair along the axis is lo, hi
      const R w = R(0.5) * (b == 1 ? w0 : w1) * (c == 1 ? w0 : w1);
      const int lo = axis == 0 ? r.row[c][b] + r.dx[0] : (axis == 1 ? r.row[c][0] + r.dx[b] : r.row[0][c] + r.dx[b]);
      const int hi = axis == 0 ? r.row[c][b] + r.dx[2] : (axis == 1 ? r.row[c][2] + r.dx[b] : r.row[2][c] + r.dx[b]);
      s += w * (g[hi] - g[lo]);
    }
  return s;
}

// Row l of the FP64 diffusion solve of one node (FP32 lattices above the
// condition bound): the whole system from the sums in shared memory.
template <class R, int M, bool EN, int NB>
__device__ __noinline__ void solve_row_fp64(const Params<R>& p, const R* S, R phi, int l, R (&v)[3]) {
  using F = SplitFields<R, M, EN>;
  typename Transport<float, 3, M>::Fp64System y;
  y.phi = phi; y.sf = S[F::kMo * NB]; y.T = S[F::kT * NB]; y.Kc = p.Kc;
  const R ss = S[F::kSS * NB];
  for (int a = 0; a < M; ++a) {
    const R sa = S[F::kSp * a * NB];
    y.sa[a] = sa;
    y.Y[a] = sa / ss;
    y.knc[a] = p.knudsen ? p.knc[a] : R(0);
    y.tiny[a] = Transport<R, 3, M>::unresolved(sa, ss, S[(F::kSp * a + 4) * NB]);
    for (int b = 0; b < M; ++b) y.D_[a][b] = p.invDmm[a][b];
    for (int b = 0; b < 3; ++b) y.ja[a][b] = S[(F::kSp * a + 1 + b) * NB];
  }
  for (int b = 0; b < 3; ++b) y.w[b] = S[(F::kW + b) * NB];
  Transport<float, 3, M>::solve_system(y);
  for (int b = 0; b < 3; ++b) v[b] = y.v[l][b];
}

// Node update of NB nodes; with SRC the reaction sources are added: Eq. 89 to
// the species, Eq. 87 to the momentum and Eq. 88 to the energy lattice
// (src: [M + 2][N] in double, mass production per species, then the change of
// the fluid internal energy).
template <class R, int M, bool EN, int NB, bool SRC, int MINB, bool PARK>
__global__ void __launch_bounds__(SplitThreads<NB, M, EN>::kAll, MINB)
    k_collide3(Params<R> p, InletTables<R> it, StepArgs<R> a, const double* srcv) {
  using F = SplitFields<R, M, EN>;
  constexpr int L = M + 1 + (EN ? 1 : 0);
  constexpr int TS = SplitThreads<NB, M, EN>::kSp, T1 = SplitThreads<NB, M, EN>::kOne;
  // barriers: 0 all; 1 state ready (last group to the species), 2 pivot rows
  // (species), 3 mixture ready (last group to the momentum group), 4
  // difference moments (species), 5 v ready (species to the last group)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  after_previous();
  const int lane = threadIdx.x % NB, l = group_of<NB, M, EN>();
  R* S = reinterpret_cast<R*>(smem_raw) + lane;
  R* D0 = reinterpret_cast<R*>(smem_raw) + F::kAll * NB + lane * F::kStride;
  const bool live = (int)(blockIdx.x * NB) + lane < p.N;
  const int n = live ? (int)(blockIdx.x * NB) + lane : p.N - 1;
  const unsigned N = (unsigned)p.N;
  R f[27];
  // what the groups need after the first barrier is loaded before it, so that
  // it waits with the pull
  R phi = R(0), Tf = R(0), dU = R(0);
  {
    int x, y, z;
    node_xyz<R, 3>(p, n, x, y, z);
    pull_lattice<R, M, EN>(p, it, a.src, a.phi, x, y, z, l, f);
    if (l == L - 1) {
      phi = a.phi[n];
      if (!EN) Tf = a.Tfix[n];
      if (SRC) dU = (R)srcv[(size_t)(unsigned)M * N + n];
    }
    if (l < M) {
      if (SRC) S[(F::kRd + l) * NB] = (R)srcv[(size_t)(unsigned)l * N + n];
      Rows3<R> r;
      r.template init<true>(p, x, y, z);
      if (EN) {
        R g[3];
        grad3<R>(r, a.mac + (size_t)(unsigned)(6 + l) * N, g);
#pragma unroll
        for (int b = 0; b < 3; ++b) S[(F::kDY + 3 * l + b) * NB] = g[b];
      }
#pragma unroll 1
      for (int q = l; q < 6; q += M)
        S[(F::kU + q) * NB] = grad_axis3<R>(r, a.mac + (size_t)(unsigned)q * N, q < 3 ? q : q - 3);
    }
  }
  R* __restrict__ parked = S + (F::kAll + M * F::kStride + 27 * l) * NB;
  auto get = [&](int i) { return PARK ? parked[i * NB] : f[i]; };
  R s0, j0[3], sabs = R(0);
  {
    auto get = [&](int i) { return f[i]; };
    R Pt[3][3];
    const int k = l < M ? F::kSp * l : (l == M ? F::kMo : F::kEn);
    if (EN && l == M) {
      lattice_sums<R, 3, 2>(get, s0, j0, Pt);
      int e = F::kMo + 4;
#pragma unroll
      for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = b; c < 3; ++c) S[(e++) * NB] = Pt[b][c];
    } else {
      lattice_sums<R, 3, 1>(get, s0, j0, Pt);
    }
    S[k * NB] = s0;
#pragma unroll
    for (int b = 0; b < 3; ++b) S[(k + 1 + b) * NB] = j0[b];
    if (ScalarTraits<R>::single && l < M) {
      sabs = fabs(f[0]);
#pragma unroll
      for (int i = 1; i < 27; ++i) sabs += fabs(f[i]);
      S[(k + 4) * NB] = sabs;
    }
    if (PARK) {
#pragma unroll
      for (int i = 0; i < 27; ++i) parked[i * NB] = f[i];
    }
  }
  __syncthreads();
  R* __restrict__ dn = a.dst + (size_t)(unsigned)(l * 27) * N + n;
  auto put = [&](int i, const R& v) {
    if (live) dn[(size_t)(unsigned)i * N] = v;
  };
  if (l < M) {
    // ---- species l: its row of the diffusion system (Eq. 23, 24, 22, 26, 29) ------
    bar_sync(1, TS + T1);
    R w[3], v[3], row[M], X[M];
#pragma unroll
    for (int b = 0; b < 3; ++b) w[b] = S[(F::kW + b) * NB];
    R h = R(0), hYl = R(0), beta, q, itk;
#pragma unroll
    for (int b = 0; b < M; ++b) {
      const R hY = S[(F::kHY + b) * NB], t = hY * p.invDmm[l][b];      // zero on the diagonal
      if (b == l) hYl = hY;
      row[b] = -t;
      h += t;
    }
    itk = p.knc[l] * S[F::kKT * NB];
    q = R(1) / (R(1) + h);
    beta = h * q;
    const R hk = R(0.5) * itk, margin = R(1) + hk;
    const bool tiny = Transport<R, 3, M>::unresolved(s0, S[F::kSS * NB], sabs);
    const R isa = R(1) / s0;
#pragma unroll
    for (int b = 0; b < 3; ++b) v[b] = (tiny ? R(0) : j0[b] * isa - w[b]) - hk * w[b];
    if (ScalarTraits<R>::single) {
      R rs = fabs(margin + h);
#pragma unroll
      for (int b = 0; b < M; ++b) rs += fabs(row[b]);
      S[(F::kCond + l) * NB] = rs;
      S[(F::kCond + M + l) * NB] = margin;
    }
#pragma unroll
    for (int b = 0; b < M; ++b)
      if (b == l) row[b] = margin + h;
    bool fp64 = false;
#pragma unroll
    for (int k = 0; k < M; ++k) {
      R* pv = S + (F::kPv + k * (M + 3)) * NB;
      if (l == k) {
        const R inv = R(1) / row[k];
#pragma unroll
        for (int c = k + 1; c < M; ++c) {
          row[c] *= inv;
          pv[c * NB] = row[c];
        }
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          v[b] *= inv;
          pv[(M + b) * NB] = v[b];
        }
      }
      bar_sync(2, TS);
      if (l != k) {
        const R g = row[k];
#pragma unroll
        for (int c = k + 1; c < M; ++c) row[c] -= g * pv[c * NB];
#pragma unroll
        for (int b = 0; b < 3; ++b) v[b] -= g * pv[(M + b) * NB];
      }
      if (ScalarTraits<R>::single && k == 0) {
        // condition bound (R12): above it the system is solved in double
        R amax = R(0), dmin = R(1e30);
#pragma unroll
        for (int b = 0; b < M; ++b) {
          const R rs = S[(F::kCond + b) * NB], d = S[(F::kCond + M + b) * NB];
          amax = rs > amax ? rs : amax;
          dmin = d < dmin ? d : dmin;
        }
        fp64 = amax > p.kappa_thr * dmin;
      }
    }
    if constexpr (ScalarTraits<R>::single) {
      if (fp64) solve_row_fp64<R, M, EN, NB>(p, S, a.phi[n], l, v);
      if (live && l == 0 && fp64) flag(a.status, 2);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) S[(F::kV + 3 * l + b) * NB] = v[b];
    bar_arrive(5, TS + T1);
    // ---- its difference moments and relaxation (Eq. 21, Eq. 25) --------------------
    const R gd = q * itk, qY = R(2) * q * hYl;         // (1 - beta) Y_l C
    SpeciesTarget<R, 3> t;
    t.th = R(0.5) * p.Ra[l] * S[F::kT * NB];
    t.gE = gd * s0;
    t.cE = R(2) * beta * s0;
    R total = s0;
    if (SRC) {
      const R rd = S[(F::kRd + l) * NB];
      t.cE += rd;                                      // Eq. 89, R^r = fdot^r dt
      total += rd;
    }
    SpeciesAxes<R, 3> ax;
    ax.set(w, v, s0, t.th);
    {
      R* d = D0 + l * NB * F::kStride;
      R m[9];
      ax.template delta<0>(m);
      store16<8>(d + F::kO0, m + 1);
      ax.template delta<1>(m);
      store16<9>(d + F::kO1, m);
      ax.template delta<2>(m);
      store16<9>(d + F::kO2, m);
    }
    bar_sync(4, TS);
#pragma unroll
    for (int b = 0; b < M; ++b) X[b] = (b == l) ? -gd : qY * p.invDmm[l][b];
    const R keep = R(1) - R(2) * beta;
    R c2[9], c1[9], m[9], acc;
    couple<R, M, F::kStride, NB, 9>(D0 + F::kO2, X, c2);
    couple<R, M, F::kStride, NB, 9>(D0 + F::kO1, X, c1);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      c2[e] += t.template entry<2>(ax, w, e % 3, e / 3);
      c1[e] += t.template entry<1>(ax, w, e % 3, e / 3);
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) m[e] = c2[e] - c1[e];
    acc = relax_dirs<R, 3, false>(get, -1, keep, m, nullptr, put);
#pragma unroll
    for (int e = 0; e < 9; ++e) m[e] = c2[e] + c1[e];
    acc += relax_dirs<R, 3, false>(get, 1, keep, m, nullptr, put);
    couple<R, M, F::kStride, NB, 8>(D0 + F::kO0, X, c1);
#pragma unroll
    for (int e = 1; e < 9; ++e)
      m[e] = (c1[e - 1] + t.template entry<0>(ax, w, e % 3, e / 3)) - R(2) * c2[e];
    acc += relax_dirs<R, 3, false>(get, 0, keep, m, nullptr, put);
    put(13, total - acc);
    return;
  }
  R m[3][9], ex[3] = {R(0), R(0), R(0)}, total, keep;
  if (l == L - 1) {
    // ---- last group: state, then mixture (and the energy lattice) -------------------
    Moments<R, 3, M, EN, true> mo;
#pragma unroll
    for (int k = 0; k < M; ++k) mo.sa[k] = S[F::kSp * k * NB];
    mo.sf = S[F::kMo * NB];
#pragma unroll
    for (int b = 0; b < 3; ++b) mo.jf[b] = S[(F::kMo + 1 + b) * NB];
    if (EN) mo.sg = s0;
    State<R, 3, M> s;
    s.template from_moments<EN, true>(p, mo, phi, Tf);
    const R inv_phi = R(1) / s.phi;
    const R kT = s.T * rsqrt_<R>(s.T) * inv_phi, hC = R(0.5) * p.Kc * s.sf * kT;      // as in Transport
#pragma unroll
    for (int b = 0; b < 3; ++b) S[(F::kW + b) * NB] = s.w[b];
    S[F::kT * NB] = s.T;
    S[F::kSS * NB] = s.ss;
    S[F::kKT * NB] = p.knudsen ? kT : R(0);
#pragma unroll
    for (int k = 0; k < M; ++k) S[(F::kHY + k) * NB] = hC * s.Y[k];
    bar_arrive(1, TS + T1);
    if (live && bad_state(s, inv_phi)) flag(a.status, 1);
    Grad<R, 3, M, EN> gr;
    gr.divu = S[F::kU * NB] + S[(F::kU + 1) * NB] + S[(F::kU + 2) * NB];
#pragma unroll
    for (int b = 0; b < 3; ++b) gr.dPi[b] = S[(F::kU + 3 + b) * NB];
    R itk[M], sum_rd = R(0);
#pragma unroll
    for (int k = 0; k < M; ++k) {
      itk[k] = p.knudsen ? p.knc[k] * kT : R(0);
      if (SRC) sum_rd += S[(F::kRd + k) * NB];
    }
    Mixture<R, 3> mix;
    mix.template scalars<M, EN>(p, s, inv_phi, gr.divu);
    bar_sync(5, TS + T1);
    R v[M][3], vbar[3];
#pragma unroll
    for (int k = 0; k < M; ++k)
#pragma unroll
      for (int b = 0; b < 3; ++b) v[k][b] = S[(F::kV + 3 * k + b) * NB];
    mix.template force<M>(s, itk, v, vbar);
    const R cf = (SRC ? mix.omega + sum_rd * s.inv_sf : mix.omega) * s.sf;            // Eq. 42, Eq. 87
    Axis<R> F3[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) mix.momentum_axis(s.w[b], s.inv_sf, b, gr.dPi[b], F3[b]);
    keep = R(1) - mix.omega;
    if constexpr (EN) {
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        S[(F::kF + 2 * b) * NB] = F3[b].m[1];
        S[(F::kF + 2 * b + 1) * NB] = F3[b].m[2];
      }
      S[F::kOm * NB] = mix.omega;
      S[F::kCf * NB] = cf;
      S[F::kTot * NB] = s.sf + sum_rd;                                                // Eq. 78
      bar_arrive(3, 2 * T1);
      // ---- energy (Eq. 43, Eq. 51, Eq. 54, Eq. 88) --------------------------------
      int e = F::kMo + 4;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        mo.q[b] = j0[b];
#pragma unroll
        for (int c = b; c < 3; ++c) mo.Pt[b][c] = mo.Pt[c][b] = S[(e++) * NB];
#pragma unroll
        for (int k = 0; k < M; ++k) gr.dY[k][b] = S[(F::kDY + 3 * k + b) * NB];
      }
      mix.template heat<M, EN>(p, mo, s, v, vbar, gr);
      R cU = mix.omega * s.sf * mix.U, c2 = mix.omega * s.sf;
      total = mo.sg;
      if (SRC) {
        // source distribution with the post-reaction density and internal
        // energy (Eq. 86): phi rho U gains dU, phi rho gains the sum of the sources
        cU += dU;
        c2 += sum_rd;
        total += dU + sum_rd * mix.hw2;
      }
#pragma unroll
      for (int b = 0; b < 3; ++b) ex[b] = mix.Dq[b];
      energy_moments<R, 3>(cU, c2, mix.RT, s.w, m);
    } else {
      total = s.sf + sum_rd;
      product_moments<R, 3>(cf, F3, m);
    }
  } else {
    // ---- momentum (Eq. 42, Eq. 44, Eq. 87) -----------------------------------------
    bar_sync(3, 2 * T1);
    Axis<R> F3[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) F3[b].set(R(1), S[(F::kF + 2 * b) * NB], S[(F::kF + 2 * b + 1) * NB]);
    product_moments<R, 3>(S[F::kCf * NB], F3, m);
    total = S[F::kTot * NB];
    keep = R(1) - S[F::kOm * NB];
  }
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

}  // namespace lbm
