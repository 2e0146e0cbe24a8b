// Instantiates the step kernels for one (precision, dimension); the including
// file defines LBM_REAL, LBM_DIM and LBM_OPS_NAME.
#include "lbm_forms.h"
#include "lbm_fused.cuh"
#include "lbm_march2d.cuh"
#include "lbm_ops.h"
#include "lbm_split2d.cuh"
#include "lbm_staged.cuh"

namespace lbm {
namespace {

constexpr size_t kMaxSmem = 227 * 1024;

template <class Kern>
int configure(Kern kern, size_t smem, bool& done) {
  if (smem > kMaxSmem) return -1;
  if (!done) {
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
      return -1;
    done = true;
  }
  return 0;
}

template <class R, int D, int M, bool EN>
struct Launch {
  // small lattices take small blocks, so that they spread over the SMs
  static int block(int N) { return N < 152 * 512 ? 64 : 256; }
  static int grid(int N) { return (N + block(N) - 1) / block(N); }
  // 3-D: the step split by lattice, NB = 32 nodes and one warp per lattice in a
  // block; small FP64 lattices take 8 or 16 nodes and several species per warp
  static constexpr int L = M + 1 + (EN ? 1 : 0);
  template <bool AUX, int NB>
  static int macro3(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, R* aux, cudaStream_t s) {
    if constexpr (D == 3) {
      constexpr size_t smem = split_smem_bytes<R, M, EN>(NB, false, false);
      return launch_after(k_macro3<R, M, EN, NB, AUX>, (p.N + NB - 1) / NB, SplitThreads<NB, M, EN>::kAll, smem, s, p,
                          it, a, aux);
    }
    return -1;
  }
  template <bool SRC, int NB, int MINB, bool PARK>
  static int collide3(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, const double* src,
                      cudaStream_t s) {
    if constexpr (D == 3) {
      constexpr size_t smem = split_smem_bytes<R, M, EN>(NB, true, PARK);
      auto kern = k_collide3<R, M, EN, NB, SRC, MINB, PARK>;
      static bool done = false;
      if (configure(kern, smem, done)) return -1;
      return launch_after(kern, (p.N + NB - 1) / NB, SplitThreads<NB, M, EN>::kAll, smem, s, p, it, a, src);
    }
    return -1;
  }
  static constexpr int kMinB = 2;
  static constexpr bool kPark = sizeof(R) == 4;
  template <bool AUX>
  static int macro_any(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, R* aux, cudaStream_t s) {
    if constexpr (sizeof(R) == 8) {
      if (p.N <= split3d_nodes8) return macro3<AUX, 8>(p, it, a, aux, s);
      if (p.N <= split3d_nodes16) return macro3<AUX, 16>(p, it, a, aux, s);
    }
    return macro3<AUX, 32>(p, it, a, aux, s);
  }
  template <bool SRC>
  static int collide_any(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, const double* src,
                         cudaStream_t s) {
    if constexpr (sizeof(R) == 8) {
      if (p.N <= split3d_nodes8) return collide3<SRC, 8, 1, false>(p, it, a, src, s);
      if (p.N <= split3d_nodes16) return collide3<SRC, 16, 1, false>(p, it, a, src, s);
    }
    return collide3<SRC, 32, kMinB, kPark>(p, it, a, src, s);
  }
  static void macro(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, cudaStream_t s) {
    if constexpr (D == 3) macro_any<false>(p, it, a, nullptr, s);
    else launch_after(k_macro<R, D, M, EN>, grid(p.N), block(p.N), 0, s, p, it, a);
  }
  static void collide(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, cudaStream_t s) {
    if constexpr (D == 3) collide_any<false>(p, it, a, nullptr, s);
    else launch_after(k_collide<R, D, M, EN>, grid(p.N), block(p.N), 0, s, p, it, a);
  }
  // fused step, shared-memory ring of macro fields, TX columns marching SEG rows
  template <int TX, int SEG>
  static int fused_tile(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, cudaStream_t s) {
    static_assert(D == 2, "fused tiles are a 2-D form");
    if (!rows_fit(p.ny, SEG)) return -1;
    constexpr size_t smem = fused_smem_bytes<R, M, EN, TX>();
    auto kern = k_fused<R, M, EN, TX, SEG>;
    static bool done = false;
    if (configure(kern, smem, done)) return -1;
    kern<<<dim3((p.nx + TX - 1) / TX, (p.ny + SEG - 1) / SEG), TX, smem, s>>>(p, it, a);
    return 0;
  }
  // tiles with the populations in registers
  template <int TX, int TY, int MINB>
  static int tile2d(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, cudaStream_t s) {
    if (!rows_fit(p.ny, TY)) return -1;
    if constexpr (D == 2)
      return launch_after(k_tile2d<R, M, EN, TX, TY, MINB>, dim3((p.nx + TX - 1) / TX, (p.ny + TY - 1) / TY), TX * TY,
                          0, s, p, it, a);
    return -1;
  }
  // tiles split by lattice, one warp each
  static int split2d(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, cudaStream_t s) {
    if (!rows_fit(p.ny, 4)) return -1;
    if constexpr (D == 2)
      return launch_after(k_split2d<R, M, EN>, dim3((p.nx + 7) / 8, (p.ny + 3) / 4), 32 * (L + 1), 0, s, p, it, a);
    return -1;
  }
  // pipelined 2-D step (cp.async staging), TX columns marching SEG rows
  template <int TX, int SEG, int MINB, int PD>
  static int march2d(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, cudaStream_t s) {
    if constexpr (D != 2) {
      return -1;
    } else {
      constexpr size_t smem = march2d_smem_bytes<R, M, EN, TX, PD>();
      if constexpr (smem > kMaxSmem) {
        return -1;
      } else {
        if (!rows_fit(p.ny, SEG)) return -1;
        // the reservoir-column path is compiled in only when a face is a reservoir
        const bool inlet = p.bc_lo == BC_INLET || p.bc_hi == BC_INLET;
        auto kern = inlet ? k_march2d<R, M, EN, TX, SEG, MINB, PD, true> : k_march2d<R, M, EN, TX, SEG, MINB, PD, false>;
        static bool done[2] = {false, false};
        if (configure(kern, smem, done[inlet ? 1 : 0])) return -1;
        dim3 g((p.nx + TX - 3) / (TX - 2), (p.ny + SEG - 1) / SEG, 1);
        return launch_after(kern, g, TX, smem, s, p, it, a, TmaMaps{});
      }
    }
  }
  // the same march with each row staged by bulk tensor copies (TMA); lattices
  // whose rows are not a multiple of 16 bytes take the cp.async form
  template <int TX, int SEG, int MINB, int PD>
  static int march2d_tma(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, cudaStream_t s) {
    if constexpr (D != 2) {
      return -1;
    } else {
      using LB = RowBoxLayout<R, M, EN, TX, PD>;
      constexpr size_t smem = LB::bytes();
      if constexpr (smem > kMaxSmem) {
        return -1;
      } else {
        if (!rows_fit(p.ny, SEG)) return -1;
        TmaMaps tm;
        if (!encode_row_maps<R>(tm, a.src, a.phi, EN ? nullptr : a.Tfix, p.nx, p.ny, Lat<D>::Q, LB::NL, LB::W))
          return march2d<TX, SEG, MINB, PD>(p, it, a, s);
        const bool inlet = p.bc_lo == BC_INLET || p.bc_hi == BC_INLET;
        auto kern = inlet ? k_march2d<R, M, EN, TX, SEG, MINB, PD, true, true>
                          : k_march2d<R, M, EN, TX, SEG, MINB, PD, false, true>;
        static bool done[2] = {false, false};
        if (configure(kern, smem, done[inlet ? 1 : 0])) return -1;
        dim3 g((p.nx + TX - 3) / (TX - 2), (p.ny + SEG - 1) / SEG, 1);
        return launch_after(kern, g, TX, smem, s, p, it, a, tm);
      }
    }
  }
  // two-pass form whose node update stages each node's pulled populations in shared memory
  template <int TB>
  static int staged(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, cudaStream_t s) {
    static_assert(D == 2, "populations are staged in 2-D only");
    constexpr size_t smem = sizeof(R) * (size_t)n_pops2<M, EN>() * TB;
    if constexpr (smem > kMaxSmem) {
      return -1;
    } else {
      auto kern = k_collide_staged<R, M, EN, TB>;
      auto kmac = k_macro_staged<R, M, EN, TB>;
      static bool done = false, done_mac = false;
      if (configure(kern, smem, done) || configure(kmac, smem, done_mac)) return -1;
      kmac<<<(p.N + TB - 1) / TB, TB, smem, s>>>(p, it, a);
      kern<<<(p.N + TB - 1) / TB, TB, smem, s>>>(p, it, a);
      return 0;
    }
  }
  static int fused(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, int v, cudaStream_t s) {
    if constexpr (D == 2) {
      switch (v) {
        case 0: return march2d<64, 8, 1, 1>(p, it, a, s);
        case 1: return march2d<64, 8, 1, 2>(p, it, a, s);
        case 2: return march2d<32, 8, 1, 1>(p, it, a, s);
        case 3: return march2d<128, 4, 1, 1>(p, it, a, s);
        case 4: return march2d<64, 16, 1, 1>(p, it, a, s);
        case 5: return fused_tile<32, 8>(p, it, a, s);
        case 6: return staged<64>(p, it, a, s);
        case 7: return staged<128>(p, it, a, s);
        case 8: return march2d_tma<32, 8, 1, 1>(p, it, a, s);
        case 9: return march2d_tma<64, 8, 1, 1>(p, it, a, s);
        case 10: return split2d(p, it, a, s);
        case 11: return tile2d<16, 8, sizeof(R) == 4 ? 3 : 1>(p, it, a, s);
        case 12: return tile2d<32, 4, sizeof(R) == 4 ? 3 : 1>(p, it, a, s);
        default: return -1;
      }
    } else {
      if (v < 3 ? macro3<false, 32>(p, it, a, nullptr, s) : macro_any<false>(p, it, a, nullptr, s)) return -1;
      switch (v) {
        case 0: return collide3<false, 32, 1, false>(p, it, a, nullptr, s);
        case 1: return collide3<false, 32, 2, false>(p, it, a, nullptr, s);
        case 2: return collide3<false, 32, sizeof(R) == 4 ? 3 : 2, false>(p, it, a, nullptr, s);
        case 3:
        case 4:
        case 5: return collide_any<false>(p, it, a, nullptr, s);
        default: return -1;
      }
    }
  }
  static constexpr int n_variants = (D == 2) ? 13 : 6;
  static void init(const Params<R>& p, const double* X, const double* T, const double* P, const double* U,
                   double cvel, double RU, R* dst, const R* phi, cudaStream_t s) {
    k_init<R, D, M, EN><<<grid(p.N), block(p.N), 0, s>>>(p, X, T, P, U, cvel, RU, dst, phi);
  }
  static void moments(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, int which, double cvel,
                      double* out, cudaStream_t s) {
    k_moments<R, D, M, EN><<<grid(p.N), block(p.N), 0, s>>>(p, it, a, which, cvel, out);
  }
  static constexpr bool has_react = (D == 3 && M == 6 && EN);
  static void react_macro(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, const ReactArgs& ra,
                          cudaStream_t s) {
    if constexpr (has_react) {
      R* aux = a.mac + (size_t)(2 * D + M) * p.N;
      macro_any<true>(p, it, a, aux, s);
      if (p.N <= source_warp_nodes<R>) {
        launch_after(k_source_warp<R, M>, p.N, 32, 0, s, p.N, aux, a.phi, a.status, ra);
      } else if (p.N <= source_wide_nodes) {
        k_source<R, M, 1><<<(p.N + 127) / 128, 128, 0, s>>>(p.N, aux, a.phi, a.status, ra);
      } else {
        k_source<R, M, sizeof(R) == 4 ? 10 : 8><<<(p.N + 127) / 128, 128, 0, s>>>(p.N, aux, a.phi, a.status, ra);
      }
    }
  }
  static void react_collide(const Params<R>& p, const InletTables<R>& it, const StepArgs<R>& a, const ReactArgs& ra,
                            cudaStream_t s) {
    if constexpr (has_react) collide_any<true>(p, it, a, ra.src, s);
  }
  static Ops<R> ops() {
    return Ops<R>{macro, collide, fused, n_variants, init, moments, has_react ? react_macro : nullptr,
                  has_react ? react_collide : nullptr};
  }
};

}  // namespace

bool LBM_OPS_NAME(int M, int energy, Ops<LBM_REAL>* out) {
  switch (M * 2 + (energy ? 1 : 0)) {
    case 4: *out = Launch<LBM_REAL, LBM_DIM, 2, false>::ops(); return true;
    case 5: *out = Launch<LBM_REAL, LBM_DIM, 2, true>::ops(); return true;
    case 6: *out = Launch<LBM_REAL, LBM_DIM, 3, false>::ops(); return true;
    case 7: *out = Launch<LBM_REAL, LBM_DIM, 3, true>::ops(); return true;
    case 12: *out = Launch<LBM_REAL, LBM_DIM, 6, false>::ops(); return true;
    case 13: *out = Launch<LBM_REAL, LBM_DIM, 6, true>::ops(); return true;
    default: return false;
  }
}

}  // namespace lbm
