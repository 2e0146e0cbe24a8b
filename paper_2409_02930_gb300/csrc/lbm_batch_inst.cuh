// Instantiates the batched-form kernels for one precision; the including file
// defines LBM_REAL and LBM_BATCH_OPS_NAME.
#include "lbm_batch.cuh"

namespace lbm {
namespace {

template <class R, int D, int M, bool EN>
struct BatchLaunch {
  // variant v < 6: two passes over runs of 64, 128 or 256 nodes (v / 2); v >= 6:
  // one pass over tiles of 8 x 4, 16 x 4 or 32 x 4 nodes; v % 2: grid mode
  static constexpr int kRuns[3] = {64, 128, 256}, kTileX[3] = {8, 16, 32};
  static void tile(int v, int* tx, int* ty) {
    *tx = v < 6 ? kRuns[v / 2] : kTileX[(v - 6) / 2];
    *ty = v < 6 ? 0 : 4;
  }
  template <class Kern>
  static int blocks(Kern kern, int threads) {
    int n = 0;
    return (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, 0) == cudaSuccess && n > 0) ? n : 1;
  }
  template <int TB>
  static int runs_occ() {
    const int a = blocks(k_batch<R, D, M, EN, TB, false>, TB), b = blocks(k_batch<R, D, M, EN, TB, true>, TB);
    return a < b ? a : b;
  }
  static int occupancy(int v) {
    switch (v / 2) {
      case 0: return runs_occ<64>();
      case 1: return runs_occ<128>();
      case 2: return runs_occ<256>();
      case 3: return blocks(k_batch_tile<R, M, EN, 8, 4>, 32);
      case 4: return blocks(k_batch_tile<R, M, EN, 16, 4>, 64);
      default: return blocks(k_batch_tile<R, M, EN, 32, 4>, 128);
    }
  }
  template <int TB>
  static void runs(const BatchArgs<R>& b, int grid, int collide, cudaStream_t s) {
    if (collide) k_batch<R, D, M, EN, TB, true><<<grid, TB, 0, s>>>(b);
    else k_batch<R, D, M, EN, TB, false><<<grid, TB, 0, s>>>(b);
  }
  static void pass(const BatchArgs<R>& b, int v, int grid, int collide, cudaStream_t s) {
    if (v >= 6 && !collide) return;                   // one pass: nothing before the node update
    switch (v / 2) {
      case 0: runs<64>(b, grid, collide, s); break;
      case 1: runs<128>(b, grid, collide, s); break;
      case 2: runs<256>(b, grid, collide, s); break;
      case 3: k_batch_tile<R, M, EN, 8, 4><<<grid, 32, 0, s>>>(b); break;
      case 4: k_batch_tile<R, M, EN, 16, 4><<<grid, 64, 0, s>>>(b); break;
      default: k_batch_tile<R, M, EN, 32, 4><<<grid, 128, 0, s>>>(b); break;
    }
  }
  static BatchOps<R> ops() { return BatchOps<R>{tile, occupancy, pass, 12}; }
};

}  // namespace

bool LBM_BATCH_OPS_NAME(int M, int energy, BatchOps<LBM_REAL>* out) {
  if (M == 2 && !energy) { *out = BatchLaunch<LBM_REAL, 2, 2, false>::ops(); return true; }
  if (M == 3 && energy) { *out = BatchLaunch<LBM_REAL, 2, 3, true>::ops(); return true; }
  return false;
}

}  // namespace lbm
