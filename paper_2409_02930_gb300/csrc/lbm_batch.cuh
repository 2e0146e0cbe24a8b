// Batched form: many independent 2-D lattices (capillaries or slabs of
// uneven size and pressure, each with its own lattice scaling) advanced by
// persistent kernels over one work list of node tiles.
//
// Every case keeps the single-lattice layout ([L][Q][N_c] populations,
// [2D+M][N_c] macro fields) at its own offset inside shared buffers, so the
// per-node code of the two-pass step (lbm_kernels.cuh) runs unchanged with
// the case's own parameters (read through the L1 cache from the case table).
// A block takes a contiguous range of the tile list, which keeps most of its
// tiles inside one case.
#pragma once

#include "lbm_tile2d.cuh"

namespace lbm {

template <class R>
struct CaseDev {
  Params<R> p;
  InletTables<R> it;
  long long pop_off;    // element offset of the case's populations
  long long node_off;   // offset of its per-node fields (porosity, temperature)
  long long mac_off;    // offset of its macro-field block
};

template <class R>
struct BatchArgs {
  const CaseDev<R>* cases;
  const int2* tiles;    // (case, first node of the tile) or (case, index of the 2-D tile)
  int ntiles;
  const R* src;
  R* dst;
  const R* phi;
  const R* Tfix;
  R* mac;
  int* status;
};

// One pass of the two-pass step over every tile: COLLIDE = false computes the
// macro fields, COLLIDE = true the node update.  Tiles are TB nodes long.
template <class R, int D, int M, bool EN, int TB, bool COLLIDE>
__global__ void __launch_bounds__(TB) k_batch(BatchArgs<R> b) {
  const int t0 = (int)((long long)blockIdx.x * b.ntiles / gridDim.x);
  const int t1 = (int)((long long)(blockIdx.x + 1) * b.ntiles / gridDim.x);
  for (int t = t0; t < t1; ++t) {
    const int2 tl = b.tiles[t];
    const CaseDev<R>& cs = b.cases[tl.x];
    const int n = tl.y + (int)threadIdx.x;
    if (n >= cs.p.N) continue;
    StepArgs<R> a{b.src + cs.pop_off, b.dst + cs.pop_off, b.phi + cs.node_off, b.Tfix + cs.node_off,
                  b.mac + cs.mac_off, b.status};
    if (COLLIDE) collide_node<R, D, M, EN>(cs.p, cs.it, a, n);
    else macro_node<R, D, M, EN>(cs.p, cs.it, a, n);
  }
}

// The single-launch form: TX x TY tiles of every case (lbm_tile2d.cuh), the
// case's parameters copied to shared memory once per tile (the node code reads
// them all over, and a block's tiles mostly stay in one case).  64 capillaries
// (0.30 M nodes, FP32): 21.2 us per step, against 24 us in two passes over
// runs and 31 us with the populations staged in shared memory.
template <class R, int M, bool EN, int TX, int TY>
__global__ void __launch_bounds__(TX * TY) k_batch_tile(BatchArgs<R> b) {
  using T = TileShape<R, M, EN, TX, TY>;
  __shared__ R mac[T::NF * T::PN];
  __shared__ CaseDev<R> cs;
  const int t0 = (int)((long long)blockIdx.x * b.ntiles / gridDim.x);
  const int t1 = (int)((long long)(blockIdx.x + 1) * b.ntiles / gridDim.x);
  int have = -1;
  for (int t = t0; t < t1; ++t) {
    const int2 tl = b.tiles[t];
    __syncthreads();                                  // the last tile's readers are done
    if (tl.x != have) {
      const int* s = reinterpret_cast<const int*>(b.cases + tl.x);
      int* d = reinterpret_cast<int*>(&cs);
      for (int k = threadIdx.x; k < (int)(sizeof(cs) / sizeof(int)); k += TX * TY) d[k] = s[k];
      have = tl.x;
      __syncthreads();
    }
    StepArgs<R> a{b.src + cs.pop_off, b.dst + cs.pop_off, b.phi + cs.node_off, b.Tfix + cs.node_off,
                  b.mac + cs.mac_off, b.status};
    const int tx = (cs.p.nx + TX - 1) / TX;
    tile2d_step<R, M, EN, TX, TY>(cs.p, cs.it, a, (tl.y % tx) * TX, (tl.y / tx) * TY, mac);
  }
}

// variants below 6 take two passes over runs of nodes, the others one over tiles
inline bool batch_two_pass(int v) { return v < 6; }

// Launch table of the batched form for one (precision, M, energy).
template <class R>
struct BatchOps {
  // tile of variant v: TX columns by TY rows (TY = 0: a run of TX nodes)
  void (*tile)(int v, int* tx, int* ty);
  // resident blocks per SM of the kernels of variant v (occupancy query)
  int (*occupancy)(int v);
  // one pass of a time step (collide = 0: macro fields, 1: node update) with
  // variant v on grid blocks
  void (*pass)(const BatchArgs<R>&, int v, int grid, int collide, cudaStream_t);
  int n_variants;
};

bool get_batch_ops_f32(int M, int energy, BatchOps<float>* out);
bool get_batch_ops_f64(int M, int energy, BatchOps<double>* out);

}  // namespace lbm
