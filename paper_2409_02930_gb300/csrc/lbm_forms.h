// Which kernel form a new single lattice or batch takes, from its configuration
// alone (host code without CUDA).
#pragma once

#include "../../include/lbm.h"

namespace lbm {

// Forms whose grid counts rows in its y dimension can launch up to this many
// units of `rows` lattice rows; taller lattices take a form with a flat grid.
constexpr int kGridRows = 65535;
inline bool rows_fit(long long ny, int rows) { return (ny + rows - 1) / rows <= kGridRows; }

// Lattices narrower than a tile leave most of its threads without a node, and
// every block still pays for the whole tile, so beyond a few blocks per SM they
// take the two-pass form, whose threads all have a node.  us per step (tiles /
// two-pass), FP32 in tiles of 32 x 4: 1x200000 579 / 32, 8x25003 77 / 33,
// 18x11114 36.8 / 34.2, 20x10003 33.2 / 34.2; 12x2500 (625 tiles) 10.9 / 7.3
// (two isothermal species 11.1 / 7.4, and 7.1 / 7.8 at 19x1900, 475 tiles).  FP64
// in tiles of 16 x 8: 1x200000 6192 / 525, 10x20003 646 / 527, 12x16669 533 / 527,
// 14x14288 459 / 526, 16x12503 420 / 525, 17x11767 757 / 528, 24x8336 534 / 526,
// 28x7145 459 / 527 (isothermal 18x8000 418 / 267): about 39 us for every 152 tiles
// against 45 us for every 152 x 128 nodes in two passes (8x1250 78 / 47, 24x800 78 /
// 48, 12x2000 78 / 90, 24x1000 78 / 90).  Split by lattice, tiles of 8 x 4: FP32
// 4x2400 (600 tiles) 6.6 / 6.6, 1x5000 (1,250) 10.3 / 5.7, 1x9000 16.7 / 6.3 (two
// isothermal species 3x3000, 750 tiles, 5.3 / 6.9, 1x9000 11.1 / 7.4); FP64 6x1600
// (400) 43.9 / 44.8, 5x1900 (475) 50.7 / 45.1, 1x9000 197 / 45.
constexpr int kSMs = 152;
constexpr long long kSplit2dNodes = 2 * kSMs * 32, kMarchNodes = 3 << 20;
inline bool narrow_lattice(long long nx, long long ny, bool single) {
  auto rows = [&](int t) { return (ny + t - 1) / t; };
  if (nx * ny <= kSplit2dNodes) return nx < 8 && rows(4) > (single ? 8 : 3) * kSMs;
  if (single) return nx < 20 && rows(4) > 4 * kSMs;
  const long long tiles = (nx + 15) / 16 * rows(8);
  return nx < 32 && 5 * ((tiles + kSMs - 1) / kSMs) > 6 * ((nx * ny + kSMs * 128 - 1) / (kSMs * 128));
}

// Kernel form of a new single lattice.  3-D: the split step.  2-D, measured in
// us per step (tiles / row march): FP32 256x256 with reservoirs 14.4 / 73,
//   512x512 27.5 / 27.4, 640x512 36.1 / 52.5, 512x768 43.0 / 54.5, 1024x512
//   55.3 / 56.5, 1024x1024 104.6 / 108.4, 1536x1536 224 / 226, 2048x2048 389 /
//   380, 701x523 with walls 45 / 58; FP64 512x512 549 / 689.
// The row march (bulk tensor copies, rows of whole 16-byte units, no
// reservoir) is taken from 3 x 2^20 FP32 nodes, where its prefetched rows read
// HBM without stalls, and from 2^18 nodes where its blocks (30 columns by 8
// rows, eight resident per SM) make one wave: there it is ahead or level
// (tiles / march: 480x560 28.6 / 27.6, 600x440 27.5 / 27.6, 1000x270 29.2 / 27.5,
// 300x900 30.1 / 29.0, 2100x128 28.0 / 27.4, 540x512 29.5 / 27.8, 256x1024 27.5 /
// 27.7; from a flushed L2 512x512 36.8 / 34.8), below it leaves SMs idle (500x500 26.5 / 27.7, 448x512 22.9 / 27.5), and
// between the two lines its long blocks leave part of a last wave empty.
// Everything else runs on tiles.  Up to two 32-node tiles per SM the lattice is
// bound by one tile's latency and the tiles are split by lattice (split / best
// other tile: FP64 256x4 20.0 / 40.1, capillary 17.5 / 34.1, 96x96 27.5 / 40.4,
// 128x128 52.2 / 44.0; FP32 64x40 4.9 / 5.5, 96x96 5.1 / 6.5, 128x128 7.4 / 6.0;
// six species 128x64 FP64 67.7 / 99.0, FP32 7.7 / 8.4, 128x128 123 / 98, 13.4 /
// 8.5); above that 32 x 4 in FP32 (whole lines) and
// 16 x 8 in FP64 (bound by operations, so the smaller halo counts; six species
// 512x512 1047 against 1064 in 32 x 4 and 1162 in two passes).  Lattices
// of one or two rows would leave most of a tile idle and take the two-pass
// form once they fill the GPU, and so do lattices with more rows than the tiles'
// grids can count.
inline int default_variant(const lbm_config* c) {
  if (c->nz > 1) return 5;
  const long long N = (long long)c->nx * c->ny;
  const bool single = c->precision == LBM_FP32;
  const bool reservoir = c->bc_lo == LBM_BC_INLET || c->bc_hi == LBM_BC_INLET;
  const bool one_wave = N >= (1 << 18) && ((c->nx + 29LL) / 30) * ((c->ny + 7LL) / 8) <= 8 * kSMs;
  if (narrow_lattice(c->nx, c->ny, single)) return -1;
  if (single && !reservoir && (one_wave || N >= kMarchNodes) && c->nx % 4 == 0 && rows_fit(c->ny, 8)) return 8;
  if (!rows_fit(c->ny, 4) || (c->ny < 3 && N >= 8192)) return -1;
  return N <= kSplit2dNodes ? 10 : (single ? 12 : 11);
}

// Form indices that launch the same kernels as another one, so that a search
// over the forms times each once: of the D3Q27 indices 3, 4 and -1 are the
// default form 5, and in FP64 2 is 1.
inline bool alias_form(int D, bool single, int v) {
  return D == 3 && (v == -1 || v == 3 || v == 4 || (v == 2 && !single));
}

// What a search over the forms settles on: the form in effect unless another takes
// less than 98 % of its time.  Closer ones are told apart by the noise of a few
// steps, and steps that follow one another find the state in the caches: 512x512
// FP32 27.4 us (form 8) and 27.5 (12) then, 34.8 and 36.8 from a flushed L2.
inline int settled_form(int held, float held_ms, int best, float best_ms) {
  return held_ms > 0.f && best_ms > 0.98f * held_ms ? held : best;
}

// Kernel form of a new batch: tiles of 32 x 4 nodes (10), or two passes over runs
// of 64 nodes (0) where the cases are so narrow or of so few rows that too many
// of the tiles' threads have no node, and the tiles are more than the SMs hold
// at once.  us per step (tiles / runs), cases x their sizes, energy lattice with
// three species unless said: FP32 8 x 3x5000 119 / 19, 8 x 12x2000 50 / 27, 8 x
// 22x600 18.8 / 15.2 but two isothermal species 13.7 / 15.8, 8 x 28x600 19.1 / 20.3,
// 64 tubes of one row 15.9 / 9.8, of two 16.8 / 15.9, of three 18.7 / 21.6; FP64
// 8 x 3x5000 2592 / 315, 8 x 22x600 317 / 238, 8 x 28x600 318 / 317 (two species 274 /
// 244), 8 x 30x600 319 / 317 (273 / 283), tubes of three rows 326 / 306, of four 403 /
// 413.  By tiles: FP32 two species 16 x 12x100 (400 tiles) 7.0 / 7.6, 24 x 12x100
// (600) 7.6 / 8.0; FP64 8 x 5x200 (400) 161 / 42, 8 tubes of nine rows (130) 38 / 37.
inline int default_batch_variant(int n_cases, const lbm_config* cfgs) {
  long long nodes = 0, tiles = 0;
  for (int c = 0; c < n_cases; ++c) {
    nodes += (long long)cfgs[c].nx * cfgs[c].ny;
    tiles += ((cfgs[c].nx + 31LL) / 32) * ((cfgs[c].ny + 3LL) / 4);
  }
  const bool single = cfgs[0].precision == LBM_FP32;
  const bool idle = 10 * nodes < (single ? 6 : 9) * 128 * tiles;
  return idle && tiles > (single ? 4 : 1) * kSMs ? 0 : 10;
}

}  // namespace lbm
