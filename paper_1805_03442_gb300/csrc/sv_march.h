// sv_march.h -- how many segments the marching axis of a 2D / 3D step is cut
// into (host only).
//
// A block marches over one segment of one transverse tile and pays up to two
// extra iterations of warm-up, so few long segments do the least work; but a grid
// of few tiles needs many segments to reach every SM, and a grid of many
// needs a count whose last wave of blocks is not nearly empty.  The rule
// minimises
//   sum over waves of  t[blocks per SM in the wave] x iterations per block,
// with t the measured relative time of an iteration at that residency.  On a
// GB300 the sum tracks the measured steps within 5 % (nseg swept from 1 to
// 152 on 17 grids); against the fixed 128- or 256-plane segments used before
// (us per step):
//   FP64 500 x 500 with walls 4851 -> 334 (8 blocks on 152 SMs before)
//   FP64 1000 x 1000          5202 -> 1069
//   FP32 1000 x 700             76 -> 25
//   FP32 2048 x 2048           111 -> 97,  4096 x 4096 332, 8192 x 8192 1235 -> 1227
//   FP32 256^3 958 -> 797, 201 x 150 x 170 431 -> 311, 64 x 48 x 200 262 -> 40
//   FP32 512^3 5494 (4 segments either way)
#pragma once

#include <stdint.h>

namespace sv {

// How a 2D / 3D step kernel is cut into blocks: the written columns of a
// transverse tile, the blocks an SM holds, and the relative time of one
// iteration of its march when 1 .. occ blocks share an SM.
struct MarchShape {
  int cols_x, cols_y;     // written columns of a tile (cols_y 0: 2D)
  int step;               // planes an iteration takes (the row pairs: 2)
  double warm;            // a segment's extra iterations, in whole ones
  int occ;                // blocks per SM
  double t[3];            // t[k - 1]: iteration time with k blocks on the SM
  int cap;                // default cap on a segment's planes
};

// Segments for a grid n[] of `dim` axes on `sms` SMs, no segment longer than
// `cap` planes.
inline int march_segments(const MarchShape& g, int dim, const int64_t* n, int64_t cap, int sms) {
  const int64_t M = n[dim - 1];
  int64_t tiles = (n[0] + g.cols_x - 1) / g.cols_x;
  if (dim == 3) tiles *= (n[1] + g.cols_y - 1) / g.cols_y;
  if (sms < 1) sms = 1;
  int64_t lo = (M + cap - 1) / cap;
  if (lo < 1) lo = 1;
  // beyond several waves more segments only add warm-up
  int64_t hi = lo + 16 + 8 * (int64_t)sms * g.occ / tiles;
  if (hi > M) hi = M;
  int64_t best = lo < M ? lo : M;
  double best_cost = 1e300;
  for (int64_t s = best; s <= hi; ++s) {
    const int64_t planes = (M + s - 1) / s;
    const double iters = (double)((planes + g.step - 1) / g.step) + g.warm;
    const int64_t blocks = tiles * s, slots = (int64_t)sms * g.occ;
    const int64_t full = blocks / slots, rem = blocks % slots;
    double cost = (double)full * g.t[g.occ - 1] * iters;
    if (rem) cost += g.t[(rem + sms - 1) / sms - 1] * iters;
    if (cost < best_cost * (1.0 - 1e-9)) {
      best_cost = cost;
      best = s;
    }
  }
  return (int)best;
}

}  // namespace sv
