// What a 2D step takes on the shared-memory tile kernel (tile2d.cu) and on the staged kernels
// (staged.cu), as estimates in microseconds for the dispatch between the two.  Host code only.
//
// A block of the tile kernel computes its tile with the halo H of the whole step, so that the pass
// farthest from the end costs up to ((32 + 2H) / 32)^2 of its cells; the staged kernels compute every
// cell once but pay a launch per sub-step and the trips through L2.  The coefficients are fitted to
// both sides on 64^2 .. 2000^2 cells, 2 to 8 passes, with and without the limiter and the third-order
// terms; the estimates are within about 15 % and the choice within 10 % of the better side.  Measured
// (us per step, tile / staged): FP32 three passes with the limiter 1024^2 70 / 111, six passes 348 / 247;
// FP64 third-order terms with two passes 1024^2 340 / 413, 64^2 34 / 15; three passes with the limiter
// 512^2 202 / 185, eight passes 1024^2 4843 / 2197.
#pragma once

#include <cstddef>
#include <initializer_list>

namespace mpd {

struct TileCase {
  int n0, n1, fields, n_iters;
  bool fct, tot, nug, dfl, fp64;
};

constexpr int kTileCols = 32;

inline int tile_reach(const TileCase& c) { return 1 + (c.fct ? 1 : 0) + (c.tot ? 1 : 0); }
inline int tile_halo(const TileCase& c) { return 1 + (c.n_iters - 1) * tile_reach(c); }

// dynamic shared memory of a block with tiles of `rows` rows
inline size_t tile_smem(const TileCase& c, int rows) {
  const size_t arrays = 6 + (c.fct ? 2 + (c.n_iters > 2 ? 2 : 0) : 0) + (c.nug ? 1 : 0) + (c.dfl ? 1 : 0);
  const int H = tile_halo(c);
  return (c.fp64 ? 8 : 4) * arrays * static_cast<size_t>(rows + 2 * H) * static_cast<size_t>(kTileCols + 2 * H);
}

// The launch of a step in tiles of `rows` rows.
inline double tile_us(const TileCase& c, int rows) {
  const double fct = c.fct ? 1.0 : 0.0, tot = c.tot ? 1.0 : 0.0;
  double area = 0.0;  // cells that the corrective passes compute, in units of 32 x 32
  for (int k = 2; k <= c.n_iters; ++k) {
    const int M = (c.n_iters - k) * tile_reach(c) + (c.fct ? 1 : 0);
    area += (rows + 2 * M + 1) * (kTileCols + 2 * M + 1) / 1024.0;
  }
  const long long tiles =
      static_cast<long long>(c.fields) * ((c.n0 + rows - 1) / rows) * ((c.n1 + kTileCols - 1) / kTileCols);
  const long long per_sm = (tiles + 151) / 152;  // tiles of the fullest SM
  const size_t room = 228 * 1024 / (tile_smem(c, rows) + 1024);  // blocks whose shared memory fits an SM
  const long long blocks = room < 1 ? 1 : (room > 8 ? 8 : static_cast<long long>(room));
  if (c.fp64) {  // bound by the SM's FP64 pipe, which one block alone does not quite fill
    const double block = 4.5 * rows / 32.0 + area * (21.5 + 19.0 * tot + 8.0 * fct) * (blocks < 2 ? 1.15 : 1.0);
    return block * (per_sm == 1 ? 1.27 : static_cast<double>(per_sm));
  }
  // one block's chain of sub-steps, or the SM's issue rate, which few blocks do not fill
  const double alone = 8.3 + area * (2.4 + 0.4 * tot + 2.3 * fct);
  const double idle = blocks == 1 ? 2.1 : (blocks == 2 ? 1.37 : (blocks == 3 ? 1.12 : 1.0));
  const double rate = static_cast<double>(per_sm) * (1.6 + area * (1.25 + 0.35 * tot + 1.15 * fct) * idle);
  const double chain = per_sm > 1 && per_sm <= blocks ? 1.15 * alone
                                                      : alone * static_cast<double>((per_sm + blocks - 1) / blocks);
  return chain > rate ? chain : rate;
}

// The same step, field by field, on the staged kernels: a launch per sub-step and the cells.
inline double staged_us(const TileCase& c) {
  const double fct = c.fct ? 1.0 : 0.0, tot = c.tot ? 1.0 : 0.0;
  const double launches = 1.0 + fct + (c.n_iters - 1) * (2.0 + 2.0 * fct);
  const double kcells = static_cast<double>(c.n0) * c.n1 / 1000.0, passes = c.n_iters - 1;
  if (c.fp64)
    return c.fields * (3.2 * launches + kcells * (0.022 + 0.007 * fct + passes * (0.223 + 0.152 * tot + 0.0735 * fct)));
  const double small = 2.0 * launches + 2.0;
  const double large = 1.9 * launches + kcells * (0.0095 + passes * (0.024 + 0.0027 * tot + 0.018 * fct));
  return c.fields * (small > large ? small : large);
}

// Rows of the tiles that a step should take (32, or in FP64 16: more halo, more blocks for a small
// field), 0 for the staged kernels (also where no tile's shared memory, `most` bytes, fits).  `always`:
// the tile kernel wherever it fits.
inline int tile_rows(const TileCase& c, size_t most, bool always) {
  int best = 0;
  double us = 0.0;
  for (int rows : {32, 16}) {
    if ((rows == 16 && !c.fp64) || tile_smem(c, rows) > most) continue;
    const double t = tile_us(c, rows);
    if (best == 0 || t < us) {
      best = rows;
      us = t;
    }
  }
  // estimates close to each other: the staged kernels, whose time varies less with the tiling
  if (best != 0 && !always && us > 0.95 * staged_us(c)) best = 0;
  return best;
}

}  // namespace mpd
