// Layout of the 2D warp march (march2d.cuh) and the choice of its lanes and tile heights for FP32
// fields, by the time a step should take.  Host code only.
#pragma once

namespace mpd {

constexpr int kLead = 4;   // computed columns left of a strip's first output column
constexpr int kWarps = 4;  // warps per block
// output columns of a strip with lanes of nc columns
constexpr int strip_stride(int nc) { return 32 * nc - 2 * kLead; }

// Tile height of the FP32 warp march and the time it should take.  Every warp of a tile height ty
// marches ty + 6 rows; with k blocks on the fullest SM one row of all of them takes it c(k)
// microseconds, more than k times one block's share only while few warps leave the issue slots idle
// (c measured on fields of 256^2 .. 4096^2: one block takes almost as long as two; three of the
// plain march with lanes of 4 fit an SM at once).  The height is the smallest that keeps the fullest
// SM at k blocks, for the k of least time, even (the march's loop takes two rows a turn, and its
// single last row of an odd height rounds the products differently, so that a result would depend
// on the height); a field with more strips than that has warps is not cut into rows.  Against the earlier list of heights (the tallest with 7.5 warps per SM): 4096^2
// 102 -> 90 us (80 rows instead of 64), 2000 x 500 13.9 -> 10.3 us (with lanes of 2).
struct MarchRows {
  int ty;
  float us;
};
inline MarchRows march_rows(int nc, int n0, int n1, bool comp) {
  constexpr float plain4[4] = {0.55f, 0.73f, 1.00f, 1.44f}, plain2[4] = {0.38f, 0.455f, 0.59f, 0.74f};
  constexpr float comp4[4] = {0.93f, 0.97f, 1.37f, 1.83f}, comp2[4] = {0.53f, 0.58f, 0.76f, 0.97f};
  const float* c = nc == 4 ? (comp ? comp4 : plain4) : (comp ? comp2 : plain2);
  const long long strips = (n1 + strip_stride(nc) - 1) / strip_stride(nc);
  constexpr long long kSms = 152;
  MarchRows best{0, 0.0f};
  // few tiles per strip: more blocks per SM give heights in between (1500 x 150000 1326 -> 1092 us,
  // 300 x 250000 454 -> 382)
  const int most = strips > 2 * kSms ? 24 : 6;
  for (long long k = 1; k <= most; ++k) {
    const long long tiles = kSms * k * kWarps / strips;
    long long ty = tiles < 1 ? n0 : (n0 + tiles - 1) / tiles;
    if (ty < 4) ty = 4;
    ty += ty & 1;
    const long long blocks = (strips * ((n0 + ty - 1) / ty) + kWarps - 1) / kWarps;
    const long long full = (blocks + kSms - 1) / kSms;
    const float us = static_cast<float>(ty + 6) * (full <= 4 ? c[full - 1] : c[2] / 3.0f * static_cast<float>(full));
    if (best.ty == 0 || us < best.us) best = {static_cast<int>(ty), us};
  }
  return best;
}

// Whether lanes of 2 columns suit an FP32 field better than lanes of 4: where the narrower strips
// leave fewer padded columns or, on a field too small to fill the GPU, their twice as many warps
// hide more latency (compensated 512^2 12.1 -> 7.4 us, plain 2000 x 500 13.9 -> 10.3).
inline bool narrow_lanes(int n0, int n1, bool comp) {
  return march_rows(2, n0, n1, comp).us < 0.98f * march_rows(4, n0, n1, comp).us;
}

}  // namespace mpd
