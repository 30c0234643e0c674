// Tiles of the FP32 3D z-marches (march3.cuh; staged.cu's scalar ones) and the choice between them by
// the time a plane step should take.  Host code only.
#pragma once

namespace mpd {

constexpr int kMarchRows = 8;  // tile rows

// Blocks on the fullest SM of a march with lanes of nc cells and chunks of zc planes
inline long long march3_blocks(const int (&n)[3], int nc, int zc) {
  const long long b = static_cast<long long>((n[2] + 32 * nc - 1) / (32 * nc)) * ((n[1] + kMarchRows - 1) / kMarchRows) *
                      ((n[0] + zc - 1) / zc);
  return (b + 151) / 152;
}

// z-planes per block, 4 to 16: the chunk of least time by the load of the fullest SM.  A block takes
// about zc + 3 plane steps (its halo planes are staged, pass 1 and the factors recomputed on two of
// them); two blocks share an SM and take 1.5 times as long as one there.  Large fields get 16
// (measured at 256^3: 8 .. 24 within 2 %); 128^3, one block per SM with 16, gets 7 and two: 206 -> 144
// us per step of three passes with third-order terms.  steps: the plane steps of the fullest SM, in units of
// those of one block alone.
struct ZChunk {
  int zc;
  float steps;
};
inline ZChunk z_chunk(const int (&n)[3], int nc) {
  ZChunk best{16, 0.0f};
  float least = 0.0f;
  for (int zc = 16; zc >= 4; --zc) {
    const long long k = march3_blocks(n, nc, zc);
    const float load = k == 1 ? 1.0f : 0.75f * static_cast<float>(k);
    const float t = static_cast<float>(zc + 3) * load;
    if (zc == 16 || t < 0.98f * least) {
      least = t;
      best = {zc, static_cast<float>((zc < n[0] ? zc : n[0]) + 3) * load};
    }
  }
  return best;
}

// The forms of the marches: staged.cu's scalar ones (32 columns, 16 planes per block, many blocks per
// SM), lanes of 4 cells with rows in 16-byte chunks, and lanes of 4 or of 2 cells staged cell by cell.
enum class March3 { kScalar, kChunks, kCells4, kCells2 };

// chunks: whether the rows can move in 16-byte chunks.  Large fields take the widest lanes that pad
// their rows little; a field of few blocks is bound by one block's plane step, shortest in the
// scalar form, and one of few planes does not fill that form's 16.  Microseconds per step of two
// passes with the limiter (three kernels), fitted to 1 .. 40 planes of 4 .. 300 rows and 48 .. 512
// columns; the choice is within 8 % of the best form there.  Measured, widest lanes -> chosen:
// 4 x 100 x 100 41 -> 24 us, 40 x 32 x 100 42 -> 28, 4 x 32 x 200 33 -> 24.  widest: those lanes always.
inline March3 march3_form(const int (&n)[3], bool chunks, bool widest) {
  const int w4 = (n[2] + 127) / 128 * 128, w2 = (n[2] + 63) / 64 * 64;
  const float two = 5.0f + 3.15f * z_chunk(n, 2).steps;
  const float four = chunks ? 0.4f + 4.55f * z_chunk(n, 4).steps : 4.0f + 5.3f * z_chunk(n, 4).steps;
  const long long k = march3_blocks(n, 1, 16);
  const float scalar = 3.6f + 2.83f * static_cast<float>((n[0] < 16 ? n[0] : 16) + 3) *
                                  (k == 1 ? 1.0f : (k == 2 ? 1.38f : 0.5f * static_cast<float>(k)));
  // lanes of 2 where their tiles cover the row with at most 3/4 of the columns that lanes of 4 compute
  March3 form = chunks ? March3::kChunks : (4 * w2 <= 3 * w4 ? March3::kCells2 : March3::kCells4);
  if (widest) return form;
  float us = 0.95f * (form == March3::kCells2 ? two : four);  // another form has to be clearly faster
  if (two < us) { form = March3::kCells2; us = two; }
  if (scalar < us) form = March3::kScalar;
  return form;
}

}  // namespace mpd
