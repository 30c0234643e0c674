// The vectorised FP32 3D z-marches (march3.cuh) for fields whose rows cannot be moved in 16-byte
// chunks (x extents that are no multiple of 4, unaligned arrays) and for fields of fewer than 128
// columns: the planes are staged cell by cell (4-byte cp.async, each cell wrapped by itself), the
// arithmetic on the staged rows is the same.  Lanes of 4 or of 2 cells (tiles of 128 or 64
// columns; march3_form).
//
// Against the scalar z-marches of staged.cu, whose threads own one cell each: 101 x 97 x 103 with
// three passes, third-order terms, limiter and G 233 -> 142 us per step, 64^3 133 -> 49,
// 256 x 256 x 255 1743 -> 1369 (256^3 with 16-byte chunks 1088).
#include "march3.cuh"

namespace mpd {

void antidiff3_cells(const Grid& g, bool two, const float* psi, const float* const* v, float vscale, const float* G,
                     bool iga, bool tot, bool abs_psi, float* const* out, bool chained, cudaStream_t st) {
  if (two) antidiff3_nc<2, false>(g, psi, v, vscale, G, iga, tot, abs_psi, out, chained, st);
  else antidiff3_nc<4, false>(g, psi, v, vscale, G, iga, tot, abs_psi, out, chained, st);
}

void p1b3_cells(const Grid& g, bool two, const float* psi, const float* const* v, float vscale, const float* G, bool kahan,
                float* p1, float* mx, float* mn, bool chained, cudaStream_t st) {
  if (two) p1b3_nc<2, false>(g, psi, v, vscale, G, kahan, p1, mx, mn, chained, st);
  else p1b3_nc<4, false>(g, psi, v, vscale, G, kahan, p1, mx, mn, chained, st);
}

void corr3_cells(const Grid& g, bool two, const float* psi, const float* const* vu, const float* G, bool iga,
                 const float* mx, const float* mn, float* const* lim, float* out, bool chained, cudaStream_t st) {
  if (two) corr3_nc<2, false>(g, psi, vu, G, iga, mx, mn, lim, out, chained, st);
  else corr3_nc<4, false>(g, psi, vu, G, iga, mx, mn, lim, out, chained, st);
}

}  // namespace mpd
