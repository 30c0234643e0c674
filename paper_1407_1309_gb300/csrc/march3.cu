// Dispatch of the vectorised FP32 3D z-marches (march3.cuh) and their form with 16-byte chunks.
#include <cstdlib>

#include "march3.cuh"

namespace mpd {
namespace {

// Fields of at least 48 columns; narrower ones take the scalar z-march of staged.cu, whose 32-column
// tiles leave fewer lanes without a cell.  MPDATA_MARCH3=0 in the environment selects the scalar
// z-march everywhere.
bool use_vec(const Grid& g) {
  static const bool off = [] {
    const char* e = std::getenv("MPDATA_MARCH3");
    return e && std::atoi(e) == 0;
  }();
  return !off && g.nd == 3 && !g.any_open() && g.n[2] >= 48;
}

bool al16(const void* p) { return p == nullptr || (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Whether rows move in 16-byte chunks: tiles of 128 columns, aligned arrays, an x extent of
// whole chunks
bool chunks(const Grid& g, const float* const* v, const float* const* w) {
  for (int d = 0; d < 3; ++d)
    if (!al16(v[d]) || !al16(w[d])) return false;
  return g.n[2] % 4 == 0 && g.n[2] >= 128;
}

}  // namespace

bool antidiff3_vec(const Grid& g, const float* psi, const float* const* v, float vscale, const float* G, bool iga,
                   bool tot, bool abs_psi, float* const* out, bool chained, cudaStream_t st) {
  if (!use_vec(g)) return false;
  if (chunks(g, v, out) && al16(psi) && al16(G)) antidiff3_nc<4, true>(g, psi, v, vscale, G, iga, tot, abs_psi, out, chained, st);
  else antidiff3_cells(g, psi, v, vscale, G, iga, tot, abs_psi, out, chained, st);
  return true;
}

bool p1b3_vec(const Grid& g, const float* psi, const float* const* v, float vscale, const float* G, bool kahan,
              float* p1, float* mx, float* mn, bool chained, cudaStream_t st) {
  if (!use_vec(g)) return false;
  const float* const o[3] = {p1, mx, mn};
  if (chunks(g, v, o) && al16(psi) && al16(G)) p1b3_nc<4, true>(g, psi, v, vscale, G, kahan, p1, mx, mn, chained, st);
  else p1b3_cells(g, psi, v, vscale, G, kahan, p1, mx, mn, chained, st);
  return true;
}

bool corr3_vec(const Grid& g, const float* psi, const float* const* vu, const float* G, bool iga, bool kahan,
               const float* mx, const float* mn, bool post, float* const* lim, float* out, bool chained, cudaStream_t st) {
  if (!use_vec(g) || kahan || post) return false;
  if (chunks(g, vu, lim) && al16(psi) && al16(G) && al16(mx) && al16(mn) && al16(out))
    corr3_nc<4, true>(g, psi, vu, G, iga, mx, mn, lim, out, chained, st);
  else corr3_cells(g, psi, vu, G, iga, mx, mn, lim, out, chained, st);
  return true;
}

}  // namespace mpd
