// Dispatch of the vectorised FP32 3D z-marches (march3.cuh) and their form with 16-byte chunks.
#include <cstdlib>

#include "march3.cuh"

namespace mpd {
namespace {

// MPDATA_MARCH3 in the environment: 0 selects the scalar z-marches of staged.cu everywhere, 2 the
// widest lanes that suit the row wherever there are 48 columns (comparison and testing).
int forced() {
  static const int v = [] {
    const char* e = std::getenv("MPDATA_MARCH3");
    return e ? std::atoi(e) : 1;
  }();
  return v;
}

bool al16(const void* p) { return p == nullptr || (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// The form of a march over these arrays: rows move in 16-byte chunks in tiles of 128 columns, with
// aligned arrays and an x extent of whole chunks.  Fields of fewer than 48 columns take the scalar
// form, whose 32-column tiles leave fewer lanes without a cell.
March3 form_of(const Grid& g, const float* const* v, const float* const* w, bool aligned) {
  if (forced() == 0 || g.nd != 3 || g.any_open() || g.n[2] < 48) return March3::kScalar;
  for (int d = 0; d < 3; ++d) aligned = aligned && al16(v[d]) && al16(w[d]);
  return march3_form(g.n, aligned && g.n[2] % 4 == 0 && g.n[2] >= 128, forced() == 2);
}

}  // namespace

bool antidiff3_vec(const Grid& g, const float* psi, const float* const* v, float vscale, const float* G, bool iga,
                   bool tot, bool abs_psi, float* const* out, bool chained, cudaStream_t st) {
  const March3 form = form_of(g, v, out, al16(psi) && al16(G));
  if (form == March3::kScalar) return false;
  if (form == March3::kChunks) antidiff3_nc<4, true>(g, psi, v, vscale, G, iga, tot, abs_psi, out, chained, st);
  else antidiff3_cells(g, form == March3::kCells2, psi, v, vscale, G, iga, tot, abs_psi, out, chained, st);
  return true;
}

bool p1b3_vec(const Grid& g, const float* psi, const float* const* v, float vscale, const float* G, bool kahan,
              float* p1, float* mx, float* mn, bool chained, cudaStream_t st) {
  const float* const o[3] = {p1, mx, mn};
  const March3 form = form_of(g, v, o, al16(psi) && al16(G));
  if (form == March3::kScalar) return false;
  if (form == March3::kChunks) p1b3_nc<4, true>(g, psi, v, vscale, G, kahan, p1, mx, mn, chained, st);
  else p1b3_cells(g, form == March3::kCells2, psi, v, vscale, G, kahan, p1, mx, mn, chained, st);
  return true;
}

bool corr3_vec(const Grid& g, const float* psi, const float* const* vu, const float* G, bool iga, bool kahan,
               const float* mx, const float* mn, bool post, float* const* lim, float* out, bool chained, cudaStream_t st) {
  if (kahan || post) return false;
  const March3 form = form_of(g, vu, lim, al16(psi) && al16(G) && al16(mx) && al16(mn) && al16(out));
  if (form == March3::kScalar) return false;
  if (form == March3::kChunks) corr3_nc<4, true>(g, psi, vu, G, iga, mx, mn, lim, out, chained, st);
  else corr3_cells(g, form == March3::kCells2, psi, vu, G, iga, mx, mn, lim, out, chained, st);
  return true;
}

}  // namespace mpd
