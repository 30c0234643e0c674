// Fused 2D step (march2d.cuh) of FP32 fields with |psi| in the psi-fractions (variable-sign fields,
// Sect. 3.1.5), the divergent-flow term (Sect. 3.1.3) or both: a translation unit of its own
// beside fused2d.cu so that the two compile side by side.
//
// Bound by issue like the plain march, whose instructions these options barely add to (the
// divergence takes four adds per cell and two fma per face).  Measured: |psi| with the limiter on
// 1021 x 1000 cells 80.3 us per step on the staged kernels, 11.3 us here.
#include "march2d.cuh"

namespace mpd {
namespace {

template <int NC, int EXT>
void launch_ext(const F2Params<float>& p, const Opts& o, cudaStream_t st) {
  if (o.fct) {
    if (o.nug) launch<float, NC, true, true, false, false, false, false, EXT>(p, st);
    else launch<float, NC, true, false, false, false, false, false, EXT>(p, st);
  } else {
    if (o.nug) launch<float, NC, false, true, false, false, false, false, EXT>(p, st);
    else launch<float, NC, false, false, false, false, false, false, EXT>(p, st);
  }
}

}  // namespace

int fused_step_ext(const Grid& g, const Opts& o, const StepArgs<float>& a, cudaStream_t st) {
  if (g.nd != 2 || o.n_iters != 2 || o.tot || o.iga || o.open || o.kahan) return MPDATA_EUNSUPPORTED;
  if (a.psi_out == a.psi_in) return MPDATA_EUNSUPPORTED;
  bool band_auto = false;
  F2Params<float> p = warp_params(g, o, a, &band_auto);
  if (o.kernel == 3 || (o.kernel == 0 && o.tile_rows == 0 && narrow_lanes(p.n0, p.n1, false))) {
    p = warp_params<float, 2>(g, o, a, &band_auto);
    if (o.abs && o.dfl) launch_ext<2, kExtAbs | kExtDfl>(p, o, st);
    else if (o.abs) launch_ext<2, kExtAbs>(p, o, st);
    else launch_ext<2, kExtDfl>(p, o, st);
  } else {
    if (o.abs && o.dfl) launch_ext<4, kExtAbs | kExtDfl>(p, o, st);
    else if (o.abs) launch_ext<4, kExtAbs>(p, o, st);
    else launch_ext<4, kExtDfl>(p, o, st);
  }
  return cudaGetLastError() == cudaSuccess ? MPDATA_OK : MPDATA_ECUDA;
}

}  // namespace mpd
