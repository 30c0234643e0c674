// Launches of the fused 2D step (march2d.cuh): the warp march of one field with every option but
// the third-order terms, |psi| and the divergent-flow term, its compensated-state and
// tape-recording variants, and the batched kernel that walks a table of tiles of many fields.
#include "march2d.cuh"

namespace mpd {
namespace {

using namespace dev;

// Ensemble of fields: a persistent grid walks a table of (field, strip, row tile) items.
template <typename T>
struct BatchParams {
  const T* psi;
  T* out;
  const T* gc0;
  const T* gc1;
  const T* G;
  const T* R;
  const BatchField* fields;
  const int* item_field;  // field of every work item
  int n_items, ty;
  T dt, scale;
  int rhs_a, rhs_b, vec_ok;
  bool chained;
};

template <typename T, int NC, bool FCT, bool NUG, bool IGA, bool KAHAN>
__global__ void __launch_bounds__(kWarps * 32) k_fused2d_batched(const BatchParams<T> b) {
  constexpr int kArr = arrs<false>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  T* ring = reinterpret_cast<T*>(smem_raw) + static_cast<size_t>(wib) * kSlots * kArr * cols<NC>();
  grid_release_small<T>(gridDim.x);
  grid_wait();  // the step before this one, when launched as its dependent
  const int total = gridDim.x * kWarps;
  for (int item = blockIdx.x * kWarps + wib; item < b.n_items; item += total) {
    const BatchField fd = b.fields[b.item_field[item]];
    const int local = item - fd.item_base;
    F2Params<T> p;
    p.psi = b.psi + fd.offset;
    p.out = b.out + fd.offset;
    p.gc0 = b.gc0 + fd.offset;
    p.gc1 = b.gc1 + fd.offset;
    p.G = NUG ? b.G + fd.offset : nullptr;
    p.R = b.R ? b.R + fd.offset : nullptr;
    p.n0 = fd.n0;
    p.n1 = fd.n1;
    p.strips = fd.strips;
    p.rowtiles = 0;
    p.ty = b.ty;
    p.dt = b.dt;
    p.scale = b.scale;
    p.rhs_a = b.rhs_a;
    p.rhs_b = b.rhs_b;
    p.vec = fd.vec && b.vec_ok;
    p.lo = nullptr;
    p.lo_out = nullptr;
    p.tape = nullptr;
    p.tape_n = 0;
    p.chained = b.chained;
    march_tile<T, NC, FCT, NUG, IGA, KAHAN, false>(p, local % fd.strips, (local / fd.strips) * b.ty, ring, lane);
  }
}

template <typename T, int NC, bool FCT, bool NUG>
void launch_mode(const F2Params<T>& p, bool iga, bool kahan, cudaStream_t st) {
  if (iga) {
    if (kahan) launch<T, NC, FCT, NUG, true, true>(p, st); else launch<T, NC, FCT, NUG, true, false>(p, st);
  } else {
    if (kahan) launch<T, NC, FCT, NUG, false, true>(p, st); else launch<T, NC, FCT, NUG, false, false>(p, st);
  }
}

template <typename T, int NC>
void launch_all(const F2Params<T>& p, const Opts& o, cudaStream_t st) {
  if (o.fct) {
    if (o.nug) launch_mode<T, NC, true, true>(p, o.iga, o.kahan, st);
    else launch_mode<T, NC, true, false>(p, o.iga, o.kahan, st);
  } else {
    if (o.nug) launch_mode<T, NC, false, true>(p, o.iga, o.kahan, st);
    else launch_mode<T, NC, false, false>(p, o.iga, o.kahan, st);
  }
}

template <typename T, int NC, bool FCT, bool NUG, bool IGA, bool KAHAN>
void launch_b(const BatchParams<T>& b, cudaStream_t st) {
  const size_t smem = static_cast<size_t>(kWarps) * kSlots * arrs<false>() * cols<NC>() * sizeof(T);
  static PerDevice<int> grid_of;  // persistent grid: every block that fits on the GPU at once
  const int grid = grid_of.get([&](int dev) {
    cudaFuncSetAttribute(k_fused2d_batched<T, NC, FCT, NUG, IGA, KAHAN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         static_cast<int>(smem));
    int per_sm = 0, sms = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fused2d_batched<T, NC, FCT, NUG, IGA, KAHAN>,
                                                  kWarps * 32, smem);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (per_sm > 0 ? per_sm : 1) * (sms > 0 ? sms : 1);
  });
  const int need = (b.n_items + kWarps - 1) / kWarps;
  const unsigned blocks = need < grid ? need : grid;
  launch_chained(b.chained, k_fused2d_batched<T, NC, FCT, NUG, IGA, KAHAN>, dim3(blocks),
                 dim3(kWarps * 32), smem, st, b);
}

template <typename T, int NC, bool FCT, bool NUG>
void launch_b_mode(const BatchParams<T>& b, bool iga, bool kahan, cudaStream_t st) {
  if (iga) {
    if (kahan) launch_b<T, NC, FCT, NUG, true, true>(b, st); else launch_b<T, NC, FCT, NUG, true, false>(b, st);
  } else {
    if (kahan) launch_b<T, NC, FCT, NUG, false, true>(b, st); else launch_b<T, NC, FCT, NUG, false, false>(b, st);
  }
}

}  // namespace

template <typename T>
int fused_batched_columns() { return sizeof(T) == 4 ? 4 : 2; }
template int fused_batched_columns<float>();
template int fused_batched_columns<double>();

int fused_strip_stride(int nc) { return 32 * nc - 2 * kLead; }

namespace {

template <typename T, int NC>
int batched_launch(const BatchTable& tab, const Opts& o, const T* psi_in, T* psi_out, const T* gc0, const T* gc1,
                   const T* G, const T* R, T dt, T scale, bool chained, cudaStream_t st) {
  BatchParams<T> b;
  b.chained = chained;
  b.psi = psi_in;
  b.out = psi_out;
  b.gc0 = gc0;
  b.gc1 = gc1;
  b.G = o.nug ? G : nullptr;
  b.R = R;
  b.fields = tab.fields;
  b.item_field = tab.item_field;
  b.n_items = tab.n_items;
  b.ty = tab.ty;
  b.dt = dt;
  b.scale = scale;
  b.rhs_a = o.rhs_a;
  b.rhs_b = o.rhs_b;
  const size_t va = NC * sizeof(T) <= 16 ? NC * sizeof(T) : 16;
  b.vec_ok = al(psi_in, va) && al(psi_out, va) && al(gc0, va) && al(gc1, va) && al(b.G, va) && al(R, va);
  if (o.fct) {
    if (o.nug) launch_b_mode<T, NC, true, true>(b, o.iga, o.kahan, st);
    else launch_b_mode<T, NC, true, false>(b, o.iga, o.kahan, st);
  } else {
    if (o.nug) launch_b_mode<T, NC, false, true>(b, o.iga, o.kahan, st);
    else launch_b_mode<T, NC, false, false>(b, o.iga, o.kahan, st);
  }
  return cudaGetLastError() == cudaSuccess ? MPDATA_OK : MPDATA_ECUDA;
}

}  // namespace

template <typename T>
int fused_batched_step(const BatchTable& tab, const Opts& o, const T* psi_in, T* psi_out, const T* gc0,
                       const T* gc1, const T* G, const T* R, T dt, T scale, bool chained, cudaStream_t st, int nc) {
  if (o.n_iters != 2 || o.tot || o.abs || o.dfl || o.open) return MPDATA_EUNSUPPORTED;
  if (sizeof(T) == 4 && nc == 2)
    return batched_launch<T, 2>(tab, o, psi_in, psi_out, gc0, gc1, G, R, dt, scale, chained, st);
  if (nc != fused_batched_columns<T>()) return MPDATA_EINVAL;
  return batched_launch<T, sizeof(T) == 4 ? 4 : 2>(tab, o, psi_in, psi_out, gc0, gc1, G, R, dt, scale, chained, st);
}

template int fused_batched_step<float>(const BatchTable&, const Opts&, const float*, float*, const float*,
                                       const float*, const float*, const float*, float, float, bool, cudaStream_t,
                                       int);
template int fused_batched_step<double>(const BatchTable&, const Opts&, const double*, double*, const double*,
                                        const double*, const double*, const double*, double, double, bool,
                                        cudaStream_t, int);

namespace {

template <bool FCT, bool NUG, int NC = 4>
void launch_comp(const F2Params<float>& p, bool iga, cudaStream_t st) {
  if (iga) launch<float, NC, FCT, NUG, true, false, true>(p, st);
  else launch<float, NC, FCT, NUG, false, false, true>(p, st);
}

}  // namespace

template <typename T>
int fused_step(const Grid& g, const Opts& o, const StepArgs<T>& a, T*, cudaStream_t st) {
  if (g.nd != 2 || o.n_iters != 2 || o.tot || o.open) return MPDATA_EUNSUPPORTED;
  if (a.psi_out == a.psi_in) return MPDATA_EUNSUPPORTED;
  if (o.abs || o.dfl) {
    if constexpr (sizeof(T) == 4) return fused_step_ext(g, o, a, st);
    else return MPDATA_EUNSUPPORTED;
  }
  constexpr int NC = sizeof(T) == 4 ? 4 : 2;
  bool band_auto = false;
  if (o.kernel == 3 && sizeof(T) == 4) {  // narrow lanes (FP32)
    launch_all<T, 2>(warp_params<T, 2>(g, o, a, &band_auto), o, st);
    return cudaGetLastError() == cudaSuccess ? MPDATA_OK : MPDATA_ECUDA;
  }
  const F2Params<T> p = warp_params(g, o, a, &band_auto);
  if (o.kernel == 2 || (o.kernel == 0 && band_auto)) return band_step<T>(g, o, a, st);
  if constexpr (sizeof(T) == 4) {
    if (o.kernel == 0 && o.tile_rows == 0 && narrow_lanes(p.n0, p.n1, false)) {
      launch_all<T, 2>(warp_params<T, 2>(g, o, a, &band_auto), o, st);
      return cudaGetLastError() == cudaSuccess ? MPDATA_OK : MPDATA_ECUDA;
    }
  }
  launch_all<T, NC>(p, o, st);
  return cudaGetLastError() == cudaSuccess ? MPDATA_OK : MPDATA_ECUDA;
}

int fused_step_comp(const Grid& g, const Opts& o, const StepArgs<float>& a, const float* lo_in, float* lo_out,
                    cudaStream_t st) {
  if (g.nd != 2 || o.n_iters != 2 || o.tot || o.abs || o.dfl || o.open) return MPDATA_EUNSUPPORTED;
  if (a.psi_out == a.psi_in || lo_out == lo_in) return MPDATA_EUNSUPPORTED;
  bool band_auto = false;
  const bool narrow = o.kernel == 3 || (o.kernel == 0 && o.tile_rows == 0 && narrow_lanes(g.n[1], g.n[2], true));
  if (narrow && o.fct && !o.nug) {  // lanes of 2 columns, the common case
    F2Params<float> p = warp_params<float, 2>(g, o, a, &band_auto, true);
    p.lo = lo_in;
    p.lo_out = lo_out;
    p.vec = p.vec && al(lo_in, 8) && al(lo_out, 8);
    launch_comp<true, false, 2>(p, o.iga, st);
    return cudaGetLastError() == cudaSuccess ? MPDATA_OK : MPDATA_ECUDA;
  }
  F2Params<float> p = warp_params(g, o, a, &band_auto, true);  // the warp march carries the low parts
  p.lo = lo_in;
  p.lo_out = lo_out;
  p.vec = p.vec && al(lo_in, 16) && al(lo_out, 16);
  if (o.fct) {
    if (o.nug) launch_comp<true, true>(p, o.iga, st); else launch_comp<true, false>(p, o.iga, st);
  } else {
    if (o.nug) launch_comp<false, true>(p, o.iga, st); else launch_comp<false, false>(p, o.iga, st);
  }
  return cudaGetLastError() == cudaSuccess ? MPDATA_OK : MPDATA_ECUDA;
}

template <typename T>
int fused_tape(const Grid& g, const Opts& o, const StepArgs<T>& a, T* tape, cudaStream_t st) {
  if (g.nd != 2 || o.n_iters != 2 || o.tot || o.abs || o.dfl || o.open || o.kahan || o.nug || o.iga || o.rhs_a || o.rhs_b)
    return MPDATA_EUNSUPPORTED;
  if (a.psi_out == nullptr || a.psi_out == a.psi_in) return MPDATA_EUNSUPPORTED;
  constexpr int NC = sizeof(T) == 4 ? 4 : 2;
  bool band_auto = false;
  F2Params<T> p = warp_params(g, o, a, &band_auto);
  if (o.kernel == 2 || (o.kernel == 0 && band_auto)) return band_tape<T>(g, o, a, tape, st);
  if constexpr (sizeof(T) == 4) {  // the lanes that the step itself takes, so that the results are its bits
    if (o.kernel == 3 || (o.kernel == 0 && o.tile_rows == 0 && narrow_lanes(p.n0, p.n1, false))) {
      p = warp_params<T, 2>(g, o, a, &band_auto);
      p.tape = tape;
      p.tape_n = g.N;
      if (o.fct) launch<T, 2, true, false, false, false, false, true>(p, st);
      else launch<T, 2, false, false, false, false, false, true>(p, st);
      return cudaGetLastError() == cudaSuccess ? MPDATA_OK : MPDATA_ECUDA;
    }
  }
  p.tape = tape;
  p.tape_n = g.N;
  if (o.fct) launch<T, NC, true, false, false, false, false, true>(p, st);
  else launch<T, NC, false, false, false, false, false, true>(p, st);
  return cudaGetLastError() == cudaSuccess ? MPDATA_OK : MPDATA_ECUDA;
}

template int fused_tape<float>(const Grid&, const Opts&, const StepArgs<float>&, float*, cudaStream_t);
template int fused_tape<double>(const Grid&, const Opts&, const StepArgs<double>&, double*, cudaStream_t);

template int fused_step<float>(const Grid&, const Opts&, const StepArgs<float>&, float*, cudaStream_t);
template int fused_step<double>(const Grid&, const Opts&, const StepArgs<double>&, double*, cudaStream_t);

}  // namespace mpd
