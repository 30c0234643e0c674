// Batched step: every field of an ensemble handle (independent 2D fields of
// uneven sizes, concatenated) advanced by one launch of the fused kernel whose
// persistent grid walks a table of (field, strip, row tile) work items.  The
// table is built on the host once per handle and tile height and kept on the
// device with the handle.
#include <cuda_runtime.h>

#include <vector>

#include "kernels.h"

namespace mpd {
namespace {

struct TableHolder {
  BatchTable tab{};
  int nc = 0;
  int rows = 0, kernel = 0;  // the MPDATA_TUNE_TILE_ROWS and MPDATA_TUNE_KERNEL it was built for
};

// Tile height of an ensemble and the time a step should take (microseconds).  The tiles are dealt out
// in turn to the warps of a persistent grid of up to `most` blocks of 4 per SM; with k blocks on the
// fullest SM a row takes their warps row_us[k - 1].
struct BatchRows {
  int ty;
  double us;
};
// What one launch of the kernel takes: FP32 marches a 6-row ramp at a row's price, and the warps of an
// SM share its issue slots, so that a warp's share is the rows of all tiles over the warps, plus on
// average half a tile that ends after the others.  FP64 is bound by the SM's FP64 pipe: two blocks
// take nearly twice one's time, the ramp's half-filled rows cost 3 (one tile of 8 .. 128 rows: 73 ..
// 852 us), and a round of tiles that not every warp gets takes almost the time of a full one.
struct BatchCost {
  int most;
  const double* row_us;
  int ramp;
  bool fp64;
};
BatchRows batch_rows(const Grid* grids, int nf, int strip, const BatchCost& c) {
  BatchRows best{32, -1.0};
  for (int ty : {8, 12, 16, 24, 32, 48, 64, 96, 128}) {
    long long tiles = 0;
    for (int f = 0; f < nf; ++f)
      tiles += static_cast<long long>((grids[f].n[2] + strip - 1) / strip) * ((grids[f].n[1] + ty - 1) / ty);
    const long long one = 152 * 4;  // warps of one block per SM
    const long long k = tiles > one * c.most ? c.most : (tiles + one - 1) / one;
    const double rounds = static_cast<double>(tiles) / static_cast<double>(one * k);
    const double full = static_cast<double>((tiles + one * k - 1) / (one * k));
    double share = full;
    if (rounds > 1.0 && !c.fp64) share = rounds + 0.5;
    else if (rounds > 2.0) share = 0.5 * (rounds + full);
    const double us = c.row_us[k - 1] * share * (ty + c.ramp);
    if (best.us < 0.0 || us < best.us) best = {ty, us};
  }
  return best;
}

}  // namespace

void batched_free(mpdata_s* h) {
  void** slot = handle_batch(h);
  auto* th = static_cast<TableHolder*>(*slot);
  if (th) {
    cudaFree(th->tab.fields);
    cudaFree(th->tab.item_field);
    delete th;
    *slot = nullptr;
  }
}

namespace {

// The handle's table for lanes of nc columns and tiles of ty rows, in place of the one it has.
int build_table(mpdata_s* h, int nc, int ty) {
  batched_free(h);
  const int nf = handle_fields(h);
  const Grid* grids = handle_grids(h);
  const long long* offs = handle_offsets(h);
  const int stride = fused_strip_stride(nc);
  std::vector<BatchField> fields(nf);
  std::vector<int> item_field;
  for (int f = 0; f < nf; ++f) {
    BatchField& b = fields[f];
    b.offset = offs[f];
    b.n0 = grids[f].n[1];
    b.n1 = grids[f].n[2];
    b.strips = (b.n1 + stride - 1) / stride;
    b.item_base = static_cast<int>(item_field.size());
    b.vec = (b.n1 % nc == 0) && (b.offset % nc == 0);
    const long long items = static_cast<long long>(b.strips) * ((b.n0 + ty - 1) / ty);
    if (item_field.size() + items > (1LL << 30)) return MPDATA_EUNSUPPORTED;
    item_field.insert(item_field.end(), static_cast<size_t>(items), f);
  }
  auto* th = new TableHolder;
  th->nc = nc;
  th->tab.ty = ty;
  th->tab.n_items = static_cast<int>(item_field.size());
  if (cudaMalloc(&th->tab.fields, sizeof(BatchField) * nf) != cudaSuccess ||
      cudaMalloc(&th->tab.item_field, sizeof(int) * item_field.size()) != cudaSuccess) {
    cudaFree(th->tab.fields);
    delete th;
    return MPDATA_ENOMEM;
  }
  cudaMemcpy(th->tab.fields, fields.data(), sizeof(BatchField) * nf, cudaMemcpyHostToDevice);
  cudaMemcpy(th->tab.item_field, item_field.data(), sizeof(int) * item_field.size(), cudaMemcpyHostToDevice);
  *handle_batch(h) = th;
  return MPDATA_OK;
}

}  // namespace

template <typename T>
int batched_step(mpdata_s* h, const T* psi_in, T* psi_out, const T* const* gc, const T* g, const T* r, T dt,
                 T gc_scale, bool chained, const Opts& o) {
  if (handle_nd(h) != 2 || o.n_iters != 2 || o.tot || o.abs || o.dfl || o.open) return MPDATA_EUNSUPPORTED;
  void** slot = handle_batch(h);
  auto* th = static_cast<TableHolder*>(*slot);
  if (th == nullptr || th->rows != o.tile_rows || th->kernel != o.kernel) {
    // FP32 lanes of 4 columns (two blocks fit an SM) or of 2 (four), whichever should be faster: the
    // narrower strips pad less and give a small ensemble more warps (100 fields of 60^2 .. 300^2: 53 ->
    // 36 us per step, 20 of 40^2 .. 120^2: 25 -> 8; 512 fields of 64^2 .. 512^2 with lanes of 4: 389,
    // with lanes of 2: 400).  MPDATA_TUNE_KERNEL = 3 asks for lanes of 2.  FP64 lanes own 2 (two blocks);
    // its heights against 32 rows throughout and the FP32 costs: 64 of 200^2 814 / 789 -> 628, 100 of 60^2 ..
    // 300^2 817 / 939 -> 818, 10 of 500^2 634 / 600 -> 559 us per step.
    constexpr bool fp64 = sizeof(T) == 8;
    constexpr int wide = fp64 ? 2 : 4;
    static const double us4[2] = {0.55, 0.73}, us2[4] = {0.38, 0.455, 0.59, 0.74}, us64[2] = {6.5, 11.6};
    const BatchRows by_wide = batch_rows(handle_grids(h), handle_fields(h), fused_strip_stride(wide),
                                         BatchCost{2, fp64 ? us64 : us4, fp64 ? 3 : 6, fp64});
    int nc = wide, ty = by_wide.ty;
    if (sizeof(T) == 4 && (o.kernel == 3 || (o.kernel == 0 && o.tile_rows == 0))) {
      const BatchRows by_2 = batch_rows(handle_grids(h), handle_fields(h), fused_strip_stride(2), BatchCost{4, us2, 6, false});
      if (o.kernel == 3 || by_2.us < by_wide.us) {
        nc = 2;
        ty = by_2.ty;
      }
    }
    if (o.tile_rows > 0) ty = o.tile_rows;
    // a setting that asks for the table there is keeps it: graphs captured from earlier calls read it
    if (th == nullptr || th->nc != nc || th->tab.ty != ty) {
      const int rc = build_table(h, nc, ty);
      if (rc != MPDATA_OK) return rc;
      th = static_cast<TableHolder*>(*slot);
    }
    th->rows = o.tile_rows;
    th->kernel = o.kernel;
  }
  return fused_batched_step<T>(th->tab, o, psi_in, psi_out, gc[0], gc[1], g, r, dt, gc_scale, chained, handle_stream(h),
                               th->nc);
}

template int batched_step<float>(mpdata_s*, const float*, float*, const float* const*, const float*, const float*,
                                 float, float, bool, const Opts&);
template int batched_step<double>(mpdata_s*, const double*, double*, const double* const*, const double*,
                                  const double*, double, double, bool, const Opts&);

}  // namespace mpd
