// One step of 2D fields as a shared-memory tile kernel: every option and any number of passes
// whose reach fits, open edges included.  It takes the cases that the register marches
// (march2d.cuh, band2d.cu) leave, the third-order terms, more than two passes, open edges
// and in FP64 the divergent-flow option, where it is the faster one: the staged kernels keep FP64
// fields below about 200^2 and most steps whose halo costs more than their launches (tile_cost.h).
//
// Why a tile: those cases ran as one kernel per sub-step (4 launches per pass), each reading every
// neighbour again through L1 and L2; the shallow-water step of three 320^2 FP64 fields took 22
// launches.  A block loads the step's input once with its halo, H = 1 + (n_iters - 1) r cells (r: 1,
// one more with the limiter, one more with the third-order terms), runs the sub-steps there,
// separated by block barriers, on regions that shrink towards the tile, and writes the tile.  The
// price is the recomputed halo (1.2x the arithmetic for a 32 x 16 tile with H = 3).  32-row tiles repeat
// less of it than 16-row tiles, which give a small FP64 field more blocks (576^2, third-order terms and
// limiter: 200 us in 32 rows, 176 in 16; 544^2 135 and 143).  FP64 is bound by the FP64 pipe, FP32 by
// shared-memory issue.  Fields of one shape with one advector (the shallow-water system) share a
// launch, one grid layer each.
//
// Measured: a shallow-water step of three 320^2 FP64 fields with open edges, |psi|, limiter and
// divergent-flow term 218 us staged, 96 here with its source kernels (the FP64 pipe's floor is about
// 65 us); sign tests in place of products, the divergence once per cell and 32-row tiles took it
// there from 108.
//
// Open edges (Sect. 2.4): only cells of the field are computed; a neighbour beyond an open edge is
// the edge cell, a face beyond it the adjacent interior face (offset clamping, in the tiles that
// touch an edge only).  Periodic dimensions wrap when the tile is loaded.
//
// The expressions and their order are those of the staged kernels (staged.cu).
#include <cuda_runtime.h>

#include "kernels.h"
#include "launch.cuh"
#include "stencil2d.cuh"
#include "tile_cost.h"

namespace mpd {
namespace {

using namespace dev;

constexpr int kThreadsT = 256;
constexpr int kCols = kTileCols;  // tile columns; rows: 32, or in FP64 16 (tile_rows)

template <typename T>
struct TileParams {
  const T* psi;
  T* out;
  const T* gc0;
  const T* gc1;
  const T* G;
  const T* R;
  long long field;  // elements from one field of psi and out to the next (grid layers)
  int n0, n1, K, reach, H;
  T dt, scale;
  bool open0, open1, tot, abs, dfl, kahan, rhs_a, rhs_b;
  bool chained;  // launched as a dependent of the kernel before it (StepArgs::chained)
};

// f(r, c) over rows [r0, r1) x columns [c0, c1), dealt to the threads cell by cell
template <class F>
__device__ __forceinline__ void over(int r0, int r1, int c0, int c1, F&& f) {
  const int W = c1 - c0, n = (r1 - r0) * W;
  if (n <= 0) return;
  const int t = static_cast<int>(threadIdx.x);
  int r = r0 + t / W, c = c0 + t % W;
  const int dr = kThreadsT / W, dc = kThreadsT % W;
  for (int k = t; k < n; k += kThreadsT) {
    f(r, c);
    r += dr;
    c += dc;
    if (c >= c1) { c -= W; ++r; }
  }
}

// Offsets in the tile, along one dimension, from a cell to its neighbours at -1, +1, +2 and to the
// storage of the faces at +1/2, -1/2, +3/2 of the component along it
struct Off { int m1, p1, p2, f0, fm, fp; };
__device__ __forceinline__ Off offs(bool edge, int x, int n, int s) {
  Off o{-s, s, 2 * s, 0, -s, s};
  if (edge) {  // neighbours clamped to 0 .. n-1, faces to 0 .. n-2
    o.m1 = x > 0 ? -s : 0;
    o.p1 = x < n - 1 ? s : 0;
    o.p2 = x < n - 2 ? 2 * s : (x < n - 1 ? s : 0);
    o.f0 = x < n - 1 ? 0 : -s;
    o.fm = x > 0 ? -s : 0;
    o.fp = x < n - 2 ? s : (x < n - 1 ? 0 : -s);
  }
  return o;
}

// n1/d and n2/d (0 for d = 0) with one guard
__device__ __forceinline__ void ratio2(float n1, float n2, float d, float& r1, float& r2) {
  const float r = rcp_normal(d);
  r1 = divisible(d) ? n1 * r : 0.0f;
  r2 = divisible(d) ? n2 * r : 0.0f;
}
__device__ __forceinline__ void ratio2(double n1, double n2, double d, double& r1, double& r2) {
  r1 = ratio(n1, d);
  r2 = ratio(n2, d);
}
__device__ __forceinline__ bool sum_counts(float x) { return x > 0.0f; }
__device__ __forceinline__ bool sum_counts(double x) { return gt0(x) && divisible(x); }
__device__ __forceinline__ bool zero(float x) { return x == 0.0f; }
__device__ __forceinline__ bool zero(double x) { return !nonzero(x); }

template <typename T, int kRows, bool FCT, bool IGA, bool NUG>
__global__ void __launch_bounds__(kThreadsT, 2) k_tile2d(const TileParams<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int H = p.H, L = kCols + 2 * H, A = (kRows + 2 * H) * L;
  T* cur = reinterpret_cast<T*>(smem_raw);  // psi^(k-1)
  T* nxt = cur + A;                         // psi^(k)
  T* C0 = nxt + A;                          // the advector that drives the pass's pseudo-advector
  T* C1 = C0 + A;
  T* W0 = C1 + A;                           // the pseudo-advector, limited in place
  T* W1 = W0 + A;
  T* const BU = W1 + A;
  T* const BD = BU + A;
  T* const MX = BD + A;                     // bounds, with more than two passes and the limiter
  T* const MN = MX + A;
  T* const Gs = FCT ? (p.K > 2 ? MN + A : MX) : BU;
  T* const DV = Gs + (NUG ? A : 0);         // the advector's difference across the cell (divergent flow)
  const int R0 = static_cast<int>(blockIdx.y) * kRows, Q0 = static_cast<int>(blockIdx.x) * kCols;
  const int x0 = R0 - H, y0 = Q0 - H;  // field row and column of the tile array's corner
  const T* const psi = p.psi + blockIdx.z * p.field;
  T* const out = p.out + blockIdx.z * p.field;
  // whether the tile's array leaves the field across an open edge
  const bool e0 = p.open0 && (x0 < 0 || x0 + kRows + 2 * H > p.n0);
  const bool e1 = p.open1 && (y0 < 0 || y0 + L > p.n1);
  auto inside = [&](int r, int c) {
    return !(e0 && (x0 + r < 0 || x0 + r >= p.n0)) && !(e1 && (y0 + c < 0 || y0 + c >= p.n1));
  };
  grid_release_small<T>(gridDim.x * gridDim.y * gridDim.z);
  grid_wait();
  over(0, kRows + 2 * H, 0, L, [&](int r, int c) {
    if (!inside(r, c)) return;
    int gr = x0 + r, gc = y0 + c;
    while (gr < 0) gr += p.n0;
    while (gr >= p.n0) gr -= p.n0;
    while (gc < 0) gc += p.n1;
    while (gc >= p.n1) gc -= p.n1;
    const long long g = static_cast<long long>(gr) * p.n1 + gc;
    const int i = r * L + c;
    T v = psi[g];
    if (p.rhs_b) v = v + p.dt * p.R[g];
    cur[i] = v;
    C0[i] = p.gc0[g] * p.scale;
    C1[i] = p.gc1[g] * p.scale;
    if (NUG) Gs[i] = p.G[g];
  });
  __syncthreads();
  // donor-cell pass (Eqs. 4-5) of cell i from psi q with advector (V0, V1)
  auto donor = [&](const T* q, const T* V0, const T* V1, int i, const Off& a, const Off& b, bool unit) {
    const T x = q[i];
    const T Gi = NUG ? Gs[i] : T(1);
    const T v0p = V0[i + a.f0], v0m = V0[i + a.fm], v1p = V1[i + b.f0], v1m = V1[i + b.fm];
    const T Fp0 = unit ? v0p : flux(x, q[i + a.p1], v0p), Fm0 = unit ? v0m : flux(q[i + a.m1], x, v0m);
    const T Fp1 = unit ? v1p : flux(x, q[i + b.p1], v1p), Fm1 = unit ? v1m : flux(q[i + b.m1], x, v1m);
    const T t[4] = {NUG ? -fdiv(Fp0, Gi) : -Fp0, NUG ? fdiv(Fm0, Gi) : Fm0, NUG ? -fdiv(Fp1, Gi) : -Fp1,
                    NUG ? fdiv(Fm1, Gi) : Fm1};
    T s = x, comp = T(0);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (p.kahan) kahan_add(s, comp, t[j]);
      else s = s + t[j];
    }
    return s;
  };
  {
    const int m = H - 1;  // pass 1 on the margin the later passes need
    over(H - m, H + kRows + m, H - m, H + kCols + m, [&](int r, int c) {
      if (!inside(r, c)) return;
      const int i = r * L + c;
      const Off a = offs(e0, x0 + r, p.n0, L), b = offs(e1, y0 + c, p.n1, 1);
      nxt[i] = donor(cur, C0, C1, i, a, b, false);
      if (p.dfl) DV[i] = (C0[i + a.f0] - C0[i + a.fm]) + (C1[i + b.f0] - C1[i + b.fm]);
    });
  }
  __syncthreads();
  T* psi0 = cur;  // for the bounds of the first corrective pass
  cur = nxt;
  nxt = psi0;
  auto fr = [&](T x) { return p.abs ? absv(x) : x; };
  for (int k = 2; k <= p.K; ++k) {
    const int m = (p.K - k) * p.reach;  // psi^(k) is needed m cells beyond the tile
    const int M = FCT ? m + 1 : m;      // and the pseudo-advector on the faces of these cells
    const int lo = H - M, hr = H + kRows + M, hc = H + kCols + M;
    // ---- pseudo-advector (Eq. 6, cross, third-order and divergent-flow terms): dimension 0 on rows
    // [lo-1, hr) x columns [lo, hc), dimension 1 on rows [lo, hr) x columns [lo-1, hc)
    over(lo - 1, hr, lo - 1, hc, [&](int r, int c) {
      if (!inside(r, c)) return;
      const int i = r * L + c;
      const Off a = offs(e0, x0 + r, p.n0, L), b = offs(e1, y0 + c, p.n1, 1);
      // the face at +1/2 along d of cell i: offsets d along it, q across it; D, Q the advector
      // components along and across it
      auto face = [&](const Off& d, const Off& q, const T* D, const T* Q) {
        const int ip = i + d.p1;
        const T rGb = NUG ? fdiv(T(1), T(0.5) * (Gs[i] + Gs[ip])) : T(1);
        const T V = D[i + d.f0];
        const T f0 = fr(cur[i]), f1 = fr(cur[ip]);
        const T Av = IGA ? (f1 - f0) * T(0.5) : ratio(f1 - f0, f0 + f1);
        T o = (absv(V) - V * V * rGb) * Av;
        const T q0 = Q[i + q.f0], q1 = Q[ip + q.f0], q2 = Q[i + q.fm], q3 = Q[ip + q.fm];
        const T Vs = (q0 + q1) + (q2 + q3);  // four times the mean transverse advector
        const T x = fr(cur[i + q.p1]), y = fr(cur[ip + q.p1]), z = fr(cur[i + q.m1]), w = fr(cur[ip + q.m1]);
        const T Tp = x + y, Bt = z + w;
        T B, D2 = T(0);
        if (IGA) {
          B = (Tp - Bt) * T(0.25);
          if (p.tot) D2 = ((y - x) - (w - z)) * T(0.25);
        } else if (p.tot) {
          ratio2(Tp - Bt, (y - x) - (w - z), Tp + Bt, B, D2);
        } else {
          B = ratio(Tp - Bt, Tp + Bt);
        }
        o = o - T(0.125) * V * Vs * rGb * B;
        if (p.tot) {
          const T fm = fr(cur[i + d.m1]), f2 = fr(cur[i + d.p2]);
          const T num = ((f2 - f1) - f0) + fm;
          const T Dd = IGA ? num * T(0.25) : ratio(num, ((f2 + f1) + f0) + fm);
          o = o + ((T(3) * V * absv(V)) * rGb - (T(2) * V * V * V) * (rGb * rGb) - V) * T(1.0 / 3.0) * Dd;
          o = o + absv(V) * (T(0.25) * Vs) * rGb * (T(1) - T(2) * absv(V) * rGb) * D2;
        }
        if (p.dfl) o = o - T(0.25) * V * (DV[i] + DV[ip]) * rGb;
        return o;
      };
      if (c >= lo) W0[i] = face(a, b, C0, C1);
      if (r >= lo) W1[i] = face(b, a, C1, C0);
    });
    __syncthreads();
    if (FCT) {
      // ---- factors (Sect. 3.1.4) on margin M; the bounds are those of the first corrective pass
      over(lo, hr, lo, hc, [&](int r, int c) {
        if (!inside(r, c)) return;
        const int i = r * L + c;
        const Off a = offs(e0, x0 + r, p.n0, L), b = offs(e1, y0 + c, p.n1, 1);
        const T q = cur[i], qu = cur[i + a.p1], qd = cur[i + a.m1], qr = cur[i + b.p1], ql = cur[i + b.m1];
        T mx, mn;
        if (k == 2) {
          mx = max3(max3(maxv(psi0[i], q), psi0[i + a.p1], qu), max3(psi0[i + a.m1], qd, psi0[i + b.p1]),
                    max3(qr, psi0[i + b.m1], ql));
          mn = min3(min3(minv(psi0[i], q), psi0[i + a.p1], qu), min3(psi0[i + a.m1], qd, psi0[i + b.p1]),
                    min3(qr, psi0[i + b.m1], ql));
          if (p.K > 2) { MX[i] = mx; MN[i] = mn; }
        } else {
          mx = MX[i];
          mn = MN[i];
        }
        const T v0p = W0[i + a.f0], v0m = W0[i + a.fm], v1p = W1[i + b.f0], v1m = W1[i + b.fm];
        const T Fp0 = IGA ? v0p : flux(q, qu, v0p), Fm0 = IGA ? v0m : flux(qd, q, v0m);
        const T Fp1 = IGA ? v1p : flux(q, qr, v1p), Fm1 = IGA ? v1m : flux(ql, q, v1m);
        T in, ou;
        flow_sums(Fm0, Fp0, Fm1, Fp1, in, ou);
        T up = posp(mx - q), dn = posp(q - mn);
        if (NUG) { up = Gs[i] * up; dn = Gs[i] * dn; }
        BU[i] = sum_counts(in) ? fdiv(up, in) : T(1);
        BD[i] = sum_counts(ou) ? fdiv(dn, ou) : T(1);
      });
      __syncthreads();
      // ---- limited pseudo-advector on the faces of margin m, in place
      const int l2 = H - m, r2 = H + kRows + m, c2 = H + kCols + m;
      over(l2 - 1, r2, l2 - 1, c2, [&](int r, int c) {
        if (!inside(r, c)) return;
        const int i = r * L + c;
        auto limit = [&](T* W, int ip) {
          // the unlimited flux V up goes right where V and the upwind value have the same sign, or,
          // where it is zero, where V > 0 (signs alone: no product on the FP64 pipe)
          const T V = W[i], up = gt0(V) ? cur[i] : cur[ip];
          const bool right = IGA || zero(up) ? gt0(V) : !zero(V) && gt0(V) == gt0(up);
          W[i] = V * min3(T(1), right ? BD[i] : BU[i], right ? BU[ip] : BD[ip]);
        };
        // an open edge's last stored face is not one of its cells' faces
        if (c >= l2 && !(e0 && x0 + r >= p.n0 - 1)) limit(W0, i + L);
        if (r >= l2 && !(e1 && y0 + c >= p.n1 - 1)) limit(W1, i + 1);
      });
      __syncthreads();
    }
    // ---- donor-cell pass
    if (k == p.K) {
      over(H, H + kRows, H, H + kCols, [&](int r, int c) {
        const int gr = x0 + r, gc = y0 + c;
        if (gr >= p.n0 || gc >= p.n1) return;
        T s = donor(cur, W0, W1, r * L + c, offs(e0, gr, p.n0, L), offs(e1, gc, p.n1, 1), IGA);
        const long long g = static_cast<long long>(gr) * p.n1 + gc;
        if (p.rhs_a) s = s + p.dt * p.R[g];
        out[g] = s;
      });
    } else {
      over(H - m, H + kRows + m, H - m, H + kCols + m, [&](int r, int c) {
        if (!inside(r, c)) return;
        const int i = r * L + c;
        nxt[i] = donor(cur, W0, W1, i, offs(e0, x0 + r, p.n0, L), offs(e1, y0 + c, p.n1, 1), IGA);
      });
      __syncthreads();
      T* t = cur; cur = nxt; nxt = t;
      t = C0; C0 = W0; W0 = t;
      t = C1; C1 = W1; W1 = t;
      if (p.dfl) {  // of the advector that drives the next pass, on the cells of its faces
        const int w = m - p.reach + (FCT ? 2 : 1);
        over(H - w, H + kRows + w, H - w, H + kCols + w, [&](int r, int c) {
          if (!inside(r, c)) return;
          const int i = r * L + c;
          const Off a = offs(e0, x0 + r, p.n0, L), b = offs(e1, y0 + c, p.n1, 1);
          DV[i] = (C0[i + a.f0] - C0[i + a.fm]) + (C1[i + b.f0] - C1[i + b.fm]);
        });
        __syncthreads();
      }
    }
  }
}

template <typename T, int kRows, bool FCT, bool IGA, bool NUG>
int launch_rows(const TileParams<T>& p, int fields, size_t smem, int most, cudaStream_t st) {
  static PerDevice<bool> attr;
  attr.get([&](int) {
    return cudaFuncSetAttribute(k_tile2d<T, kRows, FCT, IGA, NUG>, cudaFuncAttributeMaxDynamicSharedMemorySize, most) ==
           cudaSuccess;
  });
  const long long ty = (p.n0 + kRows - 1) / kRows;
  if (ty > 65535) return MPDATA_EUNSUPPORTED;
  const dim3 grid(static_cast<unsigned>((p.n1 + kCols - 1) / kCols), static_cast<unsigned>(ty),
                  static_cast<unsigned>(fields));
  launch_chained(p.chained, k_tile2d<T, kRows, FCT, IGA, NUG>, grid, dim3(kThreadsT), smem, st, p);
  return cudaGetLastError() == cudaSuccess ? MPDATA_OK : MPDATA_ECUDA;
}

template <typename T, bool FCT, bool IGA, bool NUG>
int launch_tile(const TileParams<T>& p, int fields, bool always, cudaStream_t st) {
  static PerDevice<int> most_of;
  const int most = most_of.get([](int dev) {
    int m = 0;
    cudaDeviceGetAttribute(&m, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return m;
  });
  const TileCase c{p.n0, p.n1, fields, p.K, FCT, p.tot, NUG, p.dfl, sizeof(T) == 8};
  const int rows = tile_rows(c, static_cast<size_t>(most), always);
  if (rows == 0) return MPDATA_EUNSUPPORTED;
  const size_t smem = tile_smem(c, rows);
  if constexpr (sizeof(T) == 8) {
    if (rows == 16) return launch_rows<T, 16, FCT, IGA, NUG>(p, fields, smem, most, st);
  }
  return launch_rows<T, 32, FCT, IGA, NUG>(p, fields, smem, most, st);
}

}  // namespace

template <typename T>
int tile2d_step(const Grid& g, const Opts& o, const StepArgs<T>& a, int fields, long long field, cudaStream_t st) {
  if (g.nd != 2 || o.n_iters < 2 || o.n_iters > 8 || a.psi_in == a.psi_out) return MPDATA_EUNSUPPORTED;
  // periodic FP64 |psi| without the divergent-flow term stays on the staged kernels: its step on a
  // positive field is to have the bits of the basic step there (MPDATA_STAGED), and the products here
  // are contracted differently
  if (sizeof(T) == 8 && o.abs && !o.dfl && !o.open) return MPDATA_EUNSUPPORTED;
  TileParams<T> p;
  p.psi = a.psi_in;
  p.out = a.psi_out;
  p.gc0 = a.gc[0];
  p.gc1 = a.gc[1];
  p.G = o.nug ? a.g : nullptr;
  p.R = a.r;
  p.field = field;
  p.n0 = g.n[1];
  p.n1 = g.n[2];
  p.K = o.n_iters;
  const TileCase c{p.n0, p.n1, fields, p.K, o.fct, o.tot, o.nug, o.dfl, sizeof(T) == 8};
  p.reach = tile_reach(c);
  p.H = tile_halo(c);
  p.dt = a.dt;
  p.scale = a.gc_scale;
  p.open0 = g.open[1];
  p.open1 = g.open[2];
  p.tot = o.tot;
  p.abs = o.abs;
  p.dfl = o.dfl;
  p.kahan = o.kahan;
  p.rhs_a = o.rhs_a;
  p.rhs_b = o.rhs_b;
  p.chained = a.chained;
  const bool always = o.kernel != 0;  // MPDATA_TUNE_KERNEL asks for a fused kernel
#define MPD_T(F, I) \
  (o.nug ? launch_tile<T, F, I, true>(p, fields, always, st) : launch_tile<T, F, I, false>(p, fields, always, st))
  if (o.fct) return o.iga ? MPD_T(true, true) : MPD_T(true, false);
  return o.iga ? MPD_T(false, true) : MPD_T(false, false);
#undef MPD_T
}

template int tile2d_step<float>(const Grid&, const Opts&, const StepArgs<float>&, int, long long, cudaStream_t);
template int tile2d_step<double>(const Grid&, const Opts&, const StepArgs<double>&, int, long long, cudaStream_t);

}  // namespace mpd
