// Many steps of a 1D field, or of a system of 1D equations with trapezoidal sources (Sect. 4.1), in
// one launch of one thread-block cluster.
//
// What bounds it: a 1D field of the usual size (100 .. 2000 cells) is too small to fill the GPU and
// its steps depend on each other, so the call costs n_steps times the latency of one step.  One
// kernel per sub-step pays 7 launches per step and field (58 us per step of the two-equation
// system of 1000 cells); one block with the field in shared memory pays one SM's FP64 rate (about
// 1.7 FP64 lane operations per clock) and a block barrier per sub-step (11.2 us per step of 500
// cells in FP64, two passes with the limiter).
//
// Work decomposition: the cluster's blocks (up to 16 SMs) own contiguous ranges of cells, a warp
// owns a chunk of its block's range, one cell per lane, and keeps everything in registers:
// neighbours come from warp shuffles, the advector, G and R are loaded once per call.  A step
// reaches kHalo = 1 + (n_iters - 1) r cells (r below), so the warp's outermost lanes hold copies of
// its neighbours' cells and are recomputed; after S steps the chunk's results are exchanged
// through shared memory: every block's buffer holds its range with S kHalo cells on each side, a
// warp writes its cells there and those near the range's ends also into the neighbouring
// block's buffer (distributed shared memory), then one cluster barrier.  The buffers alternate, so
// one barrier per exchange is enough: a buffer is rewritten only after the barrier that follows
// the reads of it.  S is as large as the lanes allow (a chunk of 16 cells: two steps of the
// two-pass scheme with the limiter).  A system's equations are coupled per cell, so each warp
// advects one equation's chunk and every step exchanges.  Each block gets as few warps as hold its
// cells (500 cells: 16 blocks of 2).
//
// The arithmetic is that of the staged kernels (same expressions); each face's flux is formed
// once and shuffled to the cell on its right.
//
// Measured: 500 cells, FP64, two passes with the limiter 11.2 -> 2.1 us per step, of which the chain
// of 36 dependent FP64 instructions at about 70 clocks each takes 1.2 and the exchange every second
// step and the idle sub-partitions (two warps on four) the rest; the FP64 system of two equations
// and 1000 cells 58 -> 4.0 us per step (six warps on four sub-partitions, an exchange every step).
#include <cuda_runtime.h>

#include "internal.h"
#include "launch.cuh"
#include "stencil2d.cuh"

namespace mpd {
namespace {

using namespace dev;

constexpr int kMaxCluster = 16;
constexpr int kMaxWarps = 32;
constexpr int kLeast = 8;  // cells of its own that a warp must have room for

template <typename T>
struct LineParams {
  int n, n_steps, K, E;
  int halo, S, chunks;  // halo cells of one step, steps between exchanges, chunks per block range
  bool tot, kahan, abs, rhs_a, rhs_b;
  const T* psi_in;
  T* psi_out;
  const T* gc;
  const T* G;
  const T* R;
  const T* b;  // constant part of the trapezoidal sources (SYS), nullable
  T dt;
  TrapezMat m;
};

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// store v at the address p has in the shared memory of block `rank` of the cluster
__device__ __forceinline__ unsigned remote_addr(const void* p, unsigned rank) {
  const unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(p));
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void remote_store(const float* p, unsigned rank, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote_addr(p, rank)), "f"(v) : "memory");
}
__device__ __forceinline__ void remote_store(const double* p, unsigned rank, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote_addr(p, rank)), "d"(v) : "memory");
}

template <typename T> __device__ __forceinline__ T up1(T x) { return __shfl_up_sync(kFull, x, 1); }
template <typename T> __device__ __forceinline__ T down1(T x) { return __shfl_down_sync(kFull, x, 1); }

// a flux sum that takes a limiting factor (0, or in FP64 a subnormal sum, gives the factor 1)
__device__ __forceinline__ bool positive_sum(float x) { return x > 0.0f; }
__device__ __forceinline__ bool positive_sum(double x) { return gt0(x) && divisible(x); }
__device__ __forceinline__ bool is_zero(float x) { return x == 0.0f; }
__device__ __forceinline__ bool is_zero(double x) { return !nonzero(x); }

template <typename T, bool FCT, bool IGA, bool SYS>
__global__ void __launch_bounds__(32 * kMaxWarps) k_line1d(const LineParams<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* const buf = reinterpret_cast<T*>(smem_raw);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int C = static_cast<int>(gridDim.x);  // one cluster
  const int rank = static_cast<int>(cluster_rank());
  const int n = p.n, E = SYS ? p.E : 1;
  auto start_of = [&](int r) { return static_cast<int>(static_cast<long long>(r) * n / C); };
  const int c0 = start_of(rank), c1 = start_of(rank + 1);
  const int HS = p.halo * p.S;
  const int most = (n + C - 1) / C;         // the longest range of a block
  const int pitch = most + 2 * HS;          // one equation's buffer
  const int e = SYS ? w / p.chunks : 0, chunk = SYS ? w - e * p.chunks : w;
  const int u = (most + p.chunks - 1) / p.chunks;
  const int w0 = c0 + chunk * u, w1 = w0 + u < c1 ? w0 + u : c1;
  const int c = w0 - HS + lane;             // the lane's cell (unwrapped)
  int cw = c % n;
  if (cw < 0) cw += n;
  const bool mine = c >= w0 && c < w1;
  // the cell's place in a buffer: its own block's range with HS cells on each side, or, with one
  // block, the whole field; lanes past the chunk's halo hold a copy that nothing of the chunk reads
  int at = C > 1 ? c - c0 + HS : cw;
  if (at > pitch - 1) at = pitch - 1;
  const int left = rank == 0 ? C - 1 : rank - 1, right = rank + 1 == C ? 0 : rank + 1;
  const int len_left = start_of(left + 1) - start_of(left);
  const bool to_left = C > 1 && mine && c - c0 < HS, to_right = C > 1 && mine && c1 - c <= HS;
  const long long g = static_cast<long long>(e) * n + cw;

  // per-lane constants of the call: the advector of the face right of the cell, G, 1/G of the
  // face, R
  const T v0 = p.gc[g];
  const bool nug = p.G != nullptr;
  const T Gi = nug ? p.G[g] : T(1);
  const T rGb = nug ? fdiv(T(1), T(0.5) * (Gi + down1(Gi))) : T(1);
  const T Ri = p.R ? p.R[g] : T(0);
  const T coef0 = absv(v0) - v0 * v0 * rGb;

  auto donor = [&](T q, T F, T Fm) {
    T t0 = -F, t1 = Fm;
    if (nug) { t0 = -fdiv(F, Gi); t1 = fdiv(Fm, Gi); }
    if (p.kahan) {
      T s = q, comp = T(0);
      kahan_add(s, comp, t0);
      kahan_add(s, comp, t1);
      return s;
    }
    return (q + t0) + t1;
  };
  // one step of this warp's cells
  auto step = [&](T q0) {
    if (p.rhs_b) q0 = q0 + p.dt * Ri;
    const T F0 = flux(q0, down1(q0), v0);
    T q = donor(q0, F0, up1(F0));
    if (p.K > 1) {
      T hi = T(0), lo = T(0);
      if (FCT) {
        const T h = maxv(q0, q), l = minv(q0, q);
        hi = max3(h, up1(h), down1(h));
        lo = min3(l, up1(l), down1(l));
      }
      T V = v0, coef = coef0;
      for (int k = 2; k <= p.K; ++k) {
        if (k > 2) coef = absv(V) - V * V * rGb;
        const T qR = down1(q);
        const T f0 = p.abs ? absv(q) : q, f1 = p.abs ? absv(qR) : qR;
        const T A = IGA ? (f1 - f0) * T(0.5) : ratio(f1 - f0, f0 + f1);
        T out = coef * A;
        if (p.tot) {
          const T fm = up1(f0), f2 = __shfl_down_sync(kFull, f0, 2);
          const T num = ((f2 - f1) - f0) + fm;
          const T D = IGA ? num * T(0.25) : ratio(num, ((f2 + f1) + f0) + fm);
          out = out + ((T(3) * V * absv(V)) * rGb - (T(2) * V * V * V) * (rGb * rGb) - V) * T(1.0 / 3.0) * D;
        }
        const T upw = IGA ? T(1) : (gt0(out) ? q : qR);  // the flux's upwind value
        T Fl;
        if (FCT) {
          const T F = IGA ? out : out * upw;
          const T Fm = up1(F);
          const T in = posp(Fm) - negp(F), ou = posp(F) - negp(Fm);
          T a = posp(hi - q), d = posp(q - lo);
          if (nug) { a = Gi * a; d = Gi * d; }
          const T bu = positive_sum(in) ? fdiv(a, in) : T(1);
          const T bd = positive_sum(ou) ? fdiv(d, ou) : T(1);
          const bool right_ward = gt0(F) || (is_zero(F) && gt0(out));
          const T buR = down1(bu), bdR = down1(bd);
          V = out * min3(T(1), right_ward ? bd : bu, right_ward ? buR : bdR);
          Fl = IGA ? V : V * upw;
        } else {
          V = out;
          Fl = IGA ? out : out * upw;
        }
        q = donor(q, Fl, up1(Fl));
      }
    }
    if (p.rhs_a) q = q + p.dt * Ri;
    return q;
  };
  const T half_dt = T(0.5) * p.dt;
  // psi^n + dt/2 (A psi^n + b) of equation e, from all equations of the cell
  auto before = [&](const T (&x)[kTrapezMax]) {
    T r = T(0), own = T(0);
#pragma unroll
    for (int f = 0; f < kTrapezMax; ++f) {
      if (f < E) {
        r = r + static_cast<T>(p.m.A[e * kTrapezMax + f]) * x[f];
        if (f == e) own = x[f];
      }
    }
    if (p.b) r = r + p.b[g];
    return own + half_dt * r;
  };
  // psi^{n+1} = Minv (psi* + dt/2 b) of every equation, psi* from the buffer
  auto after = [&](const T* from, T (&x)[kTrapezMax]) {
    T y[kTrapezMax];
#pragma unroll
    for (int f = 0; f < kTrapezMax; ++f) {
      y[f] = f < E ? from[f * pitch + at] : T(0);
      if (p.b && f < E) y[f] = y[f] + half_dt * p.b[static_cast<long long>(f) * n + cw];
    }
#pragma unroll
    for (int i = 0; i < kTrapezMax; ++i) {
      T s = T(0);
      if (i < E) {
#pragma unroll
        for (int f = 0; f < kTrapezMax; ++f)
          if (f < E) s = s + static_cast<T>(p.m.Minv[i * kTrapezMax + f]) * y[f];
      }
      x[i] = s;
    }
  };

  // the launch before this one, when launched as its dependent; it wrote psi, not what is read above
  grid_wait();
  T q;
  T x[kTrapezMax];
  if (SYS) {
#pragma unroll
    for (int f = 0; f < kTrapezMax; ++f) x[f] = f < E ? p.psi_in[static_cast<long long>(f) * n + cw] : T(0);
    q = before(x);
  } else {
    q = p.psi_in[g];
  }
  // every block of the cluster has started (its shared memory may be written) and has read psi_in
  // (psi_out may be the same array)
  cluster_sync();
  for (int s = 0, parity = 0; s < p.n_steps; parity ^= 1) {
    const int todo = p.n_steps - s < p.S ? p.n_steps - s : p.S;
    for (int j = 0; j < todo; ++j) q = step(q);
    s += todo;
    if (!SYS && s == p.n_steps) break;
    T* const b = buf + parity * E * pitch;
    if (mine) {
      b[e * pitch + at] = q;
      // the neighbours' halos: the left block holds this range's first cells behind its own, the
      // right block this range's last cells before its own
      if (to_left) remote_store(b + e * pitch + HS + len_left + (c - c0), left, q);
      if (to_right) remote_store(b + e * pitch + HS - (c1 - c), right, q);
    }
    cluster_sync();
    if (SYS) {
      after(b, x);
      if (s < p.n_steps) q = before(x);
    } else {
      q = b[at];
    }
  }
  if (mine) {
    if (SYS) {
      T own = T(0);
#pragma unroll
      for (int f = 0; f < kTrapezMax; ++f)
        if (f == e) own = x[f];
      p.psi_out[g] = own;
    } else {
      p.psi_out[g] = q;
    }
  }
}

// The largest cluster the device can run (a power of two up to kMaxCluster).
template <typename T, bool FCT, bool IGA, bool SYS>
int largest_cluster() {
  static PerDevice<int> of;
  return of.get([](int) {
    auto kern = k_line1d<T, FCT, IGA, SYS>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      cudaGetLastError();
      return 8;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kMaxCluster);
    cfg.blockDim = dim3(32 * kMaxWarps);
    cfg.dynamicSmemBytes = 32 << 10;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kMaxCluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int count = 0;
    if (cudaOccupancyMaxActiveClusters(&count, kern, &cfg) != cudaSuccess || count < 1) {
      cudaGetLastError();
      return 8;
    }
    return kMaxCluster;
  });
}

template <typename T, bool FCT, bool IGA, bool SYS>
int launch_line(LineParams<T> p, bool chained, cudaStream_t st) {
  const int room = 32 - 2 * p.halo;  // cells of its own per warp, one step between exchanges
  if (room < kLeast) return MPDATA_EUNSUPPORTED;
  // the smallest cluster that gives every warp's SM one chunk per equation (more blocks only add
  // barrier latency), else the largest; a range is at least one step's halo long
  const int top = largest_cluster<T, FCT, IGA, SYS>();
  int C = 1;
  while (C < top && (p.n + C - 1) / C > room && p.n / (2 * C) >= p.halo) C *= 2;
  const int most = (p.n + C - 1) / C;
  p.chunks = (most + room - 1) / room;
  if (p.chunks * p.E > kMaxWarps) return MPDATA_EUNSUPPORTED;
  // An FP64 field of many chunks per SM waits for the cluster's FP64 pipes, and the launches of the
  // staged kernels, spread over all SMs, take less: microseconds per step of either, fitted to 50 ..
  // 12000 cells and 1 .. 6 passes (K4 with third-order terms and limiter, 4000 cells 36.7 and 36.4,
  // 6000 cells 55 and 37; two passes with the limiter 10000 cells 10.8 and 12.7).  Systems, whose
  // staged form takes the launches of every equation, and FP32 are faster here at every length.
  if (sizeof(T) == 8 && !SYS) {
    const double passes = p.K - 1, fct = FCT ? 1.0 : 0.0, tot = p.tot ? 1.0 : 0.0;
    const double here = p.chunks * (0.09 + passes * (0.2 + 0.145 * fct + 0.2 * tot));
    if (here > 1.8 + passes * (4.75 + 5.2 * fct + 1.9 * tot)) return MPDATA_EUNSUPPORTED;
  }
  const int u = (most + p.chunks - 1) / p.chunks;
  p.S = 1;
  if (!SYS) {
    const int least = C > 1 ? p.n / C : 1 << 20;  // the halo comes from the adjacent blocks alone
    while (p.S < p.n_steps && u + 2 * p.halo * (p.S + 1) <= 32 && p.halo * (p.S + 1) <= least) ++p.S;
  }
  const size_t smem = sizeof(T) * 2 * p.E * (most + 2 * p.halo * p.S);
  if (smem > (size_t{48} << 10)) return MPDATA_EUNSUPPORTED;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(C));
  cfg.blockDim = dim3(static_cast<unsigned>(32 * p.chunks * p.E));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(C);
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k_line1d<T, FCT, IGA, SYS>, p) == cudaSuccess ? MPDATA_OK : MPDATA_ECUDA;
}

}  // namespace

template <typename T>
int line1d_steps(const Grid& g, const Opts& o, const T* psi_in, T* psi_out, const T* gc, const T* G, const T* R, T dt,
                 int n_steps, const TrapezMat* m, const T* b, bool chained, cudaStream_t st) {
  if (g.nd != 1 || o.dfl || o.open) return MPDATA_EUNSUPPORTED;
  // FP64 |psi| stays on the staged kernels (k_steps1d): the option's step on a positive field is to have
  // the bits of the basic step there (MPDATA_STAGED), and the products here are contracted differently
  if (o.abs && sizeof(T) == 8) return MPDATA_EUNSUPPORTED;
  if (g.N > (1 << 20) || o.n_iters > 64) return MPDATA_EUNSUPPORTED;
  LineParams<T> p{};
  p.n = static_cast<int>(g.N);
  p.n_steps = n_steps;
  p.K = o.n_iters;
  p.E = m ? m->E : 1;
  // cells a pass reaches: pass 1 one; a corrective pass one (its faces' pseudo-advectors), one more
  // with the third-order terms (psi_{i-1} .. psi_{i+2}) and one more with the limiter (the
  // neighbours' factors)
  p.halo = 1 + (p.K - 1) * (1 + (o.tot ? 1 : 0) + (o.fct ? 1 : 0));
  p.tot = o.tot;
  p.kahan = o.kahan;
  p.abs = o.abs;
  p.rhs_a = o.rhs_a;
  p.rhs_b = o.rhs_b;
  p.psi_in = psi_in;
  p.psi_out = psi_out;
  p.gc = gc;
  p.G = o.nug ? G : nullptr;
  p.R = R;
  p.b = b;
  p.dt = dt;
  if (m) {
    p.m = *m;
    if (o.fct) return o.iga ? launch_line<T, true, true, true>(p, chained, st) : launch_line<T, true, false, true>(p, chained, st);
    return o.iga ? launch_line<T, false, true, true>(p, chained, st) : launch_line<T, false, false, true>(p, chained, st);
  }
  if (o.fct) return o.iga ? launch_line<T, true, true, false>(p, chained, st) : launch_line<T, true, false, false>(p, chained, st);
  return o.iga ? launch_line<T, false, true, false>(p, chained, st) : launch_line<T, false, false, false>(p, chained, st);
}

template int line1d_steps<float>(const Grid&, const Opts&, const float*, float*, const float*, const float*,
                                 const float*, float, int, const TrapezMat*, const float*, bool, cudaStream_t);
template int line1d_steps<double>(const Grid&, const Opts&, const double*, double*, const double*, const double*,
                                  const double*, double, int, const TrapezMat*, const double*, bool, cudaStream_t);

}  // namespace mpd
