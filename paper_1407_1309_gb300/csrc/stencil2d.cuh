// Device helpers shared by the fused 2D kernels (fused2d.cu, band2d.cu): the
// donor-cell flux of Eq. 5, the guarded psi-fraction of Eq. 6, the donor update
// of Eq. 4, cp.async wrappers and the lane-neighbour shuffles of a row held as
// NC adjacent columns per lane.
#pragma once

#include <cuda_runtime.h>

namespace mpd {
namespace dev {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ int wrapi(int c, int n) {
  int r = c % n;
  return r < 0 ? r + n : r;
}

template <typename T> __device__ __forceinline__ T fdiv(T a, T b);
// FP32 n / d (2 ulp), also for a d below the smallest normal number: the limiter divides by flux
// sums, which become that small in the tail of a field.
template <> __device__ __forceinline__ float fdiv<float>(float a, float b) { return __fdividef(a, b); }
// Approximate FP32 reciprocal of a divisor known to be normal (the psi-fractions: divisible()), in
// which subnormal numbers are flushed: 0 above 2^126, as __fdividef's quotient is.
__device__ __forceinline__ float rcp_normal(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return r;
}
// Approximate FP32 reciprocal that takes and gives subnormal numbers: of d scaled by a power of two
// into the range of the form above (PTX's rcp.approx.f32 in its place: 256^3 with three passes and
// third-order terms 1086 -> 1100 us per step).
__device__ __forceinline__ float rcp(float d) {
  const float s = fabsf(d) > 1.0f ? 0.25f : 16777216.0f;
  return rcp_normal(d * s) * s;
}

// FP64 n / d for the arithmetic-bound FP64 kernels, five FP64 operations: one Newton-Raphson
// iteration r <- r + r (1 - d r) (quadratic convergence) from the PTX approximate FP64 reciprocal
// (rcp.approx.ftz.f64, full exponent range), and Markstein's remainder correction
// q <- q + r (n - d q) of the quotient: within one unit in the last place of the exact quotient for
// normal operands.  The seed carries about 20 bits, the iterated reciprocal 40, and so does the first
// quotient; the fma rounds its remainder to 53 bits of a correction of relative size 2^-40, so that
// the corrected quotient's error before its last rounding is about 2^-80.  Measured against IEEE
// division: none of 4 10^8 quotients differs, with this form and with a second iteration alike;
// without that the 1024^2 FP64 step takes 215 instead of 242 us.  A zero, infinite or NaN divisor
// gives NaN (the kernels never rely on it: the psi-ratio guards zero sums, and the FCT factors'
// min(1, x) maps the inf or NaN of a zero flux sum to 1 alike).
__device__ __forceinline__ double nr_div(double n, double d) {
  double r0;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r0) : "d"(d));
  const double r = fma(r0, fma(-d, r0, 1.0), r0);
  const double q = n * r;
  return fma(r, fma(-d, q, n), q);
}
template <> __device__ __forceinline__ double fdiv<double>(double a, double b) { return nr_div(a, b); }

template <typename T> __device__ __forceinline__ T posp(T x) { return x > T(0) ? x : T(0); }
template <typename T> __device__ __forceinline__ T negp(T x) { return x < T(0) ? x : T(0); }
template <typename T> __device__ __forceinline__ T absv(T x) { return x < T(0) ? -x : x; }
template <typename T> __device__ __forceinline__ T maxv(T a, T b) { return a > b ? a : b; }
template <typename T> __device__ __forceinline__ T minv(T a, T b) { return a < b ? a : b; }
// FP32: PTX min and max, which return the number where one operand is NaN (the ternary forms have
// to return a particular operand then), and |x|.  The 2D and 3D marches are bound by issue and the
// half-rate ALU pipe that runs comparisons and selections; these forms, the three-value extrema
// below, selected upwind values and the flushing reciprocal of the guarded psi-fractions together,
// measured per step: 4096^2 139 -> 90 us (with the tile heights of lanes2d.h), the compensated
// 1024^2 18.4 -> 13.2 us, the 512-field ensemble 539 -> 402 us, 256^3 with three passes and
// third-order terms 1248 -> 1086 us.
template <> __device__ __forceinline__ float posp<float>(float x) { return fmaxf(x, 0.0f); }
template <> __device__ __forceinline__ float negp<float>(float x) { return fminf(x, 0.0f); }
template <> __device__ __forceinline__ float absv<float>(float x) { return fabsf(x); }
template <> __device__ __forceinline__ float maxv<float>(float a, float b) { return fmaxf(a, b); }
template <> __device__ __forceinline__ float minv<float>(float a, float b) { return fminf(a, b); }
// extrema of three values: PTX's three-operand min and max in FP32
template <typename T> __device__ __forceinline__ T max3(T a, T b, T c) { return maxv(maxv(a, b), c); }
template <typename T> __device__ __forceinline__ T min3(T a, T b, T c) { return minv(minv(a, b), c); }
template <> __device__ __forceinline__ float max3<float>(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
template <> __device__ __forceinline__ float min3<float>(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// min(1, x); a NaN x gives 1 (fmin returns the non-NaN operand)
__device__ __forceinline__ float min1(float x) { return fminf(1.0f, x); }
// FP64, for x >= +0, infinities and NaN: the bits of such values below 1 are unsigned integers below
// those of 1 (fmin would compare on the FP64 pipe)
__device__ __forceinline__ double min1(double x) {
  return static_cast<unsigned long long>(__double_as_longlong(x)) < 0x3FF0000000000000ull ? x : 1.0;
}
// donor-cell flux (Eq. 5) in advector units: [V]+ L + [V]- R, one term of which is zero
template <typename T> __device__ __forceinline__ T flux(T L, T R, T V) { return V * (V > T(0) ? L : R); }
// A divisor the fast divisions can take: not zero and not below the smallest normal number (their
// approximate reciprocals flush such a divisor to zero).  A psi-sum that small counts as zero in
// the guard of the psi-fraction: the fraction it would give changes no flux by more than that.
__device__ __forceinline__ bool divisible(float d) { return fabsf(d) >= 1.17549435e-38f; }
__device__ __forceinline__ bool divisible(double d) { return ((__double_as_longlong(d) >> 52) & 0x7FF) != 0; }

// psi-fraction of Eq. 6 with the zero-denominator guard
template <typename T> __device__ __forceinline__ T ratio(T n, T d) { return divisible(d) ? fdiv(n, d) : T(0); }
template <> __device__ __forceinline__ float ratio<float>(float n, float d) {
  return divisible(d) ? n * rcp_normal(d) : 0.0f;
}

// x > 0 (the upwind choice of a flux, the limiter's direction)
__device__ __forceinline__ bool gt0(float x) { return x > 0.0f; }

// FP64: sign tests, extrema and magnitudes on the integer pipe.  GB300's FP64 pipe runs at a
// small fraction of the FP32 rate and bounds the FP64 step, so the operations that need no
// FP64 arithmetic (comparisons with zero, ordering of two values, |x|) are taken off it.  For
// finite arguments they give the floating-point forms' results, up to the sign of a zero
// result (an ordering key makes -0 < +0).
__device__ __forceinline__ bool gt0(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool lt0(double x) {
  const long long b = __double_as_longlong(x);
  return b < 0 && (b << 1) != 0;
}
__device__ __forceinline__ bool nonzero(double x) { return (__double_as_longlong(x) << 1) != 0; }
// a signed integer in the order of the doubles (finite arguments)
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFLL);
}
template <> __device__ __forceinline__ double posp<double>(double x) { return gt0(x) ? x : 0.0; }
template <> __device__ __forceinline__ double negp<double>(double x) { return lt0(x) ? x : 0.0; }
template <> __device__ __forceinline__ double absv<double>(double x) {
  return __longlong_as_double(__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFLL);
}
template <> __device__ __forceinline__ double maxv<double>(double a, double b) { return order_key(a) > order_key(b) ? a : b; }
template <> __device__ __forceinline__ double minv<double>(double a, double b) { return order_key(a) < order_key(b) ? a : b; }
template <> __device__ __forceinline__ double flux<double>(double L, double R, double V) { return V * (gt0(V) ? L : R); }

// Sums of the inflows [Fm]+ - [Fp]- and of the outflows [Fp]+ - [Fm]- of a 2D cell.  [x]- = x - [x]+ and
// [x]+ = x - [x]- hold exactly in floating point, so in FP32 the outflow sum takes the inflow sum's four
// extrema (adds instead of min/max on the half-rate pipe); FP64 takes its own, which cost integer
// selects and save four operations on the FP64 pipe.  The same bits.
template <typename T>
__device__ __forceinline__ void flow_sums(T Fm0, T Fp0, T Fm1, T Fp1, T& in, T& ou) {
  const T pFm0 = posp(Fm0), nFp0 = negp(Fp0), pFm1 = posp(Fm1), nFp1 = negp(Fp1);
  in = (pFm0 - nFp0) + (pFm1 - nFp1);
  if constexpr (sizeof(T) == 4) ou = ((Fp0 - nFp0) - (Fm0 - pFm0)) + ((Fp1 - nFp1) - (Fm1 - pFm1));
  else ou = (posp(Fp0) - negp(Fm0)) + (posp(Fp1) - negp(Fm1));
}

template <int B>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(src), "n"(B) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

template <typename T>
__device__ __forceinline__ void kahan_add(T& s, T& comp, T t) {
  const T y = t - comp;
  const T u = s + y;
  comp = (u - s) - y;
  s = u;
}

// Donor-cell update of Eq. 4 from the four face fluxes, rG = 1/G.  The flux
// differences are added first and psi last, so only one rounding happens at the
// scale of psi; with the Kahan option the terms psi - Fp0 + Fm0 - Fp1 + Fm1 are
// summed in that order with compensation instead.
template <typename T, bool NUG, bool KAHAN>
__device__ __forceinline__ T donor(T p, T Fp0, T Fm0, T Fp1, T Fm1, T rG) {
  if (KAHAN) {
    if (NUG) {
      Fp0 *= rG;
      Fm0 *= rG;
      Fp1 *= rG;
      Fm1 *= rG;
    }
    T s = p, comp = T(0);
    kahan_add(s, comp, -Fp0);
    kahan_add(s, comp, Fm0);
    kahan_add(s, comp, -Fp1);
    kahan_add(s, comp, Fm1);
    return s;
  }
  const T div = (Fm0 - Fp0) + (Fm1 - Fp1);
  return NUG ? p + div * rG : p + div;
}

// s + t = u + err exactly (Knuth's two-sum, no magnitude condition); s <- u, e += err.
template <typename T>
__device__ __forceinline__ void two_sum_acc(T& s, T& e, T t) {
  const T u = s + t;
  const T bp = u - s;
  const T err = (s - (u - bp)) + (t - bp);
  s = u;
  e = e + err;
}

// Donor-cell update of Eq. 4 on a compensated state psi = hi + lo: the flux divergence of
// the high parts is formed in FP32 as in the plain update (fluxes differenced first), added to
// hi with a two-sum whose rounding error joins lo together with the low parts' own flux
// divergence (lo_div), and the pair is renormalised so that the returned hi is the value of
// the representable sum nearest hi + lo.  The rounding of psi + divergence, at the scale of
// psi, is the one that biases the plain FP32 state over long runs; it is kept exactly.
// lo_div: the divergence of the low parts' own face fluxes (added to lo, scaled by 1/G).
template <typename T, bool NUG>
__device__ __forceinline__ T donor_comp(T p, T lo, T Fp0, T Fm0, T Fp1, T Fm1, T rG, T lo_div, T& lo_out) {
  T div = (Fm0 - Fp0) + (Fm1 - Fp1);
  if (NUG) {
    div *= rG;
    lo_div *= rG;
  }
  const T s = p + div;
  const T bp = s - p;
  const T err = (p - (s - bp)) + (div - bp);
  const T e = (lo + lo_div) + err;
  // renormalise with a full two-sum: after cancellation |e| may exceed |s|
  const T h = s + e;
  const T bq = h - s;
  lo_out = (s - (h - bq)) + (e - bq);
  return h;
}

// A row of NC columns held by one lane; the columns just outside come from the
// neighbouring lanes.
template <typename T, int NC> __device__ __forceinline__ T from_left(const T (&a)[NC]) {
  return __shfl_up_sync(kFull, a[NC - 1], 1);
}
template <typename T, int NC> __device__ __forceinline__ T from_right(const T (&a)[NC]) {
  return __shfl_down_sync(kFull, a[0], 1);
}
template <typename T, int NC> __device__ __forceinline__ T left_of(const T (&a)[NC], int c, T aL) {
  return c == 0 ? aL : a[c > 0 ? c - 1 : 0];
}
template <typename T, int NC> __device__ __forceinline__ T right_of(const T (&a)[NC], int c, T aR) {
  return c == NC - 1 ? aR : a[c < NC - 1 ? c + 1 : NC - 1];
}
template <typename T, int N> __device__ __forceinline__ void copy_row(T (&d)[N], const T (&s)[N]) {
#pragma unroll
  for (int c = 0; c < N; ++c) d[c] = s[c];
}

}  // namespace dev
}  // namespace mpd
