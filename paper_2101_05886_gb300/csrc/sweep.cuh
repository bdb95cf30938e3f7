// sweep.cuh - the directional residual sweep of the free-stream-preserving (FP)
// upwind finite-difference scheme (arXiv 2101.05886, Sec. 3.2), templated on the
// arithmetic type.
//
// One CTA owns a tile of TT lines along the swept direction and marches along
// them in chunks of S faces (S * TT = the CTA's threads, one face per thread), from
// the end of one line straight on to the next line of its work item.  Cells
// enter a shared-memory ring (2S slots per line) once and are reused by every
// face whose stencil covers them; per-cell primitives and spectral radii are
// formed once per cell.  Face fluxes go to a second ring, and each cell's
// residual contribution F'_{i+1/2} - F'_{i-1/2} (Eq. aderivative) is applied in
// the epilogue: written, accumulated, scaled into dQ/dt, or fused into the
// Runge-Kutta stage update.  The work items of a launch are laid out on the host
// (make_items in api.cu), so one launch covers every block of a batch.
//
// Face flux in difference form (Eq. my_point1 with the split of Eq.
// flux_split_detail): with Q* = Q~_{i+1/2}/(1/J)_{i+1/2} (Eq. Q_star, order-M
// interpolation, Remark 3) written as Q* = Q_i + delta,
//   dF_m = (F(Q_m) - F(Q*)) . k_m,  dQ_m = (Q_m - Q*) (1/J)_m      m = i-2..i+3
// are formed directly from the state differences (never as a difference of two
// large fluxes), projected on the Roe left eigenvectors, split with local
// Lax-Friedrichs speeds and reconstructed by WENO5-JS or linear upwind into W.
// The reference face fluxes F~*_{i+-1/2} = F(Q*_{i+-1/2}) . k_{i+-1/2} enter the
// residual of point i through the exact identity
//   F~*_+ - F~*_- = [F(Q*_+) - F(Q*_-)] . k_+ + [F(Q*_-) - F(Qbar)] . (k_+ - k_-)
//                   + F(Qbar) . (k_+ - k_-),
// with Qbar the far-field state and k_+ - k_- formed in FP64 when the metrics
// are built.  Summed over the directions the last term is F(Qbar) times the
// discrete surface-conservation residual (Eq. SCL), zero to round-off for the
// symmetric conservative metrics, and is not formed.  Every remaining term is a
// product with a difference, so FP32 arithmetic keeps its relative accuracy on
// the residual, and a uniform free stream gives exactly zero in either precision.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "fp_internal.h"

namespace fpk {

template <typename T> struct Num;
template <> struct Num<double> {
  // reciprocal of a finite nonzero x: the PTX approximation (relative error about 2^-20) and one
  // step of Householder's third-order iteration, y <- y + y (e + e^2) with e = 1 - x y, which
  // cubes the error (three operations; two Newton-Raphson steps take four): within 2^-53 (1 + 2^-4)
  // of 1/x, as tested
  static __device__ __forceinline__ double rcp(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
  }
  // max(m, |x|), m >= 0, a NaN ignored as by fmax: doubles without sign are ordered like their
  // bits, and integer compares leave the FP64 pipe alone
  static __device__ __forceinline__ double amax(double m, double x) {
    const long long a = __double_as_longlong(m), b = __double_as_longlong(fabs(x));
    return __longlong_as_double(b > a && b <= 0x7ff0000000000000LL ? b : a);
  }
  static __device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
  static __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
  static __device__ __forceinline__ double rsqrt_(double x) { return rsqrt(x); }
  // sqrt(a b): one root of the product, which stays in range up to 1e308
  static __device__ __forceinline__ double sqrt_product(double a, double b) { return sqrt(a * b); }
};
template <> struct Num<float> {
  // the PTX approximate reciprocal (one MUFU operation, max relative error 2^-23);
  // subnormal inputs are flushed, so 1/x of a value below 2^-126 is +-inf
  static __device__ __forceinline__ float rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
  }
  static __device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
  static __device__ __forceinline__ float amax(float m, float x) { return fmaxf(m, fabsf(x)); }
  static __device__ __forceinline__ float sqrt_(float x) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
  }
  static __device__ __forceinline__ float rsqrt_(float x) { return rsqrtf(x); }
  // sqrt(a b) by two roots: c^2 |k|^2 leaves the FP32 range where c |k| passes 1.8e19 (sound speeds
  // in m/s on cells of 1e8 m) though both factors are far inside it
  static __device__ __forceinline__ float sqrt_product(float a, float b) { return sqrt_(a) * sqrt_(b); }
};

// Pairs of values processed by one instruction: packed FP32x2 arithmetic (sm_100+
// FFMA2 / FADD2 / FMUL2) for float, two scalar operations for double.
struct dpair { double x, y; };
template <typename T> struct PairOf;
template <> struct PairOf<float> { using type = float2; };
template <> struct PairOf<double> { using type = dpair; };

__device__ __forceinline__ float2 pmk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ dpair pmk(double a, double b) { return dpair{a, b}; }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ dpair pfma(dpair a, dpair b, dpair c) { return dpair{fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)}; }
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ dpair padd(dpair a, dpair b) { return dpair{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ dpair pmul(dpair a, dpair b) { return dpair{a.x * b.x, a.y * b.y}; }
template <typename P> __device__ __forceinline__ P psub(P a, P b) { return pfma(b, pmk(decltype(a.x)(-1), decltype(a.x)(-1)), a); }
template <typename P> __device__ __forceinline__ P pc(decltype(P::x) v) { return pmk(v, v); }

// Three smoothness indicators (at least 1e-6) divided by the power of two that brings the largest
// below 2^181 if it is above: on their exponents, by integer operations, which leave the FP64 pipe
// alone (96^3 WENO5 FP64 step 21.08 ms with it, 21.07 without).  The weights depend on their quotients only, and
// for a largest one up to 2^511 the products of the squares neither overflow nor all underflow.
// An infinity or NaN stays as it is.
__device__ __forceinline__ void common_scale(double &a, double &b, double &c) {
  const int h = max(max(__double2hiint(a), __double2hiint(b)), __double2hiint(c));
  const int k = h < 0x7ff00000 ? max(h - ((1023 + 180) << 20), 0) & 0x7ff00000 : 0;
  a = __hiloint2double(__double2hiint(a) - k, __double2loint(a));
  b = __hiloint2double(__double2hiint(b) - k, __double2loint(b));
  c = __hiloint2double(__double2hiint(c) - k, __double2loint(c));
}

// WENO5-JS reconstruction of a pair of five-point stencils (the + side and the mirrored - side of
// one characteristic field) in first-difference form; returns the two reconstructed values.
// The stencil values come at half the size of the split values f+-, and 4 times the smoothness
// indicators of that half-size stencil are formed, (second difference)^2 13/3 + (first)^2, one
// operation per square: the same numbers as the indicators of f+-, with the same epsilon.
// FP64: the weights 1/10, 6/10, 3/10 over beta^2 are brought to the common denominator
// beta0^2 beta1^2 beta2^2, one reciprocal instead of four (a reciprocal takes three operations
// of the FP64 pipe, which bounds that sweep).  The numerator, about 6 beta^4.5, would leave the
// range at indicators of 2^227, so common_scale brings large ones down first and the form holds
// like the reciprocals, up to indicators of 2^511 (squares in range).  FP32 takes the reciprocals,
// which run on their own unit: the products would leave the FP32 range at indicators of 4e9.
template <typename T>
__device__ __forceinline__ typename PairOf<T>::type recon5_pair(
    typename PairOf<T>::type v0, typename PairOf<T>::type v1, typename PairOf<T>::type v2,
    typename PairOf<T>::type v3, typename PairOf<T>::type v4) {
  using P = typename PairOf<T>::type;
  // first differences a, b, c, d, two of them negated so that no combination needs a negation
  const P a = psub(v1, v0), nb = psub(v1, v2), c = psub(v3, v2), nd = psub(v3, v4);
  const P d0 = padd(nb, a), d1 = padd(c, nb), d2 = padd(c, nd);  // second differences (signs free)
  const P e0 = pfma(pc<P>(T(3)), nb, a), e1 = psub(c, nb), e2 = pfma(pc<P>(T(3)), c, nd);
  const P r0 = pfma(pc<P>(T(-2)), e0, nb);                       // 6 (q0 - v2) = 5 b - 2 a
  const P r1 = padd(e1, c);                                      // 6 (q1 - v2) = b + 2 c
  const P r2 = padd(e2, c);                                      // 6 (q2 - v2) = 4 c - d
  const P c133 = pc<P>(T(13.0 / 3.0)), eps = pc<P>(T(1.0e-6));
  P b0 = pfma(c133, pmul(d0, d0), pfma(e0, e0, eps));
  P b1 = pfma(c133, pmul(d1, d1), pfma(e1, e1, eps));
  P b2 = pfma(c133, pmul(d2, d2), pfma(e2, e2, eps));
  if constexpr (sizeof(T) == 8) {
    common_scale(b0.x, b1.x, b2.x);
    common_scale(b0.y, b1.y, b2.y);
  }
  const P s0 = pmul(b0, b0), s1 = pmul(b1, b1), s2 = pmul(b2, b2);
  P a0, a1, a2;                                                  // the weights times 10
  if constexpr (sizeof(T) == 8) {
    const P t2 = pmul(pc<P>(T(3)), s0), t1 = pmul(pc<P>(T(6)), s0);
    a0 = pmul(s1, s2);
    a1 = pmul(t1, s2);
    a2 = pmul(t2, s1);
  } else {
    a0 = pmk(Num<T>::rcp(s0.x), Num<T>::rcp(s0.y));
    a1 = pmul(pc<P>(T(6)), pmk(Num<T>::rcp(s1.x), Num<T>::rcp(s1.y)));
    a2 = pmul(pc<P>(T(3)), pmk(Num<T>::rcp(s2.x), Num<T>::rcp(s2.y)));
  }
  const P num = pfma(a2, r2, pfma(a1, r1, pmul(a0, r0)));
  const P den = padd(padd(a0, a1), a2);
  return pfma(pc<P>(T(1.0 / 6.0)), pmul(num, pmk(Num<T>::rcp(den.x), Num<T>::rcp(den.y))), v2);
}

// WENOCU6 (the sixth-order adaptive central-upwind WENO that Remark 2 names) for a pair
// of six-point stencils i-2..i+3, in the first differences a..e of the six values: the
// three upwind parabolic sub-stencils of WENO5 and the downwind {i+1, i+2, i+3}, linear
// weights (1, 9, 9, 1)/20 (the M6 central face value), the downwind stencil judged by the
// six-point indicator beta6 (integral definition; 120960 beta6 below), reference
// tau6 = |beta6 - (beta0 + 4 beta1 + beta2)/6|, alpha_k = d_k (20 + tau6/(beta_k + 1e-40))^2.
// The ratio is capped at 1e18 so that alpha stays finite in FP32; a cap that only binds
// where a sub-stencil is flat to 1e-18 of tau6.
template <typename T>
__device__ __forceinline__ T cu6_ratio(T tau, T beta) {
  if (!(tau > T(0))) return T(0);
  const T r = tau * Num<T>::rcp(beta + T(1.0e-40));   // +inf when the sum is below FP32 range
  return r < T(1.0e18) ? r : T(1.0e18);
}
template <typename T>
__device__ __forceinline__ typename PairOf<T>::type recon6cu_pair(const typename PairOf<T>::type v[6]) {
  using P = typename PairOf<T>::type;
  const P a = psub(v[1], v[0]), b = psub(v[2], v[1]), c = psub(v[3], v[2]);
  const P d = psub(v[4], v[3]), e = psub(v[5], v[4]);
  // 6 (q_k - v2)
  const P r0 = pfma(pc<P>(T(5)), b, pmul(pc<P>(T(-2)), a));
  const P r1 = pfma(pc<P>(T(2)), c, b);
  const P r2 = pfma(pc<P>(T(4)), c, pmul(pc<P>(T(-1)), d));
  const P r3 = pfma(pc<P>(T(2)), e, pfma(pc<P>(T(-5)), d, pmul(pc<P>(T(6)), c)));
  // WENO5 indicators of the three upwind sub-stencils
  const P d0 = psub(b, a), e0 = pfma(pc<P>(T(3)), b, pmul(pc<P>(T(-1)), a));
  const P d1 = psub(c, b), e1 = padd(b, c);
  const P d2 = psub(d, c), e2 = pfma(pc<P>(T(-3)), c, d);
  const P c13 = pc<P>(T(13.0 / 12.0)), q4 = pc<P>(T(0.25));
  const P b0 = pfma(c13, pmul(d0, d0), pmul(q4, pmul(e0, e0)));
  const P b1 = pfma(c13, pmul(d1, d1), pmul(q4, pmul(e1, e1)));
  const P b2 = pfma(c13, pmul(d2, d2), pmul(q4, pmul(e2, e2)));
  // 120960 beta6 as a quadratic form of the differences
  P f = pmul(a, pfma(pc<P>(T(271779)), a, pfma(pc<P>(T(-1837242)), b, pfma(pc<P>(T(2249110)), c,
             pfma(pc<P>(T(-1213142)), d, pmul(pc<P>(T(245620)), e))))));
  f = pfma(b, pfma(pc<P>(T(3544296)), b, pfma(pc<P>(T(-9252940)), c, pfma(pc<P>(T(5189840)), d,
             pmul(pc<P>(T(-1079386)), e)))), f);
  f = pfma(c, pfma(pc<P>(T(6713736)), c, pfma(pc<P>(T(-7947412)), d, pmul(pc<P>(T(1713274)), e))), f);
  f = pfma(d, pfma(pc<P>(T(2534504)), d, pmul(pc<P>(T(-1150710)), e)), f);
  f = pfma(e, pmul(pc<P>(T(139633)), e), f);
  const P b3 = pmul(f, pc<P>(T(1.0 / 120960.0)));
  const P tt = psub(b3, pmul(pc<P>(T(1.0 / 6.0)), pfma(pc<P>(T(4)), b1, padd(b0, b2))));
  const T tx = tt.x < T(0) ? -tt.x : tt.x, ty = tt.y < T(0) ? -tt.y : tt.y;
  const P w0 = padd(pc<P>(T(20)), pmk(cu6_ratio(tx, b0.x), cu6_ratio(ty, b0.y)));
  const P w1 = padd(pc<P>(T(20)), pmk(cu6_ratio(tx, b1.x), cu6_ratio(ty, b1.y)));
  const P w2 = padd(pc<P>(T(20)), pmk(cu6_ratio(tx, b2.x), cu6_ratio(ty, b2.y)));
  const P w3 = padd(pc<P>(T(20)), pmk(cu6_ratio(tx, b3.x), cu6_ratio(ty, b3.y)));
  const P a0 = pmul(pc<P>(T(0.05)), pmul(w0, w0)), a1 = pmul(pc<P>(T(0.45)), pmul(w1, w1));
  const P a2 = pmul(pc<P>(T(0.45)), pmul(w2, w2)), a3 = pmul(pc<P>(T(0.05)), pmul(w3, w3));
  const P num = pfma(a3, r3, pfma(a2, r2, pfma(a1, r1, pmul(a0, r0))));
  const P den = pmul(pc<P>(T(6)), padd(padd(a0, a1), padd(a2, a3)));
  return pfma(num, pmk(Num<T>::rcp(den.x), Num<T>::rcp(den.y)), v[2]);
}

// Seventh-order WENO-JS (four 4-point sub-stencils, optimal weights (1,12,18,4)/35,
// smoothness indicators of the integral definition) for a pair of seven-point stencils,
// written in the first differences d1..d6 of the seven values.
template <typename T>
__device__ __forceinline__ typename PairOf<T>::type recon7_pair(const typename PairOf<T>::type v[7]) {
  using P = typename PairOf<T>::type;
  const P d1 = psub(v[1], v[0]), d2 = psub(v[2], v[1]), d3 = psub(v[3], v[2]);
  const P d4 = psub(v[4], v[3]), d5 = psub(v[5], v[4]), d6 = psub(v[6], v[5]);
  // 12 (q_k - v3)
  const P r0 = pfma(pc<P>(T(13)), d3, pfma(pc<P>(T(-10)), d2, pmul(pc<P>(T(3)), d1)));
  const P r1 = pfma(pc<P>(T(3)), d4, pfma(pc<P>(T(4)), d3, pmul(pc<P>(T(-1)), d2)));
  const P r2 = pfma(pc<P>(T(-1)), d5, pfma(pc<P>(T(6)), d4, d3));
  const P r3 = pfma(pc<P>(T(9)), d4, pfma(pc<P>(T(-4)), d5, d6));
  // 240 beta_k as quadratic forms of the differences
  const P f0 = pfma(d1, pfma(pc<P>(T(547)), d1, pfma(pc<P>(T(-2788)), d2, pmul(pc<P>(T(1854)), d3))),
                    pfma(d2, pfma(pc<P>(T(3708)), d2, pmul(pc<P>(T(-5188)), d3)), pmul(pc<P>(T(2107)), pmul(d3, d3))));
  const P f1 = pfma(d2, pfma(pc<P>(T(267)), d2, pfma(pc<P>(T(-1108)), d3, pmul(pc<P>(T(494)), d4))),
                    pfma(d3, pfma(pc<P>(T(1468)), d3, pmul(pc<P>(T(-1428)), d4)), pmul(pc<P>(T(547)), pmul(d4, d4))));
  const P f2 = pfma(d3, pfma(pc<P>(T(547)), d3, pfma(pc<P>(T(-1428)), d4, pmul(pc<P>(T(494)), d5))),
                    pfma(d4, pfma(pc<P>(T(1468)), d4, pmul(pc<P>(T(-1108)), d5)), pmul(pc<P>(T(267)), pmul(d5, d5))));
  const P f3 = pfma(d4, pfma(pc<P>(T(2107)), d4, pfma(pc<P>(T(-5188)), d5, pmul(pc<P>(T(1854)), d6))),
                    pfma(d5, pfma(pc<P>(T(3708)), d5, pmul(pc<P>(T(-2788)), d6)), pmul(pc<P>(T(547)), pmul(d6, d6))));
  const P i240 = pc<P>(T(1.0 / 240.0)), eps = pc<P>(T(1.0e-6));
  const P b0 = pfma(f0, i240, eps), b1 = pfma(f1, i240, eps), b2 = pfma(f2, i240, eps), b3 = pfma(f3, i240, eps);
  const P s0 = pmul(b0, b0), s1 = pmul(b1, b1), s2 = pmul(b2, b2), s3 = pmul(b3, b3);
  const P a0 = pmul(pc<P>(T(1.0 / 35.0)), pmk(Num<T>::rcp(s0.x), Num<T>::rcp(s0.y)));
  const P a1 = pmul(pc<P>(T(12.0 / 35.0)), pmk(Num<T>::rcp(s1.x), Num<T>::rcp(s1.y)));
  const P a2 = pmul(pc<P>(T(18.0 / 35.0)), pmk(Num<T>::rcp(s2.x), Num<T>::rcp(s2.y)));
  const P a3 = pmul(pc<P>(T(4.0 / 35.0)), pmk(Num<T>::rcp(s3.x), Num<T>::rcp(s3.y)));
  const P num = pfma(a3, r3, pfma(a2, r2, pfma(a1, r1, pmul(a0, r0))));
  const P den = pmul(pc<P>(T(12)), padd(padd(a0, a1), padd(a2, a3)));
  return pfma(num, pmk(Num<T>::rcp(den.x), Num<T>::rcp(den.y)), v[3]);
}

// element `off` of component v of an array whose components are `stride` elements apart (both
// below 2^32, one 32 x 32 + 64 bit multiply-add each)
template <typename T>
__device__ __forceinline__ T *comp_at(T *base, unsigned off, unsigned stride, unsigned v) {
  return reinterpret_cast<T *>(reinterpret_cast<unsigned long long>(base) + (unsigned long long)off * sizeof(T) +
                               (unsigned long long)stride * (v * (unsigned)sizeof(T)));
}

// index of component v of cell `idx` in the state of an RK stage (BlockDev::q) of n cells
__device__ __forceinline__ unsigned long long state_at(int stage, unsigned long long idx, unsigned long long n, int v) {
  return stage && v < 4 ? 4 * idx + v : v * n + idx;
}

// a . b with its fused operations spelled out.  Where a cell is staged (at the start of a work item or
// within one) depends on the layout of the launch, each place is compiled by itself, and a sum of
// two products leaves the compiler the choice of the one that it fuses: linear upwind's results
// differed in the last bit from one layout to another.  So whatever is computed in several places
// (stage_cell, wall_reflect) names its fused operations.
template <typename T>
__device__ __forceinline__ T dot3(T a0, T a1, T a2, T b0, T b1, T b2) {
  return Num<T>::fma_(a2, b2, Num<T>::fma_(a1, b1, a0 * b0));
}

// Slip-wall reflection of a ghost value (the mirror cell's state Q) about the boundary
// face metric fm: m - 2 (m.k) k/|k|^2.
template <typename T>
__device__ __forceinline__ void wall_reflect(T Q[5], const T *fm) {
  const T n0 = fm[0], n1 = fm[1], n2 = fm[2];
  const T s = T(-2) * dot3<T>(Q[1], Q[2], Q[3], n0, n1, n2) / dot3<T>(n0, n1, n2, n0, n1, n2);
  Q[1] = Num<T>::fma_(s, n0, Q[1]);
  Q[2] = Num<T>::fma_(s, n1, Q[2]);
  Q[3] = Num<T>::fma_(s, n2, Q[3]);
}

// Asynchronous global -> shared copies of single elements (sm_80+ cp.async).
template <typename T>
__device__ __forceinline__ void cp_async_el(T *smem, const T *gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  if (sizeof(T) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem));
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem));
}
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem));
}
__device__ __forceinline__ void cp_async8(void *smem, const void *gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem));
}
// copies of four or six neighbouring elements, in the widest pieces that six keep aligned
template <typename T>
__device__ __forceinline__ void cp_async_2el(T *smem, const T *gmem) {
  if (sizeof(T) == 4) cp_async8(smem, gmem); else cp_async16(smem, gmem);
}
template <typename T>
__device__ __forceinline__ void cp_async_4el(T *smem, const T *gmem) {
  cp_async16(smem, gmem);
  if (sizeof(T) == 8) cp_async16(smem + 2, gmem + 2);
}
__device__ __forceinline__ void load4(const float *p, float v[4]) {
  const float4 x = *reinterpret_cast<const float4 *>(p);
  v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void load4(const double *p, double v[4]) {
  const double2 x = *reinterpret_cast<const double2 *>(p), y = *reinterpret_cast<const double2 *>(p + 2);
  v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
}
__device__ __forceinline__ void store4(float *p, const float v[4]) {
  *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store4(double *p, const double v[4]) {
  *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
  *reinterpret_cast<double2 *>(p + 2) = make_double2(v[2], v[3]);
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Weights of the order-M midpoint formula (Sec. 3, Eq. metric_discret), stencil
// i-M/2+1 .. i+M/2 for the face i+1/2.
template <int M> struct MidW;
template <> struct MidW<2> { static __device__ __forceinline__ double w(int m) { return 0.5; } };
template <> struct MidW<4> {
  static __device__ __forceinline__ double w(int m) {
    return (m == 0 || m == 3) ? -1.0 / 12.0 : 7.0 / 12.0;
  }
};
template <> struct MidW<6> {
  static __device__ __forceinline__ double w(int m) {
    return (m == 0 || m == 5) ? 1.0 / 60.0 : (m == 1 || m == 4) ? -8.0 / 60.0 : 37.0 / 60.0;
  }
};
template <> struct MidW<8> {
  static __device__ __forceinline__ double w(int m) {
    return (m == 0 || m == 7) ? -3.0 / 840.0
         : (m == 1 || m == 6) ? 29.0 / 840.0
         : (m == 2 || m == 5) ? -139.0 / 840.0 : 533.0 / 840.0;
  }
};

// [F(B) - F(A)] . k from A's state (velocity uA, momentum mA, energy EA, pressure pA),
// the difference d = B - A, and B's 1/rho and velocity; every term is a product
// with a component of d, so the result carries the relative rounding of d.
template <typename T>
__device__ __forceinline__ void dflux(T g1, T rinvB, const T uB[3], const T uA[3], const T mA[3],
                                      T EA, T pA, const T d[5], const T k[3], T out[5]) {
  T du0 = (d[1] - uA[0] * d[0]) * rinvB;
  T du1 = (d[2] - uA[1] * d[0]) * rinvB;
  T du2 = (d[3] - uA[2] * d[0]) * rinvB;
  T dke = T(0.5) * (d[1] * uB[0] + d[2] * uB[1] + d[3] * uB[2] + mA[0] * du0 + mA[1] * du1 +
                    mA[2] * du2);
  T dp = g1 * (d[4] - dke);
  T UB = uB[0] * k[0] + uB[1] * k[1] + uB[2] * k[2];
  T dU = du0 * k[0] + du1 * k[1] + du2 * k[2];
  out[0] = d[1] * k[0] + d[2] * k[1] + d[3] * k[2];
  out[1] = d[1] * UB + mA[0] * dU + dp * k[0];
  out[2] = d[2] * UB + mA[1] * dU + dp * k[1];
  out[3] = d[3] * UB + mA[2] * dU + dp * k[2];
  out[4] = (d[4] + dp) * UB + (EA + pA) * dU;
}

// dflux of two pairs of states at once.
template <typename P, typename T>
__device__ __forceinline__ void dflux_pair(T g1, P rinvB, const P uB[3], const P uA[3], const P mA[3], P EA, P pA,
                                           const P d[5], const P k[3], P out[5]) {
  P du[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) du[c] = pmul(psub(d[1 + c], pmul(uA[c], d[0])), rinvB);
  P dke = pfma(d[3], uB[2], pfma(d[2], uB[1], pmul(d[1], uB[0])));
#pragma unroll
  for (int c = 0; c < 3; ++c) dke = pfma(mA[c], du[c], dke);
  const P dp = pmul(pc<P>(g1), pfma(pc<P>(T(-0.5)), dke, d[4]));
  const P UB = pfma(uB[2], k[2], pfma(uB[1], k[1], pmul(uB[0], k[0])));
  const P dU = pfma(du[2], k[2], pfma(du[1], k[1], pmul(du[0], k[0])));
  out[0] = pfma(d[3], k[2], pfma(d[2], k[1], pmul(d[1], k[0])));
#pragma unroll
  for (int c = 0; c < 3; ++c) out[1 + c] = pfma(dp, k[c], pfma(mA[c], dU, pmul(d[1 + c], UB)));
  out[4] = pfma(padd(EA, pA), dU, pmul(padd(d[4], dp), UB));
}

// A pair of stencil points B seen from the frame that moves with the reference state's velocity
// V = u* (Galilean frame: momenta m - rho V, energy E - m.V + rho V^2/2).  d = B - Q* comes in the
// laboratory frame and leaves in the moving one, and out = [F(B) - F(Q*)] . k there.  Q* is at
// rest in that frame, so the differences of velocity, kinetic energy and momentum flux lose the
// terms with its momentum (28 operations per point instead of 35, and no velocities of B): with
// z = d_m - V d_0 = rho_B (u_B - V),
//   e = d_E - V.z - V^2/2 d_0,  dp = (gamma-1)(e - z.z/(2 rho_B)),  dU = z.k/rho_B,
//   U_B = u_B.k, V.k = U_B - dU,
//   out = (z.k + d_0 V.k,  z U_B + dp k,  e U_B + (E*+p* + dp) dU),
// every term a product with a component of d, so the result keeps the relative rounding of d.
// V is any fixed number for this: its own rounding cancels.  EpP = E* + p* = p* gamma/(gamma-1).
// With the reconstruction below and the velocities out of the shared ring: 64-block WENO5 step
// 18.04 -> 17.24 ms, 256^3 9.05 -> 8.65 ms, 96^3 FP64 24.5 -> 21.7 ms.
// z.z leaves the FP32 range where momenta differ by more than 1.8e19, and loses digits that count where
// they are below about 1e-16 (densities of 1e-24 kg/m^3).  WIDE forms the velocity differences
// w = z/rho_B first, z.z/rho_B = z.w, dU = w.k, and out[0] = d_0 U_B + rho* dU (rs = rho*): no squares of
// momenta, one operation and three registers more (64-block step 16.27 | 16.52 ms, WENO7 672 |
// 686 us), so the sweeps of ordinary states do without.
template <typename T, bool WIDE>
__device__ __forceinline__ void dflux_frame(T g1, typename PairOf<T>::type rinvB, typename PairOf<T>::type UB,
                                            T rs, const T V[3], T hV2, T EpP, typename PairOf<T>::type d[5],
                                            const typename PairOf<T>::type k[3],
                                            typename PairOf<T>::type out[5]) {
  using P = typename PairOf<T>::type;
#pragma unroll
  for (int c = 0; c < 3; ++c) d[1 + c] = pfma(pc<P>(-V[c]), d[0], d[1 + c]);
#pragma unroll
  for (int c = 0; c < 3; ++c) d[4] = pfma(pc<P>(-V[c]), d[1 + c], d[4]);
  d[4] = pfma(pc<P>(-hV2), d[0], d[4]);
  P zz, dU;                                          // z.z/rho_B, dU
  if constexpr (WIDE) {
    const P w[3] = {pmul(rinvB, d[1]), pmul(rinvB, d[2]), pmul(rinvB, d[3])};
    zz = pfma(d[3], w[2], pfma(d[2], w[1], pmul(d[1], w[0])));
    dU = pfma(w[2], k[2], pfma(w[1], k[1], pmul(w[0], k[0])));
    out[0] = pfma(d[0], UB, pmul(pc<P>(rs), dU));
  } else {
    const P zk = pfma(d[3], k[2], pfma(d[2], k[1], pmul(d[1], k[0])));
    zz = pmul(rinvB, pfma(d[3], d[3], pfma(d[2], d[2], pmul(d[1], d[1]))));
    dU = pmul(rinvB, zk);
    out[0] = pfma(d[0], psub(UB, dU), zk);
  }
  const P dp = pmul(pc<P>(g1), pfma(pc<P>(T(-0.5)), zz, d[4]));
#pragma unroll
  for (int c = 0; c < 3; ++c) out[1 + c] = pfma(dp, k[c], pmul(d[1 + c], UB));
  out[4] = pfma(padd(dp, pc<P>(EpP)), dU, pmul(d[4], UB));
}

// One value of an SSP-RK3 stage (Gottlieb & Shu) in increment form:
// Q^(s+1) = Q^(s) + a_s (Q^n - Q^(s)) + b_s dt L(Q^(s))
template <typename T> struct RkStage {
  T a, bdt;
  bool first;
  __device__ __forceinline__ RkStage(int stage, T dt)
      : a(stage == 1 ? T(0.75) : T(1.0 / 3.0)),
        bdt((stage == 0 ? T(1) : (stage == 1 ? T(0.25) : T(2.0 / 3.0))) * dt), first(stage == 0) {}
  __device__ __forceinline__ T operator()(T qk, const T *qn, T L) const {
    return Num<T>::fma_(bdt, L, first ? qk : Num<T>::fma_(a, *qn - qk, qk));
  }
};

// FIX = 1 or 2: the characteristic decomposition and the FP form on, local Lax-Friedrichs speeds,
// all fixed at compile time (the configuration of the paper's workloads but the shock test), so
// their switches fold away.  FIX = 2 is the same sweep with the alternative CTA shape of
// sweep_threads (fp_internal.h).  FIX = 0: characteristic, the FP form and the speeds read from
// the arguments and the block descriptor.  FIX = 3: component-wise, the others as FIX = 0 (one
// variant for both decompositions held the operands of both and spilled: linear upwind on
// 70 x 80 x 22 points, component-wise, 208 us a step against 149).  FIX = 4: all three read at run
// time, and no squares of momenta (dflux_frame).
template <typename T, int M, int SCHEME, bool BND, int FIX>
__global__ void __launch_bounds__(sweep_threads(sizeof(T) == 4, SCHEME, FIX), sweep_min_ctas(sizeof(T) == 4, SCHEME, FIX))
fp_sweep(const BlockDev *__restrict__ blocks, const SweepItem *__restrict__ items, int mode,
         int stage, const double *__restrict__ dtp, int fpform_arg) {
  // this variant's CTA shape (fp_internal.h): threads, ring stride of a staged field
  constexpr int kThreads = sweep_threads(sizeof(T) == 4, SCHEME, FIX);
  constexpr int kRing = sweep_ring(sizeof(T) == 4, SCHEME, FIX);
  constexpr bool kFold = FIX == 1 || FIX == 2;
  const int charwise = FIX == 3 ? 0 : (FIX == 4 ? !(fpform_arg & 2) : 1);
  const int fpform = kFold ? 1 : (FIX == 4 ? fpform_arg & 1 : fpform_arg);
  // stencil points of a face: i-2..i+3 (5th order) or i-3..i+4 (WENO7), offset index Q0
  constexpr int NS = SCHEME == 2 ? 8 : 6;
  constexpr int Q0 = SCHEME == 2 ? 0 : 1;
  // kEarly: the face ring also takes the lower cell's state and 1/J, so that the epilogue leaves the
  // cell ring alone and the next cells are staged without a barrier after it.  FP32 WENO7 has the
  // registers for it (150 x 141 x 133, M8: 711 -> 698 us a residual); WENO5 spills and loses 1 to 2 %.
  constexpr bool kEarly = sweep_early(sizeof(T) == 4, SCHEME);
  constexpr int kFace = sweep_face_fields(sizeof(T) == 4, SCHEME);
  extern __shared__ __align__(16) unsigned char smraw[];
  T *const sm = reinterpret_cast<T *>(smraw);              // cell ring: kCellFields x kRing
  T *const fr = sm + kCellFields * kRing;                   // face ring: kFace x kRing
  T *const nsb = fr + kFace * kRing;                  // next chunk's cell and face metrics, per thread
  T *const epb = nsb + kNextFields * kThreads;              // epilogue operands, per thread
  const int tid = threadIdx.x;
  // Work-item descriptors in shared memory, double-buffered: during an item's first chunk
  // the next item of this CTA and its whole block descriptor are copied in with cp.async, so an
  // item starts without a chain of dependent global loads, and the chunk loop reads buffer
  // pointers from here rather than through an L1 that the streamed cells keep evicting.
  static_assert(sizeof(BlockDev) % 16 == 0, "descriptor copied in 16-byte pieces");
  constexpr int kDescPieces = (int)(sizeof(BlockDev) / 16);
  __shared__ __align__(16) unsigned char s_desc[2][sizeof(BlockDev)];
  __shared__ __align__(16) SweepItem s_item[2];
  __shared__ T s_dt;
  __shared__ T s_lam[3];                // global Lax-Friedrichs speeds of this item's direction
  auto fetch_desc = [&](int buf, int blk) {
    for (int p = tid; p < kDescPieces; p += kThreads)
      cp_async16(s_desc[buf] + 16 * p, reinterpret_cast<const unsigned char *>(blocks + blk) + 16 * p);
  };
  // this CTA's first item and its descriptor, loaded before the loop
  fetch_desc(0, items[blockIdx.x].block);
  if (tid == 0) s_item[0] = items[blockIdx.x];
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();

  int cur = 0;
  for (int it = blockIdx.x; it >= 0; cur ^= 1) {
    const SweepItem &item = s_item[cur];
    const BlockDev *B = reinterpret_cast<const BlockDev *>(s_desc[cur]);
    const DirDev *D = &B->dir[item.dir];
    const int nit = item.next;
    // the next item: lands by this item's prologue barrier
    if (tid < 2 && nit >= 0) cp_async16(reinterpret_cast<unsigned char *>(&s_item[cur ^ 1]) + 16 * tid,
                                        reinterpret_cast<const unsigned char *>(items + nit) + 16 * tid);
    if (tid == 0) s_dt = mode == MODE_RK ? T(*dtp) : T(0);   // read after the prologue's barrier
    const int S = D->S, TT = D->TT, W = 2 * S;
    // thread roles: along-line index tf and line index tl.  The xi pass puts
    // consecutive threads along the line (coalesced, i contiguous), the other passes
    // across lines.  Shared layout: line-fast slots are TT apart; slot-fast lines 2S apart, with
    // the slots of every other run of 32/S lines turned by S, so that the lines a warp reads at
    // once lie in different banks for every S.
    const bool slotFast = item.dir == 0;
    const int tf = slotFast ? (tid % S) : (tid / TT);
    const int tl = slotFast ? (tid / S) : (tid % TT);
    const int SS = slotFast ? 1 : TT;
    const int lbase = slotFast ? tl * W : tl;
    const int turn = slotFast && S < 32 && (tl & (16 / S)) ? S : 0;
    const int nd = D->nd, nt1 = D->nt1, nt2 = D->nt2;
    const int qsd = D->qsd;
    const unsigned qc = B->qc;
    const int G = B->G;
    // The lines of a tile row are marched as one stream of positions: line after line, each with
    // its G ghost cells at both ends (period P).  `u` is a position within its line (cell
    // x = u - G) and (t1, t2) that line's transverse coordinates.  A chunk may cover the end of
    // one line and the start of the next: 2 G - 1 idle faces between two lines, where whole chunks
    // per line (32 faces along xi) left 15 idle on average, 25 % of the pass for 96 points; and
    // the next line's loads are in flight like any others (xi pass of eight batch blocks, 1.9M
    // points: 124.8 -> 102.4 us, 86.9M -> 73.6M warp instructions).
    const int P = nd + 2 * G;
    // the position w steps after the start of the item's first tile
    auto locate = [&](int w, int &u, int &t1, int &t2) {
      int line = item.tile * TT + tl;
      while (w >= P) { w -= P; line += TT * item.stride; }
      u = w;
      t2 = line / nt1;
      t1 = line - t2 * nt1;
    };
    const int step2 = TT * item.stride / nt1, step1 = TT * item.stride - step2 * nt1;
    const bool shortLines = P < S + 4;   // a step of a chunk can pass more than one line
    auto wrap = [&](int &u, int &t1, int &t2) {
      const bool p = u >= P;
      u -= p ? P : 0;
      t1 += p ? step1 : 0;
      t2 += p ? step2 : 0;
      const bool c = t1 >= nt1;
      t1 -= c ? nt1 : 0;
      t2 += c ? 1 : 0;
      if (shortLines)
#pragma unroll 1
        while (u >= P) {
          u -= P;
          t1 += step1;
          t2 += step2;
          if (t1 >= nt1) { t1 -= nt1; ++t2; }
        }
    };
    const T *__restrict__ qin = static_cast<const T *>(B->q[stage]);
    const int glf = kFold ? 0 : B->global_lf;
    // the block's constants in the arithmetic type: far-field state, its velocity and pressure,
    // gamma - 1, gamma, 1/(gamma - 1)
    const T *const cst = reinterpret_cast<const T *>(B->cst);
    const T g1 = cst[9], gam = cst[10], rg1 = cst[11];

    auto off = [&](int x) -> int {
      const int o = lbase + ((x + turn) & (W - 1)) * SS;
      FPK_CHK_ONLY(if (o < 0 || o >= kRing) { atomicOr(B->status, ST_BOUNDS); return 0; })
      return o;
    };
    // offsets of cell / face x of line (t1, t2) in the state, the ghosted metrics and the face
    // metrics (face x + 1/2): below 2^32
    auto qoff = [&](int x, int t1, int t2) { return (unsigned)t1 * D->qT1 + (unsigned)t2 * D->qT2 + (unsigned)x * qsd; };
    auto moff = [&](int x, int t1, int t2) {
      return B->moff + (unsigned)t1 * D->mT1 + (unsigned)t2 * D->mT2 + (unsigned)x * D->msd;
    };
    auto foff = [&](int x, int t1, int t2) {
      return (unsigned)t1 * D->fT1 + (unsigned)t2 * D->fT2 + (unsigned)(x + 1) * D->fsd;
    };

    // boundary rule of cell index x of line (t1, t2): the source cell (its first component
    // at src, component stride cs), or the far-field state (far); `wall` asks for the
    // momentum to be reflected about the boundary face's normal.  Codes: 0 periodic, 1 far
    // field, 2 zero gradient, 3 slip wall (mirror cell), 4 C-grid cut (mirror cell on the line
    // with t1 reversed, wall outside the cut width), 5 another block of the batch (its cells
    // next to its opposite side, same transverse indices, same RK stage), 6 the caller's halo
    // buffer of that side (the cells another process holds, refreshed for every RK stage).
    // The caller's state and halos hold each component by itself; the stage states (stage > 0) four
    // components side by side and the fifth behind them.  So component v < 4 of a source is at
    // src + v cs, cs = 1 for a stage state, and the fifth at src4.
    auto cell_of = [&](const T *base, unsigned n, unsigned o, const T *&src, const T *&src4, unsigned &cs) {
      src = base + (stage ? 4ULL * o : (unsigned long long)o);
      cs = stage ? 1u : n;
      src4 = comp_at(base, o, n, 4);
    };
    auto bc_source = [&](int x, int t1, int t2, const T *&src, const T *&src4, unsigned &cs, bool &far,
                         bool &wall FPK_CHK_ONLY(, const T *&sb, long long &sn)) {
      cell_of(qin, qc, qoff(x, t1, t2), src, src4, cs);
      far = false; wall = false;
      FPK_CHK_ONLY(sb = qin; sn = 5LL * qc;)
      if ((unsigned)x >= (unsigned)nd) {
        const int hi = x >= 0, bc = hi ? D->bchi : D->bclo;
        if (bc == 1) {
          far = true;
        } else if (BND && bc == 6) {   // halo buffer: index x + G below the line, x - nd above it
          const unsigned o = (unsigned)t1 * D->hT1 + (unsigned)t2 * D->hT2 + (unsigned)(hi ? x - nd : x + G) * D->hsd;
          src = static_cast<const T *>(D->halo[hi]) + o;
          cs = D->hc;
          src4 = comp_at(src, 0, cs, 4);
          FPK_CHK_ONLY(sb = static_cast<const T *>(D->halo[hi]); sn = 5LL * D->hc;)
        } else if (BND && bc == 5) {
          const BlockDev *NB = blocks + D->nbr[hi];
          const DirDev *ND = &NB->dir[item.dir];
          cell_of(static_cast<const T *>(NB->q[stage]), NB->qc,
                  (unsigned)t1 * ND->qT1 + (unsigned)t2 * ND->qT2 + (unsigned)(hi ? x - nd : ND->nd + x) * ND->qsd, src, src4, cs);
          FPK_CHK_ONLY(sb = static_cast<const T *>(NB->q[stage]); sn = 5LL * NB->qc;)
        } else {
          int xx, s1 = t1;
          if (bc == 0) {
            xx = x % nd;
            if (xx < 0) xx += nd;
          } else if (!BND || bc == 2) {
            xx = hi ? nd - 1 : 0;
          } else {
            xx = hi ? 2 * nd - 1 - x : -1 - x;
            const int cw = B->cut;
            if (bc == 4 && (t1 < cw || t1 >= nt1 - cw)) s1 = nt1 - 1 - t1;
            else wall = true;
          }
          cell_of(qin, qc, qoff(xx, s1, t2), src, src4, cs);
        }
      }
    };
    // slip wall: reflect about the boundary face of the line (face -1/2 or nd-1/2)
    auto reflect = [&](int x, int t1, int t2, T Q[5]) {
      const T *const fk = static_cast<const T *>(D->fk);
      wall_reflect<T>(Q, FPK_IN(fk + 6ULL * foff(x < 0 ? -1 : nd - 1, t1, t2), fk, 6LL * D->fc - 5, B->status));
    };

    // global loads of one cell (Q, metric vector, 1/J) with the boundary rule applied
    auto fetch = [&](int x, int t1, int t2, T Q[5], T k[3], T &invJ) {
      if (x >= -G && x < nd + G) {
        const T *const kj = static_cast<const T *>(D->kj);
        T kv[4];
        load4(FPK_IN(kj + 4ULL * moff(x, t1, t2), kj, 4LL * B->mc - 3, B->status), kv);
        k[0] = kv[0]; k[1] = kv[1]; k[2] = kv[2];
        invJ = kv[3];
        const T *qp, *q4;
        unsigned cs;
        bool far, wall;
        FPK_CHK_ONLY(const T *sb; long long sn;)
        bc_source(x, t1, t2, qp, q4, cs, far, wall FPK_CHK_ONLY(, sb, sn));
        if (far) {
#pragma unroll
          for (int v = 0; v < 5; ++v) Q[v] = cst[v];
        } else {
#pragma unroll
          for (int v = 0; v < 4; ++v) Q[v] = *FPK_IN(comp_at(qp, 0, cs, v), sb, sn, B->status);
          Q[4] = *FPK_IN(q4, sb, sn, B->status);
          if (BND && wall) reflect(x, t1, t2, Q);
        }
      } else {   // before the first line of the item: no face of a line uses it
#pragma unroll
        for (int v = 0; v < 5; ++v) Q[v] = cst[v];
        k[0] = T(1); k[1] = T(0); k[2] = T(0);
        invJ = T(1);
      }
    };
    // primitives and spectral radius of a fetched cell into the ring
    auto stage_cell = [&](int x, const T Q[5], const T k[3], T invJ) {
      const T rinv = Num<T>::rcp(Q[0]);
      const T u0 = Q[1] * rinv, u1 = Q[2] * rinv, u2 = Q[3] * rinv;
      const T e = Num<T>::fma_(T(-0.5), dot3<T>(Q[1], Q[2], Q[3], u0, u1, u2), Q[4]);
      const T p = g1 * e;
      const T Jc = Num<T>::rcp(invJ);
      T *cp = sm + off(x);
#pragma unroll
      for (int v = 0; v < 5; ++v) cp[(CF_Q + v) * kRing] = Q[v];
      cp[(CF_K + 0) * kRing] = k[0];
      cp[(CF_K + 1) * kRing] = k[1];
      cp[(CF_K + 2) * kRing] = k[2];
      cp[CF_INVJ * kRing] = invJ;
      cp[CF_RINV * kRing] = rinv;
      cp[CF_H * kRing] = Num<T>::fma_(g1, e, Q[4]) * rinv;
      cp[CF_SQR * kRing] = Num<T>::sqrt_(Q[0]);
      cp[CF_UC * kRing] = Jc * dot3<T>(u0, u1, u2, k[0], k[1], k[2]);
      // |J| c |k|.  The component-wise sweep takes no other square of k, so on it (and in the one for
      // units far from 1) |grad d| = |J k| keeps cells beyond 2^32 or below 2^-32 in the FP32 range
      if constexpr (sizeof(T) == 4 && FIX >= 3) {
        const T gx = Jc * k[0], gy = Jc * k[1], gz = Jc * k[2];
        cp[CF_AC * kRing] = Num<T>::sqrt_product(gam * p * rinv, dot3<T>(gx, gy, gz, gx, gy, gz));
      } else {
        cp[CF_AC * kRing] = fabs(Jc) * Num<T>::sqrt_product(gam * p * rinv, dot3<T>(k[0], k[1], k[2], k[0], k[1], k[2]));
      }
    };

    // asynchronous copy of the metrics of face x + 1/2 of line (t1, t2), and of the change of the face
    // metric over cell x, into staging slot `slot` (0/1, alternating between chunks)
    auto prefetch_face = [&](int x, int t1, int t2, int slot) {
      T *dst = nsb + (9 + 6 * slot) * kThreads + 6 * tid;
      const T *const fk = static_cast<const T *>(D->fk);
      const T *const src = FPK_IN(fk + 6ULL * foff(x, t1, t2), fk, 6LL * D->fc - 5, B->status);
#pragma unroll
      for (int c = 0; c < 6; c += 2) cp_async_2el(dst + c, src + c);
    };
    // asynchronous copy of one cell's loads (-G <= x < nd + G) into this thread's staging slots
    auto prefetch_cell = [&](int x, int t1, int t2) {
      T *const dst = nsb + 4 * tid, *const dst4 = nsb + 4 * kThreads + tid;
      const T *const kj = static_cast<const T *>(D->kj);
      cp_async_4el(nsb + 5 * kThreads + 4 * tid, FPK_IN(kj + 4ULL * moff(x, t1, t2), kj, 4LL * B->mc - 3, B->status));
      const T *qp, *q4;
      unsigned cs;
      bool far, wall;
      FPK_CHK_ONLY(const T *sb; long long sn;)
      bc_source(x, t1, t2, qp, q4, cs, far, wall FPK_CHK_ONLY(, sb, sn));
      if (far) {
#pragma unroll
        for (int v = 0; v < 4; ++v) dst[v] = cst[v];
        *dst4 = cst[4];
      } else {   // a wall ghost copies its mirror cell; the reflection is applied when staged
        if (BND ? cs == 1 : stage != 0) {
          cp_async_4el(dst, FPK_IN(qp, sb, sn - 3, B->status));
        } else {
#pragma unroll
          for (int v = 0; v < 4; ++v) cp_async_el(dst + v, FPK_IN(comp_at(qp, 0, cs, v), sb, sn, B->status));
        }
        cp_async_el(dst4, FPK_IN(q4, sb, sn, B->status));
      }
    };
    // asynchronous copy of the epilogue operands of a cell (state offset qo: residual
    // accumulator, Q^n) into this thread's slots
    auto prefetch_epilogue = [&](unsigned qo) {
      if (mode != MODE_WRITE) {
        const T *const ra = static_cast<const T *>(D->racc);
        cp_async_4el(epb + 4 * tid, FPK_IN(ra + 4ULL * qo, ra, 4LL * qc - 3, B->status));
        cp_async_el(epb + 4 * kThreads + tid, FPK_IN(comp_at(ra, qo, qc, 4), ra, 5LL * qc, B->status));
      }
      if (mode == MODE_RK && stage != 0) {
        const T *const qn = static_cast<const T *>(B->q[0]);
#pragma unroll
        for (int v = 0; v < 5; ++v)
          cp_async_el(epb + (5 + v) * kThreads + tid, FPK_IN(comp_at(qn, qo, qc, v), qn, 5LL * qc, B->status));
      }
    };

    // Within an item, faces and cells are numbered from its first cell (0, at position item.u0):
    // ring slots go by that number.  Chunk ch computes faces a .. a+S-1, a = ch S - 1, and then
    // finishes cells max(a, 0) .. a+S-1.
    const int len = item.len, nch = (len + S) / S;   // faces -1 .. len - 1
    int u, t1, t2;                       // position of this thread's face of the current chunk
    locate(item.u0 - 1 + tf, u, t1, t2);
    // prologue: the first chunk's window, cells [a-4, a+S+4), a = -1, and its faces' metrics
    {
      if (t2 < nt2 && u >= G - 1 && u < nd + G) prefetch_face(u - G, t1, t2, 0);
      cp_async_commit();
      // S >= 8, so the window's S + 8 cells are one per thread plus a second one for the
      // threads tf < 8: both loads are issued before either cell is staged
      int ua, a1, a2, ub2, b1, b2;
      locate(item.u0 - 5 + tf, ua, a1, a2);
      locate(item.u0 - 5 + tf + S, ub2, b1, b2);
      const bool one = a2 < nt2, two = tf < 8 && b2 < nt2;
      chain_wait();                      // from here on: what earlier kernels wrote
      if (sizeof(T) == 4) chain_next();
      if (!kFold && tid == 0 && B->global_lf)
        for (int c = 0; c < 3; ++c)
          s_lam[c] = *FPK_IN(static_cast<const T *>(B->lamg) + (3 * item.dir + c), static_cast<const T *>(B->lamg), 9, B->status);
      T Qa[5], ka[3], ija, Qb[5], kb[3], ijb;
      if (one) fetch(ua - G, a1, a2, Qa, ka, ija);
      if (two) fetch(ub2 - G, b1, b2, Qb, kb, ijb);
      if (one) stage_cell(-5 + tf, Qa, ka, ija);
      if (two) stage_cell(-5 + tf + S, Qb, kb, ijb);
    }
    cp_async_wait_all();
    __syncthreads();

    for (int ch = 0; ch < nch; ++ch) {
      const int a = ch * S - 1;                      // first face of the chunk
      const bool more = ch + 1 < nch;
      // this thread's face u - G + 1/2 and cell u - G of line (t1, t2)
      const bool faceOK = t2 < nt2 && u >= G - 1 && u < nd + G && a + tf < len;
      const bool cellOK = faceOK && u >= G && (ch > 0 || tf > 0);
      const unsigned qo = qoff(u - G, t1, t2);       // the cell's offset in the state
      // ---- start the loads this chunk's epilogue and the next chunk need
      if (cellOK) prefetch_epilogue(qo);
      bool stageOK = false;
      if (more) {
        u += S;                                      // this thread's face of the next chunk
        wrap(u, t1, t2);
        if (t2 < nt2 && u >= G - 1 && u < nd + G) prefetch_face(u - G, t1, t2, (ch + 1) & 1);
        int uc = u + 4, c1 = t1, c2 = t2;            // the cell it stages for the next chunk
        wrap(uc, c1, c2);
        stageOK = c2 < nt2 && a + S + tf < len;
        if (stageOK) prefetch_cell(uc - G, c1, c2);
      }
      if (ch == 0 && nit >= 0) fetch_desc(cur ^ 1, s_item[cur ^ 1].block);   // next item's descriptor
      // opaque: the compiler otherwise splits the chunk by these conditions and spills 250 bytes
      int staged = stageOK;
      asm volatile("" : "+r"(staged));
      cp_async_commit();
      // ---- one face per thread: face ff + 1/2 between cells ff and ff+1
      const int ff = a + tf;
      // the face's flux and reference-state increment, kept for the epilogue, its metric and cell
      // ff's state (kept by linear upwind, whose face leaves the registers for it)
      constexpr bool kOwn = SCHEME == 1 && sizeof(T) == 4;
      T F[5], dl[5], kf[3], Qi[5];
      if (faceOK) {
        int o[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) o[q] = off(ff - 3 + q);
#define CELL(field, q) sm[(field) * kRing + o[(q)]]
#pragma unroll
        for (int v = 0; v < 5; ++v) { Qi[v] = CELL(CF_Q + v, 3); dl[v] = T(0); }
        // face metric of this face, staged by the previous chunk (or the prologue)
#pragma unroll
        for (int c = 0; c < 3; ++c) kf[c] = nsb[(9 + 6 * (ch & 1)) * kThreads + 6 * tid + c];

        if (kEarly && mode >= MODE_RHS) fr[15 * kRing + o[3]] = CELL(CF_INVJ, 3);

        // reference face state Q* = Q_i + delta (Eqs. Q_star, QdJ_star, 1dJ at order M)
        using P = typename PairOf<T>::type;
        // The cells q = kQlo .. kQlo + M - 1 of the weighted sum are taken in mirror pairs
        // (kQlo + m, kQlo + M - 1 - m), m < M/2, whose weights are equal, two cells per packed
        // instruction.  These are the stencil loops' pairs (q, 7 - q) of the same cells, so linear
        // upwind with the switches folded keeps the pairs' Q_q - Q_i and (1/J)_q for its stencil
        // differences instead of loading and subtracting them again.
        constexpr bool kKeep = SCHEME == 1 && kFold;
        constexpr int kQlo = 3 - M / 2 + 1;
        P dqk[4][5], ijk[4];
        if (fpform) {
          P acc[5];
#pragma unroll
          for (int v = 0; v < 5; ++v) acc[v] = pc<P>(T(0));
          P wsum = pc<P>(T(0));
#pragma unroll
          for (int m = 0; m < M / 2; ++m) {
            const int q = kQlo + m, q2 = kQlo + M - 1 - m;
            const P ij = pmk(CELL(CF_INVJ, q), CELL(CF_INVJ, q2));
            const P w = pmul(pc<P>(T(MidW<M>::w(m))), ij);
            wsum = padd(wsum, w);
            if (kKeep) ijk[m] = ij;
#pragma unroll
            for (int v = 0; v < 5; ++v) {
              const P dq = psub(pmk(CELL(CF_Q + v, q), CELL(CF_Q + v, q2)), pc<P>(Qi[v]));
              if (kKeep) dqk[m][v] = dq;
              acc[v] = pfma(w, dq, acc[v]);
            }
          }
          const T wi = Num<T>::rcp(wsum.x + wsum.y);
#pragma unroll
          for (int v = 0; v < 5; ++v) dl[v] = (acc[v].x + acc[v].y) * wi;
        }
        // the frame of the face: velocity V = u* (0 for the plain scheme), see dflux_frame
        T V[3] = {T(0), T(0), T(0)}, hV2 = T(0), EpP = T(0), rhos = T(0);
        if (fpform) {
          T Qs[5];
#pragma unroll
          for (int v = 0; v < 5; ++v) Qs[v] = Qi[v] + dl[v];
          rhos = Qs[0];
          const T rinvs = Num<T>::rcp(rhos);
#pragma unroll
          for (int c = 0; c < 3; ++c) V[c] = Qs[1 + c] * rinvs;
          hV2 = T(0.5) * (V[0] * V[0] + V[1] * V[1] + V[2] * V[2]);
          EpP = gam * (Qs[4] - Qs[0] * hV2);            // p* gamma/(gamma-1)
        }

        // Lax-Friedrichs speeds: local (max over the stencil cells i-2..i+3) or global
        T lm = T(0), l0 = T(0), lp = T(0);
        if (glf) {
          lm = s_lam[0]; l0 = s_lam[1]; lp = s_lam[2];
        } else {
#pragma unroll
          for (int q = Q0; q < Q0 + NS; ++q) {
            const T U = CELL(CF_UC, q), ac = CELL(CF_AC, q);
            lm = Num<T>::amax(lm, U - ac);
            l0 = Num<T>::amax(l0, U);
            lp = Num<T>::amax(lp, U + ac);
          }
        }
        T lam[5];
        if (charwise) {
          lam[0] = lm; lam[1] = l0; lam[2] = l0; lam[3] = l0; lam[4] = lp;
        } else {
          const T lmax = fmax(lm, lp);
          lam[0] = lam[1] = lam[2] = lam[3] = lam[4] = lmax;
        }

        // Roe average of cells i, i+1 and eigenvector basis in the face normal
        const T rl = CELL(CF_SQR, 3), rr = CELL(CF_SQR, 4);
        const T rs = Num<T>::rcp(rl + rr);
        // sqrt(rho) u = (rho u) sqrt(rho)/rho
        const T ml = rl * CELL(CF_RINV, 3) * rs, mr = rr * CELL(CF_RINV, 4) * rs;
        T u[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) u[c] = ml * Qi[1 + c] + mr * CELL(CF_Q + 1 + c, 4);
        const T H = (rl * CELL(CF_H, 3) + rr * CELL(CF_H, 4)) * rs;
        const T c2 = g1 * (H - T(0.5) * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]));
        const T csi = Num<T>::rsqrt_(c2), cs = c2 * csi;
        // from here on velocities are those in the frame of the face (w = u - V)
#pragma unroll
        for (int c = 0; c < 3; ++c) u[c] -= V[c];
        const T hq2 = T(0.5) * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
        const T bb = g1 * csi * csi;
        const T knr = Num<T>::rsqrt_(kf[0] * kf[0] + kf[1] * kf[1] + kf[2] * kf[2]);
        const T n[3] = {kf[0] * knr, kf[1] * knr, kf[2] * knr};
        // first tangent, normalised: e_z x n where n is far from e_z, else n x e_x.  Chosen by
        // selects (faster for linear upwind, WENO7 and component-wise WENO5), except in the
        // folded WENO5 sweep, where the selects cost registers, and in WENOCU6: there a branch
        // measured faster.
        T t1[3], t2[3];
        const bool lowz = n[2] * n[2] <= T(0.5);
        if constexpr ((SCHEME == 0 && kFold) || SCHEME == 3) {
          if (lowz) {
            const T s = Num<T>::rsqrt_(n[0] * n[0] + n[1] * n[1]);
            t1[0] = -n[1] * s; t1[1] = n[0] * s; t1[2] = T(0);
          } else {
            const T s = Num<T>::rsqrt_(n[1] * n[1] + n[2] * n[2]);
            t1[0] = T(0); t1[1] = n[2] * s; t1[2] = -n[1] * s;
          }
        } else {
          const T s = Num<T>::rsqrt_(lowz ? n[0] * n[0] + n[1] * n[1] : n[1] * n[1] + n[2] * n[2]);
          t1[0] = lowz ? -n[1] * s : T(0);
          t1[1] = (lowz ? n[0] : n[2]) * s;
          t1[2] = lowz ? T(0) : -n[1] * s;
        }
        t2[0] = n[1] * t1[2] - n[2] * t1[1];
        t2[1] = n[2] * t1[0] - n[0] * t1[2];
        t2[2] = n[0] * t1[1] - n[1] * t1[0];
        const T Un = u[0] * n[0] + u[1] * n[1] + u[2] * n[2];
        const T ut1 = u[0] * t1[0] + u[1] * t1[1] + u[2] * t1[2];
        const T ut2 = u[0] * t2[0] + u[1] * t2[1] + u[2] * t2[2];
        // the left-eigenvector rows, scaled by kRow: the 1/2 of the Lax-Friedrichs split folded in,
        // and for WENO5 another 1/2 (see recon5_pair)
        constexpr T kRow = SCHEME == 0 ? T(0.25) : T(0.5);
        const T qbb = kRow * T(0.5) * bb, qcs = kRow * T(0.5) * csi;
        const T h1[3] = {kRow * t1[0], kRow * t1[1], kRow * t1[2]};
        const T h2[3] = {kRow * t2[0], kRow * t2[1], kRow * t2[2]};
        const T hut1 = kRow * ut1, hut2 = kRow * ut2;

        // kRow l_s . d for the five characteristic fields
        auto project = [&](const T d[5], T c[5]) {
          if (!charwise) {
#pragma unroll
            for (int v = 0; v < 5; ++v) c[v] = kRow * d[v];
            return;
          }
          const T X4 = qbb * (hq2 * d[0] - (u[0] * d[1] + u[1] * d[2] + u[2] * d[3]) + d[4]);
          const T Y4 = (Un * d[0] - (n[0] * d[1] + n[1] * d[2] + n[2] * d[3])) * qcs;
          c[0] = X4 + Y4;
          c[1] = kRow * d[0] - T(2) * X4;
          c[2] = h1[0] * d[1] + h1[1] * d[2] + h1[2] * d[3] - hut1 * d[0];
          c[3] = h2[0] * d[1] + h2[1] * d[2] + h2[2] * d[3] - hut2 * d[0];
          c[4] = X4 - Y4;
        };

        // the same projection of two stencil points at once (the rows are the face's)
        auto project_pair = [&](const P d[5], P c[5]) {
          if (!charwise) {
#pragma unroll
            for (int v = 0; v < 5; ++v) c[v] = pmul(pc<P>(kRow), d[v]);
            return;
          }
          const P ud = pfma(pc<P>(u[0]), d[1], pfma(pc<P>(u[1]), d[2], pmul(pc<P>(u[2]), d[3])));
          const P X4 = pmul(pc<P>(qbb), pfma(pc<P>(hq2), d[0], psub(d[4], ud)));
          const P nd = pfma(pc<P>(n[0]), d[1], pfma(pc<P>(n[1]), d[2], pmul(pc<P>(n[2]), d[3])));
          const P Y4 = pmul(pc<P>(qcs), psub(pmul(pc<P>(Un), d[0]), nd));
          c[0] = padd(X4, Y4);
          c[1] = pfma(pc<P>(T(-2)), X4, pmul(pc<P>(kRow), d[0]));
          c[2] = pfma(pc<P>(h1[0]), d[1], pfma(pc<P>(h1[1]), d[2], pfma(pc<P>(h1[2]), d[3], pmul(pc<P>(-hut1), d[0]))));
          c[3] = pfma(pc<P>(h2[0]), d[1], pfma(pc<P>(h2[1]), d[2], pfma(pc<P>(h2[2]), d[3], pmul(pc<P>(-hut2), d[0]))));
          c[4] = psub(X4, Y4);
        };

        // a flux in the frame of the face, seen from the laboratory
        auto to_lab = [&](P f[5]) {
          f[4] = pfma(pc<P>(hV2), f[0], f[4]);
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            f[4] = pfma(pc<P>(V[c]), f[1 + c], f[4]);
            f[1 + c] = pfma(pc<P>(V[c]), f[0], f[1 + c]);
          }
        };
        // h: the back-projected characteristic part of the face flux, cen: the part added
        // to it outside the projection (linear upwind only)
        T h[5], cen[5] = {T(0), T(0), T(0), T(0), T(0)};
        if constexpr (SCHEME == 1) {
          // Linear upwind (Eq. linear_upwind; Appendix Eq. new_form_linear_upwind) is linear in
          // the split values and the speeds are constant over the stencil, so the projection
          // commutes with the reconstruction:
          //   sum_s r_s [W+(f+_s) + W-(f-_s)] = C6(dF) + R Lambda L D(dQ~),
          // C6 = (1, -8, 37, 37, -8, 1)/60 (half the sum of the two upwind stencils) and
          // D = (1, -5, 10, -10, 5, -1)/60 (half their difference) over i-2..i+3.  One
          // projection per face instead of two per stencil point; dF and dQ~ = dQ (1/J)_m as
          // in the WENO branch (stencil point s paired with its mirror 5-s).
          constexpr T c6[3] = {T(1.0 / 60.0), T(-8.0 / 60.0), T(37.0 / 60.0)};
          constexpr T d5[3] = {T(1.0 / 60.0), T(-5.0 / 60.0), T(10.0 / 60.0)};
          P cenp[5], disp[5];
#pragma unroll
          for (int v = 0; v < 5; ++v) cenp[v] = disp[v] = pc<P>(T(0));
#pragma unroll
          for (int s = 0; s < 3; ++s) {
            const int q = s + 1, q2 = 6 - s;
            P dp[5], out[5];
            // the weighted sum's pair of these two cells, if it has one (every pair at M6 and M8)
            const int km = q - kQlo;
            const bool kept = kKeep && km >= 0;
            const int kmi = kept ? km : 0;
            const P ijp = kept ? ijk[kmi] : pmk(CELL(CF_INVJ, q), CELL(CF_INVJ, q2));
            const P rip = pmk(CELL(CF_RINV, q), CELL(CF_RINV, q2));
            if (fpform) {
              P kp2[3];
#pragma unroll
              for (int v = 0; v < 5; ++v)
                dp[v] = kept ? psub(dqk[kmi][v], pc<P>(dl[v]))
                             : psub(psub(pmk(CELL(CF_Q + v, q), CELL(CF_Q + v, q2)), pc<P>(Qi[v])), pc<P>(dl[v]));
#pragma unroll
              for (int c = 0; c < 3; ++c) kp2[c] = pmk(CELL(CF_K + c, q), CELL(CF_K + c, q2));
              const P UBp = pmul(pmk(CELL(CF_UC, q), CELL(CF_UC, q2)), ijp);
              const P dlab[3] = {dp[1], dp[2], dp[3]};
              const P elab = dp[4];
              dflux_frame<T, FIX == 4>(g1, rip, UBp, rhos, V, hV2, EpP, dp, kp2, out);
              if (!charwise) {       // the components are those of the laboratory frame
                to_lab(out);
                dp[1] = dlab[0]; dp[2] = dlab[1]; dp[3] = dlab[2]; dp[4] = elab;
              }
            } else {
              // plain scheme: F~_m and Q~_m themselves
              P uBp[3], kp2[3];
#pragma unroll
              for (int v = 0; v < 5; ++v) dp[v] = pmk(CELL(CF_Q + v, q), CELL(CF_Q + v, q2));
#pragma unroll
              for (int c = 0; c < 3; ++c) {
                kp2[c] = pmk(CELL(CF_K + c, q), CELL(CF_K + c, q2));
                uBp[c] = pmul(dp[1 + c], rip);
              }
              const P ke = pfma(dp[3], uBp[2], pfma(dp[2], uBp[1], pmul(dp[1], uBp[0])));
              const P pm = pmul(pc<P>(g1), pfma(pc<P>(T(-0.5)), ke, dp[4]));
              const P U = pfma(uBp[2], kp2[2], pfma(uBp[1], kp2[1], pmul(uBp[0], kp2[0])));
              out[0] = pmul(dp[0], U);
#pragma unroll
              for (int c = 0; c < 3; ++c) out[1 + c] = pfma(pm, kp2[c], pmul(dp[1 + c], U));
              out[4] = pmul(padd(dp[4], pm), U);
            }
            const P ds = pmk(d5[s], -d5[s]);
#pragma unroll
            for (int v = 0; v < 5; ++v) {
              cenp[v] = pfma(pc<P>(c6[s]), out[v], cenp[v]);
              disp[v] = pfma(ds, pmul(dp[v], ijp), disp[v]);
            }
          }
          T dis[5];
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            cen[v] = cenp[v].x + cenp[v].y;
            dis[v] = disp[v].x + disp[v].y;
          }
          // lambda_s l_s . D (project() carries the 1/2 of the split: twice its rows)
          T c[5];
          project(dis, c);
#pragma unroll
          for (int v = 0; v < 5; ++v) h[v] = lam[v] * c[v] * T(1 / kRow);
        } else {
          // split stencil values f+/- for the NS stencil points
          T fpl[NS][5], fmi[NS][5];
          // f+- = (1/2) l.(dF +- lambda d (1/J)_m) of one stencil point
          auto split_point = [&](int s, const T dF[5], const T d[5], T ijm) {
            T cF[5], cD[5];
            project(dF, cF);
            project(d, cD);
            const T mu0 = lam[0] * ijm, mu1 = lam[1] * ijm, mu4 = lam[4] * ijm;
            const T mu[5] = {mu0, mu1, mu1, mu1, mu4};
#pragma unroll
            for (int v = 0; v < 5; ++v) {
              fpl[s][v] = cF[v] + mu[v] * cD[v];
              fmi[s][v] = cF[v] - mu[v] * cD[v];
            }
          };
          if (fpform) {
            // reference-state differences of the stencil points two at a time (packed): points
            // s and its mirror NS-1-s, whose f+ and f- are the (+, -) lanes of the reconstruction
            // pair s; the mirror pair NS-1-s is formed lane by lane
            const P lpm[3] = {pmk(lam[0], -lam[0]), pmk(lam[1], -lam[1]), pmk(lam[4], -lam[4])};
#pragma unroll
            for (int s = 0; s < NS / 2; ++s) {
              const int mir = NS - 1 - s;
              const int q = s + Q0, q2 = mir + Q0;
              P dp[5], kp2[3], out[5];
#pragma unroll
              for (int v = 0; v < 5; ++v)
                dp[v] = psub(psub(pmk(CELL(CF_Q + v, q), CELL(CF_Q + v, q2)), pc<P>(Qi[v])), pc<P>(dl[v]));
#pragma unroll
              for (int c = 0; c < 3; ++c) kp2[c] = pmk(CELL(CF_K + c, q), CELL(CF_K + c, q2));
              const P ijp = pmk(CELL(CF_INVJ, q), CELL(CF_INVJ, q2));
              const P UBp = pmul(pmk(CELL(CF_UC, q), CELL(CF_UC, q2)), ijp);
              const P dlab[3] = {dp[1], dp[2], dp[3]};
              const P elab = dp[4];
              dflux_frame<T, FIX == 4>(g1, pmk(CELL(CF_RINV, q), CELL(CF_RINV, q2)), UBp, rhos, V, hV2, EpP, dp, kp2, out);
              if (!charwise) {       // the components are those of the laboratory frame
                to_lab(out);
                dp[1] = dlab[0]; dp[2] = dlab[1]; dp[3] = dlab[2]; dp[4] = elab;
              }
              P cF[5], cD[5];
              project_pair(out, cF);
              project_pair(dp, cD);
              // (lambda (1/J)_s, -lambda (1/J)_mirror) for the three speed classes
              const P mp[3] = {pmul(lpm[0], ijp), pmul(lpm[1], ijp), pmul(lpm[2], ijp)};
#pragma unroll
              for (int v = 0; v < 5; ++v) {
                const P &mv = mp[v == 0 ? 0 : (v == 4 ? 2 : 1)];
                const P r = pfma(mv, cD[v], cF[v]);                 // (f+ of s, f- of the mirror)
                fpl[s][v] = r.x;
                fmi[mir][v] = r.y;
                fmi[s][v] = cF[v].x - mv.x * cD[v].x;
                fpl[mir][v] = cF[v].y - mv.y * cD[v].y;
              }
            }
          } else {
            // plain scheme: F~_m and Q~_m themselves
#pragma unroll
            for (int s = 0; s < NS; ++s) {
              const int q = s + Q0;
              T dF[5], d[5];
              const T km[3] = {CELL(CF_K, q), CELL(CF_K + 1, q), CELL(CF_K + 2, q)};
#pragma unroll
              for (int v = 0; v < 5; ++v) d[v] = CELL(CF_Q + v, q);
              const T ri = CELL(CF_RINV, q);
              const T uB[3] = {d[1] * ri, d[2] * ri, d[3] * ri};
              const T pm = g1 * (d[4] - T(0.5) * (d[1] * uB[0] + d[2] * uB[1] + d[3] * uB[2]));
              const T U = uB[0] * km[0] + uB[1] * km[1] + uB[2] * km[2];
              dF[0] = d[0] * U;
              dF[1] = d[1] * U + pm * km[0];
              dF[2] = d[2] * U + pm * km[1];
              dF[3] = d[3] * U + pm * km[2];
              dF[4] = (d[4] + pm) * U;
              split_point(s, dF, d, CELL(CF_INVJ, q));
            }
          }
#undef CELL
          // reconstruct each field from both sides (the - side mirrored) and back-project
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            if constexpr (SCHEME == 2) {
              P w7[7];
#pragma unroll
              for (int t = 0; t < 7; ++t) w7[t] = pmk(fpl[t][v], fmi[7 - t][v]);   // i-3..i+3 / i+4..i-2
              const P r = recon7_pair<T>(w7);
              h[v] = r.x + r.y;
            } else if constexpr (SCHEME == 3) {
              P w6[6];
#pragma unroll
              for (int t = 0; t < 6; ++t) w6[t] = pmk(fpl[t][v], fmi[5 - t][v]);   // i-2..i+3 / i+3..i-2
              const P r = recon6cu_pair<T>(w6);
              h[v] = r.x + r.y;
            } else {
              const P r = recon5_pair<T>(pmk(fpl[0][v], fmi[5][v]), pmk(fpl[1][v], fmi[4][v]),
                                                 pmk(fpl[2][v], fmi[3][v]), pmk(fpl[3][v], fmi[2][v]),
                                                 pmk(fpl[4][v], fmi[1][v]));
              h[v] = r.x + r.y;
            }
          }
        }
        if (charwise) {
          // in the frame of the face; H' = c^2/(gamma-1) + w^2/2
          const T sa = h[0] + h[4], da = cs * (h[4] - h[0]), s1 = sa + h[1];
          F[0] = s1;
#pragma unroll
          for (int c = 0; c < 3; ++c) F[1 + c] = u[c] * s1 + n[c] * da + t1[c] * h[2] + t2[c] * h[3];
          F[4] = c2 * rg1 * sa + hq2 * s1 + Un * da + ut1 * h[2] + ut2 * h[3];
        } else {
#pragma unroll
          for (int v = 0; v < 5; ++v) F[v] = h[v];
        }
        if constexpr (SCHEME == 1) {
#pragma unroll
          for (int v = 0; v < 5; ++v) F[v] += cen[v];
        }
        if (SCHEME == 0)             // WENO5 works on half-size values (kRow)
#pragma unroll
          for (int v = 0; v < 5; ++v) F[v] += F[v];
        if (charwise && fpform) {    // back to the laboratory frame: E += V.m + V^2/2 rho, m += V rho
          F[4] += V[0] * F[1] + V[1] * F[2] + V[2] * F[3] + hV2 * F[0];
#pragma unroll
          for (int c = 0; c < 3; ++c) F[1 + c] += V[c] * F[0];
        }
        T *fp = fr + off(ff);
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          fp[v * kRing] = F[v];
          fp[(5 + v) * kRing] = dl[v];
          if (kEarly) fp[(10 + v) * kRing] = Qi[v];
        }
      }
      cp_async_wait_all();
      __syncthreads();
      // ---- residual of cell x = a + tf from its two faces (the upper one is this thread's own),
      // then the epilogue
      if (cellOK) {
        const int oxm = off(ff - 1);
        if constexpr (!kOwn) {                       // loaded again rather than held over the face's arithmetic
          const int ox = off(ff);
#pragma unroll
          for (int v = 0; v < 5; ++v) Qi[v] = kEarly ? fr[(10 + v) * kRing + ox] : sm[(CF_Q + v) * kRing + ox];
#pragma unroll
          for (int c = 0; c < 3; ++c) kf[c] = nsb[(9 + 6 * (ch & 1)) * kThreads + 6 * tid + c];
        }
        T R[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) R[v] = F[v] - fr[v * kRing + oxm];
        if (fpform) {
          // reference states of the two faces: Q*_+ = Q_x + delta_+, Q*_- = Q_{x-1} + delta_-
          T Qp[5], Qm[5], dQ[5], dqm[5], qb[5];
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            qb[v] = cst[v];
            const T qx1 = kEarly ? fr[(10 + v) * kRing + oxm] : sm[(CF_Q + v) * kRing + oxm], dm = fr[(5 + v) * kRing + oxm];
            Qp[v] = Qi[v] + dl[v];
            Qm[v] = qx1 + dm;
            dQ[v] = (Qi[v] - qx1) + (dl[v] - dm);
            dqm[v] = (qx1 - qb[v]) + dm;
          }
          const T ub[3] = {cst[5], cst[6], cst[7]}, pb = cst[8];
          const T rA = Num<T>::rcp(Qm[0]);
          const T uA[3] = {Qm[1] * rA, Qm[2] * rA, Qm[3] * rA};
          const T pA = g1 * (Qm[4] - T(0.5) * (Qm[1] * uA[0] + Qm[2] * uA[1] + Qm[3] * uA[2]));
          const T mA[3] = {Qm[1], Qm[2], Qm[3]};
          const T rB = Num<T>::rcp(Qp[0]);
          const T uBp[3] = {Qp[1] * rB, Qp[2] * rB, Qp[3] * rB};
          T dk[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) dk[c] = nsb[(9 + 6 * (ch & 1)) * kThreads + 6 * tid + 3 + c];
          // [F(Q*_+) - F(Q*_-)] . k_+ and [F(Q*_-) - F(Qbar)] . (k_+ - k_-): packed for linear upwind, which is
          // bound by instruction issue (20-block batch 2.50 -> 2.47 ms), one after the other for the
          // others, whose FMA pipe is the busier (WENO5 on 256^3 packed: 8.57 -> 8.61 ms)
          if constexpr (SCHEME == 1 && sizeof(T) == 4) {
            using P = typename PairOf<T>::type;
            P d[5], uBq[3], uAq[3], mAq[3], k[3], tv[5];
#pragma unroll
            for (int v = 0; v < 5; ++v) d[v] = pmk(dQ[v], dqm[v]);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              uBq[c] = pmk(uBp[c], uA[c]);
              uAq[c] = pmk(uA[c], ub[c]);
              mAq[c] = pmk(mA[c], qb[1 + c]);
              k[c] = pmk(kf[c], dk[c]);
            }
            dflux_pair<P>(g1, pmk(rB, rA), uBq, uAq, mAq, pmk(Qm[4], qb[4]), pmk(pA, pb), d, k, tv);
#pragma unroll
            for (int v = 0; v < 5; ++v) R[v] += tv[v].x + tv[v].y;
          } else {
            T t1v[5], t2v[5];
            dflux<T>(g1, rB, uBp, uA, mA, Qm[4], pA, dQ, kf, t1v);
            dflux<T>(g1, rA, uA, ub, qb + 1, qb[4], pb, dqm, dk, t2v);
#pragma unroll
            for (int v = 0; v < 5; ++v) R[v] += t1v[v] + t2v[v];
          }
        }
        T *const racc = static_cast<T *>(D->racc);
        // the accumulator holds four components side by side and the fifth behind them (one wide
        // access per point instead of four: the eta and zeta rows are only TT points wide)
        if (mode != MODE_WRITE) {                     // add what the passes before wrote
          T ra[4];
          load4(epb + 4 * tid, ra);
#pragma unroll
          for (int v = 0; v < 4; ++v) R[v] = ra[v] + R[v];
          R[4] = epb[4 * kThreads + tid] + R[4];
        }
        if (mode <= MODE_ADD) {
          store4(FPK_IN(racc + 4ULL * qo, racc, 4LL * qc - 3, B->status), R);
          *FPK_IN(comp_at(racc, qo, qc, 4), racc, 5LL * qc, B->status) = R[4];
        } else {
          const T Jc = Num<T>::rcp(kEarly ? fr[15 * kRing + off(ff)] : sm[CF_INVJ * kRing + off(ff)]);
          if (mode == MODE_RHS) {
            T *const out = static_cast<T *>(B->dqdt);
#pragma unroll
            for (int v = 0; v < 5; ++v)
              *FPK_IN(comp_at(out, qo, qc, v), out, 5LL * qc, B->status) = -Jc * R[v];
          } else {
            T *const qs = static_cast<T *>(B->q[(stage + 1) % 3]);
            const RkStage<T> rk(stage, s_dt);
            bool bad = false;
            T nv[5];
#pragma unroll
            for (int v = 0; v < 5; ++v) {
              nv[v] = rk(Qi[v], epb + (5 + v) * kThreads + tid, -Jc * R[v]);
              bad |= !isfinite(nv[v]);
            }
            if (stage < 2) {
              store4(FPK_IN(qs + 4ULL * qo, qs, 4LL * qc - 3, B->status), nv);
            } else {
#pragma unroll
              for (int v = 0; v < 4; ++v) *FPK_IN(comp_at(qs, qo, qc, v), qs, 5LL * qc, B->status) = nv[v];
            }
            *FPK_IN(comp_at(qs, qo, qc, 4), qs, 5LL * qc, B->status) = nv[4];
            if (bad) atomicOr(B->status, ST_NONFINITE);
          }
        }
      }
      if (!kEarly) __syncthreads();
      // ---- stage the next chunk's new cell from this thread's staging slots
      if (staged) {
        T Q[5];
        load4(nsb + 4 * tid, Q);
        Q[4] = nsb[4 * kThreads + tid];
        T kv[4];
        load4(nsb + 5 * kThreads + 4 * tid, kv);
        if (BND) {                                   // a slip-wall ghost?
          int uc = u + 4, c1 = t1, c2 = t2;
          wrap(uc, c1, c2);
          const int xs = uc - G;
          if (xs < 0 ? D->bclo >= 3 : xs >= nd && D->bchi >= 3) {
            const T *qp, *q4;
            unsigned cs;
            bool far, wall;
            FPK_CHK_ONLY(const T *sb; long long sn;)
            bc_source(xs, c1, c2, qp, q4, cs, far, wall FPK_CHK_ONLY(, sb, sn));
            if (wall) reflect(xs, c1, c2, Q);
          }
        }
        stage_cell(a + S + 4 + tf, Q, kv, kv[3]);
      }
      __syncthreads();
    }
    it = nit;
  }
}

// dynamic shared memory of a sweep variant: the cell and face rings, then the per-thread slots
template <typename T, int SCHEME, int FIX>
constexpr size_t sweep_smem() {
  return ((size_t)(kCellFields + sweep_face_fields(sizeof(T) == 4, SCHEME)) * sweep_ring(sizeof(T) == 4, SCHEME, FIX) +
          (size_t)(kNextFields + kEpiFields) * sweep_threads(sizeof(T) == 4, SCHEME, FIX)) * sizeof(T);
}

template <typename T, int M, int SCHEME, bool BND, int FIX>
cudaError_t launch_one(const SweepLaunch &L, int fp, cudaStream_t s) {
  constexpr size_t smem = sweep_smem<T, SCHEME, FIX>();
  constexpr int nt = sweep_threads(sizeof(T) == 4, SCHEME, FIX);
  if (L.grid <= 0) return cudaSuccess;
  return launch_kernel(fp_sweep<T, M, SCHEME, BND, FIX>, L.grid, nt, smem, s, L.chained, L.blocks, L.items, L.mode,
                       L.stage, L.dt, fp);
}

template <typename T, bool BND, int FIX>
cudaError_t launch_sweep_t(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s) {
#define FPK_CASE(MM, SS) \
  if (M == MM && scheme == SS) return launch_one<T, MM, SS, BND, FIX>(L, fp, s);
  FPK_CASE(2, 0) FPK_CASE(4, 0) FPK_CASE(6, 0) FPK_CASE(8, 0)
  FPK_CASE(2, 1) FPK_CASE(4, 1) FPK_CASE(6, 1) FPK_CASE(8, 1)
  FPK_CASE(2, 2) FPK_CASE(4, 2) FPK_CASE(6, 2) FPK_CASE(8, 2)
  FPK_CASE(2, 3) FPK_CASE(4, 3) FPK_CASE(6, 3) FPK_CASE(8, 3)
#undef FPK_CASE
  return cudaErrorInvalidValue;
}

// Opt in to the dynamic shared memory of a variant and return its resident CTAs per SM.
// Called before any launch or graph capture.
template <typename T, bool BND, int FIX>
int prepare_t(int M, int scheme) {
  int nb = 0;
#define FPK_OCC(MM, SS)                                                                              \
  if (M == MM && scheme == SS) {                                                                     \
    constexpr size_t smem = sweep_smem<T, SS, FIX>();                                                \
    cudaFuncSetAttribute(fp_sweep<T, MM, SS, BND, FIX>, cudaFuncAttributeMaxDynamicSharedMemorySize,  \
                         (int)smem);                                                                 \
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fp_sweep<T, MM, SS, BND, FIX>,                \
                                                  sweep_threads(sizeof(T) == 4, SS, FIX), smem);     \
  }
  FPK_OCC(2, 0) FPK_OCC(4, 0) FPK_OCC(6, 0) FPK_OCC(8, 0)
  FPK_OCC(2, 1) FPK_OCC(4, 1) FPK_OCC(6, 1) FPK_OCC(8, 1)
  FPK_OCC(2, 2) FPK_OCC(4, 2) FPK_OCC(6, 2) FPK_OCC(8, 2)
  FPK_OCC(2, 3) FPK_OCC(4, 3) FPK_OCC(6, 3) FPK_OCC(8, 3)
#undef FPK_OCC
  return nb > 0 ? nb : 1;
}

// One translation unit per (precision, boundary rules, fixed switches): the launcher and the
// preparation of its 16 (M, scheme) variants, named launch_sweep_<NAME> / prepare_sweep_<NAME>.
#define FPK_SWEEP_UNIT(NAME, T, BND, FIX)                                                           \
  cudaError_t launch_sweep_##NAME(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s) { \
    return launch_sweep_t<T, BND, FIX>(L, M, scheme, fp, s);                                        \
  }                                                                                                 \
  int prepare_sweep_##NAME(int M, int scheme) { return prepare_t<T, BND, FIX>(M, scheme); }

}  // namespace fpk
