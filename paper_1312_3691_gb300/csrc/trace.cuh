// Device code of the TPMC hot path for sm_103a (GB300): seeding and tracing.
// Included by one translation unit per BVH width (trace_w2.cu, trace_w4.cu,
// trace_w8.cu), which instantiate the kernels, and by kernels.cu (set-up).
//
//   seed_kernel<W, R>  pool path, first half: seeds a batch of particles
//                    (Eq. 11, Eq. 14a-c, Eq. 15; or the box CV), drops those
//                    that miss the mesh's front boxes and writes the others
//                    to the pool in device memory.
//   trace_kernel<R, MINB, CLL, W, COUNT, POOL>
//                    persistent, one warp = 32 particle slots refilled by
//                    ballot, from the pool (POOL) or from a queue in shared
//                    memory that the warp itself seeds; per slot: BVH closest
//                    hit with a watertight ray/triangle test (§II.A), Maxwell
//                    (or, with CLL, Cercignani-Lampis-Lord) re-emission, int64
//                    fixed-point momentum sums, until the particle misses or
//                    reaches max_bounces.  R = float (FP32 path) or double;
//                    MINB = register-capped occupancy; CLL: with the CLL
//                    branch; W: BVH width; COUNT: with the node-visit and
//                    triangle-test counters and the per-particle records
//                    (verification launches).
//
// This file shares nothing with the CPU oracle; both follow the paper and the
// published Philox4x32-10 definition (Salmon et al., SC'11).
#pragma once

#include <algorithm>
#include <cstddef>
#include <type_traits>

#include <cuda_runtime.h>
#include <math_constants.h>

#include "tpmc_internal.h"

namespace tpmc {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr double kBoltz = 1.380649e-23;
constexpr double kSqrtPiD = 1.7724538509055160273;

// ------------------------------------------------------------------ Philox
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k.x += 0x9E3779B9u;
      k.y += 0xBB67AE85u;
    }
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
  }
  return c;
}

// (k + 1/2) 2^-23 for the top 23 bits k: exact in float and double.
// In float from the bits: 1 + k 2^-23 less (1 - 2^-24), an exact difference,
// spares the conversion its quarter-rate pipe.
template <typename R>
__device__ __forceinline__ R uniform(uint32_t w) {
  if constexpr (sizeof(R) == 4) return __uint_as_float(0x3F800000u | (w >> 9)) - 0.999999940395355224609375f;
  return (R)(w >> 9) * (R)1.1920928955078125e-07 + (R)5.9604644775390625e-08;
}

// floor(f) for |f| < 2^21, as an integer and as a float: adding 1.5 2^23 rounded
// down leaves it in the low bits (two additions where two conversions take the
// quarter-rate pipe twice).
__device__ __forceinline__ int floor_bits(float f, float& as_float) {
  const float r = __fadd_rd(f, 12582912.0f);
  as_float = r - 12582912.0f;
  return __float_as_int(r) - 0x4B400000;
}

__device__ __forceinline__ uint4 draws(const QueryDev& q, uint64_t pid, uint32_t block) {
  return philox4x32_10(make_uint4((uint32_t)pid, (uint32_t)(pid >> 32), q.stream_id, block),
                       make_uint2((uint32_t)q.seed, (uint32_t)(q.seed >> 32)));
}

// ----------------------------------------------------------- math by type
template <typename R> struct Fn;
template <> struct Fn<float> {
  static __device__ __forceinline__ float exp(float x) { return expf(x); }
  static __device__ __forceinline__ float log(float x) { return logf(x); }
  static __device__ __forceinline__ float sqrt(float x) { return sqrtf(x); }
  static __device__ __forceinline__ float erfc(float x) { return erfcf(x); }
  static __device__ __forceinline__ float erfcx(float x) { return erfcxf(x); }
  static __device__ __forceinline__ float ncdfinv(float x) { return normcdfinvf(x); }
  static __device__ __forceinline__ float erfcinv(float x) { return erfcinvf(x); }
  static __device__ __forceinline__ void sincospi(float x, float* s, float* c) { sincospif(x, s, c); }
  static __device__ __forceinline__ float fabs(float x) { return fabsf(x); }
  // The hardware reciprocal (within one unit in the last place), not the
  // correctly rounded division: for the ray's slab constants, the shear
  // constant and hit distances, where the correctly rounded form cost 1-6 %
  // of throughput.  Box tests stay conservative (the builder widens every box
  // by a grid step, far more than these errors move a slab), and the
  // watertight test stays watertight (one shear for all triangles of a ray).
  static __device__ __forceinline__ float rcp(float x) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
  }
  static __device__ __forceinline__ float rsqrt(float x) { return rsqrtf(x); }
};
template <> struct Fn<double> {
  static __device__ __forceinline__ double exp(double x) { return ::exp(x); }
  static __device__ __forceinline__ double log(double x) { return ::log(x); }
  static __device__ __forceinline__ double sqrt(double x) { return ::sqrt(x); }
  static __device__ __forceinline__ double erfc(double x) { return ::erfc(x); }
  static __device__ __forceinline__ double erfcx(double x) { return ::erfcx(x); }
  static __device__ __forceinline__ double ncdfinv(double x) { return ::normcdfinv(x); }
  static __device__ __forceinline__ double erfcinv(double x) { return ::erfcinv(x); }
  static __device__ __forceinline__ void sincospi(double x, double* s, double* c) { ::sincospi(x, s, c); }
  static __device__ __forceinline__ double fabs(double x) { return ::fabs(x); }
  static __device__ __forceinline__ double rcp(double x) { return 1.0 / x; }
  static __device__ __forceinline__ double rsqrt(double x) { return 1.0 / ::sqrt(x); }
  static constexpr double kTolLat = 1e-14;
  static constexpr double kTolSpeed = 1e-14;
  static constexpr int kIter = 40;
};

// Query constants in the path's precision.
template <typename R> struct QC;
template <> struct QC<float> {
  float S, cw, r_cv, sqrtpi_4S, K1, Dinv, scale;
  float Rm[9], vhat[3], center[3], ref[3];
  __device__ __forceinline__ void load(const QueryDev& q) {
    S = q.fc[kFcS]; cw = q.fc[kFcCw]; r_cv = q.fc[kFcRcv]; sqrtpi_4S = q.fc[kFcSqrtpi4S];
    K1 = q.fc[kFcK1]; Dinv = q.fc[kFcDinv]; scale = q.fc[kFcScale];
#pragma unroll
    for (int i = 0; i < 9; ++i) Rm[i] = q.fc[kFcR + i];
#pragma unroll
    for (int i = 0; i < 3; ++i) { vhat[i] = q.fc[kFcVhat + i]; center[i] = q.fc[kFcCenter + i]; ref[i] = q.fc[kFcRef + i]; }
  }
};
template <> struct QC<double> {
  double S, cw, r_cv, sqrtpi_4S, K1, Dinv, scale;
  double Rm[9], vhat[3], center[3], ref[3];
  __device__ __forceinline__ void load(const QueryDev& q) {
    S = q.S; cw = q.cw; r_cv = q.r_cv; sqrtpi_4S = kSqrtPiD / (4.0 * q.S); K1 = q.K1; Dinv = 1.0 / q.Dnorm;
    scale = 1.0 / q.quantum;
#pragma unroll
    for (int i = 0; i < 9; ++i) Rm[i] = q.R[i];
#pragma unroll
    for (int i = 0; i < 3; ++i) { vhat[i] = q.vhat[i]; center[i] = q.center[i]; ref[i] = q.ref[i]; }
  }
};

// ------------------------------------------------------- seeding (§III.A)
// Latitude law (Eq. 11) in x = sin(phi): CDF written with erfc(-S x) = 1 + erf(S x):
//   H(x) = [ sqrt(pi)/(4S) (2 S^2 x^2 + 1) erfc(-S x) + (x/2) e^{-S^2 x^2} - K1 ] / D,
//   K1 = sqrt(pi)/(4S) (2 S^2 + 1) erfc(S) - e^{-S^2}/2,  so H(-1) = 0 exactly in the algebra.
// Its density h(x) = [e^{-S^2 x^2} + sqrt(pi) S x erfc(-S x)] / D.
template <typename R>
__device__ __forceinline__ R latitude_cdf(R x, R S, R sqrtpi_4S, R K1, R Dinv) {
  const R Sx = S * x;
  return (sqrtpi_4S * ((R)2 * Sx * Sx + (R)1) * Fn<R>::erfc(-Sx) + (R)0.5 * x * Fn<R>::exp(-Sx * Sx) - K1) * Dinv;
}
template <typename R>
__device__ __forceinline__ R latitude_pdf(R x, R S, R Dinv) {
  const R Sx = S * x;
  return (Fn<R>::exp(-Sx * Sx) + (R)kSqrtPiD * Sx * Fn<R>::erfc(-Sx)) * Dinv;
}

// Interpolated start from a query's table laid out in z = Phi^-1(u).  Plain loads:
// the set-up may write the table after the trace kernel has been launched.
__device__ __forceinline__ float z_table_start(const float* tab, int n, float z, float z_lo, float z_step) {
  const float f = (z - z_lo) / z_step;
  float fl;
  const int j = min(max(floor_bits(f, fl), 0), n - 2);
  const float w = fminf(fmaxf(f - fminf(fmaxf(fl, 0.0f), (float)(n - 2)), 0.0f), 1.0f);
  return (1.0f - w) * tab[j] + w * tab[j + 1];
}

// Float latitude solve near a pole, in w = 1 - x (up) or w = 1 + x (down).
// The probability within w of the pole is the integral of h over that end
// interval; with g = D h, g' = sqrt(pi) S erfc(-S t) and g'' = 2 S^2 e^{-S^2 t^2},
// it is the cubic c0 w + c1 w^2 + c2 w^3 (Taylor, next term below 3e-7
// relative for w < 0.002), coefficients per query from the FP64 set-up.
// Newton from w = q / c0, one step: w, and cos(phi) = sqrt(w (2 - w)), to
// ~1e-7 relative, which x itself cannot carry in float this close to +-1.
// Returns (x, cos(phi)) by value: an out-of-line call that wrote through a
// pointer would keep the caller's variable in local memory.
__device__ __noinline__ float2 latitude_pole(float q, float c0, float c1, float c2, bool up) {
  float w = q / c0;
  const float f = ((c2 * w + c1) * w + c0) * w - q;
  const float d = (3.0f * c2 * w + 2.0f * c1) * w + c0;
  w = fminf(fmaxf(w - f / d, 0.0f), 1.0f);
  return make_float2(up ? 1.0f - w : w - 1.0f, sqrtf(w * (2.0f - w)));
}

constexpr float kPoleW = 0.002f;  // pole solves within this distance of x = +-1

// x = H^-1(u), and cphi = cos(phi) = sqrt(1 - x^2).  Float: start from the
// query's table at z = Phi^-1(u) (error ~1e-4), then one Newton step (error
// ~1e-7 over all tails): a fixed step count keeps the warp converged; within
// kPoleW of a pole, the pole solve above.  Double: the same start, then a
// safeguarded Newton loop (on log H in the lower tail) to double precision.
template <typename R>
__device__ R latitude_inverse(R u, const QueryDev& q, const QC<R>& c, R* cphi) {
  const float z = normcdfinvf((float)u);
  R x = (R)z_table_start(q.htab, kHTable + 1, z, (float)kZLo, (float)((kZHi - kZLo) / kHTable));
  if constexpr (sizeof(R) == 4) {
    const R H = latitude_cdf<R>(x, c.S, c.sqrtpi_4S, c.K1, c.Dinv);
    const R h = latitude_pdf<R>(x, c.S, c.Dinv);
    if (h > (R)0) x -= (H - u) / h;
    x = fmin(fmax(x, (R)-1), (R)1);
    *cphi = Fn<R>::sqrt(((R)1 - x) * ((R)1 + x));
    // within kPoleW of a pole, the pole solve (rare; the common path stays branch-free)
    if (x > 1.0f - kPoleW || x < kPoleW - 1.0f) {
      const bool up = x > 0.0f;
      const int k = up ? kFcPole : kFcPole + 3;
      const float2 r = latitude_pole(up ? 1.0f - u : u, q.fc[k], q.fc[k + 1], q.fc[k + 2], up);
      x = r.x;
      *cphi = r.y;
    }
    return x;
  } else {
    R lo = -1, hi = 1;
    const bool logmode = u < (R)0.0625;
    const R lu = logmode ? Fn<R>::log(u) : (R)0;
#pragma unroll 1
    for (int it = 0; it < Fn<R>::kIter; ++it) {
      // the law and its density from one erfc and one exp: each is a chain of
      // branches in double, which the compiler does not merge by itself
      const R Sx = c.S * x;
      const R ec = Fn<R>::erfc(-Sx), ex = Fn<R>::exp(-Sx * Sx);
      const R H = (c.sqrtpi_4S * ((R)2 * Sx * Sx + (R)1) * ec + (R)0.5 * x * ex - c.K1) * c.Dinv;
      const R h = (ex + (R)kSqrtPiD * Sx * ec) * c.Dinv;
      R f, dx;
      if (logmode) {
        if (!(H > (R)0)) { lo = x; x = (R)0.5 * (lo + hi); continue; }
        f = Fn<R>::log(H) - lu;
        dx = -f * H / h;
      } else {
        f = H - u;
        dx = -f / h;
      }
      if (f == (R)0) break;
      if (f < (R)0) lo = x; else hi = x;
      if (Fn<R>::fabs(dx) <= Fn<R>::kTolLat * (Fn<R>::fabs(x) + (R)1e-3)) { x += dx; break; }
      x += dx;
      if (!(x > lo && x < hi)) x = (R)0.5 * (lo + hi);
    }
    x = fmin(fmax(x, (R)-1), (R)1);
    *cphi = Fn<R>::sqrt(((R)1 - x) * ((R)1 + x));
    return x;
  }
}

// Inward normal speed (Eq. 14a, numerator read as 2 v_n/c_mp): x = v_n/c_mp > 0
// with density p(x) = 2 x e^{-(x-s)^2} / Z(s), Z(s) = e^{-s^2} + sqrt(pi) s erfc(-s).
// The root of F(x) = u is found on the smaller tail, so that the solved
// probability keeps its digits in float:
//   u > 1/2: Q(x) = 1 - F(x) = [e^{-y^2} + sqrt(pi) s erfc(y)] / Z, y = x - s
//            (for s < 0 as e^{-x(x-2s)} [1 + sqrt(pi) s erfcx(y)] / [1 + sqrt(pi) s erfcx(-s)]);
//   u <= 1/2: F(x) by 4-point Gauss-Legendre on [0, x] near x = 0 (F ~ x^2 there), else
//            F = [g(s - x) - g(s)] / Z with g(w) = sqrt(pi) s erfc(w) - e^{-w^2}
//            (for s < 0 as 1 - Q).
// Newton runs on log Q (additive steps) or log F (multiplicative steps in x,
// exact for the x^2 law near 0), inside a bisection bracket.
template <typename R>
__device__ R normal_speed_inverse_adaptive(R u, R s, R x_start) {
  const R sp = (R)kSqrtPiD * s;
  const bool upper = u > (R)0.5;
  const R target = upper ? (R)1 - u : u;  // 1 - u is exact for u = (2k+1) 2^-24
  const R lt = Fn<R>::log(target);
  R Z, Zs;  // Z, and Zs = Z e^{s^2} when s < 0
  if (s >= (R)0) { Z = Fn<R>::exp(-s * s) + sp * Fn<R>::erfc(-s); Zs = Z; }
  else { Zs = (R)1 + sp * Fn<R>::erfcx(-s); Z = Zs; }
  const R xq = fmin((R)0.05, (R)0.3 / ((R)1 + Fn<R>::fabs(s)));
  const R g_s = sp * Fn<R>::erfc(s) - Fn<R>::exp(-s * s);
  R lo = 0, hi = fmax(s, (R)0) + (R)6.5;
  R x = x_start;
  if (!(x > lo && x < hi)) x = (R)0.5 * (lo + hi);
#pragma unroll 1
  for (int it = 0; it < Fn<R>::kIter; ++it) {
    const R y = x - s;
    R T, p;
    // x near 0 below the median: F by 4-point Gauss-Legendre of p on [0, x]
    const bool quad = !upper && x < xq;
    R e, q1 = (R)0;
    if (s >= (R)0) {
      // erfc(y) above the median, erfc(-y) below: one evaluation for both
      e = Fn<R>::exp(-y * y);
      const R ec = Fn<R>::erfc(upper ? y : s - x);
      p = (R)2 * x * e / Z;
      T = upper ? (e + sp * ec) / Z : ((sp * ec - e) - g_s) / Z;
    } else {
      e = Fn<R>::exp(-x * (x - (R)2 * s));
      p = (R)2 * x * e / Zs;
      q1 = e * ((R)1 + sp * Fn<R>::erfcx(y));
      T = upper ? q1 / Zs : (Zs - q1) / Zs;
    }
    if (quad) {
      const R gx[4] = {(R)0.06943184420297371, (R)0.33000947820757187, (R)0.6699905217924281, (R)0.9305681557970262};
      const R gw[4] = {(R)0.17392742256872692, (R)0.3260725774312731, (R)0.3260725774312731, (R)0.17392742256872692};
      R acc = 0;
#pragma unroll 1
      for (int k = 0; k < 4; ++k) {
        const R t = x * gx[k];
        acc += gw[k] * (R)2 * t * Fn<R>::exp(s >= (R)0 ? -(t - s) * (t - s) : -t * (t - (R)2 * s));
      }
      T = x * acc / (s >= (R)0 ? Z : Zs);
    }
    if (!(T > (R)0)) {
      // underflow or cancellation: x lies deep in the solved tail
      if (upper) hi = x; else lo = x;
      x = (R)0.5 * (lo + hi);
      continue;
    }
    const R f = Fn<R>::log(T) - lt;
    if (f == (R)0) break;
    R dx;
    if (upper) {  // Q decreases in x
      if (f > (R)0) lo = x; else hi = x;
      if (!(p > (R)0)) { x = (R)0.5 * (lo + hi); continue; }
      dx = f * T / p;
    } else {      // F increases in x; Newton in log x
      if (f < (R)0) lo = x; else hi = x;
      if (!(p > (R)0)) { x = (R)0.5 * (lo + hi); continue; }
      dx = x * (Fn<R>::exp(-f * T / (x * p)) - (R)1);
    }
    if (Fn<R>::fabs(dx) <= Fn<R>::kTolSpeed * (x + (R)1e-3)) { x += dx; break; }
    x += dx;
    if (!(x > lo && x < hi)) x = (R)0.5 * (lo + hi);
  }
  return fmax(x, (R)0);
}

// Start of the normal-speed solve from the context's table at (s, z = Phi^-1(u));
// beyond the table's s range: the Gaussian limit s + z / sqrt(2) + 1/(2s)
// (large s) or the small-x law F ~ x^2 / (Z e^{s^2}) (very negative s).
__device__ __forceinline__ float normal_speed_start(const float* tab, float s, float z, float u) {
  const float fs = (s - (float)kVnSLo) / (float)kVnStep;
  if (!(fs <= (float)(kVnNS - 1))) return s + 0.70710678f * z + 0.5f / s;  // also catches NaN
  if (!(fs >= 0.0f)) {
    const float a = -s;
    const float zs = 1.0f - 1.77245385f * a * erfcxf(a);  // e^{s^2} Z
    return fmaxf(sqrtf(u * fmaxf(zs, 1e-30f)), 1e-30f);
  }
  float fi, fj;
  const int i = min(floor_bits(fs, fi), kVnNS - 2);
  const float a = fminf(fs - fminf(fi, (float)(kVnNS - 2)), 1.0f);
  const float fz = (z - (float)kZLo) / (float)kVnStep;
  const int j = min(max(floor_bits(fz, fj), 0), kVnNZ - 2);
  const float b = fminf(fmaxf(fz - fminf(fmaxf(fj, 0.0f), (float)(kVnNZ - 2)), 0.0f), 1.0f);
  const float* r0 = tab + i * kVnNZ + j;
  const float* r1 = r0 + kVnNZ;
  const float x = (1.0f - a) * ((1.0f - b) * __ldg(r0) + b * __ldg(r0 + 1)) + a * ((1.0f - b) * __ldg(r1) + b * __ldg(r1 + 1));
  return fmaxf(x, 1e-30f);
}

// Float: one Newton step from the bilinear table start (start error ~3e-5;
// after the step ~6e-8 relative in the median, 2e-5 at the 99th percentile,
// <= 1.5e-4 at the extreme uniforms u ~ 2^-24), on the survival function
// above the median and on the CDF below it (selected per lane, no branch on
// the tail); near x = 0 the CDF comes from 4-point Gauss-Legendre.
// Double: the table start, then the adaptive loop to double precision.
template <typename R>
__device__ R normal_speed_inverse(R u, R s, const float* tab) {
  const float z = normcdfinvf((float)u);
  const R x0 = (R)normal_speed_start(tab, (float)s, z, (float)u);
  if constexpr (sizeof(R) == 8) {
    return normal_speed_inverse_adaptive<R>(u, s, x0);
  } else {
    const float sp = 1.77245385090551602730f * s;
    const bool upper = u > 0.5f;
    const float target = upper ? 1.0f - u : u;
    float Z, Zs, gs = 0.0f;
    if (s >= 0.0f) {
      const float es = expf(-s * s), ecs = erfcf(s);  // erfc(-s) = 2 - erfc(s), in [1, 2]
      Z = es + sp * (2.0f - ecs);
      Zs = Z;
      gs = sp * ecs - es;
    } else {
      Zs = 1.0f + sp * erfcxf(-s);
      Z = Zs;
    }
    const float xq = fminf(0.05f, 0.3f / (1.0f + fabsf(s)));
    float x = x0;
    {
      const float y = x - s;
      float T, p;
      if (s >= 0.0f) {
        const float e = expf(-y * y);
        p = 2.0f * x * e / Z;
        const float ec = erfcf(fabsf(y));
        const float erfc_y = y >= 0.0f ? ec : 2.0f - ec;
        const float erfc_w = y >= 0.0f ? 2.0f - ec : ec;
        T = upper ? (e + sp * erfc_y) / Z : ((sp * erfc_w - e) - gs) / Z;
      } else {
        const float e = expf(-x * (x - 2.0f * s));
        p = 2.0f * x * e / Zs;
        const float qn = e * (1.0f + sp * erfcxf(y));
        T = upper ? qn / Zs : (Zs - qn) / Zs;
      }
      if (!upper && x < xq) {
        // F near x = 0 by quadrature of p on [0, x] (F ~ x^2 keeps its digits)
        const float gx[4] = {0.06943184420297371f, 0.33000947820757187f, 0.6699905217924281f, 0.9305681557970262f};
        const float gw[4] = {0.17392742256872692f, 0.3260725774312731f, 0.3260725774312731f, 0.17392742256872692f};
        // integrand scaled by e^{s^2} when s < 0 (then divided by Zs = Z e^{s^2})
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float t = x * gx[k];
          acc += gw[k] * 2.0f * t * expf(s >= 0.0f ? -(t - s) * (t - s) : -t * (t - 2.0f * s));
        }
        T = x * acc / (s >= 0.0f ? Z : Zs);
      }
      const float f = T - target;
      const float dx = p > 0.0f ? (upper ? f / p : -f / p) : 0.0f;
      const float xn = x + dx;
      x = xn > 0.0f ? xn : 0.5f * x;
    }
    return x;
  }
}

// Seed particle pid of query q: position on the CV (body frame, m) and
// velocity (c_mp units).  Stream frame: flow along +z, upstream pole at -z;
// local frame n (inward), t1 (tangential projection of the flow), t2 = t1 x n;
// Eq. 14b-c tangential laws by Box-Muller; Eq. 15 rotation to the body frame.
// Box-CV constants in the path's precision.
template <typename R> struct BoxC;
template <> struct BoxC<float> {
  static __device__ __forceinline__ float s(const QueryDev& q, int f) { return q.fface_s[f]; }
  static __device__ __forceinline__ float lo(const QueryDev& q, int i) { return q.fbox_lo[i]; }
  static __device__ __forceinline__ float ext(const QueryDev& q, int i) { return q.fbox_ext[i]; }
  static __device__ __forceinline__ float hi(const QueryDev& q, int i) { return q.fbox_lo[i] + q.fbox_ext[i]; }
};
template <> struct BoxC<double> {
  static __device__ __forceinline__ double s(const QueryDev& q, int f) { return q.face_s[f]; }
  static __device__ __forceinline__ double lo(const QueryDev& q, int i) { return q.box_lo[i]; }
  static __device__ __forceinline__ double ext(const QueryDev& q, int i) { return q.box_hi[i] - q.box_lo[i]; }
  static __device__ __forceinline__ double hi(const QueryDev& q, int i) { return q.box_hi[i]; }
};

// Inward normal speed of the Maxwell box faces: the free-stream Maxwellian
// restricted to x = v_n / c_mp > 0 (density exp(-(x - s)^2), no flux factor),
// whose survival function erfc(x - s) / erfc(-s) = 1 - u inverts in closed
// form.  1 - u is exact for these uniforms.  A face whose erfc(-s) underflows
// carries no particle ids (its flux share is below 1e-35); the guard only
// keeps a non-finite value out of the ray set-up.
template <typename R>
__device__ __forceinline__ R truncated_normal_inverse(R u, R s) {
  R x = s + Fn<R>::erfcinv(((R)1 - u) * Fn<R>::erfc(-s));
  if (!(x > (R)0) || !(x < (R)1e30)) x = (R)1e-30;
  return x;
}

// Rectangular-CV seeding (§I, §III.A): the face owning id pid, a uniform
// point on it, the inward normal speed from the face's law, and the
// tangential components of the drifting Maxwellian (free-stream drift plus the
// same Box-Muller pair as on the sphere).
template <typename R>
__device__ __forceinline__ void seed_box(const QueryDev& q, const QC<R>& c, const float* vn_table, uint64_t pid,
                                         const uint4& w0, uint32_t w_a, R pos[3], R vel[3]) {
  int f = 0;
#pragma unroll
  for (int k = 0; k < 5; ++k) f += pid >= q.face_end[k] ? 1 : 0;
  // face axis ax; its first tangential axis (ax + 1) mod 3 takes w0.x, the second w0.y
  const int ax = f >> 1, a1 = ax == 2 ? 0 : ax + 1;
  const bool hi_face = (f & 1) == 0;
  const R s_f = BoxC<R>::s(q, f);
  const R vn = q.cv_kind == TPMC_CV_BOX_FLUX ? normal_speed_inverse<R>(uniform<R>(w0.z), s_f, vn_table)
                                             : truncated_normal_inverse<R>(uniform<R>(w0.z), s_f);
  const R rad = Fn<R>::sqrt(-Fn<R>::log(uniform<R>(w0.w)));
  R sa, ca;
  Fn<R>::sincospi((R)2 * uniform<R>(w_a), &sa, &ca);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (i == ax) {
      pos[i] = hi_face ? BoxC<R>::hi(q, i) : BoxC<R>::lo(q, i);
      vel[i] = hi_face ? -vn : vn;
    } else {
      const bool first = i == a1;
      pos[i] = BoxC<R>::lo(q, i) + uniform<R>(first ? w0.x : w0.y) * BoxC<R>::ext(q, i);
      vel[i] = c.S * c.vhat[i] + rad * (first ? ca : sa);
    }
  }
}

// One Philox block seeds a particle: u_x, u_theta, u_vn, u_r from the top 23 bits
// of its words, u_a (Box-Muller angle) from 23 low bits they leave unused.
__device__ __forceinline__ uint32_t angle_word(const uint4& w0) {
  return ((w0.x & 0x1FFu) | ((w0.y & 0x1FFu) << 9) | ((w0.z & 0x1Fu) << 18)) << 9;
}

template <typename R>
__device__ __forceinline__ void seed_particle(const QueryDev& q, const QC<R>& c, const float* vn_table, uint64_t pid,
                                              const uint4& w0, R pos[3], R vel[3]) {
  const uint32_t w_a = angle_word(w0);
  if (q.cv_kind != TPMC_CV_SPHERE) {
    seed_box<R>(q, c, vn_table, pid, w0, w_a, pos, vel);
    return;
  }
  R cphi;
  const R x = latitude_inverse<R>(uniform<R>(w0.x), q, c, &cphi);
  R st, ct;
  Fn<R>::sincospi((R)2 * uniform<R>(w0.y), &st, &ct);
  const R vn = normal_speed_inverse<R>(uniform<R>(w0.z), c.S * x, vn_table);
  const R rad = Fn<R>::sqrt(-Fn<R>::log(uniform<R>(w0.w)));
  R sa, ca;
  Fn<R>::sincospi((R)2 * uniform<R>(w_a), &sa, &ca);
  const R vt1 = c.S * cphi + rad * ca;
  const R vt2 = rad * sa;
  // stream-frame vectors: out = (cphi ct, cphi st, -x), n = -out, t1 = (x ct, x st, cphi), t2 = (st, -ct, 0)
  const R ps[3] = {cphi * ct, cphi * st, -x};
  const R vs[3] = {-vn * cphi * ct + vt1 * x * ct + vt2 * st, -vn * cphi * st + vt1 * x * st - vt2 * ct,
                   vn * x + vt1 * cphi};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const R rp = c.Rm[3 * i] * ps[0] + c.Rm[3 * i + 1] * ps[1] + c.Rm[3 * i + 2] * ps[2];
    pos[i] = c.center[i] + c.r_cv * rp;
    vel[i] = c.Rm[3 * i] * vs[0] + c.Rm[3 * i + 1] * vs[1] + c.Rm[3 * i + 2] * vs[2];
  }
}

// --------------------------------------------------- closest hit (§II.A)
template <typename R>
__device__ __forceinline__ R pick(const R v[3], int k) {
  return k == 0 ? v[0] : (k == 1 ? v[1] : v[2]);
}

template <typename R> struct TriLoad;
template <> struct TriLoad<float> {
  static __device__ __forceinline__ uint32_t load(const MeshDev& m, uint32_t k, float A[3], float B[3], float C[3]) {
    const float4 a = __ldg(&m.tris[3 * k]), b = __ldg(&m.tris[3 * k + 1]), c = __ldg(&m.tris[3 * k + 2]);
    A[0] = a.x; A[1] = a.y; A[2] = a.z;
    B[0] = b.x; B[1] = b.y; B[2] = b.z;
    C[0] = c.x; C[1] = c.y; C[2] = c.z;
    return __float_as_uint(a.w);
  }
};
template <> struct TriLoad<double> {
  static __device__ __forceinline__ uint32_t load(const MeshDev& m, uint32_t k, double A[3], double B[3],
                                                  double C[3]) {
    const double2* p = reinterpret_cast<const double2*>(m.tris64 + 12 * (size_t)k);
    const double2 p0 = __ldg(p), p1 = __ldg(p + 1), p2 = __ldg(p + 2), p3 = __ldg(p + 3), p4 = __ldg(p + 4);
    A[0] = p0.x; A[1] = p0.y; A[2] = p1.x;
    B[0] = p1.y; B[1] = p2.x; B[2] = p2.y;
    C[0] = p3.x; C[1] = p3.y; C[2] = p4.x;
    return (uint32_t)p4.y;
  }
};

// Edge function without contraction so that a shared edge evaluates to exactly
// opposite values in its two triangles (watertightness).
__device__ __forceinline__ float edge_fn(float a, float b, float c, float d) {
  return __fsub_rn(__fmul_rn(a, b), __fmul_rn(c, d));
}
__device__ __forceinline__ double edge_fn(double a, double b, double c, double d) {
  return __dsub_rn(__dmul_rn(a, b), __dmul_rn(c, d));
}

// a b - c d in float with the sign of the exact value, and exactly 0 when
// a b = c d: Kahan's algorithm, w = c d, e = w - c d (exact by an FMA),
// f = round(a b - w), result f + e, whose relative error is at most two units
// in the last place (Jeannerod, Louvet & Muller, Math. Comp. 2013).  It
// decides the watertight test's ties in float where the plain edge function
// rounds to 0.
__device__ __forceinline__ float edge_fn_exact(float a, float b, float c, float d) {
  const float w = __fmul_rn(c, d);
  const float e = __fmaf_rn(-c, d, w);
  const float f = __fmaf_rn(a, b, -w);
  return __fadd_rn(f, e);
}

// B: the arithmetic of the box tests, float also in double precision on binary
// trees.  There the boxes' distances count from t0, a little before the ray meets
// the mesh, so that they keep their digits whatever the control volume's size,
// and box tests allow their rounding (trav_inner): every triangle that the ray
// may hit is still reached, and only the triangle tests decide.  (An SM issues a
// double instruction every 16 cycles; a node visit had 40 of them.  1e5 particles
// on the 1,280-triangle icosphere: 916 -> 661 us.)
template <typename R, typename B = R>
struct Ray {
  R o[3], d[3];
  B inv[3], oi[3];
  R tlo;
  R t0;     // B != R
  B tnear;  // B != R: no distance below it counts
  // wide trees: visit position (0 first) of each child-box corner c (nibble c
  // of ptab) and the corner at each position (nibble p of stab)
  uint32_t ptab, stab;
  uint32_t nsel[3];  // binary trees: selectors of the near box planes (ray_to_grid)
};

// Woop, Benthin & Wald (JCGT 2013): shear the ray onto +z of a permuted frame.
template <typename R>
struct Shear {
  R Sx, Sy, Sz;
  int kx, ky, kz;
};

template <typename R>
__device__ __forceinline__ Shear<R> make_shear(const R d[3]) {
  Shear<R> s;
  const R ax = Fn<R>::fabs(d[0]), ay = Fn<R>::fabs(d[1]), az = Fn<R>::fabs(d[2]);
  s.kz = (ax > ay) ? (ax > az ? 0 : 2) : (ay > az ? 1 : 2);
  s.kx = s.kz == 2 ? 0 : s.kz + 1;
  s.ky = s.kx == 2 ? 0 : s.kx + 1;
  if (pick(d, s.kz) < (R)0) { const int t = s.kx; s.kx = s.ky; s.ky = t; }
  s.Sz = Fn<R>::rcp(pick(d, s.kz));
  s.Sx = pick(d, s.kx) * s.Sz;
  s.Sy = pick(d, s.ky) * s.Sz;
  return s;
}

// t0: for B != R, where the boxes' distances start (0 <= t0 <= the first hit).
template <typename R, typename B>
__device__ __forceinline__ void make_ray(Ray<R, B>& r, const R o[3], const R d[3], R tlo, R t0 = (R)0) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    r.o[i] = o[i];
    r.d[i] = d[i];
    const R di = Fn<R>::fabs(d[i]) < (R)1e-30 ? copysign((R)1e-30, d[i]) : d[i];
    if constexpr (std::is_same_v<R, B>) {
      r.inv[i] = Fn<R>::rcp(di);
      r.oi[i] = o[i] * r.inv[i];
    } else {
      r.inv[i] = Fn<B>::rcp((B)di);
    }
  }
  r.tlo = tlo;
  if constexpr (!std::is_same_v<R, B>) {
    r.t0 = t0;
    r.tnear = (B)(tlo - t0) - (B)1e-6 * Fn<B>::fabs((B)(tlo - t0));
  }
}

// A distance before a seeded particle meets the mesh's bounding sphere (see Ray).
__device__ __forceinline__ double box_start(const MeshDev& m, const double o[3], const double d[3]) {
  float od = 0.0f, dd = 0.0f;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float x = (float)(o[i] - (double)m.centre[i]), y = (float)d[i];
    od = fmaf(x, y, od);
    dd = fmaf(y, y, dd);
  }
  const float t = -od / dd - 1.001f * m.scene_radius * rsqrtf(dd);
  const float t0 = t - 1e-4f * fabsf(t);
  return t0 > 0.0f && t0 < 1e30f ? (double)t0 : 0.0;
}

// Watertight ray/triangle test; updates (tbest, best) by nearest t, then lower index.
template <typename R, typename BX>
__device__ __forceinline__ void test_triangle(const Ray<R, BX>& r, const Shear<R>& sh, const R V0[3], const R V1[3], const R V2[3],
                                              uint32_t id, R& tbest, uint32_t& best) {
  R A[3], B[3], C[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) { A[i] = V0[i] - r.o[i]; B[i] = V1[i] - r.o[i]; C[i] = V2[i] - r.o[i]; }
  const int kx = sh.kx, ky = sh.ky, kz = sh.kz;
  const R Akz = pick(A, kz), Bkz = pick(B, kz), Ckz = pick(C, kz);
  const R Ax = pick(A, kx) - sh.Sx * Akz, Ay = pick(A, ky) - sh.Sy * Akz;
  const R Bx = pick(B, kx) - sh.Sx * Bkz, By = pick(B, ky) - sh.Sy * Bkz;
  const R Cx = pick(C, kx) - sh.Sx * Ckz, Cy = pick(C, ky) - sh.Sy * Ckz;
  R U = edge_fn(Cx, By, Cy, Bx);
  R V = edge_fn(Ax, Cy, Ay, Cx);
  R W = edge_fn(Bx, Ay, By, Ax);
  if constexpr (sizeof(R) == 4) {
    if (U == 0.0f || V == 0.0f || W == 0.0f) {
      // the ray meets an edge or a vertex to float rounding: the exact signs decide
      U = edge_fn_exact(Cx, By, Cy, Bx);
      V = edge_fn_exact(Ax, Cy, Ay, Cx);
      W = edge_fn_exact(Bx, Ay, By, Ax);
    }
  }
  if ((U < (R)0 || V < (R)0 || W < (R)0) && (U > (R)0 || V > (R)0 || W > (R)0)) return;
  R det = U + V + W;
  if (det == (R)0) return;
  R T = U * (sh.Sz * Akz) + V * (sh.Sz * Bkz) + W * (sh.Sz * Ckz);
  if (det < (R)0) { det = -det; T = -T; }
  if (T <= r.tlo * det || T > tbest * det) return;
  const R t = T * Fn<R>::rcp(det);
  if (t < tbest || (t == tbest && id < best)) { tbest = t; best = id; }
}

// Three-input min and max (one instruction each for float on sm_100 and later).
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ double max3(double a, double b, double c) { return fmax(fmax(a, b), c); }
__device__ __forceinline__ double min3(double a, double b, double c) { return fmin(fmin(a, b), c); }

// Binary trees keep their boxes on the mesh's grid: plane = qorigin + q qstep.
// The ray's slab constants are turned into grid units once per segment, so
// that a node's plane q, read as the float 2^23 + q (exact), gives its
// distance t = (2^23 + q) inv' - oi' in one FMA: inv' = qstep / d (exact,
// qstep is a power of two) and oi' = 2^23 inv' - (qorigin - o) / d.  The
// rounding of oi' is below half a grid step, inside the one step by which
// the builder widens every box.  A box's lo and hi along an axis share a
// word, and nsel[a] is the byte selector that reads the plane the ray meets
// first along a (lo where it runs towards +a); the other plane's selector is
// nsel[a] ^ 0x22.  The near and far distances then need no min and max.
template <typename R, typename B>
__device__ __forceinline__ void ray_to_grid(Ray<R, B>& r, const MeshDev& m) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const B sa = (B)m.qstep[i] * r.inv[i];
    if constexpr (std::is_same_v<R, B>) {
      const R oa = fma((R)m.qorigin[i], r.inv[i], -r.oi[i]);
      r.oi[i] = fma((R)8388608.0, sa, -oa);
    } else {
      // the start at t0 in grid units, in double: half a step of rounding is all that is left
      const R g = (fma(r.t0, r.d[i], r.o[i]) - (R)m.qorigin[i]) * (R)m.qinv[i];
      r.oi[i] = (B)((g + (R)8388608.0) * (R)sa);
    }
    r.inv[i] = sa;
    r.nsel[i] = sa >= (B)0 ? 0x7610u : 0x7632u;
  }
}

// A 16-bit coordinate of word w (the half that selector sel picks) as the float 2^23 + q (exact).
__device__ __forceinline__ float grid_q(uint32_t w, uint32_t sel) {
  return __int_as_float((int)__byte_perm(w, 0x4B000000u, sel));
}

// Resumable traversal of one ray, organised as in Aila & Laine's
// "while-while" scheme with speculative traversal: a warp steps through inner
// nodes until every searching lane holds a leaf, then all of them test their
// leaves together, so node visits and triangle tests run in separate, mostly
// converged loops.  A lane that found a leaf postpones it and keeps descending
// while other lanes are still searching.
constexpr int kDone = (int)0x80000000;  // no valid leaf code: first + count would exceed 2^24

// Traversal stack entry of binary trees: a stacked child and its entry distance
// (float in both precisions: it is the box tests'), one 8-byte local-memory access
// per push and per pop (two 4-byte arrays took two).  The pool kernel with its first
// four entries in shared memory instead, and so a branch at each access and less L1:
// cylinder sweep 91.8 -> 92.7 ms, hemisphere 6.55 -> 6.59, moments 3.44 -> 3.48,
// attitude sweep 185.4 -> 186.8.
struct __align__(8) StackE { int node; float t; };
__device__ __forceinline__ void stack_put(StackE* s, int i, int node, float t) {
  *reinterpret_cast<int2*>(s + i) = make_int2(node, __float_as_int(t));
}
__device__ __forceinline__ void stack_get(const StackE* s, int i, int& node, float& t) {
  const int2 v = *reinterpret_cast<const int2*>(s + i);
  node = v.x;
  t = __int_as_float(v.y);
}

template <typename R, typename B = R>
struct Trav {
  R tbest;
  B tcull;   // B != R: not below tbest - t0 (B == R: tbest itself is compared)
  uint32_t best;
  int cur;   // inner node >= 0; a leaf found while one is postponed (< 0); kDone when the stack is empty
  int leaf;  // postponed leaf (< 0), or 0 for none
  int sp;
};

template <typename R, typename B>
__device__ __forceinline__ B trav_cull(const Trav<R, B>& t) {
  if constexpr (std::is_same_v<R, B>) return t.tbest;
  else return t.tcull;
}

template <typename R, typename B>
__device__ __forceinline__ void trav_begin(Trav<R, B>& t) {
  t.tbest = (R)CUDART_INF;
  if constexpr (!std::is_same_v<R, B>) t.tcull = (B)CUDART_INF;
  t.best = 0xFFFFFFFFu;
  t.cur = 0;
  t.leaf = 0;
  t.sp = 0;
}

// Next stacked candidate whose entry distance is still below the best hit.
template <typename R, typename B>
__device__ __forceinline__ int trav_pop(Trav<R, B>& t, StackE* stack) {
  while (t.sp > 0) {
    --t.sp;
    int node;
    B te;
    stack_get(stack, t.sp, node, te);
    if (te <= trav_cull(t)) return node;
  }
  return kDone;
}

// One inner node: test both children, continue with the nearer hit child,
// stack the farther one; the first leaf reached is postponed.  STAGE: nodes
// below n_stage come from the copy in shared memory.
template <bool STAGE, typename R, typename B>
__device__ __forceinline__ void trav_inner(const MeshDev& m, const float4* __restrict__ s_nodes, uint32_t n_stage,
                                           const Ray<R, B>& r, Trav<R, B>& t, StackE* stack,
                                           uint32_t& n_nodes) {
  ++n_nodes;
  float4 n0, n1;
  if (STAGE && (uint32_t)t.cur < n_stage) {
    n0 = s_nodes[2 * t.cur]; n1 = s_nodes[2 * t.cur + 1];
  } else {
    const float4* g = m.nodes + 2 * (size_t)t.cur;
    n0 = __ldg(g); n1 = __ldg(g + 1);
  }
  // child 0: x, y, z words n0.x, n0.y, n0.z; child 1: n0.w, n1.x, n1.y; child codes n1.z, n1.w
  const uint32_t w[6] = {__float_as_uint(n0.x), __float_as_uint(n0.y), __float_as_uint(n0.z),
                         __float_as_uint(n0.w), __float_as_uint(n1.x), __float_as_uint(n1.y)};
  B tn[2][3], tf[2][3];
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      tn[c][a] = fma((B)grid_q(w[3 * c + a], r.nsel[a]), r.inv[a], -r.oi[a]);
      tf[c][a] = fma((B)grid_q(w[3 * c + a], r.nsel[a] ^ 0x22u), r.inv[a], -r.oi[a]);
    }
  B tnear = (B)0;
  if constexpr (std::is_same_v<R, B>) tnear = r.tlo;
  else tnear = r.tnear;
  const B tmin0 = max3(tn[0][0], tn[0][1], fmax(tn[0][2], tnear));
  B tmax0 = min3(tf[0][0], tf[0][1], fmin(tf[0][2], trav_cull(t)));
  const B tmin1 = max3(tn[1][0], tn[1][1], fmax(tn[1][2], tnear));
  B tmax1 = min3(tf[1][0], tf[1][1], fmin(tf[1][2], trav_cull(t)));
  if constexpr (!std::is_same_v<R, B>) {  // the slopes' rounding, 1e-7 of each distance
    tmax0 = fma(fabs(tmax0), (B)1e-6, tmax0);
    tmax1 = fma(fabs(tmax1), (B)1e-6, tmax1);
  }
  const bool h0 = tmin0 <= tmax0, h1 = tmin1 <= tmax1;
  const int c0 = __float_as_int(n1.z), c1 = __float_as_int(n1.w);
  // the nearer hit child next, the farther one of two on the stack (which holds
  // at most one entry a level: the builder keeps the depth below its size)
  const bool second = h0 && h1 ? tmin1 < tmin0 : h1;
  if (h0 && h1) {
    stack_put(stack, t.sp, second ? c0 : c1, second ? tmin0 : tmin1);
    ++t.sp;
  }
  t.cur = second ? c1 : c0;
  // A leaf is postponed when none is; then, or when nothing was hit, the next
  // candidate of the stack whose entry distance is still below the best hit.  One
  // loop for both, which ends as each turn takes an entry off: two calls of
  // trav_pop took the hemisphere 6.67 ms instead of 6.59, moments 3.51 and 3.49
  // (branches and their barriers are a quarter of the trace kernel's instructions).
  bool next = !h0 && !h1;
  if (!next && t.cur < 0 && t.leaf == 0) {
    t.leaf = t.cur;
    next = true;
  }
  while (next) {
    if (t.sp == 0) {
      t.cur = kDone;
      break;
    }
    --t.sp;
    B te;
    stack_get(stack, t.sp, t.cur, te);
    if (te <= trav_cull(t)) {
      next = t.cur < 0 && t.leaf == 0;
      if (next) t.leaf = t.cur;
    }
  }
}

// The postponed leaf: test its triangles; then a leaf found meanwhile becomes
// the postponed one.  Returns true when the ray's traversal is finished.
template <typename R, typename B>
__device__ __forceinline__ void trav_leaf(const MeshDev& m, const Ray<R, B>& r, uint32_t last, Trav<R, B>& t,
                                          StackE* stack, uint32_t& n_tris) {
  const uint32_t code = ~(uint32_t)t.leaf;
  const uint32_t first = code & 0xFFFFFFu, count = code >> 24;
  const Shear<R> sh = make_shear<R>(r.d);
  for (uint32_t k = first; k < first + count; ++k) {
    R V0[3], V1[3], V2[3];
    const uint32_t id = TriLoad<R>::load(m, k, V0, V1, V2);
    if (id == last) continue;
    ++n_tris;
    test_triangle<R>(r, sh, V0, V1, V2, id, t.tbest, t.best);
  }
  if constexpr (!std::is_same_v<R, B>) {
    const R rel = t.tbest - r.t0;
    t.tcull = __double2float_ru(rel + 1e-6 * Fn<R>::fabs(rel));
  }
  t.leaf = 0;
  if (t.cur < 0 && t.cur != kDone) {
    t.leaf = t.cur;
    t.cur = trav_pop(t, stack);
  }
}

// ------------------------------------- compressed wide BVH traversal
// The children of a wide node are visited in the order of their slots'
// corners (bit a of a corner: the child lies towards +a) as seen along the
// ray: the corner's bits are flipped on the axes where the ray runs towards
// -a, then read most significant first along the ray's dominant axis, next
// the second, last the third.  A near child thus comes before a far one
// along the axis that matters most, with no sort.  ptab holds each slot's
// visit position (nibble s), stab the slot at each position (nibble p).
template <int W, typename R>
__device__ __forceinline__ void ray_order(Ray<R>& r) {
  const R ax = Fn<R>::fabs(r.d[0]), ay = Fn<R>::fabs(r.d[1]), az = Fn<R>::fabs(r.d[2]);
  const uint32_t flip = (r.d[0] < (R)0 ? 1u : 0u) | (r.d[1] < (R)0 ? 2u : 0u) | (r.d[2] < (R)0 ? 4u : 0u);
  // axes by decreasing |d|
  uint32_t a0 = 0, a1 = 1, a2 = 2;
  {
    R v0 = ax, v1 = ay, v2 = az;
    if (v1 > v0) { const R t = v0; v0 = v1; v1 = t; const uint32_t u = a0; a0 = a1; a1 = u; }
    if (v2 > v1) { const R t = v1; v1 = v2; v2 = t; const uint32_t u = a1; a1 = a2; a2 = u; }
    if (v1 > v0) { const uint32_t u = a0; a0 = a1; a1 = u; }
  }
  uint32_t ptab = 0, stab = 0;
#pragma unroll
  for (uint32_t slot = 0; slot < (uint32_t)W; ++slot) {
    // the slot's corner (kWide4Corner for 4-wide nodes)
    const uint32_t c = W == 8 ? slot : (slot == 0 ? 0u : (slot == 1 ? 3u : (slot == 2 ? 5u : 6u)));
    const uint32_t t = c ^ flip;
    const uint32_t pos = (((t >> a0) & 1u) << 2) | (((t >> a1) & 1u) << 1) | ((t >> a2) & 1u);
    ptab |= pos << (4 * slot);
    stab |= slot << (4 * pos);
  }
  r.ptab = ptab;
  r.stab = stab;
}

// Traversal state of one ray in a wide tree.
//   gx, gy: the current node group, the hit inner children of one node still
//           to visit: gx = child_base | (hit positions << 24), gy = (lower
//           bound on their entry distances, low 8 bits cleared) | imask;
//   tb, tm: triangles to test: tb + k for every bit k of tm.
// A stack entry is a node group (gx, gy), or a postponed triangle group
// (tm, tb | 2^31): a node group's gy is a positive float's bits, bit 31 clear.
template <typename R>
struct TravW {
  R tbest;
  uint32_t best;
  uint32_t gx, gy, tb, tm;
  int sp;
};

constexpr uint32_t kTriEntry = 0x80000000u;

template <typename R>
__device__ __forceinline__ void travw_begin(TravW<R>& t, const Ray<R>& r) {
  t.tbest = (R)CUDART_INF;
  t.best = 0xFFFFFFFFu;
  t.gx = (1u << (r.ptab & 7u)) << 24;  // the root: an inner child in slot 0 of node base 0
  t.gy = 1u;
  t.tb = 0;
  t.tm = 0;
  t.sp = 0;
}

// Next stacked work: a node group whose entry bound is still within the best
// hit becomes the current group; a postponed triangle group becomes the
// triangle mask (only taken when the mask is empty).
template <typename R>
__device__ __forceinline__ void travw_pop(TravW<R>& t, const uint2* stack) {
  while (t.sp > 0) {
    --t.sp;
    const uint2 e = stack[t.sp];
    if (e.y & kTriEntry) {
      t.tm = e.x;
      t.tb = e.y & ~kTriEntry;
      return;
    }
    if ((R)__uint_as_float(e.y & ~0xFFu) <= t.tbest) {
      t.gx = e.x;
      t.gy = e.y;
      return;
    }
  }
}

// Byte k of w as a float, exactly: 2^23 + b built in the bits, then 2^23 taken off.
__device__ __forceinline__ float byte_float(uint32_t w, uint32_t k) {
  return __int_as_float((int)__byte_perm(w, 0x4B000000u, 0x7440u + k)) - 8388608.0f;
}


// Float bound below t (its low 8 bits are cleared to make room for imask).
__device__ __forceinline__ uint32_t t_bits_down(float t) { return __float_as_uint(t) & ~0xFFu; }
__device__ __forceinline__ uint32_t t_bits_down(double t) { return __float_as_uint(__double2float_rd(t)) & ~0xFFu; }

// One node of the group: the next hit child in visit order is fetched and its
// W child boxes tested; the group's other children are stacked.  The hit
// inner children form the new group; the hit leaves' triangles become the
// triangle mask, or, when the lane still holds one (speculative descent),
// a postponed group on the stack.
template <typename R, int W>
__device__ __forceinline__ void travw_node(const MeshDev& m, const Ray<R>& r, TravW<R>& t, uint2* stack,
                                           uint32_t& n_nodes, int* err) {
  constexpr int F4 = W == 8 ? 5 : 4;
  const uint32_t hits = t.gx >> 24;
  const uint32_t pos = __ffs(hits) - 1;
  const uint32_t rest = hits & (hits - 1u);
  const uint32_t slot = (r.stab >> (4 * pos)) & 7u;
  const uint32_t node = (t.gx & 0xFFFFFFu) + __popc(t.gy & 0xFFu & ((1u << slot) - 1u));
  if (rest != 0u) {
    if (t.sp >= kMaxStackW) {
      atomicOr(err, 1);
      t.gx = 0;
      t.tm = 0;
      t.sp = 0;
      return;
    }
    stack[t.sp] = make_uint2((t.gx & 0xFFFFFFu) | (rest << 24), t.gy);
    ++t.sp;
  }
  ++n_nodes;
  float4 v[F4];
  const float4* g = m.nodes + (size_t)F4 * node;
#pragma unroll
  for (int i = 0; i < F4; ++i) v[i] = __ldg(g + i);
  const uint32_t ew = __float_as_uint(v[0].w);
  const uint32_t imask = ew >> 24;
  // per axis: grid step times 1/d, and the grid origin's distance
  R sa[3], oa[3];
  const float p[3] = {v[0].x, v[0].y, v[0].z};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    sa[a] = (R)__uint_as_float(((ew >> (8 * a)) & 0xFFu) << 23) * r.inv[a];
    oa[a] = fma((R)p[a], r.inv[a], -r.oi[a]);
  }
  // plane words (W = 8: two per plane, slots 0-3 then 4-7; W = 4: one per plane)
  constexpr int PP = W == 8 ? 2 : 1;
  uint32_t q[6 * PP];
#pragma unroll
  for (int i = 0; i < 6 * PP; ++i) {
    const float4& f = v[2 + i / 4];
    q[i] = __float_as_uint((i & 3) == 0 ? f.x : ((i & 3) == 1 ? f.y : ((i & 3) == 2 ? f.z : f.w)));
  }
  // near and far planes along each axis: lo first where the ray runs towards +a
  uint32_t qn[3][PP], qf[3][PP];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const bool pos_dir = r.inv[a] >= (R)0;
#pragma unroll
    for (int h = 0; h < PP; ++h) {
      const uint32_t lo = q[PP * a + h], hi = q[PP * (a + 3) + h];
      qn[a][h] = pos_dir ? lo : hi;
      qf[a][h] = pos_dir ? hi : lo;
    }
  }
  uint32_t hitbits = 0;
  R tmin_hit = (R)CUDART_INF;
#pragma unroll
  for (int s = 0; s < W; ++s) {
    const int h = s >> 2, k = s & 3;
    const R tn = max3(max3(fma((R)byte_float(qn[0][h], k), sa[0], oa[0]), fma((R)byte_float(qn[1][h], k), sa[1], oa[1]),
                           fma((R)byte_float(qn[2][h], k), sa[2], oa[2])), r.tlo, r.tlo);
    const R tf = min3(fma((R)byte_float(qf[0][h], k), sa[0], oa[0]), fma((R)byte_float(qf[1][h], k), sa[1], oa[1]),
                      min3(fma((R)byte_float(qf[2][h], k), sa[2], oa[2]), t.tbest, t.tbest));
    const bool hit = tn <= tf;
    hitbits |= hit ? (1u << s) : 0u;
    tmin_hit = fmin(tmin_hit, hit ? tn : (R)CUDART_INF);
  }
  // hit inner children by visit position; hit leaves' triangles
  uint32_t inner = hitbits & imask, new_hits = 0;
  while (inner != 0u) {
    const uint32_t s = __ffs(inner) - 1;
    inner &= inner - 1u;
    new_hits |= 1u << ((r.ptab >> (4 * s)) & 7u);
  }
  uint32_t leaves = hitbits & ~imask, tris = 0;
  const uint32_t meta0 = __float_as_uint(v[1].z), meta1 = __float_as_uint(v[1].w);
  while (leaves != 0u) {
    const uint32_t s = __ffs(leaves) - 1;
    leaves &= leaves - 1u;
    const uint32_t meta = ((s < 4 ? meta0 : meta1) >> (8 * (s & 3u))) & 0xFFu;
    tris |= (0xFu >> (3u - (meta >> 5))) << (meta & 31u);
  }
  t.gx = __float_as_uint(v[1].x) | (new_hits << 24);
  t.gy = t_bits_down(tmin_hit) | imask;
  if (tris != 0u) {
    if (t.tm == 0u) {
      t.tb = __float_as_uint(v[1].y);
      t.tm = tris;
    } else if (t.sp < kMaxStackW) {  // speculative step: postpone these triangles
      stack[t.sp] = make_uint2(tris, __float_as_uint(v[1].y) | kTriEntry);
      ++t.sp;
    } else {
      atomicOr(err, 1);
      t.gx = 0;
      t.tm = 0;
      t.sp = 0;
    }
  }
}

// Triangles of the mask (a node's hit leaves), in any order: nearest t wins.
template <typename R>
__device__ __forceinline__ void travw_tris(const MeshDev& m, const Ray<R>& r, uint32_t last, TravW<R>& t,
                                           uint32_t& n_tris) {
  const Shear<R> sh = make_shear<R>(r.d);
  while (t.tm != 0u) {
    const uint32_t k = __ffs(t.tm) - 1;
    t.tm &= t.tm - 1u;
    R V0[3], V1[3], V2[3];
    const uint32_t id = TriLoad<R>::load(m, t.tb + k, V0, V1, V2);
    if (id == last) continue;
    ++n_tris;
    test_triangle<R>(r, sh, V0, V1, V2, id, t.tbest, t.best);
  }
}

// ------------------------------------------------ re-emission (§II.A)
template <typename R> struct Frame;
// A triangle's frame, and its exposed sides (bit 0: the side n points to,
// bit 1: the other): sides that the whole mesh lies behind.
template <> struct Frame<float> {
  static __device__ __forceinline__ uint32_t load(const MeshDev& m, uint32_t id, float n[3], float t1[3]) {
    const float4 a = __ldg(&m.frames[2 * id]), b = __ldg(&m.frames[2 * id + 1]);
    n[0] = a.x; n[1] = a.y; n[2] = a.z;
    t1[0] = b.x; t1[1] = b.y; t1[2] = b.z;
    return __float_as_uint(b.w);
  }
};
template <> struct Frame<double> {
  static __device__ __forceinline__ uint32_t load(const MeshDev& m, uint32_t id, double n[3], double t1[3]) {
    const double* f = m.frames64 + 8 * (size_t)id;
    n[0] = __ldg(f); n[1] = __ldg(f + 1); n[2] = __ldg(f + 2);
    t1[0] = __ldg(f + 4); t1[1] = __ldg(f + 5); t1[2] = __ldg(f + 6);
    return (uint32_t)__ldg(f + 7);
  }
};

// Maxwell model: with probability eps diffuse re-emission from the
// flux-weighted half-range Maxwellian at T_W about the hit-side normal
// (normal speed c_W sqrt(-ln u1), tangential c_W sqrt(-ln u2) at angle 2 pi u3
// in the frame (t1, n x t1)); otherwise specular reflection.
template <typename R> struct CllC;
template <> struct CllC<float> {
  static __device__ __forceinline__ float get(const QueryDev& q, int k) { return q.fcll[k]; }
};
template <> struct CllC<double> {
  static __device__ __forceinline__ double get(const QueryDev& q, int k) { return q.cll[k]; }
};

// Cercignani-Lampis-Lord re-emission (Lord's sampling of the CL kernel), in
// units of c_W about the hit-side normal n_out (sgn n): with the incident
// normal speed v_n and tangential components (v_t1, v_t2) along (t1, n x t1),
//   r = sqrt(-alpha_n ln u0), theta = 2 pi u1,
//   v_n' = sqrt(r^2 + (1 - alpha_n) v_n^2 + 2 r sqrt(1 - alpha_n) v_n cos theta),
//   rho = sqrt(-alpha_t ln u2), phi = 2 pi u3,
//   v_t' = sqrt(1 - alpha_t) v_t + rho (cos phi, sin phi).
template <typename R>
__device__ __forceinline__ void reemit_cll(const QueryDev& q, R cw, const uint4& w, R sgn, const R n[3],
                                           const R t1[3], R v[3]) {
  const R t2[3] = {n[1] * t1[2] - n[2] * t1[1], n[2] * t1[0] - n[0] * t1[2], n[0] * t1[1] - n[1] * t1[0]};
  const R inv_cw = (R)1 / cw;
  const R vn = -sgn * (v[0] * n[0] + v[1] * n[1] + v[2] * n[2]) * inv_cw;
  const R vt1 = (v[0] * t1[0] + v[1] * t1[1] + v[2] * t1[2]) * inv_cw;
  const R vt2 = (v[0] * t2[0] + v[1] * t2[1] + v[2] * t2[2]) * inv_cw;
  const R r = Fn<R>::sqrt(-CllC<R>::get(q, 0) * Fn<R>::log(uniform<R>(w.x)));
  R st, ct;
  Fn<R>::sincospi((R)2 * uniform<R>(w.y), &st, &ct);
  const R b = CllC<R>::get(q, 1) * vn;
  const R vn_out = Fn<R>::sqrt(fmax(r * r + b * b + (R)2 * r * b * ct, (R)0));
  const R rho = Fn<R>::sqrt(-CllC<R>::get(q, 2) * Fn<R>::log(uniform<R>(w.z)));
  R sp, cp;
  Fn<R>::sincospi((R)2 * uniform<R>(w.w), &sp, &cp);
  const R a1 = CllC<R>::get(q, 3) * vt1 + rho * cp, a2 = CllC<R>::get(q, 3) * vt2 + rho * sp;
#pragma unroll
  for (int i = 0; i < 3; ++i) v[i] = cw * (sgn * vn_out * n[i] + a1 * t1[i] + a2 * t2[i]);
}

// CLL: compiled into the kernel variants that serve launches holding a CLL query.
template <typename R, bool CLL>
__device__ __forceinline__ void reemit(const QueryDev& q, R cw, uint64_t pid, uint32_t bounce, const R n[3],
                                       const R t1[3], R v[3]) {
  const uint4 w = draws(q, pid, 2 + bounce);
  const R vdn = v[0] * n[0] + v[1] * n[1] + v[2] * n[2];
  if constexpr (CLL) {
    if (q.gsi_model == TPMC_GSI_CLL) {
      reemit_cll<R>(q, cw, w, vdn < (R)0 ? (R)1 : (R)-1, n, t1, v);
      return;
    }
  }
  if ((w.x >> 9) < q.eps_k) {  // u < eps, decided on the integer behind u
    const R sgn = vdn < (R)0 ? (R)1 : (R)-1;
    const R vn = cw * Fn<R>::sqrt(-Fn<R>::log(uniform<R>(w.y)));
    const R vt = cw * Fn<R>::sqrt(-Fn<R>::log(uniform<R>(w.z)));
    R s, co;
    Fn<R>::sincospi((R)2 * uniform<R>(w.w), &s, &co);
    const R t2[3] = {n[1] * t1[2] - n[2] * t1[1], n[2] * t1[0] - n[0] * t1[2], n[0] * t1[1] - n[1] * t1[0]};
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = sgn * vn * n[i] + vt * (co * t1[i] + s * t2[i]);
  } else {
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = v[i] - (R)2 * vdn * n[i];
  }
}

__device__ __forceinline__ long long quantize(float x) { return __float2ll_rn(x); }
__device__ __forceinline__ long long quantize(double x) { return __double2ll_rn(x); }

// Per-lane partial sums for the query the lane is working on.  They live in
// shared memory (one slot per thread), which keeps them out of the registers
// the traversal needs.
// d2lo and d2hi hold the lane's sum of squared drag contributions as the
// 96-bit integer d2hi 2^64 + d2lo (units of the query's quantum2).
struct LaneAcc {
  long long F[3], T[3];
  unsigned long long d2lo;
  uint32_t hits, hit_particles, truncated, particles;
  int q;
  uint32_t d2hi;
  // the lane's particle: its id (bits 0-39) and the hits so far (bits 40-63),
  // kept here rather than in registers the traversal loop needs
  unsigned long long pb;
};

__device__ __forceinline__ void lane_reset(LaneAcc& a, int q) {
#pragma unroll
  for (int i = 0; i < 3; ++i) { a.F[i] = 0; a.T[i] = 0; }
  a.hits = a.hit_particles = a.truncated = a.particles = 0;
  a.d2lo = 0;
  a.d2hi = 0;
  a.q = q;
}

// Adds one particle's squared drag contribution d^2 (c_mp^2 units), rounded to
// the query's quantum2; the set-up bounds every particle's term below 2^62.
__device__ __forceinline__ unsigned long long quantize_sq(float x) { return __float2ull_rn(x); }
__device__ __forceinline__ unsigned long long quantize_sq(double x) { return __double2ull_rn(x); }
__device__ __forceinline__ void lane_add_d2(LaneAcc& a, unsigned long long x) {
  const unsigned long long lo = a.d2lo + x;
  a.d2hi += lo < x ? 1u : 0u;
  a.d2lo = lo;
}

// Adds the 96-bit sum hi 2^64 + lo of one flush to the three limbs of the
// stripe's squared-drag sum: bits 0-29, bits 30-59, and hi 2^4 + (lo >> 60).
// A flush whose sum is not 0 carries at least one finished particle and a query
// has at most 2^34, so each low limb stays below 2^34 2^30 = 2^64; the top limb
// stays below the exact total over 2^60, which is below 2^36 (each particle's term
// is below 2^62).
__device__ __forceinline__ void add_d2(AccStripe& A, unsigned long long lo, unsigned long long hi) {
  constexpr unsigned long long kM30 = (1ull << 30) - 1ull;
  const unsigned long long l0 = lo & kM30, l1 = (lo >> 30) & kM30, l2 = (hi << 4) | (lo >> 60);
  if (l0) atomicAdd(&A.d2[0], l0);
  if (l1) atomicAdd(&A.d2[1], l1);
  if (l2) atomicAdd(&A.d2[2], l2);
}

// The stripe of a query's sums that this warp adds to.
__device__ __forceinline__ int acc_stripe() {
  return (int)((blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) & (unsigned)(kAccStripes - 1));
}

// Adds the warp's sums to their queries and clears them; the whole warp calls it:
// when a lane with sums is about to take a particle of another query, and at the
// end.  The lanes of each query add up by butterflies of shuffles (the sum of
// squares with its carry) and one lane per word issues the atomic.  Integer sums,
// so the result does not depend on the order.  Lanes that flushed by themselves
// put 13 atomics each on the query's few lines, and a lane without a particle (a
// launch's last warps hold many) made all 32 do so: 60 ns a warp, 270 us of a
// 131,072-particle launch on the cylinder, now 50.  Queries are taken one after the
// other; with very many of a few particles each, where a warp holds up to 32, that
// is no slower: 65,536 queries of 1, 4, 16 and 63 particles on the cylinder 64.7 to
// 65.4 -> 7.5 to 8.3 ms a call, 2^20 of 1 and of 8 1,031 -> 120 (set-up included).
__device__ __noinline__ void warp_flush(AccStripe* acc, uint32_t stride, LaneAcc& a, int stripe) {
  const uint32_t lane = threadIdx.x & 31u;
  unsigned todo = __ballot_sync(kFull, a.q >= 0 && a.particles + a.hits > 0);
  while (todo != 0u) {
    const int q0 = __shfl_sync(kFull, a.q, __ffs(todo) - 1);
    const bool in = a.q == q0;
    AccStripe& A = acc[(size_t)stripe * stride + q0];
    unsigned long long mine = 0ull;  // the first ten words of a stripe
#pragma unroll
    for (int i = 0; i < 10; ++i) {
      unsigned long long v = 0ull;
      if (in)
        v = i < 3   ? (unsigned long long)a.F[i]
            : i < 6 ? (unsigned long long)a.T[i - 3]
                    : (i == 6 ? a.hits : (i == 7 ? a.hit_particles : (i == 8 ? a.truncated : a.particles)));
#pragma unroll
      for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(kFull, v, m);
      if (lane == (uint32_t)i) mine = v;
    }
    unsigned long long lo = in ? a.d2lo : 0ull, hi = in ? a.d2hi : 0ull;
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      const unsigned long long olo = __shfl_xor_sync(kFull, lo, m), ohi = __shfl_xor_sync(kFull, hi, m);
      const unsigned long long nlo = lo + olo;
      hi += ohi + (nlo < lo ? 1ull : 0ull);
      lo = nlo;
    }
    if (lane < 10 && mine != 0ull) atomicAdd(reinterpret_cast<unsigned long long*>(&A) + lane, mine);
    if (lane == 10) add_d2(A, lo, hi);
    if (in) lane_reset(a, a.q);
    todo &= ~__ballot_sync(kFull, in);
  }
}
static_assert(offsetof(AccStripe, particles) == 9 * 8, "warp_flush writes a stripe's first ten words");

__device__ __forceinline__ void work_flush(AccStripe* acc, uint32_t stride, int q, uint32_t n_nodes, uint32_t n_tris,
                                           int stripe) {
  if (q < 0) return;
  AccStripe& A = acc[(size_t)stripe * stride + q];
  if (n_nodes) atomicAdd(&A.nodes, (unsigned long long)n_nodes);
  if (n_tris) atomicAdd(&A.tris, (unsigned long long)n_tris);
}

// Work index g -> item (binary search over item starts).  Plain loads: the
// set-up may write the items after this kernel has been launched.
__device__ __forceinline__ uint32_t find_item(const ItemDev* items, uint32_t n_items, uint64_t g) {
  uint32_t lo = 0, hi = n_items;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (items[mid].g_begin <= g) lo = mid; else hi = mid;
  }
  return lo;
}

// Per-query constants of the traced (not seeded) part, in the path's precision.
template <typename R> struct HitConst;
template <> struct HitConst<float> {
  static __device__ __forceinline__ float cw(const QueryDev& q) { return q.fc[kFcCw]; }
  static __device__ __forceinline__ float scale(const QueryDev& q) { return q.fc[kFcScale]; }
  static __device__ __forceinline__ float ref(const QueryDev& q, int i) { return q.fc[kFcRef + i]; }
  static __device__ __forceinline__ float vhat(const QueryDev& q, int i) { return q.fc[kFcVhat + i]; }
  static __device__ __forceinline__ float scale2(const QueryDev& q) { return q.fc[kFcScale2]; }
};
template <> struct HitConst<double> {
  static __device__ __forceinline__ double cw(const QueryDev& q) { return q.cw; }
  static __device__ __forceinline__ double scale(const QueryDev& q) { return 1.0 / q.quantum; }
  static __device__ __forceinline__ double ref(const QueryDev& q, int i) { return q.ref[i]; }
  static __device__ __forceinline__ double vhat(const QueryDev& q, int i) { return q.vhat[i]; }
  static __device__ __forceinline__ double scale2(const QueryDev& q) { return 1.0 / q.quantum2; }
};

// A seeded particle waiting in its warp's queue (shared memory).
template <typename R>
struct alignas(sizeof(R) == 4 ? 16 : 8) Seeded {
  R pos[3], vel[3];
  uint64_t pq;  // particle id in bits 0-39, query slot above
};
static_assert(sizeof(Seeded<float>) == 32, "a float queue slot is two 16-byte vectors");

// Float slots are written and read as two 16-byte vectors: eight lanes'
// 16-byte accesses at a 32-byte stride take two shared-memory wavefronts,
// where 4-byte fields at that stride would conflict eight ways.
// STREAM: pool entries, written once and read once (they leave the L2 to the mesh).
template <typename R, bool STREAM = false>
__device__ __forceinline__ void slot_store(Seeded<R>& e, const R pos[3], const R vel[3], uint64_t pq) {
  if constexpr (sizeof(R) == 4) {
    float4* v = reinterpret_cast<float4*>(&e);
    const float4 v0 = make_float4(pos[0], pos[1], pos[2], vel[0]);
    const float4 v1 = make_float4(vel[1], vel[2], __uint_as_float((uint32_t)pq), __uint_as_float((uint32_t)(pq >> 32)));
    if constexpr (STREAM) {
      __stcs(v, v0);
      __stcs(v + 1, v1);
    } else {
      v[0] = v0;
      v[1] = v1;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 3; ++i) { e.pos[i] = pos[i]; e.vel[i] = vel[i]; }
    e.pq = pq;
  }
}

template <typename R, bool STREAM = false>
__device__ __forceinline__ uint64_t slot_load(const Seeded<R>& e, R pos[3], R vel[3]) {
  if constexpr (sizeof(R) == 4) {
    const float4* v = reinterpret_cast<const float4*>(&e);
    const float4 a = STREAM ? __ldcs(v) : v[0], b = STREAM ? __ldcs(v + 1) : v[1];
    pos[0] = a.x; pos[1] = a.y; pos[2] = a.z;
    vel[0] = a.w; vel[1] = b.x; vel[2] = b.y;
    return (uint64_t)__float_as_uint(b.z) | ((uint64_t)__float_as_uint(b.w) << 32);
  } else {
#pragma unroll
    for (int i = 0; i < 3; ++i) { pos[i] = e.pos[i]; vel[i] = e.vel[i]; }
    return e.pq;
  }
}

constexpr uint32_t kQueue = 64;     // queue slots per warp (two seeding batches)

// Particles of query q that missed, added to its count.
__device__ __forceinline__ void add_missed(const TraceArgs& a, int q, uint32_t n, int stripe) {
  if (q >= 0 && n > 0)
    atomicAdd(&a.acc[(size_t)stripe * a.acc_stride + q].particles, (unsigned long long)n);
}

// Whether the ray may meet the mesh: one of its front boxes beyond tlo.  Slab
// distances about a box's centre (one FMA for the centre, two for the planes),
// so that only the final comparisons use the ALU pipe.  A ray rejected here
// misses every triangle: the boxes are padded beyond the rounding (tpmc_internal.h).
// WIDER: of the boxes widened by `margin` metres.
template <int W, bool WIDER, typename R>
__device__ __forceinline__ bool meets_front(const MeshDev& m, const float* __restrict__ front, const R pos[3],
                                            const R vel[3], float margin = 0.0f) {
  float inv[3], oi[3], ainv[3];
  bool far = false;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float o = (float)pos[i], d = (float)vel[i];
    const float di = fabsf(d) < 1e-30f ? copysignf(1e-30f, d) : d;
    const float v = Fn<float>::rcp(di);
    if constexpr (W == 2) {  // grid units, as ray_to_grid
      inv[i] = m.qstep[i] * v;
      oi[i] = fmaf(8388608.0f, inv[i], -fmaf(m.qorigin[i], v, -o * v));
    } else {
      inv[i] = v;
      oi[i] = o * v;
    }
    ainv[i] = fabsf(inv[i]);
    far = far || !(fabsf(oi[i]) <= m.front_reach[i] * ainv[i]);
  }
  if (far) return m.n_front > 0;
  [[maybe_unused]] float w[3];  // the margin in distances along the ray
#pragma unroll
  for (int i = 0; i < 3; ++i) w[i] = W == 2 ? margin * (ainv[i] * m.qinv[i]) : margin * ainv[i];
  bool meet = false;
  for (uint32_t k = 0; k < m.n_front; ++k) {
    const float* f = front + 8 * k;
    const float4 c = *reinterpret_cast<const float4*>(f);
    const float2 h = *reinterpret_cast<const float2*>(f + 4);
    const float tx = fmaf(c.x, inv[0], -oi[0]), ty = fmaf(c.y, inv[1], -oi[1]), tz = fmaf(c.z, inv[2], -oi[2]);
    float tn, tf;
    if constexpr (WIDER) {
      const float hx = fmaf(c.w, ainv[0], w[0]), hy = fmaf(h.x, ainv[1], w[1]), hz = fmaf(h.y, ainv[2], w[2]);
      tn = max3(tx - hx, ty - hy, tz - hz);
      tf = min3(tx + hx, ty + hy, tz + hz);
    } else {
      tn = max3(fmaf(-c.w, ainv[0], tx), fmaf(-h.x, ainv[1], ty), fmaf(-h.y, ainv[2], tz));
      tf = min3(fmaf(c.w, ainv[0], tx), fmaf(h.x, ainv[1], ty), fmaf(h.y, ainv[2], tz));
    }
    meet = meet || (tn <= tf && tf >= 0.0f);
  }
  return meet;
}

// Phi^-1(u) to 4.5e-4 (Hastings' rational approximation; Abramowitz & Stegun
// 26.2.23), with hardware logarithm and square root.
__device__ __forceinline__ float rough_quantile(float u) {
  const float p = fminf(u, 1.0f - u);
  const float t = sqrtf(-2.0f * __logf(p));
  const float n = fmaf(fmaf(0.010328f, t, 0.802853f), t, 2.515517f);
  const float d = fmaf(fmaf(fmaf(0.001308f, t, 0.189269f), t, 1.432788f), t, 1.0f);
  return copysignf(t - __fdividef(n, d), u - 0.5f);
}

// Entry of the normal-speed table at (s, z), s in its range: normal_speed_start without the cases beyond it.
__device__ __forceinline__ float rough_normal_speed(const float* tab, float s, float z) {
  float fi, fj;
  const float fs = fmaf(s, (float)(1.0 / kVnStep), (float)(-kVnSLo / kVnStep));
  const float fz = fmaf(z, (float)(1.0 / kVnStep), (float)(-kZLo / kVnStep));
  const int i = min(max(floor_bits(fs, fi), 0), kVnNS - 2), j = min(max(floor_bits(fz, fj), 0), kVnNZ - 2);
  const float a = fs - fi, b = fz - fj;
  const float* r = tab + i * kVnNZ + j;
  const float lo = fmaf(b, __ldg(r + 1) - __ldg(r), __ldg(r));
  const float hi = fmaf(b, __ldg(r + kVnNZ + 1) - __ldg(r + kVnNZ), __ldg(r + kVnNZ));
  return fmaf(a, hi - lo, lo);
}

// Whether the particle may hit, from a rough copy of its ray: the starts of the
// two inverse-CDF solves without their Newton steps, quantiles to 4.5e-4,
// hardware sines.  The position is off by at most 1.6e-3 CV radii (in arc), the
// normal speed by 2e-3, the tangential radius by 6e-4 (units of c_mp), so the ray
// passes within fc[kFcPreMargin] (set-up) of the true one as long as its speed
// squared is at least fc[kFcPreV2]; slower ones are kept, as is what the start
// table does not cover.  About 410 instructions with the Philox block and the loop
// around it (156 of them), where the exact seeding takes 745.
template <int W>
__device__ __forceinline__ bool may_hit(const QueryDev& q, const TraceArgs& a, const float* front, uint64_t pid,
                                        const uint4& w0) {
  const float margin = q.fc[kFcPreMargin];
  if (!(margin > 0.0f)) return true;
  const float rad = sqrtf(fmaxf(-__logf(uniform<float>(w0.w)), 0.0f));
  const float an = (uniform<float>(angle_word(w0)) - 0.5f) * 6.28318531f;  // the angle less pi
  const float sa = -__sinf(an), ca = -__cosf(an);
  const float zv = rough_quantile(uniform<float>(w0.z));
  float pos[3], vel[3], s;
  if (q.cv_kind == TPMC_CV_SPHERE) {
    const float ux = uniform<float>(w0.x);
    const float f = fmaf(rough_quantile(ux), (float)(kHTable / (kZHi - kZLo)), (float)(-kZLo * kHTable / (kZHi - kZLo)));
    float fl;
    const int j = min(max(floor_bits(f, fl), 0), kHTable - 1);
    const float x0 = __ldg(&q.htab[j]), x = fmaf(f - fl, __ldg(&q.htab[j + 1]) - x0, x0);
    const float cphi = sqrtf(fmaxf((1.0f - x) * (1.0f + x), 0.0f));
    const float th = (uniform<float>(w0.y) - 0.5f) * 6.28318531f;
    const float st = -__sinf(th), ct = -__cosf(th);
    s = q.fc[kFcS] * x;
    const float vn = rough_normal_speed(a.vn_table, s, zv);
    const float vt1 = q.fc[kFcS] * cphi + rad * ca, vt2 = rad * sa;
    const float ps[3] = {cphi * ct, cphi * st, -x};
    const float vr = vt1 * x - vn * cphi;
    const float vs[3] = {vr * ct + vt2 * st, vr * st - vt2 * ct, vn * x + vt1 * cphi};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float* R = &q.fc[kFcR + 3 * i];
      pos[i] = q.fc[kFcCenter + i] + q.fc[kFcRcv] * (R[0] * ps[0] + R[1] * ps[1] + R[2] * ps[2]);
      vel[i] = R[0] * vs[0] + R[1] * vs[1] + R[2] * vs[2];
    }
  } else {
    int f = 0;
#pragma unroll
    for (int k = 0; k < 5; ++k) f += pid >= q.face_end[k] ? 1 : 0;
    const int ax = f >> 1, a1 = ax == 2 ? 0 : ax + 1;
    s = q.fface_s[f];
    const float vn = rough_normal_speed(a.vn_table, s, zv);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float at = i == ax ? ((f & 1) == 0 ? 1.0f : 0.0f) : uniform<float>(i == a1 ? w0.x : w0.y);
      pos[i] = fmaf(at, q.fbox_ext[i], q.fbox_lo[i]);
      vel[i] = i == ax ? ((f & 1) == 0 ? -vn : vn) : fmaf(q.fc[kFcS], q.fc[kFcVhat + i], rad * (i == a1 ? ca : sa));
    }
  }
  const float v2 = vel[0] * vel[0] + vel[1] * vel[1] + vel[2] * vel[2];
  if (!(v2 >= q.fc[kFcPreV2]) || !(s >= -7.9f)) return true;
  return meets_front<W, true, float>(a.mesh, front, pos, vel, margin);
}

// First half of the pool path: a warp seeds one segment of the batch, a.segment
// work indices from a.g0 + segment x a.segment, 32 at a time, and writes the
// particles that may hit to the segment's part of the pool, closed up.
//
// Why the seeding has a kernel of its own: inside the trace kernel its
// temporaries and the queue's state cost the traversal loop its registers (84
// bytes of spills at 64, none now at 56), and warps of one SM in different
// phases evicted each other's instructions (no_instruction was 1.5 to 3.7 of the
// stall cycles per issue, now 0.3).  Here every lane seeds, 745 instructions a
// particle at 85 % of the issue slots, which bound it: 4.1e10 particles/s, where
// the fused kernel on an empty mesh reaches 3.2e10.
//
// PRE: a rough ray (may_hit) decides first, and only the particles that it lets
// through, gathered in shared memory until they fill a warp, are seeded exactly.
// The host takes it when it expects less than 45 % to pass (Ctx::trace_pool):
// 7.4e10 particles/s when none does.
template <int W, typename R, bool PRE>
__global__ void __launch_bounds__(128, 8) seed_kernel(const __grid_constant__ TraceArgs a) {
  __shared__ __align__(16) float s_front[kMaxFront * 8];
  struct Cand {  // a particle that may hit: its Philox block, id and query
    uint4 w0;
    uint64_t pq;
    uint64_t pad;
  };
  __shared__ Cand s_cand[PRE ? 4 * 64 : 1];
  for (uint32_t i = threadIdx.x; i < (uint32_t)kMaxFront * 6u; i += blockDim.x)
    s_front[8 * (i / 6) + i % 6] = a.mesh.front[0][i];
  __syncthreads();
  const uint32_t seg = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31u;
  const uint32_t lt_mask = (1u << lane) - 1u;
  if (seg == 0 && lane == 0) *a.counter = 0;  // the trace kernel's segment counter
  if (seg >= a.n_seg) return;
  const uint64_t first = a.g0 + (uint64_t)seg * a.segment;
  const uint32_t n_idx = (uint32_t)(min(first + a.segment, a.total) - first);
  Seeded<R>* out = reinterpret_cast<Seeded<R>*>(a.pool) + (size_t)seg * a.segment;
  Cand* cand = s_cand + (PRE ? (threadIdx.x >> 5) * 64u : 0u);
  uint32_t n_kept = 0, n_cand = 0, missed = 0;
  // the lane's work item: where it ends and its particle id 0, both from the segment's first index
  uint32_t it_end = 0;
  uint64_t it_pid = 0;
  int it_q = -1;
  // seeds the lane's particle exactly (when it has one) and keeps it if it may hit
  auto seed = [&](bool active, uint64_t pid, int qi, const uint4& w0) {
    bool keep = false;
    R pos[3], vel[3];
    if (active) {
      const QueryDev& q = a.queries[qi];
      QC<R> c;
      c.load(q);
      seed_particle<R>(q, c, a.vn_table, pid, w0, pos, vel);
      keep = meets_front<W, false, R>(a.mesh, s_front, pos, vel);
    }
    const unsigned kept = __ballot_sync(kFull, keep);
    if (keep) slot_store<R, true>(out[n_kept + __popc(kept & lt_mask)], pos, vel, pid | ((uint64_t)qi << kSlotPidBits));
    n_kept += __popc(kept);
    return keep;
  };
  for (uint32_t i0 = 0; i0 < n_idx || (PRE && n_cand > 0); i0 += 32) {
    const uint32_t i = i0 + lane;
    const bool active = i < n_idx;
    uint64_t pid = 0;
    uint4 w0 = make_uint4(0u, 0u, 0u, 0u);
    if (active) {
      if (i >= it_end) {
        const ItemDev item = a.items[find_item(a.items, a.n_items, first + i)];
        it_end = (uint32_t)min(item.g_begin + item.count - first, (uint64_t)n_idx);
        it_pid = item.pid_begin - item.g_begin + first;
        if ((int)item.query != it_q) {
          add_missed(a, it_q, missed, acc_stripe());
          missed = 0;
          it_q = (int)item.query;
        }
      }
      pid = it_pid + i;
      w0 = draws(a.queries[it_q], pid, 0);
    }
    if constexpr (PRE) {
      const bool may = active && may_hit<W>(a.queries[it_q], a, s_front, pid, w0);
      const unsigned m = __ballot_sync(kFull, may);
      if (may) {
        Cand& e = cand[n_cand + __popc(m & lt_mask)];
        e.w0 = w0;
        e.pq = pid | ((uint64_t)it_q << kSlotPidBits);
      }
      missed += active && !may ? 1u : 0u;
      n_cand += __popc(m);
      __syncwarp();
      if (n_cand >= 32u || i0 + 32 >= n_idx) {
        const uint32_t n = min(n_cand, 32u);
        const Cand e = cand[lane];
        const int qi = (int)(e.pq >> kSlotPidBits);
        const bool keep = seed(lane < n, e.pq & ((1ull << kSlotPidBits) - 1), qi, e.w0);
        // a miss counts for its own query, which need not be the lane's item
        if (lane < n && !keep) {
          if (qi == it_q) ++missed;
          else add_missed(a, qi, 1, acc_stripe());
        }
        n_cand -= n;
        __syncwarp();
        if (lane < n_cand) cand[lane] = cand[32u + lane];
        __syncwarp();
      }
    } else {
      const bool keep = seed(active, pid, it_q, w0);
      missed += active && !keep ? 1u : 0u;
    }
  }
  // the misses are particles of their queries all the same
  const int q0 = __shfl_sync(kFull, it_q, 0);
  if (__all_sync(kFull, it_q == q0)) {
    missed = __reduce_add_sync(kFull, missed);
    if (lane == 0) add_missed(a, it_q, missed, acc_stripe());
  } else {
    add_missed(a, it_q, missed, acc_stripe());
  }
  if (lane == 0) a.seg_count[seg] = n_kept;
}

// Seeds particle pid of query qi and, unless it misses the mesh's front boxes,
// puts it into the queue, closed up behind the others of the batch (`mask`: the
// batch's lanes; `at`: the first free slot).  Returns the lanes kept.  Kept out
// of line: the seeding temporaries then do not stay live across the traversal
// loop.
template <int W, typename R, bool COUNT>
__device__ __noinline__ unsigned seed_into(const TraceArgs& a, uint32_t qi, uint64_t pid, Seeded<R>* queue, uint32_t at,
                                           unsigned mask, const float* front) {
  const QueryDev& q = a.queries[qi];
  QC<R> c;
  c.load(q);
  R pos[3], vel[3];
  seed_particle<R>(q, c, a.vn_table, pid, draws(q, pid, 0), pos, vel);
  const bool keep = meets_front<W, false, R>(a.mesh, front, pos, vel);
  const unsigned kept = __ballot_sync(mask, keep);
  if (keep)
    slot_store<R>(queue[(at + __popc(kept & ((1u << (threadIdx.x & 31u)) - 1u))) & (kQueue - 1)], pos, vel,
                  pid | ((uint64_t)qi << kSlotPidBits));
  if constexpr (COUNT) {
    if (a.rec.pos != nullptr) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        a.rec.pos[3 * pid + i] = (double)pos[i];
        a.rec.vel[3 * pid + i] = (double)vel[i];
      }
    }
    if (!keep && a.rec.n_hits != nullptr) {
      a.rec.n_hits[pid] = 0;
      a.rec.truncated[pid] = 0;
#pragma unroll
      for (int i = 0; i < 3; ++i) a.rec.dv[3 * pid + i] = 0.0;
    }
  }
  return kept;
}

// --------------------------------------------------------- trace kernel
// Persistent kernel.  POOL: lanes take particles from the pool that seed_kernel
// filled, a warp fetching a segment at a time.  Otherwise each warp keeps a queue
// of seeded particles in shared memory; when its lanes need particles and the
// queue runs low, all 32 lanes seed one particle each (so the inverse-CDF solves
// run at full warp width).
// Lanes then trace in rounds of resumable traversal steps; a round ends when
// refill_at lanes have finished their rays, and those lanes re-emit (next
// bounce) or finish their particle and take the next one from the queue.
// What bounds it, from the pool: on the cylinder sweep the issue slots (79 % full
// at 35 warps per SM; a round is 15 node steps at 22 lanes, two leaf phases at 15
// and one hit phase at 23), on concave meshes the latency of node loads as well
// (the hemisphere 17 lanes a node step).  Occupancy decides: 8 and 10 blocks per SM
// (64 and 48 registers) take the cylinder sweep 95.5 and 92.7 ms, 9 blocks 91.7.
// MINB > 0: a register-capped instantiation for 128-thread blocks with at
// least MINB resident blocks per SM (more warps to hide latency, at the cost
// of spills inside the out-of-line seeding).  MINB = 0: 256-thread blocks,
// two per SM in float (at most 128 registers), one in double.
template <int W, typename R, typename B, typename TV>
__device__ __forceinline__ void begin_trav(Ray<R, B>& r, TV& tv, const MeshDev& m) {
  if constexpr (W > 2) {
    ray_order<W>(r);
    travw_begin(tv, r);
  } else {
    ray_to_grid(r, m);
    trav_begin(tv);
  }
}

template <typename R, int MINB, bool CLL, int W, bool COUNT, bool POOL>
__global__ void __launch_bounds__(MINB > 0 ? 128 : 256, MINB > 0 ? MINB : (sizeof(R) == 4 ? 2 : 1))
    trace_kernel(TraceArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr uint32_t kNodeF4 = kBinaryNodeF4;  // float4 per binary node
  // only the binary traversal reads staged nodes
  const uint32_t n_stage = W > 2 ? 0u : min(a.smem_nodes, a.mesh.n_nodes);
  float4* s_nodes = reinterpret_cast<float4*>(smem);
  if constexpr (W == 2)
    for (uint32_t i = threadIdx.x; i < kNodeF4 * n_stage; i += blockDim.x) s_nodes[i] = __ldg(&a.mesh.nodes[i]);
  constexpr size_t kQueueBytes = POOL ? 0 : kQueue * sizeof(Seeded<R>);  // per warp
  unsigned char* smem_warps = smem + (size_t)n_stage * kNodeF4 * sizeof(float4);
  Seeded<R>* queue = reinterpret_cast<Seeded<R>*>(smem_warps + (threadIdx.x >> 5) * kQueueBytes);
  LaneAcc& acc = reinterpret_cast<LaneAcc*>(smem_warps + (blockDim.x >> 5) * kQueueBytes)[threadIdx.x];
  __shared__ __align__(16) float s_front[POOL ? 4 : kMaxFront * 8];
  __shared__ uint2 s_missed[POOL ? 1 : 8];  // per warp: query and its particles seeded that miss the mesh
  uint2& missed = s_missed[POOL ? 0 : threadIdx.x >> 5];
  if constexpr (!POOL) {
    for (uint32_t i = threadIdx.x; i < (uint32_t)kMaxFront * 6u; i += blockDim.x)
      s_front[8 * (i / 6) + i % 6] = a.mesh.front[0][i];
    if ((threadIdx.x & 31u) == 0) missed = make_uint2(0u, 0u);
  }
  lane_reset(acc, -1);
  __syncthreads();
  // The set-up may still run (its launch_after, kernels.cu): the mesh's arrays
  // above are complete, queries, items, tables and sums only from here on.
  if constexpr (!POOL) {
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
  }

  const unsigned lane = threadIdx.x & 31u;
  const unsigned lt_mask = (1u << lane) - 1u;

  // warp-uniform state.  Queue ring (its head and fill) and work indices
  // fetched; POOL: the rest of the segment being read, q_count particles from
  // pool index q_head.
  uint32_t q_head = 0, q_count = 0, seg = 0, seg_left = 0;
  uint64_t pool_base = 0;
  uint32_t pool_rem = 0;
  bool drained = false;
  // lane's cached work item (for seeding)
  uint64_t it_g1 = 0, it_off = 0;  // cached item: end of its work range, pid - g
  uint32_t it_q = 0;

  // lane's particle
  // tdone: the ray is finished (binary trees: no postponed leaf and nothing to
  // visit, which holds for lanes without a particle too)
  bool has = false, tdone = true;
  int qi = -1;
  uint32_t last = 0xFFFFFFFFu;
  R dvp[3] = {0, 0, 0};  // the particle's summed momentum change (records only)
  R dpart = 0;           // its drag component, summed over its hits (for sigma)
  using B = std::conditional_t<W == 2, float, R>;  // of the box tests
  Ray<R, B> ray;
  using TV = std::conditional_t<(W > 2), TravW<R>, Trav<R, B>>;
  using SE = std::conditional_t<(W > 2), uint2, StackE>;
  TV tv{};
  if constexpr (W == 2) tv.cur = kDone;  // nothing to do
  SE stack[W > 2 ? kMaxStackW : kMaxStack];
  uint32_t n_nodes = 0, n_tris = 0;

  for (;;) {
    // ---- 1. lanes whose ray is finished: re-emit, or finish the particle
    if constexpr (W == 2) tdone = tv.leaf == 0 && tv.cur == kDone;
    if (has && tdone) {
      const QueryDev& q = a.queries[qi];
      const uint64_t pid = acc.pb & ((1ull << kSlotPidBits) - 1);
      uint32_t bounce = (uint32_t)(acc.pb >> kSlotPidBits);
      bool finish = true;
      if (tv.best != 0xFFFFFFFFu) {
        const uint32_t hit = tv.best;
        R nrm[3], t1[3], hp[3], v_in[3];
        const uint32_t exposed = Frame<R>::load(a.mesh, hit, nrm, t1);
#pragma unroll
        for (int i = 0; i < 3; ++i) { hp[i] = ray.o[i] + tv.tbest * ray.d[i]; v_in[i] = ray.d[i]; }
        R v[3] = {ray.d[0], ray.d[1], ray.d[2]};
        reemit<R, CLL>(q, HitConst<R>::cw(q), pid, bounce, nrm, t1, v);
        R dv[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          dv[i] = v_in[i] - v[i];
          if constexpr (COUNT) dvp[i] += dv[i];
        }
        dpart += dv[0] * HitConst<R>::vhat(q, 0) + dv[1] * HitConst<R>::vhat(q, 1) + dv[2] * HitConst<R>::vhat(q, 2);
        const R r0 = hp[0] - HitConst<R>::ref(q, 0), r1 = hp[1] - HitConst<R>::ref(q, 1),
                r2 = hp[2] - HitConst<R>::ref(q, 2);
        const R tq[3] = {r1 * dv[2] - r2 * dv[1], r2 * dv[0] - r0 * dv[2], r0 * dv[1] - r1 * dv[0]};
        const R sc = HitConst<R>::scale(q);
        long long qf[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          qf[i] = quantize(dv[i] * sc);
          acc.F[i] += qf[i];
          acc.T[i] += quantize(tq[i] * sc);
        }
        long long* panel = q.panel;
        if (panel != nullptr) {
          long long* pp = panel + 3 * (size_t)hit;
#pragma unroll
          for (int i = 0; i < 3; ++i)
            if (qf[i]) atomicAdd(reinterpret_cast<unsigned long long*>(pp + i), (unsigned long long)qf[i]);
        }
        if constexpr (COUNT)
          if (a.rec.tri != nullptr && bounce < a.rec.K) a.rec.tri[(size_t)pid * a.rec.K + bounce] = hit;
        ++acc.hits;
        if (bounce == 0) ++acc.hit_particles;
        ++bounce;
        acc.pb += 1ull << kSlotPidBits;
        last = hit;
        if (bounce >= q.max_bounces) {
          ++acc.truncated;
        } else {
          // The particle leaves from the side it arrived on.  When the whole
          // mesh lies behind that side (to 1e-12 m) and it leaves at more than
          // 0.01 in cos from the plane, nothing lies ahead of it beyond 1e-10 m,
          // inside the shortest hit distance: it is done, without a traversal.
          const R vv = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
          const R vn = v[0] * nrm[0] + v[1] * nrm[1] + v[2] * nrm[2];
          const bool escapes = (exposed & (vn > (R)0 ? 1u : 2u)) != 0u && vn * vn > (R)1e-4 * vv;
          if (!escapes) {
            // the shortest hit distance, 1e-6 m (1e-9 m in double) over the speed
            make_ray(ray, hp, v, (sizeof(R) == 4 ? (R)1e-6 : (R)1e-9) * Fn<R>::rsqrt(vv));
            begin_trav<W>(ray, tv, a.mesh);
            tdone = false;
            finish = false;
          }
        }
      }
      if (finish) {
        if (dpart != (R)0) lane_add_d2(acc, quantize_sq(dpart * dpart * HitConst<R>::scale2(q)));
        ++acc.particles;
        if (COUNT && a.rec.n_hits != nullptr) {
          a.rec.n_hits[pid] = bounce;
          a.rec.truncated[pid] = (tv.best != 0xFFFFFFFFu && bounce >= q.max_bounces) ? 1u : 0u;
#pragma unroll
          for (int i = 0; i < 3; ++i) a.rec.dv[3 * pid + i] = (double)dvp[i];
        }
        has = false;
      }
    }

    // ---- 2. idle lanes take particles from the queue, filled when it runs low, or from the pool
    const unsigned need = __ballot_sync(kFull, !has);
    const uint32_t n_need = __popc(need);
    if (n_need > 0u) {
      if constexpr (POOL) {
        while (q_count == 0 && !drained) {  // the next segment, of a run of them
          // A run of segments at a time, as many as would let every warp fetch four
          // more times (64 at most): with single segments a warp met another query
          // at every fetch of an attitude sweep (its queries held 2,000 segments,
          // the grid 5,472 warps), which took 306 ms instead of 239.
          if (seg_left == 0) {
            unsigned sg = 0;
            const uint32_t left = seg < a.n_seg ? a.n_seg - seg : 0u;
            const uint32_t k = min(64u, left / (4u * gridDim.x * (blockDim.x >> 5)) + 1u);
            if (lane == 0) sg = (unsigned)atomicAdd(a.counter, (unsigned long long)k);
            seg = __shfl_sync(kFull, sg, 0);
            seg_left = k;
          } else {
            ++seg;
          }
          --seg_left;
          drained = seg >= a.n_seg;
          q_count = drained ? 0u : __ldg(&a.seg_count[seg]);
          q_head = seg * a.segment;
        }
      }
      while (!POOL && q_count < n_need && !drained && q_count + 32u <= kQueue) {
        if (pool_rem == 0) {
          unsigned long long base = 0;
          if (lane == 0) base = atomicAdd(a.counter, (unsigned long long)a.chunk);
          base = a.g0 + __shfl_sync(kFull, base, 0);
          if (base >= a.total) {
            drained = true;
            break;
          }
          pool_base = base;
          const uint64_t left = a.total - base;
          pool_rem = left < (uint64_t)a.chunk ? (uint32_t)left : a.chunk;
        }
        const uint32_t nb = min(32u, pool_rem);
        unsigned kept = 0;
        if (lane < nb) {
          const uint64_t g = pool_base + lane;
          if (g >= it_g1) {  // a lane's work indices only grow
            const ItemDev item = a.items[find_item(a.items, a.n_items, g)];
            it_g1 = item.g_begin + item.count;
            it_off = item.pid_begin - item.g_begin;
            it_q = item.query;
          }
          kept = seed_into<W, R, COUNT>(a, it_q, g + it_off, queue, q_head + q_count, kFull >> (32u - nb), s_front);
        }
        kept = __shfl_sync(kFull, kept, 0);
        // the misses: one query's wait in the warp's counter, a mixed batch's are added at once
        const uint32_t q0 = __shfl_sync(kFull, it_q, 0);
        if (__all_sync(kFull, lane >= nb || it_q == q0)) {
          if (lane == 0) {
            uint2 w = missed;
            if (w.x != q0) {
              add_missed(a, (int)w.x, w.y, acc_stripe());
              w = make_uint2(q0, 0u);
            }
            w.y += nb - __popc(kept);
            missed = w;
          }
        } else if (lane < nb && !((kept >> lane) & 1u)) {
          add_missed(a, (int)it_q, 1, acc_stripe());
        }
        pool_base += nb;
        pool_rem -= nb;
        q_count += __popc(kept);
        __syncwarp();
      }
      const uint32_t take = min(n_need, q_count);
      const uint32_t rank = __popc(need & lt_mask);
      {
        // a taking lane with another query: all lanes' sums go out first
        bool sw = false;
        if (((need >> lane) & 1u) && rank < take) {
          const uint64_t pq = POOL ? reinterpret_cast<const Seeded<R>*>(a.pool)[q_head + rank].pq : queue[(q_head + rank) & (kQueue - 1)].pq;
          sw = (int)(pq >> kSlotPidBits) != acc.q && acc.particles + acc.hits > 0;
        }
        if (__any_sync(kFull, sw)) warp_flush(a.acc, a.acc_stride, acc, acc_stripe());
      }
      if (((need >> lane) & 1u) && rank < take) {
        R pos[3], vel[3];
        const uint64_t pq = slot_load<R, POOL>(POOL ? reinterpret_cast<const Seeded<R>*>(a.pool)[q_head + rank]
                                              : queue[(q_head + rank) & (kQueue - 1)], pos, vel);
        const uint64_t pid = pq & ((1ull << kSlotPidBits) - 1);
        const int nq = (int)(pq >> kSlotPidBits);
        if (nq != acc.q) {
          if constexpr (COUNT) {
            work_flush(a.acc, a.acc_stride, acc.q, n_nodes, n_tris, acc_stripe());
            n_nodes = n_tris = 0;
          }
          acc.q = nq;
        }
        qi = nq;
        R t0 = (R)0;
        if constexpr (!std::is_same_v<R, B>) t0 = box_start(a.mesh, pos, vel);
        make_ray(ray, pos, vel,
                 (sizeof(R) == 4 ? (R)1e-6 : (R)1e-9) *
                     Fn<R>::rsqrt(vel[0] * vel[0] + vel[1] * vel[1] + vel[2] * vel[2]), t0);
        begin_trav<W>(ray, tv, a.mesh);
        tdone = false;
        has = true;
        acc.pb = pid;  // no hits yet
        last = 0xFFFFFFFFu;
        dvp[0] = dvp[1] = dvp[2] = (R)0;
        dpart = (R)0;
      }
      q_head = POOL ? q_head + take : (q_head + take) & (kQueue - 1);
      q_count -= take;
      __syncwarp();
    }

    // ---- 3. the warp is done when nothing is in flight and nothing is left to seed
    if (!__any_sync(kFull, has)) {
      if (drained && q_count == 0) break;
      continue;
    }

    // ---- 4. traversal round
    if constexpr (W > 2) {
      // Wide tree: lanes without triangles to test (searching) step through
      // nodes until each holds a triangle mask or has nothing left; lanes
      // that already hold one keep descending meanwhile (speculative), while
      // their stack has room for a postponed triangle group.  Then the
      // triangles.
      for (;;) {
        for (;;) {
          const bool work = has && !tdone;
          const bool search = work && tv.tm == 0u && ((tv.gx >> 24) != 0u || tv.sp > 0);
          if (!__any_sync(kFull, search)) break;
          if (search && (tv.gx >> 24) == 0u) travw_pop(tv, stack);
          const bool step = work && (tv.gx >> 24) != 0u &&
                            (tv.tm == 0u || tv.sp + (int)a.mesh.depth + 2 < kMaxStackW);
          if (step && (search || tv.tm != 0u)) travw_node<R, W>(a.mesh, ray, tv, stack, n_nodes, a.error);
        }
        if (has && !tdone) {
          if (tv.tm != 0u) travw_tris<R>(a.mesh, ray, last, tv, n_tris);
          tdone = (tv.gx >> 24) == 0u && tv.sp == 0;
        }
        const unsigned fin = __ballot_sync(kFull, has && tdone);
        const unsigned run = __ballot_sync(kFull, has && !tdone);
        if (run == 0u || (uint32_t)__popc(fin) >= a.refill_at) break;
      }
      continue;
    } else
    // ---- binary tree: inner nodes until every searching lane holds a leaf
    // (lanes with a leaf keep descending meanwhile), then the leaves
    for (;;) {
      // without staged nodes, the shared-memory check leaves the node loop
      if (n_stage == 0) {
        for (;;) {
          const unsigned searching = __ballot_sync(kFull, tv.cur >= 0 && tv.leaf == 0);
          if (searching == 0u) break;
          // the last few lanes wait while as many others test their leaves: cylinder
          // sweep 98.3 -> 97.5 ms, hemisphere 7.38 -> 7.17, attitude sweep 204.5 -> 197.4
          // (6 lanes: 98.9, 7.14, 197.4; 8: 101.0, 7.21, 198.7)
          if (__popc(searching) < 4 && __popc(__ballot_sync(kFull, tv.leaf != 0)) >= 4) break;
          if (tv.cur >= 0)
            trav_inner<false>(a.mesh, s_nodes, n_stage, ray, tv, stack, n_nodes);
        }
      } else {
        while (__any_sync(kFull, tv.cur >= 0 && tv.leaf == 0)) {
          if (tv.cur >= 0)
            trav_inner<true>(a.mesh, s_nodes, n_stage, ray, tv, stack, n_nodes);
        }
      }
      if (tv.leaf != 0) trav_leaf(a.mesh, ray, last, tv, stack, n_tris);
      const bool ended = tv.leaf == 0 && tv.cur == kDone;  // also lanes without a particle
      const unsigned fin = __ballot_sync(kFull, has && ended);
      const unsigned run = __ballot_sync(kFull, !ended);
      if (run == 0u || (uint32_t)__popc(fin) >= a.refill_at) break;
    }
  }
  if (!POOL && lane == 0) add_missed(a, (int)missed.x, missed.y, acc_stripe());
  if constexpr (COUNT) work_flush(a.acc, a.acc_stride, acc.q, n_nodes, n_tris, acc_stripe());
  warp_flush(a.acc, a.acc_stride, acc, acc_stripe());
}

using TraceFn = void (*)(TraceArgs);

// Kernel instantiation for a schedule: the register-capped float variants serve
// 128-thread blocks.  From the queue: 7 and 8 blocks per SM (64 registers) or 5
// and 6 (80); from the pool: 5 to 9 (56 registers).
template <int W, bool CLL, bool COUNT>
TraceFn pick_trace_t(uint32_t variant, uint32_t block, uint32_t blocks_per_sm) {
  const bool fp64 = (variant & 1u) == TPMC_FP64, small = block <= 128;
  if constexpr (!COUNT) {
    if (variant & kVariantPool) {
      if (small && blocks_per_sm >= 5) return trace_kernel<float, 9, CLL, W, false, true>;
      return trace_kernel<float, 0, CLL, W, false, true>;
    }
  }
  if (fp64) return trace_kernel<double, 0, CLL, W, COUNT, false>;
  if (small && blocks_per_sm >= 7) return trace_kernel<float, 8, CLL, W, COUNT, false>;
  if (small && blocks_per_sm >= 5) return trace_kernel<float, 6, CLL, W, COUNT, false>;
  return trace_kernel<float, 0, CLL, W, COUNT, false>;
}

template <int W>
TraceFn pick_trace_w(uint32_t variant, uint32_t block, uint32_t blocks_per_sm) {
  if (variant & kVariantCount)
    return (variant & kVariantCll) ? pick_trace_t<W, true, true>(variant, block, blocks_per_sm)
                                   : pick_trace_t<W, false, true>(variant, block, blocks_per_sm);
  return (variant & kVariantCll) ? pick_trace_t<W, true, false>(variant, block, blocks_per_sm)
                                 : pick_trace_t<W, false, false>(variant, block, blocks_per_sm);
}

template <int W>
cudaError_t launch_seed_w(const TraceArgs& a, cudaStream_t stream) {
  const uint32_t grid = (a.n_seg + 3) / 4;
  if (a.prefilter) seed_kernel<W, float, true><<<grid, 128, 0, stream>>>(a);
  else seed_kernel<W, float, false><<<grid, 128, 0, stream>>>(a);
  return cudaGetLastError();
}

}  // namespace
}  // namespace tpmc
