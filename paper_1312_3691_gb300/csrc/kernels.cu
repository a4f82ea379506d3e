// CUDA kernels around the trace for sm_103a (GB300), and the launchers.
//
//   setup_kernel     FP64: free-stream set-up per query (Nomenclature; Eq. 10
//                    flux; particle weight, §II.A), Rodrigues matrix (Eq. 15),
//                    fixed-point scale, start table of the latitude inverse CDF.
//   finalize_kernel  FP64 reduction to force, torque, C_D and its error.
//   panels_kernel    FP64 per-triangle pressure and shear.
// Seeding and tracing are in trace.cuh.
#include "trace.cuh"

namespace tpmc {
namespace {

// ---------------------------------------------------------- set-up kernel
// Set-up of query blockIdx.x, spread over the chip: gridDim.y = 1 (one block
// does it all) or kSetupParts (block y = 0: the scalars; the others: the
// latitude start table).  With `base` set, query b is a copy of *base whose
// direction / speed ratio come from dirs[b] / Svals[b] (when given) and whose
// Philox stream is base->stream_id + b; with `items` set, it also writes work
// item b = particles [0, N) of query b at work indices [b N, (b+1) N).
//
// What bounds it is double-precision latency: an SM issues a double warp
// instruction every 16 cycles or so, whether one lane is active or 32, and a
// library function is a chain of 50 to 200 of them.  So independent functions
// run in different warps, arguments of one function (erfc and exp at S, -S and
// the six box faces) in the lanes of one warp, and with few queries the table
// in blocks of its own.  The table's root searches start from a bracket and
// two Newton steps in float, which leaves two to four double evaluations of the
// law per knot; started at 2u - 1 it took up to 54 in the lower tail.  With that
// start, and one thread doing the scalars, a call took 320 us for 8 queries and
// 3.31 ms for 3,072; now 16 us and 0.33 ms.
constexpr int kSetupThreads = 160;
constexpr int kSetupParts = 6;

// The base query comes with the launch (no copy to the device before it), and
// the run's counters and error word (`zero`) are cleared here (no memset).
struct SetupBase {
  QueryDev q;
  uint32_t given;
};

__global__ void __launch_bounds__(kSetupThreads)
    setup_kernel(QueryDev* qs, const __grid_constant__ SetupBase with, const double* dirs, const double* Svals, ItemDev* items,
                 const uint32_t* slots, AccStripe* acc, uint32_t acc_stride, const double* knots, RunWords* zero) {
  cudaTriggerProgrammaticLaunchCompletion();  // see launch_after
  const QueryDev* base = with.given ? &with.q : nullptr;
  if (zero != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < sizeof(RunWords) / 4)
    reinterpret_cast<uint32_t*>(zero)[threadIdx.x] = 0u;
  const uint32_t slot = slots != nullptr ? slots[blockIdx.x] : blockIdx.x;
  QueryDev& q = qs[slot];
  const QueryDev& in = base != nullptr ? *base : q;  // the inputs (T_inf, m, V, dir, ...)
  const bool scalars = blockIdx.y == 0, table = gridDim.y == 1 || blockIdx.y != 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ double s_V, s_S, s_c, s_cw, s_dn, s_vh[3], s_erfc[8], s_exp[8], s_erf, s_erfcx, s_D, s_K1;
  __shared__ int s_st, s_shift_bad;
  __shared__ float s_H[kSetupThreads];

  if (scalars) {
    // the query's sums start at zero: its kAccStripes stripes of 16 words each
    for (uint32_t i = threadIdx.x; i < (uint32_t)kAccStripes * 16u; i += blockDim.x)
      reinterpret_cast<unsigned long long*>(&acc[(size_t)(i >> 4) * acc_stride + slot])[i & 15u] = 0ull;
    if (base != nullptr) {  // all of *base but the start table, which other blocks write
      constexpr uint32_t kTab0 = offsetof(QueryDev, htab) / 4, kTab1 = kTab0 + kHTable + 1;
      for (uint32_t i = threadIdx.x; i < sizeof(QueryDev) / 4; i += blockDim.x)
        if (i < kTab0 || i >= kTab1) reinterpret_cast<uint32_t*>(&q)[i] = reinterpret_cast<const uint32_t*>(base)[i];
      __syncthreads();
    }
  }
  if (threadIdx.x == 0) {
    s_c = sqrt(2.0 * kBoltz * in.T_inf / in.m);
    s_V = Svals != nullptr ? Svals[blockIdx.x] * s_c : in.V;
    s_S = s_V / s_c;
    s_shift_bad = 0;
  } else if (threadIdx.x == 32 && scalars) {
    const double* d = dirs != nullptr ? dirs + 3 * (size_t)blockIdx.x : in.dir;
    const double d0 = d[0], d1 = d[1], d2 = d[2];
    s_dn = sqrt(d0 * d0 + d1 * d1 + d2 * d2);
    s_vh[0] = d0 / s_dn;
    s_vh[1] = d1 / s_dn;
    s_vh[2] = d2 / s_dn;
    if (dirs != nullptr) { q.dir[0] = d0; q.dir[1] = d1; q.dir[2] = d2; }
  } else if (threadIdx.x == 64 && scalars) {
    s_cw = sqrt(q.T_W / q.T_inf);
  } else if (threadIdx.x == 96 && scalars && items != nullptr) {
    ItemDev it;
    it.g_begin = (uint64_t)blockIdx.x * q.N;
    it.pid_begin = 0;
    it.count = q.N;
    it.query = blockIdx.x;
    it.pad = 0;
    items[blockIdx.x] = it;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int st = TPMC_OK;
    if (!(isfinite(s_V) && s_V > 0.0) || (scalars && !(isfinite(s_dn) && s_dn > 0.0))) st = TPMC_EINVAL;
    if (!(s_S >= 0.01 && s_S <= 50.0)) st = TPMC_EINVAL;
    s_st = st;
    if (scalars) {
      if (base != nullptr) q.stream_id = base->stream_id + blockIdx.x;
      if (Svals != nullptr) q.V = s_V;
    }
  }
  __syncthreads();
  const bool sphere = in.cv_kind == TPMC_CV_SPHERE;
  if (s_st != TPMC_OK) {
    if (scalars && threadIdx.x == 0) q.status = s_st;
    if (table && base != nullptr)
      for (int j = threadIdx.x; j <= kHTable; j += blockDim.x) q.htab[j] = 0.0f;
    return;
  }
  const double S = s_S;

  // ---- functions of S and the faces' speed ratios, a warp to each function
  if (warp == 0 && lane < 8) {
    // lane 0: S, lane 1: -S, lanes 2-7: minus the inward-normal speed ratio of each box face
    double a = lane == 0 ? S : -S;
    if (lane >= 2 && scalars) {
      const int f = lane - 2;
      const double v = s_vh[f >> 1];
      a = -(S * (f % 2 == 0 ? -v : v));
    }
    s_erfc[lane] = erfc(a);
    s_exp[lane] = exp(-a * a);
  } else if (warp == 1 && lane == 0) {
    s_erf = erf(S);
  } else if (warp == 2 && lane == 0 && scalars) {
    s_erfcx = erfcx(S);
  } else if (warp == 3 && lane == 0 && scalars) {
    // Eq. 15: rotation about u = z x Vhat by beta = acos(z . Vhat), carrying +z onto Vhat.
    const double* vh = s_vh;
    const double ux = -vh[1], uy = vh[0];  // z x Vhat = (-Vy, Vx, 0)
    const double sb = sqrt(ux * ux + uy * uy);
    const double cb = fmin(1.0, fmax(-1.0, vh[2]));
    double Rm[9];
    if (sb < 1e-12) {
      const double sg = cb > 0.0 ? 1.0 : -1.0;  // identity, or a half turn about x
      Rm[0] = 1; Rm[1] = 0; Rm[2] = 0; Rm[3] = 0; Rm[4] = sg; Rm[5] = 0; Rm[6] = 0; Rm[7] = 0; Rm[8] = sg;
    } else {
      const double kx = ux / sb, ky = uy / sb;  // unit axis (kx, ky, 0)
      const double beta = acos(cb);
      const double cs = cos(beta), sn = sin(beta), oc = 1.0 - cs;
      Rm[0] = cs + kx * kx * oc; Rm[1] = kx * ky * oc;      Rm[2] = ky * sn;
      Rm[3] = kx * ky * oc;      Rm[4] = cs + ky * ky * oc; Rm[5] = -kx * sn;
      Rm[6] = -ky * sn;          Rm[7] = kx * sn;           Rm[8] = cs;
    }
    for (int i = 0; i < 9; ++i) { q.R[i] = Rm[i]; q.fc[kFcR + i] = (float)Rm[i]; }
    for (int i = 0; i < 3; ++i) {
      q.vhat[i] = vh[i];
      q.fc[kFcVhat + i] = (float)vh[i];
      q.fc[kFcCenter + i] = (float)q.center[i];
      q.fc[kFcRef + i] = (float)q.ref[i];
    }
  } else if (warp == 4 && lane == 0 && scalars) {
    // fixed point: worst case |v| <= max(S + 8, 8 c_W/c), so every int64 sum fits for
    // N * max_bounces hits of |dv| <= 2 |v|max and lever arms <= rmax.
    const double vmax = fmax(S + 8.0, 8.0 * s_cw);
    const double bound = (double)q.N * (double)q.max_bounces * 2.0 * 1.7320508075688772 * vmax * fmax(1.0, q.rmax);
    int shift = (int)floor(62.0 - log2(bound));
    shift = min(shift, 32);
    if (shift < 8) s_shift_bad = 1;
    q.shift = shift;
    q.quantum = ldexp(1.0, -shift);
    // squared drag contributions: a particle's |dv . Vhat| <= 2 vmax max_bounces,
    // so each quantised term stays below 2^62; the sum is a 128-bit integer
    const double dmax = 2.0 * vmax * (double)q.max_bounces;
    const int shift2 = max(0, min(32, (int)floor(62.0 - log2(dmax * dmax))));
    q.shift2 = shift2;
    q.quantum2 = ldexp(1.0, -shift2);
    q.fc[kFcScale2] = (float)ldexp(1.0, shift2);
    q.fc[kFcScale] = (float)ldexp(1.0, shift);
    q.fc[kFcS] = (float)S;
    // Rough rays (may_hit): off by `da` radians on the CV, their velocity by da |v|
    // + dv + S dc; emulated over samples of the uniforms, da and dc are at most 1.6e-3 for S
    // below 3.5 and 4.4e-4 above (tests/test_rough_rays.py), dv 2.6e-3.  They pass the body within two CV radii
    // (or the box's diagonal) of the start.  Half as much again is added.
    const double vmin = fmax(0.5, 0.5 * S), da = S < 4.0 ? 1.7e-3 : 4.5e-4, dv = 2.6e-3;
    double margin;
    if (q.cv_kind == TPMC_CV_SPHERE) {
      margin = 1.5 * q.r_cv * (da + 2.0 * (da + (dv + S * da) / vmin));
    } else {
      double d2 = 0.0;
      for (int i = 0; i < 3; ++i) d2 += (q.box_hi[i] - q.box_lo[i]) * (q.box_hi[i] - q.box_lo[i]);
      margin = 1.5 * sqrt(d2) * (1e-5 + dv / vmin);
    }
    q.fc[kFcPreMargin] = S <= 15.9 && q.cv_kind != TPMC_CV_BOX_MAXWELL ? (float)margin : 0.0f;
    q.fc[kFcPreV2] = (float)(vmin * vmin);
    q.fc[kFcCw] = (float)s_cw;
    q.fc[kFcRcv] = (float)q.r_cv;
    q.fc[kFcSqrtpi4S] = (float)(kSqrtPiD / (4.0 * S));
    q.S = S;
    q.c_mp = s_c;
    q.cw = s_cw;
    q.q_inf = 0.5 * q.n * q.m * q.V * q.V;
  }
  __syncthreads();
  const double eS = s_exp[0], erS = s_erf;
  if (threadIdx.x == 0) {
    s_D = eS + kSqrtPiD * (1.0 + 2.0 * S * S) * erS / (2.0 * S);
  } else if (threadIdx.x == 32) {
    s_K1 = kSqrtPiD / (4.0 * S) * (2.0 * S * S + 1.0) * s_erfc[0] - 0.5 * eS;
  }
  __syncthreads();

  if (scalars) {
    if (threadIdx.x == 0) {
      q.Dnorm = s_D;
      q.fc[kFcDinv] = (float)(1.0 / s_D);
      q.status = s_shift_bad ? TPMC_EINVAL : TPMC_OK;
    } else if (threadIdx.x == 32) {
      q.K1 = s_K1;
      q.fc[kFcK1] = (float)s_K1;
      // tail-mass cubics of the latitude law at the poles (see latitude_pole):
      //   x -> +1: h(1) w - h'(1) w^2 / 2 + h''(1) w^3 / 6,  x -> -1: h(-1) w + h'(-1) w^2 / 2 + h''(-1) w^3 / 6,
      //   h(1) = [e^{-S^2} + sqrt(pi) S erfc(-S)] / D,  h(-1) = e^{-S^2} [1 - sqrt(pi) S erfcx(S)] / D,
      //   h'(+-1) = sqrt(pi) S erfc(-+S) / D,  h''(+-1) = 2 S^2 e^{-S^2} / D
      q.fc[kFcPole + 0] = (float)((eS + kSqrtPiD * S * s_erfc[1]) / s_D);
      q.fc[kFcPole + 1] = (float)(-0.5 * kSqrtPiD * S * s_erfc[1] / s_D);
      q.fc[kFcPole + 2] = (float)(S * S * eS / (3.0 * s_D));
    } else if (threadIdx.x == 64) {
      q.fc[kFcPole + 3] = (float)(eS * (1.0 - kSqrtPiD * S * s_erfcx) / s_D);
      q.fc[kFcPole + 4] = (float)(0.5 * kSqrtPiD * S * s_erfc[0] / s_D);
      q.fc[kFcPole + 5] = (float)(S * S * eS / (3.0 * s_D));
    } else if (threadIdx.x == 96) {
      if (sphere) {
        q.gamma = (kSqrtPiD * eS + (CUDART_PI / (2.0 * S) + CUDART_PI * S) * erS) * s_c * q.n * q.r_cv * q.r_cv;
      } else {
        // Rectangular CV (§I, §III.A): face f receives the flat-plate number
        // flux A_f n c G(s_f), G(s) = (e^{-s^2} + sqrt(pi) s erfc(-s)) / (2 sqrt(pi)),
        // and the particle ids up to floor(N C_{f+1}), C the cumulative share.
        double flux[6], total = 0.0;
        for (int f = 0; f < 6; ++f) {
          const int ax = f / 2, a1 = (ax + 1) % 3, a2 = (ax + 2) % 3;
          const double s_f = S * (f % 2 == 0 ? -s_vh[ax] : s_vh[ax]);
          const double area = (q.box_hi[a1] - q.box_lo[a1]) * (q.box_hi[a2] - q.box_lo[a2]);
          flux[f] = area * ((s_exp[2 + f] + kSqrtPiD * s_f * s_erfc[2 + f]) / (2.0 * kSqrtPiD));
          total += flux[f];
          q.face_s[f] = s_f;
          q.fface_s[f] = (float)s_f;
        }
        double cum = 0.0;
        for (int f = 0; f < 6; ++f) {
          cum += flux[f] / total;
          q.face_end[f] = f == 5 ? q.N : (uint64_t)floor((double)q.N * cum);
        }
        for (int i = 0; i < 3; ++i) {
          q.fbox_lo[i] = (float)q.box_lo[i];
          q.fbox_ext[i] = (float)(q.box_hi[i] - q.box_lo[i]);
        }
        q.gamma = total * s_c * q.n;
      }
    }
  }
  if (!table || !sphere) return;  // the latitude table serves the sphere only

  // ---- latitude start table
  const float Sf = (float)S, q4 = (float)(kSqrtPiD / (4.0 * S)), K1f = (float)s_K1, Df = (float)(1.0 / s_D);
  s_H[threadIdx.x] = latitude_cdf<float>(-1.0f + 2.0f * (float)threadIdx.x / (float)(kSetupThreads - 1), Sf, q4, K1f, Df);
  __syncthreads();
  const double K1 = s_K1, q4d = kSqrtPiD / (4.0 * S), Dinv = 1.0 / s_D;
  // neighbouring knots in one warp: their arguments take the same branches of erfc
  const int parts = gridDim.y == 1 ? 1 : (int)gridDim.y - 1, part = gridDim.y == 1 ? 0 : (int)blockIdx.y - 1;
  const int per = (kHTable + parts) / parts;
  const int j = part * per + (int)threadIdx.x;
  if ((int)threadIdx.x < per && j <= kHTable) {
    const double u = knots[j];
    // the grid cell that brackets u, interpolated, then two steps in float (on
    // log H in the lower tail); only a start, so float rounding does not matter
    const float uf = (float)u;
    int k0 = 0, k1 = kSetupThreads - 1;
    while (k1 - k0 > 1) {
      const int mid = (k0 + k1) >> 1;
      if (s_H[mid] <= uf) k0 = mid; else k1 = mid;
    }
    const float x0 = -1.0f + 2.0f * (float)k0 / (float)(kSetupThreads - 1);
    const float x1 = -1.0f + 2.0f * (float)k1 / (float)(kSetupThreads - 1);
    const float h0 = s_H[k0], h1 = s_H[k1];
    const bool tail = uf < 0.0625f && Sf > 1.0f && h0 > 0.0f && h1 > h0;
    const float w = tail ? logf(uf / h0) / logf(h1 / h0) : (h1 > h0 ? (uf - h0) / (h1 - h0) : 0.5f);
    float xf = x0 + (x1 - x0) * fminf(fmaxf(w, 0.0f), 1.0f);
#pragma unroll 1
    for (int it = 0; it < 2; ++it) {
      const float H = latitude_cdf<float>(xf, Sf, q4, K1f, Df), h = latitude_pdf<float>(xf, Sf, Df);
      if (!(H > 0.0f && h > 0.0f)) break;
      const float xn = xf - (tail ? logf(H / uf) * H / h : (H - uf) / h);
      if (xn >= x0 && xn <= x1) xf = xn;
    }
    double lo = -1.0, hi = 1.0, x = xf;
#pragma unroll 1
    for (int it = 0; it < 200; ++it) {
      const double a = S * x, ec = erfc(-a), e = exp(-a * a);
      const double f = (q4d * (2.0 * a * a + 1.0) * ec + 0.5 * x * e - K1) * Dinv - u;
      const double dx = f / ((e + kSqrtPiD * a * ec) * Dinv);
      // Newton squares the error (times at most S^2 here): below 1e-10 this step is the last
      if (fabs(dx) < 1e-10) { x -= dx; break; }
      if (f < 0.0) lo = x; else hi = x;
      x -= dx;
      if (!(x > lo && x < hi)) x = 0.5 * (lo + hi);
    }
    q.htab[j] = (float)x;
  }
}

// The latitude table's uniforms Phi(z_j) (FP64, once per context).
__global__ void knots_kernel(double* knots) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j > kHTable) return;
  const double zj = kZLo + (kZHi - kZLo) * j / kHTable;
  knots[j] = 0.5 * erfc(-zj * 0.70710678118654752440);  // Phi(z_j)
}

// Normal-speed start table (FP64, once per context): entry (i, j) is the
// root of F(x; s_i) = Phi(z_j) by bisection, on the survival function above
// the median (the same law as Eq. 14a; see normal_speed_inverse).
__global__ void vn_table_kernel(float* tab) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= kVnNS * kVnNZ) return;
  const int i = k / kVnNZ, j = k % kVnNZ;
  const double s = kVnSLo + kVnStep * i;
  const double z = kZLo + kVnStep * j;
  const double u = 0.5 * erfc(-z * 0.70710678118654752440);
  const double sp = kSqrtPiD * s;
  const double Z = exp(-s * s) + sp * erfc(-s);
  double lo = 0.0, hi = fmax(s, 0.0) + 12.0;
  for (int it = 0; it < 200; ++it) {
    const double x = 0.5 * (lo + hi);
    if (x <= lo || x >= hi) break;
    const double y = x - s;
    bool below;
    if (u <= 0.5) {
      const double F = (exp(-s * s) - exp(-y * y) + sp * (erfc(-s) - erfc(y))) / Z;
      below = F < u;
    } else {
      const double Q = (exp(-y * y) + sp * erfc(y)) / Z;
      below = Q > 1.0 - u;
    }
    if (below) lo = x; else hi = x;
  }
  tab[k] = (float)(0.5 * (lo + hi));
}

// -------------------------------------------------------- final reduction
// Warp i reduces query slots[i] (or i) into out[i]; the first thread passes the
// trace kernel's error word on (err_out, when given).  Lanes sum the stripes'
// words side by side and compute the components side by side: a chain of double
// divisions and a square root in one thread after 120 loads took 9 us.
__global__ void __launch_bounds__(128)
    finalize_kernel(const QueryDev* qs, const AccStripe* acc, uint32_t stride, uint32_t nq, const uint32_t* slots,
                    tpmc_result* out, const int* err, int* err_out) {
  const uint32_t i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31u;
  cudaGridDependencySynchronize();  // every thread, before its first read: see launch_after
  if (err_out != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *err_out = *err;
  if (i >= nq) return;
  const uint32_t qi = slots != nullptr ? slots[i] : i;
  const QueryDev& q = qs[qi];
  // word (lane & 15) of the stripes; the limbs' sums stay below 2^64 too
  unsigned long long v = 0ull;
#pragma unroll
  for (int j = 0; j < kAccStripes / 2; ++j)
    v += reinterpret_cast<const unsigned long long*>(&acc[(size_t)(2 * j + (lane >> 4)) * stride + qi])[lane & 15u];
  v += __shfl_xor_sync(kFull, v, 16);
  const unsigned long long parts = __shfl_sync(kFull, v, 9);
  // the squared-drag limbs as one exact 128-bit integer
  const unsigned long long l0 = __shfl_sync(kFull, v, 12), l1 = __shfl_sync(kFull, v, 13), l2 = __shfl_sync(kFull, v, 14);
  unsigned long long d2lo = l0 + (l1 << 30), d2hi = (l1 >> 34) + (l2 >> 4) + (d2lo < l0 ? 1ull : 0ull);
  const unsigned long long before = d2lo;
  d2lo += l2 << 60;
  d2hi += d2lo < before ? 1ull : 0ull;
  tpmc_result& res = out[i];
  // every word of the result starts at zero; lanes then write their own parts
  for (uint32_t w = lane; w < sizeof(tpmc_result) / 8; w += 32) reinterpret_cast<unsigned long long*>(&res)[w] = 0ull;
  __syncwarp();
  int status = q.status;
  if (status == TPMC_OK) {
    const double Np = (double)parts;
    // lanes 0-2: force, lanes 3-5: torque; force = (Gamma/N) m c sum(dv) (§II.A)
    const double sum = (double)(long long)v * q.quantum;
    const double scale = Np > 0 ? q.gamma / Np * q.m * q.c_mp : 0.0;
    const double f = scale * sum;
    const double f0 = __shfl_sync(kFull, f, 0), f1 = __shfl_sync(kFull, f, 1), f2 = __shfl_sync(kFull, f, 2);
    const double s0 = __shfl_sync(kFull, sum, 0), s1 = __shfl_sync(kFull, sum, 1), s2 = __shfl_sync(kFull, sum, 2);
    if (lane < 3) {
      res.force[lane] = f;
      res.sum_dv_q[lane] = (long long)v;
      res.CF[lane] = f / (q.q_inf * q.A_ref);
      res.center[lane] = q.center[lane];
    } else if (lane < 6) {
      // force and moment coefficient vectors (the moment about ref over q_inf A_ref l_ref, §III.D.1)
      res.torque[lane - 3] = f;
      res.sum_rdv_q[lane - 3] = (long long)v;
      res.CM[lane - 3] = f / (q.q_inf * q.A_ref * q.l_ref);
    } else if (lane < 12) {
      uint64_t* const counts[6] = {&res.n_hits, &res.n_hit_particles, &res.n_truncated, &res.n_particles,
                                   &res.n_node_visits, &res.n_tri_tests};
#pragma unroll
      for (uint32_t c = 0; c < 6; ++c)
        if (lane == 6 + c) *counts[c] = v;
    } else if (lane == 12) {
      // C_D = F . Vhat / (q_inf A_ref) (Eq. 1)
      res.CD = (f0 * q.vhat[0] + f1 * q.vhat[1] + f2 * q.vhat[2]) / (q.q_inf * q.A_ref);
    } else if (lane == 13) {
      const double mean = Np > 0 ? (s0 * q.vhat[0] + s1 * q.vhat[1] + s2 * q.vhat[2]) / Np : 0.0;
      const double d2 = ((double)d2hi * 18446744073709551616.0 + (double)d2lo) * q.quantum2;
      const double var = Np > 1 ? fmax(0.0, (d2 - Np * mean * mean) / (Np - 1.0)) : 0.0;
      res.CD_sigma = Np > 0 ? q.gamma * q.m * q.c_mp / (q.q_inf * q.A_ref) * sqrt(var / Np) : 0.0;
    } else if (lane == 14) {
      res.S = q.S;
      res.S_W = q.S / q.cw;
      res.gamma = q.gamma;
      res.weight = Np > 0 ? q.gamma / Np : 0.0;
      res.q_inf = q.q_inf;
      res.c_mp = q.c_mp;
      res.r_cv = q.r_cv;
      res.fixed_quantum = q.quantum;
    }
    if (parts != q.N) status = TPMC_ECUDA;
  }
  if (lane == 31) res.status = status;
}

__global__ void panels_kernel(const QueryDev* q, const long long* panel, const double* frames64, uint32_t n_tri,
                              double* pressure, double* shear) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_tri) return;
  const double* f = frames64 + 8 * (size_t)i;
  const double area = f[3];
  double p = 0.0, s = 0.0;
  if (area > 0.0) {
    const double scale = q->gamma / (double)q->N * q->m * q->c_mp * q->quantum;
    double F[3];
    for (int k = 0; k < 3; ++k) F[k] = scale * (double)panel[3 * (size_t)i + k];
    const double fn = F[0] * f[0] + F[1] * f[1] + F[2] * f[2];
    p = -fn / area;
    const double tx = F[0] - fn * f[0], ty = F[1] - fn * f[1], tz = F[2] - fn * f[2];
    s = sqrt(tx * tx + ty * ty + tz * tz) / area;
  }
  if (pressure) pressure[i] = p;
  if (shear) shear[i] = s;
}

}  // namespace

// ------------------------------------------------------------- launchers
// A launch that may start once every block of the stream's previous kernel has
// started (cudaTriggerProgrammaticLaunchCompletion in it; at its end otherwise), so
// that its launch latency passes under that kernel.  Its threads wait in
// cudaGridDependencySynchronize for that kernel's end, and its writes, before they
// read what it wrote; as all of them do, the end of this kernel means the end of
// that one, and a chain of these is as ordered as plain launches for what follows.
// Waiting blocks hold only what the running ones left free.  A call of 4,096
// particles on the 1,280-triangle sphere: 90 -> 86 us, eight attitudes of 20,000 on the
// cylinder: 156 -> 152.  Not from the pool: those launches take milliseconds.
template <typename... P, typename... A>
cudaError_t launch_after(void (*f)(P...), uint32_t grid, uint32_t block, size_t smem, cudaStream_t stream, A... args) {
  cudaLaunchAttribute overlap{};
  overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  overlap.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = stream;
  c.attrs = &overlap;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, f, P(args)...);
}

cudaError_t launch_setup(QueryDev* d_queries, uint32_t nq, const QueryDev* h_base, const double* d_dirs,
                         const double* d_S, ItemDev* d_items, const uint32_t* d_slots, AccStripe* d_acc,
                         uint32_t acc_stride, const float* tables, RunWords* d_zero, int num_sms, cudaStream_t stream) {
  if (nq == 0) return cudaSuccess;
  static_assert(sizeof(SetupBase) <= 3800, "a kernel's parameters");
  SetupBase with{};
  with.given = h_base != nullptr ? 1u : 0u;
  if (h_base != nullptr) with.q = *h_base;
  // Blocks of their own for the table as long as the chip's SMs are not all
  // busy with other queries (beyond that the split only repeats the scalars the
  // table needs).
  const dim3 grid(nq, (uint64_t)nq * kSetupParts <= 2 * (uint64_t)num_sms ? kSetupParts : 1);
  setup_kernel<<<grid, kSetupThreads, 0, stream>>>(d_queries, with, d_dirs, d_S, d_items, d_slots, d_acc, acc_stride,
                                                   reinterpret_cast<const double*>(tables + kVnNS * kVnNZ + 1), d_zero);
  return cudaGetLastError();
}

cudaError_t launch_tables(float* d_tables, cudaStream_t stream) {
  vn_table_kernel<<<(kVnNS * kVnNZ + 127) / 128, 128, 0, stream>>>(d_tables);
  knots_kernel<<<(kHTable + 128) / 128, 128, 0, stream>>>(reinterpret_cast<double*>(d_tables + kVnNS * kVnNZ + 1));
  return cudaGetLastError();
}

size_t trace_smem_bytes(const LaunchCfg& cfg, uint32_t n_nodes, uint32_t variant) {
  const uint32_t precision = variant & 1u;
  const size_t queue = (variant & kVariantPool) ? 0
                                                : (size_t)(cfg.block / 32) * kQueue *
                                                      (precision == TPMC_FP64 ? sizeof(Seeded<double>) : sizeof(Seeded<float>));
  const size_t staged =
      variant_width(variant) > 2 ? 0 : (size_t)std::min(cfg.smem_nodes, n_nodes) * kBinaryNodeF4 * sizeof(float4);
  return staged + queue + (size_t)cfg.block * sizeof(LaneAcc);
}

namespace {
TraceKernel pick_trace(uint32_t variant, uint32_t block, uint32_t blocks_per_sm) {
  switch (variant_width(variant)) {
    case 8: return trace_kernel_w8(variant, block, blocks_per_sm);
    case 4: return trace_kernel_w4(variant, block, blocks_per_sm);
    default: return trace_kernel_w2(variant, block, blocks_per_sm);
  }
}

int occupancy(TraceKernel f, uint32_t block, size_t smem) {
  int nb = 0;
  if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, (int)block, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return nb;
}
}  // namespace

// Largest resident block count over the instantiations that can run `cfg`.
int trace_max_blocks_per_sm(uint32_t variant, const LaunchCfg& cfg, uint32_t n_nodes) {
  const size_t smem = trace_smem_bytes(cfg, n_nodes, variant);
  if (smem > 227 * 1024) return 0;
  int best = occupancy(pick_trace(variant, cfg.block, 1), cfg.block, smem);
  if ((variant & 1u) == TPMC_FP32 && cfg.block <= 128) {
    for (int minb : {6, 8, 9}) {
      const int nb = occupancy(pick_trace(variant, cfg.block, (uint32_t)minb), cfg.block, smem);
      if (nb >= minb) best = std::max(best, nb);
    }
  }
  return best;
}

cudaError_t launch_seed(const TraceArgs& args, cudaStream_t stream) {
  switch (args.mesh.width) {
    case 8: return launch_seed_w8(args, stream);
    case 4: return launch_seed_w4(args, stream);
    default: return launch_seed_w2(args, stream);
  }
}

cudaError_t launch_trace(const TraceArgs& args, uint32_t variant, const LaunchCfg& cfg, int num_sms,
                         cudaStream_t stream) {
  // the mesh's own layout decides which traversal reads its nodes, and the
  // launch's counting flag whether the counters are compiled in
  variant = (variant & ~(kVariantWide4 | kVariantWide8 | kVariantCount)) |
            (args.mesh.width == 8 ? kVariantWide8 : (args.mesh.width == 4 ? kVariantWide4 : 0u)) |
            (args.count_work || args.rec.n_hits != nullptr || args.rec.tri != nullptr ? kVariantCount : 0u);
  if (args.pool == nullptr) variant &= ~kVariantPool;
  const size_t smem = trace_smem_bytes(cfg, args.mesh.n_nodes, variant);
  const uint32_t grid = (uint32_t)num_sms * cfg.blocks_per_sm;
  const TraceKernel f = pick_trace(variant, cfg.block, cfg.blocks_per_sm);
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (variant & kVariantPool) {
    f<<<grid, cfg.block, smem, stream>>>(args);
    return cudaGetLastError();
  }
  return launch_after(f, grid, cfg.block, smem, stream, args);
}

cudaError_t launch_finalize(const QueryDev* d_queries, const AccStripe* d_acc, uint32_t acc_stride, uint32_t nq,
                            const uint32_t* d_slots, tpmc_result* d_out, const int* d_err, int* err_out,
                            cudaStream_t stream) {
  if (nq == 0) return cudaSuccess;
  return launch_after(finalize_kernel, (nq + 3) / 4, 128, 0, stream, d_queries, d_acc, acc_stride, nq, d_slots, d_out,
                      d_err, err_out);
}

cudaError_t launch_panels(const QueryDev* d_query, const long long* d_panel, const float4*, const double* frames64,
                          uint32_t n_tri, double* d_pressure, double* d_shear, cudaStream_t stream) {
  if (n_tri == 0) return cudaSuccess;
  panels_kernel<<<(n_tri + 255) / 256, 256, 0, stream>>>(d_query, d_panel, frames64, n_tri, d_pressure, d_shear);
  return cudaGetLastError();
}

}  // namespace tpmc
