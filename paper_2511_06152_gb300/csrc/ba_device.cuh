// Device helpers: SO(3), the camera model of Eq. 5 with Brown distortion,
// the Huber weight of Eq. 6, and deterministic warp reductions.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "ba_internal.h"

namespace bagpu {

#define BA_FULL_MASK 0xffffffffu

__device__ __forceinline__ float rsqrt_any(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_any(double x) { return rsqrt(x); }

// 1 / sqrt(d) of a Cholesky pivot d > 0.  A pivot can be positive but tiny
// (a block whose only term is mu * D with a tiny damping mu, down to
// subnormal values): the reciprocal square root is taken of d scaled by an
// even power of two into the normal range, and the result is scaled back.
__device__ __forceinline__ double pivot_rsqrt(double d) {
  return d < 0x1p-960 ? rsqrt(d * 0x1p960) * 0x1p480 : rsqrt(d);
}
__device__ __forceinline__ float pivot_rsqrt(float d) {
  return d < 0x1p-100f ? rsqrtf(d * 0x1p100f) * 0x1p50f : rsqrtf(d);
}
__device__ __forceinline__ float recip_any(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double recip_any(double x) { return 1.0 / x; }
// a > b for b >= 0 (false for NaN), on the bits: a binary64
// comparison occupies the binary64 pipe like a product
__device__ __forceinline__ bool above(double a, double b) {
  const long long x = __double_as_longlong(a);
  return x > __double_as_longlong(b) && x <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool above(float a, float b) { return a > b; }

// largest s in [0, n) with pre[s] <= g (pre is non-decreasing)
__device__ __forceinline__ int find_slot(const int* __restrict__ pre, int n, int g) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(pre + mid) <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Reduce v over lanes [seg_start, seg_end) of a warp to lane seg_start by a
// binary tree whose shape depends only on the segment: deterministic.
// span = the warp's longest segment (warp-uniform): the levels at or above
// it add nothing and are skipped, which leaves every sum unchanged.
template <typename T>
__device__ __forceinline__ T seg_reduce(T v, int lane, int seg_start, int seg_end, int span = 32) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    if (off >= span) break;
    const T o = __shfl_down_sync(BA_FULL_MASK, v, off);
    if (((lane - seg_start) & (2 * off - 1)) == 0 && lane + off < seg_end) v += o;
  }
  return v;
}

// Whole-warp tree sum to lane 0 (fixed order).
template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(BA_FULL_MASK, v, off);
  return v;
}

// Segment bounds of each lane from the point index of its observation
// (inactive lanes carry a unique negative key and are their own segment).
__device__ __forceinline__ void segments(int key, int lane, int& seg_start, int& seg_end) {
  const int prev = __shfl_up_sync(BA_FULL_MASK, key, 1);
  const bool head = (lane == 0) || (key != prev) || key < 0;
  const unsigned heads = __ballot_sync(BA_FULL_MASK, head);
  const unsigned upto = (2u << lane) - 1u;  // lanes 0..lane (lane 31 wraps to all ones)
  seg_start = 31 - __clz(heads & upto);
  const unsigned after = heads & ~upto;
  seg_end = after ? __ffs(after) - 1 : 32;
}

// longest segment of the warp
__device__ __forceinline__ int segment_span(int seg_start, int seg_end) {
  return (int)__reduce_max_sync(BA_FULL_MASK, (unsigned)(seg_end - seg_start));
}

template <typename Real>
__device__ __forceinline__ Real clamp_diag(Real v) {
  return v < Real(kDiagMin) ? Real(kDiagMin) : (v > Real(kDiagMax) ? Real(kDiagMax) : v);
}

// ------------------------------------------------------------------ SO(3), FP64
//
// Angles below about 0.01 rad, which is what a step's rotation and the
// distance from an IMU attitude are, take the Taylor series of the
// coefficients (truncated below 2^-60 of the leading term) instead of
// trigonometric functions, square roots and quotients: binary64 runs at 2
// lanes per clock per SM, and these are evaluated for a handful of images at
// a time, on the critical path (the cost of a 16-image window's state, priors
// included: 17.8 -> 14.1 us).  The quotients' cancellation near zero goes
// with it.
constexpr double kSmallAngle2 = 1e-4;  // t^2

// R = Exp(w) = I + a [w]x + b [w]x^2, [w]x^2 = w w^T - |w|^2 I
__device__ inline void so3_exp(const double w[3], double R[9]) {
  const double t2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
  double a, b;
  if (t2 < kSmallAngle2) {  // sin t / t, (1 - cos t) / t^2
    a = 1.0 + t2 * (-1.0 / 6.0 + t2 * (1.0 / 120.0 + t2 * (-1.0 / 5040.0 + t2 * (1.0 / 362880.0))));
    b = 0.5 + t2 * (-1.0 / 24.0 + t2 * (1.0 / 720.0 + t2 * (-1.0 / 40320.0 + t2 * (1.0 / 3628800.0))));
  } else {
    const double t = sqrt(t2);
    double s, c;
    sincos(t, &s, &c);
    a = s / t;
    b = (1.0 - c) / t2;
  }
  const double d = 1.0 - b * t2;
  R[0] = d + b * w[0] * w[0];
  R[4] = d + b * w[1] * w[1];
  R[8] = d + b * w[2] * w[2];
  R[1] = b * w[0] * w[1] - a * w[2];
  R[3] = b * w[0] * w[1] + a * w[2];
  R[2] = b * w[0] * w[2] + a * w[1];
  R[6] = b * w[0] * w[2] - a * w[1];
  R[5] = b * w[1] * w[2] - a * w[0];
  R[7] = b * w[1] * w[2] + a * w[0];
}

// The factor of the axial part (R - R^T)^v in the rotation vector of R, t / (2
// sin t) for the angle t of the trace; -1 within 1e-6 of a half turn.
__device__ __forceinline__ double log_scale(double trace) {
  double c = 0.5 * (trace - 1.0);
  c = fmin(1.0, fmax(-1.0, c));
  const double x = 1.0 - c;
  if (x < 0.5 * kSmallAngle2)  // t / sin t in powers of 1 - cos t
    return 0.5 * (1.0 + x * (1.0 / 3.0 + x * (2.0 / 15.0 + x * (2.0 / 35.0 + x * (8.0 / 315.0)))));
  const double t = acos(c);
  return t > 3.14159165358979 ? -1.0 : t / (2.0 * sin(t));
}

__device__ inline void so3_log(const double R[9], double w[3]) {
  const double v0 = R[7] - R[5], v1 = R[2] - R[6], v2 = R[3] - R[1];
  const double sc = log_scale(R[0] + R[4] + R[8]);
  if (sc < 0.0) {
    const double t = acos(fmax(-1.0, 0.5 * (R[0] + R[4] + R[8] - 1.0)));
    // axis from the column of R + I with the largest norm
    int col = 0;
    double best = -1.0;
    for (int j = 0; j < 3; ++j) {
      const double a0 = R[j] + (j == 0), a1 = R[3 + j] + (j == 1), a2 = R[6 + j] + (j == 2);
      const double nn = a0 * a0 + a1 * a1 + a2 * a2;
      if (nn > best) { best = nn; col = j; }
    }
    const double inv = 1.0 / sqrt(best);
    double ax0 = (R[col] + (col == 0)) * inv, ax1 = (R[3 + col] + (col == 1)) * inv,
           ax2 = (R[6 + col] + (col == 2)) * inv;
    if (ax0 * v0 + ax1 * v1 + ax2 * v2 < 0.0) { ax0 = -ax0; ax1 = -ax1; ax2 = -ax2; }
    w[0] = t * ax0; w[1] = t * ax1; w[2] = t * ax2;
  } else {
    w[0] = sc * v0; w[1] = sc * v1; w[2] = sc * v2;
  }
}

// c2 of the inverse right Jacobian I + 1/2 [w]x + c2 [w]x^2, t2 = |w|^2
__device__ __forceinline__ double jr_inv_c2(double t2) {
  if (t2 < kSmallAngle2) return 1.0 / 12.0 + t2 * (1.0 / 720.0 + t2 * (1.0 / 30240.0 + t2 * (1.0 / 1209600.0)));
  const double t = sqrt(t2);
  double s, c;
  sincos(t, &s, &c);
  return 1.0 / t2 - (1.0 + c) / (2.0 * t * s);
}
__device__ inline void so3_jr_inv(const double w[3], double J[9]) {
  const double t2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
  const double c2 = jr_inv_c2(t2);
  const double d = 1.0 - c2 * t2;
  J[0] = d + c2 * w[0] * w[0];
  J[4] = d + c2 * w[1] * w[1];
  J[8] = d + c2 * w[2] * w[2];
  J[1] = c2 * w[0] * w[1] - 0.5 * w[2];
  J[3] = c2 * w[0] * w[1] + 0.5 * w[2];
  J[2] = c2 * w[0] * w[2] + 0.5 * w[1];
  J[6] = c2 * w[0] * w[2] - 0.5 * w[1];
  J[5] = c2 * w[1] * w[2] - 0.5 * w[0];
  J[7] = c2 * w[1] * w[2] + 0.5 * w[0];
}

// GNSS/IMU prior of one camera at (R, T): residual phi = Log(Rp^T R),
// e = T - Tp, whitened.  Fills J^T J (6x6 row-major) and J^T r (6), and
// returns the prior cost 1/2 |r|^2.
__device__ inline double prior_terms(const double* R, const double* T, const double* Rp, const double* Tp,
                                     double sigma_imu, double sigma_gnss, double* JtJ, double* Jtr) {
  double cost = 0.0;
  if (JtJ) for (int i = 0; i < 36; ++i) JtJ[i] = 0.0;
  if (Jtr) for (int i = 0; i < 6; ++i) Jtr[i] = 0.0;
  if (sigma_imu > 0.0) {
    double E[9];
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) E[3 * i + j] = Rp[i] * R[j] + Rp[3 + i] * R[3 + j] + Rp[6 + i] * R[6 + j];
    double phi[3];
    so3_log(E, phi);
    const double iv = 1.0 / (sigma_imu * sigma_imu);
    cost += 0.5 * iv * (phi[0] * phi[0] + phi[1] * phi[1] + phi[2] * phi[2]);
    if (JtJ || Jtr) {
      double Jr[9];
      so3_jr_inv(phi, Jr);
      for (int a = 0; a < 3; ++a) {
        if (Jtr) Jtr[a] = iv * (Jr[a] * phi[0] + Jr[3 + a] * phi[1] + Jr[6 + a] * phi[2]);
        if (JtJ)
          for (int b = 0; b < 3; ++b)
            JtJ[6 * a + b] = iv * (Jr[a] * Jr[b] + Jr[3 + a] * Jr[3 + b] + Jr[6 + a] * Jr[6 + b]);
      }
    }
  }
  if (sigma_gnss > 0.0) {
    const double ig = 1.0 / (sigma_gnss * sigma_gnss);
    for (int a = 0; a < 3; ++a) {
      const double e = T[a] - Tp[a];
      cost += 0.5 * ig * e * e;
      if (Jtr) Jtr[3 + a] = ig * e;
      if (JtJ) JtJ[6 * (3 + a) + 3 + a] = ig;
    }
  }
  return cost;
}

// The priors four lanes per image (a binary64 instruction occupies its quarter
// of the SM for 64 cycles per warp, however many lanes take part, so what
// counts is the length of a lane's program): lane q of the four takes axis q,
// q = 0 .. 2 (the fourth lane repeats axis 2).  mask: the four lanes.
__device__ __forceinline__ double quad_get(unsigned mask, double v, int q) {
  return __shfl_sync(mask, v, ((threadIdx.x & 31) & ~3) | q);
}
// w: the rotation vector of Rp^T R
__device__ __forceinline__ void quad_log(unsigned mask, const double* Rp, const double* R, int q, double w[3]) {
  // E(i, j) = sum_k Rp(k, i) R(k, j); this lane: E(q, q) and the axial part
  // E(a, b) - E(b, a), (a, b) = (2, 1), (0, 2), (1, 0)
  const int a = q == 0 ? 2 : (q == 1 ? 0 : 1), b = q == 0 ? 1 : (q == 1 ? 2 : 0);
  double tr = 0.0, v = 0.0, u = 0.0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    tr += Rp[3 * k + q] * R[3 * k + q];
    v += Rp[3 * k + a] * R[3 * k + b];
    u += Rp[3 * k + b] * R[3 * k + a];
  }
  const double t0 = quad_get(mask, tr, 0), t1 = quad_get(mask, tr, 1), t2 = quad_get(mask, tr, 2);
  const double s = log_scale(t0 + t1 + t2);
  if (s >= 0.0) {
    const double wq = s * (v - u);
    for (int i = 0; i < 3; ++i) w[i] = quad_get(mask, wq, i);
  } else {  // near a half turn: the general function
    double E[9];
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) E[3 * i + j] = Rp[i] * R[j] + Rp[3 + i] * R[3 + j] + Rp[6 + i] * R[6 + j];
    so3_log(E, w);
  }
}

// Prior cost of image k at (R, T), all four lanes
static __device__ __noinline__ double prior_cost_quad(unsigned mask, const DevCluster& C, int k, const double* R,
                                               const double* T, int q) {
  double v = 0.0;
  if (C.inv_imu2 > 0.0) {
    double w[3];
    quad_log(mask, C.R_prior + 9 * k, R, q, w);
    v = 0.5 * C.inv_imu2 * (w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
  }
  if (C.inv_gnss2 > 0.0) {
    const double e = T[q] - C.T_prior[3 * k + q];
    double e2 = 0.0;
    for (int i = 0; i < 3; ++i) {
      const double ei = quad_get(mask, e, i);
      e2 += ei * ei;
    }
    v += 0.5 * C.inv_gnss2 * e2;
  }
  return v;
}

// Sum of t[0 .. m) by one warp, in a fixed order; valid in lane 0
__device__ __forceinline__ double strided_sum(const double* t, int m, int lane) {
  double v = 0.0;
  for (int j = lane; j < m; j += 32) v += t[j];
  return warp_sum(v);
}

// ------------------------------------------------------------------ Eq. 5 + Brown, Eq. 6

// FP64 robust cost term 1/2 rho(s) / sigma^2 of one observation (0 behind the camera).
__device__ __forceinline__ double obs_cost(const double* R, const double* T, const double* in, const double* X,
                                           double uo, double vo, double half_inv_s2, double delta) {
  const double dx = X[0] - T[0], dy = X[1] - T[1], dz = X[2] - T[2];
  const double x = R[0] * dx + R[3] * dy + R[6] * dz;
  const double y = R[1] * dx + R[4] * dy + R[7] * dz;
  const double z = R[2] * dx + R[5] * dy + R[8] * dz;
  if (!above(z, kMinDepth)) return 0.0;
  const double iz = recip_any(z);
  const double xn = x * iz, yn = y * iz;
  const double xx = xn * xn, yy = yn * yn, xy = 2.0 * (xn * yn);
  const double r2 = xx + yy;
  const double rad = 1.0 + r2 * (in[3] + in[4] * r2);
  const double xd = xn * rad + in[5] * xy + in[6] * (r2 + 2.0 * xx);
  const double yd = yn * rad + in[5] * (r2 + 2.0 * yy) + in[6] * xy;
  const double e0 = in[0] * xd + (in[1] - uo), e1 = in[0] * yd + (in[2] - vo);
  const double s = e0 * e0 + e1 * e1;
  const double d2 = delta * delta;
  const double rho = !above(s, d2) ? s : 2.0 * delta * sqrt(s) - d2;
  return half_inv_s2 * rho;
}

__device__ __forceinline__ double obs_error_norm(const double* R, const double* T, const double* in, const double* X,
                                                 double uo, double vo) {
  const double dx = X[0] - T[0], dy = X[1] - T[1], dz = X[2] - T[2];
  const double x = R[0] * dx + R[3] * dy + R[6] * dz;
  const double y = R[1] * dx + R[4] * dy + R[7] * dz;
  const double z = R[2] * dx + R[5] * dy + R[8] * dz;
  const double iz = 1.0 / z;
  const double xn = x * iz, yn = y * iz;
  const double r2 = xn * xn + yn * yn;
  const double rad = 1.0 + r2 * (in[3] + in[4] * r2);
  const double xd = xn * rad + 2.0 * in[5] * xn * yn + in[6] * (r2 + 2.0 * xn * xn);
  const double yd = yn * rad + in[5] * (r2 + 2.0 * yn * yn) + 2.0 * in[6] * xn * yn;
  return hypot(in[0] * xd + in[1] - uo, in[0] * yd + in[2] - vo);
}

// Whitened, robust-weighted residual and Jacobians of one observation.
// d = X - T (world), Rm camera->world (row-major), in = (f, cx, cy, k1, k2, p1, p2).
// Jc is 2x6 row-major over [dtheta, dT] (right perturbation), Jp is 2x3.
template <typename Real>
__device__ __forceinline__ bool obs_linearize(const Real* Rm, Real dx, Real dy, Real dz, const Real* in, Real uo,
                                              Real vo, Real inv_sigma, Real delta, Real& r0, Real& r1, Real Jc[12],
                                              Real Jp[6]) {
  const Real x = Rm[0] * dx + Rm[3] * dy + Rm[6] * dz;
  const Real y = Rm[1] * dx + Rm[4] * dy + Rm[7] * dz;
  const Real z = Rm[2] * dx + Rm[5] * dy + Rm[8] * dz;
  if (!above(z, Real(kMinDepth))) {
    r0 = r1 = Real(0);
#pragma unroll
    for (int i = 0; i < 12; ++i) Jc[i] = Real(0);
#pragma unroll
    for (int i = 0; i < 6; ++i) Jp[i] = Real(0);
    return false;
  }
  const Real f = in[0], k1 = in[3], k2 = in[4], p1 = in[5], p2 = in[6];
  const Real iz = recip_any(z);
  const Real xn = x * iz, yn = y * iz;
  const Real r2 = xn * xn + yn * yn;
  const Real rad = Real(1) + r2 * (k1 + k2 * r2);
  const Real xd = xn * rad + Real(2) * p1 * xn * yn + p2 * (r2 + Real(2) * xn * xn);
  const Real yd = yn * rad + p1 * (r2 + Real(2) * yn * yn) + Real(2) * p2 * xn * yn;
  const Real e0 = f * xd + in[1] - uo;
  const Real e1 = f * yd + in[2] - vo;
  const Real s = e0 * e0 + e1 * e1;
  // IRLS weight w = rho'(s); scale = sqrt(w) / sigma
  Real scale = inv_sigma;
  if (above(s, delta * delta)) scale *= sqrt(delta * rsqrt_any(s));
  r0 = scale * e0;
  r1 = scale * e1;
  // d(xd, yd)/d(xn, yn)
  const Real drad = Real(2) * k1 + Real(4) * k2 * r2;
  const Real D00 = rad + drad * xn * xn + Real(2) * p1 * yn + Real(6) * p2 * xn;
  const Real D01 = drad * xn * yn + Real(2) * p1 * xn + Real(2) * p2 * yn;
  const Real D11 = rad + drad * yn * yn + Real(6) * p1 * yn + Real(2) * p2 * xn;
  // A = f D d(xn,yn)/dXc, scaled
  const Real a = scale * f * iz;
  const Real A00 = a * D00, A01 = a * D01, A02 = -a * (D00 * xn + D01 * yn);
  const Real A10 = a * D01, A11 = a * D11, A12 = -a * (D01 * xn + D11 * yn);
  // dXc/dX = R^T: Jp[r][b] = sum_c A[r][c] R[b][c]
  Jp[0] = A00 * Rm[0] + A01 * Rm[1] + A02 * Rm[2];
  Jp[1] = A00 * Rm[3] + A01 * Rm[4] + A02 * Rm[5];
  Jp[2] = A00 * Rm[6] + A01 * Rm[7] + A02 * Rm[8];
  Jp[3] = A10 * Rm[0] + A11 * Rm[1] + A12 * Rm[2];
  Jp[4] = A10 * Rm[3] + A11 * Rm[4] + A12 * Rm[5];
  Jp[5] = A10 * Rm[6] + A11 * Rm[7] + A12 * Rm[8];
  // dXc/ddtheta = [Xc]x
  Jc[0] = A01 * z - A02 * y;
  Jc[1] = A02 * x - A00 * z;
  Jc[2] = A00 * y - A01 * x;
  Jc[6] = A11 * z - A12 * y;
  Jc[7] = A12 * x - A10 * z;
  Jc[8] = A10 * y - A11 * x;
  // dXc/dT = -R^T
  Jc[3] = -Jp[0]; Jc[4] = -Jp[1]; Jc[5] = -Jp[2];
  Jc[9] = -Jp[3]; Jc[10] = -Jp[4]; Jc[11] = -Jp[5];
  return true;
}

// The point's share of one observation in the back-substitution, Jp^T (Jc dc),
// from the image's step: with A = d(residual)/dXc, Jc dc = A (Xc x dtheta - R^T
// dT) and Jp = A R^T, so that neither Jacobian is formed (and the robust weight
// enters without its root).  d = X - T, dth = dtheta, dt = R^T dT.
template <typename Real>
__device__ __forceinline__ void obs_step(const Real* Rm, Real dx, Real dy, Real dz, const Real* in, Real uo, Real vo,
                                         Real inv_sigma, Real delta, const Real dth[3], const Real dt[3], Real g[3]) {
  const Real x = Rm[0] * dx + Rm[3] * dy + Rm[6] * dz;
  const Real y = Rm[1] * dx + Rm[4] * dy + Rm[7] * dz;
  const Real z = Rm[2] * dx + Rm[5] * dy + Rm[8] * dz;
  const bool front = above(z, Real(kMinDepth));
  const Real f = in[0], k1 = in[3], k2 = in[4], p1 = in[5], p2 = in[6];
  const Real iz = recip_any(front ? z : Real(1));
  const Real xn = x * iz, yn = y * iz;
  const Real r2 = xn * xn + yn * yn;
  const Real rad = Real(1) + r2 * (k1 + k2 * r2);
  const Real xd = xn * rad + Real(2) * p1 * xn * yn + p2 * (r2 + Real(2) * xn * xn);
  const Real yd = yn * rad + p1 * (r2 + Real(2) * yn * yn) + Real(2) * p2 * xn * yn;
  const Real e0 = f * xd + in[1] - uo;
  const Real e1 = f * yd + in[2] - vo;
  const Real s = e0 * e0 + e1 * e1;
  Real w = inv_sigma * inv_sigma;  // rho'(s) / sigma^2
  if (above(s, delta * delta)) w *= delta * rsqrt_any(s);
  const Real drad = Real(2) * k1 + Real(4) * k2 * r2;
  const Real D00 = rad + drad * xn * xn + Real(2) * p1 * yn + Real(6) * p2 * xn;
  const Real D01 = drad * xn * yn + Real(2) * p1 * xn + Real(2) * p2 * yn;
  const Real D11 = rad + drad * yn * yn + Real(6) * p1 * yn + Real(2) * p2 * xn;
  // A = a (D | -D (xn, yn)^T), a = f / z
  const Real c0 = y * dth[2] - z * dth[1] - dt[0];
  const Real c1 = z * dth[0] - x * dth[2] - dt[1];
  const Real c2 = x * dth[1] - y * dth[0] - dt[2];
  const Real h0 = c0 - xn * c2, h1 = c1 - yn * c2;
  const Real u0 = D00 * h0 + D01 * h1, u1 = D01 * h0 + D11 * h1;
  Real b0 = D00 * u0 + D01 * u1, b1 = D01 * u0 + D11 * u1;
  const Real a = f * iz;
  const Real m = front ? w * a * a : Real(0);
  // A weight of zero selects zero: in binary32 b0 and b1 are infinite for a
  // point 1e5 m beside an image and behind it (its coordinates enter to the
  // tenth power), or where the squared error overflows, and 0 times that is NaN.
  b0 = above(m, Real(0)) ? b0 * m : Real(0);
  b1 = above(m, Real(0)) ? b1 * m : Real(0);
  const Real b2 = -(xn * b0 + yn * b1);
#pragma unroll
  for (int i = 0; i < 3; ++i) g[i] = Rm[3 * i] * b0 + Rm[3 * i + 1] * b1 + Rm[3 * i + 2] * b2;
}

// The LM decision of one cluster once every tile of its back-substitution is
// done, by one thread: gain ratio from F(x + d) and pred (Fo, pp: the sums of
// the tiles' cost and pred terms), accept or reject, Nielsen's update of mu and
// nu, the step record.  Returns 1 when the step was accepted.
__device__ __forceinline__ int lm_decide(const DevCluster& C, double Fo, double pp) {
  LmState* lm = C.lm;
  const bool ok = lm->status == 0;
  const double F = lm->F;
  const double Fn = ok ? Fo + lm->prior_new : F;
  const double pred = ok ? 0.5 * (pp + lm->pred_cam) : 0.0;
  const double gain = pred > 0.0 ? (F - Fn) / pred : 0.0;
  const int accepted = ok && pred > 0.0 && gain > 0.0;
  const double mu_used = lm->mu;
  if (accepted) {
    const double tt = 2.0 * gain - 1.0;
    const double fct = 1.0 - tt * tt * tt;
    lm->mu = mu_used * (fct > 1.0 / 3.0 ? fct : 1.0 / 3.0);
    lm->nu = 2.0;
    lm->cur ^= 1;
    lm->F = Fn;
    lm->n_accepted += 1;
  } else {
    lm->mu = mu_used * lm->nu;
    lm->nu *= 2.0;
  }
  if (C.trace_cap > 0) {
    StepRec& r = C.trace[lm->iter % C.trace_cap];
    r.accepted = accepted;
    r.status = lm->status;
    r.F_before = F;
    r.F_after = Fn;
    r.predicted = pred;
    r.gain = gain;
    r.mu_used = mu_used;
    r.mu = lm->mu;
    r.nu = lm->nu;
  }
  lm->iter += 1;
  if (lm->iter >= lm->iters_target) lm->active = 0;
  // converged (serving): an accepted step, not the first since arming, that
  // lowered F by at most ftol * F
  if (lm->ftol > 0.0 && accepted && lm->iter - lm->iter0 >= 2 && F - Fn <= lm->ftol * F) lm->active = 0;
  lm->pt_fail = 0;
  lm->mu_f = (float)lm->mu;
  return accepted;
}

// binary64 path: the camera records of an accepted step's state (buffer cur),
// by nt threads, t = 0 .. nt - 1
__device__ __forceinline__ void refresh_camreal(const DevCluster& C, int cur, int t, int nt) {
  double* cr = (double*)C.camreal;
  for (int k = t; k < C.n_cams; k += nt) {
    const double* R = C.R + ((size_t)cur * C.n_cams + k) * 9;
    const double* T = C.T + ((size_t)cur * C.n_cams + k) * 3;
    double* o = cr + (size_t)kCamReal * k;
    for (int i = 0; i < 9; ++i) o[i] = R[i];
    for (int i = 0; i < 3; ++i) o[9 + i] = T[i];
  }
}

// The tiles' sums are formed in the order of k_cost_init (kCostInitThreads
// threads, thread t of warp t / 32 adds tiles t, t + 256, ... in turn; a warp
// tree; the 8 warps in order), so that F carried from one iteration to the
// next equals F evaluated afresh at the start of a solve, bit for bit.
__device__ __forceinline__ void lm_tile_run(const DevCluster& C, int first, double& a, double& b) {
  const double2* tp = reinterpret_cast<const double2*>(C.tilepart);
  a = b = 0.0;
  int i = first;
  for (; i + 3 * kCostInitThreads < C.n_tiles; i += 4 * kCostInitThreads) {  // four loads in flight
    double2 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = __ldcg(tp + i + q * kCostInitThreads);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      a += v[q].x;
      b += v[q].y;
    }
  }
  for (; i < C.n_tiles; i += kCostInitThreads) {
    const double2 v = __ldcg(tp + i);
    a += v.x;
    b += v.y;
  }
  a = warp_sum(a);
  b = warp_sum(b);
}

// the whole step by one warp
template <bool MIXED>
__device__ __forceinline__ void lm_update_warp(const DevCluster& C, int lane) {
  double Fo = 0.0, pp = 0.0;
  if (C.lm->status == 0) {
    for (int w = 0; w < kCostInitThreads / 32; ++w) {
      double a, b;
      lm_tile_run(C, 32 * w + lane, a, b);
      Fo += a;
      pp += b;
    }
  }
  int accepted = lane == 0 ? lm_decide(C, Fo, pp) : 0;
  accepted = __shfl_sync(BA_FULL_MASK, accepted, 0);
  if (!MIXED && accepted) refresh_camreal(C, __shfl_sync(BA_FULL_MASK, lane == 0 ? C.lm->cur : 0, 0), lane, 32);
}

// the whole step by a CTA of kCostInitThreads threads (red: shared [2][8] and
// one more double)
template <bool MIXED>
__device__ __forceinline__ void lm_update_cta(const DevCluster& C, double* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  constexpr int nw = kCostInitThreads / 32;
  if (C.lm->status == 0) {
    double a, b;
    lm_tile_run(C, threadIdx.x, a, b);
    if (lane == 0) {
      red[wid] = a;
      red[nw + wid] = b;
    }
  } else if (lane == 0) {
    red[wid] = red[nw + wid] = 0.0;
  }
  __syncthreads();
  int* acc = reinterpret_cast<int*>(red + 2 * nw);
  if (threadIdx.x == 0) {
    double Fo = 0.0, pp = 0.0;
    for (int w = 0; w < nw; ++w) {
      Fo += red[w];
      pp += red[nw + w];
    }
    acc[0] = lm_decide(C, Fo, pp);
    acc[1] = C.lm->cur;
  }
  __syncthreads();
  if (!MIXED && acc[0]) refresh_camreal(C, acc[1], threadIdx.x, kCostInitThreads);
  __syncthreads();  // red is free
}

}  // namespace bagpu
