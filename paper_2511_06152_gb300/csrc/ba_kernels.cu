// Kernels of one LM iteration, batched over many clusters.
//
//   k_lin_schur      one CTA per chunk of consecutive tiles (a tile is up to 32
//                    observations of whole points, one warp).  Each warp
//                    linearises its tiles: residual, Jacobians (Eq. 5-7),
//                    point blocks V = sum Jp^T Jp and g_p = -sum Jp^T r by
//                    segmented warp reductions, V* = V + mu D_p = L L^T,
//                    M = L^-1, q = M g_p and Z = Jc^T Jp M^T, so that
//                    W V*^-1 W^T = Z Z^T and W V*^-1 g_p = Z q; one record per
//                    observation goes to shared memory.  The CTA then runs the
//                    chunk's reduction jobs: per free image the sums of
//                    Jc^T Jc - Z Z^T, -Jc^T r, Z q, diag(Jc^T Jc), and per
//                    co-visible image pair the sum of Z_a Z_b^T, each job on a
//                    run of lanes sized by its cost.  One partial sum per job.
//   k_partial_reduce the chunks' partial sums of each image and each pair,
//                    added in a fixed order; the pair sums go to their places
//                    in S.
//   k_factor_solve   per cluster (ba_factor.cu): assemble S = U* - W V*^-1 W^T
//                    and rhs = g_c - W V*^-1 g_p with priors and damping,
//                    L D L^T in the shared memory of four CTAs, solve,
//                    iterative refinement, candidate camera poses.  (Clusters
//                    of more than 32 free images: the global-memory solver of
//                    ba_big.cu.)
//   k_backsub_cost   per tile: each observation's Jp^T (Jc dc) from its image's
//                    step, without Jacobians; dX = M^T M (g_p - their sum),
//                    candidate points, cost at the candidate and the predicted
//                    reduction; the CTA whose warp finishes a cluster's last
//                    tile takes its LM step: gain ratio, accept/reject, Nielsen
//                    update.
//   Four launches per LM iteration.
//
// Precision.  MIXED = false: every step in binary64.  MIXED = true: the
// per-observation linearisation, the Schur reductions and the back-
// substitution run in binary32; the state (points and cameras) is held in
// double-float, and the cost F(x) that decides the gain ratio is evaluated
// per observation in double-float and summed in binary64; the reduced
// camera system is assembled, factored and refined in binary64.
//
// Every sum runs in an order fixed by the cluster's presorted tables; the
// only atomic is the back-substitution's per-cluster tile counter, which
// chooses the CTA that takes the LM step and enters no sum.
#include <cuda_runtime.h>
#include <stdio.h>

#include <algorithm>
#include <type_traits>

#include "ba_device.cuh"
#include "ba_bulk.cuh"
#include "ba_camera.cuh"
#include "ba_dfloat.cuh"
#include "ba_internal.h"

namespace bagpu {

template <bool MIXED> struct RealOf { using T = double; };
template <> struct RealOf<true> { using T = float; };

template <typename Real> struct Vec2;
template <> struct Vec2<float> { using T = float2; };
template <> struct Vec2<double> { using T = double2; };

// ------------------------------------------------------------------ state access

__device__ __forceinline__ const float2* xdf_ptr(const DevCluster& C, int buf, int j) {
  return reinterpret_cast<const float2*>(C.X) + ((size_t)buf * C.n_pts + j) * 3;
}
__device__ __forceinline__ float2* xdf_wptr(const DevCluster& C, int buf, int j) {
  return reinterpret_cast<float2*>(C.X) + ((size_t)buf * C.n_pts + j) * 3;
}

// double-float camera record
struct CamDf {
  dfl R[9], T[3], f, k1, k2, p1, p2;
  float free_flag;
};

// Camera record layout (kCamDf = 40 floats): the part the binary32
// linearisation reads first, in six float4: R.hi [0, 9), T.hi [9, 12),
// T.lo [12, 15), f.hi 15, k1 k2 p1 p2 .hi [16, 20), free flag 20, pad; then
// R.lo [24, 33), f.lo 33, k1 k2 p1 p2 .lo [34, 38), pad.
__device__ __forceinline__ void load_f4(const float* p, int n4, float* v) {
  const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
  for (int i = 0; i < n4; ++i) {
    const float4 w = q[i];
    v[4 * i] = w.x; v[4 * i + 1] = w.y; v[4 * i + 2] = w.z; v[4 * i + 3] = w.w;
  }
}

// the linearisation's part: high words of R, f and the distortion, T in full
__device__ __forceinline__ CamDf load_camdf_lin(const float* p) {
  CamDf c;
  float v[24];
  load_f4(p, 6, v);
#pragma unroll
  for (int i = 0; i < 9; ++i) c.R[i] = dfl{v[i], 0.f};
#pragma unroll
  for (int i = 0; i < 3; ++i) c.T[i] = dfl{v[9 + i], v[12 + i]};
  c.f = dfl{v[15], 0.f};
  c.k1 = dfl{v[16], 0.f};
  c.k2 = dfl{v[17], 0.f};
  c.p1 = dfl{v[18], 0.f};
  c.p2 = dfl{v[19], 0.f};
  c.free_flag = v[20];
  return c;
}

// the whole double-float record
__device__ __forceinline__ CamDf load_camdf(const float* p) {
  CamDf c;
  float v[kCamDf];
  load_f4(p, kCamDf / 4, v);
#pragma unroll
  for (int i = 0; i < 9; ++i) c.R[i] = dfl{v[i], v[24 + i]};
#pragma unroll
  for (int i = 0; i < 3; ++i) c.T[i] = dfl{v[9 + i], v[12 + i]};
  c.f = dfl{v[15], v[33]};
  c.k1 = dfl{v[16], v[34]};
  c.k2 = dfl{v[17], v[35]};
  c.p1 = dfl{v[18], v[36]};
  c.p2 = dfl{v[19], v[37]};
  c.free_flag = v[20];
  return c;
}

__device__ __forceinline__ const float* camdf_ptr(const DevCluster& C, int buf, int k) {
  return C.camdf + ((size_t)buf * C.n_cams + k) * kCamDf;
}

// Eq. 5 with Brown distortion in double-float: residual (u - cx, v - cy) - c
// for a double-float point, every term in double-float.  X - T and the final
// difference with the observation, where the result is much smaller than the
// operands, use the accurate sum; the other sums (the rotation, the
// distortion terms, all far below the pixel accuracy the cost needs in their
// cancellation) the sloppy one; one reciprocal of the depth.
__device__ __forceinline__ bool df_residual(const CamDf& c, dfl X0, dfl X1, dfl X2, dfl c0, dfl c1, dfl& e0,
                                            dfl& e1) {
  const dfl d0 = df_sub(X0, c.T[0]), d1 = df_sub(X1, c.T[1]), d2 = df_sub(X2, c.T[2]);
  const dfl z = df_add_fast(df_add_fast(df_mul(c.R[2], d0), df_mul(c.R[5], d1)), df_mul(c.R[8], d2));
  if (!(z.hi > (float)kMinDepth)) return false;
  const dfl x = df_add_fast(df_add_fast(df_mul(c.R[0], d0), df_mul(c.R[3], d1)), df_mul(c.R[6], d2));
  const dfl y = df_add_fast(df_add_fast(df_mul(c.R[1], d0), df_mul(c.R[4], d1)), df_mul(c.R[7], d2));
  const dfl iz = df_recip(z);
  const dfl xn = df_mul(x, iz), yn = df_mul(y, iz);
  const dfl xx = df_mul(xn, xn), yy = df_mul(yn, yn), xy2 = df_mul_f(df_mul(xn, yn), 2.0f);
  const dfl r2 = df_add_fast(xx, yy);
  const dfl radm1 = df_mul(r2, df_add_fast(c.k1, df_mul(c.k2, r2)));  // rad - 1
  const dfl ddx = df_add_fast(df_add_fast(df_mul(xn, radm1), df_mul(c.p1, xy2)),
                              df_mul(c.p2, df_add_fast(r2, df_mul_f(xx, 2.0f))));
  const dfl ddy = df_add_fast(df_add_fast(df_mul(yn, radm1), df_mul(c.p1, df_add_fast(r2, df_mul_f(yy, 2.0f)))),
                              df_mul(c.p2, xy2));
  e0 = df_sub(df_mul(c.f, df_add_fast(xn, ddx)), c0);
  e1 = df_sub(df_mul(c.f, df_add_fast(yn, ddy)), c1);
  return true;
}

// 1/2 rho(s) / sigma^2 in double-float, s = e0^2 + e1^2 (Eq. 6: rho on the squared norm)
__device__ __forceinline__ dfl df_robust_cost(dfl e0, dfl e1, float delta, float half_inv_s2) {
  const dfl s = df_add_fast(df_mul(e0, e0), df_mul(e1, e1));
  const float d2 = delta * delta;
  dfl rho;
  if (s.hi <= d2) {
    rho = s;
  } else {
    rho = df_add_f(df_mul_f(df_sqrt(s), 2.0f * delta), -d2);
  }
  return df_mul_f(rho, half_inv_s2);
}

// ------------------------------------------------------------------ camera copies

// FP64 path: camera records in binary64 for the per-observation kernels.
__global__ void k_camreal(BatchView bv) {
  for (int s = blockIdx.x; s < bv.n; s += gridDim.x) {
    const DevCluster& C = bv.cl[s];
    const int cur = C.lm->cur;
    double* cr = (double*)C.camreal;
    for (int k = threadIdx.x; k < C.n_cams; k += blockDim.x) {
      const double* R = C.R + ((size_t)cur * C.n_cams + k) * 9;
      const double* T = C.T + ((size_t)cur * C.n_cams + k) * 3;
      double* o = cr + (size_t)kCamReal * k;
      for (int i = 0; i < 9; ++i) o[i] = R[i];
      for (int i = 0; i < 3; ++i) o[9 + i] = T[i];
      for (int i = 0; i < 7; ++i) o[12 + i] = C.intr[7 * k + i];
      o[19] = C.free_idx[k] >= 0 ? 1.0 : 0.0;
    }
  }
}

// both buffers of the mixed camera records from the binary64 cameras
__global__ void k_camdf_all(BatchView bv) {
  for (int s = blockIdx.x; s < bv.n; s += gridDim.x) {
    const DevCluster& C = bv.cl[s];
    for (int idx = threadIdx.x; idx < 2 * C.n_cams; idx += blockDim.x) {
      const int buf = idx / C.n_cams, k = idx - buf * C.n_cams;
      write_camdf(C, buf, k, C.R + ((size_t)buf * C.n_cams + k) * 9, C.T + ((size_t)buf * C.n_cams + k) * 3);
    }
  }
}

// ------------------------------------------------------------------ per-tile linearisation

__device__ __forceinline__ void ld4(const float* r, int at, float* o) {
  const float4 v = *reinterpret_cast<const float4*>(r + at);
  o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void ld4(const double* r, int at, double* o) {
  const double2 a = *reinterpret_cast<const double2*>(r + at);
  const double2 b = *reinterpret_cast<const double2*>(r + at + 2);
  o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}

// What one lane knows after linearising its observation of a tile: the
// whitened, robust-weighted Jacobians and residual, P = Jp L^-T, and
// (broadcast from the point's first lane) L^-1 and q = L^-1 g_p of the damped
// point block; D_p and g_p are valid on the point's first lane.
template <bool MIXED>
struct TileLin {
  using Real = typename RealOf<MIXED>::T;
  bool act, head;
  int o, k, j, seg_start, seg_end, span;
  Real Jc[12], r0, r1;
  Real P[6];  // P = Jp M^T (2x3, row-major), so that Z = Jc^T P
  Real m00, m10, m11, m20, m21, m22, q0, q1, q2;
  Real d0, d1, d2, g0, g1, g2;
};

// Where the mixed linearisation reads a chunk's observations (camera, point,
// observation relative to the principal point) and the current points: a
// shared-memory copy of the chunk's ranges (index o - o0, point j - j0), the
// points of a chunk that spans too many in global memory.
struct ObsView {
  const int* cam;
  const int* pt;
  const float2* chi;
  const float2* x;  // 3 float2 (hi, lo) per point
  int o0, j0;
};

// Linearise one tile (one warp).
template <bool MIXED>
__device__ __forceinline__ void linearize_tile(const DevCluster& C, LmState* lm, const Tile& tl, int lane,
                                               bool report_fail, TileLin<MIXED>& L, const ObsView& V) {
  using Real = typename RealOf<MIXED>::T;
  L.act = lane < tl.n_obs;
  L.o = tl.obs_begin + (L.act ? lane : 0);
  if constexpr (MIXED) {
    L.k = L.act ? V.cam[L.o - V.o0] : 0;
    L.j = L.act ? V.pt[L.o - V.o0] : -1 - lane;
  } else {
    L.k = L.act ? C.obs_cam[L.o] : 0;
    L.j = L.act ? C.obs_pt[L.o] : -1 - lane;
  }
  segments(L.j, lane, L.seg_start, L.seg_end);
  L.span = segment_span(L.seg_start, L.seg_end);
  L.head = L.act && lane == L.seg_start;
  const int cur = lm->cur;
  Real mu, inv_sigma, delta;
  if constexpr (MIXED) {
    mu = lm->mu_f;
    inv_sigma = C.inv_sigma_f;
    delta = C.delta_f;
  } else {
    mu = lm->mu;
    inv_sigma = C.inv_sigma;
    delta = C.huber_delta;
  }
  Real Jp[6];
  L.r0 = 0;
  L.r1 = 0;
#pragma unroll
  for (int i = 0; i < 12; ++i) L.Jc[i] = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) Jp[i] = 0;
  if (L.act) {
    Real Rm[9], in[7], dx, dy, dz, uo, vo;
    bool is_free;
    if constexpr (MIXED) {
      const CamDf cd = load_camdf_lin(camdf_ptr(C, cur, L.k));
      const float2* xp = V.x + (size_t)(L.j - V.j0) * 3;
      const float2 a = xp[0], b = xp[1], c = xp[2];
      dx = df_sum_to_f(dfl{a.x, a.y}, df_neg(cd.T[0]));
      dy = df_sum_to_f(dfl{b.x, b.y}, df_neg(cd.T[1]));
      dz = df_sum_to_f(dfl{c.x, c.y}, df_neg(cd.T[2]));
#pragma unroll
      for (int i = 0; i < 9; ++i) Rm[i] = cd.R[i].hi;
      in[0] = cd.f.hi; in[1] = 0.f; in[2] = 0.f;
      in[3] = cd.k1.hi; in[4] = cd.k2.hi; in[5] = cd.p1.hi; in[6] = cd.p2.hi;
      const float2 ch = V.chi[L.o - V.o0];  // observation relative to the principal point
      uo = ch.x; vo = ch.y;
      is_free = cd.free_flag != 0.0f;
    } else {
      const double* cr = (const double*)C.camreal + (size_t)kCamReal * L.k;
#pragma unroll
      for (int i = 0; i < 9; ++i) Rm[i] = cr[i];
#pragma unroll
      for (int i = 0; i < 7; ++i) in[i] = cr[12 + i];
      const double* Xd = C.X + ((size_t)cur * C.n_pts + L.j) * 3;
      dx = Xd[0] - cr[9]; dy = Xd[1] - cr[10]; dz = Xd[2] - cr[11];
      const double2 u = reinterpret_cast<const double2*>(C.obs_uv)[L.o];
      uo = u.x; vo = u.y;
      is_free = cr[19] != 0.0;
    }
    obs_linearize<Real>(Rm, dx, dy, dz, in, uo, vo, inv_sigma, delta, L.r0, L.r1, L.Jc, Jp);
    if (!is_free) {
#pragma unroll
      for (int i = 0; i < 12; ++i) L.Jc[i] = 0;
    }
  }
  {
    // point blocks by segmented reduction
    Real v00 = Jp[0] * Jp[0] + Jp[3] * Jp[3];
    Real v01 = Jp[0] * Jp[1] + Jp[3] * Jp[4];
    Real v02 = Jp[0] * Jp[2] + Jp[3] * Jp[5];
    Real v11 = Jp[1] * Jp[1] + Jp[4] * Jp[4];
    Real v12 = Jp[1] * Jp[2] + Jp[4] * Jp[5];
    Real v22 = Jp[2] * Jp[2] + Jp[5] * Jp[5];
    Real g0 = -(Jp[0] * L.r0 + Jp[3] * L.r1);
    Real g1 = -(Jp[1] * L.r0 + Jp[4] * L.r1);
    Real g2 = -(Jp[2] * L.r0 + Jp[5] * L.r1);
    v00 = seg_reduce(v00, lane, L.seg_start, L.seg_end, L.span);
    v01 = seg_reduce(v01, lane, L.seg_start, L.seg_end, L.span);
    v02 = seg_reduce(v02, lane, L.seg_start, L.seg_end, L.span);
    v11 = seg_reduce(v11, lane, L.seg_start, L.seg_end, L.span);
    v12 = seg_reduce(v12, lane, L.seg_start, L.seg_end, L.span);
    v22 = seg_reduce(v22, lane, L.seg_start, L.seg_end, L.span);
    g0 = seg_reduce(g0, lane, L.seg_start, L.seg_end, L.span);
    g1 = seg_reduce(g1, lane, L.seg_start, L.seg_end, L.span);
    g2 = seg_reduce(g2, lane, L.seg_start, L.seg_end, L.span);
    // head: damp, factor V* = L L^T, M = L^-1, q = M g_p
    Real m00 = 0, m10 = 0, m11 = 0, m20 = 0, m21 = 0, m22 = 0, q0 = 0, q1 = 0, q2 = 0;
    L.d0 = L.d1 = L.d2 = 0;
    L.g0 = g0; L.g1 = g1; L.g2 = g2;
    if (L.head) {
      const Real d0 = clamp_diag(v00), d1 = clamp_diag(v11), d2 = clamp_diag(v22);
      const Real a00 = v00 + mu * d0, a11 = v11 + mu * d1, a22 = v22 + mu * d2;
      // V* = L L^T with M = L^-1 from reciprocal square roots of the pivots
      bool ok = a00 > Real(0);
      m00 = pivot_rsqrt(ok ? a00 : Real(1));
      const Real l10 = v01 * m00, l20 = v02 * m00;
      const Real t11 = a11 - l10 * l10;
      ok = ok && t11 > Real(0);
      m11 = pivot_rsqrt(t11 > Real(0) ? t11 : Real(1));
      const Real l21 = (v12 - l20 * l10) * m11;
      const Real t22 = a22 - l20 * l20 - l21 * l21;
      ok = ok && t22 > Real(0);
      m22 = pivot_rsqrt(t22 > Real(0) ? t22 : Real(1));
      if (!ok && report_fail) lm->pt_fail = 1;  // point block not positive definite: reject this step
      m10 = -l10 * m00 * m11;
      m21 = -l21 * m11 * m22;
      m20 = -(l20 * m00 + l21 * m10) * m22;
      q0 = m00 * g0;
      q1 = m10 * g0 + m11 * g1;
      q2 = m20 * g0 + m21 * g1 + m22 * g2;
      L.d0 = d0; L.d1 = d1; L.d2 = d2;
    }
    L.m00 = __shfl_sync(BA_FULL_MASK, m00, L.seg_start);
    L.m10 = __shfl_sync(BA_FULL_MASK, m10, L.seg_start);
    L.m11 = __shfl_sync(BA_FULL_MASK, m11, L.seg_start);
    L.m20 = __shfl_sync(BA_FULL_MASK, m20, L.seg_start);
    L.m21 = __shfl_sync(BA_FULL_MASK, m21, L.seg_start);
    L.m22 = __shfl_sync(BA_FULL_MASK, m22, L.seg_start);
    L.q0 = __shfl_sync(BA_FULL_MASK, q0, L.seg_start);
    L.q1 = __shfl_sync(BA_FULL_MASK, q1, L.seg_start);
    L.q2 = __shfl_sync(BA_FULL_MASK, q2, L.seg_start);
  }
  // P = Jp M^T (2x3), so that Z = Jc^T P (6x3)
  const Real P00 = Jp[0] * L.m00;
  const Real P01 = Jp[0] * L.m10 + Jp[1] * L.m11;
  const Real P02 = Jp[0] * L.m20 + Jp[1] * L.m21 + Jp[2] * L.m22;
  const Real P10 = Jp[3] * L.m00;
  const Real P11 = Jp[3] * L.m10 + Jp[4] * L.m11;
  const Real P12 = Jp[3] * L.m20 + Jp[4] * L.m21 + Jp[5] * L.m22;
  L.P[0] = P00; L.P[1] = P01; L.P[2] = P02;
  L.P[3] = P10; L.P[4] = P11; L.P[5] = P12;
}

// ------------------------------------------------------------------ K1: linearise + Schur reductions, one CTA per chunk

// Shared record of one observation, kSrec = 28 Real, 16-byte aligned:
// Jc [0, 12), r [12, 14), u = P q [14, 16), W = I - P P^T as
// (w00, w01, w11) [16, 19), pad, P [20, 26) (P = Jp M^T, 2x3), pad.  Since
// Z = Jc^T P, the observation's share of the image block is
// Jc^T Jc - Z Z^T = Jc^T W Jc, of the right-hand side Z q = Jc^T u, and of a
// pair block Z_a Z_b^T = Jc_a^T (P_a P_b^T) Jc_b.  An image job reads the
// first five 16-byte groups, a pair job groups 0-2, 5 and 6.
// Jc (12) and P (6)
template <typename Real>
__device__ __forceinline__ void ld_rec_jcp(const Real* r, Real Jc[12], Real P[6]) {
  ld4(r, 0, Jc);
  ld4(r, 4, Jc + 4);
  ld4(r, 8, Jc + 8);
  Real t[4];
  ld4(r, 20, P);
  ld4(r, 24, t);
  P[4] = t[0];
  P[5] = t[1];
}
// Jc (12), r (2), u (2), W (3)
template <typename Real>
__device__ __forceinline__ void ld_rec_cam(const Real* r, Real Jc[12], Real rr[2], Real u[2], Real w[3]) {
  ld4(r, 0, Jc);
  ld4(r, 4, Jc + 4);
  ld4(r, 8, Jc + 8);
  Real a[4], b[4];
  ld4(r, 12, a);
  ld4(r, 16, b);
  rr[0] = a[0]; rr[1] = a[1];
  u[0] = a[2]; u[1] = a[3];
  w[0] = b[0]; w[1] = b[1]; w[2] = b[2];
}

// Store one observation's record (vector stores): Jc, r, u = P q,
// W = I - P P^T and P.
template <bool MIXED>
__device__ __forceinline__ void st_rec(typename RealOf<MIXED>::T* r, const TileLin<MIXED>& L) {
  using Real = typename RealOf<MIXED>::T;
  const Real* P = L.P;
  const Real u0 = P[0] * L.q0 + P[1] * L.q1 + P[2] * L.q2;
  const Real u1 = P[3] * L.q0 + P[4] * L.q1 + P[5] * L.q2;
  const Real w00 = Real(1) - (P[0] * P[0] + P[1] * P[1] + P[2] * P[2]);
  const Real w01 = -(P[0] * P[3] + P[1] * P[4] + P[2] * P[5]);
  const Real w11 = Real(1) - (P[3] * P[3] + P[4] * P[4] + P[5] * P[5]);
  const Real v[28] = {L.Jc[0], L.Jc[1], L.Jc[2], L.Jc[3], L.Jc[4], L.Jc[5], L.Jc[6], L.Jc[7], L.Jc[8], L.Jc[9],
                      L.Jc[10], L.Jc[11], L.r0, L.r1, u0, u1, w00, w01, w11, Real(0),
                      P[0], P[1], P[2], P[3], P[4], P[5], Real(0), Real(0)};
  if constexpr (MIXED) {
    float4* o = reinterpret_cast<float4*>(r);
#pragma unroll
    for (int i = 0; i < 7; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
  } else {
    double2* o = reinterpret_cast<double2*>(r);
#pragma unroll
    for (int i = 0; i < 14; ++i) o[i] = make_double2(v[2 * i], v[2 * i + 1]);
  }
}

// The point's block for the back-substitution (head lane of the point).
template <bool MIXED>
__device__ __forceinline__ void st_ptblk(const DevCluster& C, const TileLin<MIXED>& L) {
  using Real = typename RealOf<MIXED>::T;
  const Real v[16] = {L.m00, L.m10, L.m11, L.m20, L.m21, L.m22, L.q0, L.q1,
                      L.q2,  L.d0,  L.d1,  L.d2,  L.g0,  L.g1,  L.g2, Real(0)};
  Real* pb = reinterpret_cast<Real*>(C.ptblk) + (size_t)L.j * 16;
  if constexpr (MIXED) {
    float4* o = reinterpret_cast<float4*>(pb);
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
  } else {
    double2* o = reinterpret_cast<double2*>(pb);
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i] = make_double2(v[2 * i], v[2 * i + 1]);
  }
}

// One job's sums over its items [i0, i1).  Image job: the upper triangle of
// sum Jc^T W Jc (21), -sum Jc^T r (6), sum Jc^T u (6), diag sum Jc^T Jc (6).
// Pair job: sum Jc_a^T (P_a P_b^T) Jc_b (36, row-major).
template <typename Real>
__device__ __forceinline__ void job_sums(const DevCluster& C, const Job& J, bool cam, int i0, int i1,
                                         const Real* srec, Real acc[39]) {
#pragma unroll
  for (int i = 0; i < 39; ++i) acc[i] = 0;
  if (cam) {
    for (int e = i0; e < i1; ++e) {
      const Real* r = srec + (size_t)C.cm_list[J.item_begin + e] * kSrec;
      Real Jc[12], rr[2], u[2], w[3];
      ld_rec_cam(r, Jc, rr, u, w);
      Real WJ0[6], WJ1[6];
#pragma unroll
      for (int m = 0; m < 6; ++m) {
        WJ0[m] = w[0] * Jc[m] + w[1] * Jc[6 + m];
        WJ1[m] = w[1] * Jc[m] + w[2] * Jc[6 + m];
      }
      int t = 0;
#pragma unroll
      for (int a = 0; a < 6; ++a)
#pragma unroll
        for (int b = a; b < 6; ++b) acc[t++] += Jc[a] * WJ0[b] + Jc[6 + a] * WJ1[b];
#pragma unroll
      for (int a = 0; a < 6; ++a) {
        acc[21 + a] -= Jc[a] * rr[0] + Jc[6 + a] * rr[1];
        acc[27 + a] += Jc[a] * u[0] + Jc[6 + a] * u[1];
        acc[33 + a] += Jc[a] * Jc[a] + Jc[6 + a] * Jc[6 + a];
      }
    }
  } else {
    for (int e = i0; e < i1; ++e) {
      const unsigned int it = C.pent[J.item_begin + e];
      Real Ja[12], Pa[6], Jb[12], Pb[6];
      ld_rec_jcp(srec + (size_t)(it & 0xffffu) * kSrec, Ja, Pa);
      ld_rec_jcp(srec + (size_t)(it >> 16) * kSrec, Jb, Pb);
      // G = P_a P_b^T (2x2), H = G Jc_b (2x6)
      const Real g00 = Pa[0] * Pb[0] + Pa[1] * Pb[1] + Pa[2] * Pb[2];
      const Real g01 = Pa[0] * Pb[3] + Pa[1] * Pb[4] + Pa[2] * Pb[5];
      const Real g10 = Pa[3] * Pb[0] + Pa[4] * Pb[1] + Pa[5] * Pb[2];
      const Real g11 = Pa[3] * Pb[3] + Pa[4] * Pb[4] + Pa[5] * Pb[5];
      Real H0[6], H1[6];
#pragma unroll
      for (int m = 0; m < 6; ++m) {
        H0[m] = g00 * Jb[m] + g01 * Jb[6 + m];
        H1[m] = g10 * Jb[m] + g11 * Jb[6 + m];
      }
#pragma unroll
      for (int a = 0; a < 6; ++a)
#pragma unroll
        for (int b = 0; b < 6; ++b) acc[6 * a + b] += Ja[a] * H0[b] + Ja[6 + a] * H1[b];
    }
  }
}

// One job's partial sums as 16-byte stores (the rows are 16-byte aligned:
// kCamPart and kPairPart are multiples of 16 bytes); a camera row's last
// group carries a zero in its pad word.
static_assert(kCamPart % 4 == 0 && kPairPart % 4 == 0, "partial rows of 16-byte groups");
__device__ __forceinline__ void store_job_row(float* out, bool cam, const float acc[39]) {
  float4* o = reinterpret_cast<float4*>(out);
#pragma unroll
  for (int i = 0; i < 9; ++i) o[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
  if (cam) o[9] = make_float4(acc[36], acc[37], acc[38], 0.f);
}
__device__ __forceinline__ void store_job_row(double* out, bool cam, const double acc[39]) {
  double2* o = reinterpret_cast<double2*>(out);
#pragma unroll
  for (int i = 0; i < 18; ++i) o[i] = make_double2(acc[2 * i], acc[2 * i + 1]);
  if (cam) {
    o[18] = make_double2(acc[36], acc[37]);
    o[19] = make_double2(acc[38], 0.0);
  }
}

template <typename Real>
__device__ __forceinline__ void store_job(const DevCluster& C, const Job& J, bool cam, const Real acc[39]) {
  Real* out = cam ? (Real*)C.campart + (size_t)kCamPart * J.slot : (Real*)C.pairpart + (size_t)kPairPart * J.slot;
  store_job_row(out, cam, acc);
}

// bytes of the per-observation records (and, overlaid, the lane partials)
__host__ __device__ constexpr size_t chunk_records_bytes(bool mixed) {
  return (mixed ? sizeof(float) : sizeof(double)) *
         ((size_t)(mixed ? kChunkObsMixed : kChunkObsF64) * kSrec > (size_t)kChunkThreads * kLanePart
              ? (size_t)(mixed ? kChunkObsMixed : kChunkObsF64) * kSrec
              : (size_t)kChunkThreads * kLanePart);
}
__device__ __forceinline__ float4 vadd(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

// Shared-memory staging of one chunk's observations and points (mixed path):
// camera and point indices (int), observations relative to the principal
// point (float2 hi), points (3 float2 each), each range rounded outward to
// 16 bytes.  A chunk spanning more than kStagePts points reads its points
// from global memory instead.  Double-buffered beside them, so that the next
// chunk's copies land while this chunk's jobs still read its own: the chunk's
// head (cluster slot, state buffer, chunk record; written by the issuing
// thread), its tile headers, its job records and the job of each lane (the
// last two for chunks of at most kChunkThreads jobs).
constexpr int kStagePts = 512;
constexpr uint32_t kStageIdxBytes = kChunkObsMixed * 4 + 32;
constexpr uint32_t kStageChiBytes = kChunkObsMixed * 8 + 32;
constexpr uint32_t kStageXBytes = kStagePts * 24 + 32;
struct ChunkHead {
  int s, cur, pad0, pad1;
  Chunk ch;
};
constexpr uint32_t kHeadBytes = (sizeof(ChunkHead) + 15) / 16 * 16;
constexpr uint32_t kStageTileBytes = kChunkTilesMixed * sizeof(Tile) + 32;
constexpr uint32_t kStageJobBytes = kChunkThreads * sizeof(Job) + 32;
constexpr uint32_t kStageLaneBytes = kChunkThreads;  // one byte per lane
constexpr uint32_t kTableBytes = kHeadBytes + kStageTileBytes + kStageJobBytes + kStageLaneBytes;
constexpr uint32_t kStageBytes = 2 * kStageIdxBytes + kStageChiBytes + kStageXBytes + 2 * kTableBytes;
constexpr uint64_t kCopyWaitNs = 200000000ull;  // give up on a staged copy after 200 ms
constexpr uint64_t kInjectWaitNs = 1000000ull;  // the injected wait's limit (kInjectCopyTimeout)
static_assert(kTableBytes % 16 == 0 && kStageTileBytes % 16 == 0 && kStageJobBytes % 16 == 0, "16-byte staging");

struct Stage {
  char* idx_cam;
  char* idx_pt;
  char* chi;
  char* x;
  char* tab;  // two table buffers of kTableBytes
  uint64_t* bar;
  int* ok;
  uint64_t* never;  // failure injection: a barrier no copy or thread completes
  __device__ ChunkHead* head(int b) const { return reinterpret_cast<ChunkHead*>(tab + b * kTableBytes); }
  __device__ char* tiles(int b) const { return tab + b * kTableBytes + kHeadBytes; }
  __device__ char* jobs(int b) const { return tab + b * kTableBytes + kHeadBytes + kStageTileBytes; }
  __device__ unsigned char* lanes(int b) const {
    return reinterpret_cast<unsigned char*>(tab + b * kTableBytes + kHeadBytes + kStageTileBytes + kStageJobBytes);
  }
};

__device__ __forceinline__ bool job_table_mode(const Chunk& ch) {
  const int nj = ch.n_lc + ch.n_lp;
  return nj > 0 && nj <= kChunkThreads;
}

// Issue the copies of chunk g into table buffer b (one thread) and write its
// head.  The barrier's transaction count covers exactly the bytes issued.
__device__ __forceinline__ void stage_issue(const BatchView& bv, int g, const Stage& S, int b) {
  const int s = find_slot(bv.chunk_pre, bv.n, g);
  const DevCluster& C = bv.cl[s];
  const int local = g - bv.chunk_pre[s];
  const Chunk ch = C.chunks[local];
  const int cur = C.lm->cur;
  ChunkHead* hd = S.head(b);
  hd->s = s;
  hd->cur = cur;
  hd->ch = ch;
  const BulkRange rc = bulk_range(C.obs_cam + ch.obs_begin, (size_t)ch.n_obs * 4);
  const BulkRange rp = bulk_range(C.obs_pt + ch.obs_begin, (size_t)ch.n_obs * 4);
  const BulkRange rh = bulk_range(C.obs_chi + ch.obs_begin, (size_t)ch.n_obs * 8);
  const bool stage_x = ch.n_pts <= kStagePts;
  const float2* xb = reinterpret_cast<const float2*>(C.X) + ((size_t)cur * C.n_pts + ch.pt_begin) * 3;
  const BulkRange rx = bulk_range(xb, stage_x ? (size_t)ch.n_pts * 24 : 0);
  const BulkRange rt = bulk_range(C.tiles + ch.tile_begin, (size_t)ch.n_tiles * sizeof(Tile));
  const bool tab = job_table_mode(ch);
  const BulkRange rj = bulk_range(C.jobs + ch.job_begin, tab ? (size_t)(ch.n_lc + ch.n_lp) * sizeof(Job) : 0);
  const unsigned char* lj = C.lane_job + (size_t)local * kChunkThreads;
  fence_proxy_async_smem();
  mbar_arrive_expect_tx(S.bar, rc.bytes + rp.bytes + rh.bytes + (stage_x ? rx.bytes : 0u) + rt.bytes +
                                   (tab ? rj.bytes + kStageLaneBytes : 0u));
  bulk_copy_g2s(S.idx_cam, rc.src, rc.bytes, S.bar);
  bulk_copy_g2s(S.idx_pt, rp.src, rp.bytes, S.bar);
  bulk_copy_g2s(S.chi, rh.src, rh.bytes, S.bar);
  if (stage_x && rx.bytes) bulk_copy_g2s(S.x, rx.src, rx.bytes, S.bar);
  bulk_copy_g2s(S.tiles(b), rt.src, rt.bytes, S.bar);
  if (tab) {
    bulk_copy_g2s(S.jobs(b), rj.src, rj.bytes, S.bar);
    bulk_copy_g2s(S.lanes(b), lj, kStageLaneBytes, S.bar);
  }
}

// The view of the staged chunk (same rounding as stage_issue).
__device__ __forceinline__ ObsView stage_view(const DevCluster& C, const Chunk& ch, int cur, const Stage& S) {
  ObsView V;
  V.cam = reinterpret_cast<const int*>(S.idx_cam + bulk_range(C.obs_cam + ch.obs_begin, 4).lead);
  V.pt = reinterpret_cast<const int*>(S.idx_pt + bulk_range(C.obs_pt + ch.obs_begin, 4).lead);
  V.chi = reinterpret_cast<const float2*>(S.chi + bulk_range(C.obs_chi + ch.obs_begin, 8).lead);
  V.o0 = ch.obs_begin;
  const float2* xb = reinterpret_cast<const float2*>(C.X) + ((size_t)cur * C.n_pts + ch.pt_begin) * 3;
  if (ch.n_pts <= kStagePts) {
    V.x = reinterpret_cast<const float2*>(S.x + bulk_range(xb, 24).lead);
    V.j0 = ch.pt_begin;
  } else {
    V.x = reinterpret_cast<const float2*>(C.X) + (size_t)cur * C.n_pts * 3;
    V.j0 = 0;
  }
  return V;
}

template <bool MIXED>
__global__ void __launch_bounds__(kChunkThreads, MIXED ? kLinSchurMinBlocksMixed : 1)
    k_lin_schur(BatchView bv, int diag) {
  using Real = typename RealOf<MIXED>::T;
  extern __shared__ __align__(16) unsigned char smraw[];
  // [chunk_obs][kSrec] records; once every job has read them, the same
  // memory holds the lane partials of multi-lane jobs ([threads][kLanePart])
  Real* srec = reinterpret_cast<Real*>(smraw);
  Real* lanepart = srec;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int total = bv.tot[1];
  // a contiguous run of chunks per CTA: neighbouring chunks (Morton order of
  // the points) share images and points in the caches
  const int per = (total + (int)gridDim.x - 1) / (int)gridDim.x;
  const int g0 = (int)blockIdx.x * per, g1 = min(total, g0 + per);
  // mixed path: the next chunk's observations and points are copied into
  // shared memory by the copy engine while this chunk is reduced
  Stage S{};
  uint32_t phase = 0;
  if constexpr (MIXED) {
    char* st = reinterpret_cast<char*>(smraw) + chunk_records_bytes(true);
    S.idx_cam = st;
    S.idx_pt = st + kStageIdxBytes;
    S.chi = st + 2 * kStageIdxBytes;
    S.x = st + 2 * kStageIdxBytes + kStageChiBytes;
    S.tab = st + 2 * kStageIdxBytes + kStageChiBytes + kStageXBytes;
    S.bar = reinterpret_cast<uint64_t*>(st + kStageBytes);
    S.ok = reinterpret_cast<int*>(st + kStageBytes + 8);
    S.never = reinterpret_cast<uint64_t*>(st + kStageBytes + 16);
    if (threadIdx.x == 0) {
      mbar_init(S.bar, 1);
      mbar_init(S.never, 1);
      fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0 && g0 < g1) stage_issue(bv, g0, S, 0);
  }
  int b = 0;  // table buffer of the current chunk (mixed path)
  for (int g = g0; g < g1; ++g, b ^= 1) {
    int s;
    Chunk ch;
    if constexpr (!MIXED) {
      s = find_slot(bv.chunk_pre, bv.n, g);
      ch = bv.cl[s].chunks[g - bv.chunk_pre[s]];
    }
    ObsView V{};
    if constexpr (MIXED) {
      if (threadIdx.x == 0) {
        const bool ok = (bv.inject & kInjectCopyTimeout) ? mbar_wait_bounded(S.never, 0u, kInjectWaitNs)
                                                         : mbar_wait_bounded(S.bar, phase, kCopyWaitNs);
        *S.ok = ok ? 1 : 0;
      }
      __syncthreads();
      phase ^= 1u;
      if (!*S.ok) {
        // the copy did not complete in time: flag every cluster whose chunks
        // this CTA has still to process (their steps are rejected), wait once
        // more for the copies in flight, and stop
        if (threadIdx.x == 0) {
          for (int h = g; h < g1; ++h) {
            LmState* hl = bv.cl[find_slot(bv.chunk_pre, bv.n, h)].lm;
            hl->dev_error = kDevErrTimeout;
            hl->pt_fail = 1;
          }
          mbar_wait_bounded(S.bar, phase ^ 1u, kCopyWaitNs);
        }
        return;
      }
      const ChunkHead* hd = S.head(b);
      s = hd->s;
      ch = hd->ch;
      V = stage_view(bv.cl[s], ch, hd->cur, S);
    }
    const DevCluster& C = bv.cl[s];
    LmState* lm = C.lm;
    const bool active = lm->active != 0;
    // 1. linearise the chunk's tiles into shared memory
    if (active) {
      for (int t = warp; t < ch.n_tiles; t += nw) {
        Tile tl;
        if constexpr (MIXED) {
          tl = reinterpret_cast<const Tile*>(S.tiles(b) + bulk_range(C.tiles + ch.tile_begin, 8).lead)[t];
        } else {
          tl = C.tiles[ch.tile_begin + t];
        }
        TileLin<MIXED> L;
        linearize_tile<MIXED>(C, lm, tl, lane, true, L, V);
        if (L.act) st_rec<MIXED>(srec + (size_t)(L.o - ch.obs_begin) * kSrec, L);
        if (L.head) st_ptblk<MIXED>(C, L);
        if (diag) {  // largest |g_p| of the tile, for the gradient norm
          double gm = L.head ? fmax(fabs((double)L.g0), fmax(fabs((double)L.g1), fabs((double)L.g2))) : 0.0;
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) gm = fmax(gm, __shfl_down_sync(BA_FULL_MASK, gm, off));
          if (lane == 0) C.tilepart[2 * (ch.tile_begin + t) + 1] = gm;
        }
      }
    }
    __syncthreads();
    if constexpr (MIXED) {  // staging is free: start the copies of this CTA's next chunk
      if (threadIdx.x == 0 && g + 1 < g1) stage_issue(bv, g + 1, S, b ^ 1);
    }
    if (!active) continue;
    // 2. Schur reductions of the chunk.  Jobs: each free camera (sum of
    //    Jc^T Jc - Z Z^T, -Jc^T r, Z q, diag(Jc^T Jc) over its observations) and
    //    each co-visible camera pair (sum of Z_a Z_b^T over its point pairs).
    //    The host gave every job a run of lanes in proportion to its cost;
    //    lane i of a job sums a contiguous range of the job's items, and the
    //    lanes' partial sums are added in lane order.  A chunk with more jobs
    //    than threads runs one lane per job.
    const int n_jobs = ch.n_lc + ch.n_lp;  // 0 when every observation of the chunk is of a fixed camera
    if (n_jobs > 0 && n_jobs <= (int)blockDim.x) {
      // job whose lane run holds this thread: the last job starting at or
      // before it (jobs are in lane order); staged by the host's table on the
      // mixed path, a binary search on the other
      int lo;
      Job J;
      if constexpr (MIXED) {
        lo = S.lanes(b)[threadIdx.x];
        J = reinterpret_cast<const Job*>(S.jobs(b) + bulk_range(C.jobs + ch.job_begin, 16).lead)[lo];
      } else {
        lo = 0;
        int hi = n_jobs - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (C.jobs[ch.job_begin + mid].lane_begin <= (int)threadIdx.x) lo = mid; else hi = mid - 1;
        }
        J = C.jobs[ch.job_begin + lo];
      }
      const bool mine = (int)threadIdx.x < J.lane_begin + J.n_lanes;
      const int part = threadIdx.x - J.lane_begin;
      const bool cam = lo < ch.n_lc;
      Real acc[39];
      if (mine) {
        const int i0 = (int)(((long long)J.count * part) / J.n_lanes);
        const int i1 = (int)(((long long)J.count * (part + 1)) / J.n_lanes);
        job_sums<Real>(C, J, cam, i0, i1, srec, acc);
        if (J.n_lanes == 1) store_job<Real>(C, J, cam, acc);
      }
      __syncthreads();  // every record has been read: the lane partials may overwrite them
      if (mine && J.n_lanes > 1) {
        Real* lp = lanepart + (size_t)threadIdx.x * kLanePart;
        if constexpr (MIXED) {
          float4* o = reinterpret_cast<float4*>(lp);
#pragma unroll
          for (int i = 0; i < 9; ++i) o[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
          o[9] = make_float4(acc[36], acc[37], acc[38], 0.f);
        } else {
          double2* o = reinterpret_cast<double2*>(lp);
#pragma unroll
          for (int i = 0; i < 19; ++i) o[i] = make_double2(acc[2 * i], acc[2 * i + 1]);
          o[19] = make_double2(acc[38], 0.0);
        }
      }
      __syncthreads();
      // multi-lane jobs: the job's own lanes add its lane partials, each lane
      // a share of the 16-byte groups of the row, every element summed over
      // the job's lanes in lane order
      if (mine && J.n_lanes > 1) {
        using Vec = typename std::conditional<MIXED, float4, double2>::type;
        constexpr int kPer = 16 / sizeof(Real);  // elements of a group
        const int groups = (cam ? kCamPart : kPairPart) / kPer;
        const Vec* rows = reinterpret_cast<const Vec*>(lanepart);
        Vec* out = reinterpret_cast<Vec*>(cam ? (Real*)C.campart + (size_t)kCamPart * J.slot
                                              : (Real*)C.pairpart + (size_t)kPairPart * J.slot);
        for (int q = part; q < groups; q += J.n_lanes) {
          Vec v = rows[(size_t)J.lane_begin * (kLanePart / kPer) + q];
          for (int l = J.lane_begin + 1; l < J.lane_begin + J.n_lanes; ++l) v = vadd(v, rows[(size_t)l * (kLanePart / kPer) + q]);
          out[q] = v;
        }
      }
    } else {
      for (int jb = threadIdx.x; jb < n_jobs; jb += blockDim.x) {
        const Job J = C.jobs[ch.job_begin + jb];
        const bool cam = jb < ch.n_lc;
        Real acc[39];
        job_sums<Real>(C, J, cam, 0, J.count, srec, acc);
        store_job<Real>(C, J, cam, acc);
      }
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ partial sums -> per-camera / per-pair sums

// Running sum of binary32 partials kept in double-float (TwoSum, error-free
// to ~2^-48 of the total; binary64 adds run at 1/59 of the binary32 rate),
// or of binary64 partials in binary64.
struct AccF {
  using Raw = dfl;
  dfl v{0.f, 0.f};
  __device__ __forceinline__ void add(float x) { v = df_add_f(v, x); }
  __device__ __forceinline__ double get() const { return (double)v.hi + (double)v.lo; }
};
struct AccD {
  using Raw = double;
  double v = 0.0;
  __device__ __forceinline__ void add(double x) { v += x; }
  __device__ __forceinline__ double get() const { return v; }
};
template <typename Real> struct AccOf { using T = AccD; };
template <> struct AccOf<float> { using T = AccF; };

__device__ __forceinline__ AccF acc_join(AccF a, AccF b) { return AccF{df_add(a.v, b.v)}; }
__device__ __forceinline__ AccD acc_join(AccD a, AccD b) { return AccD{a.v + b.v}; }

// Every free camera and camera pair ("item") of the batch's clusters: its
// chunk partials, added, into camsum, and into S (pairsum for the
// global-memory solver).
//
// Per iteration on GB300: one cluster of 235 k observations 39 -> 12 us (97 ->
// 19 in binary64), 12 clusters 25 -> 21, 128 clusters 68 -> 83: their short
// lists filled the GPU as a warp each too, and the pair sums go to their rows
// in S here (a wider spread of stores, 98 us when the transposed ones went out
// column by column), which saves the factor its pair tables.
//
// What bounds it is the latency of the loads: an item is a list of rows, up
// to one per chunk of the cluster (501 of them for 235 k observations), and
// one warp per item added them a few at a time, 39 us per iteration of that
// single cluster (97 us in binary64) with most of the GPU idle.  A CTA has
// kRedSegs groups of kCamPart lanes (lane = element of the row).  A list of
// up to kRedLong rows is one group's; a longer one is cut into kRedSegs
// contiguous runs, a group each, whose sums are joined in order.  Eight rows
// are in flight per lane.  The cut depends on the list's length alone, so a
// cluster's sums are the same alone and in any batch.  With more items than
// CTAs, a CTA takes several items at a time, a grid apart (a cluster's long
// lists, its images', are neighbours), and their short lists run side by side.
constexpr int kRedSegs = 6;
constexpr int kRedLong = 48;
constexpr int kRedThreads = 256;
constexpr int kRedCtasPerSm = 16;
static_assert(kRedSegs * kCamPart <= kRedThreads && kPairPart <= kCamPart, "a group of lanes per row");

// rows [p, p1) of a list, element el, in order
template <typename Real>
__device__ __forceinline__ typename AccOf<Real>::T add_rows(const Real* part, int stride, const int* slots, int p,
                                                            int p1) {
  typename AccOf<Real>::T acc;
  for (; p + 8 <= p1; p += 8) {
    Real x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = part[(size_t)stride * slots[p + i]];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc.add(x[i]);
  }
  if (p < p1) {  // the last rows, all loads before the adds as well
    Real x[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) x[i] = p + i < p1 ? part[(size_t)stride * slots[p + i]] : Real(0);
#pragma unroll
    for (int i = 0; i < 7; ++i)
      if (p + i < p1) acc.add(x[i]);
  }
  return acc;
}

// an item's list and where its sums go
struct RedItem {
  const int* slots;
  const void* part;
  // width = 0: nothing to do (its cluster is inactive, or no such item).  An empty
  // list has n = 0 and its sums, zeros, are stored: a free image may observe
  // nothing, and the arena holds whatever an earlier cluster left in it.
  int begin, n, width;
  // lane e of the sums goes to out[(e / 6) ld + e % 6].  The pair block of a
  // cluster of up to kMaxFreeSmall free images goes negated to its place in the
  // lower triangle of S (elimination order; and mirrored to out2): where that
  // is the transposed block, lane e sums element (e % 6, e / 6), so that the
  // stores stay in runs of six.
  double *out, *out2;
  int ld, trans;
};
// the element that lane e sums
__device__ __forceinline__ int red_element(const RedItem& r, int e) { return r.trans ? (e % 6) * 6 + e / 6 : e; }
__device__ __forceinline__ RedItem red_item(const BatchView& bv, int g, int mirror) {
  const int s = find_slot(bv.item_pre, bv.n, g);
  const DevCluster& C = bv.cl[s];
  if (!C.lm->active) return RedItem{};
  const int it = g - bv.item_pre[s];
  const bool cam = it < C.n_free;
  const int key = cam ? it : it - C.n_free;
  const int* begin = (cam ? C.cam_slot_begin : C.pair_slot_begin) + key;
  RedItem r;
  r.begin = begin[0];
  r.n = begin[1] - r.begin;
  r.slots = cam ? C.cam_slots : C.pair_slots;
  r.part = cam ? C.campart : C.pairpart;
  r.out2 = nullptr;
  r.ld = 6;
  r.trans = 0;
  r.width = cam ? 39 : 36;
  if (cam) {
    r.out = C.camsum + (size_t)kCamPart * key;
  } else if (C.n_free > kMaxFreeSmall) {
    r.out = C.pairsum + (size_t)kPairPart * key;
  } else {  // -(sum Z_a Z_b^T): rows a, columns b, or its transpose below the diagonal
    const int n = 6 * C.n_free;
    const int2 ab = C.pair_key[key];
    const int pa = 6 * C.fpos[ab.x], pb = 6 * C.fpos[ab.y];
    double* const rows_a = C.S + (size_t)pa * n + pb;
    double* const rows_b = C.S + (size_t)pb * n + pa;
    r.out = pa > pb ? rows_a : rows_b;
    r.ld = n;
    r.trans = pb > pa;
    if (mirror) r.out2 = pa > pb ? rows_b : rows_a;
    r.width = -36;
  }
  return r;
}
__device__ __forceinline__ void red_store(const RedItem& r, int el, double v) {
  const int i = el / 6, c = el - 6 * i;
  if (r.width < 0) v = -v;
  r.out[(size_t)i * r.ld + c] = v;
  if (r.out2) r.out2[(size_t)c * r.ld + i] = v;
}

template <typename Real>
__global__ void __launch_bounds__(kRedThreads, 6) k_partial_reduce(BatchView bv, int mirror) {
  using Acc = typename AccOf<Real>::T;
  __shared__ typename Acc::Raw sums[2][kRedSegs][kCamPart];  // two items' worth: one barrier per long item
  __shared__ RedItem items[kRedSegs];
  const int seg = threadIdx.x / kCamPart, el = threadIdx.x - seg * kCamPart;
  const int total = bv.tot[2];
  // items a CTA takes at a time: as many as spread the batch over the grid in one round, at most one per group
  const int group = min(kRedSegs, (total + (int)gridDim.x - 1) / (int)gridDim.x);
  int buf = 0;
  for (int g0 = blockIdx.x; g0 < total; g0 += gridDim.x * group) {
    if (threadIdx.x < group) {
      const int g = g0 + threadIdx.x * gridDim.x;
      RedItem r{};
      if (g < total) r = red_item(bv, g, mirror);
      items[threadIdx.x] = r;
    }
    __syncthreads();
    if (seg < group) {  // the short lists, a group each
      const RedItem r = items[seg];
      if (r.n <= kRedLong && el < abs(r.width)) {
        const Real* part = (const Real*)r.part + red_element(r, el);
        const int stride = abs(r.width) == 36 ? kPairPart : kCamPart;
        red_store(r, el, add_rows<Real>(part, stride, r.slots, r.begin, r.begin + r.n).get());
      }
    }
    for (int i = 0; i < group; ++i) {  // the long ones, all groups together
      const RedItem r = items[i];
      if (r.n <= kRedLong) continue;
      const bool live = seg < kRedSegs && el < abs(r.width);
      if (live) {
        const Real* part = (const Real*)r.part + red_element(r, el);
        const int stride = abs(r.width) == 36 ? kPairPart : kCamPart;
        const int per = (r.n + kRedSegs - 1) / kRedSegs;
        const int p0 = r.begin + seg * per, p1 = r.begin + min(r.n, (seg + 1) * per);
        sums[buf][seg][el] = add_rows<Real>(part, stride, r.slots, p0, p1).v;
      }
      __syncthreads();
      if (seg == 0 && live) {
        Acc t{sums[buf][0][el]};
#pragma unroll
        for (int q = 1; q < kRedSegs; ++q) t = acc_join(t, Acc{sums[buf][q][el]});
        red_store(r, el, t.get());
      }
      buf ^= 1;
    }
    __syncthreads();  // items[] is read no more
  }
}

// ------------------------------------------------------------------ K5

// Back-substitution and candidate cost, warp per tile.  Each observation's
// products are formed again from its image's step (obs_step, no Jacobians)
// instead of reading per-observation records back from memory.
template <bool MIXED>
__device__ void backsub_tile(const DevCluster& C, LmState* lm, int local, int lane);

// add a warp's count of finished tiles to its cluster's total; true for the
// warp that completes the total: the cluster's LM step is due
__device__ __forceinline__ bool publish_tiles(const DevCluster& C, int count, int lane) {
  int done = 0;
  if (lane == 0) {
    __threadfence();  // this warp's partial sums before the count
    done = atomicAdd(&C.lm->tiles_done, count) + count;
  }
  done = __shfl_sync(BA_FULL_MASK, done, 0);
  if (done != C.n_tiles) return false;
  __threadfence();
  return true;
}

// Clusters that a CTA's warps complete get their LM step from the whole CTA at
// its end (the sums over a single cluster's 8,000 tiles took one warp 40 of
// the kernel's 62 us); past this many, from the completing warp itself.
constexpr int kMaxDue = 64;

template <bool MIXED>
__global__ void __launch_bounds__(kCostInitThreads) k_backsub_cost(BatchView bv) {
  using Real = typename RealOf<MIXED>::T;
  __shared__ int due[kMaxDue], n_due;
  __shared__ double red[2 * (kCostInitThreads / 32) + 1];
  if (threadIdx.x == 0) n_due = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  const int total = bv.tot[0];
  // few tiles: neighbouring ones go to different CTAs (a CTA of eight tiles
  // would queue on the binary64 pipe of one SM while others have none)
  const int warp = 2 * total <= nwarps ? (threadIdx.x >> 5) * gridDim.x + blockIdx.x
                                       : (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  // each warp takes a contiguous run of tiles, so that its tiles mostly
  // belong to one cluster: it counts them per cluster and publishes the
  // count once per cluster it leaves (one fence and one atomic each); the
  // warp whose count completes a cluster, every other tile's partial sums
  // being written by then, hands the cluster's LM step to its CTA
  const int per = (total + nwarps - 1) / nwarps;
  const int g0 = warp * per, g1 = min(total, g0 + per);
  int s = g0 < g1 ? find_slot(bv.tile_pre, bv.n, g0) : 0;
  int pending = 0;
  auto leave = [&](int slot) {
    if (!pending || !publish_tiles(bv.cl[slot], pending, lane)) return;
    int at = lane == 0 ? atomicAdd(&n_due, 1) : 0;
    at = __shfl_sync(BA_FULL_MASK, at, 0);
    if (at >= kMaxDue) lm_update_warp<MIXED>(bv.cl[slot], lane);
    else if (lane == 0) due[at] = slot;
  };
  for (int g = g0; g < g1; ++g) {
    while (g >= bv.tile_pre[s + 1]) {  // the next cluster: publish the count of this one
      leave(s);
      pending = 0;
      ++s;
    }
    const DevCluster& C = bv.cl[s];
    LmState* lm = C.lm;
    if (!lm->active) continue;
    if (lm->status == 0) backsub_tile<MIXED>(C, lm, g - bv.tile_pre[s], lane);
    ++pending;
  }
  leave(s);
  __syncthreads();
  const int n = min(n_due, kMaxDue);
  for (int i = 0; i < n; ++i) lm_update_cta<MIXED>(bv.cl[due[i]], red);
}

// back-substitution and candidate cost of one tile (one warp)
template <bool MIXED>
__device__ void backsub_tile(const DevCluster& C, LmState* lm, int local, int lane) {
  using Real = typename RealOf<MIXED>::T;
  {
    const Tile tl = C.tiles[local];
    const bool act = lane < tl.n_obs;
    const int o = tl.obs_begin + (act ? lane : 0);
    const int k = act ? C.obs_cam[o] : 0, j = act ? C.obs_pt[o] : -1 - lane;
    int seg_start, seg_end;
    segments(j, lane, seg_start, seg_end);
    const int span = segment_span(seg_start, seg_end);
    const bool head = act && lane == seg_start;
    const int cur = lm->cur;
    // this observation's share of Jp^T (Jc dc)
    Real t[3] = {0, 0, 0};
    if (act) {
      const Real* st = reinterpret_cast<const Real*>(C.dcam) + (size_t)kCamStep * k;
      Real dth[4], dt[4];
      ld4(st, 0, dth);
      ld4(st, 4, dt);
      Real Rm[9], in[7];
      if constexpr (MIXED) {
        const CamDf cd = load_camdf_lin(camdf_ptr(C, cur, k));
        const float2* xp = xdf_ptr(C, cur, j);
        const float2 a = xp[0], b = xp[1], c = xp[2];
#pragma unroll
        for (int i = 0; i < 9; ++i) Rm[i] = cd.R[i].hi;
        in[0] = cd.f.hi; in[1] = 0.f; in[2] = 0.f;
        in[3] = cd.k1.hi; in[4] = cd.k2.hi; in[5] = cd.p1.hi; in[6] = cd.p2.hi;
        const float2 ch = C.obs_chi[o];
        obs_step<Real>(Rm, df_sum_to_f(dfl{a.x, a.y}, df_neg(cd.T[0])), df_sum_to_f(dfl{b.x, b.y}, df_neg(cd.T[1])),
                       df_sum_to_f(dfl{c.x, c.y}, df_neg(cd.T[2])), in, ch.x, ch.y, C.inv_sigma_f, C.delta_f, dth, dt, t);
      } else {
        const double* cr = (const double*)C.camreal + (size_t)kCamReal * k;
#pragma unroll
        for (int i = 0; i < 9; ++i) Rm[i] = cr[i];
#pragma unroll
        for (int i = 0; i < 7; ++i) in[i] = cr[12 + i];
        const double* Xd = C.X + ((size_t)cur * C.n_pts + j) * 3;
        const double2 u = reinterpret_cast<const double2*>(C.obs_uv)[o];
        obs_step<Real>(Rm, Xd[0] - cr[9], Xd[1] - cr[10], Xd[2] - cr[11], in, u.x, u.y, C.inv_sigma, C.huber_delta,
                       dth, dt, t);
      }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) t[i] = seg_reduce(t[i], lane, seg_start, seg_end, span);
    // head: dX = M^T M (g_p - t), candidate point, pred term (M, D_p and g_p as
    // the linearise+Schur kernel of this iteration left them; the difference is
    // taken before M, where it cancels exactly)
    Real dX0 = 0, dX1 = 0, dX2 = 0;
    Real pp = 0;  // dX^T (mu Dp dX + gp)
    if (head) {
      const Real* pb = reinterpret_cast<const Real*>(C.ptblk) + (size_t)j * 16;
      Real w[16];  // m00 m10 m11 m20 m21 m22 q0 q1 q2 d0 d1 d2 g0 g1 g2
      ld4(pb, 0, w); ld4(pb, 4, w + 4); ld4(pb, 8, w + 8); ld4(pb, 12, w + 12);
      Real mu;
      if constexpr (MIXED) mu = lm->mu_f; else mu = lm->mu;
      const Real s0 = w[12] - t[0], s1 = w[13] - t[1], s2 = w[14] - t[2];
      const Real v0 = w[0] * s0;
      const Real v1 = w[1] * s0 + w[2] * s1;
      const Real v2 = w[3] * s0 + w[4] * s1 + w[5] * s2;
      dX0 = w[0] * v0 + w[1] * v1 + w[3] * v2;
      dX1 = w[2] * v1 + w[4] * v2;
      dX2 = w[5] * v2;
      pp = dX0 * (mu * w[9] * dX0 + w[12]) + dX1 * (mu * w[10] * dX1 + w[13]) + dX2 * (mu * w[11] * dX2 + w[14]);
    }
    double cost = 0.0;
    if constexpr (MIXED) {
      dfl x0{0.f, 0.f}, x1{0.f, 0.f}, x2{0.f, 0.f};
      if (head) {
        const float2* xp = xdf_ptr(C, cur, j);
        const float2 a = xp[0], b = xp[1], c = xp[2];
        x0 = df_add_f(dfl{a.x, a.y}, dX0);
        x1 = df_add_f(dfl{b.x, b.y}, dX1);
        x2 = df_add_f(dfl{c.x, c.y}, dX2);
        float2* xn = xdf_wptr(C, cur ^ 1, j);
        xn[0] = make_float2(x0.hi, x0.lo);
        xn[1] = make_float2(x1.hi, x1.lo);
        xn[2] = make_float2(x2.hi, x2.lo);
      }
      x0.hi = __shfl_sync(BA_FULL_MASK, x0.hi, seg_start); x0.lo = __shfl_sync(BA_FULL_MASK, x0.lo, seg_start);
      x1.hi = __shfl_sync(BA_FULL_MASK, x1.hi, seg_start); x1.lo = __shfl_sync(BA_FULL_MASK, x1.lo, seg_start);
      x2.hi = __shfl_sync(BA_FULL_MASK, x2.hi, seg_start); x2.lo = __shfl_sync(BA_FULL_MASK, x2.lo, seg_start);
      dfl cst{0.f, 0.f};
      if (act) {
        const CamDf cdf = load_camdf(camdf_ptr(C, cur ^ 1, k));
        const float2 ch = C.obs_chi[o], cl = C.obs_clo[o];
        dfl e0, e1;
        if (df_residual(cdf, x0, x1, x2, dfl{ch.x, cl.x}, dfl{ch.y, cl.y}, e0, e1))
          cst = df_robust_cost(e0, e1, C.delta_f, C.half_inv_s2_f);
      }
      // fixed-order warp sum in double-float, one conversion per warp
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const dfl o2{__shfl_down_sync(BA_FULL_MASK, cst.hi, off), __shfl_down_sync(BA_FULL_MASK, cst.lo, off)};
        cst = df_add(cst, o2);
      }
      if (lane == 0) cost = df_to_d(cst);
    } else {
      double x0 = 0.0, x1 = 0.0, x2 = 0.0;
      if (head) {
        const double* X = C.X + ((size_t)cur * C.n_pts + j) * 3;
        x0 = X[0] + (double)dX0;
        x1 = X[1] + (double)dX1;
        x2 = X[2] + (double)dX2;
        double* Xn = C.X + ((size_t)(cur ^ 1) * C.n_pts + j) * 3;
        Xn[0] = x0; Xn[1] = x1; Xn[2] = x2;
      }
      x0 = __shfl_sync(BA_FULL_MASK, x0, seg_start);
      x1 = __shfl_sync(BA_FULL_MASK, x1, seg_start);
      x2 = __shfl_sync(BA_FULL_MASK, x2, seg_start);
      if (act) {
        const double Xn[3] = {x0, x1, x2};
        const double* Rn = C.R + ((size_t)(cur ^ 1) * C.n_cams + k) * 9;
        const double* Tn = C.T + ((size_t)(cur ^ 1) * C.n_cams + k) * 3;
        const double2 u = reinterpret_cast<const double2*>(C.obs_uv)[o];
        cost = obs_cost(Rn, Tn, C.intr + 7 * k, Xn, u.x, u.y, C.half_inv_s2, C.huber_delta);
      }
      cost = warp_sum(cost);
    }
    double ppred;
    if constexpr (MIXED) {
      const float ps = warp_sum(pp);  // binary32 warp sum, one conversion per warp
      ppred = lane == 0 ? (double)ps : 0.0;
    } else {
      ppred = warp_sum((double)pp);
    }
    if (lane == 0) {
      C.tilepart[2 * local] = cost;
      C.tilepart[2 * local + 1] = ppred;
    }
  }
}

// ------------------------------------------------------------------ cost at the current state

template <bool MIXED>
__global__ void __launch_bounds__(256) k_cost_tiles(BatchView bv) {
  const int lane = threadIdx.x & 31;
  const int warp = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;  // few tiles spread over the SMs
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  const int total = bv.tot[0];
  for (int g = warp; g < total; g += nwarps) {
    const int s = find_slot(bv.tile_pre, bv.n, g);
    const DevCluster& C = bv.cl[s];
    const LmState* lm = C.lm;
    if (!lm->needs_init) continue;
    const int local = g - bv.tile_pre[s];
    const Tile tl = C.tiles[local];
    const int cur = lm->cur;
    double cost = 0.0;
    if constexpr (MIXED) {
      dfl cst{0.f, 0.f};
      if (lane < tl.n_obs) {
        const int o = tl.obs_begin + lane;
        const int k = C.obs_cam[o], j = C.obs_pt[o];
        const CamDf cdf = load_camdf(camdf_ptr(C, cur, k));
        const float2* xp = xdf_ptr(C, cur, j);
        const float2 a = xp[0], b = xp[1], c = xp[2];
        const float2 ch = C.obs_chi[o], cl = C.obs_clo[o];
        dfl e0, e1;
        if (df_residual(cdf, dfl{a.x, a.y}, dfl{b.x, b.y}, dfl{c.x, c.y}, dfl{ch.x, cl.x}, dfl{ch.y, cl.y}, e0, e1))
          cst = df_robust_cost(e0, e1, C.delta_f, C.half_inv_s2_f);
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const dfl o2{__shfl_down_sync(BA_FULL_MASK, cst.hi, off), __shfl_down_sync(BA_FULL_MASK, cst.lo, off)};
        cst = df_add(cst, o2);
      }
      if (lane == 0) cost = df_to_d(cst);
    } else {
      if (lane < tl.n_obs) {
        const int o = tl.obs_begin + lane;
        const int k = C.obs_cam[o], j = C.obs_pt[o];
        const double2 u = reinterpret_cast<const double2*>(C.obs_uv)[o];
        cost = obs_cost(C.R + ((size_t)cur * C.n_cams + k) * 9, C.T + ((size_t)cur * C.n_cams + k) * 3,
                        C.intr + 7 * k, C.X + ((size_t)cur * C.n_pts + j) * 3, u.x, u.y,
                        C.half_inv_s2, C.huber_delta);
      }
      cost = warp_sum(cost);
    }
    if (lane == 0) C.tilepart[2 * local] = cost;
  }
}

// fixed-order block sum of tilepart[:, which]
__device__ double block_sum_tiles(const DevCluster& C, int which, double* red) {
  double v = 0.0;
  for (int i = threadIdx.x; i < C.n_tiles; i += blockDim.x) v += C.tilepart[2 * i + which];
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double tot = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
  __syncthreads();
  return tot;  // valid in thread 0
}

// Fixed-order sum over the block (warp trees, then the warps in order);
// valid in thread 0.
__device__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double tot = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
  __syncthreads();
  return tot;
}

__global__ void __launch_bounds__(256) k_cost_init(BatchView bv) {
  __shared__ double red[8], prior[kMaxFreeSmall];
  for (int s = blockIdx.x; s < bv.n; s += gridDim.x) {
    const DevCluster& C = bv.cl[s];
    LmState* lm = C.lm;
    if (!lm->needs_init) continue;
    const double F = block_sum_tiles(C, 0, red);
    const int cur = lm->cur;
    const double* R = C.R + (size_t)cur * C.n_cams * 9;
    const double* T = C.T + (size_t)cur * C.n_cams * 3;
    double pc = 0.0;
    if (C.n_free <= kMaxFreeSmall) {
      // as the factor kernel forms it at a candidate, so that F carried from
      // there and F evaluated here are the same bits
      if (threadIdx.x < 4 * C.n_free) {
        const int f = threadIdx.x >> 2, k = C.cam_of_free[f], q = min((int)threadIdx.x & 3, 2);
        const double v = prior_cost_quad(0xfu << ((threadIdx.x & 31) & ~3), C, k, R + 9 * k, T + 3 * k, q);
        if ((threadIdx.x & 3) == 0) prior[f] = v;
      }
      __syncthreads();
      if (threadIdx.x < 32) pc = strided_sum(prior, C.n_free, threadIdx.x);
    } else {
      // thread t takes images t, t + blockDim.x, ... in order
      for (int k = threadIdx.x; k < C.n_cams; k += blockDim.x) {
        if (C.free_idx[k] < 0) continue;
        pc += prior_terms(R + 9 * k, T + 3 * k, C.R_prior + 9 * k, C.T_prior + 3 * k, C.sigma_imu, C.sigma_gnss, nullptr,
                          nullptr);
      }
      pc = block_sum(pc, red);
    }
    if (threadIdx.x == 0) {
      lm->needs_init = 0;
      lm->F = F + pc;
      lm->pt_fail = 0;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ K6

// ------------------------------------------------------------------ diagnostics

__global__ void k_grad_norm(BatchView bv, double* out) {
  __shared__ double red[8];
  for (int s = blockIdx.x; s < bv.n; s += gridDim.x) {
    const DevCluster& C = bv.cl[s];
    double m = 0.0;
    for (int i = threadIdx.x; i < 6 * C.n_free; i += blockDim.x) m = fmax(m, fabs(C.gc[i]));
    for (int t = threadIdx.x; t < C.n_tiles; t += blockDim.x) m = fmax(m, C.tilepart[2 * t + 1]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_down_sync(BA_FULL_MASK, m, off));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
      double v = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v = fmax(v, red[w]);
      out[s] = v;
    }
    __syncthreads();
  }
}

__device__ __forceinline__ void point_f64(const DevCluster& C, bool mixed, int buf, int j, double X[3]) {
  if (mixed) {
    const float2* p = xdf_ptr(C, buf, j);
    for (int i = 0; i < 3; ++i) X[i] = (double)p[i].x + (double)p[i].y;
  } else {
    const double* p = C.X + ((size_t)buf * C.n_pts + j) * 3;
    for (int i = 0; i < 3; ++i) X[i] = p[i];
  }
}

__global__ void k_reproj(const DevCluster* dcl, int mixed, double* err) {
  const DevCluster& C = *dcl;
  const int cur = C.lm->cur;
  for (int o = blockIdx.x * blockDim.x + threadIdx.x; o < C.n_obs; o += gridDim.x * blockDim.x) {
    const int k = C.obs_cam[o], j = C.obs_pt[o];
    const double2 u = reinterpret_cast<const double2*>(C.obs_uv)[o];
    double X[3];
    point_f64(C, mixed, cur, j, X);
    err[o] = obs_error_norm(C.R + ((size_t)cur * C.n_cams + k) * 9, C.T + ((size_t)cur * C.n_cams + k) * 3,
                            C.intr + 7 * k, X, u.x, u.y);
  }
}

// The current state in the caller's layout, binary64: R [nc][9] and T [nc][3]
// of the current buffer, X [np][3] in the caller's point order (any output
// may be null).
__global__ void k_export_state(const DevCluster* dcl, int mixed, double* R, double* T, double* out) {
  const DevCluster& C = *dcl;
  const int cur = C.lm->cur;
  const int stride = gridDim.x * blockDim.x;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 12 * C.n_cams; i += stride) {
    if (i < 9 * C.n_cams) {
      if (R) R[i] = C.R[(size_t)cur * C.n_cams * 9 + i];
    } else if (T) {
      T[i - 9 * C.n_cams] = C.T[(size_t)cur * C.n_cams * 3 + i - 9 * C.n_cams];
    }
  }
  if (!out) return;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < C.n_pts; j += stride) {
    double X[3];
    point_f64(C, mixed, cur, j, X);
    const int u = C.pt_perm[j];  // caller's index
    out[3 * u] = X[0];
    out[3 * u + 1] = X[1];
    out[3 * u + 2] = X[2];
  }
}

// ------------------------------------------------------------------ run control

// Arm every cluster of the batch for `iters` more iterations (iters < 0:
// mark active without a target, for the diagnostic linearisation).
__global__ void k_arm(BatchView bv, int iters) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < bv.n; s += gridDim.x * blockDim.x) {
    LmState* lm = bv.cl[s].lm;
    if (iters >= 0) {
      lm->iters_target = lm->iter + iters;
      lm->active = iters > 0;
    } else {
      lm->active = iters == -1;
    }
    lm->needs_init = 1;
    lm->pt_fail = 0;
    lm->iter0 = lm->iter;
    lm->ftol = 0.0;
  }
}

// Serving slots: arm[s] > 0 starts arm[s] more iterations for slot s (and asks
// for F at its state first), ending early on convergence when ftol[s] > 0; 0
// leaves the slot as it is.
__global__ void k_arm_slots(BatchView bv, const int* arm, const double* ftol) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < bv.n; s += gridDim.x * blockDim.x) {
    const int a = arm[s];
    if (a <= 0) continue;
    LmState* lm = bv.cl[s].lm;
    lm->iters_target = lm->iter + a;
    lm->active = 1;
    lm->needs_init = 1;
    lm->pt_fail = 0;
    lm->iter0 = lm->iter;
    lm->ftol = ftol[s];
  }
}

// Warm start: copy the current state of shared cameras and points from a live
// cluster (src) into a new one (dst): both state buffers and the reset state.
// cams / pts hold (dst index, src index) pairs in internal order.  The copy is
// representation-agnostic (8-byte words), so both clusters must use the same
// precision.
// Cluster transition (Sec. 3.2, Eq. 8): an image free in dst and shared with
// src takes the weighted average of its two current poses, weights = its
// observations in each cluster; orientation at fraction w_dst / (w_src +
// w_dst) along the geodesic from the src orientation, position the weighted
// mean.  Binary64.  pairs[i] = (camera in dst, camera in src).
__global__ void k_transition(const DevCluster* dst, const DevCluster* src, const int2* pairs, int n) {
  const DevCluster& D = *dst;
  const DevCluster& S = *src;
  const int dcur = D.lm->cur, scur = S.lm->cur;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int kd = pairs[i].x, ks = pairs[i].y;
    if (D.free_idx[kd] < 0) continue;  // fixed in dst: already the src pose
    const double wo = (double)S.cam_nobs[ks], wn = (double)D.cam_nobs[kd];
    if (!(wo + wn > 0.0)) continue;
    const double t = wn / (wo + wn);
    const double* Ro = S.R + ((size_t)scur * S.n_cams + ks) * 9;
    const double* To = S.T + ((size_t)scur * S.n_cams + ks) * 3;
    double* Rn = D.R + ((size_t)dcur * D.n_cams + kd) * 9;
    double* Tn = D.T + ((size_t)dcur * D.n_cams + kd) * 3;
    double E[9], phi[3], Q[9], Rm[9];
    for (int a = 0; a < 3; ++a)  // E = Ro^T Rn
      for (int b = 0; b < 3; ++b) E[3 * a + b] = Ro[a] * Rn[b] + Ro[3 + a] * Rn[3 + b] + Ro[6 + a] * Rn[6 + b];
    so3_log(E, phi);
    for (int a = 0; a < 3; ++a) phi[a] *= t;
    so3_exp(phi, Q);
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) Rm[3 * a + b] = Ro[3 * a] * Q[b] + Ro[3 * a + 1] * Q[3 + b] + Ro[3 * a + 2] * Q[6 + b];
    for (int a = 0; a < 9; ++a) Rn[a] = Rm[a];
    for (int a = 0; a < 3; ++a) Tn[a] = (wo * To[a] + wn * Tn[a]) / (wo + wn);
  }
}

__global__ void k_warm_copy(const DevCluster* dst, const DevCluster* src, const int2* cams, int n_cams,
                            const int2* pts, int n_pts) {
  const int scur = src->lm->cur;
  const int stride = gridDim.x * blockDim.x;
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // the damping state goes with the poses and points
    LmState* dl = dst->lm;
    const LmState* sl = src->lm;
    dl->mu = dl->mu0 = sl->mu;
    dl->mu_f = (float)sl->mu;
    dl->nu = dl->nu0 = sl->nu;
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_pts; i += stride) {
    const int2 p = pts[i];
    const double* sx = src->X + ((size_t)scur * src->n_pts + p.y) * 3;
    for (int a = 0; a < 3; ++a) {
      const double v = sx[a];
      dst->X[(size_t)p.x * 3 + a] = v;
      dst->X[((size_t)dst->n_pts + p.x) * 3 + a] = v;
      const_cast<double*>(dst->X_init)[(size_t)p.x * 3 + a] = v;
    }
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_cams; i += stride) {
    const int2 p = cams[i];
    const double* sr = src->R + ((size_t)scur * src->n_cams + p.y) * 9;
    const double* st = src->T + ((size_t)scur * src->n_cams + p.y) * 3;
    for (int b = 0; b < 2; ++b) {
      for (int a = 0; a < 9; ++a) dst->R[((size_t)b * dst->n_cams + p.x) * 9 + a] = sr[a];
      for (int a = 0; a < 3; ++a) dst->T[((size_t)b * dst->n_cams + p.x) * 3 + a] = st[a];
    }
    for (int a = 0; a < 9; ++a) const_cast<double*>(dst->R_init)[(size_t)p.x * 9 + a] = sr[a];
    for (int a = 0; a < 3; ++a) const_cast<double*>(dst->T_init)[(size_t)p.x * 3 + a] = st[a];
  }
}

// Restore the state given at create into both state buffers and reset LM
// control.  The copy is representation-agnostic (8-byte words).
__global__ void k_reset(BatchView bv) {
  for (int s = blockIdx.y; s < bv.n; s += gridDim.y) {
    const DevCluster& C = bv.cl[s];
    const size_t nr = (size_t)C.n_cams * 9, nt = (size_t)C.n_cams * 3, nx = (size_t)C.n_pts * 3;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nx; i += (size_t)gridDim.x * blockDim.x) {
      const double v = C.X_init[i];
      C.X[i] = v;
      C.X[nx + i] = v;
    }
    if (blockIdx.x == 0) {
      for (size_t i = threadIdx.x; i < nr; i += blockDim.x) { C.R[i] = C.R_init[i]; C.R[nr + i] = C.R_init[i]; }
      for (size_t i = threadIdx.x; i < nt; i += blockDim.x) { C.T[i] = C.T_init[i]; C.T[nt + i] = C.T_init[i]; }
      if (threadIdx.x == 0) {
        LmState* lm = C.lm;
        lm->mu = lm->mu0;
        lm->mu_f = (float)lm->mu0;
        lm->nu = lm->nu0;
        lm->F = 0.0;
        lm->F_new = 0.0;
        lm->cur = 0;
        lm->status = 0;
        lm->iter = 0;
        lm->n_accepted = 0;
        lm->active = 0;
        lm->iters_target = 0;
        lm->pt_fail = 0;
        lm->dev_error = 0;
      }
    }
  }
}

// Copy LM control and the last `iters` trace records of every cluster into
// contiguous buffers ([n] and [n][iters]).
__global__ void k_gather(BatchView bv, int iters, LmState* lm_out, StepRec* trace_out) {
  for (int s = blockIdx.x; s < bv.n; s += gridDim.x) {
    const DevCluster& C = bv.cl[s];
    if (threadIdx.x == 0 && lm_out) lm_out[s] = *C.lm;
    if (trace_out && C.trace_cap > 0) {
      const int end = C.lm->iter;
      for (int i = threadIdx.x; i < iters; i += blockDim.x) {
        const int it = end - iters + i;
        if (it >= 0) trace_out[(size_t)s * iters + i] = C.trace[it % C.trace_cap];
      }
    }
  }
}

// ------------------------------------------------------------------ launchers
//
// Every launch goes through LAUNCH(kind, ...): it counts the launch (as a
// direct launch, or as a kernel node when the stream is being captured) and,
// when a probe is attached to the calling thread, brackets the kernel with
// CUDA events (captured as event-record nodes inside graphs).

static thread_local Probe* t_probe = nullptr;
static thread_local unsigned long long t_direct = 0, t_captured = 0;

void set_probe(Probe* p) { t_probe = p; }
bool probe_attached() { return t_probe != nullptr; }
unsigned long long take_direct_launches() {
  const unsigned long long v = t_direct;
  t_direct = 0;
  return v;
}
unsigned long long take_captured_launches() {
  const unsigned long long v = t_captured;
  t_captured = 0;
  return v;
}

static bool capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(st, &cs);
  return cs == cudaStreamCaptureStatusActive;
}

static void probe_mark(cudaStream_t st, cudaEvent_t* out) {
  cudaEventCreate(out);
  if (capturing(st)) cudaEventRecordWithFlags(*out, st, cudaEventRecordExternal);
  else cudaEventRecord(*out, st);
}

LaunchScope::LaunchScope(int k, cudaStream_t s) : kind(k), st(s) {
  if (t_probe) probe_mark(st, &e0);
}

LaunchScope::~LaunchScope() {
  if (capturing(st)) ++t_captured; else ++t_direct;
  if (t_probe) {
    cudaEvent_t e1;
    probe_mark(st, &e1);
    t_probe->recs.push_back(ProbeRec{kind, e0, e1});
  }
}

static int grid_for(int items, int per_block, int cap) {
  int g = (items + per_block - 1) / per_block;
  if (g > cap) g = cap;
  return g < 1 ? 1 : g;
}

static int g_num_sms = 0;
int num_sms() {
  if (!g_num_sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_num_sms <= 0) g_num_sms = 1;
  }
  return g_num_sms;
}

void launch_arm(const BatchView& bv, int iters, cudaStream_t st) {
  LAUNCH(KK_OTHER, st, k_arm<<<(bv.n + 127) / 128, 128, 0, st>>>(bv, iters));
}

void launch_arm_slots(const BatchView& bv, const int* arm, const double* ftol, cudaStream_t st) {
  LAUNCH(KK_OTHER, st, k_arm_slots<<<(bv.n + 127) / 128, 128, 0, st>>>(bv, arm, ftol));
}

void launch_warm_copy(const DevCluster* dst, const DevCluster* src, const int2* cams, int n_cams, const int2* pts,
                      int n_pts, cudaStream_t st) {
  const int n = n_pts > n_cams ? n_pts : n_cams;
  LAUNCH(KK_OTHER, st,
         k_warm_copy<<<grid_for(n, 256, num_sms() * 4), 256, 0, st>>>(dst, src, cams, n_cams, pts, n_pts));
}

void launch_transition(const DevCluster* dst, const DevCluster* src, const int2* pairs, int n, cudaStream_t st) {
  LAUNCH(KK_OTHER, st, k_transition<<<grid_for(n, 128, 1024), 128, 0, st>>>(dst, src, pairs, n));
}

void launch_camreal(const BatchView& bv, bool mixed, cudaStream_t st) {
  if (mixed) LAUNCH(KK_OTHER, st, k_camdf_all<<<grid_for(bv.n, 1, 65535), 64, 0, st>>>(bv));
  else LAUNCH(KK_OTHER, st, k_camreal<<<grid_for(bv.n, 1, 65535), 64, 0, st>>>(bv));
}

void launch_reset(const BatchView& bv, bool mixed, cudaStream_t st) {
  dim3 grid(64, bv.n < 65535 ? bv.n : 65535);
  LAUNCH(KK_OTHER, st, k_reset<<<grid, 256, 0, st>>>(bv));
  launch_camreal(bv, mixed, st);
}

void launch_gather(const BatchView& bv, int iters, LmState* lm_out, StepRec* trace_out, cudaStream_t st) {
  LAUNCH(KK_OTHER, st, k_gather<<<bv.n < 65535 ? bv.n : 65535, 128, 0, st>>>(bv, iters, lm_out, trace_out));
}

// tiles a CTA of eight warps is launched for: in binary64 one where that leaves
// at most eight CTAs per SM (6 images: back-substitution 29 -> 22 us; in mixed
// precision, not bound by a pipe of the SM, 12 images took 958 instead of 908 us
// per 10 iterations that way)
static int tiles_per_cta(const BatchView& bv, bool mixed) { return !mixed && bv.total_tiles <= 8 * num_sms() ? 1 : 8; }

template <bool MIXED>
static void launch_cost_init_t(const BatchView& bv, cudaStream_t st) {
  const int sms = num_sms();
  LAUNCH(KK_COST_TILES, st, k_cost_tiles<MIXED><<<grid_for(bv.total_tiles, tiles_per_cta(bv, MIXED), sms * 16), 256, 0, st>>>(bv));
  LAUNCH(KK_COST_INIT, st, k_cost_init<<<grid_for(bv.n, 1, 65535), kCostInitThreads, 0, st>>>(bv));
}

void launch_cost_init(const BatchView& bv, bool mixed, cudaStream_t st) {
  if (mixed) launch_cost_init_t<true>(bv, st);
  else launch_cost_init_t<false>(bv, st);
}

int chunk_obs(bool mixed) { return mixed ? kChunkObsMixed : kChunkObsF64; }
int chunk_tiles(bool mixed) { return mixed ? kChunkTilesMixed : kChunkTilesF64; }

static size_t chunk_smem_bytes(bool mixed) {
  // records (later overlaid by the lane partials); mixed path: the chunk
  // staging, its barrier, a flag and the failure-injection barrier
  return chunk_records_bytes(mixed) + (mixed ? (size_t)kStageBytes + 24 : 0);
}

template <bool MIXED>
static void launch_lin_schur(const BatchView& bv, int diag, cudaStream_t st) {
  LAUNCH(KK_LIN_SCHUR, st,
         k_lin_schur<MIXED><<<grid_for(bv.total_chunks, 1, num_sms() * bv.lin_ctas_per_sm), kChunkThreads,
                              chunk_smem_bytes(MIXED),
                              st>>>(bv, diag));
}


template <bool MIXED>
static void launch_partial_reduce(const BatchView& bv, int mirror, cudaStream_t st) {
  using Real = typename RealOf<MIXED>::T;
  LAUNCH(KK_PARTIAL_REDUCE, st,
         k_partial_reduce<Real><<<grid_for(bv.total_items, 1, num_sms() * kRedCtasPerSm), kRedThreads, 0, st>>>(bv, mirror));
}

template <bool MIXED>
static void launch_iteration_t(const BatchView& bv, int refine_steps, cudaStream_t st, const std::vector<BigRef>* big) {
  const int sms = num_sms();
  launch_lin_schur<MIXED>(bv, 0, st);
  launch_partial_reduce<MIXED>(bv, refine_steps > 0, st);
  launch_factor(bv, MIXED, refine_steps, 0, st);
  if (big)
    for (const BigRef& b : *big) launch_big_solve(b, MIXED, refine_steps, 0, st);
  LAUNCH(KK_BACKSUB, st,
         k_backsub_cost<MIXED><<<grid_for(bv.total_tiles, tiles_per_cta(bv, MIXED), sms * bv.back_ctas_per_sm),
                                 kCostInitThreads, 0, st>>>(bv));
}

void launch_iteration(const BatchView& bv, bool mixed, int refine_steps, cudaStream_t st,
                      const std::vector<BigRef>* big) {
  if (mixed) launch_iteration_t<true>(bv, refine_steps, st, big);
  else launch_iteration_t<false>(bv, refine_steps, st, big);
}

template <bool MIXED>
static void launch_grad_norm_t(const BatchView& bv, double* out, cudaStream_t st, const std::vector<BigRef>* big) {
  launch_lin_schur<MIXED>(bv, 1, st);
  launch_partial_reduce<MIXED>(bv, 0, st);
  launch_factor(bv, MIXED, 0, 1, st);
  if (big)
    for (const BigRef& b : *big) launch_big_solve(b, MIXED, 0, 1, st);
  LAUNCH(KK_OTHER, st, k_grad_norm<<<grid_for(bv.n, 1, 65535), 256, 0, st>>>(bv, out));
}

void launch_grad_norm(const BatchView& bv, bool mixed, double* out, cudaStream_t st, const std::vector<BigRef>* big) {
  if (mixed) launch_grad_norm_t<true>(bv, out, st, big);
  else launch_grad_norm_t<false>(bv, out, st, big);
}

void launch_reproj(const DevCluster* dcl, const DevCluster& hcl, bool mixed, double* err_pm, cudaStream_t st) {
  LAUNCH(KK_OTHER, st, k_reproj<<<grid_for(hcl.n_obs, 256, num_sms() * 8), 256, 0, st>>>(dcl, mixed, err_pm));
}

void launch_export_state(const DevCluster* dcl, const DevCluster& hcl, bool mixed, double* R, double* T, double* X,
                         cudaStream_t st) {
  const int items = hcl.n_pts > 12 * hcl.n_cams ? hcl.n_pts : 12 * hcl.n_cams;
  LAUNCH(KK_OTHER, st, k_export_state<<<grid_for(items, 256, num_sms() * 8), 256, 0, st>>>(dcl, mixed, R, T, X));
}

// binary32 FMA-rate probe: 16 independent chains per thread (enough to
// cover the pipe's latency), the result stored only if it comes out as an
// impossible value so that nothing is optimised away
__global__ void __launch_bounds__(512) k_fma_probe(int iters, float seed, float* sink) {
  float a[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) a[i] = seed + (float)(threadIdx.x + i);
  const float m = 0.999999f, c = 1e-7f;
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = __fmaf_rn(a[i], m, c);
  }
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 16; ++i) s += a[i];
  if (s == -1.0f) *sink = s;
}

void launch_fma_probe(int ctas, int iters, float* sink, cudaStream_t st) {
  LAUNCH(KK_OTHER, st, k_fma_probe<<<ctas, 512, 0, st>>>(iters, 1.0f, sink));
}

cudaError_t set_kernel_attributes(int max_n) {
  cudaError_t e = set_factor_attributes(max_n);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_lin_schur<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)chunk_smem_bytes(true));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_lin_schur<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)chunk_smem_bytes(false));
}

}  // namespace bagpu
