// Image footprints on a DSM and their overlaps (Sec. 3.1: the four image
// corners projected onto the surface model; cross-strip overlap detection by
// comparing projected footprints, used to form the clusters of Sec. 3.2).
//
//   k_range      the raster's height range, and whether it is finite
//   k_footprint  one warp per (image, corner): the ray from the camera
//                centre through the corner pixel (no lens distortion) is
//                sampled from where it enters the DSM's height range, in
//                steps of at most half a raster cell horizontally; the first
//                sample at or below the bilinear surface brackets the first
//                hit, refined by a fixed number of bisections.  Binary64.
//   k_overlap    one thread per (footprint a, footprint b): area of the
//                intersection of the two convex ground quadrilaterals by
//                Sutherland-Hodgman clipping and the shoelace formula.
#include <cuda_runtime.h>
#include <math.h>

#include "ba_internal.h"

namespace bagpu {

namespace {

__device__ double dsm_height(const DsmView& D, double x, double y) {
  double fx = (x - D.x0) / D.dx, fy = (y - D.y0) / D.dy;
  fx = fmin(fmax(fx, 0.0), (double)(D.nx - 1));
  fy = fmin(fmax(fy, 0.0), (double)(D.ny - 1));
  int ix = (int)fx, iy = (int)fy;
  ix = min(ix, D.nx - 2);
  iy = min(iy, D.ny - 2);
  const double ax = fx - ix, ay = fy - iy;
  const double* h = D.h + (size_t)iy * D.nx + ix;
  const double h0 = h[0] * (1.0 - ax) + h[1] * ax;
  const double h1 = h[D.nx] * (1.0 - ax) + h[D.nx + 1] * ax;
  return h0 * (1.0 - ay) + h1 * ay;
}

// Height range of the raster and whether every height is finite: out[0] and
// out[1] the bits of the smallest and largest height as integers in the order of
// the numbers, out[2] nonzero when one is not finite (all set by k_range_init).
__device__ __forceinline__ long long order_of(double h) {
  const long long b = __double_as_longlong(h);
  return b < 0 ? (long long)0x8000000000000000ull - b : b;
}
__device__ __forceinline__ double of_order(long long k) {
  return __longlong_as_double(k < 0 ? (long long)0x8000000000000000ull - k : k);
}
__global__ void k_range_init(long long* out) {
  out[0] = 0x7fffffffffffffffll;
  out[1] = -0x7fffffffffffffffll;
  out[2] = 0;
}
__global__ void __launch_bounds__(256) k_range(const double* h, size_t n, long long* out) {
  long long lo = 0x7fffffffffffffffll, hi = -0x7fffffffffffffffll;
  int bad = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const double v = h[i];
    bad |= ((__double_as_longlong(v) >> 52) & 0x7ff) == 0x7ff;
    const long long k = order_of(v);
    lo = min(lo, k);
    hi = max(hi, k);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, off));
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, off));
  }
  bad = __any_sync(0xffffffffu, bad);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&out[0], lo);
    atomicMax(&out[1], hi);
    if (bad) atomicMax(&out[2], 1ll);
  }
}

// A warp per ray.  The march and the bisection are chains of evaluations that
// each wait for the raster's heights and for some thirty binary64
// instructions (64 cycles each): one thread per ray took about a hundred of
// them in a row.  The warp evaluates 32 samples of the march at once, and of
// the bisection the 31 midpoints that the next five halvings can reach, then
// walks the five outcomes: the same samples, the same midpoints, the same
// result, in 12 rounds instead of 60.
__global__ void __launch_bounds__(128) k_footprint(int n, const double* intr, double width, double height,
                                                   const double* R, const double* T, DsmView D, const long long* range,
                                                   double* corners) {
  const int lane = threadIdx.x & 31;
  if (range[2]) return;  // the call is refused
  const double hmin = of_order(range[0]), hmax = of_order(range[1]);
  for (int id = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; id < 4 * n; id += (gridDim.x * blockDim.x) >> 5) {
    const int k = id >> 2, c = id & 3;
    const double* in = intr + 7 * k;
    const double* Rk = R + 9 * k;
    const double* Tk = T + 3 * k;
    const double u = (c == 1 || c == 2) ? width : 0.0, v = (c >= 2) ? height : 0.0;
    const double a = (u - in[1]) / in[0], b = (v - in[2]) / in[0];
    double d[3];
    for (int i = 0; i < 3; ++i) d[i] = Rk[3 * i] * a + Rk[3 * i + 1] * b + Rk[3 * i + 2];
    double* P = corners + 3 * id;
    if (!(d[2] < 0.0)) {  // the ray does not point down
      if (lane < 3) P[lane] = nan("");
      continue;
    }
    auto below = [&](double t) {  // at or below the surface
      return Tk[2] + t * d[2] - dsm_height(D, Tk[0] + t * d[0], Tk[1] + t * d[1]) <= 0.0;
    };
    double t0 = (Tk[2] - hmax) / (-d[2]);
    const double t1 = (Tk[2] - hmin) / (-d[2]);
    if (t0 < 0.0) t0 = 0.0;
    const double dxy = sqrt(d[0] * d[0] + d[1] * d[1]);
    const double cell = fmin(D.dx, D.dy);
    int m = 1;
    if (dxy > 0.0) {
      const double steps = ceil((t1 - t0) * dxy / (0.5 * cell));
      m = steps < 1.0 ? 1 : (steps > (double)kDsmMaxSteps ? kDsmMaxSteps : (int)steps);
    }
    double lo = t0, hi = t1;
    for (int i0 = 1; i0 <= m; i0 += 32) {
      const int i = i0 + lane;
      const bool hit = i <= m && below(t0 + (t1 - t0) * i / m);
      const unsigned first = __ballot_sync(0xffffffffu, hit);
      if (first) {
        const int f = i0 + __ffs(first) - 1;
        hi = t0 + (t1 - t0) * f / m;
        lo = t0 + (t1 - t0) * (f - 1) / m;
        break;
      }
    }
    static_assert(kDsmBisect % 5 == 0, "five halvings a round");
    for (int it = 0; it < kDsmBisect; it += 5) {
      // lane q >= 1: node q of the tree of midpoints (children 2 q: upper half,
      // reached when the midpoint lies above the surface, and 2 q + 1: lower)
      double l = lo, h = hi;
      const int q = lane == 0 ? 1 : lane, depth = 31 - __clz(q);
      for (int s = depth - 1; s >= 0; --s) {
        const double mid = 0.5 * (l + h);
        if ((q >> s) & 1) h = mid; else l = mid;
      }
      const unsigned under = __ballot_sync(0xffffffffu, below(0.5 * (l + h)));
      int node = 1;
      for (int s = 0; s < 5; ++s) {
        const double mid = 0.5 * (lo + hi);
        const int bit = (under >> node) & 1;
        if (bit) hi = mid; else lo = mid;
        node = 2 * node + bit;
      }
    }
    if (lane < 3) P[lane] = Tk[lane] + hi * (lane == 0 ? d[0] : (lane == 1 ? d[1] : d[2]));
  }
}

__device__ double poly_area2(const double* p, int n) {
  double s = 0.0;
  for (int i = 0; i < n; ++i) {
    const int j = (i + 1 == n) ? 0 : i + 1;
    s += p[2 * i] * p[2 * j + 1] - p[2 * j] * p[2 * i + 1];
  }
  return 0.5 * s;
}

__global__ void k_overlap(int na, const double* qa, int nb, const double* qb, double* area) {
  for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < na * nb; id += gridDim.x * blockDim.x) {
    const int ia = id / nb, ib = id - ia * nb;
    const double* A = qa + 12 * ia;
    const double* B = qb + 12 * ib;
    double Bx[8];
    for (int i = 0; i < 4; ++i) {
      Bx[2 * i] = B[3 * i];
      Bx[2 * i + 1] = B[3 * i + 1];
    }
    const double sb = poly_area2(Bx, 4) >= 0.0 ? 1.0 : -1.0;  // orientation of the clipper
    double P[16], Q[16];  // a convex quadrilateral clipped by four half-planes has at most 8 vertices
    int np = 4;
    for (int i = 0; i < 4; ++i) {
      P[2 * i] = A[3 * i];
      P[2 * i + 1] = A[3 * i + 1];
    }
    for (int e = 0; e < 4 && np > 0; ++e) {
      const double ex = Bx[2 * e], ey = Bx[2 * e + 1];
      const double fx = Bx[2 * ((e + 1) & 3)], fy = Bx[2 * ((e + 1) & 3) + 1];
      int nq = 0;
      for (int i = 0; i < np; ++i) {
        const double* s = P + 2 * i;
        const double* t = P + 2 * ((i + 1 == np) ? 0 : i + 1);
        const double ds = sb * ((fx - ex) * (s[1] - ey) - (fy - ey) * (s[0] - ex));
        const double dt = sb * ((fx - ex) * (t[1] - ey) - (fy - ey) * (t[0] - ex));
        if (ds >= 0.0 && nq < 8) {
          Q[2 * nq] = s[0];
          Q[2 * nq + 1] = s[1];
          ++nq;
        }
        if ((ds >= 0.0) != (dt >= 0.0) && nq < 8) {
          const double w = ds / (ds - dt);
          Q[2 * nq] = s[0] + w * (t[0] - s[0]);
          Q[2 * nq + 1] = s[1] + w * (t[1] - s[1]);
          ++nq;
        }
      }
      np = nq;
      for (int i = 0; i < 2 * np; ++i) P[i] = Q[i];
    }
    area[id] = np >= 3 ? fabs(poly_area2(P, np)) : 0.0;
  }
}

int grid_of(int items, int per) {
  const int g = (items + per - 1) / per, cap = num_sms() * 8;
  return g < 1 ? 1 : (g > cap ? cap : g);
}

}  // namespace

void launch_footprints(int n, const double* intr, double width, double height, const double* R, const double* T,
                       const DsmView& D, long long* range, double* corners, cudaStream_t st) {
  LAUNCH(KK_OTHER, st, k_range_init<<<1, 1, 0, st>>>(range));
  const size_t nh = (size_t)D.nx * D.ny;
  LAUNCH(KK_OTHER, st, k_range<<<grid_of((int)(nh < (size_t)1 << 30 ? nh : (size_t)1 << 30), 1024), 256, 0, st>>>(D.h, nh, range));
  LAUNCH(KK_OTHER, st, k_footprint<<<grid_of(n, 1), 128, 0, st>>>(n, intr, width, height, R, T, D, range, corners));
}

void launch_overlaps(int na, const double* qa, int nb, const double* qb, double* area, cudaStream_t st) {
  LAUNCH(KK_OTHER, st, k_overlap<<<grid_of(na * nb, 128), 128, 0, st>>>(na, qa, nb, qb, area));
}

}  // namespace bagpu
