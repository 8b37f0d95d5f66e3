// The reduced camera system of a cluster of up to kMaxFreeSmall free images:
// assembly, factorisation, solve, refinement, candidate poses.
//
// One thread-block cluster of kFC CTAs per BA cluster.  The matrix (n <= 192)
// is cut into 8 x 8 blocks of 64-bit numbers (binary64, or double-float
// pairs); row block b lives in the shared memory of CTA b mod kFC, the
// diagonal blocks in every CTA.  Factorisation S = L D L^T, L unit lower, one
// block column p at a time:
//   column      blocks (i, p), i >= p, less block column p - 1 (a warp per
//               block); then one to three warps factor (p, p) and solve
//               y = A(i, p) L(p, p)^-T for three row blocks each in the same
//               sweep over the eight pivots, a row per lane (the same factor
//               in every warp of every CTA, so that nothing waits for it to be
//               passed on), keep l = y / d in place of A(i, p) and write y to
//               every CTA's shared memory;
//   trailing    all warps subtract block column p - 1 from the CTA's blocks
//               right of column p, eight lanes per block, a lane per row;
//   one cluster barrier.
// The right-hand side is one more row: its y and l are L^-1 b and
// D^-1 L^-1 b, so only the backward substitution is left after the factor.
//
// What bounds it: n sequential pivots, each a reciprocal, an update and a
// shuffle deep (a sweep over eight of them takes 1.2 k cycles alone, two to
// three times that beside the other warps' products), and per block column one
// cluster barrier; then the trailing products, 12 binary32 instructions per
// double-float product, which one SM would take longer for than the pivots
// take, hence the four SMs.  In binary64 every instruction occupies its
// quarter of an SM for 64 cycles per warp; there the sweep's 92 instructions
// and the products bound it alike.  Per iteration on GB300, against the
// predecessor (one CTA, packed rows, column-by-column panels): one cluster of
// 24 images (n = 144) 228 -> 91 us, in binary64 366 -> 186; 6 images in
// binary64 87 -> 58; 12 clusters 293 -> 119; 128 clusters 321 -> 173.  Of the
// 186 k cycles at n = 144 the factor is 122 k, the backward substitution 27 k,
// the assembly 24 k, the candidates 8 k.
//
// Nothing is computed left of a row's envelope (the elimination order makes
// the row blocks a block column reaches one run).  Double-float: the system is
// scaled by powers of two first, A' = E A E with A'(i, i) in [1/2, 4), which is
// exact and keeps every entry inside the binary32 exponent range whatever the
// scale of S.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "ba_block.cuh"
#include "ba_camera.cuh"
#include "ba_device.cuh"
#include "ba_dfloat.cuh"
#include "ba_internal.h"

namespace cg = cooperative_groups;

namespace bagpu {

namespace {

constexpr int kFC = 4;           // CTAs of a thread-block cluster
constexpr int kFactorMaxThreads = 512;

// blocks left of the diagonal in the row blocks rank, rank + kFC, ... before
// the k-th of them
__host__ __device__ __forceinline__ int own_before(int rank, int k) { return k * rank + kFC * k * (k - 1) / 2; }

// Shared memory of one CTA.
struct Smem {
  char* own;       // the CTA's row blocks, left of the diagonal; the right-hand side is row block nb
  char* y;         // two block columns of y, nb blocks each; first the images' sums and priors
  char* diag;      // diagonal blocks of A
  char* unit;      // unit lower blocks of the factor
  char* inv;       // CTA 0: their inverses, for the backward substitution
  char* lnext;     // two blocks: l of row block p + 1 in block column p
  char* rinv;      // [n8] 1 / (d s)
  char* rsc;       // [n8] s
  double* x;       // [n8] solution
  double* t;       // [n8] right-hand sides in binary64
  double* D;       // [n8] damping scale
  double* g;       // [n8] gradient
  char* v;         // [n8] working vector of the substitutions
  int* escale;     // [n8]
  int* blkfirst;   // [nb] first block column of each row block's envelope
  int* rend;       // [nb] past the last row block that block column p reaches
};

__host__ __device__ __forceinline__ size_t small_smem(int n, Smem* s, char* base) {
  const int nb = (n + 7) / 8, n8 = 8 * nb;
  int own = 0;
  for (int r = 0; r < kFC; ++r)
    if (r <= nb) {
      const int k = (nb - r) / kFC + 1, c = own_before(r, k);
      own = c > own ? c : own;
    }
  size_t o = 0;
  auto take = [&](size_t bytes) {
    char* p = base + o;
    o += (bytes + 15) & ~(size_t)15;
    return p;
  };
  Smem t;
  t.own = take((size_t)own * kBlkBytes);
  t.y = take((size_t)2 * nb * kBlkBytes);
  t.diag = take((size_t)nb * kBlkBytes);
  t.unit = take((size_t)nb * kBlkBytes);
  t.inv = t.y;  // y is read no more
  t.lnext = take((size_t)2 * kBlkBytes);
  t.rinv = take((size_t)n8 * 8);
  t.rsc = take((size_t)n8 * 8);
  t.x = (double*)take((size_t)n8 * 8);
  t.t = (double*)take((size_t)n8 * 8);
  t.D = (double*)take((size_t)n8 * 8);
  t.g = (double*)take((size_t)n8 * 8);
  t.v = take((size_t)n8 * 8);
  t.escale = (int*)take((size_t)n8 * 4);
  t.blkfirst = (int*)take((size_t)nb * 4);
  t.rend = (int*)take((size_t)nb * 4);
  if (s) *s = t;
  return o;
}
// An image's prior for the assembly: JtJ of the attitude (3 x 3, row-major)
// 0 .. 8, of the position (its equal diagonal entries) 9, Jtr 10 .. 15.
constexpr int kPr = 16;
// the images' sums (40 doubles) and priors fit the space of y (n = 6 nf)
static_assert(8 * (40 + kPr) <= 6 * 2 * kBlkBytes / 8, "assembly scratch");

// ---- factorisation

// the same place in CTA c's shared memory
template <class P>
__device__ __forceinline__ P* peer(P* p, int c) {
  return cg::this_cluster().map_shared_rank(p, c);
}

// One row (lane) of block A(i, j) less l_i y_j^T, stored (store), in every CTA
// (everywhere).
template <class A>
__device__ __forceinline__ void block_update(char* ablk, const char* lblk, const char* yblk, int r, bool store,
                                             bool everywhere) {
  using T = typename A::T;
  typename A::Acc acc[8];
#pragma unroll 1
  for (int h = 0; h < 4; ++h) {
    const Pair2<T> l = ld_grp<T>(lblk, r, h);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const Pair2<T> y = ld_grp<T>(yblk, c, h);
      acc[c].add(l.a, y.a);
      acc[c].add(l.b, y.b);
    }
  }
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const Pair2<T> v = ld_grp<T>(ablk, r, g);
    const T a = acc[2 * g].from(v.a), b = acc[2 * g + 1].from(v.b);
    if (store) st_grp<T>(ablk, r, g, a, b);
    if (everywhere) {
#pragma unroll 1
      for (int c = 0; c < kFC; ++c) st_grp<T>(peer(ablk, c), r, g, a, b);
    }
  }
}

template <class A>
struct Factor {
  using T = typename A::T;
  Smem S;
  int nb, rank, warp, lane, nw;

  // block (rb, cb) left of the diagonal, in its owner's shared memory
  __device__ const char* any_blk(int rb, int cb) const {
    const int c = rb & (kFC - 1);
    return peer(S.own, c) + (size_t)(own_before(c, rb / kFC) + cb) * kBlkBytes;
  }
  __device__ char* own_blk(int rb, int cb) const {
    return S.own + (size_t)(own_before(rank, rb / kFC) + cb) * kBlkBytes;
  }
  __device__ char* y_blk(int p, int b) const { return S.y + (size_t)((p & 1) * nb + b) * kBlkBytes; }
  __device__ char* diag_blk(int b) const { return S.diag + (size_t)b * kBlkBytes; }
  __device__ T* rinv() const { return reinterpret_cast<T*>(S.rinv); }
  __device__ typename A::S* rsc() const { return reinterpret_cast<typename A::S*>(S.rsc); }

  // the first of this CTA's row blocks at or after b
  __device__ int own_from(int b) const { return b + ((rank - b) & (kFC - 1)); }

  // Subtract block column p from the CTA's blocks (i, j), p + 1 < j <= i; the
  // warps take four blocks at a time from a shared counter.  A diagonal block
  // is its row block's CTA's to update, until the last but one update, which
  // goes to every CTA (update_column does the last).
  __device__ void trailing(int p, int* next) const {
    const int e = S.rend[p], r = lane & 7, c0 = p + 2;
    int total = 0;
    for (int b = own_from(c0); b < e; b += kFC) total += b - c0 + 1;
    if ((nb & (kFC - 1)) == rank) total += max(0, e - c0);  // the right-hand side
    for (;;) {
      int i0 = lane == 0 ? atomicAdd(next, 4) : 0;
      i0 = __shfl_sync(BA_FULL_MASK, i0, 0);
      if (i0 >= total) return;
      const int item = i0 + (lane >> 3);
      const bool live = item < total;
      int k = live ? item : total - 1, ib = own_from(c0);
      while (ib < e && k > ib - c0) {
        k -= ib - c0 + 1;
        ib += kFC;
      }
      if (ib >= e) ib = nb;
      const int jb = c0 + k;
      const bool diag = ib == jb;
      block_update<A>(diag ? diag_blk(ib) : own_blk(ib, jb), own_blk(ib, p), y_blk(p, jb), r, live,
                      live && diag && ib == c0);
    }
  }

  // the CTA's row blocks below block (p, p) that block column p reaches, the
  // right-hand side last: how many, and the t-th
  __device__ int rows_of(int p) const {
    const int f = own_from(p + 1), e = S.rend[p];
    return (f < e ? (e - 1 - f) / kFC + 1 : 0) + ((nb & (kFC - 1)) == rank ? 1 : 0);
  }
  __device__ int row_blk(int p, int t, int rows) const {
    return (nb & (kFC - 1)) == rank && t == rows - 1 ? nb : own_from(p + 1) + kFC * t;
  }

  // block column p less block column p - 1, a warp per block
  __device__ void update_column(int p, int rows) const {
    if (p == 0 || p >= S.rend[p - 1]) return;
    const char* yb = y_blk(p - 1, p);
    for (int t = warp; t <= rows; t += nw) {
      const int b = t > 0 ? row_blk(p, t - 1, rows) : p;
      product_warp<A>(t > 0 ? own_blk(b, p) : diag_blk(p),
                      t > 0 ? own_blk(b, p - 1) : S.lnext + ((p - 1) & 1) * kBlkBytes, yb, lane);
    }
  }

  // Block column p factored and solved, by the first warps, three row blocks
  // each (each warp factors the diagonal block for itself): l in place, y to
  // every CTA, and of row block p + 1 l too.  False when a pivot is not positive.
  __device__ bool solve_column(int p, int rows) const {
    if (warp > 0 && 3 * warp >= rows) return true;
    const int q = lane >> 3, t = 3 * warp + q - 1, row = lane & 7;
    const bool has = q > 0 && t < rows;
    const int b = has ? row_blk(p, t, rows) : p;
    char* blk = has ? own_blk(b, p) : diag_blk(p);
    T a[8], l[8], r = A::one();
    typename A::S s = 1;
    ld_row<T>(blk, row, a);
    const bool ok = sweep_warp<A>(a, l, r, s, lane);
    if (has) {
      st_row<T>(blk, row, l);
      if (b < nb) {
        const size_t at = (size_t)((p & 1) * nb + b) * kBlkBytes;
#pragma unroll
        for (int c = 0; c < kFC; ++c) {
          st_row<T>(peer(S.y, c) + at, row, a);
          if (b == p + 1) st_row<T>(peer(S.lnext, c) + (p & 1) * kBlkBytes, row, l);
        }
      }
    } else if (warp == 0 && q == 0) {
      // (the other warps may still be reading the diagonal block itself)
      st_row<T>(S.unit + (size_t)p * kBlkBytes, row, l);
      rinv()[8 * p + row] = r;
      rsc()[8 * p + row] = s;
    }
    return ok;
  }
};

// Inverse of a unit lower block, by one warp, to dst.
template <class A>
__device__ __forceinline__ void invert_block_warp(const char* u, char* dst, int lane) {
  using T = typename A::T;
  const int r = lane & 7, g = lane >> 3;
  T x0 = r == 2 * g ? A::one() : A::zero(), x1 = r == 2 * g + 1 ? A::one() : A::zero();
#pragma unroll 1
  for (int j = 0; j < 7; ++j) {  // rows after j less L(r, j) times row j
    const T c = *reinterpret_cast<const T*>(u + elt_off(r, j));
    const T y0 = A::shfl(x0, (g << 3) | j), y1 = A::shfl(x1, (g << 3) | j);
    if (r > j) {
      x0 = A::fms(x0, c, y0);
      x1 = A::fms(x1, c, y1);
    }
  }
  st_grp<T>(dst, r, g, x0, x1);
}

// v(8 b .. 8 b + 7) times the inverse X of the diagonal block (forward), or
// its transpose (backward), by one warp: two products per lane
template <class A, bool FWD>
__device__ __forceinline__ void solve_block_warp(const char* X, typename A::T* v, int lane) {
  using T = typename A::T;
  const int r = lane & 7, q = 2 * (lane >> 3);
  typename A::Acc a;
  a.add(*reinterpret_cast<const T*>(X + (FWD ? elt_off(r, q) : elt_off(q, r))), v[q]);
  a.add(*reinterpret_cast<const T*>(X + (FWD ? elt_off(r, q + 1) : elt_off(q + 1, r))), v[q + 1]);
  a.merge_xor(8);
  a.merge_xor(16);
  __syncwarp();
  if (lane < 8) v[r] = a.get();
}

// L^T x = v in place (rank 0, v its working vector): per row block, its 8 unknowns by one warp, then the products
// with its rows (a thread per column; loaded one block ahead).
template <class A>
__device__ void backward(const Factor<A>& F, int tid) {
  using T = typename A::T;
  T* v = reinterpret_cast<T*>(F.S.v);
  // thread tid: column tid of the row block being loaded (n8 <= 192 <= bs)
  T l[8];
  auto fetch = [&](int b) {
    const int cb = tid >> 3;
    if (tid < 8 * b && cb >= F.S.blkfirst[b]) {
      const char* blk = F.any_blk(b, cb);
#pragma unroll
      for (int r = 0; r < 8; ++r) l[r] = *reinterpret_cast<const T*>(blk + elt_off(r, tid & 7));
    }
  };
  fetch(F.nb - 1);
  for (int b = F.nb - 1; b >= 0; --b) {
    if (F.warp == 0) solve_block_warp<A, false>(F.S.inv + (size_t)b * kBlkBytes, v + 8 * b, F.lane);
    __syncthreads();
    if (tid < 8 * b && (tid >> 3) >= F.S.blkfirst[b]) {
      typename A::Acc a0, a1;
#pragma unroll
      for (int r = 0; r < 8; r += 2) {
        a0.add(l[r], v[8 * b + r]);
        a1.add(l[r + 1], v[8 * b + r + 1]);
      }
      v[tid] = a1.from(a0.from(v[tid]));
    }
    if (b > 0) fetch(b - 1);
    __syncthreads();
  }
}

// L z = v, then v = D^-1 z (rank 0), for the refinement's right-hand sides
template <class A>
__device__ void forward(const Factor<A>& F, int tid, int bs) {
  using T = typename A::T;
  T* v = reinterpret_cast<T*>(F.S.v);
  for (int b = 0; b < F.nb; ++b) {
    if (F.warp == 0) solve_block_warp<A, true>(F.S.inv + (size_t)b * kBlkBytes, v + 8 * b, F.lane);
    __syncthreads();
    const int i = tid, ib = i >> 3;  // row i
    if (ib > b && ib < F.S.rend[b]) {
      T l[8];
      ld_row<T>(F.any_blk(ib, b), i & 7, l);
      typename A::Acc a0, a1;
#pragma unroll
      for (int q = 0; q < 8; q += 2) {
        a0.add(l[q], v[8 * b + q]);
        a1.add(l[q + 1], v[8 * b + q + 1]);
      }
      v[i] = a1.from(a0.from(v[i]));
    }
    __syncthreads();
  }
  for (int i = tid; i < 8 * F.nb; i += bs) v[i] = A::scale(A::mul(v[i], F.rinv()[i]), F.rsc()[i]);
  __syncthreads();
}

// ---- priors and candidate poses, four lanes per image
//
// A binary64 instruction occupies its quarter of the SM for 64 cycles per
// warp, however many lanes take part: what counts is the length of a lane's
// program.  An image's work is dealt to four neighbouring lanes (q = 0 .. 2: an
// axis each; lane 3 repeats axis 2 and writes nothing), the images to as many
// warps as that takes.  With a lane per image, the priors took 22 k cycles and
// the candidates 21 k.

// Prior of image k at its pose (Rc, Tc: the current cameras) to o [kPr]: with
// phi the rotation vector, J = Jr^-1(phi), J^T phi = phi and
// J^T J = (1 - b |phi|^2) I + b phi phi^T, b = 2 c2 - 1/4 - c2^2 |phi|^2 (c2 of
// so3_jr_inv; K^3 = -|phi|^2 K for K = [phi]x).
__device__ __noinline__ void prior_quad(const DevCluster& C, int k, const double* Rc, const double* Tc, int lane4,
                                        double* o) {
  const unsigned mask = 0xfu << ((threadIdx.x & 31) & ~3);  // the image's four lanes
  const int q = lane4 < 3 ? lane4 : 2;
  const double ii = C.inv_imu2, ig = C.inv_gnss2;
  double row[3] = {0.0, 0.0, 0.0}, jr = 0.0;
  if (ii > 0.0) {
    double w[3];
    quad_log(mask, C.R_prior + 9 * k, Rc + 9 * k, q, w);
    const double t2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
    const double c2 = jr_inv_c2(t2);
    const double b = 2.0 * c2 - 0.25 - c2 * c2 * t2;
    const double wq = q == 0 ? w[0] : (q == 1 ? w[1] : w[2]);
    const double bw = ii * b * wq, d = ii * (1.0 - b * t2);
    for (int j = 0; j < 3; ++j) row[j] = bw * w[j] + (j == q ? d : 0.0);
    jr = ii * wq;
  }
  const double e = ig > 0.0 ? ig * (Tc[3 * k + q] - C.T_prior[3 * k + q]) : 0.0;
  if (lane4 == 3) return;
  for (int j = 0; j < 3; ++j) o[3 * q + j] = row[j];
  o[10 + q] = jr;
  o[13 + q] = e;
  if (q == 0) o[9] = ig;
}

// Candidate pose of image k (candidate_pose), a row of R and an entry of T per
// lane, stored (store), or its prior cost at the candidate (*cost, all lanes).
template <bool MIXED>
__device__ __noinline__ void candidate_quad(const DevCluster& C, int k, const double* x, int cur, bool fail, int lane4,
                                            bool store, double* cost) {
  const unsigned mask = 0xfu << ((threadIdx.x & 31) & ~3);  // the image's four lanes
  const int q = lane4 < 3 ? lane4 : 2, nc = C.n_cams;
  const double* Rc = C.R + (size_t)cur * nc * 9 + 9 * k;
  double row[3], t = C.T[(size_t)cur * nc * 3 + 3 * k + q];
  const int f = C.free_idx[k];
  const bool moves = f >= 0 && !fail;
  if (moves) {
    const double* d = x + 6 * C.fpos[f];
    double E[9];
    so3_exp(d, E);
    for (int c = 0; c < 3; ++c) row[c] = Rc[3 * q] * E[c] + Rc[3 * q + 1] * E[3 + c] + Rc[3 * q + 2] * E[6 + c];
    t += d[3 + q];
  } else {
    for (int c = 0; c < 3; ++c) row[c] = Rc[3 * q + c];
  }
  if (store) {
    if (lane4 == 3) return;
    double* Rn = C.R + (size_t)(cur ^ 1) * nc * 9 + 9 * k + 3 * q;
    for (int c = 0; c < 3; ++c) Rn[c] = row[c];
    C.T[(size_t)(cur ^ 1) * nc * 3 + 3 * k + q] = t;
    if constexpr (MIXED) write_camdf_row(C, cur ^ 1, k, q, row, t);
    store_cam_step<MIXED>(C, k, q, moves ? x + 6 * C.fpos[f] : nullptr, Rc);
    return;
  }
  double v = 0.0;
  if (moves) {
    double R[9], T[3];
    for (int i = 0; i < 9; ++i) R[i] = quad_get(mask, row[i % 3], i / 3);
    for (int i = 0; i < 3; ++i) T[i] = quad_get(mask, t, i);
    v = prior_cost_quad(mask, C, k, R, T, q);
  }
  *cost = v;
}

template <class A, bool MIXED>
__global__ void __cluster_dims__(kFC, 1, 1) __launch_bounds__(kFactorMaxThreads)
    k_factor_solve(BatchView bv, int refine_steps, int assemble_only) {
  using T = typename A::T;
  extern __shared__ __align__(16) char smem[];
  __shared__ int fail, next[2];
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x, bs = blockDim.x;
  const int rank = (int)cl.block_rank();
  Factor<A> F;
  F.rank = rank;
  F.warp = tid >> 5;
  F.lane = tid & 31;
  F.nw = bs >> 5;
  for (int so = blockIdx.x / kFC; so < bv.n; so += gridDim.x / kFC) {
    const int s = bv.factor_order[so];  // largest systems first
    const DevCluster& C = bv.cl[s];
    LmState* lm = C.lm;
    if (!lm->active && !assemble_only) continue;
    if (C.n_free > kMaxFreeSmall) continue;  // the global-memory solver takes larger systems
    const int nf = C.n_free, n = 6 * nf, nc = C.n_cams, nb = (n + 7) / 8, n8 = 8 * nb;
    const double mu = lm->mu;
    const int cur = lm->cur;
    small_smem(n, &F.S, smem);
    const Smem& S = F.S;
    F.nb = nb;
    double* cd = reinterpret_cast<double*>(S.y);  // [nf][40] sums
    double* pr = cd + (size_t)nf * 40;            // [nf][kPr] priors
    const bool keep_s = refine_steps > 0;  // S in binary64 in global memory, for the refinement

    // ---- assembly (the images in elimination order: position p = fpos[f])
    if (tid == 0) {
      fail = lm->pt_fail;
      next[0] = next[1] = 0;
    }
    for (int idx = tid; idx < 4 * nf; idx += bs) {  // four lanes per image
      const int f = idx >> 2;
      prior_quad(C, C.cam_of_free[f], C.R + (size_t)cur * nc * 9, C.T + (size_t)cur * nc * 3, idx & 3,
                 pr + kPr * C.fpos[f]);
    }
    for (int b = tid; b < nb; b += bs) S.blkfirst[b] = 6 * C.env_first[(8 * b) / 6] / 8;
    for (int idx = tid; idx < nf * 39; idx += bs) {
      const int f = idx / 39, e = idx - 39 * f;
      cd[40 * C.fpos[f] + e] = C.camsum[(size_t)kCamPart * f + e];
    }
    if (rank == 0 && tid == 0) lm->tiles_done = 0;  // the back-substitution counts its tiles from here
    __syncthreads();
    // damping, gradient, right-hand side; the scale of each row
    for (int i = tid; i < n8; i += bs) {
      if (i >= n) {  // padding rows of the identity
        S.escale[i] = 0;
        S.t[i] = 0.0;
        S.x[i] = 1.0;
        continue;
      }
      const int p = i / 6, a = i - 6 * p;
      const int ui = a * 6 - a * (a - 1) / 2;  // packed upper index of (a, a)
      const double pd = pr[kPr * p + (a < 3 ? 4 * a : 9)];
      const double D = clamp_diag(cd[40 * p + 33 + a] + pd);
      const double g = cd[40 * p + 21 + a] - pr[kPr * p + 10 + a];
      const double r = g - cd[40 * p + 27 + a];
      const double d = cd[40 * p + ui] + pd + mu * D;
      S.escale[i] = A::scale_exp(d);
      S.t[i] = r;
      S.x[i] = d;
      S.D[i] = D;
      S.g[i] = g;
    }
    // the row blocks each block column reaches: [p + 1, rend)
    for (int p = tid; p < nb; p += bs) {
      int e = p + 1;
      while (e < nb && S.blkfirst[e] <= p) ++e;
      S.rend[p] = e;
    }
    __syncthreads();
    if (rank == 0)
      for (int idx = tid; idx < n; idx += bs) {  // in the order of the free images
        const int pi = 6 * C.fpos[idx / 6] + idx % 6;
        C.gc[idx] = S.g[pi];
        C.rhs[pi] = S.t[pi];
      }
    if (assemble_only) {
      __syncthreads();
      continue;
    }
    // The 8 x 8 blocks, a warp each: the diagonal ones, then the CTA's own.
    // The images' pair blocks, -(sum Z_a Z_b^T), lie in the lower triangle of
    // S in global memory, where k_partial_reduce left them (zero between);
    // an image's own block is U + prior + mu D - sum Z Z^T.
    {
      const int r = F.lane & 7, g = F.lane >> 3;
      int total = nb;
      for (int b = F.own_from(0); b < nb; b += kFC) total += b;
      // three blocks of a warp at a time: their loads go out together
      for (int w0 = F.warp; w0 < total; w0 += 3 * F.nw) {
        double2 z[3];
        int ibs[3], jbs[3];
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const int w = w0 + u * F.nw;
          int k = w - nb, ib = w, jb = w;
          if (k >= 0) {
            for (ib = F.own_from(0); ib < nb && k >= ib; ib += kFC) k -= ib;
            jb = k;
          }
          ibs[u] = w < total ? ib : -1;
          jbs[u] = jb;
          const int i = 8 * ib + r, c = 8 * jb + 2 * g;
          z[u] = double2{0.0, 0.0};
          if (w < total && i < n && c <= i && c / 6 != i / 6)
            z[u] = *reinterpret_cast<const double2*>(C.S + (size_t)i * n + c);
        }
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const int ib = ibs[u], jb = jbs[u];
          if (ib < 0) continue;
          const int i = 8 * ib + r, c = 8 * jb + 2 * g, p = i / 6;
          if (i < n && c <= i && c / 6 == p) {
            const int b = i - 6 * p, a = c - 6 * p;  // a <= b; a even
            auto entry = [&](int a2) {
              if (a2 == b) return S.x[i];
              const double v = cd[40 * p + a2 * 6 - a2 * (a2 - 1) / 2 + b - a2];
              return b < 3 ? v + pr[kPr * p + 3 * a2 + b] : v;  // a2 < b; the position prior is diagonal
            };
            z[u].x = entry(a);
            if (a + 1 <= b) z[u].y = entry(a + 1);
            if (keep_s && (ib != jb || rank == 0)) {
              C.S[(size_t)i * n + c] = z[u].x;
              C.S[(size_t)c * n + i] = z[u].x;
              if (a + 1 <= b) {
                C.S[(size_t)i * n + c + 1] = z[u].y;
                C.S[(size_t)(c + 1) * n + i] = z[u].y;
              }
            }
          } else if (i >= n && ib == jb) {  // identity
            z[u].x = i == c ? 1.0 : 0.0;
            z[u].y = i == c + 1 ? 1.0 : 0.0;
          }
          const int ei = S.escale[i];
          st_grp<T>(ib == jb ? F.diag_blk(ib) : F.own_blk(ib, jb), r, g, A::from_double(z[u].x, ei + S.escale[c]),
                    A::from_double(z[u].y, ei + S.escale[c + 1]));
        }
      }
      if ((nb & (kFC - 1)) == rank)  // the right-hand side: row 0 of row block nb
        for (int j = F.warp; j < nb; j += F.nw) {
          const int c = 8 * j + 2 * g;
          st_grp<T>(F.own_blk(nb, j), r, g, r ? A::zero() : A::from_double(S.t[c], S.escale[c]),
                    r ? A::zero() : A::from_double(S.t[c + 1], S.escale[c + 1]));
        }
    }
    cl.sync();  // cd and pr are read no more: y may be written

    // ---- factorisation (fail is the same in every CTA: read from the LM state, then from the same pivots)
    if (!fail) {
      for (int p = 0; p < nb; ++p) {
        const int rows = F.rows_of(p);
        F.update_column(p, rows);
        __syncthreads();
        if (!F.solve_column(p, rows) && F.warp == 0 && F.lane == 0) fail = 1;
        if (p > 0) F.trailing(p - 1, &next[p & 1]);
        if (tid == 0) next[(p & 1) ^ 1] = 0;
        cl.sync();
      }
    }
    const bool bad = fail != 0;
    // ---- solve and refinement (rank 0; the other CTAs' blocks are read where they are)
    if (!bad) {
      T* v = reinterpret_cast<T*>(S.v);
      for (int b = rank + kFC * F.warp; b < nb; b += kFC * F.nw)
        invert_block_warp<A>(S.unit + (size_t)b * kBlkBytes, peer(S.inv, 0) + (size_t)b * kBlkBytes, F.lane);
      cl.sync();
      if (rank == 0) {
        for (int j = tid; j < n8; j += bs)
          v[j] = *reinterpret_cast<const T*>(F.any_blk(nb, j >> 3) + elt_off(0, j & 7));
        __syncthreads();
        backward<A>(F, tid);
        for (int j = tid; j < n; j += bs) S.x[j] = A::to_double(v[j], S.escale[j]);
      }
      for (int it = 0; it < refine_steps; ++it) {
        // t = rhs - S x over the envelope, a warp per row, the rows dealt to the CTAs
        if (rank == 0) {
          __syncthreads();
          for (int c = 1; c < kFC; ++c)
            for (int j = tid; j < n; j += bs) peer(S.x, c)[j] = S.x[j];
        }
        cl.sync();
        double* t0 = peer(S.t, 0);
        for (int r = rank + kFC * F.warp; r < n; r += kFC * F.nw) {
          const int c0 = 8 * S.blkfirst[r >> 3], c1 = min(n, 8 * S.rend[r >> 3]);
          double acc = 0.0;
          for (int c = c0 + F.lane; c < c1; c += 32) acc += C.S[(size_t)r * n + c] * S.x[c];
          acc = warp_sum(acc);
          if (F.lane == 0) t0[r] = C.rhs[r] - acc;
        }
        cl.sync();
        if (rank == 0) {
          for (int j = tid; j < n8; j += bs) v[j] = j < n ? A::from_double(S.t[j], S.escale[j]) : A::zero();
          __syncthreads();
          forward<A>(F, tid, bs);
          backward<A>(F, tid);
          for (int j = tid; j < n; j += bs) S.x[j] += A::to_double(v[j], S.escale[j]);
        }
      }
    } else if (rank == 0) {
      for (int j = tid; j < n; j += bs) S.x[j] = 0.0;
    }
    // ---- candidate poses (CTA 0), their prior cost (CTA 1), the cameras'
    // part of pred (CTA 2): three short serial binary64 jobs side by side
    __syncthreads();
    if (rank == 0)
      for (int c = 1; c < 3; ++c)
        for (int j = tid; j < n; j += bs) peer(S.x, c)[j] = S.x[j];
    cl.sync();
    if (rank == 0) {
      for (int idx = tid; idx < 4 * nc; idx += bs) candidate_quad<MIXED>(C, idx >> 2, S.x, cur, bad, idx & 3, true, nullptr);
      if (tid == 0) {
        lm->status = lm->dev_error ? lm->dev_error : (bad ? BA_STATUS_NOT_PD : 0);
        lm->dev_error = 0;
      }
    } else if (rank == 1) {
      for (int idx = tid; idx < 4 * nf; idx += bs) {
        double cost = 0.0;
        candidate_quad<MIXED>(C, C.cam_of_free[idx >> 2], S.x, cur, bad, idx & 3, false, &cost);
        if ((idx & 3) == 0) S.t[idx >> 2] = cost;
      }
    } else if (rank == 2) {  // d^T (mu D d + g), six terms per image
      for (int j = tid; j < n; j += bs) S.t[j] = bad ? 0.0 : S.x[j] * (mu * S.D[j] * S.x[j] + S.g[j]);
    }
    if (rank == 1 || rank == 2) {
      __syncthreads();
      if (F.warp == 0) {
        const double v = strided_sum(S.t, rank == 1 ? nf : n, F.lane);
        if (F.lane == 0) {
          if (rank == 1) lm->prior_new = v;
          else lm->pred_cam = v;
        }
      }
    }
    cl.sync();  // no CTA goes on while rank 0 reads its blocks
    // a cluster without observations has no back-substitution tile to count:
    // its LM step is taken here
    if (rank == 0 && C.n_tiles == 0 && tid < 32) lm_update_warp<MIXED>(C, tid);
    __syncthreads();
  }
}

template <class A, bool MIXED>
cudaError_t set_attr(size_t smem) {
  return cudaFuncSetAttribute(k_factor_solve<A, MIXED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

}  // namespace

size_t factor_smem_bytes(int max_n) { return small_smem(max_n, nullptr, nullptr); }

void launch_factor(const BatchView& bv, bool mixed, int refine_steps, int assemble_only, cudaStream_t st) {
  const int grid = kFC * (bv.n < 16384 ? bv.n : 16384);
  const size_t smem = factor_smem_bytes(bv.max_n);
  // 256 threads a CTA by default: two CTAs fit an SM's registers, which a batch
  // needs (128 clusters: 173 us per iteration against 287 with 384); a single
  // cluster of 24 images takes 91 us against 88.  At least a thread per row.
  const int th = bv.factor_threads / 2 < 192 ? 192 : bv.factor_threads / 2;
  LAUNCH(KK_FACTOR, st, {
    if (mixed) k_factor_solve<ArithDf, true><<<grid, th, smem, st>>>(bv, refine_steps, assemble_only);
    else if (bv.factor_df) k_factor_solve<ArithDf, false><<<grid, th, smem, st>>>(bv, refine_steps, assemble_only);
    else k_factor_solve<ArithD, false><<<grid, th, smem, st>>>(bv, refine_steps, assemble_only);
  });
}

cudaError_t set_factor_attributes(int max_n) {
  const size_t smem = factor_smem_bytes(max_n);
  cudaError_t e = set_attr<ArithDf, true>(smem);
  if (e == cudaSuccess) e = set_attr<ArithDf, false>(smem);
  if (e == cudaSuccess) e = set_attr<ArithD, false>(smem);
  return e;
}

}  // namespace bagpu
