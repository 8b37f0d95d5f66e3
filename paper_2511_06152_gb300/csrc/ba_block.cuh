// Blocks of 8 x 8 numbers of 64 bits (double-float pairs or binary64) in shared
// memory, and the warp-level steps of a blocked L D L^T on them; shared by the
// reduced-system solvers.
#pragma once
#include "ba_device.cuh"
#include "ba_dfloat.cuh"

namespace bagpu {

constexpr int kBlkBytes = 512;   // 8 x 8 numbers of 8 bytes

// ---- the two arithmetics

struct ArithDf {
  static constexpr bool kProductFirst = true;
  using T = dfl;
  using S = float;
  static __device__ __forceinline__ T zero() { return dfl{0.f, 0.f}; }
  static __device__ __forceinline__ T one() { return dfl{1.f, 0.f}; }
  static __device__ __forceinline__ T mul(T a, T b) { return df_mul(a, b); }
  static __device__ __forceinline__ T fms(T a, T x, T y) { return df_fms(a, x, y); }
  static __device__ __forceinline__ bool positive(T d) { return d.hi > 0.0f; }
  // 1 / (d s), s a power of two that keeps the reciprocal finite
  static __device__ __forceinline__ T recip(T d, S& s) {
    s = d.hi < 0x1p-100f ? 0x1p100f : 1.0f;
    return df_recip_fast(dfl{d.hi * s, d.lo * s});
  }
  static __device__ __forceinline__ T scale(T v, S s) { return dfl{v.hi * s, v.lo * s}; }
  static __device__ __forceinline__ T shfl(T v, int src) {
    return dfl{__shfl_sync(BA_FULL_MASK, v.hi, src), __shfl_sync(BA_FULL_MASK, v.lo, src)};
  }
  static __device__ __forceinline__ T from_double(double v, int e) { return df_from_d_pow2(v, e); }
  static __device__ __forceinline__ double to_double(T v, int e) { return ldexp(df_to_d(v), e); }
  static __device__ __forceinline__ int scale_exp(double d) {
    return (d > 0.0 && d < INFINITY) ? -(ilogb(d) / 2) : 0;
  }
  struct Acc {
    Dot2 a;
    __device__ __forceinline__ void add(T x, T y) { a.add(x, y); }
    __device__ __forceinline__ T from(T v) const { return df_sub(v, a.get()); }
    __device__ __forceinline__ void merge_xor(int off) {
      a.merge(__shfl_xor_sync(BA_FULL_MASK, a.s, off), __shfl_xor_sync(BA_FULL_MASK, a.c, off));
    }
    __device__ __forceinline__ T get() const { return a.get(); }
  };
};

struct ArithD {
  static constexpr bool kProductFirst = false;  // (a binary64 product takes as long)
  using T = double;
  using S = double;
  static __device__ __forceinline__ T zero() { return 0.0; }
  static __device__ __forceinline__ T one() { return 1.0; }
  static __device__ __forceinline__ T mul(T a, T b) { return a * b; }
  static __device__ __forceinline__ T fms(T a, T x, T y) { return fma(-x, y, a); }
  // (comparisons on the bits: a binary64 instruction, comparisons included,
  // occupies a quarter of the SM for 64 cycles)
  static __device__ __forceinline__ bool positive(T d) {
    const long long b = __double_as_longlong(d);
    return b > 0 && b <= 0x7ff0000000000000ll;
  }
  static __device__ __forceinline__ T recip(T d, S& s) {
    s = 1.0;
    if (__double_as_longlong(d) < 0x03f0000000000000ll) {  // below 2^-960
      s = 0x1p960;
      d *= s;
    }
    return 1.0 / d;
  }
  static __device__ __forceinline__ T scale(T v, S s) {
    return __double_as_longlong(s) == 0x3ff0000000000000ll ? v : v * s;
  }
  static __device__ __forceinline__ T shfl(T v, int src) { return __shfl_sync(BA_FULL_MASK, v, src); }
  static __device__ __forceinline__ T from_double(double v, int) { return v; }
  static __device__ __forceinline__ double to_double(T v, int) { return v; }
  static __device__ __forceinline__ int scale_exp(double) { return 0; }
  struct Acc {
    double a = 0.0;
    __device__ __forceinline__ void add(T x, T y) { a += x * y; }
    __device__ __forceinline__ T from(T v) const { return v - a; }
    __device__ __forceinline__ void merge_xor(int off) { a += __shfl_xor_sync(BA_FULL_MASK, a, off); }
    __device__ __forceinline__ T get() const { return a; }
  };
};

// ---- 8 x 8 blocks in shared memory
//
// Row r takes 64 bytes, four groups of two numbers; group g sits at position
// (g + r / 2) mod 4, so that eight lanes reading the same group of eight rows
// touch all 32 banks once.
__device__ __forceinline__ int grp_off(int r, int g) { return r * 64 + (((g + (r >> 1)) & 3) << 4); }
__device__ __forceinline__ int elt_off(int r, int c) { return grp_off(r, c >> 1) + ((c & 1) << 3); }

template <class T>
struct alignas(16) Pair2 {
  T a, b;
};

template <class T>
__device__ __forceinline__ Pair2<T> ld_grp(const char* blk, int r, int g) {
  return *reinterpret_cast<const Pair2<T>*>(blk + grp_off(r, g));
}
template <class T>
__device__ __forceinline__ void st_grp(char* blk, int r, int g, T a, T b) {
  *reinterpret_cast<Pair2<T>*>(blk + grp_off(r, g)) = Pair2<T>{a, b};
}
template <class T>
__device__ __forceinline__ void ld_row(const char* blk, int r, T (&v)[8]) {
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const Pair2<T> p = ld_grp<T>(blk, r, g);
    v[2 * g] = p.a;
    v[2 * g + 1] = p.b;
  }
}
template <class T>
__device__ __forceinline__ void st_row(char* blk, int r, const T (&v)[8]) {
#pragma unroll
  for (int g = 0; g < 4; ++g) st_grp<T>(blk, r, g, v[2 * g], v[2 * g + 1]);
}

// A block less l y^T, by one warp: row lane mod 8, columns 2 g and 2 g + 1
// (g = lane / 8) per lane.
template <class A>
__device__ __forceinline__ void product_warp(char* blk, const char* lblk, const char* yblk, int lane) {
  using T = typename A::T;
  const int r = lane & 7, g = lane >> 3;
  typename A::Acc c0, c1;
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const Pair2<T> l = ld_grp<T>(lblk, r, h);
    const Pair2<T> y0 = ld_grp<T>(yblk, 2 * g, h), y1 = ld_grp<T>(yblk, 2 * g + 1, h);
    c0.add(l.a, y0.a);
    c1.add(l.a, y1.a);
    c0.add(l.b, y0.b);
    c1.add(l.b, y1.b);
  }
  const Pair2<T> v = ld_grp<T>(blk, r, g);
  st_grp<T>(blk, r, g, c0.from(v.a), c1.from(v.b));
}

// One warp, a row per lane: lanes 0 .. 7 the diagonal block, the others rows
// below it, a -> y (in place) and l = y / d, in one sweep over the eight
// pivots; the diagonal block's l is the unit lower factor (left of the
// diagonal).  (r, s): 1 / (d s) and s of pivot lane mod 8.  Returns false when
// a pivot is not positive.
template <class A>
__device__ __forceinline__ bool sweep_warp(typename A::T (&a)[8], typename A::T (&l)[8], typename A::T& r,
                                           typename A::S& s, int lane) {
  using T = typename A::T;
  bool ok = true;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const T d = A::shfl(a[j], j);
    ok = ok && A::positive(d);  // (past a pivot that is not, the numbers no longer matter)
    typename A::S sj;
    const T rj = A::recip(d, sj);
    l[j] = A::scale(A::mul(a[j], rj), sj);
    if constexpr (A::kProductFirst) {
      // the column of the next pivot as a - (a_j y) / d: the product runs
      // beside the reciprocal that everything waits for
      if (j < 7) a[j + 1] = A::fms(a[j + 1], A::scale(A::mul(a[j], A::shfl(a[j], j + 1)), sj), rj);
    }
#pragma unroll
    for (int k = j + (A::kProductFirst ? 2 : 1); k < 8; ++k) a[k] = A::fms(a[k], l[j], A::shfl(a[j], k));
    if ((lane & 7) == j) {
      r = rj;
      s = sj;
    }
  }
  return ok;
}

}  // namespace bagpu
