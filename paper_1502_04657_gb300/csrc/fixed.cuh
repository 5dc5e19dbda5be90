// 64-bit fixed-point arithmetic with a block exponent for the FP64 cubic-load kernels.
//
// On this part an FP64 operation issues at 2 lanes per clock and SM, a 64-bit integer addition
// at 42 and a 32 x 32 -> 64 multiply-add at about 27 (measured).  The cubic-load and density
// kernels sum products of at most three nodal values over a small neighbourhood, so a block
// (3D) or a warp (2D) that covers a tile of nodes takes one exponent e for it, |u| < 2^e over
// the tile, and computes in integers: a quantity of degree d in u is the integer
//     I = value 2^(B_d - d e),  B_d = K - 3 d,
// so every product is (I J) >> K, rounded, whatever the degrees, and a sum is an exact integer
// addition.  Only products round, and u when it is read.  2D takes K = 61: u keeps 2^-59 of the
// tile's maximum, squares 2^-56 and cubes 2^-53 of their maxima; 3D, whose sums of 24
// tetrahedra need the headroom, K = 59.  The results are converted to FP64 and scaled once.
//
// The error is relative to the tile's maximum, FP64's to each node's own terms.  So the tile has
// to have one sign (no cancellation; the ground state's iterates do): a tile whose values of
// the rarer sign exceed 2^-12 of the others, with nonzero values below 2^-32 of its largest,
// whose exponent lies outside +-kFxMaxExp (infinities and NaN included), or of zeros, is
// computed in FP64 by the same walk (a called
// function: inlined, its register pressure spilled the fixed-point path).  And a node whose
// results are short of bits, because its star lies far below the tile's largest value (next to a
// corner of the box, or on a steep slope), is evaluated again in FP64: a cubic load below 2^36 (2D)
// or 2^40 (3D) units, a density entry below 2^44 (the whole tile where these are half of its nodes,
// or half of its columns lie 2^-7 below its largest value).  The roundings add up to at most 20 (2D) or 400
// (3D) units of a cubic load and 20 or 150 of a density entry, so every load keeps 4e-10 and every
// density entry 1e-11 of itself in the worst case.  The right-hand side lambda M u - zeta N needs no
// more of N than M u has of u: it takes its nodes in FP64 where the mean of u around them lies 2^-21
// below the largest value, which keeps 2^-32 of |lambda| M |u| + zeta N |u| (for a lambda of the size
// of zeta u^2 or above), and no tile for its columns.  (With the load's rule a right-hand side
// on 64^3 cells took 59 us instead of 43: the box's edges and corners.)  Measured
// against 113-bit arithmetic on ground-state-like inputs, relative 2-norm of the cubic load,
// fixed point and FP64: 2D sine mode 6.6e-17 and 9.1e-17, 3D sine mode 1.56e-16 and 1.70e-16,
// 3D steep trap 1.64e-16 both.
#pragma once

#include <stdint.h>

#include "dfloat.cuh"

namespace fmg {

template <int K>
struct fx {
  static constexpr int B1 = K - 3;
  long long v;
  fx() = default;
  __device__ constexpr explicit fx(int i) : v(i) {}  // raw (zero)
  __device__ constexpr explicit fx(long long i) : v(i) {}
};

template <int K>
__device__ __forceinline__ fx<K> operator+(fx<K> x, fx<K> y) {
  return fx<K>(x.v + y.v);
}
// (x y) >> K to nearest: |x| < 2^(K - 1) (the callers put the smaller factor first), so x is
// shifted to give the high word.  Both factors are split at a signed low half, which makes
// every partial product a signed 32 x 32 one and bounds what the dropped low x low product
// contributes by a quarter of a unit: three multiply-adds instead of four.
template <int K>
__device__ __forceinline__ fx<K> operator*(fx<K> x, fx<K> y) {
  const long long a = x.v << (64 - K), b = y.v;
  const int al = (int)a, bl = (int)b;
  const int ah = (int)(a >> 32) + (int)((uint32_t)al >> 31);
  const int bh = (int)(b >> 32) + (int)((uint32_t)bl >> 31);
  const long long m = (long long)al * bh + ((long long)ah * bl + 0x80000000ll);
  return fx<K>((long long)ah * bh + (m >> 32));
}
template <int K>
__device__ __forceinline__ fx<K> fma(fx<K> x, fx<K> y, fx<K> z) {
  return x * y + z;
}
template <int K>
__device__ __forceinline__ fx<K> twice(fx<K> x) {
  return fx<K>(x.v << 1);
}
// 2 u^3 from u and u^2
__device__ __forceinline__ double twice_cube(double u, double u2) { return twice(u2 * u); }
__device__ __forceinline__ dfloat twice_cube(dfloat u, dfloat u2) { return twice(u2 * u); }
template <int K>
__device__ __forceinline__ fx<K> twice_cube(fx<K> u, fx<K> u2) {
  return twice(u) * u2;
}

// C x + y for a small integer C (one operation in FP64 and double-float)
template <int C>
__device__ __forceinline__ double madd(double x, double y) {
  return fma((double)C, x, y);
}
template <int C>
__device__ __forceinline__ dfloat madd(dfloat x, dfloat y) {
  return fma(dfloat(C), x, y);
}
template <int C, int K>
__device__ __forceinline__ fx<K> madd(fx<K> x, fx<K> y) {
  return fx<K>(C * x.v + y.v);
}

__device__ __forceinline__ double fx_pow2(int e) {  // 2^e, -1022 <= e <= 1023
  return __longlong_as_double((long long)(e + 1023) << 52);
}
// the factor of a result of degree d: s 2^(d e - B_d)
template <int K>
__device__ __forceinline__ double fx_scale(double s, int d, int e) {
  return s * fx_pow2(d * e - (K - 3 * d));
}
template <int K>
__device__ __forceinline__ double to_double(fx<K> x, double scale) {
  return __ll2double_rn(x.v) * scale;
}

// v as an integer in units of 2^(e - B), |v| <= 2^e, rounded, on the integer pipes (a conversion
// occupies the FP64 pipe like an FP64 operation); shift = e + 1084 - B
__device__ __forceinline__ long long fx_rounded(double v, int shift) {
  const int hi = __double2hiint(v);
  const unsigned long long m =
      ((unsigned long long)(((uint32_t)hi & 0xfffffu) | 0x100000u) << 32 |
       (uint32_t)__double2loint(v)) << 10;
  const int sh = min(shift - ((hi >> 20) & 0x7ff), 63);
  const long long t = (long long)(((m >> sh) + 1) >> 1), sg = hi >> 31;
  return (t ^ sg) - sg;
}

// |x| < 2^T (T > 32): too few bits for the result of a single node
template <int T, int K>
__device__ __forceinline__ bool fx_short(fx<K> x) {
  return (unsigned)((int)(x.v >> 32) + (1 << (T - 32))) < (2u << (T - 32));
}

// the same, truncated; shift = e + 1085 - B
__device__ __forceinline__ long long fx_truncated(double v, int shift) {
  const int hi = __double2hiint(v);
  const unsigned long long m =
      ((unsigned long long)(((uint32_t)hi & 0xfffffu) | 0x100000u) << 32 |
       (uint32_t)__double2loint(v)) << 10;
  const int sh = min(shift - ((hi >> 20) & 0x7ff), 63);
  const long long t = (long long)(m >> sh), sg = hi >> 31;
  return (t ^ sg) - sg;
}

// high word of a 64 x 64 product (|a|, |b| < 2^63 - 2^31), within a unit and a half
__device__ __forceinline__ long long fx_mul_hi(long long a, long long b) {
  const int al = (int)a, bl = (int)b;
  const int ah = (int)(a >> 32) + (int)((uint32_t)al >> 31);
  const int bh = (int)(b >> 32) + (int)((uint32_t)bl >> 31);
  return (long long)ah * bh + (((long long)al * bh + (long long)ah * bl) >> 32);
}

// high word of |v|
__device__ __forceinline__ int fx_high(double v) { return __double2hiint(v) & 0x7fffffff; }

// u read in fixed point: scale = 2^(B1 - e)
struct FxVec {
  const double* __restrict__ u;
  double scale;
};
template <typename T>
__device__ __forceinline__ T get(const FxVec& u, size_t k) {
  return T(__double2ll_rn(u.u[k] * u.scale));
}

constexpr int kFxMaxExp = 250;
constexpr int kFxRange = 32;      // a tile with values below 2^-32 of its largest is left to FP64
constexpr int kFxLow = 7;         // a column 2^-7 below the largest is short of bits all over
constexpr int kFxNone = -100000;  // no fixed-point exponent: compute the tile in FP64
// The largest high words (without sign) of a tile's positive and negative values, and its
// smallest nonzero one (less 1).
struct FxTop {
  int pos = 0, neg = 0;
  unsigned low = 0xffffffffu;
  __device__ __forceinline__ void add(double v) {
    const int h = __double2hiint(v);
    pos = max(pos, h);
    neg = max(neg, h ^ (int)0x80000000);  // negative for h >= 0
    low = min(low, (h & 0x7fffffffu) - 1u);
  }
  __device__ __forceinline__ void warp_max() {
    pos = __reduce_max_sync(0xffffffffu, pos);
    neg = __reduce_max_sync(0xffffffffu, neg);
    low = __reduce_min_sync(0xffffffffu, low);
  }
  // whether these values, not all zero (or outside the mesh), are below 2^(e - kFxLow)
  __device__ __forceinline__ bool far_below(int e) const {
    const int top = max(pos, neg);
    return top > 0 && ((top + 1) >> 20) - 1022 + kFxLow < e;
  }
  // e with |u| <= 2^e (1 - 2^-20) (the margin keeps the signed splits of products in range),
  // or kFxNone
  __device__ __forceinline__ int exponent() const {
    const int e = ((max(pos, neg) + 1) >> 20) - 1022, minor = (min(pos, neg) >> 20) - 1022;
    const int least = (int)(low >> 20) - 1022;
    return e >= -kFxMaxExp && e <= kFxMaxExp && minor + 12 <= e && least + kFxRange >= e ? e : kFxNone;
  }
};

}  // namespace fmg
