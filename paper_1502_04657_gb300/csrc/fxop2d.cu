// The 2D level operator L = A + W on the large levels in 64-bit fixed point: damped Jacobi,
// residual (FP64, or rounded to single precision for the mixed modes) and operator apply.
//
// The FP64 kernels (grid2d.cu) need 7 to 8 FP64 operations per node, 4 clocks of an SM's FP64
// pipe (2 lanes per clock), and read the four stored coupling arrays.  Here a warp covers a
// tile of 64 columns (62 produced, two per lane) x 4 rows (and one more on each side), takes
// one exponent e for its x and f, and computes the stencil in integers in units of 2^(e - 58):
//   - the stiffness 4x - E - W - N - S exactly (integer additions);
//   - the potential's part from closed forms instead of stored couplings.  With node (i, j),
//     the six neighbours and the P1 integrals at the head of grid2d.cu,
//       W x = a (6x + sum of the six) + bx Dx + by Dy + small,
//       a  = h^2 W(x_i, y_j) / 12 + h^4 (wx + wy) / 40,   bx = h^4 wx i / 12,   by = h^4 wy j / 12,
//       Dx = (E - W) + (NE - SW),    Dy = (N - S) + (NE - SW),
//       small = -h^4 [ 17/180 (wx + wy) x + 7/360 wy (E + W) + 7/360 wx (N + S) ],
//     with a = ax[i] + ay[j], bx[i], by[j] from 1D tables, scaled by 2^(61 + sa) so that they
//     fill the integers, and the small terms (h^2 below the others) from the high words.
// Only the products, x and f round, at 2^-58 of the tile's maximum, and the small terms at 2^-50 of
// it or below (2^-26 of h^4 (wx + wy)).  FP64 rounds each of its operations at 2^-53, and each
// stored coupling -1 + O(h^2) at 2^-53: a relative perturbation of W by 2^-53 / h^2, 4e-9 at h =
// 1/4096, that this form does not have.  FP64's rounding is relative to each node's own stencil, so
// a tile where some lane's values (of its and the neighbouring lanes' columns) lie 2^-7 or more
// below the largest takes an exponent per lane, which costs a second conversion of each neighbour's
// value (16.8M nodes, every tile so: Jacobi 15 us more, apply 23).
// The operator apply of the augmented pass also stores M x = h^2/12 (6x + sum of the six), whose
// sum is at hand: the two applies took 117 and 227 us on 16.8M nodes, together 152 us.
// The update x + (omega / D) r is one FP64 operation as before.  What is left is the instruction
// rate (about 200 integer instructions per node) and the latency between a tile's loads and its
// arithmetic: 4 rows a warp and 5 blocks per SM took 156 us (Jacobi) and 127 us (residual) on
// 16.8M nodes, 8 rows and 4 blocks 180 and 142; the FP64 form took 225 and 198.
//
// Tiles with infinities, NaN, all zeros or an exponent outside +-kFxMaxExp run the FP64 expressions
// of grid2d.cu.  Instances whose potential is too large for the fixed formats (fxop2d_scale: h^2 |W|
// > 12/64 or h^4 (|wx| + |wy|) > 2^-22) take grid2d.cu's kernels and stored couplings: forming the
// couplings from their 1D tables at every use, 15 FP64 operations per node where those kernels need
// 8, took 2.00 ms for two V-cycles at h = 20/2048, the FP64 kernels 1.25.
#include <cuda_bf16.h>

#include "dfloat.cuh"
#include "fixed.cuh"
#include "fmg_internal.h"

namespace fmg {
namespace {

constexpr int kB = 58;         // x = I 2^(e - kB)
constexpr int kRows = 4;       // rows a warp produces
constexpr int kWarps = 4;      // warps of a block, stacked in y
constexpr int kCols = 62;      // columns a warp produces
constexpr int kBlocks = 5;     // resident blocks per SM
constexpr int kLaneRange = 7;  // lanes of a tile of one exponent: within 2^-7 of its largest

// Tables ax, ay, bx, by (n + 1 entries each) and the header of each instance.
__global__ void k_fxop2d_tables(int n, double h, const PotentialParams* __restrict__ pp,
                                long long* __restrict__ tab, FxHead2D* __restrict__ head) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x > n) return;
  const PotentialParams p = pp[blockIdx.y];
  tab += (size_t)blockIdx.y * 4 * (n + 1);
  const double wl = p.operator_form == FMG_W_LEFT ? 1.0 : 0.0;
  const double h2 = h * h, h4 = h2 * h2;
  const double w0 = wl * p.w0, wx = wl * p.wx, wy = wl * p.wy;
  const FxScale fs = fxop2d_scale(n, h, p);
  const int sa = fs.sa, ss = fs.ss;
  const double s = ldexp(1.0, 61 + sa), d = x;
  tab[x] = __double2ll_rn(s * (h2 * w0 / 12.0 + h4 * (wx + wy) / 40.0 + h4 * wx * d * d / 12.0));
  tab[(n + 1) + x] = __double2ll_rn(s * (h4 * wy * d * d / 12.0));
  tab[2 * (n + 1) + x] = __double2ll_rn(s * (h4 * wx * d / 12.0));
  tab[3 * (n + 1) + x] = __double2ll_rn(s * (h4 * wy * d / 12.0));
  if (x == 0) {
    FxHead2D q;
    q.sa = sa - 3;       // shift of the products' sum
    q.sm = min(63, ss - sa + 1);  // shift of the small terms to the products' units
    const double t = ldexp(h4, 30 + ss);
    q.P = (int)__double2ll_rn(t * (wx + wy) * (-17.0 / 180.0));
    q.Q = (int)__double2ll_rn(t * wy * (-7.0 / 360.0));
    q.R = (int)__double2ll_rn(t * wx * (-7.0 / 360.0));
    q.omega = p.omega;
    head[blockIdx.y] = q;
  }
}

// v 2^e by the exponent field: v normal and nonzero, the result in the normal range
__device__ __forceinline__ double times_pow2(double v, int e) {
  return __hiloint2double(__double2hiint(v) + e * (1 << 20), __double2loint(v));
}

// kJacobiTabMode: Jacobi with omega / D from the tables (levels that don't store it)
enum Mode { kJacobiMode, kJacobiTabMode, kResidualMode, kApplyMode, kApplyMassMode };
constexpr bool jacobi(int mode) { return mode == kJacobiMode || mode == kJacobiTabMode; }
constexpr bool applies(int mode) { return mode == kApplyMode || mode == kApplyMassMode; }

__device__ __forceinline__ void store(double* o, size_t k, double v) { o[k] = v; }
__device__ __forceinline__ void store(float* o, size_t k, double v) { o[k] = d2f_rn(v); }
__device__ __forceinline__ void store(__nv_bfloat16* o, size_t k, double v) {
  o[k] = __float2bfloat16(d2f_rn(v));
}

// The tile in FP64, with the expressions of grid2d.cu / mixed.cu (the couplings, which these
// instances don't store, from the same tables).
template <int MODE, typename S>
__device__ __noinline__ void tile_fp64(int n, int pitch, size_t base, int ib, int i0, int j0,
                                       const Coef2D& c, const double* __restrict__ f,
                                       const double* __restrict__ x, S* __restrict__ out,
                                       double mscale, double* __restrict__ mx) {
  const int s = n + 1;
  const double* t = c.tab + (size_t)ib * 8 * s;
  auto cC = [&](int i, int j) { return t[i] + t[4 * s + j]; };
  auto cE = [&](int i, int j) { return t[s + i] + t[5 * s + j]; };
  auto cN = [&](int i, int j) { return t[2 * s + i] + t[6 * s + j]; };
  auto cNE = [&](int i, int j) { return t[3 * s + i] + t[7 * s + j]; };
  for (int j = j0; j < min(j0 + kRows, n); ++j)
    for (int q = 0; q < 2; ++q) {
      const int i = i0 + q, lane = threadIdx.x;
      if (i < 1 || i > n - 1 || (lane == 0 && q == 0) || (lane == 31 && q == 1)) continue;
      const size_t k = base + (size_t)j * pitch + i;
      double r;
      if (applies(MODE)) {
        r = cC(i, j) * x[k];
        r = fma(cE(i, j), x[k + 1], r);
        r = fma(cE(i - 1, j), x[k - 1], r);
        r = fma(cN(i, j), x[k + pitch], r);
        r = fma(cN(i, j - 1), x[k - pitch], r);
        r = fma(cNE(i, j), x[k + pitch + 1], r);
        r = fma(cNE(i - 1, j - 1), x[k - pitch - 1], r);
      } else {
        r = fma(-cC(i, j), x[k], f[k]);
        r = fma(-cE(i, j), x[k + 1], r);
        r = fma(-cE(i - 1, j), x[k - 1], r);
        r = fma(-cN(i, j), x[k + pitch], r);
        r = fma(-cN(i, j - 1), x[k - pitch], r);
        r = fma(-cNE(i, j), x[k + pitch + 1], r);
        r = fma(-cNE(i - 1, j - 1), x[k - pitch - 1], r);
        if (jacobi(MODE)) {
          const double di = MODE == kJacobiMode ? c.dinv[k] : ratio(c.fxh[ib].omega, cC(i, j));
          r = fma(di, r, x[k]);
        }
      }
      store(out, k, r);
      if (MODE == kApplyMassMode)
        mx[k] = mscale * fma(6.0, x[k], ((x[k + 1] + x[k - 1]) + (x[k + pitch] + x[k - pitch])) +
                                            (x[k + pitch + 1] + x[k - pitch - 1]));
    }
}

// The tile of a warp, rows j0 - 1 .. j0 + kRows of x in xv (this lane's columns i0, i0 + 1), in units
// of 2^(e - kB).  LANES: e is the lane's own; lanes with fp64 set pass their values on and are
// evaluated in FP64 at the end.
template <int MODE, typename S, bool LANES>
__device__ __forceinline__ void tile_fixed(int n, int pitch, size_t base, int ib, int i0, int j0,
                                           const Coef2D& c, const double* __restrict__ f,
                                           const double* __restrict__ x, S* __restrict__ out,
                                           double mscale, double* __restrict__ mx,
                                           const double2 (&xv)[kRows + 2], int e, bool fp64) {
  const int lane = threadIdx.x;
  const bool in = i0 <= n;
  const double2 zero = make_double2(0.0, 0.0);
  auto f_row = [&](int r) {
    return in && r < n ? *reinterpret_cast<const double2*>(f + base + (size_t)r * pitch + i0) : zero;
  };
  const FxHead2D hd = c.fxh[ib];
  const int shift = e + 1085 - kB;
  const double back = fx_pow2(e - kB), mback = mscale * back;
  const long long* tab = c.fxt + (size_t)ib * 4 * (n + 1);
  const int ia = min(i0, n), ic = min(i0 + 1, n);
  const long long axa = tab[ia], axb = tab[ic], bxa = tab[2 * (n + 1) + ia],
                  bxb = tab[2 * (n + 1) + ic];
  const long long half = 1ll << (hd.sa - 1);
  // a row: this lane's pair (a, b), the left neighbour of a and the right one of b
  struct Row {
    long long l, a, b, r;
  };
  auto row = [&](const double2& v) {
    Row q;
    q.a = fx_truncated(v.x, shift);
    q.b = fx_truncated(v.y, shift);
    if (LANES) {  // the lanes beside have their own units
      q.l = fx_truncated(__shfl_up_sync(0xffffffffu, v.y, 1), shift);
      q.r = fx_truncated(__shfl_down_sync(0xffffffffu, v.x, 1), shift);
    } else {
      q.l = __shfl_up_sync(0xffffffffu, q.b, 1);
      q.r = __shfl_down_sync(0xffffffffu, q.a, 1);
    }
    return q;
  };
  // one node: (A + W) x in units of 2^(e - kB)
  auto node = [&](long long x0, long long xe, long long xw, long long xn, long long xs,
                  long long xne, long long xsw, long long a, long long bx, long long by,
                  long long& s6) {
    const long long ew = xe + xw, ns = xn + xs, d = xne + xsw, g = xne - xsw;
    const long long t = ew + ns;
    s6 = 6 * x0 + t + d;
    long long sm = (long long)hd.P * (int)(x0 >> 32) + (long long)hd.Q * (int)(ew >> 32) +
                   (long long)hd.R * (int)(ns >> 32);
    long long w = fx_mul_hi(a, s6) + fx_mul_hi(bx, (xe - xw) + g) + fx_mul_hi(by, (xn - xs) + g);
    w += (sm >> hd.sm) + half;
    return 4 * x0 - t + (w >> hd.sa);
  };
  Row s = row(xv[0]), m = row(xv[1]);
#pragma unroll
  for (int t = 0; t < kRows; ++t) {
    const int j = j0 + t;
    const Row p = row(xv[t + 2]);
    if (j < n) {
      const long long ay = tab[(n + 1) + j], by = tab[3 * (n + 1) + j];
      long long ma, mb;  // 12 / h^2 of the mass apply
      long long ra = node(m.a, m.b, m.l, p.a, s.a, p.b, s.l, axa + ay, bxa, by, ma);
      long long rb = node(m.b, m.r, m.a, p.b, s.b, p.r, s.a, axb + ay, bxb, by, mb);
      if (!applies(MODE)) {
        const double2 v = f_row(j);
        ra = fx_truncated(v.x, shift) - ra;
        rb = fx_truncated(v.y, shift) - rb;
      }
      const size_t k = base + (size_t)j * pitch + i0;
      const bool oka = lane > 0 && i0 <= n - 1 && !(LANES && fp64),
                 okb = lane < 31 && i0 + 1 <= n - 1 && !(LANES && fp64);
      double va = __ll2double_rn(ra), vb = __ll2double_rn(rb);
      if (jacobi(MODE)) {
        double2 di;
        if (MODE == kJacobiMode) {
          di = in ? *reinterpret_cast<const double2*>(c.dinv + k) : zero;
        } else {
          const double* t8 = c.tab + (size_t)ib * 8 * (n + 1);
          const double y = t8[4 * (n + 1) + j];
          di = make_double2(ratio(hd.omega, t8[ia] + y), ratio(hd.omega, t8[ic] + y));
        }
        va = fma(times_pow2(di.x, e - kB), va, xv[t + 1].x);
        vb = fma(times_pow2(di.y, e - kB), vb, xv[t + 1].y);
      } else {
        va *= back;
        vb *= back;
      }
      if (sizeof(S) == 8 && oka && okb) {
        *reinterpret_cast<double2*>(reinterpret_cast<double*>(out) + k) = make_double2(va, vb);
      } else {
        if (oka) store(out, k, va);
        if (okb) store(out, k + 1, vb);
      }
      if (MODE == kApplyMassMode) {
        const double za = __ll2double_rn(ma) * mback, zb = __ll2double_rn(mb) * mback;
        if (oka && okb) {
          *reinterpret_cast<double2*>(mx + k) = make_double2(za, zb);
        } else {
          if (oka) mx[k] = za;
          if (okb) mx[k + 1] = zb;
        }
      }
    }
    s = m;
    m = p;
  }
  if (LANES && fp64) tile_fp64<MODE, S>(n, pitch, base, ib, i0, j0, c, f, x, out, mscale, mx);
}

// The same with an exponent per lane, for the tiles whose lanes differ (called, and x read again: the
// common path keeps its registers).
template <int MODE, typename S>
__device__ __noinline__ void tile_lanes(int n, int pitch, size_t base, int ib, int i0, int j0,
                                        const Coef2D& c, const double* __restrict__ f,
                                        const double* __restrict__ x, S* __restrict__ out,
                                        double mscale, double* __restrict__ mx, int top) {
  double2 xv[kRows + 2];
#pragma unroll
  for (int t = 0; t < kRows + 2; ++t) {
    const int r = j0 - 1 + t;
    xv[t] = i0 <= n && r <= n ? *reinterpret_cast<const double2*>(x + base + (size_t)r * pitch + i0)
                              : make_double2(0.0, 0.0);
  }
  const int e = ((top + 1) >> 20) - 1022;
  const bool fp64 = e < -kFxMaxExp || e > kFxMaxExp;
  tile_fixed<MODE, S, true>(n, pitch, base, ib, i0, j0, c, f, x, out, mscale, mx, xv, fp64 ? 0 : e,
                            fp64);
}

template <int MODE, typename S>
__global__ void __launch_bounds__(32 * kWarps, kBlocks)
    k_fxop2d(int n, int pitch, size_t st, const __grid_constant__ Coef2D c,
             const double* __restrict__ f, const double* __restrict__ x, S* __restrict__ out,
             double mscale, double* __restrict__ mx) {
  const int lane = threadIdx.x, ib = blockIdx.z;
  const int i0 = kCols * blockIdx.x + 2 * lane;  // this lane's columns i0, i0 + 1
  const int j0 = 1 + kRows * (blockIdx.y * kWarps + threadIdx.y);
  if (j0 >= n) return;  // uniform over the warp
  const size_t base = ib * st;
  const bool in = i0 <= n;  // (i0 + 1 <= n + 1 < pitch then)
  double2 xv[kRows + 2];
#pragma unroll
  for (int t = 0; t < kRows + 2; ++t) {
    const int r = j0 - 1 + t;
    xv[t] = in && r <= n ? *reinterpret_cast<const double2*>(x + base + (size_t)r * pitch + i0)
                         : make_double2(0.0, 0.0);
  }
  // the largest of the lane's x and its neighbours', and of its f, which counts an eighth (|f| <=
  // 8 2^e fits beside the stencil of x).  f is read here and again, from L1, when its row is due.
  int top = 0;
#pragma unroll
  for (int t = 0; t < kRows + 2; ++t) top = max(top, max(fx_high(xv[t].x), fx_high(xv[t].y)));
  top = max(top, max(__shfl_up_sync(0xffffffffu, top, 1), __shfl_down_sync(0xffffffffu, top, 1)));
  if (!applies(MODE)) {
    int topf = 0;
#pragma unroll
    for (int t = 0; t < kRows; ++t)
      if (in && j0 + t < n) {
        const double2 v =
            *reinterpret_cast<const double2*>(f + base + (size_t)(j0 + t) * pitch + i0);
        topf = max(topf, max(fx_high(v.x), fx_high(v.y)));
      }
    top = max(top, topf - (3 << 20));
  }
  if (c.fits && !c.fits[ib]) return;  // an instance of the FP64 form
  // the tile's exponent, and its least lane's (lanes of zeros: none)
  const int most = __reduce_max_sync(0xffffffffu, top);
  const unsigned least = __reduce_min_sync(0xffffffffu, (unsigned)top - 1u);
  const int e = ((most + 1) >> 20) - 1022;
  if (e < -kFxMaxExp || e > kFxMaxExp)
    tile_fp64<MODE, S>(n, pitch, base, ib, i0, j0, c, f, x, out, mscale, mx);
  else if ((int)(least >> 20) - 1022 + kLaneRange < e)
    tile_lanes<MODE, S>(n, pitch, base, ib, i0, j0, c, f, x, out, mscale, mx, top);
  else
    tile_fixed<MODE, S, false>(n, pitch, base, ib, i0, j0, c, f, x, out, mscale, mx, xv, e, false);
}

template <int MODE, typename S>
void launch(const Grid& g, const Coef2D& c, const double* f, const double* x, S* out,
            cudaStream_t s, double* mx = nullptr) {
  const dim3 grid((g.n - 1 + kCols - 1) / kCols,
                  (g.n - 1 + kRows * kWarps - 1) / (kRows * kWarps), g.nb);
  k_fxop2d<MODE, S><<<grid, dim3(32, kWarps), 0, s>>>(g.n, g.pitch, g.stride, c, f, x, out,
                                                     g.h * g.h / 12.0, mx);
}

}  // namespace

void fxop2d_tables(const Grid& g, const PotentialParams* p, const Coef2D& c, cudaStream_t s) {
  k_fxop2d_tables<<<dim3((g.n + 1 + 127) / 128, g.nb), 128, 0, s>>>(g.n, g.h, p, c.fxt, c.fxh);
}
void fxop2d_apply(const Grid& g, const Coef2D& c, const double* x, double* y, cudaStream_t s) {
  launch<kApplyMode>(g, c, nullptr, x, y, s);
}
void fxop2d_apply_mass(const Grid& g, const Coef2D& c, const double* x, double* y, double* mx,
                       cudaStream_t s) {
  launch<kApplyMassMode>(g, c, nullptr, x, y, s, mx);
}
void fxop2d_jacobi(const Grid& g, const Coef2D& c, const double* f, const double* x, double* xo,
                   cudaStream_t s) {
  if (c.dinv) launch<kJacobiMode>(g, c, f, x, xo, s);
  else launch<kJacobiTabMode>(g, c, f, x, xo, s);
}
void fxop2d_residual(const Grid& g, const Coef2D& c, const double* f, const double* x, double* r,
                     cudaStream_t s) {
  launch<kResidualMode>(g, c, f, x, r, s);
}
void fxop2d_residual32(const Grid& g, const Coef2D& c, const double* f, const double* x, float* r,
                       bool bf, cudaStream_t s) {
  if (bf) launch<kResidualMode>(g, c, f, x, reinterpret_cast<__nv_bfloat16*>(r), s);
  else launch<kResidualMode>(g, c, f, x, r, s);
}

}  // namespace fmg
