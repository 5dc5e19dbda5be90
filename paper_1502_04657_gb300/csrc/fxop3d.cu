// The 3D level operator L = A + W on the large levels in 64-bit fixed point: damped Jacobi,
// residual and operator apply of the FP64 mode (fxop2d.cu is the 2D form).
//
// The FP64 kernels (grid3d.cu) need 15 to 16 FP64 operations per node, 8 clocks of an SM's
// FP64 pipe (2 lanes per clock), and read the eight stored coupling arrays (64 B per node).
// Here a block covers a 32 x 8 x kZ tile of nodes, holds x of the tile and its halo in shared
// memory as integers in units of 2^(e - kB), e one exponent for the block's x and f, and
// computes L / h:
//   - the stiffness 6x - (sum of the six axis neighbours) exactly;
//   - the potential's part from closed forms.  With the node's indices a_d, the neighbour
//     pairs p_o = x(+o) + x(-o) and differences d_o = x(+o) - x(-o) of the 7 directions
//     (X, Y, Z, XY, XZ, YZ, XYZ) and the P1 integrals of grid3d.cu,
//       W x / h = al S + sum_d be_d D_d + small,
//       al   = h^2 W(x) / 60 + h^4 s / 504,   be_d = h^4 w_d a_d / 60,   s = wx + wy + wz,
//       S    = 24 x + 3 (p_X + p_Y + p_Z + p_XYZ) + 2 (p_XY + p_XZ + p_YZ),
//       D_d  = 3 (d_d + d_XYZ) + 2 (the differences of the two face diagonals along d),
//       small = h^4 [ 23/2520 s p_XYZ + sum_d (w_d / 90 - s / 504) p_d
//                     + sum_faces (s / 168 - w_o / 120) p_face ],  o the axis across the face;
//       al = ax[i] + ay[j] + az[l] and be_d come from 1D tables scaled to fill the integers, the
//       small terms (h^2 below the others) take the upper 30 bits of the pairs.
// Only the products, x and f round, at 2^-57 of the tile's maximum, and the small terms at 2^-50 of
// it or below (2^-33 of h^4 s); f / h, up to 8 times the maximum, is rounded by FP64.  FP64 rounds each
// of its 15 operations and every stored coupling at 2^-53, relative to the node's own stencil: a
// block where three nodes in a column lie 2^-20 or more below its largest value (or, for x = 0,
// where f does) is left to FP64, so that every node keeps 2^-30 of its own stencil.
//
// Measured on 16.6M nodes: Jacobi 438 -> 247 us, residual 413 -> 224 us.  The instruction rate
// bounds it (some 400 integer instructions per node, half of the issue slots used), then the
// latency of a block's loads: the whole tile is loaded at once (walking the planes through a
// ring of four with a pass ahead for the exponent took 300 and 285 us).
//
// The operator apply of the augmented pass also stores M x = h^3/60 S: the two applies took 195
// and 573 us on 16.6M nodes, together 203 us.
//
// Blocks with infinities, NaN, all zeros or an exponent outside +-kFxMaxExp run the FP64 expressions
// of grid3d.cu, too.  Instances whose potential is too large for the formats (fxop3d_scale: h^2 |W| >
// 60/64 or h^4 s > 2^-17) take grid3d.cu's kernels and stored couplings: with the couplings formed
// from their 1D tables at every use (46 FP64 operations per node and more, where those kernels need
// 16) two V-cycles at h = 10/256 took 16.4 ms, the FP64 kernels 5.8.
#include "dfloat.cuh"
#include "fixed.cuh"
#include "fmg_internal.h"

namespace fmg {
namespace {

constexpr int kB = 57;                       // x = I 2^(e - kB); |S| <= 60 2^kB
constexpr int kX = 32, kY = 8, kZ = 8;       // tile of columns (= threads), planes per block
constexpr int kRange = 20;                   // range of a block, in bits
constexpr int kNX = kX + 2, kNodes = (kX + 2) * (kY + 2);

// Tables ax, ay, az, bx, by, bz (n + 1 entries each) and the header of each instance.
__global__ void k_fxop3d_tables(int n, double h, const PotentialParams* __restrict__ pp,
                                long long* __restrict__ tab, FxHead3D* __restrict__ head) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x > n) return;
  const PotentialParams p = pp[blockIdx.y];
  tab += (size_t)blockIdx.y * 6 * (n + 1);
  const double wl = p.operator_form == FMG_W_LEFT ? 1.0 : 0.0;
  const double h2 = h * h, h4 = h2 * h2;
  const double w[3] = {wl * p.wx, wl * p.wy, wl * p.wz}, w0 = wl * p.w0;
  const double s = w[0] + w[1] + w[2];
  const FxScale fs = fxop3d_scale(n, h, p);
  const int sa = fs.sa, ss = fs.ss;
  const double sc = ldexp(1.0, 61 + sa), d = x;
  const double c0 = h2 * w0 / 60.0 + h4 * s / 504.0;
  for (int q = 0; q < 3; ++q) {
    tab[q * (n + 1) + x] = __double2ll_rn(sc * ((q == 0 ? c0 : 0.0) + h4 * w[q] * d * d / 60.0));
    tab[(3 + q) * (n + 1) + x] = __double2ll_rn(sc * (h4 * w[q] * d / 60.0));
  }
  if (x == 0) {
    FxHead3D q;
    q.sa = sa - 3;                 // shift of the products' sum
    q.sm = min(63, ss - sa + 11);  // shift of the small terms to the products' units
    const double t = ldexp(h4, 36 + ss);
    q.P = (int)__double2ll_rn(t * s * (23.0 / 2520.0));
    for (int a = 0; a < 3; ++a) {
      q.A[a] = (int)__double2ll_rn(t * (w[a] / 90.0 - s / 504.0));
      // faces XY, XZ, YZ: the axis across is z, y, x
      q.F[a] = (int)__double2ll_rn(t * (s / 168.0 - w[2 - a] / 120.0));
    }
    // the constant parts of the couplings, as k_coef3d forms them
    const double w3 = wl * (h * h * h) * p.w0;
    const double axis = -h + w3 * (1.0 / 20.0), face = w3 * (1.0 / 30.0);
    const double K[8] = {6.0 * h + w3 * 0.4, axis, axis, axis, face, face, face, w3 * (1.0 / 20.0)};
    for (int a = 0; a < 8; ++a) q.K[a] = K[a];
    head[blockIdx.y] = q;
  }
}

enum Mode { kJacobiMode, kResidualMode, kApplyMode, kApplyMassMode };
constexpr bool applies(int mode) { return mode == kApplyMode || mode == kApplyMassMode; }

__device__ __forceinline__ long dir(int d, int pitch, long plane) {
  constexpr int ox[7] = {1, 0, 0, 1, 1, 0, 1}, oy[7] = {0, 1, 0, 1, 0, 1, 1},
                oz[7] = {0, 0, 1, 0, 1, 1, 1};
  return ox[d] + (long)oy[d] * pitch + oz[d] * plane;
}

// The block's nodes in FP64, with the expressions of grid3d.cu (the couplings, which these instances
// don't store, from k_coef3d's tables and constants).
template <int MODE>
__device__ __noinline__ void tile_fp64(int n, int pitch, size_t base, int ib, int x, int y, int z0,
                                       int z1,
                                       const Coef3D& c, const double* __restrict__ f,
                                       const double* __restrict__ v, double* __restrict__ out,
                                       double mscale, double* __restrict__ mv) {
  if (x > n - 1 || y > n - 1) return;
  const long plane = (long)(n + 1) * pitch;
  constexpr int kQ[8][3] = {{0, 0, 0}, {1, 2, 2}, {2, 1, 2}, {2, 2, 1},
                            {3, 3, 4}, {3, 4, 3}, {4, 3, 3}, {1, 1, 1}};
  const int s = n + 1;
  const double* T = c.tab + (size_t)ib * 15 * s;
  // coupling q of the node (x, y, z) - b d(q - 1)
  auto a = [&](int q, int z, int b) {
    const int ox = b && (q == 1 || q == 4 || q == 5 || q == 7),
              oy = b && (q == 2 || q == 4 || q == 6 || q == 7),
              oz = b && (q == 3 || q == 5 || q == 6 || q == 7);
    return ((c.fxh[ib].K[q] + T[(5 + kQ[q][1]) * s + y - oy]) + T[(10 + kQ[q][2]) * s + z - oz]) +
           T[kQ[q][0] * s + x - ox];
  };
  for (int z = z0; z < z1; ++z) {
    const size_t k = base + z * plane + (long)y * pitch + x;
    double r = applies(MODE) ? a(0, z, 0) * v[k] : fma(-a(0, z, 0), v[k], f[k]);
    double m = 24.0 * v[k];
    for (int d = 0; d < 7; ++d) {
      const long o = dir(d, pitch, plane);
      const double sg = applies(MODE) ? 1.0 : -1.0;
      r = fma(sg * a(1 + d, z, 0), v[k + o], r);
      r = fma(sg * a(1 + d, z, 1), v[k - o], r);
      if (MODE == kApplyMassMode) m = fma(d >= 3 && d < 6 ? 2.0 : 3.0, v[k + o] + v[k - o], m);
    }
    if (MODE == kApplyMassMode) mv[k] = mscale * m;
    out[k] = MODE == kJacobiMode ? fma(c.dinv[k], r, v[k]) : r;
  }
}

template <int MODE>
__global__ void __launch_bounds__(kX * kY, 3)
    k_fxop3d(int n, int pitch, size_t st, double h, double hinv, int hexp,
             const __grid_constant__ Coef3D c, const double* __restrict__ f,
             const double* __restrict__ v, double* __restrict__ out, double mscale,
             double* __restrict__ mv) {
  __shared__ long long su[kZ + 2][kNodes];  // planes z0 - 1 .. z0 + kZ
  __shared__ int top[2];
  __shared__ unsigned low[2];
  const int nzc = (n - 1 + kZ - 1) / kZ, ib = blockIdx.z / nzc;
  const int z0 = 1 + (int)(blockIdx.z - ib * nzc) * kZ, z1 = min(z0 + kZ, n);
  const int x0 = 1 + blockIdx.x * kX, y0 = 1 + blockIdx.y * kY;
  const long plane = (long)(n + 1) * pitch;
  const size_t base = ib * st;
  const int tid = threadIdx.y * kX + threadIdx.x;
  const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
  const bool active = x <= n - 1 && y <= n - 1;
  // the two plane elements this thread stages (the second one for tid < kNodes - kX kY)
  const int e1 = tid + kX * kY;
  const int xa = x0 - 1 + tid % kNX, ya = y0 - 1 + tid / kNX;
  const int xb = x0 - 1 + e1 % kNX, yb = y0 - 1 + e1 / kNX;
  const bool ina = xa <= n && ya <= n, inb = e1 < kNodes && xb <= n && yb <= n;
  const double* pa = v + base + (long)ya * pitch + xa;
  const double* pb = v + base + (long)yb * pitch + xb;
  const double* pf = f + base + (long)y * pitch + x;
  if (tid < 2) {
    top[tid] = 0;
    low[tid] = 0xffffffffu;
  }
  __syncthreads();
  // the whole tile is loaded first (a block's loads in flight at once), its exponent taken, and
  // its integers stored to shared memory, so that the planes below need no barrier
  double va[kZ + 2], vb[kZ + 2];
  {
    int m = 0, mf = 0;
    unsigned lx = 0xffffffffu, lf = 0xffffffffu;  // least nonzero values, less 1
#pragma unroll
    for (int t = 0; t < kZ + 2; ++t) {
      const int z = z0 - 1 + t;
      va[t] = ina && z <= n ? pa[z * plane] : 0.0;
      vb[t] = inb && z <= n ? pb[z * plane] : 0.0;
    }
    if (!applies(MODE) && active) {
#pragma unroll
      for (int t = 0; t < kZ; ++t)
        if (z0 + t < z1) {
          const int v = fx_high(pf[(z0 + t) * plane]);
          mf = max(mf, v);
          lf = min(lf, (unsigned)v - 1u);
        }
    }
#pragma unroll
    for (int t = 1; t <= kZ; ++t) {
      const int a = max(max(fx_high(va[t - 1]), fx_high(va[t])), fx_high(va[t + 1])),
                b = max(max(fx_high(vb[t - 1]), fx_high(vb[t])), fx_high(vb[t + 1]));
      m = max(m, max(a, b));
      lx = min(lx, min((unsigned)a - 1u, (unsigned)b - 1u));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    lx = __reduce_min_sync(0xffffffffu, lx);
    if (!applies(MODE)) {
      mf = __reduce_max_sync(0xffffffffu, mf);
      lf = __reduce_min_sync(0xffffffffu, lf);
    }
    if ((tid & 31) == 0) {
      atomicMax(&top[0], m);
      atomicMax(&top[1], mf);
      atomicMin(&low[0], lx);
      atomicMin(&low[1], lf);
    }
  }
  __syncthreads();
  // f / h counts an eighth (exponents are added as such: the sum of high words may wrap)
  const int ex = ((top[0] + 1) >> 20) - 1022, ef = ((top[1] + 1) >> 20) - 1022 + hexp - 3;
  const int e = top[1] == 0 ? ex : max(ex, ef);
  const FxHead3D hd = c.fxh[ib];
  if (c.fits && !c.fits[ib]) return;  // an instance of the FP64 form
  const int least = top[0] ? (int)(low[0] >> 20) - 1022 : (int)(low[1] >> 20) - 1022 + hexp - 3;
  if (top[1] >= 0x7ff00000 || e < -kFxMaxExp || e > kFxMaxExp || least + kRange < e) {
    tile_fp64<MODE>(n, pitch, base, ib, x, y, z0, z1, c, f, v, out, mscale, mv);
    return;
  }
  const int shift = e + 1085 - kB;
  const double fs = hinv * fx_pow2(kB - e), back = h * fx_pow2(e - kB);
  const double mback = mscale * fx_pow2(e - kB);
  const long long* tab = c.fxt + (size_t)ib * 6 * (n + 1);
  const int xc = min(x, n), yc = min(y, n);
  const long long axy = tab[xc] + tab[(n + 1) + yc], bx = tab[3 * (n + 1) + xc],
                  by = tab[4 * (n + 1) + yc];
  const long long half = 1ll << (hd.sa - 1);
  // the small terms drop the lower bits of the pairs: half a unit each on average
  const long long q0 = ((long long)hd.P + hd.A[0] + hd.A[1] + hd.A[2] + hd.F[0] + hd.F[1] +
                        hd.F[2]) / 2;
#pragma unroll
  for (int t = 0; t < kZ + 2; ++t) {
    su[t][tid] = fx_truncated(va[t], shift);
    if (e1 < kNodes) su[t][e1] = fx_truncated(vb[t], shift);
  }
  __syncthreads();
  if (!active) return;
  const int nd = (threadIdx.y + 1) * kNX + threadIdx.x + 1;
  size_t k = base + z0 * plane + (long)y * pitch + x;
#pragma unroll 2
  for (int t = 1; z0 + t <= z1; ++t, k += plane) {
    const int z = z0 + t - 1;
    const double fv = !applies(MODE) ? f[k] : 0.0;
    const double di = MODE == kJacobiMode ? c.dinv[k] : 0.0;
    const double xv = MODE == kJacobiMode ? v[k] : 0.0;
    const long long* s0 = su[t] + nd;
    const long long* sp = su[t + 1] + nd;
    const long long* sm = su[t - 1] + nd;
    {
      // sums and differences of the neighbours +o and -o, direction by direction
      const long long u = s0[0];
      long long q, dx, dy, dz, pa2, pf2;
      {
        const long long a = s0[1], b = s0[-1], p = a + b;
        dx = a - b;
        pa2 = p;
        q = q0 + (long long)hd.A[0] * (int)(p >> 28);
      }
      {
        const long long a = s0[kNX], b = s0[-kNX], p = a + b;
        dy = a - b;
        pa2 += p;
        q += (long long)hd.A[1] * (int)(p >> 28);
      }
      {
        const long long a = sp[0], b = sm[0], p = a + b;
        dz = a - b;
        pa2 += p;
        q += (long long)hd.A[2] * (int)(p >> 28);
      }
      const long long r6 = 6 * u - pa2;  // the stiffness
      {
        const long long a = sp[kNX + 1], b = sm[-kNX - 1], p = a + b, d = a - b;
        dx += d;
        dy += d;
        dz += d;
        pa2 += p;
        q += (long long)hd.P * (int)(p >> 28);
      }
      // D = 3 (axis and body) + 2 (faces): the first three carry 1, the sum below doubles both
      long long ex, ey, ez;
      {
        const long long a = s0[kNX + 1], b = s0[-kNX - 1], p = a + b, d = a - b;
        ex = dx + d;
        ey = dy + d;
        pf2 = p;
        q += (long long)hd.F[0] * (int)(p >> 28);
      }
      {
        const long long a = sp[1], b = sm[-1], p = a + b, d = a - b;
        ex += d;
        ez = dz + d;
        pf2 += p;
        q += (long long)hd.F[1] * (int)(p >> 28);
      }
      {
        const long long a = sp[kNX], b = sm[-kNX], p = a + b, d = a - b;
        ey += d;
        ez += d;
        pf2 += p;
        q += (long long)hd.F[2] * (int)(p >> 28);
      }
      const long long t = 8 * u + pa2, S = 2 * (t + pf2) + t;
      long long w = fx_mul_hi(axy + tab[2 * (n + 1) + z], S) + fx_mul_hi(bx, 2 * ex + dx) +
                    fx_mul_hi(by, 2 * ey + dy) + fx_mul_hi(tab[5 * (n + 1) + z], 2 * ez + dz);
      w += (q >> hd.sm) + half;
      long long r = r6 + (w >> hd.sa);
      if (!applies(MODE)) r = __double2ll_rn(fv * fs) - r;
      const double rd = __ll2double_rn(r);
      out[k] = MODE == kJacobiMode ? fma(di * back, rd, xv) : rd * back;
      if (MODE == kApplyMassMode) mv[k] = __ll2double_rn(S) * mback;
    }
  }
}

template <int MODE>
void launch(const Grid& g, const Coef3D& c, const double* f, const double* x, double* out,
            cudaStream_t s, double* mx = nullptr) {
  const dim3 grid((g.n - 1 + kX - 1) / kX, (g.n - 1 + kY - 1) / kY,
                  g.nb * ((g.n - 1 + kZ - 1) / kZ));
  int ex = 0;
  frexp(1.0 / g.h, &ex);  // 1 / h < 2^ex
  k_fxop3d<MODE><<<grid, dim3(kX, kY), 0, s>>>(g.n, g.pitch, g.stride, g.h, 1.0 / g.h, ex, c,
                                               applies(MODE) ? x : f, x, out,
                                               g.h * g.h * g.h / 60.0, mx);
}

}  // namespace

void fxop3d_tables(const Grid& g, const PotentialParams* p, const Coef3D& c, cudaStream_t s) {
  k_fxop3d_tables<<<dim3((g.n + 1 + 127) / 128, g.nb), 128, 0, s>>>(g.n, g.h, p, c.fxt, c.fxh);
}
void fxop3d_apply(const Grid& g, const Coef3D& c, const double* x, double* y, cudaStream_t s) {
  launch<kApplyMode>(g, c, nullptr, x, y, s);
}
void fxop3d_apply_mass(const Grid& g, const Coef3D& c, const double* x, double* y, double* mx,
                       cudaStream_t s) {
  launch<kApplyMassMode>(g, c, nullptr, x, y, s, mx);
}
void fxop3d_jacobi(const Grid& g, const Coef3D& c, const double* f, const double* x, double* xo,
                   cudaStream_t s) {
  launch<kJacobiMode>(g, c, f, x, xo, s);
}
void fxop3d_residual(const Grid& g, const Coef3D& c, const double* f, const double* x, double* r,
                     cudaStream_t s) {
  launch<kResidualMode>(g, c, f, x, r, s);
}

}  // namespace fmg
