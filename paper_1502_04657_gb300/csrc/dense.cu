// Small dense FP64 solves: the nonlinear eigenproblem on V_{h_1} (Algorithm 3.2 step 1) and
// on the augmented space V_H + span{u~} (Algorithm 3.1 step 2), plus the coarsest-level
// inverse used by the V-cycle.
//
// The nonlinear problem on an n-dimensional space with basis psi is
//     F(c, lambda) = (K0 + zeta G(c)) c - lambda M c = 0,   c^T M c = 1,
// G(c)_ij = int w^2 psi_i psi_j, w = sum_j c_j psi_j.  Section 3.2 allows self-consistent
// or Newton-type iterations; both converge to the same ground state, which is what the
// result is.  This kernel takes inverse-power steps c <- (K0 + zeta G(c))^{-1} M c while the
// relative residual is large (they pull any positive start into the ground state's basin),
// then Newton steps, which converge quadratically.  A Newton step solves the bordered system
//     [A    -M c] [dc]   [-r]        A = K0 + 3 zeta G(c) - lambda M,  r = F(c, lambda)
//     [-c^T M  0] [dl] = [ 0]        (d/dc of G(c) c is 3 G(c) for the cubic term)
// by block elimination with A' = A + lambda (M c)(M c)^T: the constraint (M c)^T dc = 0 makes
// A' dc = A dc, and A' is positive definite near the ground state (A is semidefinite there,
// singular only along c), so elimination without pivoting applies:
//     y1 = A'^{-1} r,  y2 = A'^{-1} M c,  dl = (Mc.y1)/(Mc.y2),  dc = -y1 + dl y2.
// lambda is reported as c^T (K0 + zeta G(c)) c at the final c.
//
// What bounds it.  One CTA works on one SM, whose four FP64 units take 64 cycles per warp
// instruction each whether its lanes do useful work or not, so the cost is the number of
// FP64 warp instructions on the longest chain, then barriers.  Hence:
//   - The residual never needs G(c): its FP64 evaluation forms the load int w^3 psi_i
//     (evaluate below).  With w = w_H + c_u u~ that is, per coarse row a,
//         int w_H^3 phi_a + 3 c_u X c + 3 c_u^2 B1 c + c_u^3 t1,   X_ab = sum_T sum_c w_c T3_abc,
//     from the fine-pass integrals (augment2d.cu): T3 (summed over the simplices that share a
//     vertex triple when the kernel starts, dense_lists.h), B1 = int u~^2 phi phi,
//     t1 = int u~^3 phi, T0 = int u~^4; and int_T w_H^3 mu_a = |T| 3! d!/(d + 4)!
//     h_3(w_1 .. w_nv, w_a) = .. [h_3 + w_a h_2 + w_a^2 h_1 + w_a^3], h_q the complete
//     homogeneous symmetric polynomials of the vertex values, so each simplex forms h_1, h_2,
//     h_3 once for its vertices.  K0, M and B1 are kept as their nonzeros.
//   - c is not rescaled before an evaluation: every term is homogeneous in c, so the factor
//     f = +-(c^T M c)^{-1/2} is applied to the sums.
//   - The small scalar chains are Horner evaluations in c_u, one chain per lane.
//   - The Jacobian A' (and K0 + zeta G) is assembled and inverted in single precision, whose
//     pipes issue 64 times faster; what the ~1e-6 relative error of a step leaves is removed
//     by further steps with the same inverse against the FP64 residual (a chord step costs one
//     evaluation), so c and lambda are exact to the FP64 residual as before.
// Measured (ncu, every dense launch of one solve summed): 2D h = 1/64 983 -> 359 us, 2D
// coarse 7 x 7 h = 1/896 1452 -> 530 us, 3D h = 1/32 1061 -> 367 us, against the all-FP64
// assembly of G(c) per evaluation with refined single-precision solves that this replaced.
#include <math.h>
#include <stdint.h>

#include "dense_lists.h"
#include "fmg_internal.h"

namespace fmg {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr double kSwitch = 1e-2;  // relative residual below which Newton takes over
constexpr int kMaxChord = 2;      // steps with an inverse of an earlier iterate, per inverse
constexpr int kMaxN = kDenseMaxNh + 1;
constexpr int kSide = 16;         // the sweep's threads: kSide x kSide
constexpr int kMaxTile = 6;       // at most kMaxTile x kMaxTile elements each (n <= 96)

// Capacities of a CTA's shared arrays per dimension (vertices of a simplex), covering every
// coarse mesh that dense_smem_bytes accepts (2D: 9 cells per side, 3D: 4).
template <int NV>
struct Cap {
  static constexpr int nh = NV == 3 ? 64 : 27, pat = NV == 3 ? 386 : 223,
                       tri = NV == 3 ? 162 : 384, trip = NV == 3 ? 484 : 343,
                       lists = NV == 3 ? 3872 : 3716;
};

// One float matrix row: a multiple of 4 words that is 4 times an odd number, so that the 8
// rows x 4 columns a warp reads at once fall into 32 banks.
__host__ __device__ inline int row_stride(int n) { return ((n + 3) / 4 | 1) * 4; }

template <int NV>
struct Smem {
  static constexpr int H = Cap<NV>::nh + 1, P = Cap<NV>::pat, T = Cap<NV>::tri;
  // nonzeros of the coarse blocks, sum_c w_c tau_abc per nonzero, and tau itself
  double K[P], M[P], B1[P], X[P], tau[Cap<NV>::trip];
  double h1[T], h2[T], h3[T];    // h_1, 2 h_2, 6 h_3 of each simplex's vertex values
  double w[H], w2[H], w3[H];     // c_H, its squares and doubled cubes; entry nh (boundary) is 0
  double Kc[H], Mc[H], Bc[H], Xc[H], S1[H], S2[H], S3[H], Q[H];
  double gA[H], gM[H], t1[H];
  double m64[H], r64[H];         // M c and the residual of the rescaled c
  double dots[kWarps], red[2][kWarps];
  double cu, f, zf3, lam, auu, buu, t0;
  float h1f[T], h2f[T];
  float r[kMaxN], m[kMaxN], y1[kMaxN], y2[kMaxN];
  alignas(16) float piv[2][2][kSide * kMaxTile];  // the sweep's pivot rows, double-buffered
  float rn;
  uint16_t tri[T * NV], lists[Cap<NV>::lists];
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 1 / d by Newton's iteration from the hardware's approximate reciprocal (about 2^-20 relative
// error; two steps reach FP64 rounding).
__device__ __forceinline__ double recip(double d) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  y = fma(y, fma(-d, y, 1.0), y);
  y = fma(y, fma(-d, y, 1.0), y);
  return y;
}

// Views of the staged lists (dense_lists.h)
struct Lists {
  const uint16_t *row, *pair, *simptr, *sim, *x3ptr, *x3;
};
__device__ __forceinline__ Lists lists_of(const uint16_t* base, const DenseLists& d, int nh) {
  return Lists{base, base + d.pair(nh), base + d.simptr(nh), base + d.sim(nh),
               base + d.x3ptr(nh), base + d.x3(nh)};
}

// Sums at the iterate (w, cu): X, h_q per simplex; per row K0_HH w, M_HH w, B1 w, X w, the
// sums S_q of h_q over the row's simplices and Q = 6 sum_T h_3(w.., w_a); and the dot
// products with w: dots = [K0 w, Q, gA (level 1: sum w), gM, X w, B1 w, t1, M w].
template <int NV>
__device__ void sums(const DenseProblem& p, Smem<NV>& s) {
  const int tid = threadIdx.x, nh = p.nh, npat = p.dims.npat;
  const Lists li = lists_of(s.lists, p.dims, nh);
  const int nx = p.aug ? npat : 0;
  for (int e = tid; e < nx + p.ntri; e += kThreads) {
    if (e < nx) {
      double x = 0.0;
      for (int k = li.x3ptr[e]; k < li.x3ptr[e + 1]; ++k) {
        const int c = li.x3[k];
        x = fma(s.w[c & 63], s.tau[c >> 6], x);
      }
      s.X[e] = x;
    } else {
      const int t = e - nx;
      const uint16_t* v = s.tri + t * NV;
      double p1 = s.w[v[0]] + s.w[v[1]], p2 = s.w2[v[0]] + s.w2[v[1]],
             p3 = s.w3[v[0]] + s.w3[v[1]];
#pragma unroll
      for (int q = 2; q < NV; ++q) {
        p1 += s.w[v[q]];
        p2 += s.w2[v[q]];
        p3 += s.w3[v[q]];  // the doubled cubes: 2 p_3
      }
      const double q1 = p1 * p1, h2 = q1 + p2;        // 2 h_2 = p_1^2 + p_2
      s.h1[t] = p1;
      s.h2[t] = h2;
      s.h3[t] = fma(p1, fma(3.0, p2, q1), p3);        // 6 h_3 = p_1^3 + 3 p_1 p_2 + 2 p_3
      s.h1f[t] = (float)p1;
      s.h2f[t] = (float)h2;
    }
  }
  __syncthreads();
  // seven row sums: one (sum, row) pair per thread
  const int lg = nh <= 32 ? 5 : 6, kinds = p.aug ? 7 : 5;
  for (int q = tid; q < kinds << lg; q += kThreads) {
    const int kind = q >> lg, a = q & ((1 << lg) - 1);
    if (a >= nh) continue;
    const int e0 = li.row[a];
    double v = 0.0;
    if (kind >= 2 && kind < 5) {
      const double* h = kind == 2 ? s.h1 : kind == 3 ? s.h2 : s.h3;
      for (int k = li.simptr[e0]; k < li.simptr[e0 + 1]; ++k) v += h[li.sim[k]];
      (kind == 2 ? s.S1 : kind == 3 ? s.S2 : s.S3)[a] = v;
    } else {
      const double* m = kind == 0 ? s.K : kind == 1 ? s.M : kind == 5 ? s.B1 : s.X;
      for (int e = e0; e < li.row[a + 1]; ++e) v = fma(m[e], s.w[li.pair[e] & 255], v);
      (kind == 0 ? s.Kc : kind == 1 ? s.Mc : kind == 5 ? s.Bc : s.Xc)[a] = v;
    }
  }
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31;
  const bool used = p.aug || warp < 3 || warp == 7;
  double d = 0.0;
  if (used) {
    const double* y = warp == 0 ? s.Kc : warp == 2 ? s.gA : warp == 3 ? s.gM : warp == 4 ? s.Xc
                    : warp == 5 ? s.Bc : warp == 6 ? s.t1 : s.Mc;
    for (int a = lane; a < nh; a += 32) {
      const double w = s.w[a];
      double v;
      if (warp == 1) {
        const double cnt = (double)(li.simptr[li.row[a] + 1] - li.simptr[li.row[a]]);
        // 6 sum_T [h_3 + w h_2 + w^2 h_1 + w^3] = S3 + w (3 S2 + 6 w (S1 + cnt w))
        v = fma(w, fma(6.0 * w, fma(cnt, w, s.S1[a]), 3.0 * s.S2[a]), s.S3[a]);
        s.Q[a] = v;
      } else {
        v = warp == 2 && !p.aug ? 1.0 : y[a];
      }
      d = fma(v, w, d);
    }
    d = warp_sum(d);
  }
  if (lane == 0) s.dots[warp] = d;
  __syncthreads();
}

// The residual at the iterate c = (w, cu), which it rescales to c^T M c = 1 with the sign of
// the ground state: lambda, the relative residual s.rn, and in single precision the residual
// r and M c.  Leaves s.f, the factor that was applied, for the sums that refer to the old c.
template <int NV>
__device__ void evaluate(const DenseProblem& p, Smem<NV>& s, double zeta) {
  sums<NV>(p, s);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nh = p.nh, n = nh + p.aug;
  constexpr int kRowWarps = (kMaxN + 31) / 32;
  if (warp < kRowWarps) {
    // polynomials in c_u, one per lane: c^T K0 c, c^T M c, the load's u~ entry N_u, c^T N,
    // (K0 c)_u and (M c)_u
    const double cu = p.aug ? s.cu : 0.0;
    const double d2 = p.aug ? s.dots[2] : 0.0, d3 = s.dots[3], d4 = s.dots[4], d5 = s.dots[5],
                 d6 = s.dots[6], qo = 0.5 * p.quart_off;
    double k0 = 0.0, k1 = 0.0, k2 = 0.0, k3 = 0.0, k4 = 0.0, m1 = 1.0, m2 = 1.0, m3 = 1.0;
    switch (lane) {
      case 0: k0 = s.dots[0]; k1 = d2; m1 = 2.0; k2 = s.auu; break;
      case 1: k0 = s.dots[7]; k1 = d3; m1 = 2.0; k2 = s.buu; break;
      case 2: k0 = d4; k1 = d5; m1 = 3.0; k2 = d6; m2 = 3.0; k3 = s.t0; break;
      case 3: k0 = qo * s.dots[1]; k1 = d4; m1 = 4.0; k2 = d5; m2 = 6.0; k3 = d6; m3 = 4.0;
              k4 = s.t0; break;
      case 4: k0 = d2; k1 = s.auu; break;
      case 5: k0 = d3; k1 = s.buu; break;
    }
    const double v = fma(cu, fma(cu, fma(cu, fma(cu, k4, m3 * k3), m2 * k2), m1 * k1), k0);
    const double cKc = __shfl_sync(0xffffffffu, v, 0), cMc = __shfl_sync(0xffffffffu, v, 1),
                 Nu = __shfl_sync(0xffffffffu, v, 2), cN = __shfl_sync(0xffffffffu, v, 3),
                 Ku = __shfl_sync(0xffffffffu, v, 4), Mu = __shfl_sync(0xffffffffu, v, 5);
    const double dm = cMc - 1.0;
    double f;
    if (fabs(dm) <= 1e-3)  // (1 + dm)^{-1/2}, the next term below 3e-16
      f = fma(dm, fma(dm, fma(dm, fma(dm, 0.2734375, -0.3125), 0.375), -0.5), 1.0);
    else
      f = 1.0 / sqrt(cMc);
    if ((p.aug ? cu : s.dots[2]) < 0.0) f = -f;
    const double f2 = f * f, zf2 = zeta * f2, zf3 = zf2 * f;
    const double lam = f2 * fma(zf2, cN, cKc);
    const int a = tid;
    double rr = 0.0, mm = 0.0;
    if (a < n) {
      double k, m, nl;
      if (a < nh) {
        k = s.Kc[a];
        m = s.Mc[a];
        nl = qo * s.Q[a];
        if (p.aug) {
          k = fma(cu, s.gA[a], k);
          m = fma(cu, s.gM[a], m);
          nl = fma(cu, fma(3.0, s.Xc[a], cu * fma(3.0, s.Bc[a], cu * s.t1[a])), nl);
        }
        s.w[a] *= f;
      } else {
        k = Ku;
        m = Mu;
        nl = Nu;
      }
      m *= f;
      const double r = fma(-lam, m, fma(zf3, nl, f * k));
      s.m64[a] = m;
      s.r64[a] = r;
      s.m[a] = (float)m;
      s.r[a] = (float)r;
      rr = r * r;
      mm = m * m;
    }
    rr = warp_sum(rr);
    mm = warp_sum(mm);
    if (lane == 0) {
      s.red[0][warp] = rr;
      s.red[1][warp] = mm;
    }
    if (tid == 0) {
      s.f = f;
      s.zf3 = zf3;
      s.lam = lam;
    }
  }
  __syncthreads();
  if (tid == 0) {
    double rr = 0.0, mm = 0.0;
    for (int q = 0; q < kRowWarps; ++q) {
      rr += s.red[0][q];
      mm += s.red[1][q];
    }
    const double den = s.lam * s.lam * mm;
    s.red[0][0] = rr;
    s.red[1][0] = den;
    s.rn = sqrtf((float)(rr * recip(den)));
    if (p.aug) s.cu *= s.f;
  }
  __syncthreads();
}

// G(c)_ab of nonzero e = (a, b) at c = f (w_old, cu_old), from the sums of `sums` at the old
// c and the rescaled w, in T (float: the Jacobian; double: the assembled system, and the
// Jacobian of the fallback): sum_T int_T w_H^2 mu_a mu_b + 2 c_u X_ab + c_u^2 B1_ab, with
//   int_T w^2 mu_a mu_b = |T| 2 d! / (d + 4)! h_2(w_1 .. w_nv, w_a, w_b)  (twice for a = b).
template <int NV, typename T>
__device__ __forceinline__ T coarse_G(const DenseProblem& p, const Smem<NV>& s, const Lists& li,
                                      int e, T f, T cu) {
  const int a = li.pair[e] >> 8, b = li.pair[e] & 255;
  const int k0 = li.simptr[e], k1 = li.simptr[e + 1];
  const T cnt = (T)(k1 - k0), wa = (T)s.w[a], wb = (T)s.w[b];
  T g;
  if (a == b) {
    const T s1 = f * (T)s.S1[a], s2 = f * f * (T)s.S2[a];
    g = (T)p.quart_off * (s2 + wa * ((T)4 * s1 + (T)6 * cnt * wa));
  } else {
    T s1 = 0, s2 = 0;
    for (int k = k0; k < k1; ++k) {
      const int t = li.sim[k];
      if constexpr (sizeof(T) == 4) {
        s1 += s.h1f[t];
        s2 += s.h2f[t];
      } else {
        s1 += s.h1[t];
        s2 += s.h2[t];
      }
    }
    const T ws = wa + wb;
    g = (T)(0.5 * p.quart_off) *
        (f * f * s2 + (T)2 * (ws * f * s1 + cnt * (ws * ws - wa * wb)));
  }
  if (p.aug) g += cu * ((T)2 * f * (T)s.X[e] + cu * (T)s.B1[e]);
  return g;
}

// G(c)_au, a < nh, and G(c)_uu (a = nh), as above
template <int NV, typename T>
__device__ __forceinline__ T border_G(const Smem<NV>& s, int a, int nh, T f, T cu) {
  if (a < nh)
    return f * f * (T)s.Xc[a] + cu * ((T)2 * f * (T)s.Bc[a] + cu * (T)s.t1[a]);
  return f * f * (T)s.dots[5] + cu * ((T)2 * f * (T)s.dots[6] + cu * (T)s.t0);
}

// J += K0 - lam M + gz G at the current iterate, on the structural nonzeros (the others stay
// zero), row stride ns
template <int NV, typename T>
__device__ void jacobian(const DenseProblem& p, const Smem<NV>& s, T* J, int ns, double lam,
                         T gz) {
  const int nh = p.nh;
  const Lists li = lists_of(s.lists, p.dims, nh);
  const T f = (T)s.f, cu = p.aug ? (T)s.cu : (T)0;
  for (int e = threadIdx.x; e < p.dims.npat; e += kThreads) {
    const int a = li.pair[e] >> 8, b = li.pair[e] & 255;
    J[a * ns + b] = (T)fma(-lam, s.M[e], s.K[e]) + gz * coarse_G<NV, T>(p, s, li, e, f, cu);
  }
  if (p.aug)
    for (int a = kThreads - 1 - threadIdx.x; a <= nh; a += kThreads) {
      const double k = a < nh ? s.gA[a] : s.auu, m = a < nh ? s.gM[a] : s.buu;
      const T v = (T)fma(-lam, m, k) + gz * border_G<NV, T>(s, a, nh, f, cu);
      J[a * ns + nh] = v;
      J[nh * ns + a] = v;
    }
  __syncthreads();
}

// -A^{-1} (into Ainv, row stride ns) of the SPD matrix A = J + tau m m^T (n <= 16 TS) in
// single precision by the sweep operator (Gauss-Jordan elimination without pivoting, stable
// for SPD matrices).  Sweeping a set P of indices maps M to M' with H = (M_PP)^{-1}:
//     M'_PP = -H,  M'_Pj = H M_Pj,  M'_iP = M_iP H,  M'_ij = M_ij - M_iP H M_Pj  (i, j not in P),
// and after sweeping every index the matrix is -A^{-1}.  All four cases are one update
// M_ij - F_i R_j once the pivot rows and columns of M are set to zero, with F_i = M_iP H
// (pivot row: -H_i) and R_j = M_Pj (pivot column: -e_j), so no lane takes a branch of its own.
// The indices go in pairs, one barrier per pair; 16 x 16 threads hold TS x TS elements each in
// registers, and the owners of the next two pivot rows publish them to s.piv.  M stays
// symmetric, so F is read from the pivot rows too.  A pair's chain (publish, barrier, read,
// 2 x 2 inverse, update) is about 190 cycles: 50 x 50 takes 25 pairs.  Returns false at a
// non-positive pivot (all threads read the same pivots, so all return together).
template <int TS>
__device__ __forceinline__ bool sweep_tiles(const float* J, float* Ainv, int ns, float tau,
                                            const float* m, float (*piv)[2][kSide * kMaxTile],
                                            int n) {
  const int ti = threadIdx.x / kSide, tj = threadIdx.x % kSide, i0 = ti * TS, j0 = tj * TS;
  float v[TS][TS];
#pragma unroll
  for (int r = 0; r < TS; ++r)
#pragma unroll
    for (int c = 0; c < TS; ++c) {
      const int i = i0 + r, j = j0 + c;
      v[r][c] = i < n && j < n ? J[i * ns + j] : (i == j ? 1.0f : 0.0f);
      if (tau != 0.0f && i < n && j < n) v[r][c] = fmaf(tau * m[i], m[j], v[r][c]);
    }
  if (ti == 0) {
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < TS; c += 2)
        *reinterpret_cast<float2*>(&piv[0][r][j0 + c]) = make_float2(v[r][c], v[r][c + 1]);
  }
  __syncthreads();
  int buf = 0;
  for (int kt = 0; kt * TS < n; ++kt) {
#pragma unroll
    for (int q = 0; q < TS; q += 2) {
      const int k = kt * TS + q;
      if (k >= n) break;
      const float* p0 = piv[buf][0];
      const float* p1 = piv[buf][1];
      const float a = p0[k], b = p0[k + 1], d = p1[k + 1];
      const float det = fmaf(a, d, -b * b);
      if (!(a > 0.0f) || !(det > 0.0f)) return false;
      const float inv = __fdividef(1.0f, det);
      const float h00 = d * inv, h01 = -b * inv, h11 = a * inv;
      float f0[TS], f1[TS], r0[TS], r1[TS];
#pragma unroll
      for (int r = 0; r < TS; r += 2) {
        const float2 x = *reinterpret_cast<const float2*>(&p0[i0 + r]);
        const float2 y = *reinterpret_cast<const float2*>(&p1[i0 + r]);
        f0[r] = fmaf(x.x, h00, y.x * h01);
        f1[r] = fmaf(x.x, h01, y.x * h11);
        f0[r + 1] = fmaf(x.y, h00, y.y * h01);
        f1[r + 1] = fmaf(x.y, h01, y.y * h11);
        const float2 z = *reinterpret_cast<const float2*>(&p0[j0 + r]);
        const float2 w = *reinterpret_cast<const float2*>(&p1[j0 + r]);
        r0[r] = z.x;
        r0[r + 1] = z.y;
        r1[r] = w.x;
        r1[r + 1] = w.y;
      }
      const bool prow = ti == kt, pcol = tj == kt;
      if (prow) {
        f0[q] = -h00;
        f1[q] = -h01;
        f0[q + 1] = -h01;
        f1[q + 1] = -h11;
      }
      if (pcol) {
        r0[q] = -1.0f;
        r1[q] = 0.0f;
        r0[q + 1] = 0.0f;
        r1[q + 1] = -1.0f;
      }
#pragma unroll
      for (int r = 0; r < TS; ++r)
#pragma unroll
        for (int c = 0; c < TS; ++c) {
          const bool zr = r == q || r == q + 1, zc = c == q || c == q + 1;
          float x = v[r][c];
          if (zr) x = prow ? 0.0f : x;
          if (zc) x = pcol ? 0.0f : x;
          v[r][c] = fmaf(-f0[r], r0[c], fmaf(-f1[r], r1[c], x));
        }
      // publish the next pair of pivot rows: of this tile row, or of the next one
      if (q + 2 < TS ? prow : ti == kt + 1) {
        constexpr int wrap = TS;
        const int nr = (q + 2) % wrap;
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int c = 0; c < TS; c += 2)
            *reinterpret_cast<float2*>(&piv[buf ^ 1][r][j0 + c]) =
                make_float2(v[nr + r][c], v[nr + r][c + 1]);
      }
      buf ^= 1;
      __syncthreads();
    }
  }
#pragma unroll
  for (int r = 0; r < TS; ++r)
#pragma unroll
    for (int c = 0; c < TS; ++c)
      if (i0 + r < n && j0 + c < n) Ainv[(i0 + r) * ns + j0 + c] = v[r][c];
  __syncthreads();
  return true;
}

__device__ __noinline__ bool sweep_inverse(const float* J, float* Ainv, int ns, float tau,
                                           const float* m, float (*piv)[2][kSide * kMaxTile],
                                           int n) {
  if (n <= 2 * kSide) return sweep_tiles<2>(J, Ainv, ns, tau, m, piv, n);
  if (n <= 4 * kSide) return sweep_tiles<4>(J, Ainv, ns, tau, m, piv, n);
  return sweep_tiles<kMaxTile>(J, Ainv, ns, tau, m, piv, n);
}

// y = A^{-1} x for one or two vectors, Ainv = -A^{-1} in single precision: 4 threads per row
__device__ __forceinline__ void apply_inverse(const float* Ainv, int ns, const float* x1,
                                              float* y1, const float* x2, float* y2, int n) {
  const int part = threadIdx.x & 3;
  for (int row0 = 0; row0 < n; row0 += kThreads / 4) {
    const int row = row0 + (threadIdx.x >> 2);
    float a = 0.0f, b = 0.0f;
    if (row < n)
      for (int j = part; j < n; j += 4) {
        const float v = Ainv[row * ns + j];
        a = fmaf(v, x1[j], a);
        if (x2) b = fmaf(v, x2[j], b);
      }
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    b += __shfl_xor_sync(0xffffffffu, b, 1);
    b += __shfl_xor_sync(0xffffffffu, b, 2);
    if (part == 0 && row < n) {
      y1[row] = -a;
      if (x2) y2[row] = -b;
    }
  }
  __syncthreads();
}

// the new iterate: entry a of c (a < n), with the squares and doubled cubes the sums read
template <int NV>
__device__ __forceinline__ void set_entry(const DenseProblem& p, Smem<NV>& s, int a, double c) {
  if (a < p.nh) {
    const double q = c * c;
    s.w[a] = c;
    s.w2[a] = q;
    s.w3[a] = 2.0 * (q * c);
  } else {
    s.cu = c;
  }
}

// c += dc = -y1 + dl y2 of the bordered Newton system; returns dl
template <int NV>
__device__ float newton_update(const DenseProblem& p, Smem<NV>& s) {
  const int n = p.nh + p.aug, lane = threadIdx.x & 31;
  float p1 = 0.0f, p2 = 0.0f;
  for (int a = lane; a < n; a += 32) {
    p1 = fmaf(s.m[a], s.y1[a], p1);
    p2 = fmaf(s.m[a], s.y2[a], p2);
  }
  const float dl = warp_sum(p1) / warp_sum(p2);
  for (int a = threadIdx.x; a < n; a += kThreads)
    set_entry(p, s, a, (a < p.nh ? s.w[a] : s.cu) + (double)fmaf(dl, s.y2[a], -s.y1[a]));
  __syncthreads();
  return dl;
}

// In-place symmetric elimination A = L D L^T (no pivoting) on the lower triangle: after it,
// A_kk = D_k and A_ik = L_ik D_k (i > k); dinv[k] = 1 / D_k.  At step k every thread updates
// its elements (i >= j > k) of the trailing triangle, and the thread that updates the next
// pivot also forms its reciprocal, so each step needs one barrier.  Returns false at a
// non-positive pivot (every thread reads the same pivot, so all return together).
__device__ __noinline__ bool ldlt(double* A, int n, double* dinv) {
  if (threadIdx.x == 0) dinv[0] = A[0] > 0.0 ? recip(A[0]) : 0.0;
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    const double d = A[k * n + k];
    if (!(d > 0.0)) return false;
    const double inv = dinv[k];
    const int m = n - k - 1;
    const int tri = m * (m + 1) / 2;
    for (int e = threadIdx.x; e < tri; e += kThreads) {
      // e -> (r, c), c <= r, rows of the trailing lower triangle in order
      int r = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
      while ((r + 1) * (r + 2) / 2 <= e) ++r;
      while (r * (r + 1) / 2 > e) --r;
      const int c = e - r * (r + 1) / 2;
      const int i = k + 1 + r, j = k + 1 + c;
      const double v = fma(-(A[i * n + k] * inv), A[j * n + k], A[i * n + j]);
      A[i * n + j] = v;
      if (e == 0) dinv[k + 1] = v > 0.0 ? recip(v) : 0.0;  // (k+1, k+1): the next pivot
    }
    __syncthreads();
  }
  return true;
}

// Solve (L D L^T) x = b for x held in `x` (b on entry), by one warp, column by column: once
// an entry is final, the lanes update the remaining ones (only warp-level synchronisation).
// Reads the lower triangle written by ldlt.
__device__ __noinline__ void ldlt_solve_warp(const double* A, const double* dinv, int n,
                                             double* x) {
  const int lane = threadIdx.x & 31;
  for (int k = 0; k < n; ++k) {  // forward: w_k = z_k / D_k, z_i -= A_ik w_k (i > k)
    const double wk = x[k] * dinv[k];
    __syncwarp();
    if (lane == 0) x[k] = wk;
    for (int i = k + 1 + lane; i < n; i += 32) x[i] = fma(-A[i * n + k], wk, x[i]);
    __syncwarp();
  }
  for (int k = n - 1; k >= 0; --k) {  // backward: x_i -= (A_ki / D_i) x_k (i < k)
    const double xk = x[k];
    for (int i = lane; i < k; i += 32) x[i] = fma(-A[k * n + i] * dinv[i], xk, x[i]);
    __syncwarp();
  }
}

// The step's linear solves in FP64 (LDL^T) for a matrix whose single-precision elimination
// met a non-positive pivot: y1 = A^{-1} r, y2 = A^{-1} M c (Newton), or y1 = A^{-1} M c.  A64
// (n x n doubles) takes the space of both float matrices; the zeros of J are restored.
// noinline: keeps the rare path's registers and instructions out of the iteration.
template <int NV>
__device__ __noinline__ bool solve_fp64(const DenseProblem& p, Smem<NV>& s, double* A64,
                                        float* J, int ns, double lam, double gz, double tau,
                                        bool newton) {
  const int n = p.nh + p.aug;
  __syncthreads();
  for (int e = threadIdx.x; e < n * n; e += kThreads) A64[e] = 0.0;
  __syncthreads();
  jacobian<NV, double>(p, s, A64, n, lam, gz);
  for (int e = threadIdx.x; e < n * n; e += kThreads) {
    const int a = e / n, b = e - a * n;
    A64[e] = fma(tau * s.m64[a], s.m64[b], A64[e]);
  }
  __syncthreads();
  double* dinv = s.S3;  // free until the next evaluation (and S1, S2 once A64 is formed)
  const bool ok = ldlt(A64, n, dinv);
  if (ok) {
    double *x1 = s.S1, *x2 = s.S2;
    for (int a = threadIdx.x; a < n; a += kThreads) {
      x1[a] = newton ? s.r64[a] : s.m64[a];
      x2[a] = s.m64[a];
    }
    __syncthreads();
    if (threadIdx.x < 32) ldlt_solve_warp(A64, dinv, n, x1);
    else if (threadIdx.x < 64 && newton) ldlt_solve_warp(A64, dinv, n, x2);
    __syncthreads();
    for (int a = threadIdx.x; a < n; a += kThreads) {
      s.y1[a] = (float)x1[a];
      s.y2[a] = (float)x2[a];
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 2 * n * ns; e += kThreads) J[e] = 0.0f;
  __syncthreads();
  return ok;
}

// One CTA of 256 threads per problem, a batch of problems one CTA each (two resident per SM:
// at most 128 registers and half of the shared memory).  The iteration count is bounded by
// max_iter (chord steps, at most kMaxChord per inverse, are not counted: they replace the
// refinement of the Newton correction); hitting it sets status 1.
template <int NV>
__global__ void __launch_bounds__(kThreads, 2) k_dense_scf(const __grid_constant__ DenseProblem p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem<NV>& s = *reinterpret_cast<Smem<NV>*>(smem_raw);
  const int tid = threadIdx.x, nh = p.nh, n = nh + p.aug, ns = row_stride(n);
  // two n x ns float matrices (the Jacobian and its inverse), or one n x n FP64 matrix
  float* J = reinterpret_cast<float*>(smem_raw + (sizeof(Smem<NV>) + 15) / 16 * 16);
  float* Pinv = J + n * ns;
  const size_t ib = blockIdx.x;  // the instance, whose arrays lie at its slices
  const double *L1 = p.L1 + ib * nh * nh, *M1 = p.M1 + ib * nh * nh;
  const double zeta = p.params[ib].zeta;
  for (int e = tid; e < p.dims.tripptr(nh); e += kThreads) s.lists[e] = p.lists[e];
  for (int e = tid; e < p.ntri * NV; e += kThreads) {
    const int v = p.tri[e];
    s.tri[e] = (uint16_t)(v < 0 ? nh : v);
  }
  for (int e = tid; e < 2 * n * ns; e += kThreads) J[e] = 0.0f;
  if (tid < kWarps) s.dots[tid] = 0.0;
  if (tid <= nh) {
    double c = 0.0;
    if (p.c_init) c = tid < n ? p.c_init[ib * (nh + 1) + tid] : 0.0;
    else if (tid == nh) c = 1.0;
    if (tid == nh) {  // entry nh of w is the boundary value
      s.cu = p.aug ? c : 0.0;
      c = 0.0;
    }
    s.w[tid] = c;
    s.w2[tid] = c * c;
    s.w3[tid] = 2.0 * (c * c * c);
  }
  if (p.aug) {
    if (tid < nh) {
      s.gA[tid] = p.gA[ib * nh + tid];
      s.gM[tid] = p.gM[ib * nh + tid];
      s.t1[tid] = p.t1[ib * nh + tid];
    }
    const uint16_t* tp = p.lists + p.dims.tripptr(nh);
    const uint16_t* ti = p.lists + p.dims.trip(nh);
    const double* t3 = p.t3 + ib * p.ntri * p.nt3;
    for (int q = tid; q < p.dims.nq; q += kThreads) {
      double v = 0.0;
      for (int k = tp[q]; k < tp[q + 1]; ++k) v += t3[ti[k]];
      s.tau[q] = v;
    }
  }
  if (tid == 0) {
    s.auu = p.aug ? p.auu[ib] : 0.0;
    s.buu = p.aug ? p.buu[ib] : 0.0;
    s.t0 = p.aug ? p.t0[ib] : 0.0;
  }
  {
    const uint16_t* pr = p.lists + p.dims.pair(nh);
    for (int e = tid; e < p.dims.npat; e += kThreads) {
      const int k = (pr[e] >> 8) * nh + (pr[e] & 255);
      s.K[e] = L1[k];
      s.M[e] = M1[k];
      if (p.aug) s.B1[e] = p.B1[ib * nh * nh + k];
    }
  }
  __syncthreads();
  if (p.K_out) {  // assemble-only mode: K0, M and G(c_init) as given
    sums<NV>(p, s);
    const Lists li = lists_of(s.lists, p.dims, nh);
    for (int e = tid; e < n * n; e += kThreads) p.K_out[e] = p.M_out[e] = p.G_out[e] = 0.0;
    __syncthreads();
    for (int e = tid; e < p.dims.npat; e += kThreads) {
      const int k = (li.pair[e] >> 8) * n + (li.pair[e] & 255);
      p.K_out[k] = s.K[e];
      p.M_out[k] = s.M[e];
      p.G_out[k] = coarse_G<NV, double>(p, s, li, e, 1.0, s.cu);
    }
    if (p.aug)
      for (int a = tid; a <= nh; a += kThreads) {
        const int k = a * n + nh, l = nh * n + a;
        p.K_out[k] = p.K_out[l] = a < nh ? s.gA[a] : s.auu;
        p.M_out[k] = p.M_out[l] = a < nh ? s.gM[a] : s.buu;
        p.G_out[k] = p.G_out[l] = border_G<NV, double>(s, a, nh, 1.0, s.cu);
      }
    return;
  }

  int it = 0, status = 1, chords = kMaxChord;  // kMaxChord: no inverse to step with
  float last = 0.0f;                           // the residual before the latest Newton step
  double dlam = 0.0;
  for (;;) {
    evaluate<NV>(p, s, zeta);
    const float rn = s.rn;
    const bool converged = s.red[0][0] <= p.tol * p.tol * s.red[1][0];
    // A step with the inverse of an earlier iterate cuts the residual by about twice what the
    // latest step did (the Jacobian is off by the distance moved since, and by ~1e-6): it
    // replaces a new inverse where that reaches the tolerance.  On convergence the same step,
    // without another evaluation, takes c and lambda from the tolerance to rounding.
    const bool chord = chords < kMaxChord && rn < 0.05f * last &&
                       (converged || 4.0f * rn * rn <= last * (float)p.tol);
    if (chord) {
      ++chords;
      apply_inverse(Pinv, ns, s.r, s.y1, s.m, s.y2, n);
      const float dl = newton_update(p, s);
      last = rn;
      if (converged) {
        dlam = (double)dl;
        status = 0;
        break;
      }
      continue;
    }
    if (converged) {
      status = 0;
      break;
    }
    if (it >= p.max_iter) break;
    const double lam = s.lam;
    bool newton = rn <= (float)kSwitch, have = false;
    if (newton) {
      const double tau = fabs(lam);
      jacobian<NV, float>(p, s, J, ns, lam, (float)(3.0 * zeta));
      have = sweep_inverse(J, Pinv, ns, (float)tau, s.m, s.piv, n);
      if (have) {
        apply_inverse(Pinv, ns, s.r, s.y1, s.m, s.y2, n);
        chords = 0;
        last = rn;
      } else {
        chords = kMaxChord;
        newton = have = solve_fp64<NV>(p, s, reinterpret_cast<double*>(J), J, ns, lam,
                                       3.0 * zeta, tau, true);
      }
      if (newton) newton_update(p, s);
    }
    if (!newton) {
      // inverse-power step: c <- (K0 + zeta G)^{-1} M c
      chords = kMaxChord;
      jacobian<NV, float>(p, s, J, ns, 0.0, (float)zeta);
      if (sweep_inverse(J, Pinv, ns, 0.0f, s.m, s.piv, n))
        apply_inverse(Pinv, ns, s.m, s.y1, nullptr, nullptr, n);
      else if (!solve_fp64<NV>(p, s, reinterpret_cast<double*>(J), J, ns, 0.0, zeta, 0.0, false))
        break;
      for (int a = tid; a < n; a += kThreads) set_entry(p, s, a, (double)s.y1[a]);
      __syncthreads();
    }
    ++it;
  }
  for (int a = tid; a < n; a += kThreads) p.c_out[ib * (nh + 1) + a] = a < nh ? s.w[a] : s.cu;
  if (tid == 0) {
    p.lam_out[ib] = s.lam + dlam;
    p.iters_out[ib] = it;
    p.status_out[ib] = status;
  }
}

// L^{-1} by LDL^T in FP64, all columns at once (rows sequential, columns spread over the
// threads); false when L is not positive definite.  A, Y: n x n doubles, dinv: n.
__device__ __noinline__ bool inverse_fp64(const double* L, double* A, double* Y, double* dinv,
                                          int n) {
  __syncthreads();
  for (int e = threadIdx.x; e < n * n; e += kThreads) {
    A[e] = L[e];
    const int i = e / n, j = e - i * n;
    Y[e] = i == j ? 1.0 : 0.0;
  }
  __syncthreads();
  if (!ldlt(A, n, dinv)) return false;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // forward: rows of W with (C D) W = I: W_k = (Y_k - sum_{i<k} A_ki W_i) / D_k
  for (int k = 0; k < n; ++k) {
    const double inv = dinv[k];
    for (int j = threadIdx.x; j < n; j += kThreads) Y[k * n + j] *= inv;
    __syncthreads();
    for (int i = k + 1 + warp; i < n; i += kWarps) {
      const double l = A[i * n + k];
      for (int j = lane; j < n; j += 32) Y[i * n + j] = fma(-l, Y[k * n + j], Y[i * n + j]);
    }
    __syncthreads();
  }
  // backward: C^T X = W, X_i = W_i - sum_{k>i} (A_ki / D_i) X_k
  for (int k = n - 1; k >= 0; --k) {
    for (int i = warp; i < k; i += kWarps) {
      const double l = A[k * n + i] * dinv[i];
      for (int j = lane; j < n; j += 32) Y[i * n + j] = fma(-l, Y[k * n + j], Y[i * n + j]);
    }
    __syncthreads();
  }
  return true;
}

constexpr int kInverseRounds = 2;

// L^{-1} of the SPD level-1 operator, one CTA per instance: the single-precision inverse of
// the sweep operator (~1e-6), then X <- X + Y (I - L X) with Y that inverse: the residual in
// FP64 over the nonzeros of L (15 or 7 per row, so the FP64 work is n^2 x that, not n^3), the
// product in single precision on a residual that shrinks by ~1e6 a round; two rounds leave the
// rounding of I - L X.  An L whose single-precision elimination meets a non-positive pivot
// takes the FP64 LDL^T.
__global__ void __launch_bounds__(kThreads) k_spd_inverse(const double* __restrict__ L,
                                                          double* __restrict__ Linv, int n,
                                                          const uint16_t* __restrict__ lists,
                                                          DenseLists dims) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) float piv[2][2][kSide * kMaxTile];
  L += blockIdx.x * (size_t)n * n;  // instance blockIdx.x
  Linv += blockIdx.x * (size_t)n * n;
  const int ns = row_stride(n), tid = threadIdx.x;
  float* R = reinterpret_cast<float*>(smem_raw);
  float* Y = R + n * ns;  // -(single-precision inverse)
  double* X = reinterpret_cast<double*>(Y + n * ns);
  double* dinv = X + n * n;
  for (int e = tid; e < n * n; e += kThreads) R[(e / n) * ns + e % n] = (float)L[e];
  __syncthreads();
  if (!sweep_inverse(R, Y, ns, 0.0f, nullptr, piv, n)) {
    const bool ok = inverse_fp64(L, reinterpret_cast<double*>(R), X, dinv, n);
    for (int e = tid; e < n * n; e += kThreads) Linv[e] = ok ? X[e] : nan("");
    return;
  }
  for (int e = tid; e < n * n; e += kThreads) X[e] = -(double)Y[(e / n) * ns + e % n];
  const uint16_t* pair = lists + dims.pair(n);
  const int nq = (n + 3) / 4;
  for (int round = 0; round < kInverseRounds; ++round) {
    __syncthreads();
    for (int e = tid; e < n * n; e += kThreads) {
      const int i = e / n, j = e - i * n;
      double r = i == j ? 1.0 : 0.0;
      for (int q = lists[i]; q < lists[i + 1]; ++q) {
        const int k = pair[q] & 255;
        r = fma(-L[i * n + k], X[k * n + j], r);
      }
      R[i * ns + j] = (float)r;
    }
    __syncthreads();
    for (int e = tid; e < n * nq; e += kThreads) {
      const int i = e / nq, j = 4 * (e - i * nq);
      float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      for (int k = 0; k < n; ++k) {
        const float y = Y[i * ns + k];
        const float4 r = *reinterpret_cast<const float4*>(R + k * ns + j);
        a = make_float4(fmaf(y, r.x, a.x), fmaf(y, r.y, a.y), fmaf(y, r.z, a.z),
                        fmaf(y, r.w, a.w));
      }
      const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (j + c < n) X[i * n + j + c] -= (double)av[c];
    }
  }
  __syncthreads();
  for (int e = tid; e < n * n; e += kThreads) Linv[e] = X[e];
}

// y = Linv x on the interior of level 1: one CTA, x gathered to shared memory, one warp per
// row with coalesced loads and a shuffle reduction.
__device__ __forceinline__ size_t level1_index(int dim, int m, int pitch, int q) {
  if (dim == 2) return (size_t)(1 + q / m) * pitch + 1 + q % m;
  return ((size_t)(1 + q / (m * m)) * (m + 2) + 1 + (q / m) % m) * pitch + 1 + q % m;
}

__global__ void __launch_bounds__(kThreads) k_coarse_matvec(int dim, int n, int pitch, size_t st,
                                                            const double* __restrict__ Linv,
                                                            const double* __restrict__ x,
                                                            double* __restrict__ y) {
  __shared__ double xs[1024];
  const int m = n - 1, nh = dim == 2 ? m * m : m * m * m;
  Linv += blockIdx.x * (size_t)nh * nh;  // instance blockIdx.x
  x += blockIdx.x * st;
  y += blockIdx.x * st;
  for (int q = threadIdx.x; q < nh; q += kThreads) xs[q] = x[level1_index(dim, m, pitch, q)];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int p = warp; p < nh; p += kWarps) {
    const double* row = Linv + (size_t)p * nh;
    double s = 0.0;
    for (int q = lane; q < nh; q += 32) s = fma(row[q], xs[q], s);
    s = warp_sum(s);
    if (lane == 0) y[level1_index(dim, m, pitch, p)] = s;
  }
}

}  // namespace

// The acceptance rule of coarse meshes: the shared memory of the all-FP64 form of the solve,
// which keeps K0, M, G and a work matrix dense.  The kernels above need less (Cap holds every
// mesh the rule accepts).
size_t dense_smem_bytes(int n, int ntri, int nvert, int aug) {
  const int L = nvert + 1, nh = n - aug;
  const size_t nt3 = nvert == 3 ? 10 : 20;
  const size_t maxadj = nvert == 3 ? 6 : 24;
  const bool loc_in_A = (size_t)ntri * L * L <= (size_t)n * n;
  const size_t loc = loc_in_A ? 0 : (size_t)ntri * L * L;
  return sizeof(double) * ((size_t)4 * n * n + loc + 8 * (size_t)n + 4 * kThreads + nh +
                           (aug ? (size_t)ntri * nt3 : 0) + ((size_t)ntri * nvert + 1) / 2 +
                           ((size_t)nh * maxadj + 1) / 2);
}

namespace {
size_t scf_smem(int n, int nvert) {
  const size_t s = nvert == 3 ? sizeof(Smem<3>) : sizeof(Smem<4>);
  return (s + 15) / 16 * 16 + (size_t)2 * n * row_stride(n) * sizeof(float);
}
size_t inverse_smem(int n) {
  return (size_t)2 * n * row_stride(n) * sizeof(float) + sizeof(double) * ((size_t)n * n + n);
}
}  // namespace

void dense_scf(const DenseProblem& p, int nb, cudaStream_t s) {
  const size_t smem = scf_smem(p.nh + p.aug, p.nvert);
  if (p.nvert == 3) k_dense_scf<3><<<nb, kThreads, smem, s>>>(p);
  else k_dense_scf<4><<<nb, kThreads, smem, s>>>(p);
}

// The attributes are per function, shared by every handle in the process, so they are always
// set to what the largest accepted mesh needs (never to one caller's smaller need).
cudaError_t dense_prepare(size_t need) {
  if (need > kDenseSmemLimit) return cudaErrorInvalidValue;
  const struct { const void* f; size_t smem; } k[] = {
      {(const void*)k_dense_scf<3>, scf_smem(Cap<3>::nh + 1, 3)},
      {(const void*)k_dense_scf<4>, scf_smem(Cap<4>::nh + 1, 4)},
      {(const void*)k_spd_inverse, inverse_smem(kDenseMaxNh)}};
  for (const auto& q : k) {
    cudaError_t e = cudaFuncSetAttribute(q.f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)q.smem);
    // all of the unified L1 as shared memory, so that instances of a batch share an SM
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(q.f, cudaFuncAttributePreferredSharedMemoryCarveout,
                               (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

void dense_spd_inverse(const double* L, double* Linv, int n, const uint16_t* lists,
                       const DenseLists& dims, int nb, cudaStream_t s) {
  k_spd_inverse<<<nb, kThreads, inverse_smem(n), s>>>(L, Linv, n, lists, dims);
}

void coarse_matvec(const Grid& g, const double* Linv, const double* x, double* y,
                   cudaStream_t s) {
  k_coarse_matvec<<<g.nb, kThreads, 0, s>>>(g.dim, g.n, g.pitch, g.stride, Linv, x, y);
}

}  // namespace fmg
