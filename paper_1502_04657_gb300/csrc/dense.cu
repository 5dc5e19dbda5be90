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
//   - c is rescaled only when c^T M c is off 1 by more than 1e-3 (the start, an inverse-power
//     step), by a factor f applied to the sums: every term is homogeneous in c.  Otherwise the
//     Newton system carries the constraint's defect, (M c)^T dc = -(c^T M c - 1) / 2.
//   - The small scalar chains are Horner evaluations in c_u, one chain per lane.
//   - The Jacobian A' (and K0 + zeta G) is assembled and inverted in single precision, whose
//     pipes issue 64 times faster; what the ~1e-6 relative error of a step leaves is removed
//     by further steps with the same inverse against the FP64 residual (a chord step costs one
//     evaluation), so c and lambda are exact to the FP64 residual as before.
// Measured (ncu, every dense launch of one solve summed): 2D h = 1/64 983 -> 262 us, 2D
// coarse 7 x 7 h = 1/896 1452 -> 386 us, 3D h = 1/32 1061 -> 291 us, against the all-FP64
// assembly of G(c) per evaluation with refined single-precision solves that this replaced.
#include <math.h>
#include <stdint.h>

#include "dense_lists.h"
#include "dfloat.cuh"
#include "fmg_internal.h"

namespace fmg {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
// Relative residual below which Newton takes over (where its matrix is positive definite).  Over
// coarse meshes of 3 to 9 (2D) and 3, 4 (3D) cells, zeta 1 to 5000 and traps 1 to 1000, 0.1
// needed 3 to 22 steps where 1e-2 needed 3 to 47, never more, for the same ground state; 0.3
// sometimes needed more (33 against 22).  Beyond (zeta to 1e5, large negative or positive w_const,
// under-resolved meshes) Newton from so far can wander to the cap: the problem then starts again
// with 1e-2.
constexpr float kSwitch = 0.1f, kSwitchAgain = 1e-2f;
constexpr int kMaxChord = 2;      // steps with an inverse of an earlier iterate, per inverse
constexpr int kMaxN = kDenseMaxNh + 1;
constexpr int kTile = 4;          // elements per side of a thread's tile in the FP32 sweep
constexpr int kMaxSweep = 88;     // largest matrix the sweep takes: 22 x 23 / 2 tiles

// Capacities of a CTA's shared arrays per dimension (vertices of a simplex), covering every
// coarse mesh that dense_smem_bytes accepts (2D: 9 cells per side, 3D: 4).
template <int NV>
struct Cap {
  static constexpr int nh = NV == 3 ? 64 : 27, pat = NV == 3 ? 386 : 223,
                       tri = NV == 3 ? 162 : 384, trip = NV == 3 ? 484 : 343,
                       lists = NV == 3 ? 5488 : 5984;  // multiples of 8 (16-byte copies)
};

// One float matrix row: a multiple of 4 words that is 4 times an odd number, so that the 8
// rows x 4 columns a warp reads at once fall into 32 banks.
__host__ __device__ inline int row_stride(int n) { return ((n + 3) / 4 | 1) * 4; }

template <int NV>
struct Smem {
  static constexpr int H = Cap<NV>::nh + 1, P = Cap<NV>::pat, T = Cap<NV>::tri;
  // nonzeros of the coarse blocks, sum_c w_c tau_abc per nonzero, and tau itself
  alignas(16) uint16_t lists[Cap<NV>::lists];
  double K[P], M[P], B1[P], X[P], tau[Cap<NV>::trip];
  double h1[T], h2[T], h3[T];    // h_1, 2 h_2, 6 h_3 of each simplex's vertex values
  double w[H], w2[H], w3[H];     // c_H, its squares and doubled cubes; entry nh (boundary) is 0
  double Kc[H], Mc[H], Bc[H], Xc[H], S1[H], S2[H], S3[H], Q[H];
  double gA[H], gM[H], t1[H];
  double m64[H], r64[H];         // M c and the residual of the rescaled c
  double cnt[H];                 // simplices around each coarse node
  double dots[9];
  double cu, f, g, lam, auu, buu, t0;
  float h1f[T], h2f[T], wf[H];   // single precision, at the rescaled c (Jacobian)
  float r[kMaxN], m[kMaxN], y1[kMaxN], y2[kMaxN];
  alignas(16) float piv[2][kTile][kMaxSweep];  // the sweep's pivot rows, double-buffered
  float red[2][kWarps];
  int pivots_ok;
  uint16_t tri[T * NV];
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Both sums by one butterfly: a's in the lower half of the warp, b's in the upper (five
// additions instead of ten; order fixed).
template <typename T>
__device__ __forceinline__ T half_sums(T a, T b) {
  const bool upper = threadIdx.x & 16;
  T v = (upper ? b : a) + __shfl_xor_sync(0xffffffffu, upper ? a : b, 16);
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The exponent of v, and 2^e as a float (clamped to its range)
__device__ __forceinline__ int exponent_of(double v) {
  return ((__double2hiint(v) >> 20) & 0x7ff) - 1023;
}
__device__ __forceinline__ float pow2f(int e) {
  return __int_as_float(min(max(e + 127, 1), 254) << 23);
}

// Views of the staged lists (dense_lists.h)
struct Lists {
  const uint16_t *row, *pair, *simptr, *sim, *x3ptr, *x3;
};
__device__ __forceinline__ Lists lists_of(const uint16_t* base, const DenseLists& d, int nh) {
  return Lists{base, base + d.pair(nh), base + d.simptr(nh), base + d.sim(nh),
               base + d.x3ptr(nh), base + d.x3(nh)};
}

// Sums at the iterate c = (w, cu): X, h_q per simplex; per row (K0 c)_a, (M c)_a, B1 w, X w, the
// sums S_q of h_q over the row's simplices and Q = 6 sum_T h_3(w.., w_a); and the dot
// products with w: dots = [K0 c, gA (level 1: sum w), M c, gM, X w, B1 w, t1, and Q over the
// rows of warps 0 and 1].  zero: w = 0 (every augmented solve starts so).
template <int NV>
__device__ __forceinline__ void sums(const DenseProblem& p, Smem<NV>& s, bool zero) {
  const int tid = threadIdx.x, nh = p.nh, npat = p.dims.npat;
  const Lists li = lists_of(s.lists, p.dims, nh);
  const int nx = p.aug ? npat : 0;
  const int lg = nh <= 32 ? 5 : 6, kinds = p.aug ? 7 : 5;
  for (int e = tid; e < nx + p.ntri; e += kThreads) {
    if (e < nx) {
      double x = 0.0;
      if (!zero) {
        const int k1 = li.x3ptr[e + 1];
#pragma unroll 2
        for (int k = li.x3ptr[e]; k < k1; ++k) {
          const int c = li.x3[k];
          x = fma(s.w[c & 63], s.tau[c >> 6], x);
        }
      }
      s.X[e] = x;
    } else {
      const int t = e - nx;
      double p1 = 0.0, p2 = 0.0, p3 = 0.0;
      if (!zero) {
        const uint16_t* v = s.tri + t * NV;
        p1 = s.w[v[0]] + s.w[v[1]];
        p2 = s.w2[v[0]] + s.w2[v[1]];
        p3 = s.w3[v[0]] + s.w3[v[1]];
#pragma unroll
        for (int q = 2; q < NV; ++q) {
          p1 += s.w[v[q]];
          p2 += s.w2[v[q]];
          p3 += s.w3[v[q]];  // the doubled cubes: 2 p_3
        }
        const double q1 = p1 * p1;
        p3 = fma(p1, fma(3.0, p2, q1), p3);  // 6 h_3 = p_1^3 + 3 p_1 p_2 + 2 p_3
        p2 = q1 + p2;                        // 2 h_2 = p_1^2 + p_2
      }
      s.h1[t] = p1;
      s.h2[t] = p2;
      s.h3[t] = p3;
    }
  }
  __syncthreads();
  // seven row sums: one (sum, row) pair per thread
  for (int q = tid; q < kinds << lg; q += kThreads) {
    const int kind = q >> lg, a = q & ((1 << lg) - 1);
    if (a >= nh) continue;
    const int e0 = li.row[a];
    double v = 0.0;
    if (kind >= 2 && kind < 5) {
      const double* h = kind == 2 ? s.h1 : kind == 3 ? s.h2 : s.h3;
      const int k1 = zero ? 0 : li.simptr[e0 + 1];
#pragma unroll 2
      for (int k = li.simptr[e0]; k < k1; ++k) v += h[li.sim[k]];
      (kind == 2 ? s.S1 : kind == 3 ? s.S2 : s.S3)[a] = v;
    } else {
      const double* m = kind == 0 ? s.K : kind == 1 ? s.M : kind == 5 ? s.B1 : s.X;
      const int e1 = zero ? 0 : li.row[a + 1];
      if (p.aug && kind < 2) v = s.cu * (kind == 0 ? s.gA : s.gM)[a];
#pragma unroll 2
      for (int e = e0; e < e1; ++e) v = fma(m[e], s.w[li.pair[e] & 255], v);
      (kind == 0 ? s.Kc : kind == 1 ? s.Mc : kind == 5 ? s.Bc : s.Xc)[a] = v;
    }
  }
  __syncthreads();
  // dot products: Q's rows on warps 0 and 1, pairs of the others on warps 2, 3, 6, 7 (an even
  // load on the SM's four FP64 units)
  const int warp = tid >> 5, lane = tid & 31;
  if (warp < 2) {
    const int a = tid;
    double d = 0.0;
    if (a < nh) {
      // 6 sum_T [h_3 + w h_2 + w^2 h_1 + w^3] = S3 + 3 w (S2 + 2 w (S1 + cnt w))
      const double w = s.w[a], w3 = 3.0 * w;
      d = fma(w3, fma(w + w, fma(s.cnt[a], w, s.S1[a]), s.S2[a]), s.S3[a]);
      s.Q[a] = d;
      d *= w;
    }
    d = warp_sum(d);
    if (lane == 0) s.dots[7 + warp] = d;
  } else if ((warp & 2) && (warp < 4 || p.aug)) {
    const int q = warp == 2 ? 0 : warp == 3 ? 2 : warp == 6 ? 4 : 6;
    const double* y0 = q == 0 ? s.Kc : q == 2 ? s.Mc : q == 4 ? s.Xc : s.t1;
    const double* y1 = q == 0 ? s.gA : q == 2 ? s.gM : s.Bc;
    double d0 = 0.0, d1 = 0.0;
    for (int a = lane; a < nh; a += 32) {
      const double w = s.w[a];
      d0 = fma(y0[a], w, d0);
      if (!p.aug) d1 += w;
      else if (q != 6) d1 = fma(y1[a], w, d1);
    }
    d0 = half_sums(d0, d1);
    if ((lane & 15) == 0 && q + (lane >> 4) < 7) s.dots[q + (lane >> 4)] = d0;
  }
  __syncthreads();
}

// lambda and the residual r = (K0 + zeta G(c)) c - lambda M c at the iterate c = (w, cu), in
// single precision with M c; returns the relative residual |r| / (|lambda| |M c|).  When
// c^T M c is off 1 by more than 1e-3 (or c has the wrong sign) c is rescaled, by the factor
// s.f that the sums at the old c still need; otherwise s.f = 1, and s.g = (c^T M c - 1) / 2 is
// left to the Newton system (then lambda is off by a multiple of g, which r shows).
template <int NV>
__device__ __forceinline__ float evaluate(const DenseProblem& p, Smem<NV>& s, double zeta, bool zero) {
  sums<NV>(p, s, zero);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nh = p.nh, n = nh + p.aug;
  constexpr int kRowWarps = (kMaxN + 31) / 32;
  if (warp < kRowWarps) {
    // polynomials in c_u, one per lane: c^T K0 c, c^T M c, the load's u~ entry N_u, c^T N,
    // (K0 c)_u and (M c)_u
    const double cu = p.aug ? s.cu : 0.0, qo = 0.5 * p.quart_off;
    double k0 = 0.0, k1 = 0.0, k2 = 0.0, k3 = 0.0, k4 = 0.0, m1 = 1.0, m2 = 1.0, m3 = 1.0;
    if (lane == 3) k0 = s.dots[7] + s.dots[8];
    if (p.aug) {
      const double d1 = s.dots[1], d3 = s.dots[3], d4 = s.dots[4], d5 = s.dots[5],
                   d6 = s.dots[6];
      switch (lane) {
        case 0: k1 = d1; k2 = s.auu; break;
        case 1: k1 = d3; k2 = s.buu; break;
        case 2: k0 = d4; k1 = d5; m1 = 3.0; k2 = d6; m2 = 3.0; k3 = s.t0; break;
        case 3: k1 = d4; m1 = 4.0; k2 = d5; m2 = 6.0; k3 = d6; m3 = 4.0; k4 = s.t0; break;
        case 4: k0 = d1; k1 = s.auu; break;
        case 5: k0 = d3; k1 = s.buu; break;
      }
    }
    k0 = lane == 0 ? s.dots[0] : lane == 1 ? s.dots[2] : lane == 3 ? qo * k0 : k0;
    const double v = fma(cu, fma(cu, fma(cu, fma(cu, k4, m3 * k3), m2 * k2), m1 * k1), k0);
    const double cKc = __shfl_sync(0xffffffffu, v, 0), cMc = __shfl_sync(0xffffffffu, v, 1),
                 Nu = __shfl_sync(0xffffffffu, v, 2), cN = __shfl_sync(0xffffffffu, v, 3),
                 Ku = __shfl_sync(0xffffffffu, v, 4), Mu = __shfl_sync(0xffffffffu, v, 5);
    // tests on the high words: FP64 comparisons occupy the FP64 unit like any other operation
    const double dm = cMc - 1.0;
    const bool rescale = (__double2hiint(dm) & 0x7fffffff) > 0x3f50624d ||  // |dm| > 1e-3
                         __double2hiint(p.aug ? cu : s.dots[1]) < 0;
    double f = 1.0, zf2 = zeta, g = 0.5 * dm, lam;
    if (rescale) {
      f = copysign(1.0 / sqrt(cMc), p.aug ? cu : s.dots[1]);
      zf2 = zeta * (f * f);
      g = 0.0;
      lam = f * f * fma(zf2, cN, cKc);
    } else {
      lam = fma(zeta, cN, cKc);
    }
    const int a = tid;
    float rr = 0.0f, mm = 0.0f;
    if (a < n) {
      double k = Ku, m = Mu, nl = Nu;
      if (a < nh) {
        k = s.Kc[a];
        m = s.Mc[a];
        nl = qo * s.Q[a];
        if (p.aug) nl = fma(cu, fma(3.0, s.Xc[a], cu * fma(3.0, s.Bc[a], cu * s.t1[a])), nl);
        double w = s.w[a];
        if (rescale) {
          w *= f;
          s.w[a] = w;
        }
        s.wf[a] = d2f_rn(w);
      }
      double h = fma(zf2, nl, k);
      if (rescale) {
        m *= f;
        h *= f;
      }
      const double r = fma(-lam, m, h);
      s.m64[a] = m;
      s.r64[a] = r;
      const float rf = d2f_rn(r), mf = d2f_rn(m);
      s.m[a] = mf;
      s.r[a] = rf;
      // norms in single precision, scaled by powers of two to the size of |M c| ~ sqrt(M_aa)
      // and of lambda, so that their squares stay in range
      const int em = exponent_of(s.M[0]) / 2, el = exponent_of(lam);
      const float rs = rf * pow2f(-em - el), ms = mf * pow2f(-em);
      rr = rs * rs;
      mm = ms * ms;
    }
    rr = half_sums(rr, mm);
    if ((lane & 15) == 0) s.red[lane >> 4][warp] = rr;
    if (tid == 0) {
      s.f = f;
      s.g = g;
      s.lam = lam;
      s.wf[nh] = 0.0f;
    }
  }
  __syncthreads();
  // cu belongs to the thread of its row from here on (others read it after a barrier)
  if (p.aug && tid == nh) s.cu *= s.f;
  float rr = 0.0f, mm = 0.0f;
  for (int q = 0; q < kRowWarps; ++q) {
    rr += s.red[0][q];
    mm += s.red[1][q];
  }
  const double lam = s.lam;  // its significand, in [1, 2)
  const float l = __int_as_float((127 << 23) | (__double2hiint(lam) & 0xfffff) << 3);
  return exponent_of(lam) < 1024 ? sqrtf(rr / mm) / l : __int_as_float(0x7fffffff);
}

// G(c)_ab of nonzero e = (a, b) at c = f (w_old, cu_old), from the sums of `sums` at the old
// c, in T: sum_T int_T w_H^2 mu_a mu_b + 2 c_u X_ab + c_u^2 B1_ab, with
//   int_T w^2 mu_a mu_b = |T| 2 d! / (d + 4)! h_2(w_1 .. w_nv, w_a, w_b)  (twice for a = b).
// float (the Jacobian): the simplex sums h1f, h2f and wf are those of the rescaled c already.
// double: the assembled system, and the Jacobian of the fallback.
template <int NV, typename T>
__device__ __forceinline__ T coarse_G(const DenseProblem& p, const Smem<NV>& s, const Lists& li,
                                      int e, T f, T cu) {
  constexpr bool single = sizeof(T) == 4;
  const int a = li.pair[e] >> 8, b = li.pair[e] & 255;
  const int k0 = li.simptr[e], k1 = li.simptr[e + 1];
  T s1 = 0, s2 = 0, wa, wb;
  for (int k = k0; k < k1; ++k) {
    const int t = li.sim[k];
    if constexpr (single) {
      s1 += s.h1f[t];
      s2 += s.h2f[t];
    } else {
      s1 += s.h1[t];
      s2 += s.h2[t];
    }
  }
  if constexpr (single) {
    wa = s.wf[a];
    wb = s.wf[b];
  } else {
    wa = s.w[a];
    wb = s.w[b];
    s1 *= f;
    s2 *= f * f;
  }
  const T ws = wa + wb, cnt = (T)(k1 - k0);
  const T quart = (T)(a == b ? p.quart_off : 0.5 * p.quart_off);
  T g = quart * (s2 + (T)2 * (ws * s1 + cnt * (ws * ws - wa * wb)));
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
__device__ __forceinline__ void jacobian(const DenseProblem& p, Smem<NV>& s, T* J, int ns, double lam, T gz) {
  const int nh = p.nh;
  const Lists li = lists_of(s.lists, p.dims, nh);
  if constexpr (sizeof(T) == 4) {
    for (int t = threadIdx.x; t < p.ntri; t += kThreads) {
      const uint16_t* v = s.tri + t * NV;
      float p1 = 0.0f, p2 = 0.0f;
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        const float w = s.wf[v[q]];
        p1 += w;
        p2 = fmaf(w, w, p2);
      }
      s.h1f[t] = p1;
      s.h2f[t] = fmaf(p1, p1, p2);
    }
  }
  __syncthreads();
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
// The indices go in blocks of 4, one barrier per block, and M stays symmetric, so only its
// upper triangle is kept: one 4 x 4 tile (ti <= tj) in the registers of each participating
// thread (91 threads for n = 50, 28 for n = 28).  The owners of the next pivot rows publish
// them to piv (double-buffered), tiles above the diagonal from their transposed columns.
// A block takes about 940 cycles for n = 50 (its chain: publish, barrier, read, 4 x 4 inverse,
// update; 3 cycles per instruction of the one warp on each partition), 12.2k cycles in all;
// pairs of pivots with 2 x 2 inverses took 560 cycles a pair (14k), on full rows over all 256
// threads 520 a pair, and 4 x 4 blocks of full rows with sequential pivots 28.8k in all.
// Leaves whether every pivot was positive in *pivots_ok.
__device__ __forceinline__ bool sweep_inverse(const float* J, float* Ainv, int ns, float tau,
                                           const float* m, float (*piv)[kTile][kMaxSweep],
                                           int n, int* pivots_ok) {
  const int t = threadIdx.x, nt = (n + kTile - 1) / kTile, tiles = nt * (nt + 1) / 2;
  const int team = (tiles + 31) & ~31;  // participating threads, whole warps
  if (t < team) {
    int tj = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
    if ((tj + 1) * (tj + 2) / 2 <= t) ++tj;
    if (tj * (tj + 1) / 2 > t) --tj;
    int ti = t - tj * (tj + 1) / 2;
    const bool own = t < tiles;
    if (!own) ti = tj = nt - 1;  // idle lanes of the last warp: a copy that publishes nothing
    const int i0 = ti * kTile, j0 = tj * kTile;
    float v[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int i = i0 + r, j = j0 + c;
        float x = i == j ? 1.0f : 0.0f;
        if (i < n && j < n) {
          x = J[i * ns + j];
          if (tau != 0.0f) x = fmaf(tau * m[i], m[j], x);
        }
        v[r][c] = x;
      }
    if (ti == 0 && own) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
        *reinterpret_cast<float4*>(&piv[0][r][j0]) = make_float4(v[r][0], v[r][1], v[r][2], v[r][3]);
    }
    bool ok = true;
    for (int kt = 0; kt < nt; ++kt) {
      asm volatile("bar.sync 1, %0;" ::"r"(team) : "memory");
      const float(*p)[kMaxSweep] = piv[kt & 1];
      float h[4][4];  // H = (M_PP)^{-1} by its 2 x 2 blocks [A B; B^T D]
      {
        const float4 q0 = *reinterpret_cast<const float4*>(&p[0][kTile * kt]),
                     q1 = *reinterpret_cast<const float4*>(&p[1][kTile * kt]),
                     q2 = *reinterpret_cast<const float4*>(&p[2][kTile * kt]),
                     q3 = *reinterpret_cast<const float4*>(&p[3][kTile * kt]);
        const float da = fmaf(q0.x, q1.y, -q0.y * q0.y), ia = __fdividef(1.0f, da);
        const float a00 = q1.y * ia, a01 = -q0.y * ia, a11 = q0.x * ia;
        const float t00 = fmaf(a00, q0.z, a01 * q1.z), t01 = fmaf(a00, q0.w, a01 * q1.w),
                    t10 = fmaf(a01, q0.z, a11 * q1.z), t11 = fmaf(a01, q0.w, a11 * q1.w);
        const float s00 = fmaf(-q0.z, t00, fmaf(-q1.z, t10, q2.z)),
                    s01 = fmaf(-q0.z, t01, fmaf(-q1.z, t11, q2.w)),
                    s11 = fmaf(-q0.w, t01, fmaf(-q1.w, t11, q3.w));
        const float ds = fmaf(s00, s11, -s01 * s01), is = __fdividef(1.0f, ds);
        ok = q0.x > 0.0f && da > 0.0f && s00 > 0.0f && ds > 0.0f;
        if (!ok) break;
        h[2][2] = s11 * is;
        h[2][3] = h[3][2] = -s01 * is;
        h[3][3] = s00 * is;
        const float u00 = fmaf(t00, h[2][2], t01 * h[2][3]), u01 = fmaf(t00, h[2][3], t01 * h[3][3]),
                    u10 = fmaf(t10, h[2][2], t11 * h[2][3]), u11 = fmaf(t10, h[2][3], t11 * h[3][3]);
        h[0][0] = fmaf(u00, t00, fmaf(u01, t01, a00));
        h[0][1] = h[1][0] = fmaf(u00, t10, fmaf(u01, t11, a01));
        h[1][1] = fmaf(u10, t10, fmaf(u11, t11, a11));
        h[0][2] = h[2][0] = -u00;
        h[0][3] = h[3][0] = -u01;
        h[1][2] = h[2][1] = -u10;
        h[1][3] = h[3][1] = -u11;
      }
      float f[4][4], y[4][4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 x = *reinterpret_cast<const float4*>(&p[q][i0]);
        const float4 z = *reinterpret_cast<const float4*>(&p[q][j0]);
        const float xr[4] = {x.x, x.y, x.z, x.w};
        y[q][0] = z.x; y[q][1] = z.y; y[q][2] = z.z; y[q][3] = z.w;
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) f[r][c] = q == 0 ? xr[r] * h[0][c] : fmaf(xr[r], h[q][c], f[r][c]);
      }
      if (ti == kt || tj == kt) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            v[r][c] = 0.0f;
            if (ti == kt) f[r][c] = -h[r][c];
            if (tj == kt) y[r][c] = r == c ? -1.0f : 0.0f;
          }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int q = 0; q < 4; ++q) v[r][c] = fmaf(-f[r][q], y[q][c], v[r][c]);
      if (own && ti == kt + 1) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
          *reinterpret_cast<float4*>(&piv[(kt + 1) & 1][r][j0]) =
              make_float4(v[r][0], v[r][1], v[r][2], v[r][3]);
      } else if (own && tj == kt + 1) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          *reinterpret_cast<float4*>(&piv[(kt + 1) & 1][c][i0]) =
              make_float4(v[0][c], v[1][c], v[2][c], v[3][c]);
      }
    }
    if (own && ok) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (i0 + r < n && j0 + c < n) {
            Ainv[(i0 + r) * ns + j0 + c] = v[r][c];
            if (ti != tj) Ainv[(j0 + c) * ns + i0 + r] = v[r][c];
          }
    }
    if (t == 0) *pivots_ok = ok;  // every participating thread saw the same pivots
  }
  __syncthreads();
  const bool ok = *pivots_ok != 0;
  __syncthreads();  // pivots_ok may be written again
  return ok;
}

// y = A^{-1} x for two vectors, Ainv = -A^{-1} in single precision: 4 threads per row
__device__ __forceinline__ void apply_inverse(const float* Ainv, int ns, const float* x1,
                                              float* y1, const float* x2, float* y2, int n) {
  const int part = threadIdx.x & 3;
  for (int row0 = 0; row0 < n; row0 += kThreads / 4) {
    const int row = row0 + (threadIdx.x >> 2);
    float a = 0.0f, b = 0.0f;
    if (row < n)
#pragma unroll 4
      for (int j = part; j < n; j += 4) {
        const float v = Ainv[row * ns + j];
        a = fmaf(v, x1[j], a);
        b = fmaf(v, x2[j], b);
      }
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    b += __shfl_xor_sync(0xffffffffu, b, 1);
    b += __shfl_xor_sync(0xffffffffu, b, 2);
    if (part == 0 && row < n) {
      y1[row] = -a;
      y2[row] = -b;
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

// c += dc = -y1 + dl y2 of the bordered Newton system with (M c)^T dc = -g; returns dl
template <int NV>
__device__ __forceinline__ float newton_update(const DenseProblem& p, Smem<NV>& s) {
  const int n = p.nh + p.aug, lane = threadIdx.x & 31;
  float p1 = 0.0f, p2 = 0.0f;
  for (int a = lane; a < n; a += 32) {
    p1 = fmaf(s.m[a], s.y1[a], p1);
    p2 = fmaf(s.m[a], s.y2[a], p2);
  }
  const float v = half_sums(p1, p2), g = d2f_rn(s.g);
  const float dl =
      (__shfl_sync(0xffffffffu, v, 0) - g) / __shfl_sync(0xffffffffu, v, 16);
  for (int a = threadIdx.x; a < n; a += kThreads)
    set_entry(p, s, a, (a < p.nh ? s.w[a] : s.cu) + f2d_exact(fmaf(dl, s.y2[a], -s.y1[a])));
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

// (The steps of the iteration are inlined at one call site each: called functions would take
// their shared arrays as generic pointers, whose loads are slower.)
// One CTA of 256 threads per problem, a batch of problems one CTA each (two resident per SM:
// at most 128 registers and half of the shared memory).  The iteration count is bounded by
// max_iter (chord steps, at most kMaxChord per inverse, are not counted: they replace the
// refinement of the Newton correction); hitting it a second time, after a fresh start with
// kSwitchAgain, sets status 1.
// ASSEMBLE: only assemble K0, M and G(c_init) into K_out, M_out, G_out.
template <int NV, bool ASSEMBLE>
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
  {  // 16 bytes a load (the lists are padded to that on the device)
    const uint4* from = reinterpret_cast<const uint4*>(p.lists);
    uint4* to = reinterpret_cast<uint4*>(s.lists);
    for (int e = tid; e < (p.dims.total(nh) + 7) / 8; e += kThreads) to[e] = from[e];
  }
  for (int e = tid; e < p.ntri * NV; e += kThreads) {
    const int v = p.tri[e];
    s.tri[e] = (uint16_t)(v < 0 ? nh : v);
  }
  auto start = [&] {
    if (tid > nh) return;
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
  };
  start();
  if (p.aug && tid < nh) {
    s.gA[tid] = p.gA[ib * nh + tid];
    s.gM[tid] = p.gM[ib * nh + tid];
    s.t1[tid] = p.t1[ib * nh + tid];
  }
  if (tid == kThreads - 1) {
    s.auu = p.aug ? p.auu[ib] : 0.0;
    s.buu = p.aug ? p.buu[ib] : 0.0;
    s.t0 = p.aug ? p.t0[ib] : 0.0;
  }
  for (int e = tid; e < 2 * n * ns / 4; e += kThreads)
    reinterpret_cast<float4*>(J)[e] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  __syncthreads();
  {
    const Lists li = lists_of(s.lists, p.dims, nh);
    for (int e = tid; e < p.dims.npat; e += kThreads) {
      const int k = (li.pair[e] >> 8) * nh + (li.pair[e] & 255);
      s.K[e] = L1[k];
      s.M[e] = M1[k];
      if (p.aug) s.B1[e] = p.B1[ib * nh * nh + k];
    }
    if (tid < nh) s.cnt[tid] = (double)(li.simptr[li.row[tid] + 1] - li.simptr[li.row[tid]]);
  }
  if (p.aug) {
    const uint16_t* tp = s.lists + p.dims.tripptr(nh);
    const uint16_t* ti = s.lists + p.dims.trip(nh);
    const double* t3 = p.t3 + ib * p.ntri * p.nt3;
    for (int q = tid; q < p.dims.nq; q += kThreads) {
      double v = 0.0;
      const int k1 = tp[q + 1];
      for (int k = tp[q]; k < k1; k += 6) {  // 6 loads in flight
        double x[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) x[j] = k + j < k1 ? t3[ti[k + j]] : 0.0;
#pragma unroll
        for (int j = 0; j < 6; ++j)
          if (k + j < k1) v += x[j];
      }
      s.tau[q] = v;
    }
  }
  __syncthreads();
  if constexpr (ASSEMBLE) {
    sums<NV>(p, s, false);
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
  bool zero = p.aug && !p.c_init;              // the start c = u~
  bool newton = false;
  bool failed = false;  // the Newton matrix of this iterate had a non-positive pivot
  float rn = 0.0f, reach = kSwitch;
  for (;;) {
    bool converged = false, chord = false;
    if (!failed) {
      rn = evaluate<NV>(p, s, zeta, zero);
      zero = false;
      converged = rn <= (float)p.tol;
      // A step with the inverse of an earlier iterate cuts the residual by about twice what
      // the latest step did (the Jacobian is off by the distance moved since, and by ~1e-6):
      // it replaces a new inverse where that reaches the tolerance.  On convergence the same
      // step, without another evaluation, takes c and lambda from the tolerance to rounding.
      chord = chords < kMaxChord && rn < 0.05f * last &&
              (converged || 4.0f * rn * rn <= last * (float)p.tol);
      if (converged) status = 0;
      if (!chord && it >= p.max_iter && !converged && reach == kSwitch) {
        start();
        reach = kSwitchAgain;
        zero = p.aug && !p.c_init;
        it = 0;
        chords = kMaxChord;
        __syncthreads();
        continue;
      }
      if (!chord && (converged || it >= p.max_iter)) break;
      if (!chord) newton = rn <= reach;
    } else {
      newton = false;
    }
    if (chord) {
      ++chords;
    } else {
      // Newton: A' = K0 + 3 zeta G - lambda M + |lambda| (Mc)(Mc)^T; otherwise an
      // inverse-power step c <- (K0 + zeta G)^{-1} M c
      const double lam = newton ? s.lam : 0.0, gz = newton ? 3.0 * zeta : zeta;
      jacobian<NV, float>(p, s, J, ns, lam, (float)gz);
      const bool have = sweep_inverse(J, Pinv, ns, newton ? fabsf(d2f_rn(lam)) : 0.0f, s.m, s.piv,
                                      n, &s.pivots_ok);
      chords = have && newton ? 0 : kMaxChord;
      if (!have && !solve_fp64<NV>(p, s, reinterpret_cast<double*>(J), J, ns, lam, gz,
                                   newton ? fabs(lam) : 0.0, newton)) {
        if (!newton) break;
        failed = true;  // the same iterate again, by an inverse-power step
        continue;
      }
      failed = false;
      ++it;
      chord = have;  // step with the inverse (the FP64 fallback has solved already)
    }
    if (chord) apply_inverse(Pinv, ns, newton ? s.r : s.m, s.y1, s.m, s.y2, n);
    if (newton) {
      const float dl = newton_update(p, s);
      last = rn;
      if (converged) {
        dlam = (double)dl;
        break;
      }
    } else {
      for (int a = tid; a < n; a += kThreads) set_entry(p, s, a, f2d_exact(s.y1[a]));
      __syncthreads();
    }
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
// Largest entry of I - L X0 for which two rounds reach FP64 rounding (each about multiplies the
// residual by that much): 1e-7 for the operators of any resolved potential, above it from condition
// numbers of some 1e3 on (an A + W that a negative potential brings near singularity).
constexpr float kInverseStart = 3.8e-6f;

// L^{-1} of the SPD level-1 operator, one CTA per instance: the single-precision inverse of
// the sweep operator (~1e-6), then X <- X + Y (I - L X) with Y that inverse: the residual in
// FP64 over the nonzeros of L (15 or 7 per row, so the FP64 work is n^2 x that, not n^3), the
// product in single precision on a residual that shrinks by ~1e6 a round; two rounds leave the
// rounding of I - L X.  An L whose single-precision elimination meets a non-positive pivot, or
// leaves a residual above kInverseStart, takes the FP64 LDL^T.
__global__ void __launch_bounds__(kThreads) k_spd_inverse(const double* __restrict__ L,
                                                          double* __restrict__ Linv, int n,
                                                          const uint16_t* __restrict__ lists,
                                                          DenseLists dims) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) float piv[2][kTile][kMaxSweep];
  __shared__ int pivots_ok;
  L += blockIdx.x * (size_t)n * n;  // instance blockIdx.x
  Linv += blockIdx.x * (size_t)n * n;
  const int ns = row_stride(n), tid = threadIdx.x;
  float* R = reinterpret_cast<float*>(smem_raw);
  float* Y = R + n * ns;  // -(single-precision inverse)
  double* X = reinterpret_cast<double*>(Y + n * ns);
  double* dinv = X + n * n;
  for (int e = tid; e < n * n; e += kThreads) R[(e / n) * ns + e % n] = (float)L[e];
  __syncthreads();
  auto in_fp64 = [&] {
    const bool ok = inverse_fp64(L, reinterpret_cast<double*>(R), X, dinv, n);
    for (int e = tid; e < n * n; e += kThreads) Linv[e] = ok ? X[e] : nan("");
  };
  if (!sweep_inverse(R, Y, ns, 0.0f, nullptr, piv, n, &pivots_ok)) {
    in_fp64();
    return;
  }
  for (int e = tid; e < n * n; e += kThreads) X[e] = -(double)Y[(e / n) * ns + e % n];
  const uint16_t* pair = lists + dims.pair(n);
  const int nq = (n + 3) / 4;
  for (int round = 0; round < kInverseRounds; ++round) {
    __syncthreads();
    bool large = false;
    for (int e = tid; e < n * n; e += kThreads) {
      const int i = e / n, j = e - i * n;
      double r = i == j ? 1.0 : 0.0;
      for (int q = lists[i]; q < lists[i + 1]; ++q) {
        const int k = pair[q] & 255;
        r = fma(-L[i * n + k], X[k * n + j], r);
      }
      R[i * ns + j] = (float)r;
      large = large || !(fabsf((float)r) <= kInverseStart);
    }
    if (__syncthreads_or(round == 0 && large)) {
      in_fp64();
      return;
    }
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
  if (p.K_out) {
    if (p.nvert == 3) k_dense_scf<3, true><<<nb, kThreads, smem, s>>>(p);
    else k_dense_scf<4, true><<<nb, kThreads, smem, s>>>(p);
  } else {
    if (p.nvert == 3) k_dense_scf<3, false><<<nb, kThreads, smem, s>>>(p);
    else k_dense_scf<4, false><<<nb, kThreads, smem, s>>>(p);
  }
}

// The attributes are per function, shared by every handle in the process, so they are always
// set to what the largest accepted mesh needs (never to one caller's smaller need).
cudaError_t dense_prepare(size_t need) {
  if (need > kDenseSmemLimit) return cudaErrorInvalidValue;
  const struct { const void* f; size_t smem; } k[] = {
      {(const void*)k_dense_scf<3, false>, scf_smem(Cap<3>::nh + 1, 3)},
      {(const void*)k_dense_scf<4, false>, scf_smem(Cap<4>::nh + 1, 4)},
      {(const void*)k_dense_scf<3, true>, scf_smem(Cap<3>::nh + 1, 3)},
      {(const void*)k_dense_scf<4, true>, scf_smem(Cap<4>::nh + 1, 4)},
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
