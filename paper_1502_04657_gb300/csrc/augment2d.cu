// Fine-grid pass of the augmented nonlinear problem (Algorithm 3.1 step 2), 2D.
//
// On V_{H,h_k} = V_H + span{u~}, with w = w_H + c_u u~, the nonlinear matrix
// G(c)_ij = int w^2 psi_i psi_j needs four integrals of u~ against coarse hats phi^H:
//   T0    = int u~^4                       = u~ . N(u~),       N(u)_p = int u^3 phi_p
//   T1_a  = int u~^3 phi^H_a               = (P^T ... P^T N(u~))_a   (repeated restriction)
//   T2_ab = int u~^2 phi^H_a phi^H_b       = (P^T ... P^T B(u~) P ... P)_ab,
//           B(u)_pq = int u^2 phi_p phi_q, the FE matrix of a form on V_{h_k}; restricting a
//           form to the nested subspace is exact, level by level (Galerkin coarsening)
//   T3^T_abc = int_T u~ mu_a mu_b mu_c     per coarse triangle T (barycentrics mu of T)
// (the paper re-assembles the augmented matrix with a fine pass per nonlinear iteration,
// Section 3.2; these four quantities make every iteration independent of the fine grid).
//
// T3 is linear in u~: T3^T = sum_v u~_v int_T phi_v q, q = mu_a mu_b mu_c a cubic.  Taylor
// expansion of q about node v is exact, so int_T phi_v q = sum_{i+j<=3} d^{ij}q(v)/(i!j!) m_ij
// with m_ij the moments of phi_v over the fine triangles of v's star that lie in T.  Those
// depend only on v's class (interior of T, one of T's three edges, one of its vertices), so
// T3 follows from monomial sums of u~ per class: 4 FP64 operations per interior node.
#include "fmg_internal.h"
#include "reduce_dev.cuh"
#include "dfloat.cuh"
#include "star2d.cuh"

namespace fmg {
namespace {

__device__ __forceinline__ size_t at(int i, int j, int pitch) { return (size_t)j * pitch + i; }

// N(u)_p and the density stencil B(u) at p (coupling to p, E, N, NE).  Star triangles of p
// are the consecutive pairs of its hexagon of neighbours E, NE, N, W, SW, S; on a triangle
// (p, q, r) of area |K|:
//   int u^2 lambda_p^2       = |K|/90  [6u_p^2 + u_q^2 + u_r^2 + 3u_p u_q + 3u_p u_r + u_q u_r]
//   int u^2 lambda_p lambda_q = |K|/180 [3u_p^2 + 3u_q^2 + u_r^2 + 4u_p u_q + 2u_p u_r + 2u_q u_r]
// Summed over the star, and written with the per-edge numbers of the column walk
// (star2d.cuh: s, F = s^2 + a^2 + b^2 of an edge (a, b), M1 and sum F over the opposite
// edges):
//   B_pp = |K|/180 [u_p (72 u_p + 6 M1) + sum F]
//   B_pq = |K|/180 [2 (F_pq + s_pq (s_pq + u_r1 + u_r2)) + u_r1^2 + u_r2^2]
// for the edge p-q shared by the triangles closed by r1 and r2 (E: NE, S; N: NE, W;
// NE: E, N).  s60, s180 = |K| / 60, / 180 (computed on the host: an FP64 division per node
// would cost as much as a quarter of the kernel's arithmetic).
template <int R>
__device__ __noinline__ void nload_density2d_fp64(int n, int pitch, size_t st, double s60,
                                                  double s180, const double* __restrict__ u,
                                                  double* __restrict__ nl,
                                                  double* __restrict__ bC, double* __restrict__ bE,
                                                  double* __restrict__ bN,
                                                  double* __restrict__ bNE) {
  using T = double;
  star2d_walk<T, R>(n, pitch, st, u, [&](size_t k, const Star2D<T>& p) {
    nl[k] = s60 * star_cubic(p);
    bC[k] = s180 * fma(p.u, fma(T(72), p.u, T(6) * p.M1), p.SF);
    bE[k] = s180 * fma(T(2), fma(p.H.s, p.H.s + (p.uNE + p.uS), p.H.F), p.qNE + p.qS);
    bN[k] = s180 * fma(T(2), fma(p.V.s, p.V.s + (p.uNE + p.uW), p.V.F), p.qNE + p.qW);
    bNE[k] = s180 * fma(T(2), fma(p.D.s, p.D.s + (p.uE + p.uN), p.D.F), p.qE + p.qN);
  });
}

// N and the density stencil of one node in FP64: the cubic load through the pair sums m_k = n_k +
// n_{k+1} (nload_at in grid2d.cu) and the density stencil from the two triangle formulas above.
// s60, s90, s180 = |K| / 60, / 90, / 180.
__device__ __forceinline__ void nload_density_at(size_t k, int pitch, double s60, double s90,
                                                 double s180, const double* __restrict__ u,
                                                 double* __restrict__ nl, double* __restrict__ bC,
                                                 double* __restrict__ bE, double* __restrict__ bN,
                                                 double* __restrict__ bNE) {
  const double up = u[k];
  const double nE = u[k + 1], nNE = u[k + pitch + 1], nN = u[k + pitch];
  const double nW = u[k - 1], nSW = u[k - pitch - 1], nS = u[k - pitch];
  // the cubic load through the pair sums m_k = n_k + n_{k+1} (see nload_at in grid2d.cu)
  const double m0 = nE + nNE, m1 = nNE + nN, m2 = nN + nW, m3 = nW + nSW, m4 = nSW + nS,
          m5 = nS + nE;
  const double qE = nE * nE, qNE = nNE * nNE, qN = nN * nN, qW = nW * nW, qSW = nSW * nSW,
          qS = nS * nS;
  const double M1 = ((m0 + m1) + (m2 + m3)) + (m4 + m5);  // 2 S1
  double M2 = m0 * m0;
  M2 = fma(m1, m1, M2);
  M2 = fma(m2, m2, M2);
  M2 = fma(m3, m3, M2);
  M2 = fma(m4, m4, M2);
  M2 = fma(m5, m5, M2);
  const double s2 = ((qE + qNE) + (qN + qW)) + (qSW + qS);
  double M3 = m0 * (qE + qNE);
  M3 = fma(m1, qNE + qN, M3);
  M3 = fma(m2, qN + qW, M3);
  M3 = fma(m3, qW + qSW, M3);
  M3 = fma(m4, qSW + qS, M3);
  M3 = fma(m5, qS + qE, M3);
  const double u2 = up * up;
  const double s2p = fma(0.5, M2, s2);  // 2 S2 + P
  nl[k] = s60 * (fma(2.0 * up, s2p, u2 * fma(24.0, up, 3.0 * M1)) + M3);
  // density stencil, diagonal: sum over the six triangles
  bC[k] = s90 * fma(36.0, u2, fma(3.0 * up, M1, s2p));
  // edge p-q shared by the triangles closed by r1 and r2
  const double u26 = 6.0 * u2;
  bE[k] = s180 * fma(6.0, qE,
                     u26 + fma(8.0 * up, nE, fma(2.0 * (up + nE), nNE + nS, qNE + qS)));
  bN[k] = s180 * fma(6.0, qN,
                     u26 + fma(8.0 * up, nN, fma(2.0 * (up + nN), nNE + nW, qNE + qW)));
  bNE[k] = s180 * fma(6.0, qNE,
                      u26 + fma(8.0 * up, nNE, fma(2.0 * (up + nNE), nE + nN, qE + qN)));
}

// the same, called for the nodes that the fixed-point walk leaves short of bits
__device__ __noinline__ void nload_density2d_redo(size_t k, int pitch, double s60, double s180,
                                                  const double* __restrict__ u,
                                                  double* __restrict__ nl, double* __restrict__ bC,
                                                  double* __restrict__ bE, double* __restrict__ bN,
                                                  double* __restrict__ bNE) {
  nload_density_at(k, pitch, s60, 2.0 * s180, s180, u, nl, bC, bE, bN, bNE);
}

template <int R>
__global__ void __launch_bounds__(32 * kStarWarps, 4)
    k_nload_density2d(int n, int pitch, size_t st, double s60, double s180,
                      const double* __restrict__ u, double* __restrict__ nl,
                      double* __restrict__ bC, double* __restrict__ bE,
                      double* __restrict__ bN, double* __restrict__ bNE) {
  const int e = star2d_exponent<R, true>(n, pitch, st, u);
  if (e == kFxNone) {
    nload_density2d_fp64<R>(n, pitch, st, s60, s180, u, nl, bC, bE, bN, bNE);
    return;
  }
  const double a3 = fx_scale<kFx2>(s60, 3, e), a2 = fx_scale<kFx2>(s180, 2, e);
  unsigned redo = 0;
  star2d_walk_fx<true, R>(n, pitch, st, u, e, [&](size_t k, const Star2DFx& p) {
    const fx<kFx2> v = star_cubic(p);
    bool lack = fx_short<kShortLoad2>(v);
    auto put = [&](double* b, fx<kFx2> w) {
      lack = lack || fx_short<kShortDensity2>(w);
      b[k] = to_double(w, a2);
    };
    nl[k] = to_double(v, a3);
    put(bC, madd<6>(p.u * madd<12>(p.u, p.M1), p.SF));
    put(bE, madd<2>(fma(p.Hs, p.Hs + (p.uNE + p.uS), p.HF), p.qNE + p.qS));
    put(bN, madd<2>(fma(p.Vs, p.Vs + (p.uNE + p.uW), p.VF), p.qNE + p.qW));
    put(bNE, madd<2>(fma(p.Ds, p.Ds + (p.uE + p.uN), p.DF), p.qE + p.qN));
    redo = redo << 1 | (unsigned)lack;
  });
  star2d_redo<R>(n, pitch, st, redo, [&](size_t k) {
    nload_density2d_redo(k, pitch, s60, s180, u, nl, bC, bE, bN, bNE);
  }, [&] { nload_density2d_fp64<R>(n, pitch, st, s60, s180, u, nl, bC, bE, bN, bNE); });
}

// The same quantities node by node, for levels below n = 64
__global__ void k_nload_density2d_node(int n, int pitch, size_t st, double s60, double s90,
                                       double s180, const double* __restrict__ u,
                                       double* __restrict__ nl, double* __restrict__ bC,
                                       double* __restrict__ bE, double* __restrict__ bN,
                                       double* __restrict__ bNE) {
  const int i = 1 + blockIdx.x * blockDim.x + threadIdx.x;
  const int j = 1 + blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= n || j >= n) return;
  nload_density_at(blockIdx.z * st + at(i, j, pitch), pitch, s60, s90, s180, u, nl, bC, bE, bN, bNE);
}

// ---- T3 class sums -----------------------------------------------------------------------
// Per coarse triangle, 25 sums in normalised coordinates (sg, tg) = (s, t) / r of the coarse
// cell (s, t the fine offsets from its corner, 0..r):
//   [0..9]   interior: sum u sg^k tg^l, (k,l) in kMono order
//   [10..13] edge A: sum u x^m  (T0: bottom t = 0, x = sg;  T1: left s = 0, x = tg)
//   [14..17] edge B: sum u x^m  (T0: right s = r, x = tg;   T1: top t = r,  x = sg)
//   [18..21] diagonal s = t: sum u sg^m
//   [22..24] vertex values (T0: V00, V10, V11;  T1: V00, V11, V01)
//
// Interior: a thread takes a column s of the cell over kSumRows rows and adds its nodes to T0
// (t < s) or T1 (t > s), so every column is the same length and every node is read once; the rows
// are loaded 16 at a time (a row at a time, with the class of each node decided as it came,
// waited out a memory latency per row: 532 us on 16.8M nodes) and summed in integers: 153 -> 107 us.
// Only the 32 rows around a warp's diagonal need the comparison per lane.  Edges, diagonals and
// vertices (one block per cell) go apart.
constexpr int kSums = 25;
constexpr int kSumThreads = 128;
constexpr int kSumRows = 128;
constexpr int kInner = 20;  // interior sums of a cell: 10 of T0, 10 of T1
constexpr int kLines = 24;  // sum u x^m, m < 4, of bottom, right, left, top, diagonal; vertices

// Sixteen rows t0 .. t0 + 15 of a column as integers in units of 2^(e - 51), |v| <= 2^e.  Adding
// up running sums, c0 += v, c1 += c0, c2 += c1, c3 += c2, gives with j = 16 .. 1 counting down
// the rows sum v, sum v j, sum v j (j + 1) / 2 and sum v j (j + 1) (j + 2) / 6 (< 2^63), exactly:
// four integer additions per node where sums of FP64 monomials take four FP64 operations, which
// then cost 25 per 16 nodes.  t / r = (b - j) / r with b = t0 + 16 turns them into the sums of
// (t / r)^m: pb[m] = (b / r)^m, p1[m] = r^-m.
// Against exact sums over columns of 63 and 511 nodes: sine, linear and slowly falling u 2e-16 to 9e-16
// for every m, where FP64 sums leave 2e-16 to 2.5e-15; u falling by a bit per node 7e-16 to 1e-13
// (m = 0 to 3; FP64 8e-16), since a run is rounded at 2^-52 of its largest value.
constexpr int kRun = 16, kRunB = 51;
__device__ __forceinline__ void run_sums(const double (&v)[kRun], int e,
                                         const double* __restrict__ pb,
                                         const double* __restrict__ p1, double (&c)[4]) {
  const int shift = e + 1084 - kRunB;
  long long i0 = 0, i1 = 0, i2 = 0, i3 = 0;
#pragma unroll
  for (int q = 0; q < kRun; ++q) {
    i0 += fx_rounded(v[q], shift);
    i1 += i0;
    i2 += i1;
    i3 += i2;
  }
  const double sc = fx_pow2(e - kRunB);
  const double a0 = __ll2double_rn(i0) * sc, s1 = __ll2double_rn(i1);
  const double t1 = s1 * (sc * p1[1]), t2 = __ll2double_rn(2 * i2 - i1) * (sc * p1[2]),
               t3 = fma(6.0, __ll2double_rn(i3 - i2), s1) * (sc * p1[3]);
  c[0] += a0;
  c[1] = fma(pb[1], a0, c[1]) - t1;
  c[2] = fma(pb[2], a0, c[2]) + fma(-2.0 * pb[1], t1, t2);
  c[3] = fma(pb[3], a0, c[3]) + fma(3.0 * pb[1], t2, fma(-3.0 * pb[2], t1, -t3));
}

// c_m += sum_{ta <= t < tb} col[t pf] (t / r)^m.  Runs of 16 rows in integers, with an exponent
// per lane and run (FP64 when it lies out of range: zeros, infinities, NaN).
__device__ __forceinline__ void column_sums(const double* __restrict__ col, int pf,
                                            const double* __restrict__ pw, int ta, int tb,
                                            double (&c)[4]) {
  int t = ta;
  for (; t + kRun <= tb; t += kRun) {
    double v[kRun];
    int top = 0;
#pragma unroll
    for (int q = 0; q < kRun; ++q) v[q] = col[(size_t)(t + q) * pf];
#pragma unroll
    for (int q = 0; q < kRun; ++q) top = max(top, __double2hiint(v[q]) & 0x7fffffff);
    const int e = ((top + 1) >> 20) - 1022;
    if (e >= -900 && e <= 900) {
      run_sums(v, e, pw + 4 * (t + kRun), pw + 4, c);
    } else {
      for (int q = 0; q < kRun; ++q) {
        const double x = col[(size_t)(t + q) * pf];
        const double* p = pw + 4 * (t + q);
        c[0] += x;
        for (int m = 1; m < 4; ++m) c[m] = fma(x, p[m], c[m]);
      }
    }
  }
  for (; t < tb; ++t) {
    const double v = col[(size_t)t * pf];
    const double* p = pw + 4 * t;
    c[0] += v;
#pragma unroll
    for (int m = 1; m < 4; ++m) c[m] = fma(v, p[m], c[m]);
  }
}

__global__ void __launch_bounds__(kSumThreads)
    k_t3_sums2d(int pf, int n1, int r, size_t st, size_t pst, const double* __restrict__ u,
                const double* __restrict__ pw, double* __restrict__ partials, int col_blocks,
                int chunks) {
  __shared__ double sh[kSumThreads];
  const int cell = blockIdx.y, I = cell % n1, J = cell / n1;
  u += blockIdx.z * st + (size_t)(J * r) * pf + (size_t)I * r;  // the cell's corner
  partials += blockIdx.z * pst;
  double acc[kInner];
  if ((int)blockIdx.x < chunks) {
    const int cb = blockIdx.x % col_blocks, seg = blockIdx.x / col_blocks;
    const int s = 1 + cb * blockDim.x + threadIdx.x;
    const int ta = 1 + seg * kSumRows, tb = min(ta + kSumRows, r);
    const int s0 = s - (int)(threadIdx.x & 31), s1 = min(s0 + 31, r - 1);  // the warp's columns
    const double* col = u + min(s, r - 1);
    double c0[4] = {0.0, 0.0, 0.0, 0.0}, c1[4] = {0.0, 0.0, 0.0, 0.0};
    column_sums(col, pf, pw, ta, min(tb, s0), c0);
    for (int t = max(ta, s0); t < min(tb, s1 + 1); ++t) {
      const double v = col[(size_t)t * pf], v0 = t < s ? v : 0.0, v1 = t > s ? v : 0.0;
      const double* p = pw + 4 * t;
      c0[0] += v0;
      c1[0] += v1;
#pragma unroll
      for (int m = 1; m < 4; ++m) {
        c0[m] = fma(v0, p[m], c0[m]);
        c1[m] = fma(v1, p[m], c1[m]);
      }
    }
    column_sums(col, pf, pw, max(ta, s1 + 1), tb, c1);
    const double* ps = pw + 4 * min(s, r - 1);  // sg^m
    const double p1 = ps[1], p2 = ps[2], p3 = ps[3];
    auto monomials = [&](const double (&c)[4], double* o) {
      // kMono order: (0,0),(1,0),(0,1),(2,0),(1,1),(0,2),(3,0),(2,1),(1,2),(0,3)
      const bool ok = s < r;
      const double a0 = ok ? c[0] : 0.0, a1 = ok ? c[1] : 0.0, a2 = ok ? c[2] : 0.0,
                   a3 = ok ? c[3] : 0.0;
      o[0] = a0; o[1] = p1 * a0; o[2] = a1; o[3] = p2 * a0; o[4] = p1 * a1; o[5] = a2;
      o[6] = p3 * a0; o[7] = p2 * a1; o[8] = p1 * a2; o[9] = a3;
    };
    monomials(c0, acc);
    monomials(c1, acc + 10);
    block_sum_to<kInner>(acc, sh, partials + ((size_t)cell * chunks + blockIdx.x) * kInner);
    return;
  }
  double* out = partials + (size_t)n1 * n1 * chunks * kInner + (size_t)cell * kLines;
#pragma unroll
  for (int m = 0; m < kInner; ++m) acc[m] = 0.0;
  for (int x = 1 + threadIdx.x; x < r; x += blockDim.x) {
    const double v[5] = {u[x], u[(size_t)x * pf + r], u[(size_t)x * pf], u[(size_t)r * pf + x],
                         u[(size_t)x * pf + x]};
    const double* p = pw + 4 * x;
#pragma unroll
    for (int e = 0; e < 5; ++e) {
      acc[4 * e] += v[e];
#pragma unroll
      for (int m = 1; m < 4; ++m) acc[4 * e + m] = fma(v[e], p[m], acc[4 * e + m]);
    }
  }
  block_sum_to<kInner>(acc, sh, out);
  if (threadIdx.x == 0) {
    out[kInner] = u[0];
    out[kInner + 1] = u[r];
    out[kInner + 2] = u[(size_t)r * pf + r];
    out[kInner + 3] = u[(size_t)r * pf];
  }
}

// Finalise: T3^T_e = h^2 sum_m map[T][e][m] S_m, a fixed linear map of the 25 class sums per
// triangle type, built on the host for the level's r (t3_map2d).
__global__ void k_t3_finalize2d(int cells, int chunks, double h2, size_t pst, size_t tst,
                                const double* __restrict__ partials,
                                const double* __restrict__ map, double* __restrict__ t3) {
  partials += blockIdx.y * pst;
  t3 += blockIdx.y * tst;
  const int tri = blockIdx.x, cell = tri >> 1, T = tri & 1;
  __shared__ double sums[kSums];
  const int m = threadIdx.x;
  if (m < 10) {
    const double* p = partials + (size_t)cell * chunks * kInner + T * 10 + m;
    double s = 0.0;
#pragma unroll 8
    for (int c = 0; c < chunks; ++c) s += p[(size_t)c * kInner];
    sums[m] = s;
  } else if (m < kSums) {
    const double* e = partials + (size_t)cells * chunks * kInner + (size_t)cell * kLines;
    // edge A: bottom (T0) / left (T1); edge B: right / top; diagonal; vertices
    const int q = m - 10;
    int at;
    if (q < 4) at = (T == 0 ? 0 : 8) + q;
    else if (q < 8) at = (T == 0 ? 4 : 12) + q - 4;
    else if (q < 12) at = 16 + q - 8;
    else if (q == 12) at = kInner;
    else if (q == 13) at = kInner + (T == 0 ? 1 : 2);
    else at = kInner + (T == 0 ? 2 : 3);
    sums[m] = e[at];
  }
  __syncthreads();
  const int e = threadIdx.x;
  if (e >= 10) return;
  const double* row = map + ((size_t)T * 10 + e) * kSums;
  double acc = 0.0;
#pragma unroll
  for (int q = 0; q < kSums; ++q) acc = fma(row[q], sums[q], acc);
  t3[(size_t)tri * 10 + e] = h2 * acc;
}

__global__ void k_gather_level1_2d(int n, int pitch, size_t st, const double* __restrict__ gA_pad,
                                   const double* __restrict__ gM_pad,
                                   const double* __restrict__ t1_pad, Density2D b,
                                   double* __restrict__ gA, double* __restrict__ gM,
                                   double* __restrict__ t1, double* __restrict__ B1) {
  const int m = n - 1;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= m * m) return;
  const int i = 1 + p % m, j = 1 + p / m;
  const size_t nh = (size_t)m * m;
  const size_t k = blockIdx.y * st + at(i, j, pitch);
  const size_t q = blockIdx.y * nh + p;
  gA[q] = gA_pad[k];
  gM[q] = gM_pad[k];
  t1[q] = t1_pad[k];
  double* row = B1 + blockIdx.y * nh * nh + (size_t)p * nh;
  for (int q = 0; q < m * m; ++q) row[q] = 0.0;
  row[p] = b.C[k];
  auto put = [&](int di, int dj, const double* a, size_t ka) {
    const int ii = i + di, jj = j + dj;
    if (ii < 1 || jj < 1 || ii >= n || jj >= n) return;
    row[(ii - 1) + (jj - 1) * m] = a[ka];
  };
  put(1, 0, b.E, k);
  put(-1, 0, b.E, k - 1);
  put(0, 1, b.N, k);
  put(0, -1, b.N, k - pitch);
  put(1, 1, b.NE, k);
  put(-1, -1, b.NE, k - pitch - 1);
}

// a block takes blockDim.x interior columns (whole warps, up to kSumThreads) of kSumRows rows
int t3_threads2d(int r) { return warps_for(r - 1, kSumThreads); }
int t3_col_blocks(int r) { return (r - 1 + t3_threads2d(r) - 1) / t3_threads2d(r); }
int t3_chunks2d(int r) { return t3_col_blocks(r) * ((r - 1 + kSumRows - 1) / kSumRows); }

dim3 grid_of(const Grid& g, int cx, int cy) {
  return dim3((cx + g.bx - 1) / g.bx, (cy + g.by - 1) / g.by, g.nb);
}

}  // namespace

void nload_density2d(const Grid& g, const double* u, double* nl, const Density2D& b,
                     cudaStream_t s) {
  if (!star2d_rows(g)) {
    k_nload_density2d_node<<<grid_of(g, g.n - 1, g.n - 1), dim3(g.bx, g.by), 0, s>>>(
        g.n, g.pitch, g.stride, g.h * g.h / 120.0, g.h * g.h / 180.0, g.h * g.h / 360.0, u, nl,
        b.C, b.E, b.N, b.NE);
    return;
  }
  star2d_dispatch(g, [&](auto r) {
    k_nload_density2d<r><<<star2d_grid(g.n, g.nb, r), star2d_block(), 0, s>>>(
        g.n, g.pitch, g.stride, g.h * g.h / 120.0, g.h * g.h / 360.0, u, nl, b.C, b.E, b.N,
        b.NE);
  });
}

void gather_level1_2d(const Grid& g1, const double* gA_pad, const double* gM_pad,
                      const double* t1_pad, const Density2D& b1, double* gA, double* gM,
                      double* t1, double* B1, cudaStream_t s) {
  const int m = g1.n - 1;
  k_gather_level1_2d<<<dim3((m * m + 63) / 64, g1.nb), 64, 0, s>>>(
      g1.n, g1.pitch, g1.stride, gA_pad, gM_pad, t1_pad, b1, gA, gM, t1, B1);
}

size_t t3_partials2d(const Grid& fine, int n1) {
  return (size_t)n1 * n1 * ((size_t)t3_chunks2d(fine.n / n1) * kInner + kLines);
}

void t3_moments2d(const Grid& fine, int n1, const double* u, const double* pw,
                  const double* map, double* partials, double* t3, cudaStream_t s) {
  const int r = fine.n / n1, chunks = t3_chunks2d(r);
  const size_t pst = t3_partials2d(fine, n1);
  k_t3_sums2d<<<dim3(chunks + 1, n1 * n1, fine.nb), t3_threads2d(r), 0, s>>>(
      fine.pitch, n1, r, fine.stride, pst, u, pw, partials, t3_col_blocks(r), chunks);
  k_t3_finalize2d<<<dim3(2 * n1 * n1, fine.nb), 32, 0, s>>>(
      n1 * n1, chunks, fine.h * fine.h, pst, (size_t)2 * n1 * n1 * 10, partials, map, t3);
}

// Host: moments m_ij = int_K lambda_v (ds)^i (dt)^j over each star triangle of a node (fine
// units, h = 1), summed per class of each coarse-triangle type.  Exact, from the barycentric
// monomial rule int_K lambda^alpha = 2|K| alpha! / (|alpha| + 2)! with |K| = 1/2.
void t3_class_moments2d(double out[2 * 7 * 10]) {
  // star triangles as neighbour pairs of the hexagon E, NE, N, W, SW, S
  const int nb[6][2] = {{1, 0}, {1, 1}, {0, 1}, {-1, 0}, {-1, -1}, {0, -1}};
  auto fact = [](int k) {
    double r = 1.0;
    for (int i = 2; i <= k; ++i) r *= i;
    return r;
  };
  auto binom = [&](int n, int k) { return fact(n) / (fact(k) * fact(n - k)); };
  double star[6][10];
  const int mk[10] = {0, 1, 0, 2, 1, 0, 3, 2, 1, 0}, ml[10] = {0, 0, 1, 0, 1, 2, 0, 1, 2, 3};
  for (int t = 0; t < 6; ++t) {
    const int* q = nb[t];
    const int* rr = nb[(t + 1) % 6];
    for (int m = 0; m < 10; ++m) {
      const int i = mk[m], j = ml[m];
      // lambda_v (q_s lq + r_s lr)^i (q_t lq + r_t lr)^j, expanded
      double acc = 0.0;
      for (int a = 0; a <= i; ++a)
        for (int b = 0; b <= j; ++b) {
          const double coef = binom(i, a) * binom(j, b) * pow((double)q[0], a) *
                              pow((double)rr[0], i - a) * pow((double)q[1], b) *
                              pow((double)rr[1], j - b);
          if (coef == 0.0) continue;
          const int eq = a + b, er = (i - a) + (j - b);  // exponents of lambda_q, lambda_r
          acc += coef * 2.0 * 0.5 * fact(1) * fact(eq) * fact(er) / fact(1 + eq + er + 2);
        }
      star[t][m] = acc;
    }
  }
  // classes: 0 interior, 1 edge A, 2 edge B, 3 diagonal, 4..6 vertices (see the T3 class sums above);
  // star triangle t = pair (nb[t], nb[t+1]): 0 (E,NE) 1 (NE,N) 2 (N,W) 3 (W,SW) 4 (SW,S) 5 (S,E)
  const int sets[2][7][6] = {
      {{0, 1, 2, 3, 4, 5}, {0, 1, 2, -1}, {2, 3, 4, -1}, {4, 5, 0, -1}, {0, -1}, {2, -1}, {4, -1}},
      {{0, 1, 2, 3, 4, 5}, {5, 0, 1, -1}, {3, 4, 5, -1}, {1, 2, 3, -1}, {1, -1}, {3, -1}, {5, -1}}};
  for (int T = 0; T < 2; ++T)
    for (int c = 0; c < 7; ++c)
      for (int m = 0; m < 10; ++m) {
        double s = 0.0;
        for (int e = 0; e < 6 && sets[T][c][e] >= 0; ++e) s += star[sets[T][c][e]][m];
        if (c == 0) {
          s = 0.0;
          for (int e = 0; e < 6; ++e) s += star[e][m];
        }
        out[(T * 7 + c) * 10 + m] = s;
      }
}

// Host: table of (x / r)^m, m = 0..3, x = 0..r (exact: r is a power of two times n1-free)
void t3_power_table(int r, double* out) {
  for (int x = 0; x <= r; ++x) {
    const double v = (double)x / r;
    out[4 * x + 0] = 1.0;
    out[4 * x + 1] = v;
    out[4 * x + 2] = v * v;
    out[4 * x + 3] = v * v * v;
  }
}

// Host: the linear map from the 25 class sums to T3 (without the h^2 factor) for one level:
//   T3_abc = sum_class sum_{i+j<=3} m^class_ij r^-(i+j) / (i! j!)
//            sum_{k+l<=3} c^abc_kl (k)_i (l)_j S^class_{k-i, l-j},
// with q_abc(sg, tg) = mu_a mu_b mu_c = sum c_kl sg^k tg^l and (k)_i the falling factorial;
// S^class_{a,b} = sum over the class of u sg^a tg^b, one of the 25 sums or zero.
void t3_map2d(int r, double out[2 * 10 * 25]) {
  double mom[2 * 7 * 10];
  t3_class_moments2d(mom);
  const int mk[10] = {0, 1, 0, 2, 1, 0, 3, 2, 1, 0}, ml[10] = {0, 0, 1, 0, 1, 2, 0, 1, 2, 3};
  const double fall[4][4] = {{1, 0, 0, 0}, {1, 1, 0, 0}, {1, 2, 2, 0}, {1, 3, 6, 6}};
  const double fact[4] = {1, 1, 2, 6};
  // index of S^class_{a,b} among the 25 sums (-1: identically zero); see the T3 class sums above
  auto sum_index = [](int T, int cls, int a, int b) -> int {
    switch (cls) {
      case 0: { const int d = a + b; return d * (d + 1) / 2 + b; }
      case 1: return T == 0 ? (b == 0 ? 10 + a : -1) : (a == 0 ? 10 + b : -1);
      case 2: return T == 0 ? 14 + b : 14 + a;
      case 3: return 18 + a + b;
      case 4: return (a == 0 && b == 0) ? 22 : -1;
      case 5: return T == 0 ? (b == 0 ? 23 : -1) : 23;
      default: return T == 0 ? 24 : (a == 0 ? 24 : -1);
    }
  };
  for (int i = 0; i < 2 * 10 * 25; ++i) out[i] = 0.0;
  for (int T = 0; T < 2; ++T) {
    double mu[3][3];
    if (T == 0) {
      const double v[3][3] = {{1, -1, 0}, {0, 1, -1}, {0, 0, 1}};
      for (int x = 0; x < 3; ++x) for (int y = 0; y < 3; ++y) mu[x][y] = v[x][y];
    } else {
      const double v[3][3] = {{1, 0, -1}, {0, 1, 0}, {0, -1, 1}};
      for (int x = 0; x < 3; ++x) for (int y = 0; y < 3; ++y) mu[x][y] = v[x][y];
    }
    int e = 0;
    for (int a = 0; a < 3; ++a)
      for (int b = a; b < 3; ++b)
        for (int c = b; c < 3; ++c, ++e) {
          double cq[4][4] = {};
          cq[0][0] = 1.0;
          const int f3[3] = {a, b, c};
          for (int f = 0; f < 3; ++f) {
            double nq[4][4] = {};
            const double* m = mu[f3[f]];
            for (int k = 0; k < 4; ++k)
              for (int l = 0; l + k < 4; ++l) {
                if (cq[k][l] == 0.0) continue;
                nq[k][l] += cq[k][l] * m[0];
                if (k + l + 1 < 4) {
                  nq[k + 1][l] += cq[k][l] * m[1];
                  nq[k][l + 1] += cq[k][l] * m[2];
                }
              }
            for (int k = 0; k < 4; ++k) for (int l = 0; l < 4; ++l) cq[k][l] = nq[k][l];
          }
          double* row = out + ((size_t)T * 10 + e) * 25;
          for (int cls = 0; cls < 7; ++cls)
            for (int q = 0; q < 10; ++q) {
              const int i = mk[q], j = ml[q];
              const double mij = mom[(T * 7 + cls) * 10 + q];
              if (mij == 0.0) continue;
              const double w = mij * pow((double)r, -(i + j)) / (fact[i] * fact[j]);
              for (int k = i; k < 4; ++k)
                for (int l = j; l + k < 4; ++l) {
                  if (cq[k][l] == 0.0) continue;
                  const int si = sum_index(T, cls, k - i, l - j);
                  if (si >= 0) row[si] += w * cq[k][l] * fall[k][i] * fall[l][j];
                }
            }
        }
  }
}

}  // namespace fmg
