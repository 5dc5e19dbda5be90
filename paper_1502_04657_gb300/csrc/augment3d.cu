// Fine-grid pass of the augmented nonlinear problem on the 3D Kuhn mesh: the per-coarse-
// tetrahedron integrals T3^T_abc = int_T u~ mu_a mu_b mu_c (the other moments, T0, T1 and
// the density stencil B(u~), come from grid3d.cu exactly as in 2D, see augment2d.cu).
//
// Coarse cell (I,J,L) holds 6 Kuhn tetrahedra T_s = {x_s0 >= x_s1 >= x_s2}; in the chain
// coordinates (a, b, c) = (x_s0, x_s1, x_s2) / r of a fine node (r fine cells per coarse
// cell) the barycentrics are mu = (1 - a, a - b, b - c, c) for every s, and the Kuhn mesh is
// symmetric under axis permutations, so one description serves all six.  T3 is linear in u~:
//   T3^T = sum_v u~_v int_T phi_v q,   q = mu_a mu_b mu_c (a cubic),
// and a Taylor expansion of q about node v is exact: int_T phi_v q = sum_{|b|<=3} D^b q(v)/b!
// m_b, m_b the moments of phi_v over the star tetrahedra of v inside T.  Those depend only
// on v's class - interior of T, one of 4 faces, 6 edges or 4 vertices - so T3 is a fixed
// linear map of the 15 x 20 class monomial sums S^class_g = sum u~ (a,b,c)^g, |g| <= 3.
#include <math.h>

#include <algorithm>
#include <map>
#include <vector>

#include "fmg_internal.h"
#include "reduce_dev.cuh"

namespace fmg {
namespace {

constexpr int kThreads = 256;
constexpr int kMono = 20;       // monomials of degree <= 3 in 3 variables
constexpr int kClasses = 15;    // interior, F0..F3, E01 E02 E03 E12 E13 E23, V0..V3
constexpr int kPerm[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
__constant__ int kPermDev[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};

// monomial order: degree 0; a b c; a^2 ab ac b^2 bc c^2; a^3 a^2b a^2c ab^2 abc ac^2 b^3 b^2c bc^2 c^3
__device__ __forceinline__ void monomials(double a, double b, double c, double* m) {
  m[0] = 1.0;
  m[1] = a; m[2] = b; m[3] = c;
  m[4] = a * a; m[5] = a * b; m[6] = a * c; m[7] = b * b; m[8] = b * c; m[9] = c * c;
  m[10] = m[4] * a; m[11] = m[4] * b; m[12] = m[4] * c; m[13] = a * m[7]; m[14] = m[5] * c;
  m[15] = a * m[9]; m[16] = m[7] * b; m[17] = m[7] * c; m[18] = b * m[9]; m[19] = m[9] * c;
}

// Interior class: a thread takes (x0, x2) lines of the coarse cell along x1, x0 fastest across
// the threads (coalesced loads), and adds their monomial sums before one block reduction.  x1
// runs through three tetrahedra of the line, x1 < f2, f2 < x1 < f1 and x1 > f1 with f1 > f2 the
// line's fixed coordinates, so one pass over a line serves all three, every node is read and
// summed once, and the lanes of a warp read the same x1 (a pass per tetrahedron that started
// each lane at its own x1 read uncoalesced and spent most of its FP64 slots on lanes outside
// the tetrahedron: 464 us on 16.6M nodes).  Lines with x0 > x2 and x0 < x2 lie in different
// tetrahedra and go to different blocks; their index runs over the pairs f1 > f2.  Every
// monomial is (powers of f1 / r and f2 / r) x (a power of x1 / r): a thread sums u (x1/r)^e,
// e = 0..3, with the powers from the level's table pw (4 FP64 operations per node) and then
// adds the 3 x 20 monomial sums of its line.
__device__ constexpr int kExpDev[20][3] = {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {2, 0, 0},
                                       {1, 1, 0}, {1, 0, 1}, {0, 2, 0}, {0, 1, 1}, {0, 0, 2},
                                       {3, 0, 0}, {2, 1, 0}, {2, 0, 1}, {1, 2, 0}, {1, 1, 1},
                                       {1, 0, 2}, {0, 3, 0}, {0, 2, 1}, {0, 1, 2}, {0, 0, 3}};

__device__ __forceinline__ double pick4(double v0, double v1, double v2, double v3, int e) {
  return e == 0 ? v0 : (e == 1 ? v1 : (e == 2 ? v2 : v3));
}

// tetrahedron (kPerm index) of a line's phase: [x0 < x2][x1 < f2, f2 < x1 < f1, x1 > f1]
__constant__ int kPhaseTet[2][3] = {{1, 0, 2}, {4, 5, 3}};

constexpr int kLineThreads = 128;
constexpr int kLinesPerThread = 2;  // lines summed per thread before the block reduction

__global__ void __launch_bounds__(kLineThreads)
    k_t3_interior3d(int pf, long planef, int n1, int r, size_t st, size_t pst,
                    const double* __restrict__ u, const double* __restrict__ pw,
                    double* __restrict__ partials) {
  __shared__ double sh[2][kLineThreads];
  u += blockIdx.z * st;  // instance blockIdx.z
  partials += blockIdx.z * pst;
  const int cell = blockIdx.y >> 1, o = blockIdx.y & 1;  // o: x0 < x2
  const int I = cell % n1, J = (cell / n1) % n1, L = cell / (n1 * n1);
  double acc[3][kMono];
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int m = 0; m < kMono; ++m) acc[p][m] = 0.0;
  const int lines = (r - 1) * (r - 2) / 2;
  for (int line = blockIdx.x * blockDim.x + threadIdx.x; line < lines;
       line += gridDim.x * blockDim.x) {
    // line -> (g1, g2), 1 <= g2 < g1 <= r - 1, g2 fastest
    int g1 = (int)((sqrtf(8.0f * line + 1.0f) + 1.0f) * 0.5f);  // g1 - 1
    while (g1 * (g1 - 1) / 2 > line) --g1;
    while ((g1 + 1) * g1 / 2 <= line) ++g1;
    const int g2 = line - g1 * (g1 - 1) / 2 + 1;
    ++g1;
    // x0 < x2: x0 = g2, x2 = g1; x0 > x2: mirrored, so that x0 is fastest too
    const int x0 = o ? g2 : r - g2, x2 = o ? g1 : r - g1;
    const int f1 = max(x0, x2), f2 = min(x0, x2);
    const double* col =
        u + (size_t)(L * r + x2) * planef + (size_t)(J * r) * pf + (size_t)(I * r + x0);
    double m[4] = {0.0, 0.0, 0.0, 0.0}, m0[4], m1[4];  // the running phase, phases 0 and 1
    constexpr int kAhead = 8;
    for (int x1 = 1; x1 < r; x1 += kAhead) {
      double v[kAhead];
#pragma unroll
      for (int q = 0; q < kAhead; ++q) v[q] = x1 + q < r ? col[(size_t)(x1 + q) * pf] : 0.0;
#pragma unroll
      for (int q = 0; q < kAhead; ++q) {
        const int x = x1 + q;
        if (x < r) {
          if (x == f2) {  // the diagonal planes belong to the boundary classes
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              m0[e] = m[e];
              m[e] = 0.0;
            }
          } else if (x == f1) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              m1[e] = m[e];
              m[e] = 0.0;
            }
          } else {
            const double* p = pw + 4 * x;  // (x1/r)^e
            m[0] += v[q];
#pragma unroll
            for (int e = 1; e < 4; ++e) m[e] = fma(v[q], p[e], m[e]);
          }
        }
      }
    }
    double g[4][4];  // (f1/r)^i (f2/r)^j
    {
      const double *a = pw + 4 * f1, *b = pw + 4 * f2;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; i + j < 4; ++j) g[i][j] = i == 0 ? b[j] : (j == 0 ? a[i] : a[i] * b[j]);
    }
#pragma unroll
    for (int q = 0; q < kMono; ++q) {
      const int ea = kExpDev[q][0], eb = kExpDev[q][1], ec = kExpDev[q][2];
      acc[0][q] = fma(g[ea][eb], m0[ec], acc[0][q]);  // (a, b, c) = (f1, f2, x1)
      acc[1][q] = fma(g[ea][ec], m1[eb], acc[1][q]);  // (f1, x1, f2)
      acc[2][q] = fma(g[eb][ec], m[ea], acc[2][q]);   // (x1, f1, f2)
    }
  }
  // block totals of the 60 sums, 30 at a time (as block_sum_to)
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    double w[30];
#pragma unroll
    for (int q = 0; q < 30; ++q) w[q] = acc[(30 * h + q) / kMono][(30 * h + q) % kMono];
    sh[h][threadIdx.x] = warp_transpose_sum<30>(w);
  }
  __syncthreads();
  for (int q = threadIdx.x; q < 60; q += blockDim.x) {
    const int warps = blockDim.x >> 5, h = q / 30;
    double t = 0.0;
    for (int w = 0; w < warps; ++w) t += sh[h][w * 32 + q - 30 * h];
    const int tet = 6 * cell + kPhaseTet[o][q / kMono];
    partials[((size_t)tet * gridDim.x + blockIdx.x) * kMono + q % kMono] = t;
  }
}

// Boundary classes: block (class - 1, tet, instance).
//  * faces (F0..F3): two free chain coordinates p > q; a thread takes a row (fixed p) and
//    walks q (a fixed stride per class), summing u (q/r)^e, e = 0..3, then adds the row's 20 monomial sums (each
//    monomial is a power of p/r times a power of q/r on a face);
//  * edges: one free coordinate, a thread per node; vertices: one node.
// Chain coordinates (a, b, c) of each class as functions of the free ones p > q > 0 (r fine
// cells per coarse cell): faces F0 (r, p, q), F1 (p, p, q), F2 (p, q, q), F3 (p, q, 0); edges
// E01 (r, r, p), E02 (r, p, p), E03 (r, p, 0), E12 (p, p, p), E13 (p, p, 0), E23 (p, 0, 0);
// vertices (0,0,0), (r,0,0), (r,r,0), (r,r,r).
__global__ void __launch_bounds__(kThreads)
    k_t3_boundary3d(int pf, long planef, int n1, int r, size_t st, size_t pst,
                    const double* __restrict__ u, const double* __restrict__ pw,
                    double* __restrict__ partials) {
  __shared__ double sh[kThreads];
  u += blockIdx.z * st;  // instance blockIdx.z
  partials += blockIdx.z * pst;
  const int cls = 1 + blockIdx.x;
  const int tet = blockIdx.y;
  const int cell = tet / 6, s = tet % 6;
  const int I = cell % n1, J = (cell / n1) % n1, L = cell / (n1 * n1);
  const double* base = u + (size_t)(L * r) * planef + (size_t)(J * r) * pf + (size_t)I * r;
  // element strides of the chain coordinates (a, b, c)
  auto stride = [&](int q) {
    const int axis = kPermDev[s][q];
    return axis == 0 ? 1l : (axis == 1 ? (long)pf : planef);
  };
  const long sa = stride(0), sb = stride(1), sc = stride(2);
  double acc[kMono];
#pragma unroll
  for (int m = 0; m < kMono; ++m) acc[m] = 0.0;
  if (cls <= 4) {
    // face rows: p = 2 .. r - 1 (F0..F2) with q in (0, p), F0 with p < r; F3: a = p, b = q
    for (int p = 2 + threadIdx.x; p < r; p += blockDim.x) {
      // the row's first element and the stride of q, then u (q/r)^e over 0 < q < p, eight
      // loads in flight
      const double* row = base + (cls == 1 ? r * sa + p * sb : cls == 2 ? p * (sa + sb) : p * sa);
      const long sq = cls <= 2 ? sc : cls == 3 ? sb + sc : sb;
      double m0 = 0.0, m1 = 0.0, m2 = 0.0, m3 = 0.0;
      constexpr int kAhead = 8;
      for (int q0 = 1; q0 < p; q0 += kAhead) {
        double v[kAhead];
#pragma unroll
        for (int j = 0; j < kAhead; ++j) v[j] = q0 + j < p ? row[(q0 + j) * sq] : 0.0;
#pragma unroll
        for (int j = 0; j < kAhead; ++j)
          if (q0 + j < p) {
            const double* t = pw + 4 * (q0 + j);
            m0 += v[j];
            m1 = fma(v[j], t[1], m1);
            m2 = fma(v[j], t[2], m2);
            m3 = fma(v[j], t[3], m3);
          }
      }
      const double* g = pw + 4 * p;
#pragma unroll
      for (int k = 0; k < kMono; ++k) {
        const int ea = kExpDev[k][0], eb = kExpDev[k][1], ec = kExpDev[k][2];
        int ep, eq;  // exponents of p / r and q / r of a^ea b^eb c^ec on the face
        bool zero = false;
        switch (cls) {
          case 1: ep = eb; eq = ec; break;           // (r, p, q)
          case 2: ep = ea + eb; eq = ec; break;      // (p, p, q)
          case 3: ep = ea; eq = eb + ec; break;      // (p, q, q)
          default: ep = ea; eq = eb; zero = ec > 0; break;  // (p, q, 0)
        }
        if (!zero && ep <= 3 && eq <= 3)
          acc[k] = fma(g[ep], pick4(m0, m1, m2, m3, eq), acc[k]);
      }
    }
  } else {
    // edges (one free coordinate p in (0, r)) and vertices (one node)
    const bool vertex = cls >= 11;
    for (int p = 1 + threadIdx.x; vertex ? (p == 1 && threadIdx.x == 0) : p < r;
         p += blockDim.x) {
      int abc[3];
      switch (cls) {
        case 5: abc[0] = r; abc[1] = r; abc[2] = p; break;   // E01
        case 6: abc[0] = r; abc[1] = p; abc[2] = p; break;   // E02
        case 7: abc[0] = r; abc[1] = p; abc[2] = 0; break;   // E03
        case 8: abc[0] = p; abc[1] = p; abc[2] = p; break;   // E12
        case 9: abc[0] = p; abc[1] = p; abc[2] = 0; break;   // E13
        case 10: abc[0] = p; abc[1] = 0; abc[2] = 0; break;  // E23
        case 11: abc[0] = 0; abc[1] = 0; abc[2] = 0; break;  // V0
        case 12: abc[0] = r; abc[1] = 0; abc[2] = 0; break;  // V1
        case 13: abc[0] = r; abc[1] = r; abc[2] = 0; break;  // V2
        default: abc[0] = r; abc[1] = r; abc[2] = r; break;  // V3
      }
      const double val = base[abc[0] * sa + abc[1] * sb + abc[2] * sc];
      double m[kMono];
      monomials(pw[4 * abc[0] + 1], pw[4 * abc[1] + 1], pw[4 * abc[2] + 1], m);
#pragma unroll
      for (int k = 0; k < kMono; ++k) acc[k] = fma(val, m[k], acc[k]);
    }
  }
  block_sum_to<kMono>(acc, sh, partials + ((size_t)tet * (kClasses - 1) + blockIdx.x) * kMono);
}

// T3_e = h^3 sum_{class, g} map[e][class][g] S^class_g
__global__ void k_t3_finalize3d(int chunks, double h3, size_t pst, size_t tst,
                                const double* __restrict__ pin, const double* __restrict__ pbd,
                                const double* __restrict__ map, double* __restrict__ t3) {
  pin += blockIdx.y * pst;  // instance blockIdx.y
  pbd += blockIdx.y * pst;
  t3 += blockIdx.y * tst;
  const int tet = blockIdx.x;
  __shared__ double S[kClasses * kMono];
  for (int m = threadIdx.x; m < kMono; m += blockDim.x) {
    double acc = 0.0;
    for (int c = 0; c < chunks; ++c) acc += pin[((size_t)tet * chunks + c) * kMono + m];
    S[m] = acc;
  }
  for (int e = threadIdx.x; e < (kClasses - 1) * kMono; e += blockDim.x)
    S[kMono + e] = pbd[(size_t)tet * (kClasses - 1) * kMono + e];
  __syncthreads();
  // eight lanes per entry, each every eighth term (a lane per entry was one chain of 300)
  const int e = threadIdx.x >> 3, part = threadIdx.x & 7;
  const double* row = map + (size_t)e * kClasses * kMono;
  double acc = 0.0;
#pragma unroll 4
  for (int q = part; q < kClasses * kMono; q += 8) acc = fma(row[q], S[q], acc);
  for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (part == 0) t3[(size_t)tet * 20 + e] = h3 * acc;
}

// Interior: a block takes kLinesPerThread lines per thread (whole warps, up to kLineThreads)
// of the (r - 1)(r - 2) / 2 lines of a cell with x0 < x2 (or x0 > x2).  Boundary: the face rows
// and edge nodes of a class number fewer than r, so a block of boundary_threads(r) covers them
// in one or a few passes.
int interior_threads(int r) { return warps_for((long)(r - 1) * (r - 2) / 2, kLineThreads); }
int interior_chunks(int r) {
  const long lines = (long)(r - 1) * (r - 2) / 2;
  const long per_block = (long)interior_threads(r) * kLinesPerThread;
  return std::max(1, (int)((lines + per_block - 1) / per_block));
}
int boundary_threads(int r) { return warps_for(r, kThreads); }

// ---- host: class moments and the linear map ---------------------------------------------
// Polynomials in the 4 barycentrics of a tetrahedron, exponents packed in a key.
using Poly = std::map<int, double>;
int key(const int* e) { return e[0] | e[1] << 4 | e[2] << 8 | e[3] << 12; }
double fact(int k) {
  double r = 1.0;
  for (int i = 2; i <= k; ++i) r *= i;
  return r;
}
Poly mul(const Poly& x, const Poly& y) {
  Poly z;
  for (auto& a : x)
    for (auto& b : y) {
      int e[4];
      for (int i = 0; i < 4; ++i) e[i] = ((a.first >> (4 * i)) & 15) + ((b.first >> (4 * i)) & 15);
      z[key(e)] += a.second * b.second;
    }
  return z;
}
// int_K lambda^alpha for a tetrahedron of volume 1/6 (fine units): 6 |K| alpha! / (|alpha|+3)!
double integrate(const Poly& x) {
  double s = 0.0;
  for (auto& a : x) {
    int tot = 0;
    double num = 1.0;
    for (int i = 0; i < 4; ++i) {
      const int ei = (a.first >> (4 * i)) & 15;
      tot += ei;
      num *= fact(ei);
    }
    s += a.second * num / fact(tot + 3);
  }
  return s;
}

const int kMonoExp[20][3] = {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {2, 0, 0},
                             {1, 1, 0}, {1, 0, 1}, {0, 2, 0}, {0, 1, 1}, {0, 0, 2},
                             {3, 0, 0}, {2, 1, 0}, {2, 0, 1}, {1, 2, 0}, {1, 1, 1},
                             {1, 0, 2}, {0, 3, 0}, {0, 2, 1}, {0, 1, 2}, {0, 0, 3}};

int mono_index(int a, int b, int c) {
  for (int q = 0; q < 20; ++q)
    if (kMonoExp[q][0] == a && kMonoExp[q][1] == b && kMonoExp[q][2] == c) return q;
  return -1;
}

// Moments m[class][g] = sum over the star tetrahedra of a class-representative node that lie
// in T = {R >= x0 >= x1 >= x2 >= 0} of int_K lambda_v (x - x_v)^g (fine units).
void class_moments3d(double mom[kClasses][kMono]) {
  const int R = 12;
  const int rep[kClasses][3] = {{9, 6, 3},   {12, 8, 4}, {8, 8, 4},  {8, 4, 4},   {8, 4, 0},
                                {12, 12, 6}, {12, 6, 6}, {12, 6, 0}, {6, 6, 6},   {6, 6, 0},
                                {6, 0, 0},   {0, 0, 0},  {12, 0, 0}, {12, 12, 0}, {12, 12, 12}};
  for (int cls = 0; cls < kClasses; ++cls) {
    for (int g = 0; g < kMono; ++g) mom[cls][g] = 0.0;
    const int* v = rep[cls];
    // the 8 cells around v and their Kuhn tetrahedra
    for (int o = 0; o < 8; ++o) {
      const int c0[3] = {v[0] - (o & 1), v[1] - ((o >> 1) & 1), v[2] - ((o >> 2) & 1)};
      for (int s = 0; s < 6; ++s) {
        int vt[4][3];
        for (int a = 0; a < 3; ++a) vt[0][a] = c0[a];
        for (int a = 0; a < 3; ++a) vt[1][a] = vt[0][a] + (a == kPerm[s][0]);
        for (int a = 0; a < 3; ++a) vt[2][a] = vt[1][a] + (a == kPerm[s][1]);
        for (int a = 0; a < 3; ++a) vt[3][a] = c0[a] + 1;
        int iv = -1;
        for (int w = 0; w < 4; ++w)
          if (vt[w][0] == v[0] && vt[w][1] == v[1] && vt[w][2] == v[2]) iv = w;
        if (iv < 0) continue;
        double cen[3] = {0, 0, 0};
        for (int w = 0; w < 4; ++w)
          for (int a = 0; a < 3; ++a) cen[a] += vt[w][a] / 4.0;
        if (!(R > cen[0] && cen[0] > cen[1] && cen[1] > cen[2] && cen[2] > 0)) continue;
        // x - x_v = sum_w lambda_w (x_w - x_v)
        Poly lin[3];
        for (int a = 0; a < 3; ++a)
          for (int w = 0; w < 4; ++w) {
            const double d = vt[w][a] - v[a];
            if (d == 0.0) continue;
            int e[4] = {0, 0, 0, 0};
            e[w] = 1;
            lin[a][key(e)] += d;
          }
        int ev[4] = {0, 0, 0, 0};
        ev[iv] = 1;
        for (int g = 0; g < kMono; ++g) {
          Poly p;
          p[key(ev)] = 1.0;
          for (int a = 0; a < 3; ++a)
            for (int k = 0; k < kMonoExp[g][a]; ++k) p = mul(p, lin[a]);
          mom[cls][g] += integrate(p);
        }
      }
    }
  }
}

// Every class sum is taken with the node's actual chain coordinates, so S^class_g is simply
// slot class * 20 + g.
void class_sum_terms(int cls, int ga, int gb, int gc, std::vector<std::pair<int, double>>& out) {
  out.clear();
  const int q = mono_index(ga, gb, gc);
  if (q >= 0) out.push_back({cls * kMono + q, 1.0});
}

}  // namespace

size_t t3_partials3d(const Grid& fine, int n1) {
  const int r = fine.n / n1;
  const size_t tets = (size_t)6 * n1 * n1 * n1;
  return tets * kMono * ((size_t)interior_chunks(r) + (kClasses - 1));
}

void t3_moments3d(const Grid& fine, int n1, const double* u, const double* pw,
                  const double* map, double* partials, double* t3, cudaStream_t s) {
  const int r = fine.n / n1;
  const int tets = 6 * n1 * n1 * n1;
  const int chunks = interior_chunks(r);
  const long planef = (long)(fine.n + 1) * fine.pitch;
  const size_t pst = t3_partials3d(fine, n1);  // per instance
  double* pin = partials;
  double* pbd = partials + (size_t)tets * chunks * kMono;
  k_t3_interior3d<<<dim3(chunks, tets / 3, fine.nb), interior_threads(r), 0, s>>>(
      fine.pitch, planef, n1, r, fine.stride, pst, u, pw, pin);
  k_t3_boundary3d<<<dim3(kClasses - 1, tets, fine.nb), boundary_threads(r), 0, s>>>(
      fine.pitch, planef, n1, r, fine.stride, pst, u, pw, pbd);
  k_t3_finalize3d<<<dim3(tets, fine.nb), 160, 0, s>>>(chunks, fine.h * fine.h * fine.h, pst,
                                                     (size_t)tets * 20, pin, pbd, map, t3);
}

// Host: map[e][class][g] for T3_e = h^3 sum map S^class_g (r fine cells per coarse cell),
//   T3_e = sum_class sum_{|b|<=3} m^class_b r^-|b| / b! sum_{|g|<=3} c^e_g (g)_b S^class_{g-b},
// c^e the monomial coefficients of q_e = mu_a mu_b mu_c in chain coordinates and (g)_b the
// falling factorials.
void t3_map3d(int r, double* out) {
  double mom[kClasses][kMono];
  class_moments3d(mom);
  for (int i = 0; i < 20 * kClasses * kMono; ++i) out[i] = 0.0;
  // barycentrics (const, a, b, c) coefficients
  const double mu[4][4] = {{1, -1, 0, 0}, {0, 1, -1, 0}, {0, 0, 1, -1}, {0, 0, 0, 1}};
  auto ff = [](int g, int b) {  // falling factorial (g)_b
    double r = 1.0;
    for (int i = 0; i < b; ++i) r *= (g - i);
    return r;
  };
  std::vector<std::pair<int, double>> terms;
  int e = 0;
  for (int x = 0; x < 4; ++x)
    for (int y = x; y < 4; ++y)
      for (int z = y; z < 4; ++z, ++e) {
        double cq[4][4][4] = {};
        cq[0][0][0] = 1.0;
        const int f3[3] = {x, y, z};
        for (int f = 0; f < 3; ++f) {
          double nq[4][4][4] = {};
          const double* m = mu[f3[f]];
          for (int a = 0; a < 4; ++a)
            for (int b = 0; a + b < 4; ++b)
              for (int c = 0; a + b + c < 4; ++c) {
                if (cq[a][b][c] == 0.0) continue;
                nq[a][b][c] += cq[a][b][c] * m[0];
                if (a + b + c + 1 < 4) {
                  nq[a + 1][b][c] += cq[a][b][c] * m[1];
                  nq[a][b + 1][c] += cq[a][b][c] * m[2];
                  nq[a][b][c + 1] += cq[a][b][c] * m[3];
                }
              }
          for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b)
              for (int c = 0; c < 4; ++c) cq[a][b][c] = nq[a][b][c];
        }
        double* row = out + (size_t)e * kClasses * kMono;
        for (int cls = 0; cls < kClasses; ++cls)
          for (int bq = 0; bq < kMono; ++bq) {
            const double mb = mom[cls][bq];
            if (mb == 0.0) continue;
            const int b0 = kMonoExp[bq][0], b1 = kMonoExp[bq][1], b2 = kMonoExp[bq][2];
            const double w = mb * pow((double)r, -(b0 + b1 + b2)) / (fact(b0) * fact(b1) * fact(b2));
            for (int g0 = b0; g0 < 4; ++g0)
              for (int g1 = b1; g0 + g1 < 4; ++g1)
                for (int g2 = b2; g0 + g1 + g2 < 4; ++g2) {
                  const double cg = cq[g0][g1][g2];
                  if (cg == 0.0) continue;
                  const double coef = w * cg * ff(g0, b0) * ff(g1, b1) * ff(g2, b2);
                  class_sum_terms(cls, g0 - b0, g1 - b1, g2 - b2, terms);
                  for (auto& t : terms) row[t.first] += coef * t.second;
                }
          }
      }
}

}  // namespace fmg
