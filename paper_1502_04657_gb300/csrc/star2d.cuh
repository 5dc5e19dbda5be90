// Column-streamed star sums of the 2D cubic load and density stencil (device code shared by
// grid2d.cu and augment2d.cu).
//
// On the right-triangle mesh the star of node p is the hexagon of neighbours E, NE, N, W,
// SW, S; each consecutive pair (a, b) closes one triangle with p, and (a, b) is an edge of
// the mesh opposite p.  The exact cubic load int u^3 phi_p (Section 2, P1 functions,
// barycentric monomial integrals) is
//   |K|/60 [u^2 (24u + 3 M1) + u sum_e F_e + sum_e E3_e]
// over the six opposite edges e = (a, b), with s_e = a + b, F_e = s_e^2 + a^2 + b^2
// (= 2 (a^2 + ab + b^2)), E3_e = s_e (a^2 + b^2) and M1 = sum_e s_e (twice the neighbour
// sum).  These three numbers depend on the edge alone, and every mesh edge is opposite two
// nodes, so each is computed once per edge instead of once per node that needs it: a node
// owns its edges towards E (H), N (V) and NE (D) and takes the other opposite edges from
// the lanes beside it and the rows below it.
//
// Layout of the work: a warp covers 32 consecutive columns (lanes 1..30 produce, lanes 0 and
// 31 only supply edges and neighbour values) and R consecutive rows, which one thread walks
// upwards; edges of the rows before and after the block come from one extra row at each
// end.  Every node's arithmetic is the same whichever lane and block computes it, so the
// result does not depend on the launch shape.
#pragma once
#include <type_traits>

#include "fixed.cuh"
#include "fmg_internal.h"

namespace fmg {

constexpr int kFx2 = 61;  // fixed-point format of the walk (fixed.cuh)
constexpr int kShortLoad2 = 36, kShortDensity2 = 44;  // results that a node takes in FP64
constexpr int kShortMass2 = 41;  // 12 u + M1 of the right-hand side

template <typename T>
struct StarEdge {
  T s, F, E3;
};

// what a producing node hands to its epilogue
template <typename T>
struct Star2D {
  T u, q;            // u_p and u_p^2
  T M1, SF, SE;      // sums over the six opposite edges of s, F and E3
  StarEdge<T> H, V, D;  // p's own edges towards E, N and NE
  T uE, uN, uW, uS, uNE;  // neighbour values (apexes of the density stencil's edges)
  T qE, qN, qW, qS, qNE;
};

__device__ __forceinline__ double shfl_up1(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double shfl_down1(double v) {
  return __shfl_down_sync(0xffffffffu, v, 1);
}
template <typename T>
__device__ __forceinline__ StarEdge<T> shfl_up1(const StarEdge<T>& e) {
  return {shfl_up1(e.s), shfl_up1(e.F), shfl_up1(e.E3)};
}
template <typename T>
__device__ __forceinline__ StarEdge<T> shfl_down1(const StarEdge<T>& e) {
  return {shfl_down1(e.s), shfl_down1(e.F), shfl_down1(e.E3)};
}

template <typename T>
__device__ __forceinline__ StarEdge<T> star_edge(T a, T qa, T b, T qb) {
  const T s = a + b, qs = qa + qb;
  return {s, fma(s, s, qs), s * qs};
}

// the bracket of the cubic load, u^2 (24u + 3 M1) + u sum F + sum E3
template <typename T>
__device__ __forceinline__ T star_cubic(const Star2D<T>& p) {
  return fma(T(3), p.q * fma(T(8), p.u, p.M1), fma(p.u, p.SF, p.SE));
}

constexpr int kStarWarps = 4;   // warps of a block, stacked in y
constexpr int kStarCols = 30;   // producing columns of a warp

inline dim3 star2d_grid(int n, int nb, int rows) {
  return dim3((n - 1 + kStarCols - 1) / kStarCols,
              (n - 1 + rows * kStarWarps - 1) / (rows * kStarWarps), nb);
}
inline dim3 star2d_block() { return dim3(32, kStarWarps); }

// Rows one thread walks on a level (the kernels' template argument), or 0: node by node in FP64.
// A walk is a chain of dependent row steps (about 0.8 us each), so small levels take short
// walks, which are more and shorter chains but compute more rows twice (R + 2 for R).  The
// density kernel on one instance took, in us, node by node 8.2, 14.4 and 47 at n = 128, 256 and
// 512, 16 in 16-row walks at each, and 6.1, 6.5 (R = 4) and 12.7 (R = 8) at n = 112, 224 and
// 448; filled with instances, 8 rows cost 8% more per node than 16.
// The rule depends on n alone, so an instance gives the same bits alone and in a batch.
// (FMG_FLAG_STAR_WALKS walks below n = 64 as well.)
inline int star2d_rows(const Grid& lv) {
  return lv.n >= 1024 ? 16 : lv.n >= 256 ? 8 : lv.n >= 64 || lv.walk_all ? 4 : 0;
}
// f(std::integral_constant<int, rows>) for the level's rows
template <typename F>
void star2d_dispatch(const Grid& lv, F f) {
  switch (star2d_rows(lv)) {
    case 16: f(std::integral_constant<int, 16>()); break;
    case 8: f(std::integral_constant<int, 8>()); break;
    default: f(std::integral_constant<int, 4>());
  }
}

// The fixed-point exponent of this warp's tile (its 32 columns, R rows and the row before and
// after them), or kFxNone; uniform over the warp.  The walk reads the tile again from L1.  LOAD: half of the
// columns far below the largest value leave the tile to FP64.
template <int R, bool LOAD>
__device__ __forceinline__ int star2d_exponent(int n, int pitch, size_t st, const double* u) {
  const int i = kStarCols * blockIdx.x + threadIdx.x;
  const int j0 = 1 + R * (blockIdx.y * blockDim.y + threadIdx.y);
  const double* p = u + blockIdx.z * st + i;
  FxTop m;
#pragma unroll
  for (int t = 0; t <= R + 2; ++t) {
    const int r = j0 - 1 + t;
    if (i <= n && r <= n) m.add(p[(size_t)r * pitch]);
  }
  const FxTop column = m;
  m.warp_max();
  const int e = m.exponent();
  return LOAD && 2 * __popc(__ballot_sync(0xffffffffu, column.far_below(e))) > 32 ? kFxNone : e;
}

// The walk in fixed point.  Sums of fixed-point values are exact, so the three opposite edges a
// node takes from the row below it, the two of its own row and the one of the row above are
// added up as the rows pass (start, acc), and neighbours' edges are exchanged as sums: 12
// registers of state where eight carried edges take 48, and 9 exchanged words a row where the
// FP64 walk exchanges 12.
struct Star2DFx {
  using T = fx<kFx2>;
  T u, q, M1, SF, SE;                            // as Star2D
  T Hs, HF, Vs, VF, Ds, DF;                      // own edges (density)
  T uE, uN, uW, uS, uNE, qE, qN, qW, qS, qNE;    // neighbours (density)
};

// In units of the tile's maximum: 8u + M1 <= 20 and 12u + M1 <= 24 (of 2^5 that fit in 63
// bits), the density sums <= 180 (of 2^8), the cubic load <= 120 (of 2^11).
__device__ __forceinline__ fx<kFx2> star_cubic(const Star2DFx& p) {
  return madd<3>(p.q * madd<8>(p.u, p.M1), fma(p.u, p.SF, p.SE));
}

template <int K>
__device__ __forceinline__ fx<K> shfl_up1(fx<K> v) {
  return fx<K>(__shfl_up_sync(0xffffffffu, v.v, 1));
}
template <int K>
__device__ __forceinline__ fx<K> shfl_down1(fx<K> v) {
  return fx<K>(__shfl_down_sync(0xffffffffu, v.v, 1));
}
// e: the warp's exponent (star2d_exponent).  Calls out(k, star) as star2d_walk does.
template <bool DENSITY, int R, typename Out>
__device__ __forceinline__ void star2d_walk_fx(int n, int pitch, size_t st,
                                               const double* __restrict__ u, int e, Out out) {
  using T = fx<kFx2>;
  const int lane = threadIdx.x;
  const int i = kStarCols * blockIdx.x + lane;
  const int j0 = 1 + R * (blockIdx.y * blockDim.y + threadIdx.y);
  if (j0 >= n) return;  // uniform over the warp
  const double scale = fx_pow2(T::B1 - e);
  const double* col = u + blockIdx.z * st + i;
  const bool produce = lane >= 1 && lane <= kStarCols && i <= n - 1;
  auto ld = [&](int r) { return i <= n && r <= n ? col[(size_t)r * pitch] : 0.0; };
  auto fix = [&](double v) { return T(__double2ll_rn(v * scale)); };
  const T zero(0);
  T u0 = fix(ld(j0 - 1)), q0 = u0 * u0;
  T u0R = shfl_down1(u0), q0R = shfl_down1(q0);
  double next = ld(j0);
  T um1 = zero, qm1 = zero, um2 = zero, qm2 = zero;
  T uRm1 = zero, qRm1 = zero, uLm1 = zero, qLm1 = zero;
  T Hs = zero, HF = zero, Vs = zero, VF = zero, Ds = zero, DF = zero;  // own edges, row r - 1
  T start[3] = {zero, zero, zero}, acc[3] = {zero, zero, zero};        // sums of (s, F, E3)
#pragma unroll 2
  for (int t = 0; t < R + 2; ++t) {
    const int r = j0 - 1 + t;
    const T u1 = fix(next);
    next = ld(r + 2);
    const T q1 = u1 * u1;
    const T u1R = shfl_down1(u1), q1R = shfl_down1(q1);
    T V[3], H[3], D[3];
    auto edge = [&](T a, T qa, T b, T qb, T* o) {
      const T s = a + b, qs = qa + qb;
      o[0] = s;
      o[1] = fma(s, s, qs);
      o[2] = s * qs;
    };
    edge(u0, q0, u1, q1, V);
    edge(u0, q0, u0R, q0R, H);
    edge(u0, q0, u1R, q1R, D);
    if (t >= 2 && produce && r - 1 <= n - 1) {
      Star2DFx p;
      p.u = um1;
      p.q = qm1;
      p.M1 = acc[0] + H[0];
      p.SF = acc[1] + H[1];
      p.SE = acc[2] + H[2];
      if (DENSITY) {
        p.Hs = Hs; p.HF = HF; p.Vs = Vs; p.VF = VF; p.Ds = Ds; p.DF = DF;
        p.uE = uRm1; p.qE = qRm1;
        p.uN = u0; p.qN = q0;
        p.uW = uLm1; p.qW = qLm1;
        p.uS = um2; p.qS = qm2;
        p.uNE = u0R; p.qNE = q0R;
      }
      out(blockIdx.z * st + (size_t)(r - 1) * pitch + i, p);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      acc[c] = start[c] + (shfl_up1(D[c]) + shfl_down1(V[c]));  // node r: its own row's edges
      start[c] = D[c] + shfl_up1(V[c] + H[c]);                  // node r + 1: the row below
    }
    if (DENSITY) {
      um2 = um1; qm2 = qm1;
      uRm1 = u0R; qRm1 = q0R;
      uLm1 = shfl_up1(u0); qLm1 = shfl_up1(q0);
      Hs = H[0]; HF = H[1]; Vs = V[0]; VF = V[1]; Ds = D[0]; DF = D[1];
    }
    um1 = u0; qm1 = q0;
    u0 = u1; q0 = q1;
    u0R = u1R; q0R = q1R;
  }
}

// node(k) for the nodes that a fixed-point walk of this warp left short of bits, or tile() for half
// of its nodes and more.  redo: one bit per row that the lane produced, the latest lowest.  The nodes
// are spread over the lanes: an FP64 instruction takes a warp the same time for one node as for 32.
template <int R, typename Node, typename Tile>
__device__ __forceinline__ void star2d_redo(int n, int pitch, size_t st, unsigned redo, Node node,
                                            Tile tile) {
  __shared__ unsigned short list[kStarWarps][32 * R];
  __shared__ int count[kStarWarps];
  if (!__any_sync(0xffffffffu, redo)) return;
  if (__reduce_add_sync(0xffffffffu, __popc(redo)) > kStarCols * R / 2) {
    tile();
    return;
  }
  const int lane = threadIdx.x, w = threadIdx.y;
  const int j0 = 1 + R * (blockIdx.y * blockDim.y + w), last = min(j0 + R, n) - 1;
  if (lane == 0) count[w] = 0;
  __syncwarp();
  for (; redo; redo &= redo - 1)
    list[w][atomicAdd(&count[w], 1)] = (unsigned short)(lane * R + (last - (__ffs(redo) - 1) - j0));
  __syncwarp();
  for (int q = lane; q < count[w]; q += 32)
    node(blockIdx.z * st + (size_t)(j0 + list[w][q] % R) * pitch + kStarCols * blockIdx.x +
         list[w][q] / R);
}

// Walks the rows of this thread's strip of instance blockIdx.z and calls out(k, star) for
// every interior node it produces (k = the node's index in the batched arrays).  blockDim = (32,
// kStarWarps).
template <typename T, int R, typename U, typename Out>
__device__ __forceinline__ void star2d_walk(int n, int pitch, size_t st, const U& u, Out out) {
  const int lane = threadIdx.x;
  const int i = kStarCols * blockIdx.x + lane;  // lane 0 = first produced column - 1
  const int j0 = 1 + R * (blockIdx.y * blockDim.y + threadIdx.y);
  if (j0 >= n) return;  // uniform over the warp
  const size_t base = blockIdx.z * st;
  const bool produce = lane >= 1 && lane <= kStarCols && i <= n - 1;
  auto ld = [&](int r) -> T {
    return (i <= n && r <= n) ? get<T>(u, base + (size_t)r * pitch + i) : T(0);
  };
  // row r = j0 - 1 + t: u0/q0 this column, u0R/q0R the next one, u0L/q0L the previous one
  T u0 = ld(j0 - 1);
  T q0 = u0 * u0;
  T u0R = shfl_down1(u0), q0R = shfl_down1(q0);
  // state carried from earlier rows (names say which row: m1 = r - 1, m2 = r - 2)
  T um1 = T(0), qm1 = T(0), um2 = T(0), qm2 = T(0);
  T uRm1 = T(0), qRm1 = T(0), uLm1 = T(0), qLm1 = T(0);
  StarEdge<T> Dm1{}, Dm2{}, VLm1{}, VLm2{}, HLm1{}, HLm2{}, DLm1{}, VRm1{}, Hm1{}, Vm1{};
#pragma unroll
  for (int t = 0; t < R + 2; ++t) {
    const int r = j0 - 1 + t;
    const T u1 = ld(r + 1);
    const T q1 = u1 * u1;
    const T u1R = shfl_down1(u1), q1R = shfl_down1(q1);
    const T u0L = shfl_up1(u0), q0L = shfl_up1(q0);
    const StarEdge<T> V = star_edge(u0, q0, u1, q1);
    const StarEdge<T> H = star_edge(u0, q0, u0R, q0R);
    const StarEdge<T> D = star_edge(u0, q0, u1R, q1R);
    const StarEdge<T> VL = shfl_up1(V), HL = shfl_up1(H), DL = shfl_up1(D), VR = shfl_down1(V);
    if (t >= 2 && produce && r - 1 <= n - 1) {
      // node (i, r - 1): opposite edges D(i, r-2), V(i-1, r-2), H(i-1, r-2), D(i-1, r-1),
      // V(i+1, r-1) and H(i, r)
      Star2D<T> p;
      p.u = um1;
      p.q = qm1;
      p.M1 = ((Dm2.s + VLm2.s) + (HLm2.s + DLm1.s)) + (VRm1.s + H.s);
      p.SF = ((Dm2.F + VLm2.F) + (HLm2.F + DLm1.F)) + (VRm1.F + H.F);
      p.SE = ((Dm2.E3 + VLm2.E3) + (HLm2.E3 + DLm1.E3)) + (VRm1.E3 + H.E3);
      p.H = Hm1;
      p.V = Vm1;
      p.D = Dm1;
      p.uE = uRm1;
      p.qE = qRm1;
      p.uN = u0;
      p.qN = q0;
      p.uW = uLm1;
      p.qW = qLm1;
      p.uS = um2;
      p.qS = qm2;
      p.uNE = u0R;
      p.qNE = q0R;
      out(base + (size_t)(r - 1) * pitch + i, p);
    }
    // shift the rows
    um2 = um1;
    qm2 = qm1;
    um1 = u0;
    qm1 = q0;
    uRm1 = u0R;
    qRm1 = q0R;
    uLm1 = u0L;
    qLm1 = q0L;
    Dm2 = Dm1;
    Dm1 = D;
    VLm2 = VLm1;
    VLm1 = VL;
    HLm2 = HLm1;
    HLm1 = HL;
    DLm1 = DL;
    VRm1 = VR;
    Hm1 = H;
    Vm1 = V;
    u0 = u1;
    q0 = q1;
    u0R = u1R;
    q0R = q1R;
  }
}

}  // namespace fmg
