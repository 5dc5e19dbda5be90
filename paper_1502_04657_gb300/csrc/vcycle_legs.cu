// The legs of the FP64 V-cycle on its middle levels, one kernel each: down (nu_pre damped Jacobi
// sweeps, the residual and its restriction) and up (prolongation and nu_post sweeps).
//
// Between the levels that run in one CTA (vcycle_small.cu, 2D) and those that fill the GPU, a
// level visit of seven launches (two sweeps, residual, P^T, P, two sweeps) costs their latency,
// 3 to 5 us each, and hardly any work.  Here a block owns 16 x 8 (4 x 4 x 4) fine nodes, keeps x
// of its tile in shared memory with a halo wide enough for every step and recomputes the halo
// instead of exchanging it (as vcycle32_mid.cu does in single precision).  Small tiles, because
// an SM's FP64 rate (2 lanes per clock) bounds a block: with nu = 2 a down leg costs 1.5 (2D) and
// 4 (3D) times the FP64 work, 0.8 and 2 us per block (8 x 8 x 4 nodes: 2.5 times, but 5 us).
// Every node is evaluated with the expressions of grid2d.cu / grid3d.cu in the same order, so the
// results are bit-identical to the separate kernels.  Measured: 2D legs of 64 to 256 cells 5.5 to
// 9 us, 3D ones of 8 and 16 cells 6 to 8.
//
// A halo holds nodes that other blocks own, so each leg reads x from one buffer and writes the
// other (the caller swaps them).
#include <utility>

#include "fmg_internal.h"

namespace fmg {
namespace {

template <int DIM>
struct Tile;
template <>
struct Tile<2> {
  static constexpr int kX = 16, kY = 8, kZ = 1, kDirs = 3, kThreads = 256;
};
template <>
struct Tile<3> {
  static constexpr int kX = 4, kY = 4, kZ = 4, kDirs = 7, kThreads = 256;
};

// the directions of the couplings (2D: X, Y, XY; 3D: X, Y, Z, XY, XZ, YZ, XYZ)
template <int DIM>
__device__ constexpr int dirx(int d) { return DIM == 2 ? d != 1 : (d == 0 || d == 3 || d == 4 || d == 6); }
template <int DIM>
__device__ constexpr int diry(int d) { return DIM == 2 ? d != 0 : (d == 1 || d == 3 || d == 5 || d == 6); }
template <int DIM>
__device__ constexpr int dirz(int d) { return DIM == 2 ? 0 : (d == 2 || d == 4 || d == 5 || d == 6); }

template <int DIM>
struct LegLevel {
  int n, pitch;
  size_t st;
  const double* a[DIM == 2 ? 4 : 8];  // diagonal, couplings with +d
  const double* dinv;
};

// A tile: origin (ox, oy, oz), extents w x h x d; element (x, y, z) is node (ox + x, ...).
template <int DIM>
struct Box {
  int ox, oy, oz, w, h, d;

  // halo: around the block's nodes and, in the down leg (plus = 1), the next one in each axis
  __device__ Box(int halo, int plus) {
    using T = Tile<DIM>;
    ox = 1 + blockIdx.x * T::kX - halo;
    oy = 1 + blockIdx.y * T::kY - halo;
    w = T::kX + plus + 2 * halo;
    h = T::kY + plus + 2 * halo;
    oz = 0;
    d = 1;
  }
  __device__ void set_z(int z0, int halo, int plus) {
    oz = z0 - halo;
    d = Tile<DIM>::kZ + plus + 2 * halo;
  }
  __device__ int elements() const { return w * h * d; }

  // f(e, i, j, l) for the interior nodes at distance >= b from the border (this thread's)
  template <typename F>
  __device__ __forceinline__ void each(int n, int b, F f) const {
    const int rw = w - 2 * b, rh = h - 2 * b, rd = DIM == 3 ? d - 2 * b : 1;
    for (int q = threadIdx.x; q < rw * rh * rd; q += blockDim.x) {
      const int r = q / rw, x = b + q - r * rw;
      const int zz = DIM == 3 ? r / rh : 0;
      const int y = b + r - zz * rh, z = DIM == 3 ? b + zz : 0;
      const int i = ox + x, j = oy + y, l = oz + z;
      if (i < 1 || i >= n || j < 1 || j >= n) continue;
      if (DIM == 3 && (l < 1 || l >= n)) continue;
      f((z * h + y) * w + x, i, j, l);
    }
  }
};

template <int DIM>
__device__ __forceinline__ size_t node(const LegLevel<DIM>& g, int ib, int i, int j, int l) {
  return ib * g.st + ((size_t)l * (DIM == 3 ? g.n + 1 : 0) + j) * g.pitch + i;
}

// f - L x at a node, as defect / defect3 of grid2d.cu / grid3d.cu
template <int DIM>
__device__ __forceinline__ double defect(const LegLevel<DIM>& g, size_t k, double f,
                                         const double* x, int e, int w, int h) {
  const long plane = DIM == 3 ? (long)(g.n + 1) * g.pitch : 0;
  double r = fma(-g.a[0][k], x[e], f);
#pragma unroll
  for (int d = 0; d < Tile<DIM>::kDirs; ++d) {
    const long o = dirx<DIM>(d) + (long)diry<DIM>(d) * g.pitch + dirz<DIM>(d) * plane;
    const int t = dirx<DIM>(d) + (diry<DIM>(d) + dirz<DIM>(d) * h) * w;
    r = fma(-g.a[1 + d][k], x[e + t], r);
    r = fma(-g.a[1 + d][k - o], x[e - t], r);
  }
  return r;
}

// x += omega D^-1 (f - L x) at the nodes at distance >= b from the border, from X into Y
template <int DIM>
__device__ __forceinline__ void sweep(const LegLevel<DIM>& g, int ib, const Box<DIM>& box, int b,
                                      const double* __restrict__ f, const double* X, double* Y) {
  box.each(g.n, b, [&](int e, int i, int j, int l) {
    const size_t k = node(g, ib, i, j, l);
    Y[e] = fma(g.dinv[k], defect(g, k, f[k], X, e, box.w, box.h), X[e]);
  });
}

// blockIdx.z: (instance, plane block)
template <int DIM>
__device__ __forceinline__ int locate(int n, int& z0) {
  const int zb = DIM == 3 ? (n - 1 + Tile<DIM>::kZ - 1) / Tile<DIM>::kZ : 1;
  const int ib = blockIdx.z / zb;
  z0 = DIM == 3 ? 1 + (int)(blockIdx.z - ib * zb) * Tile<DIM>::kZ : 0;
  return ib;
}

template <int DIM>
__global__ void __launch_bounds__(Tile<DIM>::kThreads)
    k_leg_down(const __grid_constant__ LegLevel<DIM> g, int pc, size_t stc, int nu, int zero,
               const double* __restrict__ f, const double* __restrict__ x,
               double* __restrict__ xo, double* __restrict__ fc) {
  extern __shared__ double sm[];
  using T = Tile<DIM>;
  int z0;
  const int ib = locate<DIM>(g.n, z0);
  const int halo = zero ? max(nu, 1) : nu + 1;
  Box<DIM> box(halo, 1);
  if (DIM == 3) box.set_z(z0, halo, 1);
  const int m = box.elements();
  double *X = sm, *Y = sm + m;
  for (int e = threadIdx.x; e < 2 * m; e += blockDim.x) sm[e] = 0.0;
  __syncthreads();
  if (!zero)
    box.each(g.n, 0, [&](int e, int i, int j, int l) { X[e] = x[node(g, ib, i, j, l)]; });
  else if (nu > 0)
    box.each(g.n, 0, [&](int e, int i, int j, int l) {
      const size_t k = node(g, ib, i, j, l);
      X[e] = g.dinv[k] * f[k];
    });
  __syncthreads();
  for (int t = zero ? 1 : 0; t < nu; ++t) {
    sweep(g, ib, box, zero ? t : t + 1, f, X, Y);
    __syncthreads();
    double* s = X;
    X = Y;
    Y = s;
  }
  // the block's own nodes of x, and the residual on them and the next ones
  box.each(g.n, halo, [&](int e, int i, int j, int l) {
    const size_t k = node(g, ib, i, j, l);
    if (i < box.ox + halo + T::kX && j < box.oy + halo + T::kY && (DIM == 2 || l < z0 + T::kZ))
      xo[k] = X[e];
    Y[e] = defect(g, k, f[k], X, e, box.w, box.h);
  });
  __syncthreads();
  // P^T: coarse node (I, J, L) at fine (2I, 2J, 2L), the odd corner nodes being the block's first
  const int nc = g.n / 2, cx = T::kX / 2, cy = T::kY / 2, cz = DIM == 3 ? T::kZ / 2 : 1;
  for (int q = threadIdx.x; q < cx * cy * cz; q += blockDim.x) {
    const int a = q % cx, b = q / cx % cy, c = q / (cx * cy);
    const int I = 1 + blockIdx.x * cx + a, J = 1 + blockIdx.y * cy + b,
              L = DIM == 3 ? (z0 + 1) / 2 + c : 0;
    if (I >= nc || J >= nc || (DIM == 3 && L >= nc)) continue;
    const int e = ((DIM == 3 ? 2 * L - box.oz : 0) * box.h + 2 * J - box.oy) * box.w + 2 * I - box.ox;
    double s = 0.0;
#pragma unroll
    for (int d = 0; d < T::kDirs; ++d) {
      const int t = dirx<DIM>(d) + (diry<DIM>(d) + dirz<DIM>(d) * box.h) * box.w;
      s += Y[e + t] + Y[e - t];
    }
    fc[ib * stc + ((size_t)L * (DIM == 3 ? nc + 1 : 0) + J) * pc + I] = fma(0.5, s, Y[e]);
  }
}

template <int DIM>
__global__ void __launch_bounds__(Tile<DIM>::kThreads)
    k_leg_up(const __grid_constant__ LegLevel<DIM> g, int pc, size_t stc, int nu,
             const double* __restrict__ f, const double* __restrict__ ec,
             const double* __restrict__ x, double* __restrict__ xo) {
  extern __shared__ double sm[];
  int z0;
  const int ib = locate<DIM>(g.n, z0);
  Box<DIM> box(nu, 0);
  if (DIM == 3) box.set_z(z0, nu, 0);
  const int m = box.elements(), nc = g.n / 2;
  double *X = sm, *Y = sm + m;
  for (int e = threadIdx.x; e < 2 * m; e += blockDim.x) sm[e] = 0.0;
  __syncthreads();
  const long planec = DIM == 3 ? (long)(nc + 1) * pc : 0;
  box.each(g.n, 0, [&](int e, int i, int j, int l) {
    const double* c = ec + ib * stc + (l >> 1) * planec + (size_t)(j >> 1) * pc + (i >> 1);
    const double v = x[node(g, ib, i, j, l)];
    const int ai = i & 1, aj = j & 1, al = DIM == 3 ? l & 1 : 0;
    X[e] = ai | aj | al ? fma(0.5, c[0] + c[ai + aj * (long)pc + al * planec], v) : c[0] + v;
  });
  __syncthreads();
  for (int t = 0; t < nu; ++t) {
    sweep(g, ib, box, t + 1, f, X, Y);
    __syncthreads();
    double* s = X;
    X = Y;
    Y = s;
  }
  box.each(g.n, nu, [&](int e, int i, int j, int l) { xo[node(g, ib, i, j, l)] = X[e]; });
}

template <int DIM>
dim3 leg_grid(const Grid& g) {
  using T = Tile<DIM>;
  const int m = g.n - 1;
  return dim3((m + T::kX - 1) / T::kX, (m + T::kY - 1) / T::kY,
              g.nb * (DIM == 3 ? (m + T::kZ - 1) / T::kZ : 1));
}
template <int DIM>
size_t leg_smem(int halo, int plus) {
  using T = Tile<DIM>;
  const int r = plus + 2 * halo;
  return 2 * sizeof(double) * (T::kX + r) * (T::kY + r) * (DIM == 3 ? T::kZ + r : 1);
}
LegLevel<2> leg_level(const Grid& g, const Coef2D& c) {
  return {g.n, g.pitch, g.stride, {c.cC, c.cE, c.cN, c.cNE}, c.dinv};
}
LegLevel<3> leg_level(const Grid& g, const Coef3D& c) {
  LegLevel<3> l{g.n, g.pitch, g.stride, {}, c.dinv};
  for (int q = 0; q < 8; ++q) l.a[q] = c.a[q];
  return l;
}
template <int DIM>
void leg_down(const LegLevel<DIM>& l, const Grid& g, const Grid& gc, const double* f,
              const double* x, double* xo, double* fc, int nu, bool zero, cudaStream_t s) {
  const int halo = zero ? (nu > 1 ? nu : 1) : nu + 1;
  k_leg_down<DIM><<<leg_grid<DIM>(g), Tile<DIM>::kThreads, leg_smem<DIM>(halo, 1), s>>>(
      l, gc.pitch, gc.stride, nu, zero ? 1 : 0, f, x, xo, fc);
}
template <int DIM>
void leg_up(const LegLevel<DIM>& l, const Grid& g, const Grid& gc, const double* f,
            const double* ec, const double* x, double* xo, int nu, cudaStream_t s) {
  k_leg_up<DIM><<<leg_grid<DIM>(g), Tile<DIM>::kThreads, leg_smem<DIM>(nu, 0), s>>>(
      l, gc.pitch, gc.stride, nu, f, ec, x, xo);
}

}  // namespace

void vcycle_down(const Grid& g, const Coef2D& c2, const Coef3D& c3, const Grid& gc,
                 const double* f, const double* x, double* xo, double* fc, int nu, bool zero,
                 cudaStream_t s) {
  if (g.dim == 2) leg_down(leg_level(g, c2), g, gc, f, x, xo, fc, nu, zero, s);
  else leg_down(leg_level(g, c3), g, gc, f, x, xo, fc, nu, zero, s);
}
void vcycle_up(const Grid& g, const Coef2D& c2, const Coef3D& c3, const Grid& gc, const double* f,
               const double* ec, const double* x, double* xo, int nu, cudaStream_t s) {
  if (g.dim == 2) leg_up(leg_level(g, c2), g, gc, f, ec, x, xo, nu, s);
  else leg_up(leg_level(g, c3), g, gc, f, ec, x, xo, nu, s);
}

}  // namespace fmg
