// Internal declarations shared by the CUDA translation units of libfmg_eig.
//
// Device layout of a level vector (2D): the (n+1) x (n+1) grid of ALL nodes, boundary
// included, row-major with x fastest and a row pitch of `pitch` elements (a multiple of 32).
// Boundary entries and the pitch padding are zero and are never written, so stencils need no
// boundary branches.  3D adds planes of (n+1) rows each.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/fmg_eig.h"
#include "dense_lists.h"

namespace fmg {

// Batched launches: every per-level array holds its instances back to back, instance b's
// vector starting at element b * stride; every launcher runs instances 0 .. nb - 1 of the
// arrays it is given, and per-instance scalars (lambda, parameters, dots) are indexed by b.
struct Grid {
  int dim = 2;
  int n = 0;          // cells per side
  int pitch = 0;      // elements per row
  int rows = 0;       // rows per plane (n + 1)
  size_t stride = 0;  // elements per vector of one instance
  double h = 0;
  int nb = 1;         // instances of a launch
  int bx = 32, by = 8;  // thread-block shape of the stencil kernels on this level
  bool walk_all = false;  // FP64 cubic-load kernels as walks whatever the launch size
  size_t interior() const {
    size_t m = (size_t)(n - 1);
    return dim == 2 ? m * m : m * m * m;
  }
};

// A vector split into double-float halves (hi + lo, FP32 each) for the nonlinear kernels of
// the mixed-precision modes, which compute in double-float arithmetic on the FP32 pipes.
// up to two vectors restricted by one launch
struct RestrictVecs {
  const double* rf[2];
  double* rc[2];
};

struct SplitVec {
  const float* hi;
  const float* lo;
};

// Problem parameters that may change between solves of one handle.  They live in device
// memory (uploaded at the start of every solve), so kernels take a device pointer to them.
struct PotentialParams {
  double w0, wx, wy, wz;
  double zeta;
  double omega;
  int operator_form;
  int pad;
};

// Fixed-point form of the 2D operator (fxop2d.cu), per instance: the shifts of the product sum
// and of the small terms, and their coefficients.
struct FxHead2D {
  int sa, sm, P, Q, R;
  double omega;
};

// Stencil coefficients of L = A + W on one 2D level (see grid2d.cu for the closed forms).  The
// instances of the fixed-point form need the couplings only for the Chebyshev smoother and the
// paper-literal form, and in the mixed modes no omega / cC either (null: their sweeps are single
// precision; a Jacobi sweep of the component call forms it from tab).
struct Coef2D {
  double* cC;    // diagonal
  double* cE;    // coupling (i,j)-(i+1,j)
  double* cN;    // coupling (i,j)-(i,j+1)
  double* cNE;   // coupling (i,j)-(i+1,j+1)
  double* dinv;  // omega / cC
  double* tab;   // 8 * (n + 1) separable parts of the coefficients per instance
  // levels with instances of the fixed-point form: 4 (n + 1) table entries and a header per
  // instance
  long long* fxt;
  FxHead2D* fxh;
  // levels with instances of both forms: whether the instance takes the fixed-point one.  The
  // kernels of each form leave the other's instances out.
  const int* fits;
};

// Levels whose operator runs in fixed point (fxop2d.cu): from 512 cells per side on a sweep is
// bound by the FP64 pipe (262k nodes: 3.3 us of it); below, by launch latency.  The instances
// whose potential the formats do not hold (fxop2d_scale) keep the stored couplings and the FP64
// kernels.  The choice depends on n and the instance alone, so an instance of a batch takes the
// same form as alone.
inline bool fxop2d_applies(const Grid& g) { return g.dim == 2 && g.n >= 512; }
// Scales of the fixed-point form: the potential's coefficients are below 2^-sa, the small ones
// below 2^-ss.  holds: the formats hold them (see fxop2d.cu).
struct FxScale {
  int sa, ss;
  bool holds;
};
__host__ __device__ inline FxScale fxop2d_scale(int n, double h, const PotentialParams& p) {
  const double wl = p.operator_form == FMG_W_LEFT ? 1.0 : 0.0, h2 = h * h, L = n * h;
  const double wsum = wl * (fabs(p.wx) + fabs(p.wy));
  const double amax = h2 / 12.0 * (wl * fabs(p.w0) + wsum * (L * L + 0.3 * h2));
  const double pmax = h2 * h2 * wsum;  // bounds the small coefficients
  FxScale q;
  q.sa = amax > 0.0 ? -(ilogb(amax) + 1) : 40;
  q.sa = q.sa < 0 ? 0 : q.sa > 40 ? 40 : q.sa;
  q.ss = pmax > 0.0 ? -(ilogb(pmax) + 1) : 90;
  q.ss = q.ss < 0 ? 0 : q.ss > 90 ? 90 : q.ss;
  // the small terms are 0.2 pmax of the maximum at most and lose 2^-26 of that: with pmax <=
  // 2^-22 the loss is below 2^-50 (each rounding of the FP64 form at 4x: 2^-51)
  q.holds = amax <= 1.0 / 64.0 && pmax <= 1.0 / 4194304.0 && q.ss - q.sa + 1 >= 0;
  return q;
}
void fxop2d_tables(const Grid& g, const PotentialParams* p, const Coef2D& c, cudaStream_t s);
void fxop2d_apply(const Grid& g, const Coef2D& c, const double* x, double* y, cudaStream_t s);
void fxop2d_apply_mass(const Grid& g, const Coef2D& c, const double* x, double* y, double* mx,
                       cudaStream_t s);
void fxop2d_jacobi(const Grid& g, const Coef2D& c, const double* f, const double* x, double* xo,
                   cudaStream_t s);
void fxop2d_residual(const Grid& g, const Coef2D& c, const double* f, const double* x, double* r,
                     cudaStream_t s);
// the residual rounded to single precision (float, or bfloat16 behind the float pointer)
void fxop2d_residual32(const Grid& g, const Coef2D& c, const double* f, const double* x, float* r,
                       bool bf, cudaStream_t s);

// ---- 2D level kernels (grid2d.cu) -------------------------------------------------------
// ratio_fx: omega / D of the fixed-point instances beside others as of such instances alone
void coef2d_setup(const Grid& g, const PotentialParams* p_dev, const Coef2D& c, bool ratio_fx,
                  cudaStream_t s);
void apply2d(const Grid& g, const Coef2D& c, const double* x, double* y, cudaStream_t s);
void mass2d(const Grid& g, const double* x, double* y, cudaStream_t s);
// y = L x, z = M x
void apply_mass2d(const Grid& g, const Coef2D& c, const double* x, double* y, double* z,
                  cudaStream_t s);
// f -= W u, W u = (A + W) u - A u from the coefficient sets cw (A + W) and ca (A)
void sub_wmass2d(const Grid& g, const Coef2D& cw, const Coef2D& ca, const double* u, double* f,
                 cudaStream_t s);
void jacobi2d(const Grid& g, const Coef2D& c, const double* f, const double* x, double* xo,
              bool x_is_zero, cudaStream_t s);
void residual2d(const Grid& g, const Coef2D& c, const double* f, const double* x, double* r,
                cudaStream_t s);
// Chebyshev step: d = (first ? 0 : alpha d) + beta D^{-1} (f - L x), xo = x + d (x = 0 when
// x_zero); needs the coefficients built with omega = 1 (dinv = 1/D)
void cheb2d(const Grid& g, const Coef2D& c, const double* f, const double* x, double* d,
            double* xo, double alpha, double beta, bool first, bool x_zero, cudaStream_t s);
// rc = P^T rf; with rf2 given, also rc2 = P^T rf2 in the same launch
// Levels whose restriction sums in integers: those above the V-cycle legs' (vcycle_legs.cu), to
// whose FP64 sums the separate kernels are bit-identical.  (In 3D the same took a launch from 65
// to 55 us and no time off a solve.)
inline bool restrict_ints(const Grid& fine) { return fine.n >= 512; }
void restrict2d(const Grid& fine, const Grid& coarse, const double* rf, double* rc,
                cudaStream_t s, const double* rf2 = nullptr, double* rc2 = nullptr);
// xf = (add ? xf : 0) + P ec (+ scale[b * scale_stride] * extra for instance b when extra is
// given)
void prolong2d(const Grid& fine, const Grid& coarse, const double* ec, double* xf, bool add,
               const double* extra, const double* scale, int scale_stride, cudaStream_t s);
void nload2d(const Grid& g, const double* u, double* out, cudaStream_t s);
// f = lam[b] * M u - p[b].zeta * N(u) for instance b
void rhs2d(const Grid& g, const double* lam, const PotentialParams* p_dev, const double* u,
           double* f, cudaStream_t s);
// the same right-hand side evaluated in FP32 (mixed-precision iteration), stored in FP64
void rhs2d_f32(const Grid& g, const double* lam, const PotentialParams* p_dev, const double* u,
               double* f, cudaStream_t s);
// Dense level-1 matrices L_1 and M_1 (n1-1)^2 square, row-major, interior numbering (one
// pair per instance, back to back).
void dense_level1_2d(const Grid& g, const Coef2D& c, double* L, double* M, cudaStream_t s);
// sin-product start vector for the level-1 nonlinear solve (instance b at c + b * cstride)
void start_vector(const Grid& g, double* c, int cstride, cudaStream_t s);

// ---- 3D level kernels (grid3d.cu) -------------------------------------------------------
// Couplings of L on the Kuhn mesh: a[0] diagonal, a[1 + d] the coupling of p with p + d for
// d = X, Y, Z, XY, XZ, YZ, XYZ (the coupling with p - d is a[1 + d] at p - d).
// The levels of the fixed-point form keep a as Coef2D says.
struct FxHead3D {  // as FxHead2D, for fxop3d.cu
  int sa, sm, P, A[3], F[3];
  double K[8];  // constant parts of the couplings (the others are in tab)
};
struct Coef3D {
  double* a[8];
  double* dinv;  // omega / diagonal
  double* tab;   // 15 * (n + 1) separable parts per instance
  // FP64-mode levels with instances of the fixed-point form: 6 (n + 1) table entries and a
  // header per instance
  long long* fxt;
  FxHead3D* fxh;
  const int* fits;  // as Coef2D
};
// Levels whose operator runs in fixed point (fxop3d.cu), FP64 mode only: the mixed modes'
// single-precision V-cycles amplify the rounding of the FP64 steps around them (see
// dense_pinned.cu).  Below 96 cells per side the plane walk has too few blocks.
inline bool fxop3d_applies(const Grid& g) { return g.dim == 3 && g.n >= 96; }
// as fxop2d_scale
__host__ __device__ inline FxScale fxop3d_scale(int n, double h, const PotentialParams& p) {
  const double wl = p.operator_form == FMG_W_LEFT ? 1.0 : 0.0, h2 = h * h, L = n * h;
  const double wsum = wl * (fabs(p.wx) + fabs(p.wy) + fabs(p.wz));
  const double amax = h2 / 60.0 * (wl * fabs(p.w0) + wsum * (L * L + 0.31 * h2));
  const double pmax = h2 * h2 * wsum;  // bounds the small coefficients (and their sum over a stencil)
  FxScale q;
  q.sa = amax > 0.0 ? -(ilogb(amax) + 1) : 40;
  q.sa = q.sa < 0 ? 0 : q.sa > 40 ? 40 : q.sa;
  q.ss = pmax > 0.0 ? -(ilogb(pmax) + 1) : 90;
  q.ss = q.ss < 0 ? 0 : q.ss > 90 ? 90 : q.ss;
  // the small terms are 0.06 pmax of the maximum at most; 30 bits of the pairs and of the
  // coefficients (each below pmax / 89, hence 36 + ss) leave 2^-33 pmax of it: with pmax <=
  // 2^-17, 2^-50 of the maximum against the 6 times the maximum that L / h reaches
  q.holds = amax <= 1.0 / 64.0 && pmax <= 1.0 / 131072.0 && q.ss - q.sa + 11 >= 0;
  return q;
}
void fxop3d_tables(const Grid& g, const PotentialParams* p, const Coef3D& c, cudaStream_t s);
void fxop3d_apply(const Grid& g, const Coef3D& c, const double* x, double* y, cudaStream_t s);
void fxop3d_apply_mass(const Grid& g, const Coef3D& c, const double* x, double* y, double* mx,
                       cudaStream_t s);
void fxop3d_jacobi(const Grid& g, const Coef3D& c, const double* f, const double* x, double* xo,
                   cudaStream_t s);
void fxop3d_residual(const Grid& g, const Coef3D& c, const double* f, const double* x, double* r,
                     cudaStream_t s);
struct Density3D {
  double* a[8];  // same layout as Coef3D::a
};
struct Stencil15 {
  const double* a[8];
};
void coef3d_setup(const Grid& g, const PotentialParams* p_dev, const Coef3D& c, bool ratio_fx,
                  cudaStream_t s);
void apply3d(const Grid& g, const Coef3D& c, const double* x, double* y, cudaStream_t s);
void mass3d(const Grid& g, const double* x, double* y, cudaStream_t s);
// y = L x, z = M x
void apply_mass3d(const Grid& g, const Coef3D& c, const double* x, double* y, double* z,
                  cudaStream_t s);
void mass3d_df(const Grid& g, SplitVec x, double* y, cudaStream_t s);
void sub_wmass3d(const Grid& g, const Coef3D& cw, const Coef3D& ca, const double* u, double* f,
                 cudaStream_t s);
void jacobi3d(const Grid& g, const Coef3D& c, const double* f, const double* x, double* xo,
              bool x_is_zero, cudaStream_t s);
void residual3d(const Grid& g, const Coef3D& c, const double* f, const double* x, double* r,
                cudaStream_t s);
void cheb3d(const Grid& g, const Coef3D& c, const double* f, const double* x, double* d,
            double* xo, double alpha, double beta, bool first, bool x_zero, cudaStream_t s);
void restrict3d(const Grid& fine, const Grid& coarse, const double* rf, double* rc,
                cudaStream_t s, const double* rf2 = nullptr, double* rc2 = nullptr);
void prolong3d(const Grid& fine, const Grid& coarse, const double* ec, double* xf, bool add,
               const double* extra, const double* scale, int scale_stride, cudaStream_t s);
void nload3d(const Grid& g, const double* u, double* out, cudaStream_t s);
void rhs3d(const Grid& g, const double* lam, const PotentialParams* p_dev, const double* u,
           double* f, cudaStream_t s);
void rhs3d_f32(const Grid& g, const double* lam, const PotentialParams* p_dev, const double* u,
               double* f, cudaStream_t s);
void nload_density3d(const Grid& g, const double* u, double* nl, const Density3D& b,
                     cudaStream_t s);
// double-float versions from the split u (3D mixed-precision modes)
void rhs3d_df(const Grid& g, const double* lam, const PotentialParams* p_dev, SplitVec u,
              double* f, cudaStream_t s);
// (the _df versions write the density stencil as double-float splits: see put_entry)
void nload_density3d_df(const Grid& g, SplitVec u, double* nl, const Density3D& b,
                        cudaStream_t s);
void coarsen_density3d(const Grid& fine, const Grid& coarse, const Density3D& bf,
                       const Density3D& bc, cudaStream_t s);
void coarsen_density3d_df(const Grid& fine, const Grid& coarse, const Density3D& bf,
                          const Density3D& bc, cudaStream_t s);
void dense_level1_3d(const Grid& g, const Coef3D& c, double* L, double* M, cudaStream_t s);
void density_dense3d(const Grid& g, const Density3D& b, double* B, cudaStream_t s,
                     bool split = false);
void gather_vec3d(const Grid& g, const double* a, const double* b, const double* c, double* oa,
                  double* ob, double* oc, cudaStream_t s);
void start_vector3d(const Grid& g, double* c, int cstride, cudaStream_t s);

// ---- 3D augmented pass (augment3d.cu) -----------------------------------------------------
// T3 per coarse Kuhn tetrahedron (20 per tetrahedron, sorted triples of its 4 vertices;
// partials: t3_partials3d doubles per instance, t3: 20 per tetrahedron per instance),
// tetrahedron index 6 * (I + n1 (J + n1 L)) + s, s the axis permutation in lexicographic
// order, vertices (V, V + e_s0, V + e_s0 + e_s1, V + (1,1,1)).
size_t t3_partials3d(const Grid& fine, int n1);
// pw: the level's (x/r)^m table (t3_power_table)
void t3_moments3d(const Grid& fine, int n1, const double* u, const double* pw,
                  const double* map, double* partials, double* t3, cudaStream_t s);
void t3_map3d(int r, double* out);  // 20 * 15 * 20 doubles

// ---- Mixed precision (mixed.cu) ------------------------------------------------------------
// FP32 separable coefficient tables of one level for the single-precision V-cycle: tab =
// the level's FP64 tables (2D: 8, 3D: 15 per instance, n + 1 entries each) rounded to FP32
// and tablo their remainders (tab + tablo is their double-float split); cst = kCst floats
// per instance: the 3D constants (C, axis, face, body) at 0..3 with their remainders at
// kCstLo + 0..3, and omega at kCstOmega with its remainder at kCstOmegaLo.
struct CoefT {
  float* tab;
  float* tablo;
  float* cst;
};
// 3D single-precision sweeps: coupling = ((x part + y part) + z part) + class constant, the
// large constant (6h, -h) added last so that each coefficient is one rounding from its FP64
// value.  (Adding the constant first and three rounded table entries after it left the
// smooth-mode part of the operator off by several roundings of the constant, which showed
// as |d lambda| up to 3e-8 on strongly nonlinear 3D problems.)
constexpr int kCst = 16;
constexpr int kCstOmega = 4;
constexpr int kCstOmegaLo = 5;
constexpr int kCstLo = 8;

// hi[i] + lo[i] = u[i] to 2^-47 relative (hi: u[i]'s significand cut to 24 bits), i < n;
// n even, the arrays allocation-aligned
void split_df(const double* u, float* hi, float* lo, size_t n, cudaStream_t s);
// Storage of the single-precision V-cycle arrays (the float* below): FP32, or bfloat16 when
// `bf` is set (FMG_MIXED_BF16; arithmetic stays FP32).  Bytes per element:
size_t mixed_elem_bytes(bool bf16_storage);
// contiguous conversions over n entries (all instances of a level at once)
void add_f32(const float* e, double* x, size_t n, cudaStream_t s, bool bf = false);  // x += e
// r = f - L x with the FP64 operator of the level (2D uses c2, 3D c3), stored single
void residual_mixed(const Grid& g, const Coef2D& c2, const Coef3D& c3, const double* f,
                    const double* x, float* r, cudaStream_t s, bool bf = false);
// the split tables and constants of level g from its FP64 tables (c2.tab / c3.tab written)
void tables_f32(const Grid& g, const Coef2D& c2, const Coef3D& c3,
                const PotentialParams* pp, const CoefT& ct, cudaStream_t s);
// TMA-fed single-precision sweeps of the large levels (sweep_tma.cu).  A TMAMap holds a
// tensor map (CUtensorMap) of one level vector: columns, rows and instances, with a box of
// one tile (halo = true: the x box, 2 rows taller).
struct TMAMap {
  alignas(64) unsigned char bytes[128];
};
constexpr int kTMAMinCells2 = 512;  // 2D levels with n >= this use the TMA sweeps
constexpr int kTMAMinCells3 = 128;  // 3D levels likewise
bool tma_sweep_applies(const Grid& g);
bool encode_level_map(const Grid& g, int cap, const float* base, bool bf, bool halo,
                      TMAMap* out);
// mode 0: residual y = f - L x; 1: Jacobi y = x + omega D^-1 (f - L x); 2: Jacobi from x = 0.
// A tile wait that runs out sets wait_fail[b] = 1 for its instance b (wait_fail: g.nb ints);
// `expire` makes every tile wait give up at once (the FMG_FLAG_EXPIRE_WAITS test hook).
void sweep32_tma(const Grid& g, const CoefT& ct, const TMAMap& mx, const TMAMap& mf, float* y,
                 int mode, int* wait_fail, bool expire, cudaStream_t s, bool bf = false);
// damped Jacobi sweep / residual with coefficients rebuilt from the FP32 tables
void jacobi32(const Grid& g, const CoefT& ct, const float* f, const float* x, float* xo,
              bool zero, cudaStream_t s, bool bf = false);
void residual32(const Grid& g, const CoefT& ct, const float* f, const float* x, float* r,
                cudaStream_t s, bool bf = false);
void restrict32(const Grid& fine, const Grid& coarse, const float* rf, float* rc,
                cudaStream_t s, bool bf = false);
void prolong32_add(const Grid& fine, const Grid& coarse, const float* ec, float* xf,
                   cudaStream_t s, bool bf = false);
void coarse32(const Grid& g, const double* Linv, const float* x, float* y, cudaStream_t s,
              bool bf = false);
// The levels of a single-precision V-cycle below the TMA-fed ones (vcycle32_mid.cu), two
// kernels per level, bit-identical to the separate sweep, residual and transfer kernels:
//   down: xo = nu_pre Jacobi sweeps from x = 0 on L(g) x = f, rc = P^T (f - L xo);
//   up:   xo = nu_post Jacobi sweeps from x + P ec (xo and x distinct).
// They take 2D levels of up to kMid32MaxCells cells per side with at most 4 + 4 sweeps, and
// 3D levels of up to kMid32MaxCells3 with at most 2 + 2.
constexpr int kMid32MaxCells = 256;
constexpr int kMid32MaxCells3 = 32;  // measured: 64 no faster than the separate kernels
bool vcycle32_mid_applies(const Grid& g, int nu_pre, int nu_post);
void vcycle32_down(const Grid& g, const CoefT& ct, const Grid& gc, const float* f, float* xo,
                   float* rc, int nu_pre, cudaStream_t s, bool bf = false);
void vcycle32_up(const Grid& g, const CoefT& ct, const Grid& gc, const float* f,
                 const float* x, float* xo, const float* ec, int nu_post, cudaStream_t s,
                 bool bf = false);

// ---- FP64 V-cycle legs of the middle levels (vcycle_legs.cu) -----------------------------
// Launch-bound levels, by cells per side and by the instances' nodes together: 2D both legs to
// 256 cells, 65,536 nodes (solve at h = 1/256 1.13 -> 1.01 ms, h = 1/896 1.92 -> 1.72 ms); 3D up
// to 32 cells, 32,768 nodes (launches of 16 us -> 11), down to 24 cells, 13,824 nodes (18 -> 8;
// at 32 cells its 512 blocks take 27 us where the four kernels take 19).  Results are
// bit-identical to the separate kernels', so the choice may depend on nb.
inline bool vcycle_leg_applies(const Grid& g, int nu, bool down) {
  const size_t n = g.n, m = g.nb * n * n;
  if (g.dim == 2) return nu <= 3 && n <= 256 && m <= 256 * 256;
  const size_t most = down ? 24 : 32;
  return nu <= 2 && n <= most && m * n <= most * most * most;
}
// xo = nu sweeps on L x = f from x (not read if zero), fc = P^T (f - L xo)
void vcycle_down(const Grid& g, const Coef2D& c2, const Coef3D& c3, const Grid& gc,
                 const double* f, const double* x, double* xo, double* fc, int nu, bool zero,
                 cudaStream_t s);
// xo = nu sweeps from x + P ec
void vcycle_up(const Grid& g, const Coef2D& c2, const Coef3D& c3, const Grid& gc, const double* f,
               const double* ec, const double* x, double* xo, int nu, cudaStream_t s);

// ---- Reductions (reduce.cu) -------------------------------------------------------------
// out[b] = sum_i a[b vst + i] * b[b vst + i] over n entries for instances b < nb;
// deterministic two-stage tree whose order depends on n only.  `partials` holds
// nb * kReduceBlocks doubles.
constexpr int kReduceBlocks = 1024;
// Elements per block, at least: 2048, 8 per thread (a reduction over a small level is bound by a
// thread's chain of loads and sums; 8192 took 15.7 us for both dots of a 1.1M-node level, 2048
// takes 12.8 for a 0.83M-node one).  The 3D mixed modes keep 8192, whose order of summation their
// amplified rounding shows.
constexpr size_t kDotElements = 2048, kDotPinned = 8192;
void dot(const double* a, const double* b, size_t n, double* partials, double* out,
         cudaStream_t s, int nb, size_t vst, size_t per_block);
// out = a . b and out2 = a . c in one pass (each as dot sums it); partials: 2 kReduceBlocks nb
void dot2(const double* a, const double* b, const double* c, size_t n, double* partials,
          double* out, double* out2, cudaStream_t s, int nb, size_t vst, size_t per_block);
// Conjugate gradient smoother over nb instances of n elements (one level's stride; even),
// kReduceBlocks partial sums per instance and dot product:
//   start      p = r, rr_parts = parts of r.r
//   dot        pq_parts = parts of p.q
//   update     a = rr / pq, x += a p, r -= a q, parts = parts of the new r.r; rr[b] is read, or
//              (rr_parts given) summed from rr_parts and written
//   direction  rr_new[b] = sum of parts, p = r + (rr_new / rr_old) p
void cg_start(size_t n, int nb, const double* r, double* p, double* rr_parts, cudaStream_t s);
void cg_dot(size_t n, int nb, const double* p, const double* q, double* pq_parts, cudaStream_t s);
void cg_update(size_t n, int nb, double* rr, const double* rr_parts, const double* pq_parts,
               const double* p, const double* q, double* x, double* r, double* parts,
               cudaStream_t s);
void cg_direction(size_t n, int nb, const double* rr_old, const double* parts, double* rr_new,
                  const double* r, double* p, cudaStream_t s);

// ---- Interior <-> padded packing (pack.cu) ----------------------------------------------
// (instance b: interior vector at b * g.interior(), padded one at b * g.stride)
void pack_interior(const Grid& g, const double* interior, double* padded, cudaStream_t s);
void unpack_interior(const Grid& g, const double* padded, double* interior, cudaStream_t s);
// The interior of one instance's padded vector into a pinned host buffer by one strided
// copy-engine transfer (2D: a pitched 2D copy, 3D: a pitched 3D copy), no staging buffer.
cudaError_t copy_interior_to_host(const Grid& g, const double* padded, double* host,
                                  cudaStream_t s);
// dst[i] = src[idx[i]], i < n
void gather_by_index(const double* src, const int* idx, double* dst, int n, cudaStream_t s);
// padded level-1 vectors from dense coefficient vectors c (instance b at c + b * cstride)
void scatter_level1(const Grid& g, const double* c, size_t cstride, double* padded,
                    cudaStream_t s);

// ---- Augmented-space fine pass (augment2d.cu) ---------------------------------------------
// Density stencil B(u)_pq = int u^2 phi_p phi_q of one 2D level (couplings to p, E, N, NE).
struct Density2D {
  double *C, *E, *N, *NE;
};
// nl = N(u) (int u^3 phi_p) and the density stencil of u on level g, in one pass.
void nload_density2d(const Grid& g, const double* u, double* nl, const Density2D& b,
                     cudaStream_t s);
// Galerkin coarsening of the density stencil: bc = P^T bf P (coarsen_fx.cu).
void coarsen_density2d(const Grid& fine, const Grid& coarse, const Density2D& bf,
                       const Density2D& bc, cudaStream_t s);
// T3^T_abc = int_T u mu_a mu_b mu_c per coarse triangle (10 per triangle, a <= b <= c,
// lexicographic), from per-class monomial sums.  pw: (x/r)^m table of the level, map: the
// level's 2 x 10 x 25 map (t3_map2d), partials: t3_partials2d(fine, n1) doubles.
size_t t3_partials2d(const Grid& fine, int n1);
void t3_moments2d(const Grid& fine, int n1, const double* u, const double* pw,
                  const double* map, double* partials, double* t3, cudaStream_t s);
void t3_class_moments2d(double out[2 * 7 * 10]);
void t3_map2d(int r, double out[2 * 10 * 25]);
void t3_power_table(int r, double* out);  // 4 * (r + 1) doubles
// dense level-1 data for the augmented solve: gA, gM, t1 (nh) and B1 (nh x nh) from padded
// level-1 vectors and the level-1 density stencil (per instance, back to back)
void gather_level1_2d(const Grid& g1, const double* gA_pad, const double* gM_pad,
                      const double* t1_pad, const Density2D& b1, double* gA, double* gM,
                      double* t1, double* B1, cudaStream_t s);

// ---- Dense small solves (dense.cu) -------------------------------------------------------
// A batch of problems shares the geometry (tri, lists) and keeps the per-instance arrays
// back to back: L1, M1, B1 nh*nh; gA, gM, t1 nh; t3 ntri*nt3; c_init, c_out nh + 1;
// auu, buu, t0, lam_out, iters_out, status_out and params one each.
struct DenseProblem {
  int nh;              // coarse unknowns (interior nodes of level 1)
  int aug;             // 1: basis (phi^H, u~), n = nh + 1; 0: basis phi^H, n = nh
  int ntri;            // coarse simplices
  int nvert;           // vertices per simplex (3 in 2D, 4 in 3D)
  int nt3;             // entries of T3 per simplex (10 in 2D, 20 in 3D)
  const int* tri;      // ntri * nvert coarse interior indices, -1 on the boundary
  // sparsity lists of the coarse block and of T3 (dense_lists.h), device memory
  const uint16_t* lists;
  DenseLists dims;
  double quart_off;    // |T| 2 d! / (d + 4)!, d = nvert - 1 (int_T w^2 mu_a mu_b / h_2)
  const double* L1;    // nh*nh, operator of level 1
  const double* M1;    // nh*nh, mass of level 1
  // augmented problem only:
  const double* gA;    // nh: P^T..P^T L u~
  const double* gM;    // nh: P^T..P^T M u~
  const double* t1;    // nh: int u~^3 phi^H_a
  const double* B1;    // nh*nh: int u~^2 phi^H_a phi^H_b
  const double* t3;    // ntri * nt3: int_T u~ mu_a mu_b mu_c (sorted triples)
  const double* auu;   // u~^T L u~
  const double* buu;   // u~^T M u~
  const double* t0;    // int u~^4
  const PotentialParams* params;  // device; zeta read from here
  double tol;
  int max_iter;
  const double* c_init;  // nullptr: augmented start e_u / sqrt(buu); level-1: caller fills
  double* c_out;         // n
  double* lam_out;       // 1
  int* iters_out;        // 1
  int* status_out;       // 1 (0 converged, 1 cap hit)
  // optional (a single problem only): assemble K0, M, G(c_init) into these n x n outputs
  double* K_out;
  double* M_out;
  double* G_out;
};
constexpr size_t kDenseSmemLimit = 200 * 1024;  // dynamic shared memory of the dense solve
size_t dense_smem_bytes(int n, int ntri, int nvert, int aug);
cudaError_t dense_prepare(size_t max_smem);  // opt in to large dynamic shared memory
void dense_scf(const DenseProblem& p, int nb, cudaStream_t s);  // one CTA per problem
// The form of the small solves and of the third moments that 3D mixed-precision solves with
// single-precision V-cycles keep, bit for bit (dense_pinned.cu, t3_pinned3d.cu).  Tables: the
// adjacency codes (simplex << 3 | local vertex, -1 terminated) adj[nh * maxadj], and gather
// lists of the coarse block of G(c): the npat structurally nonzero entries gent[q] = a nh + b,
// and for each the simplex-local indices gidx[gstart[q] .. gstart[q + 1]).
struct PinnedTables {
  const int *adj = nullptr, *gent = nullptr, *gstart = nullptr, *gidx = nullptr;
  int maxadj = 24, npat = 0;
};
cudaError_t dense_prepare_pinned();
void dense_scf_pinned(const DenseProblem& p, const PinnedTables& pt, int nb, cudaStream_t s);
void dense_spd_inverse_pinned(const double* L, double* Linv, int n, int nb, cudaStream_t s);
size_t t3_partials3d_pinned(const Grid& fine, int n1);
void t3_moments3d_pinned(const Grid& fine, int n1, const double* u, const double* pw,
                         const double* map, double* partials, double* t3, cudaStream_t s);
// Linv = L^{-1} for the SPD n x n level-1 operators (nonzeros in `lists`), one CTA each.
void dense_spd_inverse(const double* L, double* Linv, int n, const uint16_t* lists,
                       const DenseLists& dims, int nb, cudaStream_t s);
// y(padded level 1) = Linv * x(padded level 1) on the interior nodes (2D or 3D)
void coarse_matvec(const Grid& g, const double* Linv, const double* x, double* y,
                   cudaStream_t s);

// ---- the small levels of a 2D V-cycle in one kernel (vcycle_small.cu) ---------------------
constexpr int kSmallMaxLevels = 6;    // entry level and the levels below it
constexpr int kSmallMaxCells = 32;    // cells per side of the entry level
constexpr size_t kSmallSmemLimit = 96 * 1024;
struct SmallLevel2D {
  int n, pitch;
  size_t stride;
  Coef2D c;  // the V-cycle's operator on this level
};
struct SmallVcycle {
  int levels;  // the entry level; levels 1 .. levels take part
  int nu_pre, nu_post, x_zero;
  SmallLevel2D lv[kSmallMaxLevels];  // level j at index j - 1
  const double* Linv;                // level-1 inverse, nh x nh per instance
  const double* f;                   // the entry level's right-hand side (batched arrays)
  double* x;                         // the entry level's iterate, read unless x_zero
};
size_t vcycle_small_smem(const SmallVcycle& v);
// One V-cycle from the entry level for instances 0 .. nb - 1; an error (before launching)
// when the levels need more shared memory than kSmallSmemLimit.
cudaError_t vcycle_small(const SmallVcycle& v, int nb, cudaStream_t s);

}  // namespace fmg
