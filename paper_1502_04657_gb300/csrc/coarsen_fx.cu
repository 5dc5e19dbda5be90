// Galerkin coarsening of the density stencil (entries FP64), 2D (7-point) and 3D (15-point):
//   Bc(a, b) = sum_{v, w} P_va P_wb B(v, w),
// the fine support of the coarse hat a being 2a (weight 1) and its neighbours (weight 1/2).
//
// A coarse node takes its 4 (8) entries from 30 (138) stored fine ones in 64 (290) weighted
// sums, which in FP64 (2 lanes per clock) cost more than reading the 16 (64) entries per coarse
// node that memory has to deliver.  The entries int u^2 phi phi are non-negative for a u of one
// sign, so a thread takes one exponent e for its coarse node, reads each entry as an integer in
// units of 2^(e - 55) and adds multiples 1, 2 or 4 of it (the weights in quarters) to the sums of
// all its targets; each target is converted once.  Only the truncation to 55 bits of the largest
// entry around the node rounds (its mean, half a unit each, is added back), where the FP64 form
// rounds every sum.  Measured: 16.6M 3D nodes 931 -> 280 us, 16.8M 2D nodes 370 -> 145 us
// (in 3D 623 us with one load per entry: half of each sector was used, and L2 had to deliver the
// rest again; 245 and 137 us with one exponent per warp, which lost the entries far below its
// largest; an exponent per thread with the neighbour's value shuffled, not its integer, spilled 1.3 KB
// per thread in 3D).
//
// e comes from the diagonal entries of 2a and of the corners of its cell.  Nodes with an entry of
// 2^(e + 1) or more, a negative one, infinities or NaN, a sum below 2^-9 of the largest entry (one
// that is exactly zero, or kept too few bits), zeros only or e outside +-kMaxExp are summed in FP64.
#include <utility>

#include "fixed.cuh"
#include "fmg_internal.h"

namespace fmg {
namespace {

constexpr int kB = 55;  // entry = I 2^(e - kB); I < 2^(kB + 1), a sum < 2^(kB + 1) 146 < 2^64
// From e = -965 on zeros and denormals are shifted out (by 63 or more), and the exponent field of
// the smallest sum stays positive when e - kB - 2 is added to it.
constexpr int kMaxExp = 900;
constexpr int kLeast = 46;  // bits a sum has at least (73 units, at most, are lost to truncation)

template <int DIM>
struct Mesh {
  static constexpr int kEnt = 1 << DIM;            // stored entries per node: self, + directions
  static constexpr int kPos = DIM == 2 ? 9 : 27;   // fine nodes 2a + {-1, 0, 1}^DIM
  // direction of an entry (the order of Density2D and Density3D)
  __host__ __device__ static constexpr int dx(int d) { return DIM == 2 ? (d == 1 || d == 3) : (d == 1 || d == 4 || d == 5 || d == 7); }
  __host__ __device__ static constexpr int dy(int d) { return DIM == 2 ? (d == 2 || d == 3) : (d == 2 || d == 4 || d == 6 || d == 7); }
  __host__ __device__ static constexpr int dz(int d) { return DIM == 2 ? 0 : (d == 3 || d == 5 || d == 6 || d == 7); }
  __host__ __device__ static constexpr int px(int v) { return v % 3 - 1; }
  __host__ __device__ static constexpr int py(int v) { return v / 3 % 3 - 1; }
  __host__ __device__ static constexpr int pz(int v) { return DIM == 2 ? 0 : v / 9 - 1; }
};

// weight, in quarters, of the entry d stored at the fine position v in the target T
template <int DIM>
struct Weights {
  unsigned char w[Mesh<DIM>::kEnt][Mesh<DIM>::kPos][Mesh<DIM>::kEnt] = {};
  int total[Mesh<DIM>::kEnt] = {};
  bool inside = true;  // every entry is stored at one of the kPos positions
  __host__ __device__ constexpr Weights() {
    using M = Mesh<DIM>;
    for (int T = 0; T < M::kEnt; ++T)
      for (int p = 0; p < 2 * M::kEnt - 1; ++p)    // self, +1, -1, +2, -2 .. directions
        for (int q = 0; q < 2 * M::kEnt - 1; ++q) {
          const int dp = (p + 1) / 2, sp = p & 1 ? 1 : -1, dq = (q + 1) / 2, sq = q & 1 ? 1 : -1;
          const int vx = sp * M::dx(dp), vy = sp * M::dy(dp), vz = sp * M::dz(dp);
          const int ox = 2 * M::dx(T) + sq * M::dx(dq) - vx, oy = 2 * M::dy(T) + sq * M::dy(dq) - vy,
                    oz = 2 * M::dz(T) + sq * M::dz(dq) - vz;
          for (int d = 0; d < M::kEnt; ++d)
            for (int s = 1; s >= (d ? -1 : 1); s -= 2) {
              if (ox != s * M::dx(d) || oy != s * M::dy(d) || oz != s * M::dz(d)) continue;
              // stored at v for +d, at v + o for -d
              const int x = vx + (s < 0 ? ox : 0), y = vy + (s < 0 ? oy : 0), z = vz + (s < 0 ? oz : 0);
              if (x < -1 || x > 1 || y < -1 || y > 1 || z < -1 || z > 1) inside = false;
              else w[d][x + 1 + 3 * (y + 1) + (DIM == 3 ? 9 * (z + 1) : 0)][T] +=
                  (p == 0 ? 2 : 1) * (q == 0 ? 2 : 1);
              total[T] += (p == 0 ? 2 : 1) * (q == 0 ? 2 : 1);
            }
        }
  }
  __host__ __device__ constexpr bool used(int d, int v) const {
    for (int T = 0; T < Mesh<DIM>::kEnt; ++T)
      if (w[d][v][T]) return true;
    return false;
  }
};
template <int DIM>
struct Tab {
  static constexpr Weights<DIM> k{};
  static_assert(k.inside && k.total[0] <= 146, "entries within the cell, sums within 64 bits");
};
template <int DIM>
struct Entries {
  double* a[1 << DIM];
};

template <int DIM>
__device__ __forceinline__ long offset(int v, int pitch, long plane) {
  using M = Mesh<DIM>;
  return M::px(v) + (long)M::py(v) * pitch + (DIM == 3 ? M::pz(v) * plane : 0);
}

// The node's targets in FP64, entry by entry (unrolled: 64 or 290 multiply-adds, 10 us of a warp;
// with the weights looked up at run time a small level with one such node took 100 us more)
template <int DIM, int D, int V, int... T>
__device__ __forceinline__ void add_targets_fp64(double e, double (&acc)[1 << DIM],
                                                 std::integer_sequence<int, T...>) {
  ((acc[T] = Tab<DIM>::k.w[D][V][T] ? fma(0.25 * Tab<DIM>::k.w[D][V][T], e, acc[T]) : acc[T]), ...);
}
template <int DIM, int... Q>
__device__ __forceinline__ void add_entries_fp64(const Entries<DIM>& f, size_t kf, int pitch,
                                                 long plane, double (&acc)[1 << DIM],
                                                 std::integer_sequence<int, Q...>) {
  constexpr int E = 1 << DIM;
  constexpr auto targets = std::make_integer_sequence<int, E>();
  ((Tab<DIM>::k.used(Q % E, Q / E)
        ? add_targets_fp64<DIM, Q % E, Q / E>(f.a[Q % E][kf + offset<DIM>(Q / E, pitch, plane)], acc,
                                              targets)
        : (void)0),
   ...);
}
template <int DIM>
__device__ __noinline__ void node_fp64(const Entries<DIM>& f, const Entries<DIM>& c, size_t kf,
                                       size_t kc, int pitch, long plane) {
  using M = Mesh<DIM>;
  double acc[M::kEnt] = {};
  add_entries_fp64<DIM>(f, kf, pitch, plane, acc,
                        std::make_integer_sequence<int, M::kEnt * M::kPos>());
#pragma unroll
  for (int T = 0; T < M::kEnt; ++T) c.a[T][kc] = acc[T];
}

// the mean of what the truncations drop, half a unit per quarter weight
template <int DIM, int... T>
__device__ __forceinline__ void start_targets(unsigned long long (&acc)[1 << DIM],
                                              std::integer_sequence<int, T...>) {
  ((acc[T] = std::integral_constant<int, Tab<DIM>::k.total[T] / 2>::value), ...);
}

template <int DIM, int D, int V, int... T>
__device__ __forceinline__ void add_targets(unsigned long long i,
                                            unsigned long long (&acc)[1 << DIM],
                                            std::integer_sequence<int, T...>) {
  ((acc[T] += std::integral_constant<int, Tab<DIM>::k.w[D][V][T]>::value * i), ...);
}

// an entry in units of 2^(e - kB); bad turns negative for one below 0 or from 2^(e + 1) on
__device__ __forceinline__ unsigned long long entry_fixed(double e, int shift, int& bad) {
  const int hi = __double2hiint(e), sh = shift - (hi >> 20);
  bad |= hi | (sh - 7);
  const unsigned long long m =
      ((unsigned long long)(((uint32_t)hi & 0xfffffu) | 0x100000u) << 32 |
       (uint32_t)__double2loint(e)) << 10;
  return m >> min((unsigned)sh, 63u);
}

// Integers of the lane before in this lane's units: 2^k larger ones lose k bits (at most
// kMaxStep; nodes whose left neighbour's exponent is further above theirs are summed in FP64).
constexpr int kMaxStep = 12;
struct Left {
  int up, down;
  __device__ __forceinline__ unsigned long long units(unsigned long long i, int& bad) const {
    bad |= (1 << (kB + 1 - 32 - up)) - 1 - (int)(i >> 32);  // an entry from 2^(e + 1) on
    return i >> down << up;
  }
};

// The entries D of one row of the cell (fine nodes 2a - 1, 2a, 2a + 1 in x): a thread loads the
// pair from 2a on and takes 2a - 1 from the lane before it.
template <int DIM, int D, int R>
__device__ __forceinline__ void add_row(const Entries<DIM>& f, size_t kf, int pitch, long plane,
                                        int shift, const Left& left, int& bad,
                                        unsigned long long (&acc)[1 << DIM]) {
  constexpr bool l = Tab<DIM>::k.used(D, 3 * R), m = Tab<DIM>::k.used(D, 3 * R + 1),
                 r = Tab<DIM>::k.used(D, 3 * R + 2);
  constexpr auto targets = std::make_integer_sequence<int, 1 << DIM>();
  if constexpr (l || m || r) {
    const double* p = f.a[D] + kf + offset<DIM>(3 * R + 1, pitch, plane);
    const double2 v = __ldg(reinterpret_cast<const double2*>(p));
    if constexpr (m) add_targets<DIM, D, 3 * R + 1>(entry_fixed(v.x, shift, bad), acc, targets);
    if constexpr (l || r) {
      const unsigned long long i = entry_fixed(v.y, shift, bad);
      if constexpr (r) add_targets<DIM, D, 3 * R + 2>(i, acc, targets);
      if constexpr (l) {
        unsigned long long j = __shfl_up_sync(0xffffffffu, i, 1);
        if (threadIdx.x == 0) j = entry_fixed(__ldg(p - 1), shift, bad);
        else j = left.units(j, bad);
        add_targets<DIM, D, 3 * R>(j, acc, targets);
      }
    }
  }
}

template <int DIM, int... Q>
__device__ __forceinline__ void add_entries(const Entries<DIM>& f, size_t kf, int pitch,
                                            long plane, int shift, const Left& left, int& bad,
                                            unsigned long long (&acc)[1 << DIM],
                                            std::integer_sequence<int, Q...>) {
  constexpr int E = 1 << DIM;
  (add_row<DIM, Q % E, Q / E>(f, kf, pitch, plane, shift, left, bad, acc), ...);
}

// blockDim (32, kY): a warp per coarse row piece (the lanes pass on the entry left of their
// pair); planes and instances share blockIdx.z.
// Entries towards coarse boundary nodes are formed as well (from interior fine entries only);
// nothing but the next coarsening reads them, for its own boundary entries.
constexpr int kY = 4;
template <int DIM>
__global__ void __launch_bounds__(32 * kY, 4)
    k_coarsen_fx(int nc, int pc, int pf, size_t stc, size_t stf,
                 const __grid_constant__ Entries<DIM> f, const __grid_constant__ Entries<DIM> c) {
  using M = Mesh<DIM>;
  const int I = 1 + blockIdx.x * 32 + threadIdx.x, J = 1 + blockIdx.y * kY + threadIdx.y;
  if (J >= nc) return;  // uniform over the warp
  const int planes = DIM == 3 ? nc - 1 : 1, ib = blockIdx.z / planes;
  const int L = DIM == 3 ? 1 + (int)blockIdx.z - ib * planes : 0;
  const long planef = (long)(2 * nc + 1) * pf;
  const size_t kf = ib * stf + 2 * L * planef + (size_t)(2 * J) * pf + 2 * min(I, nc - 1);
  int top = 0;
#pragma unroll
  for (int v = 0; v < M::kPos; ++v) {
    // 2a and the corners of its cell
    const bool corner = M::px(v) != 0 && M::py(v) != 0 && (DIM == 2 || M::pz(v) != 0);
    if (v == M::kPos / 2 || corner)
      top = max(top, __double2hiint(__ldg(f.a[0] + kf + offset<DIM>(v, pf, planef))));
  }
  const int e0 = ((top + 1) >> 20) - 1022;
  const size_t kc = ib * stc + ((size_t)L * (nc + 1) + J) * pc + I;
  int bad = e0 < -kMaxExp || e0 > kMaxExp ? -1 : 0;
  if (__any_sync(0xffffffffu, bad == 0)) {
    const int e = bad == 0 ? e0 : 0;
    const int before = __shfl_up_sync(0xffffffffu, bad == 0 ? e0 : 4096, 1);
    const int step = threadIdx.x == 0 ? 0 : before - e;
    if (step > kMaxStep) bad = -1;
    const Left left{min(max(step, 0), kMaxStep), min(max(-step, 0), 63)};
    unsigned long long acc[M::kEnt];
    start_targets<DIM>(acc, std::make_integer_sequence<int, M::kEnt>());
    add_entries<DIM>(f, kf, pf, planef, e + 1085 - kB, left, bad, acc,
                     std::make_integer_sequence<int, M::kEnt * M::kPos / 3>());
    // an entry that the lane before could not take in (and passed on)
    const int passed = __shfl_up_sync(0xffffffffu, bad, 1);
    if (threadIdx.x && passed < 0) bad = -1;
#pragma unroll
    for (int T = 0; T < M::kEnt; ++T) {
      const bool inner = (!M::dx(T) || I + 1 < nc) && (!M::dy(T) || J + 1 < nc) &&
                         (!M::dz(T) || L + 1 < nc);
      if (inner && (acc[T] >> kLeast) == 0) bad = -1;
    }
    if (bad >= 0 && I < nc) {
#pragma unroll
      for (int T = 0; T < M::kEnt; ++T) {
        const double d = __ull2double_rn(acc[T]);
        c.a[T][kc] = __hiloint2double(__double2hiint(d) + (e - kB - 2) * (1 << 20),
                                      __double2loint(d));
      }
    }
  }
  if (bad < 0 && I < nc) node_fp64<DIM>(f, c, kf, kc, pf, planef);
}

template <int DIM>
void launch(const Grid& fine, const Grid& coarse, const Entries<DIM>& f, const Entries<DIM>& c,
            cudaStream_t s) {
  const int m = coarse.n - 1;
  const dim3 grid((m + 31) / 32, (m + kY - 1) / kY, fine.nb * (DIM == 3 ? m : 1));
  k_coarsen_fx<DIM><<<grid, dim3(32, kY), 0, s>>>(coarse.n, coarse.pitch, fine.pitch,
                                                  coarse.stride, fine.stride, f, c);
}

}  // namespace

void coarsen_density2d(const Grid& fine, const Grid& coarse, const Density2D& bf,
                       const Density2D& bc, cudaStream_t s) {
  launch<2>(fine, coarse, {bf.C, bf.E, bf.N, bf.NE}, {bc.C, bc.E, bc.N, bc.NE}, s);
}

void coarsen_density3d(const Grid& fine, const Grid& coarse, const Density3D& bf,
                       const Density3D& bc, cudaStream_t s) {
  Entries<3> f, c;
  for (int d = 0; d < 8; ++d) {
    f.a[d] = bf.a[d];
    c.a[d] = bc.a[d];
  }
  launch<3>(fine, coarse, f, c, s);
}

}  // namespace fmg
