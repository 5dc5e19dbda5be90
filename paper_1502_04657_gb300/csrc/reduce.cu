// Deterministic FP64 dot products: fixed block count and fixed-order trees, so the result
// does not depend on scheduling (no atomics).
#include "fmg_internal.h"

namespace fmg {
namespace {

constexpr int kThreads = 256;

// Fixed-order block reduction for thread 0: lane trees inside each warp, then warp 0 over the
// warp sums.
__device__ double block_sum_warps(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double t = 0.0;
  if (w == 0) {
    t = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  }
  return t;
}

// instance blockIdx.y: a, b at blockIdx.y * vst, partials at blockIdx.y * kReduceBlocks.
// Block blockIdx.x sums elements [beg, end) of a chunk (an even number of elements, so the
// pairs are 16-byte aligned): each thread takes pairs in a fixed order into two accumulators
// per lane of the pair, then the block tree.
__global__ void k_dot_partial(const double* __restrict__ a, const double* __restrict__ b,
                              size_t n, size_t vst, size_t chunk, double* __restrict__ partials) {
  __shared__ double sh[kThreads / 32];
  a += blockIdx.y * vst;
  b += blockIdx.y * vst;
  partials += (size_t)blockIdx.y * kReduceBlocks;
  const size_t beg = blockIdx.x * chunk;
  // a block past n (the even chunk may leave the last one empty) contributes 0
  const size_t end = beg >= n ? beg : (beg + chunk < n ? beg + chunk : n);
  const size_t pend = beg + ((end - beg) & ~(size_t)1);
  double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
  size_t i = beg + 2 * threadIdx.x;
  for (; i + 2 * kThreads < pend; i += 4 * kThreads) {
    const double2 x0 = *reinterpret_cast<const double2*>(a + i);
    const double2 y0 = *reinterpret_cast<const double2*>(b + i);
    const double2 x1 = *reinterpret_cast<const double2*>(a + i + 2 * kThreads);
    const double2 y1 = *reinterpret_cast<const double2*>(b + i + 2 * kThreads);
    s0 = fma(x0.x, y0.x, s0);
    s1 = fma(x0.y, y0.y, s1);
    s2 = fma(x1.x, y1.x, s2);
    s3 = fma(x1.y, y1.y, s3);
  }
  if (i < pend) {
    const double2 x0 = *reinterpret_cast<const double2*>(a + i);
    const double2 y0 = *reinterpret_cast<const double2*>(b + i);
    s0 = fma(x0.x, y0.x, s0);
    s1 = fma(x0.y, y0.y, s1);
  }
  if (threadIdx.x == 0 && pend < end) s0 = fma(a[pend], b[pend], s0);
  const double t = block_sum_warps((s0 + s1) + (s2 + s3), sh);
  if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

// a . b into partials, a . c into the second half (gridDim.y instances on): each in the order
// of k_dot_partial, with a read once
__global__ void k_dot2_partial(const double* __restrict__ a, const double* __restrict__ b,
                               const double* __restrict__ c, size_t n, size_t vst, size_t chunk,
                               double* __restrict__ partials) {
  __shared__ double sh[2][kThreads / 32];
  a += blockIdx.y * vst;
  b += blockIdx.y * vst;
  c += blockIdx.y * vst;
  const size_t beg = blockIdx.x * chunk;
  const size_t end = beg >= n ? beg : (beg + chunk < n ? beg + chunk : n);
  const size_t pend = beg + ((end - beg) & ~(size_t)1);
  double s[2][4] = {};
  auto pair = [&](size_t i, int q) {
    const double2 x = *reinterpret_cast<const double2*>(a + i);
    const double2 y = *reinterpret_cast<const double2*>(b + i);
    const double2 z = *reinterpret_cast<const double2*>(c + i);
    s[0][q] = fma(x.x, y.x, s[0][q]);
    s[0][q + 1] = fma(x.y, y.y, s[0][q + 1]);
    s[1][q] = fma(x.x, z.x, s[1][q]);
    s[1][q + 1] = fma(x.y, z.y, s[1][q + 1]);
  };
  size_t i = beg + 2 * threadIdx.x;
  for (; i + 2 * kThreads < pend; i += 4 * kThreads) {
    pair(i, 0);
    pair(i + 2 * kThreads, 2);
  }
  if (i < pend) pair(i, 0);
  if (threadIdx.x == 0 && pend < end) {
    s[0][0] = fma(a[pend], b[pend], s[0][0]);
    s[1][0] = fma(a[pend], c[pend], s[1][0]);
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const double t = block_sum_warps((s[q][0] + s[q][1]) + (s[q][2] + s[q][3]), sh[q]);
    if (threadIdx.x == 0)
      partials[((size_t)q * gridDim.y + blockIdx.y) * kReduceBlocks + blockIdx.x] = t;
  }
}

// instance blockIdx.x of the dot blockIdx.y
__global__ void k_sum_final(const double* __restrict__ partials, int m, double* out,
                            double* out2) {
  __shared__ double sh[kThreads / 32];
  partials += ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * kReduceBlocks;
  out = (blockIdx.y ? out2 : out) + blockIdx.x;
  double s = 0.0;
  for (int i = threadIdx.x; i < m; i += kThreads) s += partials[i];
  const double t = block_sum_warps(s, sh);
  if (threadIdx.x == 0) out[0] = t;
}

// the split of a dot product of n elements
unsigned dot_blocks(size_t n, size_t per_block, size_t& chunk) {
  // at least per_block elements per block, at most kReduceBlocks blocks: the split does not
  // depend on nb, so an instance sums in the same order alone and in a batch
  size_t blocks = (n + per_block - 1) / per_block;
  if (blocks > (size_t)kReduceBlocks) blocks = kReduceBlocks;
  if (blocks < 1) blocks = 1;
  chunk = (n + blocks - 1) / blocks;
  chunk += chunk & 1;  // even: every block's pairs start 16-byte aligned
  return (unsigned)blocks;
}

}  // namespace

void dot(const double* a, const double* b, size_t n, double* partials, double* out,
         cudaStream_t s, int nb, size_t vst, size_t per_block) {
  size_t chunk;
  const unsigned blocks = dot_blocks(n, per_block, chunk);
  k_dot_partial<<<dim3(blocks, nb), kThreads, 0, s>>>(a, b, n, vst, chunk, partials);
  k_sum_final<<<nb, kThreads, 0, s>>>(partials, (int)blocks, out, nullptr);
}

void dot2(const double* a, const double* b, const double* c, size_t n, double* partials,
          double* out, double* out2, cudaStream_t s, int nb, size_t vst, size_t per_block) {
  size_t chunk;
  const unsigned blocks = dot_blocks(n, per_block, chunk);
  k_dot2_partial<<<dim3(blocks, nb), kThreads, 0, s>>>(a, b, c, n, vst, chunk, partials);
  k_sum_final<<<dim3(nb, 2), kThreads, 0, s>>>(partials, (int)blocks, out, out2);
}

namespace {

// Conjugate gradient steps over whole level vectors (boundary and padding entries are zero in
// p, q and r and stay zero), instance blockIdx.y.  On the levels the smoother runs on, launches
// and their gaps count for more than the memory passes, so the dot products are formed where
// their factors are written (r . r in the update of r, or with the first copy of r to p), and
// the blocks of the kernel that needs a dot product add up its partial sums themselves, in one
// fixed order, instead of a launch for it: 4 launches per step (3 in the last) and 1 to start
// where one per operation and sum took 7 and 4: a solve on 3D h = 1/64 went from 2.86 to 2.25 ms.
// Block blockIdx.x takes elements [beg, end) of an even chunk, 2048 (8 per thread) or more.

// the sum of m partial sums, for thread 0
__device__ __forceinline__ double sum_partials(const double* __restrict__ partials, int m,
                                               double* sh) {
  double s = 0.0;
  for (int i = threadIdx.x; i < m; i += kThreads) s += partials[i];
  return block_sum_warps(s, sh);
}

// f(i) for this thread's pairs of elements (i, i + 1), in a fixed order (n is even)
template <typename F>
__device__ __forceinline__ void for_chunk(size_t n, size_t chunk, F f) {
  const size_t beg = blockIdx.x * chunk, end = beg + chunk < n ? beg + chunk : n;
  for (size_t i = beg + 2 * threadIdx.x; i < end; i += 2 * kThreads) f(i);
}

__global__ void __launch_bounds__(kThreads)
    k_cg_start(size_t n, size_t chunk, const double* __restrict__ r, double* __restrict__ p,
               double* __restrict__ partials) {
  __shared__ double sh[kThreads / 32];
  const size_t b = blockIdx.y * n;
  double s0 = 0.0, s1 = 0.0;
  for_chunk(n, chunk, [&](size_t i) {
    const double2 v = *reinterpret_cast<const double2*>(r + b + i);
    *reinterpret_cast<double2*>(p + b + i) = v;
    s0 = fma(v.x, v.x, s0);
    s1 = fma(v.y, v.y, s1);
  });
  const double t = block_sum_warps(s0 + s1, sh);
  if (threadIdx.x == 0) partials[(size_t)blockIdx.y * kReduceBlocks + blockIdx.x] = t;
}

__global__ void __launch_bounds__(kThreads)
    k_cg_dot(size_t n, size_t chunk, const double* __restrict__ p, const double* __restrict__ q,
             double* __restrict__ partials) {
  __shared__ double sh[kThreads / 32];
  const size_t b = blockIdx.y * n;
  double s0 = 0.0, s1 = 0.0;
  for_chunk(n, chunk, [&](size_t i) {
    const double2 v = *reinterpret_cast<const double2*>(p + b + i);
    const double2 w = *reinterpret_cast<const double2*>(q + b + i);
    s0 = fma(v.x, w.x, s0);
    s1 = fma(v.y, w.y, s1);
  });
  const double t = block_sum_warps(s0 + s1, sh);
  if (threadIdx.x == 0) partials[(size_t)blockIdx.y * kReduceBlocks + blockIdx.x] = t;
}

// x += a p, r -= a q with a = r.r / p.q (a zero denominator gives a zero step, as in the
// oracle), and the partial sums of the new r . r.  r.r comes from its partial sums rr_parts and
// is kept in rr, or, where rr_parts is null, from rr.
__global__ void __launch_bounds__(kThreads)
    k_cg_update(size_t n, size_t chunk, double* __restrict__ rr,
                const double* __restrict__ rr_parts, const double* __restrict__ pq_parts,
                const double* __restrict__ p, const double* __restrict__ q,
                double* __restrict__ x, double* __restrict__ r, double* __restrict__ partials) {
  __shared__ double sh[2][kThreads / 32], step;
  const size_t b = blockIdx.y * n, pb = (size_t)blockIdx.y * kReduceBlocks;
  const double pq = sum_partials(pq_parts + pb, gridDim.x, sh[0]);
  const double sum = rr_parts ? sum_partials(rr_parts + pb, gridDim.x, sh[1]) : 0.0;
  if (threadIdx.x == 0) {
    const double rr_old = rr_parts ? sum : rr[blockIdx.y];
    if (rr_parts && blockIdx.x == 0) rr[blockIdx.y] = rr_old;
    step = pq > 0.0 ? rr_old / pq : 0.0;
  }
  __syncthreads();
  const double a = step;
  double s0 = 0.0, s1 = 0.0;
  for_chunk(n, chunk, [&](size_t i) {
    const double2 pv = *reinterpret_cast<const double2*>(p + b + i);
    const double2 qv = *reinterpret_cast<const double2*>(q + b + i);
    double2 xv = *reinterpret_cast<double2*>(x + b + i), rv = *reinterpret_cast<double2*>(r + b + i);
    xv.x = fma(a, pv.x, xv.x);
    xv.y = fma(a, pv.y, xv.y);
    rv.x = fma(-a, qv.x, rv.x);
    rv.y = fma(-a, qv.y, rv.y);
    *reinterpret_cast<double2*>(x + b + i) = xv;
    *reinterpret_cast<double2*>(r + b + i) = rv;
    s0 = fma(rv.x, rv.x, s0);
    s1 = fma(rv.y, rv.y, s1);
  });
  const double t = block_sum_warps(s0 + s1, sh[0]);
  if (threadIdx.x == 0) partials[pb + blockIdx.x] = t;
}

// p = r + b p, b = rr_new / rr_old (rr_new from its partial sums, kept in rr_new)
__global__ void __launch_bounds__(kThreads)
    k_cg_direction(size_t n, size_t chunk, const double* __restrict__ rr_old,
                   const double* __restrict__ parts, double* __restrict__ rr_new,
                   const double* __restrict__ r, double* __restrict__ p) {
  __shared__ double sh[kThreads / 32], ratio;
  const double rn = sum_partials(parts + (size_t)blockIdx.y * kReduceBlocks, gridDim.x, sh);
  if (threadIdx.x == 0) {
    const double ro = rr_old[blockIdx.y];
    if (blockIdx.x == 0) rr_new[blockIdx.y] = rn;
    ratio = ro > 0.0 ? rn / ro : 0.0;
  }
  __syncthreads();
  const double c = ratio;
  const size_t b = blockIdx.y * n;
  for_chunk(n, chunk, [&](size_t i) {
    const double2 rv = *reinterpret_cast<const double2*>(r + b + i);
    double2 pv = *reinterpret_cast<double2*>(p + b + i);
    pv.x = fma(c, pv.x, rv.x);
    pv.y = fma(c, pv.y, rv.y);
    *reinterpret_cast<double2*>(p + b + i) = pv;
  });
}

// the split of a level's vectors (n elements each, n even): it depends on n alone
dim3 cg_grid(size_t n, int nb, size_t& chunk) {
  size_t blocks = (n + 2047) / 2048;
  if (blocks > (size_t)kReduceBlocks) blocks = kReduceBlocks;
  chunk = (n + blocks - 1) / blocks;
  chunk += chunk & 1;
  return dim3((unsigned)((n + chunk - 1) / chunk), nb);
}

}  // namespace

void cg_start(size_t n, int nb, const double* r, double* p, double* rr_parts, cudaStream_t s) {
  size_t chunk;
  const dim3 g = cg_grid(n, nb, chunk);
  k_cg_start<<<g, kThreads, 0, s>>>(n, chunk, r, p, rr_parts);
}
void cg_dot(size_t n, int nb, const double* p, const double* q, double* pq_parts, cudaStream_t s) {
  size_t chunk;
  const dim3 g = cg_grid(n, nb, chunk);
  k_cg_dot<<<g, kThreads, 0, s>>>(n, chunk, p, q, pq_parts);
}
void cg_update(size_t n, int nb, double* rr, const double* rr_parts, const double* pq_parts,
               const double* p, const double* q, double* x, double* r, double* parts,
               cudaStream_t s) {
  size_t chunk;
  const dim3 g = cg_grid(n, nb, chunk);
  k_cg_update<<<g, kThreads, 0, s>>>(n, chunk, rr, rr_parts, pq_parts, p, q, x, r, parts);
}
void cg_direction(size_t n, int nb, const double* rr_old, const double* parts, double* rr_new,
                  const double* r, double* p, cudaStream_t s) {
  size_t chunk;
  const dim3 g = cg_grid(n, nb, chunk);
  k_cg_direction<<<g, kThreads, 0, s>>>(n, chunk, rr_old, parts, rr_new, r, p);
}

}  // namespace fmg
