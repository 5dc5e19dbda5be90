// Host-built index lists of the small dense solves (dense.cu): the sparsity of the coarse
// block and of the third moments T3 on the coarse mesh T_H.  No heap use, so the
// allocation-free coarse solve can build them too.
#pragma once

#include <stdint.h>

namespace fmg {

constexpr int kDenseMaxNh = 64;        // coarse unknowns (2D: 9 coarse cells per side)
constexpr int kDenseMaxTriples = 512;  // distinct interior vertex triples of one simplex
constexpr int kDenseMaxLists = 6144;   // entries of all lists together

// Sizes of the lists, which lie one after another in one array of 16-bit entries:
//   rowptr[nh + 1]  entries of coarse row a, the diagonal first, then by column
//   pair[npat]      entry -> a << 8 | b (a, b share a simplex)
//   simptr[npat + 1], sim[nsim]  the simplices that contain a and b
//   x3ptr[npat + 1], x3[nx]      c | q << 6: the triples q that contain a, b, and their third
//                                vertex c, so that sum_T sum_c w_c T3_abc = sum w_c tau_q
//   tripptr[nq + 1], trip[ntrip] triple q -> the entries t nt3 + i of T3 that it sums (tau_q)
struct DenseLists {
  int npat = 0, nsim = 0, nx = 0, nq = 0, ntrip = 0;
  __host__ __device__ int pair(int nh) const { return nh + 1; }
  __host__ __device__ int simptr(int nh) const { return pair(nh) + npat; }
  __host__ __device__ int sim(int nh) const { return simptr(nh) + npat + 1; }
  __host__ __device__ int x3ptr(int nh) const { return sim(nh) + nsim; }
  __host__ __device__ int x3(int nh) const { return x3ptr(nh) + npat + 1; }
  __host__ __device__ int tripptr(int nh) const { return x3(nh) + nx; }  // end of the staged part
  __host__ __device__ int trip(int nh) const { return tripptr(nh) + nq + 1; }
  __host__ __device__ int total(int nh) const { return trip(nh) + ntrip; }
  // entries kept on the device, whose kernels copy 16 bytes at a time: none for a mesh whose lists
  // could not be built (it is refused)
  int stored(int nh) const { return npat ? (total(nh) + 7) / 8 * 8 : 0; }
};

// Fill `out` (capacity kDenseMaxLists) for the ntri simplices tri[t * nv + v] (coarse interior
// index, -1 on the boundary); false when a capacity does not hold them.
inline bool build_dense_lists(int nh, int ntri, int nv, const int* tri, uint16_t* out,
                              DenseLists* dims) {
  if (nh < 1 || nh > kDenseMaxNh) return false;
  *dims = DenseLists{};
  // entry index of (a, b), the diagonal first in each row
  uint16_t entry[kDenseMaxNh][kDenseMaxNh];
  for (int a = 0; a < nh; ++a)
    for (int b = 0; b < nh; ++b) entry[a][b] = 0;
  auto interior = [&](int t, int* v) {
    int m = 0;
    for (int i = 0; i < nv; ++i)
      if (tri[t * nv + i] >= 0) v[m++] = i;
    return m;
  };
  int lv[4];
  for (int t = 0; t < ntri; ++t) {  // count the simplices of each entry
    const int m = interior(t, lv);
    for (int i = 0; i < m; ++i)
      for (int j = 0; j < m; ++j) entry[tri[t * nv + lv[i]]][tri[t * nv + lv[j]]]++;
  }
  int npat = 0, nsim = 0;
  for (int a = 0; a < nh; ++a)
    for (int b = 0; b < nh; ++b)
      if (entry[a][b]) {
        ++npat;
        nsim += entry[a][b];
      }
  // the distinct triples a <= b <= c of interior vertices of a simplex, by open addressing
  constexpr int kSlots = 2048;
  uint32_t key[kDenseMaxTriples];
  uint16_t slot[kSlots], count[kDenseMaxTriples];
  for (int s = 0; s < kSlots; ++s) slot[s] = 0xffff;
  int nq = 0, ntrip = 0;
  auto find = [&](int a, int b, int c, bool insert) -> int {
    if (a > b) { const int x = a; a = b; b = x; }
    if (b > c) { const int x = b; b = c; c = x; }
    if (a > b) { const int x = a; a = b; b = x; }
    const uint32_t k = (uint32_t)a << 16 | (uint32_t)b << 8 | (uint32_t)c;
    for (uint32_t s = (k * 2654435761u) >> 21;; s = (s + 1) % kSlots) {
      if (slot[s] == 0xffff) {
        if (!insert || nq >= kDenseMaxTriples) return -1;
        key[nq] = k;
        count[nq] = 0;
        slot[s] = (uint16_t)nq;
        return nq++;
      }
      if (key[slot[s]] == k) return slot[s];
    }
  };
  // numbered by their vertex count (1, 2, 3), so that the lists of neighbouring triples have
  // about the same length
  for (int verts = 1; verts <= 3; ++verts)
    for (int t = 0; t < ntri; ++t) {
      const int m = interior(t, lv);
      for (int i = 0; i < m; ++i)
        for (int j = i; j < m; ++j)
          for (int k = j; k < m; ++k) {
            if (1 + (i != j) + (j != k) != verts) continue;
            const int q = find(tri[t * nv + lv[i]], tri[t * nv + lv[j]], tri[t * nv + lv[k]], true);
            if (q < 0) return false;
            ++count[q];
            ++ntrip;
          }
    }
  // (a, b) entries of a triple with the remaining vertex c, by distinct ordered pairs
  auto pairs_of = [&](int q, auto&& f) {
    const int x = key[q] >> 16, y = key[q] >> 8 & 255, z = key[q] & 255;
    if (x == y && y == z) {
      f(x, x, x);
    } else if (x == y || y == z) {
      const int d = y, o = x == y ? z : x;  // the doubled vertex and the other one
      f(d, d, o);
      f(d, o, d);
      f(o, d, d);
    } else {
      f(x, y, z); f(y, x, z); f(x, z, y); f(z, x, y); f(y, z, x); f(z, y, x);
    }
  };
  int nx = 0;
  for (int q = 0; q < nq; ++q) pairs_of(q, [&](int, int, int) { ++nx; });
  dims->npat = npat;
  dims->nsim = nsim;
  dims->nx = nx;
  dims->nq = nq;
  dims->ntrip = ntrip;
  if (dims->total(nh) > kDenseMaxLists) return false;
  // rows, and the start of every entry's simplex list
  uint16_t *rowptr = out, *pair = out + dims->pair(nh), *simptr = out + dims->simptr(nh),
           *sim = out + dims->sim(nh), *x3ptr = out + dims->x3ptr(nh), *x3 = out + dims->x3(nh),
           *tripptr = out + dims->tripptr(nh), *trip = out + dims->trip(nh);
  int e = 0, ns = 0;
  for (int a = 0; a < nh; ++a) {
    rowptr[a] = (uint16_t)e;
    for (int b = -1; b < nh; ++b) {
      const int col = b < 0 ? a : b;
      if (b == a || !entry[a][col]) continue;
      pair[e] = (uint16_t)(a << 8 | col);
      simptr[e] = (uint16_t)ns;
      ns += entry[a][col];
      entry[a][col] = (uint16_t)e++;
    }
  }
  rowptr[nh] = (uint16_t)e;
  simptr[e] = (uint16_t)ns;
  for (int t = 0; t < ntri; ++t) {
    const int m = interior(t, lv);
    for (int i = 0; i < m; ++i)
      for (int j = 0; j < m; ++j)
        sim[simptr[entry[tri[t * nv + lv[i]]][tri[t * nv + lv[j]]]]++] = (uint16_t)t;
  }
  for (int i = npat; i > 0; --i) simptr[i] = simptr[i - 1];  // undo the fill's advance
  simptr[0] = 0;
  // third-moment lists
  for (int i = 0; i <= npat; ++i) x3ptr[i] = 0;
  for (int q = 0; q < nq; ++q) pairs_of(q, [&](int a, int b, int) { ++x3ptr[entry[a][b] + 1]; });
  for (int i = 0; i < npat; ++i) x3ptr[i + 1] = (uint16_t)(x3ptr[i + 1] + x3ptr[i]);
  for (int q = 0; q < nq; ++q)
    pairs_of(q, [&](int a, int b, int c) { x3[x3ptr[entry[a][b]]++] = (uint16_t)(c | q << 6); });
  for (int i = npat; i > 0; --i) x3ptr[i] = x3ptr[i - 1];
  x3ptr[0] = 0;
  tripptr[0] = 0;
  for (int q = 0; q < nq; ++q) tripptr[q + 1] = (uint16_t)(tripptr[q] + count[q]);
  const int nt3 = nv == 3 ? 10 : 20;
  for (int t = 0; t < ntri; ++t) {
    const int m = interior(t, lv);
    for (int i = 0; i < m; ++i)
      for (int j = i; j < m; ++j)
        for (int k = j; k < m; ++k) {
          // index of the sorted local triple (lv is ascending)
          const int a = lv[i], b = lv[j], c = lv[k];
          int idx = 0;
          for (int x = 0; x < a; ++x) idx += (nv - x) * (nv - x + 1) / 2;
          for (int y = a; y < b; ++y) idx += nv - y;
          const int q = find(tri[t * nv + a], tri[t * nv + b], tri[t * nv + c], false);
          trip[tripptr[q]++] = (uint16_t)(t * nt3 + idx + (c - b));
        }
  }
  for (int i = nq; i > 0; --i) tripptr[i] = tripptr[i - 1];
  tripptr[0] = 0;
  return true;
}

}  // namespace fmg
