// pecc_cells.cuh -- cell binning of whole instances for the standalone kernels (list build, feasibility
// check, features), in two forms:
//   one block per instance (at most kCellsBlockN circles): everything in shared memory;
//   several blocks per instance (pecc_kernels.cu): one kernel per step over tiles of all such instances.
// Both sort the circles by (cell, index) and keep their coordinates in that order rounded to binary32.
//
// GB300 has two binary64 lanes per SM and clock, so the searches work on the binary32 copies and
// decide in binary64 only what those cannot: a cell index within kCellSlack of a cell's edge, a
// distance within `slack` of the cutoff.  The results are those of the binary64 operations throughout.
#pragma once

#include "pecc_internal.h"

namespace pecc {

// The coordinates a search reads.
template <typename T> struct Coords;
template <> struct Coords<float> {
  using point = float2;
  const float2 *x;
  double l_cut;
  __device__ __forceinline__ float2 at(int i) const { return x[i]; }
  __device__ __forceinline__ float2 low(int i) const { return x[i]; }
};
template <> struct Coords<double> {
  using point = double2;
  const double2 *x;
  const float2 *x32;  // if set: binary32 coordinates, widened
  double l_cut;
  __device__ __forceinline__ double2 at(int i) const {
    if (x32) { const float2 f = x32[i]; return make_double2((double)f.x, (double)f.y); }
    return x[i];
  }
  __device__ __forceinline__ float2 low(int i) const {
    if (x32) return x32[i];
    const double2 v = x[i];
    return make_float2((float)v.x, (float)v.y);
  }
};

// The neighbor predicate of Sec. 4.3 for circle i (binary32 coordinates xf, given to set()) against the
// circle at sorted position q.
template <typename T> struct Near;
template <> struct Near<float> {
  float lc2;
  float2 xf;
  __device__ __forceinline__ explicit Near(double l_cut) : lc2((float)(l_cut * l_cut)) {}
  __device__ __forceinline__ void set(float2 x) { xf = x; }
  template <typename I>
  __device__ __forceinline__ bool operator()(int, float2 xq, const Coords<float> &, const I *, int) const {
    return nbr_pred(xf, xq, lc2);
  }
};
template <> struct Near<double> {
  double lc2;
  float lc;
  float2 xf;
  float lo, hi;
  __device__ __forceinline__ explicit Near(double l_cut) : lc2(l_cut * l_cut), lc((float)l_cut) {}
  __device__ __forceinline__ void set(float2 x) {
    xf = x;
    near_bounds(x, lc, lo, hi);
  }
  template <typename I>
  __device__ __forceinline__ bool operator()(int i, float2 xq, const Coords<double> &X, const I *ord, int q) const {
    const float dx = xf.x - xq.x, dy = xf.y - xq.y, s = dx * dx + dy * dy;
    if (s > hi) return false;
    if (s < lo) return true;
    return nbr_pred(X.at(i), X.at(ord[q]), lc2);
  }
};

// A coordinate that is not finite, without a binary64 operation.
__device__ __forceinline__ bool not_finite(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }
__device__ __forceinline__ bool not_finite(float v) { return (__float_as_uint(v) & 0x7f800000u) == 0x7f800000u; }

// ---- one block per instance ----
// Shared-memory layout for an instance of n circles: coordinates in cell order (binary64 searches: and
// in index order, so that each is converted once), then three 16-bit arrays, then `extra` bytes of the kernel's own, then the cell table when it fits its share (1.25 cells
// per circle: the layouts of this library have about 0.8), else the table in global memory.
__host__ __device__ inline int cell_share(int n) { return n + n / 4 + 64 < 256 ? 256 : n + n / 4 + 64; }
__host__ __device__ inline size_t cells_r16(size_t b) { return (b + 15) & ~size_t(15); }
__host__ __device__ inline size_t cells_smem(int n, size_t extra, bool wide) {
  return (wide ? 2 : 1) * cells_r16(8 * (size_t)n) + 3 * cells_r16(2 * (size_t)n) + extra + 4 * (size_t)(cell_share(n) + 1);
}
struct BlockCells {
  float2 *xs;            // coordinates in cell order (rounded to binary32)
  const float2 *xi;      // ... in index order (binary32 searches: the caller's)
  uint16_t *key, *ord;   // cell of circle i; circle at sorted position p
  int32_t *start;        // cell starts, ncell + 1
  unsigned char *extra;
};

// Sort the n circles by (cell, index).  ckey / corder (may be null): the cells and the order for export.
// visit(point, binary32 point, i): called once per circle by its thread while its coordinates are at hand.
template <typename T, typename Visit>
__device__ __forceinline__ BlockCells block_cells(const Coords<T> &X, int n, double R, double inv, int nc,
                                                  unsigned char *sm, size_t extra, int32_t *cells_g, uint32_t *ckey,
                                                  int32_t *corder, int32_t *sh, Visit visit) {
  const int tid = threadIdx.x, B = blockDim.x;
  BlockCells C;
  const size_t nb = cells_r16(2 * (size_t)n);
  C.xs = (float2 *)sm;
  sm += cells_r16(8 * (size_t)n);
  float2 *xi = nullptr;
  if constexpr (sizeof(T) == 8) {
    C.xi = xi = (float2 *)sm;
    sm += cells_r16(8 * (size_t)n);
  } else {
    C.xi = X.x;
  }
  C.key = (uint16_t *)sm;
  uint16_t *tmp = (uint16_t *)((unsigned char *)C.key + nb);
  C.ord = (uint16_t *)((unsigned char *)tmp + nb);  // until the last step: arrival rank within the cell
  C.extra = (unsigned char *)C.ord + nb;
  const int ncell = nc * nc;
  C.start = ncell <= cell_share(n) ? (int32_t *)(C.extra + extra) : cells_g;
  for (int c = tid; c <= ncell; c += B) C.start[c] = 0;
  __syncthreads();
  for (int i = tid; i < n; i += B) {
    const typename Coords<T>::point p = X.at(i);
    const float2 f = make_float2((float)p.x, (float)p.y);
    if constexpr (sizeof(T) == 8) xi[i] = f;
    const int key = cell_key_fast(p, f, R, inv, nc);
    C.key[i] = (uint16_t)key;
    if (ckey) ckey[i] = (uint32_t)key;
    C.ord[i] = (uint16_t)atomicAdd(&C.start[key + 1], 1);
    visit(p, f, i);
  }
  __syncthreads();
  block_scan_inplace(C.start + 1, ncell, sh);
  for (int i = tid; i < n; i += B) tmp[C.start[C.key[i]] + C.ord[i]] = (uint16_t)i;
  __syncthreads();
  // arrival order to index order: a circle's place in its cell is the number of smaller indices there
  for (int p = tid; p < n; p += B) {
    const int i = tmp[p], c = C.key[i];
    int r = C.start[c];
    for (int q = C.start[c], hi = C.start[c + 1]; q < hi; ++q) r += tmp[q] < i;
    C.ord[r] = (uint16_t)i;
    C.xs[r] = C.xi[i];
    if (corder) corder[r] = i;
  }
  __syncthreads();
  return C;
}

}  // namespace pecc
