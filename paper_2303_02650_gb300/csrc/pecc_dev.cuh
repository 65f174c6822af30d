// pecc_dev.cuh -- device building blocks shared by the library's kernels.
//
// Elastic model of Sec. 3.2 (Eq. 3, Eq. 5), neighbor sets of Sec. 4.3, and
// the arithmetic forms the descent runs in:
//   Arith32  binary32 coordinates, pair math, gradient, energy accumulation
//   Arith64  binary64 everywhere (the plain FP64 form)
//   ArithMix binary64 coordinates, pair differences and the near-contact
//            quantities 4 - l^2 (two fused multiply-adds) and r^2 - (R-1)^2
//            (exact by Sterbenz' lemma where it cancels); binary32 for
//            everything that only needs relative accuracy (the overlap depth
//            from them, unit vectors, gradient, quasi-Newton vectors), binary64
//            energy sums.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace pecc {

constexpr int kMaxSlots = 11;        // m + 1 physical secant slots, m <= 10
constexpr int kBasis = 2 * kMaxSlots + 1;  // S slots, Y slots, g
constexpr int kMaxK = 64;            // batches per instance
constexpr int kMetaInts = 24;        // per batch: count, stage, ring[kMaxSlots], ...
constexpr int kMaxThreads = 1024;

// ---------------------------------------------------------------- layout ----
struct InstDesc {
  int32_t n, k, ncx, cap;   // circles, batches, cells per side, CSR capacity per buffer
  int32_t big, pad_;        // 1: descended by the whole GPU (pecc_grid.cu), not by one block
  int64_t off;              // first circle (positions, per-circle scratch)
  int64_t rp_off;           // 2 * (n + 1) row pointers (two CSR buffers)
  int64_t col_off;          // 2 * cap column entries (descent lists)
  int64_t col_s_off;        // cap column entries (standalone lists; row pointers at off + index)
  int64_t cell_off;         // cell table: cell_grid_cap(n)^2 + 1 counters
  int64_t gram_off;         // k * kGram Gram entries
  int64_t meta_off;         // k * kMetaInts ring metadata
  double R, inv_cs;
  float inv_f;              // binary32 grid of the FP32 descent: 1 / side, side >= l_cut (1 + 2^-10)
  int32_t ncx_f;            // its cells per side (<= ncx)
};

struct InstOut {
  int32_t iters, status, builds, changes, trials, resets, stalls, polished;
  int32_t iters32, status32, trials32, cur;
  double E, E32, max_overlap, pad;
};

// ------------------------------------------------------------ vec types ----
template <typename T> struct V2;
template <> struct V2<float> { using type = float2; };
template <> struct V2<double> { using type = double2; };
template <typename T> using v2 = typename V2<T>::type;

template <typename T> __device__ __forceinline__ v2<T> mk2(T a, T b) { v2<T> r; r.x = a; r.y = b; return r; }

// ---------------------------------------------------------------- philox ---
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11).
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) { k.x += 0x9E3779B9u; k.y += 0xBB67AE85u; }
    uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    uint4 n;
    n.x = hi1 ^ c.y ^ k.x;
    n.y = lo1;
    n.z = hi0 ^ c.w ^ k.y;
    n.w = lo0;
    c = n;
  }
  return c;
}

__device__ __forceinline__ double u53(uint32_t hi, uint32_t lo) {
  uint64_t w = ((uint64_t)hi << 32) | (uint64_t)lo;
  return __dmul_rn((double)(w >> 11), 1.0 / 9007199254740992.0);
}

// ---------------------------------------------------------------- cells ----
__device__ __forceinline__ int cell_coord(double v, double R, double inv, int nc) {
  double f = __dmul_rn(__dadd_rn(v, R), inv);
  if (!(f >= 0.0)) return 0;
  if (f >= (double)nc) return nc - 1;
  return (int)f;
}

// Cell coordinate of v (the value of cell_coord) decided in binary32 where that is certain.  In
// binary32 (v + R) inv is off by less than nc 2^-22 (three roundings of the operands, two of the
// operations, each relative 2^-24 of at most 2 R, and R inv <= nc / 2 up to a rounding), a quarter of
// the slack; a value further than the slack from an integer lies in the same cell.
template <typename V>
__device__ __forceinline__ int cell_coord_fast(V v, float vf, double R, double inv, int nc, float Rf, float invf,
                                               float slack) {
  const float f = (vf + Rf) * invf;
  const float fl = floorf(f), fr = f - fl;
  if (f < -slack) return 0;
  if (f > (float)nc + slack) return nc - 1;
  if (fr > slack && fr < 1.f - slack && f > 0.f && f < (float)nc) return (int)fl;
  return cell_coord((double)v, R, inv, nc);
}
// inv for it in binary32: NaN, which leaves every coordinate to binary64, for radii near the end of
// binary32's range, where v + R would overflow (and inv lose bits).
__device__ __forceinline__ float fast_inv(float Rf, double inv) {
  return Rf < 1e37f ? (float)inv : __int_as_float(0x7fc00000);
}
template <typename P>
__device__ __forceinline__ int cell_key_fast(P p, float2 f, double R, double inv, int nc) {
  const float Rf = (float)R, invf = fast_inv(Rf, inv), slack = (float)nc * (1.f / 1048576.f);
  const int cx = cell_coord_fast(p.x, f.x, R, inv, nc, Rf, invf, slack);
  return cell_coord_fast(p.y, f.y, R, inv, nc, Rf, invf, slack) * nc + cx;
}

// Distance slack around a circle whose coordinates are at most M in absolute value, for pairs near a
// distance l: the binary32 distance of the rounded coordinates is off by less than 2^-22 (M + l).
__device__ __forceinline__ float dist_slack(float M, float l) { return (M + l + 8.f) * (1.f / 1048576.f); }

// Bounds of the binary32 squared distances from a circle at x that decide the predicate for cutoff lc by
// themselves: below lo inside, above hi outside, the rest in binary64.
__device__ __forceinline__ void near_bounds(float2 x, float lc, float &lo, float &hi) {
  const float m = dist_slack(fabsf(x.x) + fabsf(x.y), lc);
  const bool ok = m <= 0.25f;  // else (far out, not finite): every distance in binary64
  lo = ok ? (lc - m) * (lc - m) : -1.f;
  hi = ok ? (lc + m) * (lc + m) : __int_as_float(0x7f800000);
}

// Neighbor predicate of Sec. 4.3: dx*dx + dy*dy < l_cut^2 with every operation
// correctly rounded (no contraction), in the coordinates' own precision.
__device__ __forceinline__ bool nbr_pred(float2 a, float2 b, float lc2) {
  float dx = __fsub_rn(a.x, b.x), dy = __fsub_rn(a.y, b.y);
  float s = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
  return s < lc2;
}
__device__ __forceinline__ bool nbr_pred(double2 a, double2 b, double lc2) {
  double dx = __dsub_rn(a.x, b.x), dy = __dsub_rn(a.y, b.y);
  double s = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
  return s < lc2;
}

// ------------------------------------------------------------ reductions ---
template <typename T> __device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <typename T> __device__ __forceinline__ T warp_max(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Block-wide sum of NV values per thread; every thread receives the totals in out[].
// scratch: at least (blockDim/32) * NV elements of T in shared memory.
template <typename T, int NV>
__device__ __forceinline__ void block_sum(T (&v)[NV], T *scratch, T *out) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    T s = warp_sum(v[q]);
    if (lane == 0) scratch[w * NV + q] = s;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < NV; q += blockDim.x) {
    T s = T(0);
    for (int u = 0; u < nw; ++u) s += scratch[u * NV + q];
    out[q] = s;
  }
  __syncthreads();
}

// Reduce-scatter of NV values over the 32 lanes of a warp (NV a multiple of 32): after the
// call, lane L holds in v[0 .. NV/32) the warp totals of the values with indices
// (NV/32) * L + j.  Takes NV - NV/32 shuffles instead of 5 NV for NV separate reductions.
template <typename T, int NV>
__device__ __forceinline__ void warp_reduce_scatter(T (&v)[NV]) {
  static_assert(NV % 32 == 0, "NV must be a multiple of 32");
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16, len = NV; o > 0; o >>= 1, len >>= 1) {
    const bool hi = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < len / 2; ++j) {
      T keep = hi ? v[j + len / 2] : v[j];
      T send = hi ? v[j] : v[j + len / 2];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
}

// Entry counts and row starts saturate here: above every list capacity (1e9 at most), and the sum of two
// such counts still fits 32 bits.
constexpr int32_t kMaxEntries = 0x3fffffff;

__device__ __forceinline__ int32_t sat_add(int32_t a, int32_t b) { return min(a + b, kMaxEntries); }

// Inclusive prefix sum of a[0..len) in place (int32), whole block.  SAT: the sums stop at kMaxEntries
// (entry counts of lists).
template <bool SAT = false>
__device__ inline void block_scan_inplace(int32_t *a, int len, int32_t *sh /*>=33 ints*/) {
  const int T = blockDim.x, t = threadIdx.x, lane = t & 31, w = t >> 5, nw = T >> 5;
  auto add = [](int32_t x, int32_t y) { return SAT ? sat_add(x, y) : x + y; };
  int ch = (len + T - 1) / T;
  int lo = min(len, t * ch), hi = min(len, lo + ch);
  int32_t s = 0;
  for (int i = lo; i < hi; ++i) s = add(s, a[i]);
  int32_t incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int32_t u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl = add(incl, u);
  }
  if (lane == 31) sh[w] = incl;
  __syncthreads();
  if (w == 0) {
    int32_t v = lane < nw ? sh[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int32_t u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v = add(v, u);
    }
    if (lane < nw) sh[lane] = v;
  }
  __syncthreads();
  int32_t run = w > 0 ? sh[w - 1] : 0;
  if constexpr (SAT) {  // a saturated sum cannot be taken back
    const int32_t prev = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane) run = sat_add(run, prev);
  } else {
    run += incl - s;
  }
  for (int i = lo; i < hi; ++i) { run = add(run, a[i]); a[i] = run; }
  __syncthreads();
}

// ------------------------------------------------------- neighbor build ----
// Cell grid of one instance.  Binary64 keys use the grid of the host (side l_cut (1 + 2^-20));
// the binary32 descent uses its own grid with side l_cut (1 + 2^-10), a margin far above the
// rounding of (x + R) / side in binary32, so that circles closer than l_cut are never two
// cells apart.  Either grid only accelerates the search: the set Gamma(i) is fixed by the
// predicate alone.
struct CellGrid {
  double R, inv;
  float Rf, invf;
  int nc;
  bool f32;
};

// Cell of a circle as cx | cy << 16 (a grid has at most 65535 cells per side).
template <typename T>
__device__ __forceinline__ uint32_t grid_cell(v2<T> p, const CellGrid &G) {
  int cx, cy;
  if (G.f32) {
    const float fx = ((float)p.x + G.Rf) * G.invf, fy = ((float)p.y + G.Rf) * G.invf;
    cx = !(fx >= 0.f) ? 0 : (fx >= (float)G.nc ? G.nc - 1 : (int)fx);
    cy = !(fy >= 0.f) ? 0 : (fy >= (float)G.nc ? G.nc - 1 : (int)fy);
  } else {
    const float Rf = (float)G.R, invf = fast_inv(Rf, G.inv), slack = (float)G.nc * (1.f / 1048576.f);
    cx = cell_coord_fast(p.x, (float)p.x, G.R, G.inv, G.nc, Rf, invf, slack);
    cy = cell_coord_fast(p.y, (float)p.y, G.R, G.inv, G.nc, Rf, invf, slack);
  }
  return (uint32_t)cx | ((uint32_t)cy << 16);
}
template <typename T>
__device__ __forceinline__ uint32_t grid_key(v2<T> p, const CellGrid &G) {
  const uint32_t c = grid_cell<T>(p, G);
  return (c >> 16) * (uint32_t)G.nc + (c & 0xffffu);
}

// 32-bit integer finaliser (xor-shift-multiply); a pair's digest term.  The digest only
// decides ANM's deferral length, never which list is used, so a collision costs nothing but
// a schedule change.
__device__ __forceinline__ unsigned long long mix32(uint32_t x) {
  x ^= x >> 16; x *= 0x7feb352du;
  x ^= x >> 15; x *= 0x846ca68bu;
  x ^= x >> 16;
  return (unsigned long long)x;
}

// Cell binning and stable key sort of one instance (the first half of a list build): ckey[i] = cell
// of circle i (cx | cy << 16), corder = circles sorted by (cell, index), cells[0..ncell] = cell starts,
// xs[q] = coordinates of corder[q] rounded to binary32.  tmp: n int32 of scratch.  A circle keeps its
// arrival rank from the count, so the scatter needs no second cursor, and then finds its place in its
// cell as the number of smaller indices there: every step one circle per thread (cells sorted one per
// thread, circle after circle, left most threads waiting).
template <typename T>
__device__ void cta_cell_sort(const v2<T> *__restrict__ x, int n, const CellGrid &G, uint32_t *ckey,
                              int32_t *corder, int32_t *cells, float2 *xs, int32_t *tmp, int32_t *sh) {
  const int T_ = blockDim.x, t = threadIdx.x;
  const int nc = G.nc, ncell = nc * nc;
  int32_t *cstart = cells;  // ncell + 1
  for (int c = t; c <= ncell; c += T_) cstart[c] = 0;
  __syncthreads();
  for (int i = t; i < n; i += T_) {
    const uint32_t c = grid_cell<T>(x[i], G);
    ckey[i] = c;
    corder[i] = atomicAdd(&cstart[(int)(c >> 16) * nc + (int)(c & 0xffffu) + 1], 1);
  }
  __syncthreads();
  block_scan_inplace(cstart + 1, ncell, sh);
  for (int i = t; i < n; i += T_) {
    const uint32_t c = ckey[i];
    tmp[cstart[(int)(c >> 16) * nc + (int)(c & 0xffffu)] + corder[i]] = i;
  }
  __syncthreads();
  for (int p = t; p < n; p += T_) {
    const int i = tmp[p];
    const uint32_t c = ckey[i];
    const int key = (int)(c >> 16) * nc + (int)(c & 0xffffu);
    const int lo = cstart[key], hi = cstart[key + 1];
    int r = lo;
    for (int q = lo; q < hi; ++q) r += tmp[q] < i;
    const v2<T> v = x[i];
    corder[r] = i;
    xs[r] = make_float2((float)v.x, (float)v.y);
  }
  __syncthreads();
}

// The predicate for the circle at sorted position q0 against the one at qq.  Binary64: decided by the
// binary32 copies except within the slack of the cutoff (about one pair in a million), so that a build
// leaves the two binary64 lanes of the SM alone: they took most of a polish's and an adjustment's builds.
template <typename T> struct SortedNear;
template <> struct SortedNear<float> {
  const float2 *xs;
  float lc2;
  float2 a;
  __device__ __forceinline__ SortedNear(const float2 *, const int32_t *, const float2 *xs_, float lc2_)
      : xs(xs_), lc2(lc2_) {}
  __device__ __forceinline__ void set(int q0) { a = xs[q0]; }
  __device__ __forceinline__ bool operator()(int qq) const { return nbr_pred(a, xs[qq], lc2); }
};
template <> struct SortedNear<double> {
  const double2 *x;
  const int32_t *order;
  const float2 *xs;
  double lc2;
  float lc, lo, hi;
  float2 a;
  int i;
  __device__ __forceinline__ SortedNear(const double2 *x_, const int32_t *o, const float2 *xs_, double lc2_)
      : x(x_), order(o), xs(xs_), lc2(lc2_), lc(sqrtf((float)lc2_)) {}
  __device__ __forceinline__ void set(int q0) {
    a = xs[q0];
    i = order[q0];
    near_bounds(a, lc, lo, hi);
  }
  __device__ __forceinline__ bool operator()(int qq) const {
    const float2 b = xs[qq];
    const float dx = a.x - b.x, dy = a.y - b.y, s = dx * dx + dy * dy;
    if (s > hi) return false;
    if (s < lo) return true;
    return nbr_pred(x[i], x[order[qq]], lc2);
  }
};

// Cell binning and stable key sort of one instance of fewer than kGridMinN circles (its entries fit 32
// bits), then CSR rows over the 3x3 cells.  x: n positions; lists go to rp[0..n], col[0..cap).  cells:
// nc^2 + 1 int32 of scratch; ckey/corder: n each; xs_: room for n positions, which takes the binary32
// coordinates in cell order, so that the three cells of a row of the 3x3 block are one contiguous range.
// All pointers may be shared or global memory.  Rows come in cell-scan order (deterministic).  Returns the
// number of entries (block-uniform); > cap means overflow: the rows are then not written, rp holds no list.
// hash (shared, may be null) receives an order-independent 64-bit digest of the pair set, used to tell
// Gamma' from Gamma.
template <typename T, typename IdxT>
__device__ int cta_build_neighbors(const v2<T> *__restrict__ x, int n, const CellGrid &G, T lc2,
                                   uint32_t *ckey, int32_t *corder, int32_t *cells, v2<T> *xs_, int32_t *rp,
                                   IdxT *col, int cap, int32_t *sh, unsigned long long *hash) {
  const int T_ = blockDim.x, t = threadIdx.x;
  const int nc = G.nc;
  int32_t *cstart = cells;
  float2 *const xs = (float2 *)xs_;
  if (t == 0 && hash) *hash = 0ull;
  cta_cell_sort<T>(x, n, G, ckey, corder, cells, xs, rp, sh);  // rp is free until the count
  if (t == 0) rp[0] = 0;
  __syncthreads();
  SortedNear<T> near(x, corder, xs, lc2);
  // count: circles visited in cell order, candidates as three contiguous row ranges
  for (int q0 = t; q0 < n; q0 += T_) {
    const int i = corder[q0];
    near.set(q0);
    const uint32_t cell = ckey[i];
    const int cx = (int)(cell & 0xffffu), cy = (int)(cell >> 16);
    const int bx0 = max(cx - 1, 0), bx1 = min(cx + 1, nc - 1);
    int cntn = 0;
    for (int by = max(cy - 1, 0); by <= min(cy + 1, nc - 1); ++by) {
      const int lo = cstart[by * nc + bx0], hi = cstart[by * nc + bx1 + 1];
      for (int qq = lo; qq < hi; ++qq) cntn += near(qq) && qq != q0;
    }
    rp[i + 1] = cntn;
  }
  __syncthreads();
  block_scan_inplace(rp + 1, n, sh);
  const int total = rp[n];
  if (total <= cap) {
    unsigned long long h = 0ull;
    for (int q0 = t; q0 < n; q0 += T_) {
      const int i = corder[q0];
      near.set(q0);
      const uint32_t cell = ckey[i];
      const int cx = (int)(cell & 0xffffu), cy = (int)(cell >> 16);
      const int bx0 = max(cx - 1, 0), bx1 = min(cx + 1, nc - 1);
      int w = rp[i];
      for (int by = max(cy - 1, 0); by <= min(cy + 1, nc - 1); ++by) {
        const int lo = cstart[by * nc + bx0], hi = cstart[by * nc + bx1 + 1];
        for (int qq = lo; qq < hi; ++qq) {
          if (near(qq) && qq != q0) {
            const int j = corder[qq];
            col[w++] = (IdxT)j;
            if (hash) h += mix32((uint32_t)i * 0x9E3779B1u ^ (uint32_t)j);
          }
        }
      }
    }
    if (hash) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
      if ((t & 31) == 0) atomicAdd(hash, h);
    }
  }
  __syncthreads();
  return total;
}

// ------------------------------------------------------------- partition ---
// Order-preserving map of a double onto uint64 (for sorting keys of either sign).
__device__ __forceinline__ uint64_t sortable(double v) {
  uint64_t b = (uint64_t)__double_as_longlong(v);
  return (b & 0x8000000000000000ull) ? ~b : (b | 0x8000000000000000ull);
}

// Partition key of Sec. 4.1 with correctly rounded operations: 0 sector (a pseudo-angle,
// strictly increasing in the polar angle on [0, 2 pi)), 1 annulus (radius), 2 fence (x).
__device__ __forceinline__ double part_key(double x, double y, int mode) {
  if (mode == 1) return __dsqrt_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)));
  if (mode == 2) return x;
  double s = __dadd_rn(fabs(x), fabs(y));
  if (s == 0.0) return 0.0;
  double t = __ddiv_rn(x, s);
  return (y >= 0.0) ? __dsub_rn(1.0, t) : __dadd_rn(3.0, t);
}

// Key of the random partition of Sec. 4.1 (mode 3): 53 bits of Philox4x32-10 counter
// (i, 0, q, 3 * 2^30) under the partition seed; the order by (key, index) is a uniform permutation.
__device__ __forceinline__ double random_part_key(uint64_t seed, int i, int q) {
  const uint4 w = philox4x32_10(make_uint4((uint32_t)i, 0u, (uint32_t)q, 0xC0000000u),
                                make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
  return u53(w.x, w.y);
}

// ---------------------------------------------------------- quasi-Newton ---
constexpr int KS = kMaxSlots;      // basis index of Y slot a is KS + a
constexpr int GI = 2 * kMaxSlots;  // basis index of g
// The dots of the first reduction of a batch step come in chunks of 32 values, one chunk per six
// physical slots a: in chunk a / 6, from 4 (a % 6): g's_a, g'y_a, y's_a, y'y_a, where (s, y) is the
// pending pair; chunk 0 also carries g'g, s's, s'y and y'y at 24..27.  The two-loop on the Gram
// matrix reads an s only against the y's of its own or a newer pair, and no s against another s, so
// s's_a and s'y_a are not taken: four values per slot instead of six put the six slots of m = 5 in
// one chunk (one pass over the slots and one reduce-scatter instead of two), the eleven of m = 10
// in two instead of three.
constexpr int kSlotsPerChunk = 6;
constexpr int kChunks = (kMaxSlots + kSlotsPerChunk - 1) / kSlotsPerChunk;
constexpr int kPA = 32 * kChunks;  // per-warp partial values of the first reduction
constexpr int PA_GG = 24, PA_SS = 25, PA_SY = 26, PA_YY = 27;
__device__ __forceinline__ int pa_idx(int a, int kind) {
  return 32 * (a / kSlotsPerChunk) + 4 * (a % kSlotsPerChunk) + kind;
}
// Gram matrix of a batch: s_a'y_b at a KS + b (a not newer than b), then y_a'y_b at KS KS + a KS + b.
constexpr int kGram = 2 * KS * KS;
constexpr int kYY = KS * KS;

// One secant pair of one circle: s and y side by side, one 16-byte access in binary32 (two in
// binary64) where separate arrays took two.
template <typename T> struct alignas(16) SecantPair { v2<T> s, y; };
__device__ __forceinline__ SecantPair<float> ld_pair(const SecantPair<float> *p) {
  const float4 v = *(const float4 *)p;
  return SecantPair<float>{make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ SecantPair<double> ld_pair(const SecantPair<double> *p) { return *p; }
__device__ __forceinline__ void st_pair(SecantPair<float> *p, float2 s, float2 y) {
  *(float4 *)p = make_float4(s.x, s.y, y.x, y.y);
}
__device__ __forceinline__ void st_pair(SecantPair<double> *p, double2 s, double2 y) { p->s = s; p->y = y; }

// The pairs of circle pos in the physical slots [A0, A0 + N), of mm in all.  Every load is issued
// whether its slot is in use or not (its value is then ignored; a slot past the last is read as slot
// 0), so that all of them are in flight together: behind a test of its own each slot waited for its
// own L2 round trip (the 4096-instance batch at m = 5: 210.5 ms, with the groups 191.2).  Six slots
// per group, those of m = 5, and one circle per thread at a time: seven slots, or two circles, take
// registers the kernel does not have (196.0 and 192.6 ms, and a single instance gets slower).
// I: type of the index arithmetic (the number of circles n comes in it).
template <int A0, int N, typename T, typename I>
__device__ __forceinline__ void load_slots(const SecantPair<T> *SY, int mm, I n, int pos, SecantPair<T> *pr) {
#pragma unroll
  for (int j = 0; j < N; ++j) pr[j] = ld_pair(SY + (A0 + j < mm ? A0 + j : 0) * n + pos);
}

// ------------------------------------------------------- pair arithmetic ---
// pair(): for circles a (the row owner) and b, returns the overlap depth d >= 0
// (0 when l >= 2) and the gradient contribution to a: -2 d (a - b) / l.
// A coincident pair contributes d = 2 and no gradient.
struct Arith32 {
  using pos_t = float;
  using vec_t = float;
  using acc_t = float;
  static constexpr int kId = 1;
  // Without branches: every lane of a warp takes the same instructions whether its pair is in
  // contact or not (a list row holds both kinds), and the selects give the values of the case split.
  __device__ static __forceinline__ acc_t pair(float2 a, float2 b, float &fx, float &fy) {
    float dx = a.x - b.x, dy = a.y - b.y;
    float s = dx * dx + dy * dy;
    const bool act = s < 4.f, pos = s > 0.f, ap = act && pos;
    float rl = rsqrtf(pos ? s : 1.f);
    float d = 2.f - s * rl;
    float c = -2.f * d * rl;
    fx = ap ? c * dx : 0.f;
    fy = ap ? c * dy : 0.f;
    return act ? (pos ? fmaxf(d, 0.f) : 2.f) : 0.f;
  }
  // The same values with the arithmetic of pairs beyond contact skipped by a branch: the standalone
  // energy + gradient kernel's rows at converged layouts hold many such pairs, and there the skip
  // saves more than keeping the lanes together (3 % on the batch's final layouts).
  __device__ static __forceinline__ acc_t pair_skip(float2 a, float2 b, float &fx, float &fy) {
    float dx = a.x - b.x, dy = a.y - b.y;
    float s = dx * dx + dy * dy;
    fx = 0.f; fy = 0.f;
    if (!(s < 4.f)) return 0.f;
    if (s > 0.f) {
      float rl = rsqrtf(s);
      float d = 2.f - s * rl;
      float c = -2.f * d * rl;
      fx = c * dx; fy = c * dy;
      return fmaxf(d, 0.f);
    }
    return 2.f;
  }
  // container term: depth d_i0 and gradient 2 d_i0 c_i / |c_i|
  __device__ static __forceinline__ acc_t wall(float2 a, float R, float Rm1sq, float &fx, float &fy) {
    float r2 = a.x * a.x + a.y * a.y;
    float r = sqrtf(r2);
    float d = r + 1.f - R;
    fx = 0.f; fy = 0.f;
    if (!(d > 0.f)) return 0.f;
    if (r > 0.f) { float c = 2.f * d / r; fx = c * a.x; fy = c * a.y; }
    return d;
  }
};

__device__ __forceinline__ double rsqrt_d(double s) {
  // binary32 estimate refined by two Newton steps in binary64 (s >= 1e-30)
  double y = (double)rsqrtf((float)s);
  double h = 0.5 * s;
  y = y * fma(-h * y, y, 1.5);
  y = y * fma(-h * y, y, 1.5);
  return y;
}

struct Arith64 {
  using pos_t = double;
  using vec_t = double;
  using acc_t = double;
  static constexpr int kId = 0;
  __device__ static __forceinline__ acc_t pair(double2 a, double2 b, double &fx, double &fy) {
    double dx = a.x - b.x, dy = a.y - b.y;
    double s = fma(dx, dx, dy * dy);
    fx = 0.0; fy = 0.0;
    if (!(s < 4.0)) return 0.0;
    if (s > 1e-30) {
      double rl = rsqrt_d(s);
      double d = 2.0 - s * rl;
      double c = -2.0 * d * rl;
      fx = c * dx; fy = c * dy;
      return d > 0.0 ? d : 0.0;
    }
    if (s > 0.0) {
      double l = sqrt(s);
      double c = -2.0 * (2.0 - l) / l;
      fx = c * dx; fy = c * dy;
      return 2.0 - l;
    }
    return 2.0;
  }
  // pair() already skips the pairs beyond contact
  __device__ static __forceinline__ acc_t pair_skip(double2 a, double2 b, double &fx, double &fy) {
    return pair(a, b, fx, fy);
  }
  // Rm1sq = (R - 1)^2 when R >= 1, else -1 (every circle then touches the wall)
  __device__ static __forceinline__ acc_t wall(double2 a, double R, double Rm1sq, double &fx, double &fy) {
    double r2 = fma(a.x, a.x, a.y * a.y);
    fx = 0.0; fy = 0.0;
    if (!(r2 > Rm1sq)) return 0.0;  // |c| <= R - 1: no contact
    if (r2 <= 1e-30) { double d = sqrt(r2) + 1.0 - R; return d > 0.0 ? d : 0.0; }
    double rl = rsqrt_d(r2);
    double r = r2 * rl;
    double d = r + 1.0 - R;
    if (!(d > 0.0)) return 0.0;
    double c = 2.0 * d * rl;
    fx = c * a.x; fy = c * a.y;
    return d;
  }
};

struct ArithMix {
  using pos_t = double;
  using vec_t = float;
  using acc_t = double;
  static constexpr int kId = 2;
  // 4 - l^2 = 4 - dy^2 - dx^2 by two fused multiply-adds (one rounding of size ulp64(4) / 2 at
  // most, then the exact cancellation near contact and one rounding of the small result); its
  // sign is the contact test, and everything after it is binary32.
  __device__ static __forceinline__ float pair(double2 a, double2 b, float &fx, float &fy) {
    const double dx = a.x - b.x, dy = a.y - b.y;
    const float e = (float)fma(-dx, dx, fma(-dy, dy, 4.0));
    fx = 0.f; fy = 0.f;
    if (!(e > 0.f)) return 0.f;
    const float dxf = (float)dx, dyf = (float)dy;
    const float s = fmaf(dxf, dxf, dyf * dyf);
    if (s > 1e-30f) {
      const float rl = rsqrtf(s);
      const float l = s * rl;
      const float d = e / (2.f + l);    // 2 - l = (4 - l^2) / (2 + l)
      const float c = -2.f * d * rl;
      fx = c * dxf; fy = c * dyf;
      return d;
    }
    return 2.f;
  }
  // pair() already skips the pairs beyond contact
  __device__ static __forceinline__ float pair_skip(double2 a, double2 b, float &fx, float &fy) {
    return pair(a, b, fx, fy);
  }
  __device__ static __forceinline__ acc_t wall(double2 a, double R, double Rm1sq, float &fx, float &fy) {
    double r2 = fma(a.x, a.x, a.y * a.y);
    fx = 0.f; fy = 0.f;
    if (!(r2 > Rm1sq)) return 0.0;
    if (Rm1sq < 0.0 || r2 <= 1e-30) {   // degenerate container R < 1, or a centred circle
      double r = sqrt(r2), d = r + 1.0 - R;
      if (r > 0.0) { float c = (float)(2.0 * d / r); fx = c * (float)a.x; fy = c * (float)a.y; }
      return d > 0.0 ? d : 0.0;
    }
    float e = (float)(r2 - Rm1sq);      // |c|^2 - (R-1)^2, exact near contact
    float r = sqrtf((float)r2);
    float d = e / (r + (float)(R - 1.0));  // |c| - (R - 1)
    float c = 2.f * d / r;
    fx = c * (float)a.x; fy = c * (float)a.y;
    return (double)d;
  }
};

// Exact container depth with correctly rounded operations (feasibility check).
__device__ __forceinline__ double wall_depth_exact(double2 a, double R) {
  double r = __dsqrt_rn(__dadd_rn(__dmul_rn(a.x, a.x), __dmul_rn(a.y, a.y)));
  double d = __dsub_rn(__dadd_rn(r, 1.0), R);
  return d > 0.0 ? d : 0.0;
}
__device__ __forceinline__ double pair_depth_exact(double2 a, double2 b) {
  double dx = __dsub_rn(a.x, b.x), dy = __dsub_rn(a.y, b.y);
  double s = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
  return __dsub_rn(2.0, __dsqrt_rn(s));
}

__device__ __forceinline__ long long globaltimer_ns() {
  long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

}  // namespace pecc
