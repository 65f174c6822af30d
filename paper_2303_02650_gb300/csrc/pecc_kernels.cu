// pecc_kernels.cu -- standalone kernels: random init (Sec. 5.1), neighbor build
// (Sec. 4.3), fused energy + gradient (Eq. 3, Eq. 5), feasibility (Eq. 1, Eq. 2).
#include "pecc_cells.cuh"
#include "pecc_internal.h"

namespace pecc {

namespace {

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// Asynchronous copy of BYTES (8 or 16) from global to shared memory (cp.async; completed by
// cp.async.wait_all).  Both addresses must be BYTES-aligned.
template <int BYTES> __device__ __forceinline__ void cp_async_shared(void *dst, const void *src) {
  static_assert(BYTES == 8 || BYTES == 16, "cp.async copies 4, 8 or 16 bytes");
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}

// threads per block of the block-per-instance energy + gradient kernel (measured on the
// 4096-instance batch's final layouts: 128 threads 41.2 us, 256 threads 43.3 us, 512 threads 49.5 us)
constexpr int kEgBlock = 128;

// ------------------------------------------------------------------ init ----
// Circle i of instance q: Philox4x32-10, key (seed lo, seed hi), counter (i, attempt, q, 0);
// (w0, w1) and (w2, w3) give two 53-bit uniforms u, v; candidate (R-1)(2u-1, 2v-1),
// accepted inside the disk of radius R-1 (mode 0), or R (2u-1, 2v-1) in the square (mode 1).
__global__ void init_kernel(StandaloneParams P, uint64_t seed, int mode, int prec) {
  int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= P.total) return;
  const int q = P.inst_of[gi];
  const InstDesc D = P.desc[q];
  const uint32_t i = (uint32_t)(gi - D.off);
  const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
  const double R = D.R, rr = __dsub_rn(R, 1.0);
  double x = 0.0, y = 0.0;
  if (mode == 1) {
    uint4 w = philox4x32_10(make_uint4(i, 0u, (uint32_t)q, 0u), key);
    x = __dmul_rn(R, __dsub_rn(__dmul_rn(2.0, u53(w.x, w.y)), 1.0));
    y = __dmul_rn(R, __dsub_rn(__dmul_rn(2.0, u53(w.z, w.w)), 1.0));
  } else if (rr > 0.0) {
    for (uint32_t a = 0; a < 64u; ++a) {
      uint4 w = philox4x32_10(make_uint4(i, a, (uint32_t)q, 0u), key);
      double cx = __dmul_rn(rr, __dsub_rn(__dmul_rn(2.0, u53(w.x, w.y)), 1.0));
      double cy = __dmul_rn(rr, __dsub_rn(__dmul_rn(2.0, u53(w.z, w.w)), 1.0));
      if (__dadd_rn(__dmul_rn(cx, cx), __dmul_rn(cy, cy)) <= __dmul_rn(rr, rr)) { x = cx; y = cy; break; }
    }
  }
  if (prec == 0) {
    P.x64[gi] = make_double2(x, y);
  } else {
    float2 f = make_float2((float)x, (float)y);
    P.x32[gi] = f;
    P.x64[gi] = make_double2((double)f.x, (double)f.y);
  }
}

__global__ void set_pos_kernel(StandaloneParams P, const double *__restrict__ xy, int prec) {
  int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= P.total) return;
  double x = xy[2 * gi], y = xy[2 * gi + 1];
  if (prec == 0) {
    P.x64[gi] = make_double2(x, y);
  } else {
    float2 f = make_float2((float)x, (float)y);
    P.x32[gi] = f;
    P.x64[gi] = make_double2((double)f.x, (double)f.y);
  }
}

__global__ void get_pos_kernel(StandaloneParams P, double *__restrict__ xy, int from32) {
  int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= P.total) return;
  double2 v;
  if (from32) { float2 f = P.x32[gi]; v = make_double2((double)f.x, (double)f.y); }
  else v = P.x64[gi];
  xy[2 * gi] = v.x;
  xy[2 * gi + 1] = v.y;
}

__global__ void set_radius_kernel(InstDesc *desc, const double *__restrict__ R, int num, double l_cut) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= num) return;
  InstDesc &D = desc[q];
  const double r = R[q];
  double inv;
  int nc;
  float invf;
  int ncf;
  if (r > 0.0 && isfinite(r)) {
    host_cell_grid(r, l_cut, D.n, &inv, &nc);
    f32_cell_grid(r, l_cut, D.n, nc, &invf, &ncf);
    D.R = r;
  } else {  // the instance's energies, descents and checks come out NaN (status PECC_DESC_NONFINITE)
    host_cell_grid(1.0, l_cut, D.n, &inv, &nc);
    f32_cell_grid(1.0, l_cut, D.n, nc, &invf, &ncf);
    nc = ncf = 1;
    D.R = __longlong_as_double(0x7ff8000000000000ll);
  }
  D.inv_cs = inv;
  D.ncx = nc;
  D.inv_f = invf;
  D.ncx_f = ncf;
}

// ----------------------------------------------------------------- build ----
// Lists of Sec. 4.3 as CSR rows ascending in j, from the cells (pecc_cells.cuh).  A warp takes 32
// consecutive circles, a lane a row: the lane collects its hits (kRowHits 16- or 32-bit indices at
// most, a column of the warp's buffer), ranks them among themselves, and the warp writes its 32 rows as
// one contiguous piece.  A row with more hits sends its warp to the general path below (second walk,
// entries straight to global memory, insertion sort).
constexpr int kRowHits = 16;

// Hits of circle i (cell key; near.set() done) over the 3x3 cells, in scan order: f(q) for each.
template <typename T, typename I, typename F>
__device__ __forceinline__ void for_neighbors(const Coords<T> &X, int i, int key, int nc,
                                              const int32_t *start, const float2 *xs, const I *ord,
                                              const Near<T> &near, F f) {
  const int cy = key / nc, cx = key - cy * nc;
  const int bx0 = max(cx - 1, 0), bx1 = min(cx + 1, nc - 1);
  for (int by = max(cy - 1, 0); by <= min(cy + 1, nc - 1); ++by) {
    const int lo = start[by * nc + bx0], hi = start[by * nc + bx1 + 1];
    for (int q = lo; q < hi; ++q)
      if (near(i, xs[q], X, ord, q) && (int)ord[q] != i) f(q);
  }
}

// The 32 rows of a warp, once every lane knows where its row starts: buf holds the lane's hits at
// buf[32 h + lane] (cnt of them when cnt <= kRowHits), row0 is the lane's row start.  Called only where the
// block's rows end within the list's capacity: rows of an overflowed list are not written (nor sorted: in
// a crowd they can hold every circle).
template <typename T, typename I>
__device__ __forceinline__ void write_rows(const Coords<T> &X, bool act, int i, int key, int nc, const int32_t *start,
                                           const float2 *xs, const I *ord, I *buf, int cnt, int row0, int32_t *col) {
  const int lane = threadIdx.x & 31;
  if (__any_sync(0xffffffffu, cnt > kRowHits)) {
    if (act) {
      Near<T> near(X.l_cut);
      near.set(X.low(i));
      int w = row0;
      for_neighbors<T, I>(X, i, key, nc, start, xs, ord, near, [&](int q) {
        const int v = (int)ord[q];
        int t = w++ - 1;
        while (t >= row0 && col[t] > v) { col[t + 1] = col[t]; --t; }  // insert in ascending order
        col[t + 1] = v;
      });
    }
    return;
  }
  // ranks among the lane's own hits, all of them in registers
  int h[kRowHits], rank[kRowHits];
#pragma unroll
  for (int u = 0; u < kRowHits; ++u) {
    h[u] = u < cnt ? (int)buf[32 * u + lane] : 0x7fffffff;
    rank[u] = 0;
  }
#pragma unroll
  for (int u = 0; u < kRowHits / 2; ++u)
#pragma unroll
    for (int v = u + 1; v < kRowHits / 2; ++v) {
      const bool less = h[v] < h[u];
      rank[u] += less;
      rank[v] += !less;
    }
  if (__any_sync(0xffffffffu, cnt > kRowHits / 2)) {
#pragma unroll
    for (int v = kRowHits / 2; v < kRowHits; ++v)
#pragma unroll
      for (int u = 0; u < v; ++u) {
        const bool less = h[v] < h[u];
        rank[u] += less;
        rank[v] += !less;
      }
  }
  const int base = __shfl_sync(0xffffffffu, row0, 0);
  const int total = __shfl_sync(0xffffffffu, row0 + cnt, 31) - base;  // lanes past the last row have none
  __syncwarp();
#pragma unroll
  for (int u = 0; u < kRowHits; ++u)
    if (u < cnt) buf[row0 - base + rank[u]] = (I)h[u];
  __syncwarp();
  for (int t = lane; t < total; t += 32) col[base + t] = (int)buf[t];
  __syncwarp();  // the next rows' hits go into the same buffer
}

// Exclusive prefix sum of one value per thread over the block; total: the block's sum.  sh: 33 ints.
// SAT: the sums stop at kMaxEntries (entry counts of instances of any size).
template <bool SAT = false>
__device__ __forceinline__ int block_exclusive(int v, int32_t *sh, int &total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  auto add = [](int a, int b) { return SAT ? sat_add(a, b) : a + b; };
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl = add(incl, u);
  }
  __syncthreads();  // the previous call's reads of sh
  if (lane == 31) sh[w] = incl;
  __syncthreads();
  int before = 0;
  total = 0;
  for (int u = 0; u < nw; ++u) {
    const int t = sh[u];
    before = add(before, u < w ? t : 0);
    total = add(total, t);
  }
  if constexpr (SAT) {  // a saturated sum cannot be taken back
    const int prev = __shfl_up_sync(0xffffffffu, incl, 1);
    return lane ? sat_add(before, prev) : before;
  }
  return before + incl - v;
}

template <typename T> __device__ __forceinline__ Coords<T> coords_of(const StandaloneParams &P, int64_t off, int from32);
template <> __device__ __forceinline__ Coords<float> coords_of<float>(const StandaloneParams &P, int64_t off, int) {
  return Coords<float>{P.x32 + off, P.l_cut};
}
template <> __device__ __forceinline__ Coords<double> coords_of<double>(const StandaloneParams &P, int64_t off,
                                                                        int from32) {
  return Coords<double>{P.x64 + off, from32 ? P.x32 + off : nullptr, P.l_cut};
}

// Instances of at most kCellsBlockN circles, one block each, everything on chip: the coordinates come
// in once, the rows, cells and order go out once.  What bounds it is instruction issue (81 % of the slots)
// and shared-memory wavefronts (61 %) of the candidate walks.  The 4096-instance batch's new positions,
// lists, energy and gradient take 209 us with it, 152 us of them here; 966 us with lists built and sorted
// in global memory (901 us).
constexpr int kBuildWarpBytes = 32 * kRowHits * (int)sizeof(uint16_t);
template <typename T>
__global__ void __launch_bounds__(512, 3) build_block_kernel(StandaloneParams P, int force, int32_t *rebuilt) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int32_t sh[40];
  using PP = v2<T>;
  const int q = P.eorder[blockIdx.x];
  const InstDesc &D = P.desc[q];
  const int n = D.n;
  if (n > kCellsBlockN) return;
  const int64_t off = D.off;
  const Coords<T> X = coords_of<T>(P, off, 0);
  PP *xb = (PP *)P.xbuild + off;
  int go = force;
  if (!go) {
    // largest displacement since the last standalone build
    double m = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const PP a = X.at(i), b = xb[i];
      const double dx = (double)a.x - (double)b.x, dy = (double)a.y - (double)b.y;
      m = fmax(m, dx * dx + dy * dy);
    }
    go = __syncthreads_or(m > P.rebuild_disp * P.rebuild_disp);
  }
  if (threadIdx.x == 0 && rebuilt) rebuilt[q] = go;
  if (!go) return;
  const int nc = D.ncx, cap = D.cap;
  const size_t extra = (size_t)(blockDim.x >> 5) * kBuildWarpBytes;
  const BlockCells C = block_cells<T>(X, n, D.R, D.inv_cs, nc, sm, extra, P.cells + D.cell_off, P.ckey + off,
                                      P.corder + off, sh, [&](PP p, float2, int i) { xb[i] = p; });
  int32_t *rp = P.rp + off + q, *col = P.col + D.col_s_off;
  uint16_t *buf = (uint16_t *)(C.extra + (threadIdx.x >> 5) * kBuildWarpBytes);
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) rp[0] = 0;
  int run = 0;
  Near<T> near(P.l_cut);
  for (int i0 = 0; i0 < n; i0 += blockDim.x) {
    const int i = i0 + threadIdx.x;
    const bool act = i < n;
    int cnt = 0, key = 0;
    if (act) {
      key = C.key[i];
      near.set(C.xi[i]);
      for_neighbors<T, uint16_t>(X, i, key, nc, C.start, C.xs, C.ord, near, [&](int qq) {
        if (cnt < kRowHits) buf[32 * cnt + lane] = C.ord[qq];
        ++cnt;
      });
    }
    int total;
    const int row0 = run + block_exclusive(cnt, sh, total);
    if (act) rp[i + 1] = row0 + cnt;
    run += total;
    if (run <= cap) write_rows<T, uint16_t>(X, act, i, key, nc, C.start, C.xs, C.ord, buf, cnt, row0, col);
  }
}

// ---- larger instances: one kernel per step over tiles of all of them (pecc_cells.cuh); each step reads
// what the one before it wrote.  One block per instance left the GPU idle: new positions, lists, energy
// and gradient of 100000 circles took 3842 us, now 80 us, most of it the launches' own latency.  The line
// to the block form is where its shared memory and one block's time end; from 1000 circles on a block
// takes longer than the eight launches, but a batch of such instances fills the GPU with blocks.
struct LargeDest { uint32_t *ckey; int32_t *corder; float2 *xs; };  // per circle (offset by the instance)

template <typename T>
__global__ void __launch_bounds__(kTileRows) large_go_kernel(StandaloneParams P, LargeTiles L, int force) {
  const int2 t = L.rows[blockIdx.x];
  const InstDesc &D = P.desc[t.x];
  const int i = t.y * kTileRows + threadIdx.x, n = D.n;
  // the instance's cell counters, four per thread of its row tiles, the last tile to the end
  int32_t *cells = P.cells + D.cell_off;
  const int ncell = D.ncx * D.ncx, last = (n - 1) / kTileRows;
  const int c1 = t.y == last ? ncell + 1 : min(ncell + 1, (t.y + 1) * 4 * kTileRows);
  for (int c = t.y * 4 * kTileRows + threadIdx.x; c < c1; c += kTileRows) cells[c] = 0;
  if (force) {
    if (threadIdx.x == 0 && t.y == 0) L.go[t.x] = 1;
  } else {
    using PP = v2<T>;
    double m = 0.0;
    if (i < n) {
      const PP a = coords_of<T>(P, D.off, 0).at(i), b = ((const PP *)P.xbuild + D.off)[i];
      const double dx = (double)a.x - (double)b.x, dy = (double)a.y - (double)b.y;
      m = dx * dx + dy * dy;
    }
    const int go = __syncthreads_or(m > P.rebuild_disp * P.rebuild_disp);
    if (threadIdx.x == 0 && go) atomicOr(&L.go[t.x], 1);  // cleared before this launch
  }
}

// cells of every circle and its arrival rank in its cell; for the list build also the reference
// coordinates, for the feasibility check the largest radius and the finiteness
template <typename T, bool CHECK>
__global__ void __launch_bounds__(kTileRows) large_key_kernel(StandaloneParams P, LargeTiles L, LargeDest O, int from32,
                                                              v2<T> *xbuild) {
  const int2 t = L.rows[blockIdx.x];
  if (!CHECK && !L.go[t.x]) return;
  const InstDesc &D = P.desc[t.x];
  const int i = t.y * kTileRows + threadIdx.x;
  float r2 = 0.f;
  int bad = 0;
  if (i < D.n) {
    const typename Coords<T>::point p = coords_of<T>(P, D.off, from32).at(i);
    const float2 f = make_float2((float)p.x, (float)p.y);
    const int key = cell_key_fast(p, f, D.R, D.inv_cs, D.ncx);
    O.ckey[D.off + i] = (uint32_t)key;
    L.rank[D.off + i] = atomicAdd(P.cells + D.cell_off + key + 1, 1);
    if (xbuild) xbuild[D.off + i] = p;
    if (CHECK) {
      r2 = f.x * f.x + f.y * f.y;
      bad = not_finite(p.x) || not_finite(p.y);
    }
  }
  if (CHECK) {
    bad = __syncthreads_or(bad);
    r2 = warp_max(r2);
    if ((threadIdx.x & 31) == 0 && r2 > 0.f) atomicMax(&L.rmax32[t.x], __float_as_uint(r2));
    if (threadIdx.x == 0 && bad) atomicOr(&L.bad[t.x], 1);
  }
}

// inclusive sums of the cell counts within a tile of cells, and the tile's total
__global__ void __launch_bounds__(256) large_cells_kernel(StandaloneParams P, LargeTiles L) {
  __shared__ int32_t sh[40];
  const int2 t = L.cells[blockIdx.x];
  if (!L.go[t.x]) return;
  const InstDesc &D = P.desc[t.x];
  const int ncell = D.ncx * D.ncx, c0 = t.y * kTileCells;
  int32_t *a = P.cells + D.cell_off + 1 + c0;
  const int m = min(kTileCells, ncell - c0);
  int v[4], s = 0;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int c = 4 * threadIdx.x + u;
    v[u] = c < m ? a[c] : 0;
    s += v[u];
  }
  int total, run = block_exclusive(s, sh, total);
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int c = 4 * threadIdx.x + u;
    run += v[u];
    if (c < m) a[c] = run;
  }
  if (threadIdx.x == 0) L.cell_total[blockIdx.x] = m > 0 ? total : 0;
}

// Sum of the totals of the earlier tiles of tile b's instance (its tile t.y of the instance), saturated.
__device__ __forceinline__ int tiles_before(const int32_t *total, int b, int ty, int32_t *sh) {
  int s = 0;
  for (int u = threadIdx.x; u < ty; u += blockDim.x) s = sat_add(s, total[b - ty + u]);
  int all;
  block_exclusive<true>(s, sh, all);
  return all;
}

__global__ void __launch_bounds__(256) large_cells_base_kernel(StandaloneParams P, LargeTiles L) {
  __shared__ int32_t sh[40];
  const int2 t = L.cells[blockIdx.x];
  if (!L.go[t.x]) return;
  const InstDesc &D = P.desc[t.x];
  const int ncell = D.ncx * D.ncx, c0 = t.y * kTileCells;
  if (c0 >= ncell) return;
  const int base = tiles_before(L.cell_total, blockIdx.x, t.y, sh);
  int32_t *a = P.cells + D.cell_off + 1 + c0;
  for (int c = threadIdx.x; c < min(kTileCells, ncell - c0); c += blockDim.x) a[c] += base;
}

__global__ void __launch_bounds__(kTileRows) large_scatter_kernel(StandaloneParams P, LargeTiles L, LargeDest O) {
  const int2 t = L.rows[blockIdx.x];
  if (!L.go[t.x]) return;
  const InstDesc &D = P.desc[t.x];
  const int i = t.y * kTileRows + threadIdx.x;
  if (i < D.n) L.tmp[D.off + P.cells[D.cell_off + O.ckey[D.off + i]] + L.rank[D.off + i]] = i;
}

template <typename T>
__global__ void __launch_bounds__(kTileRows) large_order_kernel(StandaloneParams P, LargeTiles L, LargeDest O,
                                                                int from32) {
  const int2 t = L.rows[blockIdx.x];
  if (!L.go[t.x]) return;
  const InstDesc &D = P.desc[t.x];
  const int p = t.y * kTileRows + threadIdx.x;
  if (p >= D.n) return;
  const int32_t *tmp = L.tmp + D.off, *start = P.cells + D.cell_off;
  const int i = tmp[p], c = (int)O.ckey[D.off + i];
  int r = start[c];
  for (int q = start[c], hi = start[c + 1]; q < hi; ++q) r += tmp[q] < i;
  O.corder[D.off + r] = i;
  O.xs[D.off + r] = coords_of<T>(P, D.off, from32).low(i);
}

// FILL = false: the entries of every tile of rows; true: the rows.  Counts and row starts saturate: 50000
// circles in one place have 2.5e9 entries, and a start that wrapped to a negative one would pass every
// test against the capacity.
template <typename T, bool FILL>
__global__ void __launch_bounds__(kTileRows) large_rows_kernel(StandaloneParams P, LargeTiles L, LargeDest O,
                                                               int32_t *rebuilt) {
  __shared__ int32_t sh[40];
  __shared__ int32_t bufs[FILL ? kTileRows * kRowHits : 1];
  const int2 t = L.rows[blockIdx.x];
  const int go = L.go[t.x];
  if (FILL && rebuilt && t.y == 0 && threadIdx.x == 0) rebuilt[t.x] = go;
  if (!go) return;
  const InstDesc &D = P.desc[t.x];
  const int n = D.n, i = t.y * kTileRows + threadIdx.x, lane = threadIdx.x & 31, nc = D.ncx;
  const Coords<T> X = coords_of<T>(P, D.off, 0);
  const int32_t *start = P.cells + D.cell_off, *ord = O.corder + D.off;
  const float2 *xs = O.xs + D.off;
  int32_t *buf = bufs + (FILL ? (threadIdx.x >> 5) * 32 * kRowHits : 0);
  const bool act = i < n;
  int cnt = 0, key = 0;
  if (act) {
    key = (int)O.ckey[D.off + i];
    Near<T> near(P.l_cut);
    near.set(X.low(i));
    for_neighbors<T, int32_t>(X, i, key, nc, start, xs, ord, near, [&](int q) {
      if (FILL && cnt < kRowHits) buf[32 * cnt + lane] = ord[q];
      ++cnt;
    });
  }
  if (!FILL) {
    int total;
    block_exclusive<true>(cnt, sh, total);
    if (threadIdx.x == 0) L.row_total[blockIdx.x] = total;
    return;
  }
  const int base = tiles_before(L.row_total, blockIdx.x, t.y, sh);
  int total;
  const int row0 = sat_add(base, block_exclusive<true>(cnt, sh, total));
  int32_t *rp = P.rp + D.off + t.x;
  if (act) rp[i + 1] = sat_add(row0, cnt);
  if (i == 0) rp[0] = 0;
  if (sat_add(base, total) <= D.cap)
    write_rows<T, int32_t>(X, act, i, key, nc, start, xs, ord, buf, cnt, row0, P.col + D.col_s_off);
}

// Cells, order and sorted coordinates of every large instance (flags in L.go, or all of them).
template <typename T, bool CHECK>
cudaError_t large_cells(const StandaloneParams &p, const LargeTiles &L, const LargeDest &O, int from32, int force,
                        v2<T> *xbuild, cudaStream_t s) {
  if (!force)
    if (cudaError_t e = cudaMemsetAsync(L.go, 0, sizeof(int32_t) * (size_t)p.num, s)) return e;
  large_go_kernel<T><<<L.nrows, kTileRows, 0, s>>>(p, L, force);
  large_key_kernel<T, CHECK><<<L.nrows, kTileRows, 0, s>>>(p, L, O, from32, xbuild);
  large_cells_kernel<<<L.ncells, 256, 0, s>>>(p, L);
  large_cells_base_kernel<<<L.ncells, 256, 0, s>>>(p, L);
  large_scatter_kernel<<<L.nrows, kTileRows, 0, s>>>(p, L, O);
  large_order_kernel<T><<<L.nrows, kTileRows, 0, s>>>(p, L, O, from32);
  return cudaGetLastError();
}

// ------------------------------------------------- fused energy + gradient ----
// A radius that pecc_set_radius did not accept is NaN (binary64: told by its bits, as the arithmetic units of
// that width are few: a comparison took 2 % of the 4096-instance batch's energies).
__device__ __forceinline__ bool rejected(float R) { return R != R; }
__device__ __forceinline__ bool rejected(double R) { return not_finite(R); }

// One thread per circle (gather over its row, no atomics):
//   g_i = sum_{j in Gamma(i)} -2 d_ij (c_i - c_j) / l_ij + 2 d_i0 c_i / |c_i|
//   e_i = sum_{j in Gamma(i), j < i} d_ij^2 + d_i0^2      (so that E = sum_i e_i, Eq. 5)
template <class A>
__global__ void __launch_bounds__(256) energy_grad_kernel(StandaloneParams P, int stage_n, void *__restrict__ grad_,
                                                          void *__restrict__ ecirc_) {
  using pos_t = typename A::pos_t;
  using vec_t = typename A::vec_t;
  using acc_t = typename A::acc_t;
  using PP = v2<pos_t>;
  using VV = v2<vec_t>;
  int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= P.total) return;
  const int q = __ldg(P.inst_of + gi);
  if (P.desc[q].n <= stage_n) return;  // the block kernel's instance
  const int64_t off = P.desc[q].off;
  const int64_t col_off = P.desc[q].col_s_off;
  const double Rd = P.desc[q].R;
  const acc_t R = (acc_t)Rd;
  const acc_t Rm1sq = (acc_t)((Rd >= 1.0) ? (Rd - 1.0) * (Rd - 1.0) : -1.0);
  const PP *x = (sizeof(pos_t) == 4) ? (const PP *)(P.x32 + off) : (const PP *)(P.x64 + off);
  const int i = (int)(gi - off);
  const int32_t *rp = P.rp + off + q;
  const int32_t *cl = P.col + col_off;
  PP xi = x[i];
  vec_t gx = 0, gy = 0;
  acc_t e = 0;
  const int lo = __ldg(rp + i), hi = __ldg(rp + i + 1);
  if (__ldg(rp + P.desc[q].n) > P.desc[q].cap) {  // the last build overflowed the list's capacity: no valid list
    VV gv; gv.x = gv.y = (vec_t)NAN;
    ((VV *)grad_)[gi] = gv;
    ((acc_t *)ecirc_)[gi] = (acc_t)NAN;
    return;
  }
  // two entries per step (their index and coordinate loads in flight together); the sums take the
  // entries in row order
  for (int t = lo; t < hi; t += 2) {
    const bool two = t + 1 < hi;
    const int j1 = __ldg(cl + t);
    const int j2 = two ? __ldg(cl + t + 1) : j1;
    const PP x1 = x[j1], x2 = x[j2];
    vec_t fx, fy;
    const acc_t d1 = A::pair(xi, x1, fx, fy);
    gx += fx; gy += fy;
    if (j1 < i) e += d1 * d1;
    if (two) {
      const acc_t d2 = A::pair(xi, x2, fx, fy);
      gx += fx; gy += fy;
      if (j2 < i) e += d2 * d2;
    }
  }
  vec_t fx, fy;
  acc_t d0 = A::wall(xi, R, Rm1sq, fx, fy);
  gx += fx; gy += fy;
  e += d0 * d0;
  if (rejected(R)) {  // tested here, where the radius has come in
    gx = gy = (vec_t)NAN;
    e = (acc_t)NAN;
  }
  VV gv; gv.x = gx; gv.y = gy;
  ((VV *)grad_)[gi] = gv;
  ((acc_t *)ecirc_)[gi] = e;
}

// One block per instance whose coordinates fit the staging limit (stage_n circles at most): the
// coordinates are staged in shared memory by one coalesced read, so every neighbor gather is an
// on-chip load; row pointers and lists stream through once, the gradient is written once, and the
// energy is reduced in the block in a fixed order (deterministic) and written once.  Larger
// instances are left to energy_grad_kernel + energy_reduce_kernel.  Blocks take the instances
// largest first (the last blocks to start are the shortest), kEgBlock threads each: sixteen
// blocks share an SM.
template <class A>
__global__ void __launch_bounds__(kEgBlock) energy_grad_block_kernel(StandaloneParams P, int stage_n,
                                                                void *__restrict__ grad_, double *E) {
  using pos_t = typename A::pos_t;
  using vec_t = typename A::vec_t;
  using acc_t = typename A::acc_t;
  using PP = v2<pos_t>;
  using VV = v2<vec_t>;
  extern __shared__ __align__(16) unsigned char stage[];
  __shared__ acc_t red[32];
  const int q = P.eorder[blockIdx.x];
  const int n = P.desc[q].n;
  if (n > stage_n) return;  // the per-circle kernels' instance (uniform across the block)
  if (n == 0) {
    if (threadIdx.x == 0) E[q] = 0.0;
    return;
  }
  const int64_t off = P.desc[q].off;
  const int64_t col_off = P.desc[q].col_s_off;
  const double Rd = P.desc[q].R;
  const acc_t R = (acc_t)Rd;
  const acc_t Rm1sq = (acc_t)((Rd >= 1.0) ? (Rd - 1.0) * (Rd - 1.0) : -1.0);
  const PP *x = (sizeof(pos_t) == 4) ? (const PP *)(P.x32 + off) : (const PP *)(P.x64 + off);
  const int32_t *rp = P.rp + off + q;
  const int32_t *cl = P.col + col_off;
  VV *grad = (VV *)grad_ + off;
  const int end = __ldg(rp + n);  // in flight with the coordinates
  PP *xs = (PP *)stage;
  // the staging copies are asynchronous (cp.async, 8 or 16 bytes each): all of a thread's copies
  // are in flight together instead of one load round trip per coordinate
  for (int i = threadIdx.x; i < n; i += blockDim.x) cp_async_shared<sizeof(PP)>(xs + i, x + i);
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  // the last build overflowed the list's capacity (no valid list), or the radius was rejected
  if (end > P.desc[q].cap || rejected(R)) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) { VV gv; gv.x = gv.y = (vec_t)NAN; grad[i] = gv; }
    if (threadIdx.x == 0) E[q] = NAN;
    return;
  }
  __syncthreads();
  acc_t e = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const PP xi = xs[i];
    vec_t gx = 0, gy = 0;
    const int lo = __ldg(rp + i), hi = __ldg(rp + i + 1);
    // two entries per step (both loads in flight); the sums take the entries in row order
    for (int t = lo; t < hi; t += 2) {
      const bool two = t + 1 < hi;
      const int j1 = __ldg(cl + t);
      const int j2 = two ? __ldg(cl + t + 1) : j1;
      const PP x1 = xs[j1], x2 = xs[j2];
      vec_t fx, fy;
      const acc_t d1 = A::pair_skip(xi, x1, fx, fy);
      gx += fx; gy += fy;
      if (j1 < i) e += d1 * d1;
      if (two) {
        const acc_t d2 = A::pair_skip(xi, x2, fx, fy);
        gx += fx; gy += fy;
        if (j2 < i) e += d2 * d2;
      }
    }
    vec_t fx, fy;
    acc_t d0 = A::wall(xi, R, Rm1sq, fx, fy);
    gx += fx; gy += fy;
    e += d0 * d0;
    VV gv; gv.x = gx; gv.y = gy;
    grad[i] = gv;
  }
  e = warp_sum(e);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x < 32) {
    acc_t v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : acc_t(0);
    v = warp_sum(v);
    if (threadIdx.x == 0) E[q] = (double)v;
  }
}

// Per-instance sum of the per-circle energies (fixed order: deterministic), for the instances the
// block kernel left (more than stage_n circles).  Each thread keeps kRed partial sums over
// interleaved circles, so that kRed loads are in flight at a time, and adds them in a fixed order.
constexpr int kRed = 8;
template <typename acc_t>
__global__ void __launch_bounds__(1024) energy_reduce_kernel(StandaloneParams P, int stage_n,
                                                             const acc_t *__restrict__ ecirc, double *E) {
  __shared__ acc_t sh[32];
  const int q = blockIdx.x;
  const InstDesc D = P.desc[q];
  if (D.n <= stage_n) return;
  const acc_t *e = ecirc + D.off;
  const int B = blockDim.x;
  acc_t part[kRed];
#pragma unroll
  for (int u = 0; u < kRed; ++u) part[u] = 0;
  for (int i0 = threadIdx.x; i0 < D.n; i0 += kRed * B) {
#pragma unroll
    for (int u = 0; u < kRed; ++u) {
      const int i = i0 + u * B;
      if (i < D.n) part[u] += e[i];
    }
  }
  acc_t s = part[0];
#pragma unroll
  for (int u = 1; u < kRed; ++u) s += part[u];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    acc_t v = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : acc_t(0);
    v = warp_sum(v);
    if (threadIdx.x == 0) E[q] = (double)v;
  }
}

// ----------------------------------------------------------- feasibility ----
// The largest overlap depth over all pairs (Eq. 1) and walls (Eq. 2), with correctly rounded binary64
// operations: a pair's depth fl(2 - fl(sqrt(s))) never rises with its squared distance s, a wall's never
// falls with the squared radius, so the two extremes decide and only they take the square root.  The
// search runs in binary32; the binary64 values are formed for the pairs and circles whose binary32 ones
// lie within the slack of the extreme.  The entries a list with cutoff l_cut > 2 would hold (it holds
// every overlapping pair) are counted: past twice the capacity the instance is not checkable.
// The 4096-instance batch: 149 us (446 us on its finished layouts, where every contact is near the extreme),
// against 2212 us (2084) for a binary64 list build and a walk over it, which the two binary64 lanes of an
// SM bound.  40 registers let six 256-thread blocks share an SM (170 us with 64 registers and four).
__device__ __forceinline__ double dist2_exact(double2 a, double2 b) {
  const double dx = __dsub_rn(a.x, b.x), dy = __dsub_rn(a.y, b.y);
  return __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
}
__device__ __forceinline__ double norm2_exact(double2 a) { return __dadd_rn(__dmul_rn(a.x, a.x), __dmul_rn(a.y, a.y)); }

// v = the larger of 0 and the two depths; s2 / r2: smallest squared distance (below 4, or infinity) and
// largest squared radius
__device__ __forceinline__ void feasible_result(const StandaloneParams &P, int q, double R, bool bad, double s2,
                                                double r2, double tol, uint8_t *feasible, double *max_overlap) {
  double v = 0.0;
  if (s2 < 4.0) v = fmax(v, __dsub_rn(2.0, __dsqrt_rn(s2)));
  const double d = __dsub_rn(__dadd_rn(__dsqrt_rn(r2), 1.0), R);
  v = fmax(v, d > 0.0 ? d : 0.0);
  bad |= !(R > 0.0);  // a rejected radius (NaN here) contains nothing, however the circles lie
  if (P.desc[q].n == 0) { v = 0.0; bad = false; }
  if (bad) v = __longlong_as_double(0x7ff8000000000000ll);  // NaN: not checkable
  const bool ok = !bad && v <= tol;
  if (feasible) feasible[q] = ok ? 1 : 0;
  if (max_overlap) max_overlap[q] = v;
  P.out[q].max_overlap = v;
}

// Bounds for the exact pass from the extremes of the binary32 search: pairs up to *s_hi, circles from
// *r_lo on.  m: the slack at the instance's largest coordinate.
__device__ __forceinline__ void exact_bounds(float smin, float rmax, float *s_hi, float *r_lo) {
  const float r = sqrtf(rmax), m = dist_slack(1.5f * r, 2.f);
  const bool ok = m <= 0.25f;  // else every pair and circle in binary64
  const float l = sqrtf(smin) + 2.f * m, w = fmaxf(r - 2.f * m, 0.f);
  *s_hi = ok ? fminf(l * l, (2.f + m) * (2.f + m)) : __int_as_float(0x7f800000);
  *r_lo = ok ? w * w : -1.f;
}

// Visit the circles around sorted position p: f(q, squared distance in binary32) for every other circle
// of its 3x3 cells.
template <typename F>
__device__ __forceinline__ void for_candidates(int p, int key, int nc, const int32_t *start, const float2 *xs, F f) {
  const int cy = key / nc, cx = key - cy * nc;
  const int bx0 = max(cx - 1, 0), bx1 = min(cx + 1, nc - 1);
  const float2 a = xs[p];
  for (int by = max(cy - 1, 0); by <= min(cy + 1, nc - 1); ++by) {
    const int lo = start[by * nc + bx0], hi = start[by * nc + bx1 + 1];
    for (int q = lo; q < hi; ++q) {
      if (q == p) continue;
      const float dx = a.x - xs[q].x, dy = a.y - xs[q].y;
      f(q, dx * dx + dy * dy);
    }
  }
}

__global__ void __launch_bounds__(512, 3) feasible_block_kernel(StandaloneParams P, int from32, double tol,
                                                             uint8_t *feasible, double *max_overlap) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int32_t sh[40];
  __shared__ float f_s[32], f_r[32];
  __shared__ int h_n[32];
  __shared__ double d_s[32], d_r[32];
  const int q = P.eorder[blockIdx.x];  // largest instance first
  const InstDesc &D = P.desc[q];
  const int n = D.n;
  if (n > kCellsBlockN) return;
  const Coords<double> X = coords_of<double>(P, D.off, from32);
  const int nc = D.ncx, lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float rmax = 0.f;
  int bad = 0;
  const BlockCells C =
      block_cells<double>(X, n, D.R, D.inv_cs, nc, sm, 0, P.cells + D.cell_off, nullptr, nullptr, sh,
                          [&](double2 p, float2 f, int) {
                            rmax = fmaxf(rmax, f.x * f.x + f.y * f.y);
                            bad |= not_finite(p.x) || not_finite(p.y);
                          });
  const float inf = __int_as_float(0x7f800000);
  float smin = inf;
  int hits = 0;
  Near<double> near(P.l_cut);
  for (int p = threadIdx.x; p < n; p += blockDim.x) {
    const int i = C.ord[p];
    near.set(C.xs[p]);
    for_candidates(p, (int)C.key[i], nc, C.start, C.xs, [&](int qq, float s) {
      smin = fminf(smin, s);
      if (s > near.hi) return;
      hits += (s < near.lo) || nbr_pred(X.at(i), X.at(C.ord[qq]), near.lc2);
    });
  }
  const float my_s = smin;
  smin = -warp_max(-smin);
  rmax = warp_max(rmax);
  hits = warp_sum(hits);
  if (lane == 0) { f_s[w] = smin; f_r[w] = rmax; h_n[w] = hits; }
  bad = __syncthreads_or(bad);
  long long tot = 0;
  for (int u = 0; u < nw; ++u) {
    smin = fminf(smin, f_s[u]);
    rmax = fmaxf(rmax, f_r[u]);
    tot += h_n[u];
  }
  bad |= tot > 2ll * D.cap;
  unsigned long long sb = 0x7ff0000000000000ull;  // squared distances compare as integers
  double r2 = 0.0;
  if (!bad) {
    float s_hi, r_lo;
    exact_bounds(smin, rmax, &s_hi, &r_lo);
    const bool pairs = !(my_s > s_hi);
    for (int p = threadIdx.x; p < n; p += blockDim.x) {
      const float2 a = C.xs[p];
      const int i = C.ord[p];
      if (!(a.x * a.x + a.y * a.y < r_lo)) r2 = fmax(r2, norm2_exact(X.at(i)));
      if (pairs) {  // each pair once; in a finished layout every contact lies within the slack
        const double2 xi = X.at(i);
        for_candidates(p, (int)C.key[i], nc, C.start, C.xs, [&](int qq, float s) {
          if (qq > p && !(s > s_hi))
            sb = min(sb, (unsigned long long)__double_as_longlong(dist2_exact(xi, X.at(C.ord[qq]))));
        });
      }
    }
  }
  double s2 = __longlong_as_double((long long)sb);
  s2 = -warp_max(-s2);
  r2 = warp_max(r2);
  if (lane == 0) { d_s[w] = s2; d_r[w] = r2; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int u = 1; u < nw; ++u) { s2 = fmin(s2, d_s[u]); r2 = fmax(r2, d_r[u]); }
    feasible_result(P, q, D.R, bad, s2, r2, tol, feasible, max_overlap);
  }
}

// the same over the tiles of the larger instances: the binary32 search, the exact pass, the result
template <bool EXACT>
__global__ void __launch_bounds__(kTileRows) large_check_kernel(StandaloneParams P, LargeTiles L, LargeDest O,
                                                                int from32) {
  const int2 t = L.rows[blockIdx.x];
  const InstDesc &D = P.desc[t.x];
  const int n = D.n, p = t.y * kTileRows + threadIdx.x, nc = D.ncx, lane = threadIdx.x & 31;
  const Coords<double> X = coords_of<double>(P, D.off, from32);
  const int32_t *start = P.cells + D.cell_off, *ord = O.corder + D.off;
  const float2 *xs = O.xs + D.off;
  const float inf = __int_as_float(0x7f800000);
  if (!EXACT) {
    float smin = inf;
    int hits = 0;
    if (p < n) {
      const int i = ord[p];
      Near<double> near(P.l_cut);
      near.set(xs[p]);
      for_candidates(p, (int)O.ckey[D.off + i], nc, start, xs, [&](int q, float s) {
        smin = fminf(smin, s);
        if (s > near.hi) return;
        hits += (s < near.lo) || nbr_pred(X.at(i), X.at(ord[q]), near.lc2);
      });
    }
    smin = -warp_max(-smin);
    hits = warp_sum(hits);
    if (lane == 0) {
      atomicMin(&L.smin32[t.x], __float_as_uint(smin));
      if (hits) atomicAdd(&L.hits[t.x], (unsigned long long)hits);
    }
  } else {
    if (L.bad[t.x] || L.hits[t.x] > 2ull * (unsigned long long)D.cap) return;
    float s_hi, r_lo;
    exact_bounds(__uint_as_float(L.smin32[t.x]), __uint_as_float(L.rmax32[t.x]), &s_hi, &r_lo);
    if (p >= n) return;
    const int i = ord[p];
    const float2 a = xs[p];
    if (!(a.x * a.x + a.y * a.y < r_lo))
      atomicMax(&L.rmax[t.x], (unsigned long long)__double_as_longlong(norm2_exact(X.at(i))));
    unsigned long long sb = 0x7ff0000000000000ull;  // squared distances compare as integers
    for_candidates(p, (int)O.ckey[D.off + i], nc, start, xs, [&](int q, float s) {
      if (q > p && !(s > s_hi))  // each pair once; in a finished layout every contact lies within the slack
        sb = min(sb, (unsigned long long)__double_as_longlong(dist2_exact(X.at(i), X.at(ord[q]))));
    });
    if (sb < 0x7ff0000000000000ull) atomicMin(&L.smin[t.x], sb);
  }
}
__global__ void large_check_init_kernel(StandaloneParams P, LargeTiles L) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= L.nrows) return;
  const int2 t = L.rows[b];
  if (t.y) return;
  L.hits[t.x] = 0;
  L.smin[t.x] = 0x7ff0000000000000ull;
  L.rmax[t.x] = 0;
  L.smin32[t.x] = 0x7f800000u;
  L.rmax32[t.x] = 0;
  L.bad[t.x] = 0;
}
__global__ void large_check_result_kernel(StandaloneParams P, LargeTiles L, double tol, uint8_t *feasible,
                                          double *max_overlap) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= L.nrows) return;
  const int2 t = L.rows[b];
  if (t.y) return;
  const InstDesc &D = P.desc[t.x];
  const bool bad = L.bad[t.x] || L.hits[t.x] > 2ull * (unsigned long long)D.cap;
  feasible_result(P, t.x, D.R, bad, __longlong_as_double((long long)L.smin[t.x]),
                  __longlong_as_double((long long)L.rmax[t.x]), tol, feasible, max_overlap);
}

// ---------------------------------------------------------------- export ----
__global__ void export_csr_kernel(StandaloneParams P, const int64_t *__restrict__ base, int32_t *row_ptr,
                                  int32_t *col) {
  int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= P.total) {
    if (gi == P.total && P.num > 0) row_ptr[P.total] = (int32_t)base[P.num];
    return;
  }
  const int q = P.inst_of[gi];
  const InstDesc D = P.desc[q];
  const int i = (int)(gi - D.off);
  const int32_t *rp = P.rp + D.off + q;
  const int lo = rp[i], hi = rp[i + 1];
  const int64_t b = base[q];
  row_ptr[gi] = (int32_t)(b + lo);
  for (int t = lo; t < hi; ++t) col[b + t] = (int32_t)(D.off + P.col[D.col_s_off + t]);
}

__global__ void export_cells_kernel(StandaloneParams P, uint32_t *key, int32_t *order) {
  int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= P.total) return;
  key[gi] = P.ckey[gi];
  order[gi] = P.corder[gi];
}

__global__ void nnz_kernel(StandaloneParams P, int64_t *nnz) {
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= P.num) return;
  const InstDesc D = P.desc[q];
  nnz[q] = (int64_t)P.rp[D.off + q + D.n];
}

__global__ void outputs_kernel(const InstOut *out, int num, int32_t *iters, int32_t *status, double *E,
                               int32_t *builds, int32_t *changes, int32_t *trials) {
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= num) return;
  if (iters) iters[q] = out[q].iters;
  if (status) status[q] = out[q].status;
  if (E) E[q] = out[q].E;
  if (builds) builds[q] = out[q].builds;
  if (changes) changes[q] = out[q].changes;
  if (trials) trials[q] = out[q].trials;
}

__global__ void stats_kernel(const InstOut *out, int num, int32_t *st) {
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= num) return;
  const InstOut o = out[q];
  int32_t *r = st + 10 * (int64_t)q;
  r[0] = o.iters; r[1] = o.status; r[2] = o.builds; r[3] = o.changes; r[4] = o.trials;
  r[5] = o.resets; r[6] = o.stalls; r[7] = o.polished; r[8] = o.iters32; r[9] = o.trials32;
}

}  // namespace

cudaError_t raise_smem_limit(const void *kernel) {
  int dev = 0, optin = 0;
  cudaFuncAttributes a;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, kernel);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)a.sharedSizeBytes);
}

cudaError_t standalone_smem_limits(int n_small, const int (&eg_small)[3]) {
  const size_t rows = 16 * (size_t)kBuildWarpBytes;  // of 512 threads
  const int n = std::max(n_small, 0);
  const struct { const void *kernel; size_t bytes; } most[] = {
      {(const void *)build_block_kernel<float>, cells_smem(n, rows, false)},
      {(const void *)build_block_kernel<double>, cells_smem(n, rows, true)},
      {(const void *)feasible_block_kernel, cells_smem(n, 0, true)},
      {(const void *)energy_grad_block_kernel<Arith64>, sizeof(double2) * (size_t)std::max(eg_small[0], 0)},
      {(const void *)energy_grad_block_kernel<Arith32>, sizeof(float2) * (size_t)std::max(eg_small[1], 0)},
      {(const void *)energy_grad_block_kernel<ArithMix>, sizeof(double2) * (size_t)std::max(eg_small[2], 0)}};
  for (const auto &k : most)
    if (cudaError_t e = raise_smem_limit(k.kernel, k.bytes)) return e;
  return cudaSuccess;
}

cudaError_t launch_init(const StandaloneParams &p, uint64_t seed, int mode, int prec, cudaStream_t s) {
  if (p.total > 0) init_kernel<<<blocks_for(p.total, 256), 256, 0, s>>>(p, seed, mode, prec);
  return cudaGetLastError();
}

cudaError_t launch_set_positions(const StandaloneParams &p, const double *xy, int prec, cudaStream_t s) {
  if (p.total > 0) set_pos_kernel<<<blocks_for(p.total, 256), 256, 0, s>>>(p, xy, prec);
  return cudaGetLastError();
}

cudaError_t launch_get_positions(const StandaloneParams &p, double *xy, int from32, cudaStream_t s) {
  if (p.total > 0) get_pos_kernel<<<blocks_for(p.total, 256), 256, 0, s>>>(p, xy, from32);
  return cudaGetLastError();
}

cudaError_t launch_set_radius(InstDesc *desc, const double *R, int num, double l_cut, cudaStream_t s) {
  if (num > 0) set_radius_kernel<<<blocks_for(num, 128), 128, 0, s>>>(desc, R, num, l_cut);
  return cudaGetLastError();
}

// Threads of a block per instance: one circle per thread up to 256; 512 when the instances leave SMs
// idle anyway.
static int cells_threads(int n_small, int num, int sms) {
  if (n_small > 512 && num <= sms) return 512;
  return n_small <= 64 ? 64 : (n_small <= 128 ? 128 : 256);
}

template <typename T>
static cudaError_t build_t(const StandaloneParams &p, const LargeTiles &L, int n_small, int sms, int force,
                           int32_t *rebuilt, cudaStream_t s) {
  if (n_small >= 0) {
    const int block = cells_threads(n_small, p.num, sms);
    const size_t smem = cells_smem(n_small, (size_t)(block / 32) * kBuildWarpBytes, sizeof(T) == 8);
    build_block_kernel<T><<<p.num, block, smem, s>>>(p, force, rebuilt);
  }
  if (L.nrows > 0) {
    const LargeDest O{p.ckey, p.corder, (float2 *)p.xtmp};
    cudaError_t e = large_cells<T, false>(p, L, O, 0, force, (v2<T> *)p.xbuild, s);
    if (e != cudaSuccess) return e;
    large_rows_kernel<T, false><<<L.nrows, kTileRows, 0, s>>>(p, L, O, nullptr);
    large_rows_kernel<T, true><<<L.nrows, kTileRows, 0, s>>>(p, L, O, rebuilt);
  }
  return cudaGetLastError();
}

cudaError_t launch_build(const StandaloneParams &p, const LargeTiles &L, int n_small, int sms, int prec, int force,
                         int32_t *rebuilt, cudaStream_t s) {
  if (p.num <= 0) return cudaSuccess;
  return prec == 1 ? build_t<float>(p, L, n_small, sms, force, rebuilt, s)
                   : build_t<double>(p, L, n_small, sms, force, rebuilt, s);
}

cudaError_t launch_large_cells32(const StandaloneParams &p, const LargeTiles &L, cudaStream_t s) {
  return large_cells<float, false>(p, L, LargeDest{p.ckey_t, p.corder_t, (float2 *)p.xtmp}, 0, 1, nullptr, s);
}

template <class A> static cudaError_t launch_eg_block(const StandaloneParams &p, int stage_n, size_t smem,
                                                     void *grad, double *E, cudaStream_t s) {
  energy_grad_block_kernel<A><<<p.num, kEgBlock, smem, s>>>(p, stage_n, grad, E);
  return cudaGetLastError();
}

// max_small_n: the largest instance of at most stage_n(eval) circles (-1: none; instances of 0
// circles get E = 0 from the block kernel); any_large: some instance has more.
cudaError_t launch_energy_grad(const StandaloneParams &p, int eval, double *E, void *grad, void *ecirc,
                               int max_small_n, bool any_large, cudaStream_t s) {
  if (p.num <= 0) return cudaSuccess;
  const int stage_n = energy_stage_n(eval);
  cudaError_t e = cudaSuccess;
  if (max_small_n >= 0) {
    const size_t smem = std::max<size_t>(16, (size_t)max_small_n * (eval == 1 ? sizeof(float2) : sizeof(double2)));
    if (eval == 0) e = launch_eg_block<Arith64>(p, stage_n, smem, grad, E, s);
    else if (eval == 1) e = launch_eg_block<Arith32>(p, stage_n, smem, grad, E, s);
    else e = launch_eg_block<ArithMix>(p, stage_n, smem, grad, E, s);
    if (e != cudaSuccess) return e;
  }
  if (any_large && p.total > 0) {
    unsigned nb = blocks_for(p.total, 256);
    if (eval == 0) energy_grad_kernel<Arith64><<<nb, 256, 0, s>>>(p, stage_n, grad, ecirc);
    else if (eval == 1) energy_grad_kernel<Arith32><<<nb, 256, 0, s>>>(p, stage_n, grad, ecirc);
    else energy_grad_kernel<ArithMix><<<nb, 256, 0, s>>>(p, stage_n, grad, ecirc);
    if (eval == 1) energy_reduce_kernel<float><<<p.num, 1024, 0, s>>>(p, stage_n, (const float *)ecirc, E);
    else energy_reduce_kernel<double><<<p.num, 1024, 0, s>>>(p, stage_n, (const double *)ecirc, E);
  }
  return cudaGetLastError();
}

cudaError_t launch_feasible(const StandaloneParams &p, const LargeTiles &L, int n_small, int sms, int from32,
                            double tol, uint8_t *feasible, double *max_overlap, cudaStream_t s) {
  if (p.num <= 0) return cudaSuccess;
  if (n_small >= 0) {
    const size_t smem = cells_smem(n_small, 0, true);
    feasible_block_kernel<<<p.num, cells_threads(n_small, p.num, sms), smem, s>>>(p, from32, tol, feasible, max_overlap);
  }
  if (L.nrows > 0) {
    const LargeDest O{p.ckey_t, p.corder_t, (float2 *)p.xtmp2};
    const unsigned nb = blocks_for(L.nrows, 128);
    large_check_init_kernel<<<nb, 128, 0, s>>>(p, L);
    cudaError_t e = large_cells<double, true>(p, L, O, from32, 1, nullptr, s);
    if (e != cudaSuccess) return e;
    large_check_kernel<false><<<L.nrows, kTileRows, 0, s>>>(p, L, O, from32);
    large_check_kernel<true><<<L.nrows, kTileRows, 0, s>>>(p, L, O, from32);
    large_check_result_kernel<<<nb, 128, 0, s>>>(p, L, tol, feasible, max_overlap);
  }
  return cudaGetLastError();
}

cudaError_t launch_export_csr(const StandaloneParams &p, const int64_t *base, int32_t *row_ptr, int32_t *col,
                              cudaStream_t s) {
  export_csr_kernel<<<blocks_for(p.total + 1, 256), 256, 0, s>>>(p, base, row_ptr, col);
  return cudaGetLastError();
}

cudaError_t launch_export_cells(const StandaloneParams &p, uint32_t *key, int32_t *order, cudaStream_t s) {
  if (p.total > 0) export_cells_kernel<<<blocks_for(p.total, 256), 256, 0, s>>>(p, key, order);
  return cudaGetLastError();
}

cudaError_t launch_nnz(const StandaloneParams &p, int64_t *nnz, cudaStream_t s) {
  if (p.num > 0) nnz_kernel<<<blocks_for(p.num, 128), 128, 0, s>>>(p, nnz);
  return cudaGetLastError();
}

cudaError_t launch_outputs(const InstOut *out, int num, int32_t *iters, int32_t *status, double *E,
                           int32_t *builds, int32_t *changes, int32_t *trials, cudaStream_t s) {
  if (num > 0) outputs_kernel<<<blocks_for(num, 128), 128, 0, s>>>(out, num, iters, status, E, builds, changes, trials);
  return cudaGetLastError();
}

cudaError_t launch_stats(const InstOut *out, int num, int32_t *stats, cudaStream_t s) {
  if (num > 0) stats_kernel<<<blocks_for(num, 128), 128, 0, s>>>(out, num, stats);
  return cudaGetLastError();
}

}  // namespace pecc
