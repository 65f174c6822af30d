// pecc_mlp.cu -- the learned warm start: a per-circle MLP that reads the relative offsets of a
// circle's 12 nearest neighbours and its distance to the container wall and proposes a
// displacement; training (forward, backward, Adam) and inference are the kernels below, with the
// 128-wide GEMMs of every layer on the fifth-generation tensor cores (tcgen05.mma, BF16 inputs,
// FP32 accumulators in TMEM).
//
// Features of circle i (binary32, every operation correctly rounded so that a plain CPU
// restatement reproduces them bit for bit): the frame e_r = c_i / |c_i| (e_r = (1, 0) at the
// origin), e_t = (-e_r.y, e_r.x); the 12 nearest other centres within 4.5 (by squared distance,
// then index) as offsets d = c_j - c_i projected on (e_r, e_t), zero where fewer exist; and
// b = min(R - |c_i| - 1, 4.5).  The network 25 -> 128 -> 128 -> 128 -> 2 (ReLU) outputs the
// displacement in the same frame.
#include <cuda_bf16.h>

#include "pecc_cells.cuh"
#include "pecc_internal.h"
#include "pecc_tc.cuh"

namespace pecc {
namespace {

using bf16 = __nv_bfloat16;

constexpr int KNN = 12;
constexpr float kKnnR2 = 4.5f * 4.5f;
constexpr int H = 128;
constexpr int F = 25;      // features
constexpr int SA = 136;    // padded row stride (bf16) of 128-wide tiles: conflict-free fragments
constexpr int S1 = 40;     // padded row stride of 32-wide tiles

// ---------------------------------------------------------------------------- parameters ----
// Flat binary32 parameter vector: W1[128][25] b1[128] W2[128][128] b2[128] W3[128][128] b3[128]
// W4[2][128] b4[2].
constexpr int OW1 = 0, OB1 = OW1 + H * F, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H, OB3 = OW3 + H * H,
              OW4 = OB3 + H, OB4 = OW4 + 2 * H, NPAR = OB4 + 2;
// BF16 copies in the padded layouts the kernels read: W1[128][40] W2[128][136] W3[128][136] W4[16][136].
constexpr int BW1 = 0, BW2 = BW1 + H * S1, BW3 = BW2 + H * SA, BW4 = BW3 + H * SA, NBW = BW4 + 16 * SA;

__device__ __forceinline__ uint32_t pack2(bf16 lo, bf16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}


// ------------------------------------------------------------------------------- features ----
__device__ __forceinline__ float2 frame_er(float2 c) {
  const float r = __fsqrt_rn(__fadd_rn(__fmul_rn(c.x, c.x), __fmul_rn(c.y, c.y)));
  if (!(r > 0.f)) return make_float2(1.f, 0.f);
  return make_float2(__fdiv_rn(c.x, r), __fdiv_rn(c.y, r));
}

// Cells that 4.5 spans: the grid's side is at least l_cut (1 + 2^-20), l_cut above 2.  (The margin covers
// the binary32 distances: one below 4.5 is below 4.5 (1 + 2^-22) in exact terms.)
static int knn_reach(double l_cut) { return l_cut >= 2.25 ? 2 : 3; }

// A lane takes one circle: it collects the circles within 4.5 (at most `reach` cells away) as positions in
// a column of its warp's buffer, then keeps the twelve least (squared distance, index) of them as ascending
// 64-bit keys: the distance's bits, then the index (and, where both fit 16 bits, the sorted position, which
// gives the coordinates without a search).  Collecting first lets the insertions of a warp's lanes run
// together.  The warp's 32 rows of 25 values leave through shared memory as one contiguous piece.
constexpr int kKnnBuf = 32;                               // collected per lane before they are inserted
constexpr int kKnnWarpBytes = 32 * F * (int)sizeof(float);  // the rows of a warp
static_assert(kKnnWarpBytes >= 32 * kKnnBuf * (int)sizeof(uint16_t), "the rows take the 16-bit buffer's place");
static_assert(kKnnWarpBytes <= 32 * kKnnBuf * (int)sizeof(int32_t), "and fit the 32-bit one's");

// I: type of the sorted order's entries (16-bit: keys carry the position).
template <typename I>
__device__ __forceinline__ void feature_rows(const float2 *__restrict__ x, int n, int i, float Rf, int key, int nc,
                                             int reach, const int32_t *start, const float2 *xs, const I *ord, void *scratch,
                                             float *__restrict__ feat) {
  constexpr bool pack = sizeof(I) == 2;
  const int lane = threadIdx.x & 31;
  const bool act = i < n;
  unsigned long long best[KNN];
#pragma unroll
  for (int u = 0; u < KNN; ++u) best[u] = ~0ull;
  const float2 xi = act ? x[i] : make_float2(0.f, 0.f);
  if (act) {
    I *buf = (I *)scratch + lane;
    int cnt = 0;
    auto dist2 = [&](int q) {
      const float2 xj = xs[q];
      const float dx = __fsub_rn(xj.x, xi.x), dy = __fsub_rn(xj.y, xi.y);
      return __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
    };
    auto insert_all = [&]() {
      for (int h = 0; h < cnt; ++h) {
        const int q = (int)buf[32 * h];
        const int j = (int)ord[q];
        if (j == i) continue;
        unsigned long long k = ((unsigned long long)__float_as_uint(dist2(q)) << 32) |
                               (pack ? ((unsigned)j << 16) | (unsigned)q : (unsigned)j);
#pragma unroll
        for (int u = 0; u < KNN; ++u) {
          const unsigned long long b = best[u];
          const bool less = k < b;
          best[u] = less ? k : b;
          k = less ? b : k;
        }
      }
      cnt = 0;
    };
    const int cy = key / nc, cx = key - cy * nc;
    const int bx0 = max(cx - reach, 0), bx1 = min(cx + reach, nc - 1);
    for (int yy = max(cy - reach, 0); yy <= min(cy + reach, nc - 1); ++yy) {
      const int lo = start[yy * nc + bx0], hi = start[yy * nc + bx1 + 1];
      for (int q = lo; q < hi; ++q) {
        if (!(dist2(q) < kKnnR2)) continue;
        buf[32 * cnt] = (I)q;
        if (++cnt == kKnnBuf) insert_all();
      }
    }
    insert_all();
  }
  __syncwarp();  // the rows take the buffer's place
  float *rows = (float *)scratch;
  if (act) {
    const float2 er = frame_er(xi);
    float *f = rows + F * lane;
#pragma unroll
    for (int u = 0; u < KNN; ++u) {
      const bool has = best[u] != ~0ull;
      float2 xj = xi;
      if (has) xj = pack ? xs[best[u] & 0xffffu] : x[best[u] & 0xffffffffu];
      const float dx = __fsub_rn(xj.x, xi.x), dy = __fsub_rn(xj.y, xi.y);
      f[2 * u] = has ? __fadd_rn(__fmul_rn(dx, er.x), __fmul_rn(dy, er.y)) : 0.f;
      f[2 * u + 1] = has ? __fsub_rn(__fmul_rn(dy, er.x), __fmul_rn(dx, er.y)) : 0.f;
    }
    const float r = __fsqrt_rn(__fadd_rn(__fmul_rn(xi.x, xi.x), __fmul_rn(xi.y, xi.y)));
    const float b = __fsub_rn(__fsub_rn(Rf, r), 1.0f);
    f[24] = fminf(b, 4.5f);
  }
  __syncwarp();
  const int i0 = i - lane, m = min(32, n - i0) * F;
  for (int t = lane; t < m; t += 32) feat[(size_t)i0 * F + t] = rows[t];
  __syncwarp();
}

// Instances of at most kCellsBlockN circles, one block each (pecc_cells.cuh).  Bound by instruction issue
// of the collecting and inserting walks: 145 us for 665 000 circles in 1024 instances, 460 us when cells
// and lists lay in global memory and every lane inserted as it walked.
__global__ void __launch_bounds__(256) features_block_kernel(StandaloneParams P, int reach, float *feat) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int32_t sh[40];
  const int q = P.eorder[blockIdx.x];
  const InstDesc &D = P.desc[q];
  const int n = D.n;
  if (n > kCellsBlockN) return;
  const Coords<float> X{P.x32 + D.off, P.l_cut};
  const size_t extra = (size_t)(blockDim.x >> 5) * kKnnWarpBytes;
  const BlockCells C = block_cells<float>(X, n, D.R, D.inv_cs, D.ncx, sm, extra, P.cells + D.cell_off, nullptr, nullptr,
                                          sh, [](float2, float2, int) {});
  void *scratch = C.extra + (threadIdx.x >> 5) * kKnnWarpBytes;
  for (int i0 = threadIdx.x & ~31; i0 < n; i0 += blockDim.x) {
    const int i = i0 + (threadIdx.x & 31);
    feature_rows<uint16_t>(X.x, n, i, (float)D.R, i < n ? (int)C.key[i] : 0, D.ncx, reach, C.start, C.xs, C.ord,
                           scratch, feat + (size_t)D.off * F);
  }
}

// Tiles of the larger instances, over the cells that launch_large_cells32 left in the scratch.
__global__ void __launch_bounds__(kTileRows) features_tile_kernel(StandaloneParams P, LargeTiles L, int reach,
                                                                  float *feat) {
  __shared__ __align__(16) unsigned char sm[(kTileRows / 32) * 32 * kKnnBuf * 4];
  const int2 t = L.rows[blockIdx.x];
  const InstDesc &D = P.desc[t.x];
  const int n = D.n, i = t.y * kTileRows + threadIdx.x;
  if (i - (int)(threadIdx.x & 31) >= n) return;  // the whole warp
  feature_rows<int32_t>(P.x32 + D.off, n, i, (float)D.R, i < n ? (int)P.ckey_t[D.off + i] : 0, D.ncx, reach,
                        P.cells + D.cell_off, (const float2 *)P.xtmp + D.off, P.corder_t + D.off,
                        sm + (threadIdx.x >> 5) * 32 * kKnnBuf * 4, feat + (size_t)D.off * F);
}

// Target of circle i: its displacement from x_before to now, in the frame of x_before.
__global__ void targets_kernel(StandaloneParams P, const double *__restrict__ xbefore, float *target) {
  const int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= P.total) return;
  const float2 x0 = make_float2((float)xbefore[2 * gi], (float)xbefore[2 * gi + 1]);
  const float2 x1 = P.x32[gi];
  const float2 er = frame_er(x0);
  const float dx = __fsub_rn(x1.x, x0.x), dy = __fsub_rn(x1.y, x0.y);
  target[2 * gi] = __fadd_rn(__fmul_rn(dx, er.x), __fmul_rn(dy, er.y));
  target[2 * gi + 1] = __fsub_rn(__fmul_rn(dy, er.x), __fmul_rn(dx, er.y));
}

// ------------------------------------------------------------------ tensor-core network ----
// Both kernels below keep every weight and activation tile in shared memory in the core layout of
// pecc_tc.cuh and run the 128-wide GEMMs as tcgen05 MMAs (M = 128 rows of a tile, K = 16 per
// instruction) issued by one thread, with FP32 accumulators in TMEM; a thread owns a row of a tile
// (TMEM lane r) in every epilogue, or a quarter of its columns.  The 2-wide output layer runs on the CUDA
// cores inside the epilogues.
constexpr int TM = 128;                  // rows per tile
constexpr int FPAD = 32;                 // padded input width
constexpr uint32_t kW1B = TM * FPAD * 2;  // bytes of a [128][32] bf16 core tile
constexpr uint32_t kHB = TM * H * 2;      // bytes of a [128][128] bf16 core tile
constexpr long long kWaitNs = 2000000000ll;  // bound of every wait on the MMA barrier
constexpr uint32_t kColStep = 2 * 128;       // a K step of 16 along the columns: two cores

// weights of the block: W1 [128][32], W2, W3 [128][128] in the core layout, from the padded bf16
// copies; biases b1 b2 b3 [128], the output layer W4 (bf16 values; both rows' entries of a column side
// by side: [128][2]) and b4 [2] as floats
__device__ void tc_load_weights(const bf16 *__restrict__ wb, const float *__restrict__ params, unsigned char *w1,
                                unsigned char *w2, unsigned char *w3, float *fb) {
  for (int u = threadIdx.x; u < TM * (FPAD / 8); u += blockDim.x) {
    const int o = u / (FPAD / 8), c8 = u % (FPAD / 8);
    *(uint4 *)(w1 + tc::core_off(o, 8 * c8, FPAD)) = *(const uint4 *)(wb + BW1 + o * S1 + 8 * c8);
  }
  for (int u = threadIdx.x; u < TM * (H / 8); u += blockDim.x) {
    const int o = u / (H / 8), c8 = u % (H / 8);
    *(uint4 *)(w2 + tc::core_off(o, 8 * c8, H)) = *(const uint4 *)(wb + BW2 + o * SA + 8 * c8);
    *(uint4 *)(w3 + tc::core_off(o, 8 * c8, H)) = *(const uint4 *)(wb + BW3 + o * SA + 8 * c8);
  }
  for (int u = threadIdx.x; u < H; u += blockDim.x) {
    fb[u] = params[OB1 + u];
    fb[H + u] = params[OB2 + u];
    fb[2 * H + u] = params[OB3 + u];
    fb[3 * H + 2 * u] = __bfloat162float(wb[BW4 + u]);
    fb[3 * H + 2 * u + 1] = __bfloat162float(wb[BW4 + SA + u]);
  }
  if (threadIdx.x < 2) fb[5 * H + threadIdx.x] = params[OB4 + threadIdx.x];
}

// Two floats rounded to bf16, low half first, and back.
__device__ __forceinline__ uint32_t pack2f(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);  // one conversion instruction
  return *(const uint32_t *)&v;
}
__device__ __forceinline__ float lo2f(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi2f(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// 32 bf16 values (16 words) of row r starting at column c0 of a [128][C] core tile
__device__ __forceinline__ void tc_store32(unsigned char *t, int r, int c0, int C, const uint32_t (&w)[16]) {
#pragma unroll
  for (int c8 = 0; c8 < 4; ++c8)
    *(uint4 *)(t + tc::core_off(r, c0 + 8 * c8, C)) = make_uint4(w[4 * c8], w[4 * c8 + 1], w[4 * c8 + 2], w[4 * c8 + 3]);
}
__device__ __forceinline__ void trace32(float *t, const uint32_t (&w)[16]) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    t[2 * j] = lo2f(w[j]);
    t[2 * j + 1] = hi2f(w[j]);
  }
}

// Hidden layer, columns [c0, c0 + 32) of this thread's row: accumulator plus bias, ReLU, rounded to bf16.
__device__ __forceinline__ void tc_hidden32(uint32_t taddr, const float *bias, uint32_t (&w)[16]) {
  float v[32];
  tc::ld32(taddr, v);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float4 b = *(const float4 *)(bias + 4 * j);
    w[2 * j] = pack2f(fmaxf(v[4 * j] + b.x, 0.f), fmaxf(v[4 * j + 1] + b.y, 0.f));
    w[2 * j + 1] = pack2f(fmaxf(v[4 * j + 2] + b.z, 0.f), fmaxf(v[4 * j + 3] + b.w, 0.f));
  }
}
// The output layer over 32 columns: o0 / o1 += h W4^T from the rounded values, columns in order.
__device__ __forceinline__ void tc_out32(const uint32_t (&w)[16], const float *w4, float &o0, float &o1) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const float4 a = *(const float4 *)(w4 + 4 * j);
    o0 = fmaf(lo2f(w[j]), a.x, o0);
    o1 = fmaf(lo2f(w[j]), a.y, o1);
    o0 = fmaf(hi2f(w[j]), a.z, o0);
    o1 = fmaf(hi2f(w[j]), a.w, o1);
  }
}

// One thread issues D = A B^T over K (K / 16 MMAs).  The operand descriptors advance by `astep` /
// `bstep` bytes per K step of 16.
__device__ __forceinline__ void tc_gemm(uint32_t d, uint32_t a_addr, bool a_krows, int a_cols, uint32_t astep,
                                        uint32_t b_addr, bool b_krows, int b_cols, uint32_t bstep, int N, int K,
                                        bool accumulate) {
  const uint32_t id = tc::idesc_bf16(TM, N, a_krows ? 1 : 0, b_krows ? 1 : 0);
  uint64_t ad = a_krows ? tc::desc_k_rows(a_addr, a_cols) : tc::desc_k_cols(a_addr, a_cols);
  uint64_t bd = b_krows ? tc::desc_k_rows(b_addr, b_cols) : tc::desc_k_cols(b_addr, b_cols);
#pragma unroll
  for (int ks = 0; ks < K / 16; ++ks) {  // the start address is the descriptors' low field, in 16-byte units
    tc::mma(d, ad, bd, id, (accumulate || ks > 0) ? 1 : 0);
    ad += astep >> 4;
    bd += bstep >> 4;
  }
}

// Barrier of one 128-thread group of the block (named barrier 1 + g; g < 0: of the block); whether any of
// its threads passed bad.
__device__ __forceinline__ bool group_any(bool bad, int g) {
  if (g < 0) return __syncthreads_or(bad);
  uint32_t any;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.b32 p, %1, 0;\nbarrier.cta.red.or.pred q, %2, 128, p;\nselp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(any)
      : "r"((uint32_t)bad), "r"(1 + g)
      : "memory");
  return any != 0;
}

// Make this group's shared-memory writes visible to the tensor cores and order TMEM accesses around a
// barrier of the group (g < 0: of the block).  ok: this thread's waits so far ended in time; returns
// whether all threads' did.
__device__ __forceinline__ bool tc_sync(bool ok = true, int g = -1) {
  tc::fence_smem_to_async();
  tc::fence_before();
  const bool any = group_any(!ok, g);
  tc::fence_after();
  return !any;
}

// Every warp waits for the barrier's current phase itself (a wait that runs out is reported to the
// group at its next barrier, so that all of them leave together).  The answer is the warp's: a lane that
// left out the next wait or a TMEM load, both warp-wide, would leave the others standing there.
__device__ __forceinline__ bool tc_wait(uint64_t *mbar, uint32_t &phase) {
  const bool ok = tc::mbar_wait_warp(mbar, phase, kWaitNs);
  phase ^= 1u;
  tc::fence_after();
  return ok;
}

// Forward: out[rows][2] for rows of feat[rows][25]; trace (may be null): float[rows][3][128], the bf16
// activations of the three hidden layers.  One block per SM, four groups of 128 threads that share the
// weights; each group takes a tile of 128 rows at a time through the chain MMA, epilogue, MMA by itself,
// so that three tiles' epilogues run while another's MMAs do.  A group's tile of inputs and its hidden
// activations take the same 32 KB (the inputs are dead once the first MMAs are done).  The features of
// the next tile are loaded, coalesced, while the last layer runs.
// 665 000 rows: 96 us, bound by shared-memory wavefronts and issue of the epilogues; 283 us with one group
// per SM and row-wise feature loads.
constexpr int kFwdGroups = 4;
constexpr int kRowLoads = F;  // 32 rows of F floats per warp, one per lane and load
constexpr uint32_t kFwdW1 = 0, kFwdW2 = kFwdW1 + kW1B, kFwdW3 = kFwdW2 + kHB, kFwdT = kFwdW3 + kHB,
                   kFwdF = kFwdT + kFwdGroups * kHB, kFwdBar = kFwdF + (5 * H + 4) * 4;
constexpr size_t kFwdSmem = (size_t)kFwdBar + 8 * kFwdGroups + 16 + 128;  // barriers, TMEM address; alignment

// the warp's 32 rows from row0 on, coalesced: float e = lane + 32 u of the 800 (zero past rows)
__device__ __forceinline__ void load_rows32(const float *__restrict__ feat, int64_t row0, int64_t rows, float (&v)[kRowLoads]) {
  const int lane = threadIdx.x & 31;
  const int64_t n = min((int64_t)32, rows - row0) * F;  // floats that exist (<= 0 past the end)
#pragma unroll
  for (int u = 0; u < kRowLoads; ++u) {
    const int e = lane + 32 * u;
    v[u] = e < n ? __ldg(feat + row0 * F + e) : 0.f;
  }
}
// ... to the [128][32] core tile x, rows r0 .. r0 + 31; columns 25 .. 31 zero
__device__ __forceinline__ void store_rows32(unsigned char *x, int r0, const float (&v)[kRowLoads]) {
  const int lane = threadIdx.x & 31;
  *(uint4 *)(x + tc::core_off(r0 + lane, 24, FPAD)) = make_uint4(0u, 0u, 0u, 0u);
  __syncwarp();
  int row = lane / F, c = lane % F;
#pragma unroll
  for (int u = 0; u < kRowLoads; ++u) {
    *(bf16 *)(x + tc::core_off(r0 + row, c, FPAD)) = __float2bfloat16_rn(v[u]);
    c += 32 - F;
    row += 1;
    if (c >= F) { c -= F; row += 1; }
  }
}

__global__ void __launch_bounds__(128 * kFwdGroups, 1)
forward_tc_kernel(const bf16 *__restrict__ wb, const float *__restrict__ params, const float *__restrict__ feat,
                  int64_t rows, float *out, float *trace) {
  extern __shared__ unsigned char sm_raw[];
  unsigned char *sm = (unsigned char *)(((uintptr_t)sm_raw + 127) & ~(uintptr_t)127);
  unsigned char *w1 = sm + kFwdW1, *w2 = sm + kFwdW2, *w3 = sm + kFwdW3;
  float *fb = (float *)(sm + kFwdF);
  const int g = threadIdx.x >> 7, r = threadIdx.x & 127, r0 = r & ~31;
  uint64_t *mbar = (uint64_t *)(sm + kFwdBar) + g;
  uint32_t *tslot = (uint32_t *)(sm + kFwdBar + 8 * kFwdGroups);
  unsigned char *h = sm + kFwdT + g * kHB;
  const bool issuer = r == 0;
  tc_load_weights(wb, params, w1, w2, w3, fb);
  if (issuer) tc::mbar_init(mbar);
  if (threadIdx.x < 32) tc::tmem_alloc<128 * kFwdGroups>(tslot);
  tc_sync();
  const uint32_t tacc = *tslot + 128 * g, lanes = (uint32_t)r0 << 16;
  const uint32_t sw1 = tc::smem_u32(w1), sw2 = tc::smem_u32(w2), sw3 = tc::smem_u32(w3), sh = tc::smem_u32(h);
  uint32_t phase = 0;
  bool ok = true;
  const int64_t tiles = (rows + TM - 1) / TM, stride = (int64_t)gridDim.x * kFwdGroups;
  int64_t tl = (int64_t)g * gridDim.x + blockIdx.x;  // the first tiles go to different SMs
  float v[kRowLoads];
  if (tl < tiles) load_rows32(feat, tl * TM + r0, rows, v);
  for (; tl < tiles; tl += stride) {
    const int64_t gr = tl * TM + r;
    float *tr = (trace && gr < rows) ? trace + gr * 3 * H : nullptr;
    store_rows32(h, r0, v);
    if (!(ok = tc_sync(ok, g))) break;
    if (issuer) { tc_gemm(tacc, sh, false, FPAD, kColStep, sw1, false, FPAD, kColStep, H, FPAD, false); tc::commit(mbar); }
    ok = tc_wait(mbar, phase);
    float o0 = 0.f, o1 = 0.f;
    for (int layer = 0; layer < 2; ++layer) {
      for (int c0 = 0; c0 < H; c0 += 32) {
        uint32_t w[16];
        tc_hidden32(tacc + lanes + (uint32_t)c0, fb + layer * H + c0, w);
        tc_store32(h, r, c0, H, w);
        if (tr) trace32(tr + layer * H + c0, w);
      }
      if (!(ok = tc_sync(ok, g))) break;
      if (issuer) {
        tc_gemm(tacc, sh, false, H, kColStep, layer == 0 ? sw2 : sw3, false, H, kColStep, H, H, false);
        tc::commit(mbar);
      }
      if (layer == 1 && tl + stride < tiles) load_rows32(feat, (tl + stride) * TM + r0, rows, v);
      ok = tc_wait(mbar, phase);
    }
    for (int c0 = 0; ok && c0 < H; c0 += 32) {
      uint32_t w[16];
      tc_hidden32(tacc + lanes + (uint32_t)c0, fb + 2 * H + c0, w);
      if (tr) trace32(tr + 2 * H + c0, w);
      tc_out32(w, fb + 3 * H + 2 * c0, o0, o1);
    }
    if (gr < rows) {
      out[gr * 2] = o0 + fb[5 * H];
      out[gr * 2 + 1] = o1 + fb[5 * H + 1];
    }
  }
  ok = !group_any(!ok, g);  // the last tile's wait
  if (!ok)  // the tensor cores did not answer in time: NaN outputs, nothing left waiting
    for (tl = (int64_t)g * gridDim.x + blockIdx.x; tl < tiles; tl += stride)
      if (tl * TM + r < rows) out[(tl * TM + r) * 2] = out[(tl * TM + r) * 2 + 1] = __int_as_float(0x7fc00000);
  tc::fence_before();
  __syncthreads();
  if (threadIdx.x < 32) {
    tc::fence_after();
    tc::tmem_free<128 * kFwdGroups>(*tslot);
  }
}

// ------------------------------------------------------------------------------- training ----
// One block of 512 threads per SM, persistent over tiles of 128 rows; in every epilogue four threads
// share a row, 32 columns each, so that an epilogue is one TMEM load deep.  Per tile: forward (keeping X,
// H1, H2, H3), then
//   dO = 2 (out - target) / rows (rounded to bf16)                          (CUDA cores)
//   dZ3 = (dO W4) o [H3 > 0]                                                (CUDA cores)
//   dH2 = dZ3 W3, dW4 += dO' H3, dW3 += dZ3' [H2 1];  dZ2 = dH2 o [H2 > 0]  (tensor cores)
//   dH1 = dZ2 W2, dW2 += dZ2' [H1 1];                 dZ1 = dH1 o [H1 > 0]  (tensor cores)
//   dW1 += dZ1' [X 1]                                                       (tensor cores)
// Every GEMM input is bf16 (dZ rounded like the activations).  The bias gradients are the columns of
// ones: column 128 of the 144-wide H1 and H2 tiles, column 25 of X (W1 is zero there).  The ReLU masks
// stay in registers, a word per layer.  dH2 and dH1 are issued before the weight gradients of their
// stage, which then run behind the next epilogue; dZ2 takes H3's room for that.  The accumulators dW1 to
// dW4 stay in TMEM until the block's last tile; the block then writes its partial gradient to
// part[block][NPAR] and its loss to loss_part[block].
// 333 000 rows: 161 us, bound by the chain of six MMA and epilogue stages per tile; 484 us with one
// 128-thread group, the column sums as scalar reads of shared memory and every MMA waited for.
// bwd_trace (may be null): float[rows][4][128], the bf16 dZ3, dZ2, dZ1 of every row, then its bf16
// dO (2 values) and its outputs (2 values).
constexpr int kTrT = 512;                      // threads
constexpr int HX = H + 16;                     // columns of the H1, H2 tiles: the activations, ones, zeros
constexpr uint32_t kHXB = TM * HX * 2, kDOB = TM * 16 * 2;
constexpr uint32_t kTrW1 = 0, kTrW2 = kTrW1 + kW1B, kTrW3 = kTrW2 + kHB, kTrX = kTrW3 + kHB, kTrH1 = kTrX + kW1B,
                   kTrH2 = kTrH1 + kHXB, kTrH3 = kTrH2 + kHXB, kTrZ = kTrH3 + kHB, kTrO = kTrZ + kHB,
                   kTrF = kTrO + kDOB;
// floats after kTrF: biases and W4 (5 H + 4), the partial outputs of the row quarters [4][128][2]
constexpr int kTrFo = 5 * H + 4, kTrFn = kTrFo + 8 * TM;
constexpr uint32_t kTrBar = kTrF + kTrFn * 4;  // two barriers, TMEM address
constexpr size_t kTrainSmem = (size_t)kTrBar + 32;
static_assert(kTrainSmem <= 227 * 1024, "one block per SM");
constexpr int kTrLoads = (TM * F + kTrT - 1) / kTrT;
// TMEM columns: [0, 128) the layer accumulator, then dW3 [144], dW2 [144], dW1 [32], dW4 [16]
constexpr uint32_t kTcW3 = 128, kTcW2 = 288, kTcW1 = 448, kTcW4 = 480;

__global__ void __launch_bounds__(kTrT, 1) train_tc_kernel(const bf16 *__restrict__ wb, const float *__restrict__ params,
                                                           const float *__restrict__ feat, const float *__restrict__ target,
                                                           int64_t rows, float *part, float *loss_part,
                                                           float *fwd_trace, float *bwd_trace) {
  extern __shared__ __align__(128) unsigned char sm_train[];
  unsigned char *const sm = sm_train;
  unsigned char *w1 = sm + kTrW1, *w2 = sm + kTrW2, *w3 = sm + kTrW3, *x = sm + kTrX;
  unsigned char *h1 = sm + kTrH1, *h2 = sm + kTrH2, *h3 = sm + kTrH3, *z = sm + kTrZ, *dot = sm + kTrO;
  float *fb = (float *)(sm + kTrF), *opart = fb + kTrFo;
  uint64_t *mbar = (uint64_t *)(sm + kTrBar), *mbar2 = mbar + 1;
  uint32_t *tslot = (uint32_t *)(mbar + 2);
  const int tid = threadIdx.x, r = tid & 127, cq = tid >> 7, c0 = 32 * cq;
  const bool issuer = tid == 0;
  tc_load_weights(wb, params, w1, w2, w3, fb);
  const bf16 one = __float2bfloat16_rn(1.f);
  for (int u = tid; u < 2 * TM; u += kTrT) {  // the columns past the activations: a one, zeros
    unsigned char *t = u < TM ? h1 : h2;
    *(uint4 *)(t + tc::core_off(u % TM, H, HX)) = make_uint4(pack2(one, __float2bfloat16_rn(0.f)), 0u, 0u, 0u);
    *(uint4 *)(t + tc::core_off(u % TM, H + 8, HX)) = make_uint4(0u, 0u, 0u, 0u);
  }
  if (tid < TM) {
    *(uint4 *)(x + tc::core_off(tid, 24, FPAD)) = make_uint4(pack2(__float2bfloat16_rn(0.f), one), 0u, 0u, 0u);
    *(uint4 *)(dot + tc::core_off(tid, 0, 16)) = make_uint4(0u, 0u, 0u, 0u);
    *(uint4 *)(dot + tc::core_off(tid, 8, 16)) = make_uint4(0u, 0u, 0u, 0u);
  }
  if (issuer) { tc::mbar_init(mbar); tc::mbar_init(mbar2); }
  if (tid < 32) tc::tmem_alloc<512>(tslot);
  tc_sync();
  const uint32_t tacc = *tslot, lanes = (uint32_t)(r & ~31) << 16;
  const uint32_t sw1 = tc::smem_u32(w1), sw2 = tc::smem_u32(w2), sw3 = tc::smem_u32(w3), sx = tc::smem_u32(x);
  const uint32_t sh1 = tc::smem_u32(h1), sh2 = tc::smem_u32(h2), sh3 = tc::smem_u32(h3), sz = tc::smem_u32(z),
                 sdo = tc::smem_u32(dot);
  // bytes of two 8-row core groups (a K step of 16 along the rows) by width
  constexpr uint32_t kStepH = 2 * (H / 8) * 128, kStepHX = 2 * (HX / 8) * 128, kStepX = 2 * (FPAD / 8) * 128,
                     kStepO = 2 * 2 * 128;
  const float scale = 2.f / (float)rows;
  float lsum = 0.f, sg0 = 0.f, sg1 = 0.f;
  uint32_t phase = 0, phase2 = 0;
  bool ok = true, first = true;
  const int64_t tiles = (rows + TM - 1) / TM;
  float v25[kTrLoads];
  auto load_tile = [&](int64_t t) {  // 128 rows of F floats, coalesced (zero past rows)
    const int64_t n = min((int64_t)TM, rows - t * TM) * F;
#pragma unroll
    for (int u = 0; u < kTrLoads; ++u) {
      const int e = tid + kTrT * u;
      v25[u] = e < n ? __ldg(feat + t * TM * F + e) : 0.f;
    }
  };
  int64_t tl = blockIdx.x;
  if (tl < tiles) load_tile(tl);
  for (; tl < tiles; tl += gridDim.x) {
    const int64_t gr = tl * TM + r;
    const bool live = gr < rows;
    float *ft = (fwd_trace && live) ? fwd_trace + gr * 3 * H + c0 : nullptr;
    float *bt = (bwd_trace && live) ? bwd_trace + gr * 4 * H + c0 : nullptr;
    // ---- forward
#pragma unroll
    for (int u = 0; u < kTrLoads; ++u) {
      const int e = tid + kTrT * u;
      if (e < TM * F) *(bf16 *)(x + tc::core_off(e / F, e % F, FPAD)) = __float2bfloat16_rn(v25[u]);
    }
    const float2 tg = live ? make_float2(__ldg(target + 2 * gr), __ldg(target + 2 * gr + 1)) : make_float2(0.f, 0.f);
    if (!(ok = tc_sync(ok))) break;
    if (issuer) { tc_gemm(tacc, sx, false, FPAD, kColStep, sw1, false, FPAD, kColStep, H, FPAD, false); tc::commit(mbar); }
    ok = ok && tc_wait(mbar, phase);
    uint32_t w[16], mask[3];
    auto positive = [&]() {  // bit j: column c0 + j of the rounded activation is positive
      uint32_t m = 0;
#pragma unroll
      for (int j = 0; j < 16; ++j)
        m |= ((w[j] & 0x7fffu) ? 1u << (2 * j) : 0u) | ((w[j] & 0x7fff0000u) ? 2u << (2 * j) : 0u);
      return m;
    };
    tc_hidden32(tacc + lanes + c0, fb + c0, w);
    tc_store32(h1, r, c0, HX, w);
    if (ft) trace32(ft, w);
    mask[0] = positive();
    if (!(ok = tc_sync(ok))) break;
    if (issuer) { tc_gemm(tacc, sh1, false, HX, kColStep, sw2, false, H, kColStep, H, H, false); tc::commit(mbar); }
    ok = ok && tc_wait(mbar, phase);
    tc_hidden32(tacc + lanes + c0, fb + H + c0, w);
    tc_store32(h2, r, c0, HX, w);
    if (ft) trace32(ft + H, w);
    mask[1] = positive();
    if (!(ok = tc_sync(ok))) break;
    if (issuer) { tc_gemm(tacc, sh2, false, HX, kColStep, sw3, false, H, kColStep, H, H, false); tc::commit(mbar); }
    ok = ok && tc_wait(mbar, phase);
    tc_hidden32(tacc + lanes + c0, fb + 2 * H + c0, w);
    tc_store32(h3, r, c0, H, w);
    if (ft) trace32(ft + 2 * H, w);
    mask[2] = positive();
    {
      float p0 = 0.f, p1 = 0.f;
      tc_out32(w, fb + 3 * H + 2 * c0, p0, p1);
      *(float2 *)(opart + 2 * (cq * TM + r)) = make_float2(p0, p1);
    }
    __syncthreads();
    // ---- output layer: dO of this row, rounded to bf16 (the same in the row's four threads)
    float o0 = fb[5 * H], o1 = fb[5 * H + 1];
    {
      const float2 a = *(float2 *)(opart + 2 * r), b = *(float2 *)(opart + 2 * (TM + r)),
                   c = *(float2 *)(opart + 2 * (2 * TM + r)), d = *(float2 *)(opart + 2 * (3 * TM + r));
      o0 += (a.x + b.x) + (c.x + d.x);
      o1 += (a.y + b.y) + (c.y + d.y);
    }
    const float d0 = live ? o0 - tg.x : 0.f, d1 = live ? o1 - tg.y : 0.f;
    const uint32_t gw = pack2f(d0 * scale, d1 * scale);
    const float g0 = lo2f(gw), g1 = hi2f(gw);
    if (cq == 0) {
      lsum += d0 * d0 + d1 * d1;
      sg0 += g0;
      sg1 += g1;
      *(uint32_t *)(dot + tc::core_off(r, 0, 16)) = gw;
      if (bt) {
        bt[3 * H] = g0;
        bt[3 * H + 1] = g1;
        bt[3 * H + 2] = o0;
        bt[3 * H + 3] = o1;
      }
    }
    // dZ3 of this row from dO and W4, masked by H3
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const float4 a = *(const float4 *)(fb + 3 * H + 2 * (c0 + 2 * j));
      const float za = (mask[2] >> (2 * j)) & 1u ? fmaf(g1, a.y, g0 * a.x) : 0.f;
      const float zb = (mask[2] >> (2 * j)) & 2u ? fmaf(g1, a.w, g0 * a.z) : 0.f;
      w[j] = pack2f(za, zb);
    }
    tc_store32(z, r, c0, H, w);
    if (bt) trace32(bt, w);
    if (!(ok = tc_sync(ok))) break;
    if (issuer) {
      tc_gemm(tacc, sz, false, H, kColStep, sw3, true, H, kStepH, H, H, false);
      tc_gemm(tacc + kTcW4, sh3, true, H, kStepH, sdo, true, 16, kStepO, 16, TM, !first);
      tc::commit(mbar);
      tc_gemm(tacc + kTcW3, sz, true, H, kStepH, sh2, true, HX, kStepHX, HX, TM, !first);
      tc::commit(mbar2);
    }
    ok = ok && tc_wait(mbar, phase);
    // dZ = dH o [layer > 0], 32 columns of this row
    auto back = [&](uint32_t m, unsigned char *t, float *tr) {
      float v[32];
      tc::ld32(tacc + lanes + c0, v);
#pragma unroll
      for (int j = 0; j < 16; ++j)
        w[j] = pack2f((m >> (2 * j)) & 1u ? v[2 * j] : 0.f, (m >> (2 * j)) & 2u ? v[2 * j + 1] : 0.f);
      tc_store32(t, r, c0, H, w);
      if (tr) trace32(tr, w);
    };
    back(mask[1], h3, bt ? bt + H : nullptr);  // dZ2 to H3's room: dW4 is done with it
    if (!(ok = tc_sync(ok))) break;
    if (issuer) {
      tc_gemm(tacc, sh3, false, H, kColStep, sw2, true, H, kStepH, H, H, false);
      tc::commit(mbar);
    }
    ok = ok && tc_wait(mbar2, phase2);  // dW3 is done with dZ3's room
    if (issuer) {
      tc_gemm(tacc + kTcW2, sh3, true, H, kStepH, sh1, true, HX, kStepHX, HX, TM, !first);
      tc::commit(mbar2);
    }
    if (tl + gridDim.x < tiles) load_tile(tl + gridDim.x);
    ok = ok && tc_wait(mbar, phase);
    back(mask[0], z, bt ? bt + 2 * H : nullptr);
    if (!(ok = tc_sync(ok))) break;
    if (issuer) {
      tc_gemm(tacc + kTcW1, sz, true, H, kStepH, sx, true, FPAD, kStepX, FPAD, TM, !first);
      tc::commit(mbar);
    }
    first = false;
    ok = ok && tc_wait(mbar2, phase2) && tc_wait(mbar, phase);
  }
  ok = !group_any(!ok, -1);  // the last tile's waits
  // ---- the block's partial gradient: row r of each, a quarter of the columns
  float *gp = part + (size_t)blockIdx.x * NPAR;
  const float nanv = __int_as_float(0x7fc00000);
  if (ok && !first) {
    float v[32];
    tc::ld32(tacc + kTcW3 + lanes + c0, v);
#pragma unroll
    for (int j = 0; j < 32; ++j) gp[OW3 + r * H + c0 + j] = v[j];
    tc::ld32(tacc + kTcW2 + lanes + c0, v);
#pragma unroll
    for (int j = 0; j < 32; ++j) gp[OW2 + r * H + c0 + j] = v[j];
    if (cq == 0) {
      tc::ld32(tacc + kTcW1 + lanes, v);
#pragma unroll
      for (int j = 0; j < F; ++j) gp[OW1 + r * F + j] = v[j];
      gp[OB1 + r] = v[F];
    } else if (cq == 1) {
      tc::ld32(tacc + kTcW3 + H + lanes, v);  // the ones column (the columns past 144 are not read further)
      gp[OB3 + r] = v[0];
    } else if (cq == 2) {
      tc::ld32(tacc + kTcW2 + H + lanes, v);
      gp[OB2 + r] = v[0];
    } else {
      tc::ld32(tacc + kTcW4 + lanes, v);
      gp[OW4 + r] = v[0];
      gp[OW4 + H + r] = v[1];
    }
  } else {
    const float fill = ok ? 0.f : nanv;  // a block without tiles adds nothing
    for (int u = tid; u < OB4; u += kTrT) gp[u] = fill;
  }
  // loss and output bias: the sums of the first 128 threads' rows
  __syncthreads();
  if (tid < TM) {
    lsum = warp_sum(lsum);
    sg0 = warp_sum(sg0);
    sg1 = warp_sum(sg1);
    if ((tid & 31) == 0) {
      opart[tid >> 5] = lsum;
      opart[4 + (tid >> 5)] = sg0;
      opart[8 + (tid >> 5)] = sg1;
    }
  }
  tc::fence_before();
  __syncthreads();
  if (tid < 3) {
    const float t = (opart[4 * tid] + opart[4 * tid + 1]) + (opart[4 * tid + 2] + opart[4 * tid + 3]);
    if (tid == 0) loss_part[blockIdx.x] = ok ? t : nanv;
    else gp[OB4 + tid - 1] = ok ? t : nanv;
  }
  if (tid < 32) {
    tc::fence_after();
    tc::tmem_free<512>(tacc);
  }
}

// grad[p] = sum over blocks of part[b][p]; loss = sum of the blocks' losses / rows.  Four threads per
// parameter, each a quarter of the blocks with eight loads in flight (one thread and one chain per
// parameter took 13.4 us for 152 partials of 36 610 values).
constexpr int kRedP = 64;
__global__ void __launch_bounds__(4 * kRedP) grad_reduce_kernel(const float *__restrict__ part, int nb, float *grad,
                                                                const float *__restrict__ lp, int64_t rows, float *loss) {
  __shared__ float sh[4][kRedP];
  const int t = threadIdx.x % kRedP, w = threadIdx.x / kRedP, p = blockIdx.x * kRedP + t;
  float s = 0.f;
  if (p < NPAR) {
#pragma unroll 8
    for (int b = w; b < nb; b += 4) s += part[(size_t)b * NPAR + p];
  }
  sh[w][t] = s;
  __syncthreads();
  if (w == 0 && p < NPAR) grad[p] = (sh[0][t] + sh[1][t]) + (sh[2][t] + sh[3][t]);
  if (blockIdx.x == 0 && threadIdx.x >= 32 && threadIdx.x < 64 && loss) {
    float l = 0.f;
    for (int b = threadIdx.x - 32; b < nb; b += 32) l += lp[b];
    l = warp_sum(l);
    if (threadIdx.x == 32) *loss = l / (float)rows;
  }
}

// bf16 padded index of parameter p (-1 for biases)
__device__ __forceinline__ int bf_index(int p) {
  if (p < OB1) return BW1 + (p / F) * S1 + (p % F);
  if (p >= OW2 && p < OB2) return BW2 + ((p - OW2) / H) * SA + (p - OW2) % H;
  if (p >= OW3 && p < OB3) return BW3 + ((p - OW3) / H) * SA + (p - OW3) % H;
  if (p >= OW4 && p < OB4) return BW4 + ((p - OW4) / H) * SA + (p - OW4) % H;
  return -1;
}

// Adam (Kingma & Ba): m = b1 m + (1-b1) g, v = b2 v + (1-b2) g^2, p -= lr mhat / (sqrt(vhat) + eps)
__global__ void adam_kernel(float *params, float *m, float *v, const float *__restrict__ grad, bf16 *wb, float lr,
                            float b1c, float b2c) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= NPAR) return;
  const float g = grad[p];
  const float mm = 0.9f * m[p] + 0.1f * g;
  const float vv = 0.999f * v[p] + 0.001f * g * g;
  m[p] = mm;
  v[p] = vv;
  const float w = params[p] - lr * (mm / b1c) / (sqrtf(vv / b2c) + 1e-8f);
  params[p] = w;
  const int bi = bf_index(p);
  if (bi >= 0) wb[bi] = __float2bfloat16_rn(w);
}

__global__ void sync_bf16_kernel(const float *__restrict__ params, bf16 *wb) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= NPAR) return;
  const int bi = bf_index(p);
  if (bi >= 0) wb[bi] = __float2bfloat16_rn(params[p]);
}

// He-uniform initial weights from Philox4x32-10 (key = seed, counter = (p, 0, 0, 1)), zero biases
__global__ void init_params_kernel(float *params, uint64_t seed) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= NPAR) return;
  int fan = 0;
  if (p < OB1) fan = F;
  else if ((p >= OW2 && p < OB2) || (p >= OW3 && p < OB3) || (p >= OW4 && p < OB4)) fan = H;
  float w = 0.f;
  if (fan > 0) {
    const uint4 r = philox4x32_10(make_uint4((uint32_t)p, 0u, 0u, 1u), make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
    const float u = (float)(r.x >> 8) * (1.0f / 16777216.0f);
    const float a = sqrtf(6.0f / (float)fan);
    w = (2.f * u - 1.f) * a;
    if (p >= OW4 && p < OB4) w *= 0.1f;  // small output layer: the first proposals stay small
  }
  params[p] = w;
}

// ------------------------------------------------------------------------------ warm start ----
// x += clip(du e_r + dv e_t, max_move) per circle; the old coordinates go to backup
__global__ void apply_kernel(StandaloneParams P, const float *__restrict__ dout, float2 *backup, float max_move) {
  const int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= P.total) return;
  const float2 x = P.x32[gi];
  backup[gi] = x;
  const float2 er = frame_er(x);
  const float du = dout[2 * gi], dv = dout[2 * gi + 1];
  float dx = du * er.x - dv * er.y, dy = du * er.y + dv * er.x;
  const float nrm = sqrtf(dx * dx + dy * dy);
  if (nrm > max_move) { dx *= max_move / nrm; dy *= max_move / nrm; }
  if (!isfinite(dx) || !isfinite(dy)) { dx = 0.f; dy = 0.f; }
  const float2 nx = make_float2(x.x + dx, x.y + dy);
  P.x32[gi] = nx;
  P.x64[gi] = make_double2((double)nx.x, (double)nx.y);
}

// keep the move of an instance only if its energy did not rise; accepted[q] counts kept rounds
__global__ void revert_kernel(StandaloneParams P, const float2 *__restrict__ backup, const double *__restrict__ Eb,
                              const double *__restrict__ Ea, int32_t *accepted) {
  const int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= P.total) return;
  const int q = P.inst_of[gi];
  const bool keep = Ea[q] <= Eb[q];
  if (!keep) {
    const float2 x = backup[gi];
    P.x32[gi] = x;
    P.x64[gi] = make_double2((double)x.x, (double)x.y);
  }
  if (accepted && gi == P.desc[q].off) accepted[q] += keep ? 1 : 0;
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// Self-test of that wait: a warp waits for a barrier that another opens after open_after_ns; the lanes of
// short_lanes give up at once, the others a second later than that.  *yes: the lanes whose answer was yes.
__global__ void wait_selftest_kernel(long long open_after_ns, uint32_t short_lanes, int *yes) {
  __shared__ uint64_t mbar;
  if (threadIdx.x == 0) tc::mbar_init(&mbar);
  __syncthreads();
  if (threadIdx.x == 32) {
    const long long t0 = tc::now_ns();
    while (tc::now_ns() - t0 < open_after_ns) __nanosleep(1000);
    tc::mbar_arrive(&mbar);
  }
  if (threadIdx.x >= 32) return;
  const bool give_up = (short_lanes >> threadIdx.x) & 1u;
  const bool ok = tc::mbar_wait_warp(&mbar, 0, give_up ? 0 : open_after_ns + 1000000000ll);
  atomicAdd(yes, ok ? 1 : 0);
}

cudaError_t selftest_mma_wait(long long open_after_ns, uint32_t short_lanes, int *yes_host) {
  int *yes = nullptr;
  cudaError_t e = cudaMalloc(&yes, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(yes, 0, sizeof(int));
  if (e == cudaSuccess) {
    wait_selftest_kernel<<<1, 64>>>(open_after_ns, short_lanes, yes);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(yes_host, yes, sizeof(int), cudaMemcpyDeviceToHost);
  cudaFree(yes);
  return e;
}

int mlp_num_params() { return NPAR; }
int mlp_num_bf16() { return NBW; }

cudaError_t mlp_init(float *params, bf16 *wb, uint64_t seed, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(wb, 0, sizeof(bf16) * NBW, s);
  if (e) return e;
  init_params_kernel<<<nblk(NPAR, 256), 256, 0, s>>>(params, seed);
  sync_bf16_kernel<<<nblk(NPAR, 256), 256, 0, s>>>(params, wb);
  return cudaGetLastError();
}

cudaError_t mlp_sync_bf16(const float *params, bf16 *wb, cudaStream_t s) {
  sync_bf16_kernel<<<nblk(NPAR, 256), 256, 0, s>>>(params, wb);
  return cudaGetLastError();
}

cudaError_t features_smem_limit(int n_small) {
  return raise_smem_limit((const void *)features_block_kernel,
                          cells_smem(std::max(n_small, 0), 8 * (size_t)kKnnWarpBytes, false));
}

cudaError_t mlp_features(const StandaloneParams &p, const LargeTiles &L, int n_small, float *feat, cudaStream_t s) {
  if (p.num <= 0) return cudaSuccess;
  if (n_small >= 0) {
    const int block = n_small <= 64 ? 64 : (n_small <= 128 ? 128 : 256);
    const size_t smem = cells_smem(n_small, (size_t)(block / 32) * kKnnWarpBytes, false);
    features_block_kernel<<<p.num, block, smem, s>>>(p, knn_reach(p.l_cut), feat);
  }
  if (L.nrows > 0) {
    cudaError_t e = launch_large_cells32(p, L, s);
    if (e != cudaSuccess) return e;
    features_tile_kernel<<<L.nrows, kTileRows, 0, s>>>(p, L, knn_reach(p.l_cut), feat);
  }
  return cudaGetLastError();
}

cudaError_t mlp_targets(const StandaloneParams &p, const double *xbefore, float *target, cudaStream_t s) {
  if (p.total > 0) targets_kernel<<<nblk(p.total, 256), 256, 0, s>>>(p, xbefore, target);
  return cudaGetLastError();
}

cudaError_t mlp_forward(const bf16 *wb, const float *params, const float *feat, int64_t rows, float *out, int sms,
                        cudaStream_t s, float *trace) {
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(forward_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFwdSmem);
    if (e) return e;
    attr = true;
  }
  if (rows <= 0) return cudaSuccess;
  const int64_t tiles = (rows + TM - 1) / TM;
  const int grid = (int)std::min<int64_t>(tiles, (int64_t)sms);
  forward_tc_kernel<<<grid, TM * kFwdGroups, kFwdSmem, s>>>(wb, params, feat, rows, out, trace);
  return cudaGetLastError();
}

int mlp_train_blocks(int sms) { return sms; }

cudaError_t mlp_grad(const bf16 *wb, const float *params, const float *feat, const float *target, int64_t rows,
                     float *part, float *lpart, float *grad, float *loss, int sms, cudaStream_t s, float *fwd_trace,
                     float *bwd_trace) {
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(train_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTrainSmem);
    if (e) return e;
    attr = true;
  }
  const int nb = (int)std::min<int64_t>((rows + TM - 1) / TM, (int64_t)mlp_train_blocks(sms));
  train_tc_kernel<<<nb, kTrT, kTrainSmem, s>>>(wb, params, feat, target, rows, part, lpart, fwd_trace, bwd_trace);
  grad_reduce_kernel<<<nblk(NPAR, kRedP), 4 * kRedP, 0, s>>>(part, nb, grad, lpart, rows, loss);
  return cudaGetLastError();
}

cudaError_t mlp_adam(float *params, float *m, float *v, const float *grad, bf16 *wb, float lr, int step,
                     cudaStream_t s) {
  const float b1c = 1.f - powf(0.9f, (float)step), b2c = 1.f - powf(0.999f, (float)step);
  adam_kernel<<<nblk(NPAR, 256), 256, 0, s>>>(params, m, v, grad, wb, lr, b1c, b2c);
  return cudaGetLastError();
}

cudaError_t mlp_apply(const StandaloneParams &p, const float *dout, float2 *backup, float max_move, cudaStream_t s) {
  if (p.total > 0) apply_kernel<<<nblk(p.total, 256), 256, 0, s>>>(p, dout, backup, max_move);
  return cudaGetLastError();
}

cudaError_t mlp_revert(const StandaloneParams &p, const float2 *backup, const double *Eb, const double *Ea,
                       int32_t *accepted, cudaStream_t s) {
  if (p.total > 0) revert_kernel<<<nblk(p.total, 256), 256, 0, s>>>(p, backup, Eb, Ea, accepted);
  return cudaGetLastError();
}

}  // namespace pecc
