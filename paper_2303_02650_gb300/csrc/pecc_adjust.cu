// pecc_adjust.cu -- container adjustment (Sec. 4.2, Algorithm adjust_container, Eq. 12) on the GPU.
//
// z = (x, R) and U(z, lambda) = E(x, R) + lambda R^2.  For each of `rounds` rounds a limited-memory
// BFGS minimises U over all of z (one batch; a fresh memory each round), then lambda is halved.
// dU/dx is the gradient of E; dU/dR = -2 sum_i d_i0 + 2 lambda R.  One thread block per instance
// (persistent over a work queue), the two-loop recursion written out over the stored pairs (each
// dot product one block reduction in a fixed order: deterministic).  The lists are maintained as
// in the descent: a cell-list build, the Verlet rule before a step and ANM after each iteration.
// Two arithmetic forms:
//   <Arith64, double>  binary64 throughout (the binary64 contexts);
//   <ArithMix, float>  the descent's polish arithmetic for the pair and wall terms (binary64
//                      coordinates, differences and the near-contact quantities 4 - l^2 and
//                      |c|^2 - (R - 1)^2, binary32 depths and forces), binary32 gradients and
//                      quasi-Newton vectors, binary64 energy sums and everything about R.
// GB300 issues few binary64 operations per clock; in the binary64 form the pair terms and the
// two-loop recursion keep that pipe about 80 % busy.  The binary32 depths put a relative jitter of
// about 1e-7 on E, so the Armijo test on U resolves U's minimum only to about 1e-6 of R while E is
// large (a large lambda); the schedule's late rounds, where the radius is settled, have E near 0.
#include "pecc_internal.h"

namespace pecc {

namespace {

constexpr int kAdjT = 256;  // threads per instance block
constexpr int kAdjW = kAdjT / 32;
constexpr int kAdjM = kMaxSlots - 1;  // memory pairs at most

struct AdjSmem {
  double val[4][kAdjT + 4 * kAdjW];  // one value per thread and reduction slot, four words between warps' rows
  double tot[4];
  double qR;                                 // the radius's component of the two-loop's vector
  double coef;                               // and the coefficient of its current step
  double sR[kAdjM], yR[kAdjM], rho[kAdjM], yy[kAdjM], alpha[kAdjM];
  int32_t sh[40];
  unsigned long long hash;
  int q;
};

// The butterfly over each warp's 32 values of S.val[q] (distances 16, 8, 4, 2, 1), then the warps in
// order; the result in every lane of the calling warp.  A lane takes eight values of one warp, so the
// first three stages are its own additions and the eight butterflies share the warp's instructions: 16
// binary64 additions per value instead of 47, with two binary64 lanes per SM and clock.
template <bool MAX> __device__ __forceinline__ double block_combine(const AdjSmem &S, int q) {
  const int lane = threadIdx.x & 31;
  auto op = [](double a, double b) { return MAX ? fmax(a, b) : a + b; };
  const double *x = S.val[q] + 36 * (lane >> 2) + (lane & 3);
  double t[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) t[m] = x[4 * m];
#pragma unroll
  for (int o = 4; o > 0; o >>= 1)
#pragma unroll
    for (int m = 0; m < o; ++m) t[m] = op(t[m], t[m + o]);
  double a = t[0];
  a = op(a, __shfl_xor_sync(0xffffffffu, a, 2));
  a = op(a, __shfl_xor_sync(0xffffffffu, a, 1));
  double s = __shfl_sync(0xffffffffu, a, 0);
#pragma unroll
  for (int u = 1; u < kAdjW; ++u) s = op(s, __shfl_sync(0xffffffffu, a, 4 * u));
  return s;
}

// Block reduction of NV values (sum, or max where mx[q]); every thread gets the totals in v.  A thread
// leaves its values in shared memory, and warp q combines value q.
template <int NV>
__device__ __forceinline__ void bred(AdjSmem &S, double (&v)[NV], const bool (&mx)[NV]) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
#pragma unroll
  for (int q = 0; q < NV; ++q) S.val[q][tid + 4 * w] = v[q];
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    if (w != q) continue;
    const double s = mx[q] ? block_combine<true>(S, q) : block_combine<false>(S, q);
    if (lane == 0) S.tot[q] = s;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NV; ++q) v[q] = S.tot[q];
}

// Block sum of v, with which one thread forms the scalars of a two-loop step (fin): formed by every
// thread they were eight times the binary64 instructions.
template <class F> __device__ __forceinline__ void sum_then(AdjSmem &S, double v, F fin) {
  const int tid = threadIdx.x, w = tid >> 5;
  S.val[0][tid + 4 * w] = v;
  __syncthreads();
  if (w == 0) {
    const double s = block_combine<false>(S, 0);
    if (tid == 0) fin(s);
  }
  __syncthreads();
}

constexpr int kAdjOwn = 4;  // circles of a thread that the two-loop keeps in registers (n <= 1024)

// Two-loop recursion (Nocedal & Wright, Alg. 7.4) over the stored pairs from q = (g, gR): d = -q into dv,
// and this thread's parts of g'd and of the largest move.  S.qR: q's radius component in and out.
// OWN: the vector stays in the threads' registers, and each pair's vectors are loaded a step ahead, behind
// the reduction of the step before; else (n > 1024) everything goes through memory.
template <bool OWN, typename VT, typename GT>
__device__ __forceinline__ void two_loop(AdjSmem &S, int n, int m, int head, int count, const v2<GT> *g, v2<VT> *dv,
                                         const v2<VT> *Sv, const v2<VT> *Yv, GT &gd, VT &dm) {
  using V2 = v2<VT>;
  const int tid = threadIdx.x, T = kAdjT;
  V2 d[kAdjOwn], a0[kAdjOwn], a1[kAdjOwn], a2[kAdjOwn];
  auto slot = [&](const V2 *B, int c) { return B + (int64_t)((head + c) % m) * n; };
  auto load = [&](V2 (&a)[kAdjOwn], const V2 *p) {
#pragma unroll
    for (int u = 0; u < kAdjOwn; ++u) {
      const int i = tid + u * T;
      if (i < n) a[u] = p[i];
    }
  };
  // f(vector element, circle) for this thread's circles in order
  auto each = [&](auto f) {
    if constexpr (OWN) {
#pragma unroll
      for (int u = 0; u < kAdjOwn; ++u) {
        const int i = tid + u * T;
        if (i < n) f(d[u], i, u);
      }
    } else {
      for (int i = tid; i < n; i += T) {
        V2 b = dv[i];
        f(b, i, 0);
        dv[i] = b;
      }
    }
  };
  // the same without a change of the vector
  auto look = [&](auto f) {
    if constexpr (OWN) {
#pragma unroll
      for (int u = 0; u < kAdjOwn; ++u) {
        const int i = tid + u * T;
        if (i < n) f(d[u], i, u);
      }
    } else {
      for (int i = tid; i < n; i += T) f(dv[i], i, 0);
    }
  };
  each([&](V2 &b, int i, int) { const v2<GT> gi = g[i]; b = mk2<VT>((VT)gi.x, (VT)gi.y); });
  if (OWN && count > 0) load(a0, slot(Sv, count - 1));
  for (int c = count - 1; c >= 0; --c) {
    const int sl = (head + c) % m;
    const V2 *s_ = Sv + (int64_t)sl * n, *y_ = Yv + (int64_t)sl * n;
    if (OWN) {
      load(a1, y_);
      if (c > 0) load(a2, slot(Sv, c - 1));
    }
    VT pv = 0;
    look([&](const V2 &b, int i, int u) {
      const V2 a = OWN ? a0[u] : s_[i];
      pv += a.x * b.x + a.y * b.y;
    });
    sum_then(S, (double)pv, [&](double t) {
      const double a = S.rho[sl] * (t + S.sR[sl] * S.qR);
      S.alpha[c] = a;
      S.coef = a;
      S.qR -= a * S.yR[sl];
    });
    const VT av = (VT)S.coef;
    each([&](V2 &b, int i, int u) {
      const V2 yv = OWN ? a1[u] : y_[i];
      b.x -= av * yv.x;
      b.y -= av * yv.y;
    });
    if (OWN) {
#pragma unroll
      for (int u = 0; u < kAdjOwn; ++u) a0[u] = a2[u];
    }
  }
  if (count > 0) {
    const int nw_ = (head + count - 1) % m;
    if (OWN) load(a0, slot(Yv, 0));
    __syncthreads();  // the last coefficient has been read
    if (tid == 0) {
      const double gam = 1.0 / (S.rho[nw_] * S.yy[nw_]);  // s'y / y'y of the newest pair
      S.coef = gam;
      S.qR *= gam;
    }
    __syncthreads();
    const VT gv = (VT)S.coef;
    each([&](V2 &b, int, int) { b.x *= gv; b.y *= gv; });
  }
  for (int c = 0; c < count; ++c) {
    const int sl = (head + c) % m;
    const V2 *s_ = Sv + (int64_t)sl * n, *y_ = Yv + (int64_t)sl * n;
    if (OWN) {
      load(a1, s_);
      if (c + 1 < count) load(a2, slot(Yv, c + 1));
    }
    VT pv = 0;
    look([&](const V2 &b, int i, int u) {
      const V2 a = OWN ? a0[u] : y_[i];
      pv += a.x * b.x + a.y * b.y;
    });
    sum_then(S, (double)pv, [&](double t) {
      const double bta = S.rho[sl] * (t + S.yR[sl] * S.qR);
      const double w = S.alpha[c] - bta;
      S.coef = w;
      S.qR += w * S.sR[sl];
    });
    const VT wv = (VT)S.coef;
    each([&](V2 &b, int i, int u) {
      const V2 sa = OWN ? a1[u] : s_[i];
      b.x += wv * sa.x;
      b.y += wv * sa.y;
    });
    if (OWN) {
#pragma unroll
      for (int u = 0; u < kAdjOwn; ++u) a0[u] = a2[u];
    }
  }
  // d = -q; g'd and the largest move
  each([&](V2 &b, int i, int) {
    b.x = -b.x;
    b.y = -b.y;
    if (OWN) dv[i] = b;
    const v2<GT> gi = g[i];
    gd += gi.x * (GT)b.x + gi.y * (GT)b.y;
    dm = max(dm, b.x * b.x + b.y * b.y);
  });
}

template <class A, typename VT>
__global__ void __launch_bounds__(kAdjT, 2) adjust_kernel(AdjustParams P) {
  using V2 = v2<VT>;
  using GT = typename A::vec_t;  // the forces' and the stored gradient's type
  using GV2 = v2<GT>;
  __shared__ AdjSmem S;
  const int tid = threadIdx.x, T = blockDim.x;
  const double lc2 = P.l_cut * P.l_cut;
  for (;;) {
    if (tid == 0) S.q = atomicAdd(P.queue, 1);
    __syncthreads();
    const int q = S.q;
    __syncthreads();
    if (q >= P.num) break;
    const InstDesc D = P.desc[q];
    const int n = D.n;
    double R = P.R[q];
    double2 *x = P.x64 + D.off;
    if (n == 0 || D.big) {
      if (tid == 0) {
        P.iters[q] = 0; P.status[q] = n == 0 ? 0 : 4;
        if (P.stats) { P.stats[2 * q] = 0; P.stats[2 * q + 1] = 0; }
      }
      __syncthreads();
      continue;
    }
    if (P.from32)
      for (int i = tid; i < n; i += T) { const float2 f = P.x32[D.off + i]; x[i] = make_double2(f.x, f.y); }
    // gradients in the forces' type, the direction and the pairs in VT (the buffers are sized for
    // double2)
    GV2 *g = (GV2 *)(P.g + D.off), *gn = (GV2 *)(P.gn + D.off);
    V2 *dv = (V2 *)(P.d + D.off), *sv = (V2 *)(P.sv + D.off);
    double2 *zo = P.zo + D.off, *xb = P.xb + D.off, *xs = P.xs + D.off;
    V2 *Sv = (V2 *)(P.S + (int64_t)kAdjM * D.off), *Yv = (V2 *)(P.Y + (int64_t)kAdjM * D.off);
    int32_t *rp = P.rp + D.rp_off, *col = P.col + D.col_off;
    const int cap = 2 * D.cap;
    const CellGrid G{D.R, D.inv_cs, 0.f, 0.f, D.ncx, false};
    uint32_t *ckey = P.ckey + D.off;
    int32_t *corder = P.corder + D.off, *cells = P.cells + D.cell_off;

    int status = 3, iters = 0, cnt = 0, len = 1, trials = 0, visits = 0;
    unsigned long long hcur = 0ull;
    double Dmax = 0.0;
    // list build with ANM bookkeeping; false on a capacity overflow
    auto rebuild = [&](bool anm) -> bool {
      const int tot = cta_build_neighbors<double, int32_t>(x, n, G, lc2, ckey, corder, cells, xs, rp, col, cap, S.sh,
                                                          &S.hash);
      if (tot > cap) return false;
      if (anm) {
        const unsigned long long h = S.hash;
        if (h != hcur) { hcur = h; len = 1; }
        else if (len < (1 << 30)) len *= 2;
        cnt = 0;
      } else {
        hcur = S.hash;
      }
      for (int i = tid; i < n; i += T) xb[i] = x[i];
      Dmax = 0.0;
      __syncthreads();
      return true;
    };
    // U, its gradient over x into gout with its squared norm g2, and dU/dR, at the current x and radius Rz
    auto eval = [&](GV2 *gout, double Rz, double lam, double &U, double &gR, double &g2) {
      const double Rm1sq = (Rz >= 1.0) ? (Rz - 1.0) * (Rz - 1.0) : -1.0;
      double v[3] = {0.0, 0.0, 0.0};
      const bool mx[3] = {false, false, false};
      GT p1 = 0;
      for (int i = tid; i < n; i += T) {
        const double2 xi = x[i];
        GT gx = 0, gy = 0;
        double e = 0.0;
        // two entries per step (both coordinate loads in flight); the sums take the entries in row order
        const int t1 = rp[i + 1];
        for (int t = rp[i]; t < t1; t += 2) {
          const bool two = t + 1 < t1;
          const int j1 = col[t];
          const int j2 = two ? col[t + 1] : j1;
          const double2 x1 = x[j1], x2 = x[j2];
          GT fx, fy;
          const double d1 = A::pair(xi, x1, fx, fy);
          gx += fx; gy += fy;
          if (j1 < i) e += d1 * d1;
          if (two) {
            const double d2 = A::pair(xi, x2, fx, fy);
            gx += fx; gy += fy;
            if (j2 < i) e += d2 * d2;
          }
        }
        GT fx, fy;
        const double d0 = A::wall(xi, Rz, Rm1sq, fx, fy);
        gx += fx; gy += fy;
        v[0] += e + d0 * d0;
        v[1] += d0;
        gout[i] = mk2<GT>(gx, gy);
        p1 += gx * gx + gy * gy;
      }
      v[2] = (double)p1;
      bred<3>(S, v, mx);
      g2 = v[2];
      U = v[0] + lam * Rz * Rz;
      gR = -2.0 * v[1] + 2.0 * lam * Rz;
    };

    bool ok = rebuild(false);
    if (!ok) status = 4;
    double lam = P.lambda0;
    for (int round = 0; round < P.rounds && ok; ++round) {
      int head = 0, count = 0;
      double U0, gR, g2;
      eval(g, R, lam, U0, gR, g2);
      status = 3;
      for (int it = 0; it < P.max_iter; ++it) {
        if (2.0 * Dmax + P.step_max > 2.0 * P.rebuild_disp) {
          if (!rebuild(true)) { ok = false; status = 4; break; }
        }
        ++iters;
        const double gg = g2 + gR * gR, gnorm = sqrt(gg);
        if (!(gnorm > P.gsum_tol)) { status = 1; break; }
        for (int i = tid; i < n; i += T) zo[i] = x[i];
        const double Ro = R;
        bool accepted = false;
        double Ut = U0, gnR = gR, gn2 = g2;
        for (int attempt = 0; attempt < 2 && !accepted; ++attempt) {
          if (attempt == 1) {
            if (count == 0) break;
            count = 0;
            head = 0;
          }
          visits += count;
          if (tid == 0) S.qR = gR;  // read by thread 0 alone until the steps below are done
          const bool mx2[2] = {false, true};
          GT p2 = 0;
          VT m2 = 0;
          // binary64 vectors would take the registers of a block per SM
          if (sizeof(VT) == 4 && n <= kAdjOwn * kAdjT) two_loop<sizeof(VT) == 4, VT, GT>(S, n, P.m, head, count, g, dv, Sv, Yv, p2, m2);
          else two_loop<false, VT, GT>(S, n, P.m, head, count, g, dv, Sv, Yv, p2, m2);
          double v2[2] = {(double)p2, (double)m2};
          bred<2>(S, v2, mx2);
          double dR = -S.qR;
          double gd = v2[0] + gR * dR;
          double dmax = sqrt(fmax(v2[1], dR * dR));
          if (!(gd < 0.0)) {  // not a descent direction: drop the memory, take -g
            count = 0;
            head = 0;
            GT m3 = 0;
            for (int i = tid; i < n; i += T) {
              const GV2 gi = g[i];
              dv[i] = mk2<VT>((VT)-gi.x, (VT)-gi.y);
              m3 = max(m3, gi.x * gi.x + gi.y * gi.y);
            }
            double v3[1] = {(double)m3};
            const bool mx3[1] = {true};
            bred<1>(S, v3, mx3);
            dR = -gR;
            gd = -gg;
            dmax = sqrt(fmax(v3[0], dR * dR));
          }
          double al = (dmax > P.step_max) ? P.step_max / dmax : 1.0;
          for (int tr = 0; tr < P.max_trials; ++tr) {
            for (int i = tid; i < n; i += T) {
              const double2 a = zo[i];
              const V2 b = dv[i];
              x[i] = make_double2(a.x + al * (double)b.x, a.y + al * (double)b.y);
            }
            R = Ro + al * dR;
            __syncthreads();
            ++trials;
            eval(gn, R, lam, Ut, gnR, gn2);
            if (Ut <= U0 + P.c1 * al * gd) { accepted = true; break; }
            al *= 0.5;
          }
          if (!accepted) {
            for (int i = tid; i < n; i += T) x[i] = zo[i];
            R = Ro;
            __syncthreads();
          }
        }
        if (!accepted) { status = 2; break; }
        // ---- the secant pair: s into sv, y into dv (the new gradient is gn); displacement
        const bool mx4[4] = {false, false, false, true};
        VT p40 = 0, p41 = 0, p42 = 0;
        double m43 = 0.0;
        for (int i = tid; i < n; i += T) {
          const double2 xn = x[i], x0 = zo[i], b0 = xb[i];
          const GV2 gnew = gn[i], gold = g[i];
          const V2 s_ = mk2<VT>((VT)(xn.x - x0.x), (VT)(xn.y - x0.y));
          const V2 y_ = mk2<VT>((VT)(gnew.x - gold.x), (VT)(gnew.y - gold.y));
          sv[i] = s_;
          dv[i] = y_;
          p40 += s_.x * y_.x + s_.y * y_.y;
          p41 += s_.x * s_.x + s_.y * s_.y;
          p42 += y_.x * y_.x + y_.y * y_.y;
          const double ex = xn.x - b0.x, ey = xn.y - b0.y;
          m43 = fmax(m43, ex * ex + ey * ey);
        }
        double v4[4] = {(double)p40, (double)p41, (double)p42, m43};
        bred<4>(S, v4, mx4);
        const double sR = R - Ro, yR = gnR - gR;
        const double sy = v4[0] + sR * yR, ss = v4[1] + sR * sR, yy = v4[2] + yR * yR;
        Dmax = fmax(Dmax, sqrt(v4[3]));
        if (P.m > 0 && sy > P.curv_eps * sqrt(ss) * sqrt(yy)) {
          int sl;
          if (count < P.m) { sl = (head + count) % P.m; ++count; }
          else { sl = head; head = (head + 1) % P.m; }
          V2 *s_ = Sv + (int64_t)sl * n, *y_ = Yv + (int64_t)sl * n;
          for (int i = tid; i < n; i += T) { s_[i] = sv[i]; y_[i] = dv[i]; }
          if (tid == 0) { S.sR[sl] = sR; S.yR[sl] = yR; S.rho[sl] = 1.0 / sy; S.yy[sl] = yy; }
        }
        { GV2 *t_ = g; g = gn; gn = t_; }  // the trial's gradient is the next iteration's
        U0 = Ut;
        gR = gnR;
        g2 = gn2;
        __syncthreads();
        if (P.anm) {
          ++cnt;
          if (cnt >= len && !rebuild(true)) { ok = false; status = 4; break; }
        }
      }
      lam *= 0.5;
    }
    // the adjusted layout: binary64 and its binary32 copy
    for (int i = tid; i < n; i += T) {
      const double2 v = x[i];
      if (P.x32) P.x32[D.off + i] = make_float2((float)v.x, (float)v.y);
    }
    if (tid == 0) {
      P.R[q] = R; P.iters[q] = iters; P.status[q] = status;
      if (P.stats) { P.stats[2 * q] = trials; P.stats[2 * q + 1] = visits; }
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_adjust(const AdjustParams &p, int mixed, int grid, cudaStream_t s) {
  if (p.num <= 0 || grid <= 0) return cudaSuccess;
  if (mixed) adjust_kernel<ArithMix, float><<<grid, kAdjT, 0, s>>>(p);
  else adjust_kernel<Arith64, double><<<grid, kAdjT, 0, s>>>(p);
  return cudaGetLastError();
}

int adjust_max_m() { return kAdjM; }

}  // namespace pecc
