// The register-resident level-0 Krylov solves: one cooperative launch runs a whole pipelined CG (Picard steps, FP64 or
// FP32) or BiCGStab (Newton steps) whose cells' state stays in registers and whose matrix rows stay in shared memory
// (see psync.cuh for the grid synchronisation; larger meshes run the memory-resident kernels of persist.cu).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "kernels.cuh"
#include "persist.cuh"
#include "psync.cuh"

namespace nlmg {

namespace {

// Warps that hold cells at most; one more, the server, adds up the sums (with 11 warps and more cells each, and with it
// 168 registers a thread instead of 128, an iteration on 48^3 cells took 6.7 us instead of 5.7).
constexpr int kFWarps = 15;
constexpr int kFThreads = 32 * (kFWarps + 1);
constexpr size_t kFDyn = 218 * 1024;             // shared memory for the rows at most

// The cells of a thread: a block takes an equal run of consecutive slices of 32 cells (the SELL slices; equal within one,
// where a thread with a stride of the whole grid held up to 19% more on some SMs: an SM's FP64 issue, 19 clocks per warp
// operation, bounds the large meshes), its warps take the run's slices in turn. Consecutive cells are mostly each
// other's neighbours, so a block also keeps its own cells' values of the vector it multiplies in shared memory (xl) and
// gathers only the others' through L2: with every gather through L2 the product of 64^3 cells took 14.5k clocks, twice
// its FP64 issue. The rows are copied once into shared memory, entry j of slice u of a warp at 32 (off + j) + lane, with
// the column's index in xl, or the complement of its cell. Rows that do not fit (ST false: unstructured meshes, small
// shares of the SMs) are read from memory by the FP32 CG and the BiCGStab; the FP64 CG then runs the memory-resident
// kernel, whose full blocks hide the reads better (microseconds an iteration of a Voronoi mesh, streamed and in memory:
// FP64 85,184 cells 15.5 and 12.7, on 38 SMs 34.6 and 16.7; FP32 on 76 SMs 8.1 and 12.2; BiCGStab 27.7 and 30.4). A choice
// per load instead of per kernel cost both: 20.8 and 53.9 (FP64), 18.4 (FP32), 42.1 (BiCGStab) for the same, and 10.9
// instead of 10.0 on 64^3 cells in shared memory.
template <int R, class T, bool ST>
struct FRows {
  int K[R];        // cell (< 0: none)
  int n[R];        // entries of its slice
  int off[R];      // shared memory: first entry / 32; memory: first entry of the row
  int K0;          // first cell of the block
  const T* v;
  const int* c;
  T* xl;           // the block's own values
  static constexpr bool staged = ST;
};

template <int R, class T, bool ST>
__device__ __forceinline__ void rows_init(FRows<R, T, ST>& X, const FineDev& F, int nw) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int s0 = (int)((long long)F.nslice * blockIdx.x / gridDim.x);
  const int s1 = (int)((long long)F.nslice * (blockIdx.x + 1) / gridDim.x);
  X.K0 = 32 * s0;
#pragma unroll
  for (int u = 0; u < R; ++u) {
    const int s = s0 + warp + nw * u, K = 32 * s + lane;
    const bool in = warp < nw && s < s1;
    X.K[u] = in && K < F.N ? K : -1;
    X.n[u] = in ? F.sell_w[s] : 0;
    X.off[u] = in ? F.sell_off[s] + lane : 0;
  }
}

// Copies the rows into shared memory, entries scaled by S_K S_L; every thread reads back only what it wrote.
template <int R, class T, bool ST>
__device__ __forceinline__ void rows_stage(FRows<R, T, ST>& X, const FineDev& F, const double* __restrict__ A,
                                           const double* __restrict__ S, T* dv, int* dc, int nw) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int own = 32 * (int)((long long)F.nslice * (blockIdx.x + 1) / gridDim.x) - X.K0;   // cells of the block
#pragma unroll
  for (int u = 0; u < R; ++u) {
    const int K = X.K[u], e0 = X.off[u];
    X.off[u] = F.wmax * (warp + nw * u);
    const double sK = K >= 0 ? S[K] : 0.0;
    for (int j = 0; j < X.n[u]; ++j) {
      const int d = 32 * (X.off[u] + j) + lane, L = K >= 0 ? F.nbr[e0 + 32 * j] : X.K0;
      dv[d] = K >= 0 ? (T)(A[e0 + 32 * j] * sK * S[L]) : (T)0;
      dc[d] = L >= X.K0 && L < X.K0 + own ? L - X.K0 : ~L;
    }
  }
  X.v = dv;
  X.c = dc;
}

// xl[c], or v[~c] through L2 for c < 0: two predicated loads into one register, without a branch.
__device__ __forceinline__ double gather(const double* xl, const double* v, int c) {
  double x;
  asm volatile("{.reg .pred q; setp.ge.s32 q, %1, 0; @q ld.shared.f64 %0, [%2]; @!q ld.global.cg.f64 %0, [%3];}"
               : "=d"(x)
               : "r"(c), "r"((unsigned)__cvta_generic_to_shared(xl) + 8u * (unsigned)c), "l"(v + ~c)
               : "memory");
  return x;
}
__device__ __forceinline__ float gather(const float* xl, const float* v, int c) {
  float x;
  asm volatile("{.reg .pred q; setp.ge.s32 q, %1, 0; @q ld.shared.f32 %0, [%2]; @!q ld.global.cg.f32 %0, [%3];}"
               : "=f"(x)
               : "r"(c), "r"((unsigned)__cvta_generic_to_shared(xl) + 4u * (unsigned)c), "l"(v + ~c)
               : "memory");
  return x;
}

// The gathered value of entry e of slice u, from xl (LOCAL) where the column is the block's own; entry e times x onto acc.
template <bool LOCAL, int R, class T, bool ST>
__device__ __forceinline__ T row_value(const FRows<R, T, ST>& X, const T* v, int u, int e) {
  if (X.staged) {
    const int c = X.c[e];
    return LOCAL ? gather(X.xl, v, c) : __ldcg(&v[c >= 0 ? c + X.K0 : ~c]);
  }
  return X.K[u] >= 0 ? __ldcg(&v[__ldg(&X.c[e])]) : (T)0;
}
template <bool DIAG, int R, class T, bool ST>
__device__ __forceinline__ T row_add(const FRows<R, T, ST>& X, T acc, int u, int e, T x) {
  const T a = X.staged ? X.v[e] : X.K[u] >= 0 ? __ldg(&X.v[e]) : (T)0;
  return DIAG ? fma(a, x, acc) : fma(-a, x, acc);
}

// out = dg own + sum of the row's entries times v (DIAG), or own - that sum. In FP64 the gathers of slice u + 1 are on
// their way while slice u is summed: the scheduler moves a sub-partition's warps along together, so without that they
// all wait for memory at once and leave the FP64 pipe idle (11.6k clocks a product of 64^3 cells, of which 5.5k waiting).
// FP32 has no such pipe to fill, and the registers of the second set cost more there than they save (5.8 -> 6.9 us an
// iteration), and in the BiCGStab they spill (0.9 KB a thread, 46 instead of 28 us an iteration of 64^3 cells): those take a
// slice's entries eight at a time.
template <bool DIAG, bool LOCAL, int R, class T, bool ST>
__device__ __forceinline__ void rows_product(const FRows<R, T, ST>& X, const T* v, const T (&own)[R], const T (&dg)[R],
                                             T (&out)[R]) {
  const int lane = threadIdx.x & 31;
  auto first = [&](int u) { return X.staged ? 32 * X.off[u] + lane : X.off[u]; };
  if constexpr (std::is_same_v<T, double> && R > 1 && !DIAG) {
    constexpr int Q = 6;
    T x[2][Q];
    auto fetch = [&](int u, T(&y)[Q]) {
#pragma unroll
      for (int q = 0; q < Q; ++q)
        if (q < X.n[u]) y[q] = row_value<LOCAL>(X, v, u, first(u) + 32 * q);
    };
    fetch(0, x[0]);
#pragma unroll
    for (int u = 0; u < R; ++u) {
      if (u + 1 < R) fetch(u + 1 < R ? u + 1 : u, x[(u + 1) & 1]);
      T acc = DIAG ? dg[u] * own[u] : own[u];
      const int e0 = first(u);
#pragma unroll
      for (int q = 0; q < Q; ++q)
        if (q < X.n[u]) acc = row_add<DIAG>(X, acc, u, e0 + 32 * q, x[u & 1][q]);
      for (int j = Q; j < X.n[u]; ++j)   // wider rows
        acc = row_add<DIAG>(X, acc, u, e0 + 32 * j, row_value<LOCAL>(X, v, u, e0 + 32 * j));
      out[u] = acc;
    }
  } else {
#pragma unroll
    for (int u = 0; u < R; ++u) {
      T acc = DIAG ? dg[u] * own[u] : own[u];
      const int e0 = first(u);
      for (int j0 = 0; j0 < X.n[u]; j0 += 8) {
        T a[8], x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const bool in = j0 + q < X.n[u] && (X.staged || X.K[u] >= 0);
          const int e = e0 + 32 * (j0 + q);
          x[q] = a[q] = (T)0;
          if (in) {
            a[q] = X.staged ? X.v[e] : __ldg(&X.v[e]);
            x[q] = row_value<LOCAL>(X, v, u, e);
          }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (j0 + q < X.n[u]) acc = DIAG ? fma(a[q], x[q], acc) : fma(-a[q], x[q], acc);
      }
      out[u] = acc;
    }
  }
}

__device__ __forceinline__ double wide(double v) { return v; }
__device__ __forceinline__ double wide(float v) { return widen(v); }

// Pipelined CG (Ghysels and Vanroose) on the symmetrically Jacobi-scaled system of kp_fine_cg: n = A w, z = n + beta z,
// s = w + beta s, p = r + beta p, y += alpha p, r -= alpha s, w -= alpha z, gamma = (r, r), delta = (w, r). A thread owns
// the same cells for the whole solve, so y, r, p, s, z and w stay in its registers; only w, which the neighbours
// gather, is written to memory (double-buffered). The barrier that publishes w publishes the partial sums too; while
// the other warps form n = A w the server warp adds them up and derives beta and alpha, so the serial part of the
// reduction hides behind the product (one product is spent in vain at the end of a solve).
// What bounds it: 14 FP64 operations a cell at 19 clocks per warp operation and SM on large meshes (6.9 us an iteration
// of 262,144 cells), the chain gather - product - updates - sums - barrier on small ones.
// T = float runs the vectors, the matrix and a thread's partial sums in FP32, block and grid sums in FP64. In FP32 the
// recurrences drift away from the true residual on the six-decade channelized field (the iteration count grew fivefold),
// so every `replace` iterations the residual and the auxiliary vectors are recomputed from their definitions --
// r = b - A y and s = A p, then w = A r and z = A s (residual replacement, Cools and Vanroose) -- which costs four
// products and two extra synchronisations.
template <class T, int R, bool ST>
__global__ void __launch_bounds__(kFThreads, 1) kp_fine_cg_reg(FineDev F, const double* __restrict__ Tval,
                                                               const T* __restrict__ Ts, const double* __restrict__ sdiag,
                                                               const double* __restrict__ b, double bscale,
                                                               double* __restrict__ dx, FineCgBufs<T> B, double* partial,
                                                               GridSync gs, double tol, int maxit, int replace, int staged,
                                                               PcgResult* res) {
  __shared__ double sm[kSmDoubles];
  __shared__ double sc[4];   // beta, alpha, gamma, gamma_0
  __shared__ int stop;
  extern __shared__ double dyn[];
  const int server = (blockDim.x >> 5) - 1, warp = threadIdx.x >> 5;
  Grid g = grid_start(gs, partial, sm);
  FRows<R, T, ST> X;
  rows_init(X, F, server);
  if constexpr (ST) {
    X.xl = (T*)((int*)((T*)dyn + staged) + staged);
    rows_stage(X, F, Tval, sdiag, (T*)dyn, (int*)((T*)dyn + staged), server);
  } else {
    X.v = Ts;
    X.c = F.nbr;
  }
  T y[R], r[R], p[R], sv[R], z[R], w[R], n[R];
  T* wc = B.wb;   // published w of the current iteration
  T* wn = B.wa;   // next w
#pragma unroll
  for (int u = 0; u < R; ++u) {
    const int K = X.K[u];
    y[u] = p[u] = sv[u] = z[u] = r[u] = w[u] = (T)0;
    if (K >= 0) {
      r[u] = (T)(sdiag[K] * bscale * b[K]);
      wn[K] = r[u];   // the first product is A r
      if (X.staged) X.xl[K - X.K0] = r[u];
    }
  }
  if (!grid_barrier(g)) return;
  rows_product<false, true>(X, wn, r, r, w);
  __syncthreads();   // xl is read
  T t0 = (T)0, t1 = (T)0;
#pragma unroll
  for (int u = 0; u < R; ++u)
    if (X.K[u] >= 0) {
      wc[X.K[u]] = w[u];
      if (X.staged) X.xl[X.K[u] - X.K0] = w[u];
      t0 = fma(r[u], r[u], t0);
      t1 = fma(w[u], r[u], t1);
    }
  {
    const double d[2] = {wide(t0), wide(t1)};
    if (!grid_sum_arrive<2>(g, d, server)) return;
  }
  double tol2 = 0.0, ig = 0.0, ia = 0.0;   // the server's: 1 / gamma and 1 / alpha of the last iteration
  int it = 0;
  while (true) {
    if (warp == server) {
      double t[2];
      grid_sum_finish<2>(g, t);
      if (it == 0) tol2 = tol * tol * t[0];
      const double beta = t[0] * ig;                      // gamma / gamma_old (first: 0)
      const double den = fma(-beta, t[0] * ia, t[1]);     // delta - beta gamma / alpha_old
      const double alpha = den != 0.0 ? t[0] * fast_rcp(den) : 0.0;
      if ((threadIdx.x & 31) == 0) {
        if (it == 0) sc[3] = t[0];
        sc[0] = beta;
        sc[1] = alpha;
        sc[2] = t[0];
        stop = !(sc[3] > 0.0 && t[0] > tol2 && it < maxit) || !(alpha != 0.0);
      }
      __syncthreads();
      ig = t[0] != 0.0 ? fast_rcp(t[0]) : 0.0;
      ia = fast_rcp(alpha);
    } else {
      rows_product<false, true>(X, wc, w, w, n);
      __syncthreads();
    }
    if (stop) break;
    const T be = (T)sc[0], al = (T)sc[1];
    t0 = t1 = (T)0;
    if (X.K[0] >= 0) {
#pragma unroll
      for (int u = 0; u < R; ++u)
        if (u == 0 || X.K[u] >= 0) {
          z[u] = fma(be, z[u], n[u]);
          sv[u] = fma(be, sv[u], w[u]);
          w[u] = fma(-al, z[u], w[u]);
          wn[X.K[u]] = w[u];
          if (X.staged) X.xl[X.K[u] - X.K0] = w[u];
          p[u] = fma(be, p[u], r[u]);
          r[u] = fma(-al, sv[u], r[u]);
          t0 = fma(r[u], r[u], t0);
          t1 = fma(w[u], r[u], t1);
        }
    }
    bool replaced = false;
    if constexpr (std::is_same_v<T, float>) {
      if (replace > 0 && (it + 1) % replace == 0) {
        T q[R];
        replaced = true;
#pragma unroll
        for (int u = 0; u < R; ++u)
          if (X.K[u] >= 0) {
            y[u] = fma(al, p[u], y[u]);
            B.y[X.K[u]] = y[u];
            B.p[X.K[u]] = p[u];
          }
        if (!grid_barrier(g)) return;
        rows_product<false, false>(X, B.y, y, y, q);
        rows_product<false, false>(X, B.p, p, p, sv);
#pragma unroll
        for (int u = 0; u < R; ++u) {
          const int K = X.K[u];
          r[u] = K >= 0 ? (T)(sdiag[K] * bscale * b[K]) - q[u] : (T)0;
          if (K >= 0) {
            B.r[K] = r[u];
            B.s[K] = sv[u];
          }
        }
        if (!grid_barrier(g)) return;
        rows_product<false, false>(X, B.r, r, r, w);
        rows_product<false, false>(X, B.s, sv, sv, z);
        t0 = t1 = (T)0;
#pragma unroll
        for (int u = 0; u < R; ++u)
          if (X.K[u] >= 0) {
            wn[X.K[u]] = w[u];
            if (X.staged) X.xl[X.K[u] - X.K0] = w[u];
            t0 = fma(r[u], r[u], t0);
            t1 = fma(w[u], r[u], t1);
          }
      }
    }
    const double d[2] = {wide(t0), wide(t1)};
    if (!grid_sum_arrive<2>(g, d, server, [&] {   // y waits for nothing: off the chain to the next product
          if (!replaced && X.K[0] >= 0) {
#pragma unroll
            for (int u = 0; u < R; ++u) y[u] = fma(al, p[u], y[u]);
          }
        }))
      return;
    T* t = wc;
    wc = wn;
    wn = t;
    ++it;
  }
#pragma unroll
  for (int u = 0; u < R; ++u)
    if (X.K[u] >= 0) dx[X.K[u]] = sdiag[X.K[u]] * (double)y[u];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    res->err = 0;
    res->iters = it;
    res->rr0 = sc[3];
    res->rr = sc[2];
  }
}

// BiCGStab (van der Vorst) on the symmetrically scaled Newton system of kp_fine_bicgstab with a thread's r (and s), p, v
// and t in registers and its y, rh and diagonal in shared memory (all in registers they spilled, and an iteration of
// 64^3 cells took 42 us); p and s, which the neighbours gather, are published, and a block's own copy of them stays in
// shared memory. One iteration: v = J p and (rh, v) give alpha; s = r - alpha v; t = J s and (t, s), (t, t), (rh, t),
// (rh, s), (s, s) give omega and, since r = s - omega t, also (rh, r) = (rh, s) - omega (rh, t) and (r, r) = (s, s) -
// 2 omega (t, s) + omega^2 (t, t), hence rho, beta and the stopping test without a reduction of their own: two sums
// and two barriers an iteration instead of three and two. Where (r, r) comes out below a quarter of (s, s) both are summed
// from the vectors after all, so the difference costs (r, r) two bits at most, and (rh, r), whose terms are bounded by
// |rh| |s| where the direct sum's are by |rh| |r|, as many; the sums themselves are more than a bit better than a tree's
// (isum.cuh). That is one iteration in sixty on channelized fields. Bounded like the CG: 26 FP64 operations a cell, and
// four synchronisations.
template <int R, bool ST>
__global__ void __launch_bounds__(kFThreads, 1) kp_fine_bicgstab_reg(FineDev F, const double* __restrict__ Joff,
                                                                     const double* __restrict__ Js,
                                                                     const double* __restrict__ jdiag,
                                                                     const double* __restrict__ D,
                                                                     const double* __restrict__ S,
                                                                     const double* __restrict__ b, double bscale,
                                                                     double* __restrict__ dx, double* pg, double* sg,
                                                                     double* partial, GridSync gs, double tol, int maxit,
                                                                     int staged, PcgResult* res) {
  __shared__ double sm[kSmDoubles];
  __shared__ double sc[3];   // alpha, omega, beta
  __shared__ double sv[4];   // the server's: (r_0, r_0), (r, r), rho, the stopping value
  __shared__ int state;      // 0 go on, 1 stop, 2 sum (rh, r) and (r, r) from the vectors
  extern __shared__ double dyn[];
  const int server = (blockDim.x >> 5) - 1, warp = threadIdx.x >> 5;
  Grid g = grid_start(gs, partial, sm);
  FRows<R, double, ST> X;
  rows_init(X, F, server);
  // per thread and slice: y, rh and the diagonal, then the rows
  const int T = blockDim.x;
  double *ys = dyn + threadIdx.x, *rhs = ys + R * T, *jds = rhs + R * T, *rows = dyn + 3 * R * T;
  if constexpr (ST) {
    X.xl = (double*)((int*)(rows + staged) + staged);
    rows_stage(X, F, Joff, S, rows, (int*)(rows + staged), server);
  } else {
    X.v = Js;
    X.c = F.nbr;
  }
  double r[R], p[R], v[R];
#pragma unroll
  for (int u = 0; u < R; ++u) {
    const int K = X.K[u];
    r[u] = v[u] = 0.0;
    double jd = 0.0;
    if (K >= 0) {
      r[u] = S[K] * bscale * b[K];
      jd = jdiag[K] * D[K];
      pg[K] = r[u];
      if (X.staged) X.xl[K - X.K0] = r[u];
    }
    p[u] = r[u];
    ys[u * T] = 0.0;
    rhs[u * T] = r[u];
    jds[u * T] = jd;
  }
  auto diag = [&](double(&d)[R]) {
#pragma unroll
    for (int u = 0; u < R; ++u) d[u] = jds[u * T];
  };
  {
    double d[1] = {0.0}, t[1];
#pragma unroll
    for (int u = 0; u < R; ++u) d[0] = fma(r[u], r[u], d[0]);
    if (!grid_sum_arrive<1>(g, d, server)) return;   // its barrier also publishes p
    if (warp == server) {
      grid_sum_finish<1>(g, t);
      if ((threadIdx.x & 31) == 0) {
        sv[0] = sv[1] = sv[2] = t[0];
        sv[3] = tol * tol * t[0];
        state = t[0] > 0.0 && t[0] > sv[3] && maxit > 0 ? 0 : 1;
      }
    }
    __syncthreads();
  }
  int it = 0;
  while (state != 1) {
    double d1[1] = {0.0};
    {
      double jd[R];
      diag(jd);
      rows_product<true, true>(X, pg, p, jd, v);
    }
    if (X.K[0] >= 0) {
#pragma unroll
      for (int u = 0; u < R; ++u) d1[0] = fma(rhs[u * T], v[u], d1[0]);
    }
    if (!grid_sum_arrive<1>(g, d1, server)) return;
    if (warp == server) {
      double t[1];
      grid_sum_finish<1>(g, t);
      const double alpha = t[0] != 0.0 ? sv[2] * fast_rcp(t[0]) : 0.0;
      if ((threadIdx.x & 31) == 0) {
        sc[0] = alpha;
        state = alpha != 0.0 ? 0 : 1;
      }
    }
    __syncthreads();
    if (state == 1) break;
    const double al = sc[0];
    if (X.K[0] >= 0) {
#pragma unroll
      for (int u = 0; u < R; ++u) {
        r[u] = fma(-al, v[u], r[u]);
        if (X.K[u] >= 0) {
          sg[X.K[u]] = r[u];
          if (X.staged) X.xl[X.K[u] - X.K0] = r[u];
        }
      }
    }
    if (!grid_barrier(g)) return;
    double t[R], d5[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    {
      double jd[R];
      diag(jd);
      rows_product<true, true>(X, sg, r, jd, t);
    }
    if (X.K[0] >= 0) {
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const double rh = rhs[u * T];
        d5[0] = fma(t[u], r[u], d5[0]);
        d5[1] = fma(t[u], t[u], d5[1]);
        d5[2] = fma(rh, t[u], d5[2]);
        d5[3] = fma(rh, r[u], d5[3]);
        d5[4] = fma(r[u], r[u], d5[4]);
      }
    }
    if (!grid_sum_arrive<5>(g, d5, server)) return;
    if (warp == server) {
      double s[5];
      grid_sum_finish<5>(g, s);
      const double rho = sv[2], omega = s[1] != 0.0 ? s[0] * fast_rcp(s[1]) : 0.0;
      const double rn = fma(-omega, s[2], s[3]), rr = fma(omega, fma(omega, s[1], -2.0 * s[0]), s[4]);
      const bool direct = rr <= 0.25 * s[4];
      const double beta = rho != 0.0 && omega != 0.0 ? rn * fast_rcp(rho) * (al * fast_rcp(omega)) : 0.0;
      __syncwarp();
      if ((threadIdx.x & 31) == 0) {
        sc[1] = omega;
        sc[2] = beta;
        if (!direct) {
          sv[1] = rr;
          sv[2] = rn;
        }
        state = direct ? 2 : !(omega != 0.0) || !(rn != 0.0) || !(rr > sv[3] && it + 1 < maxit) ? 1 : 0;
      }
    }
    __syncthreads();
    ++it;
    const double om = sc[1];
    if (X.K[0] >= 0) {
#pragma unroll
      for (int u = 0; u < R; ++u) {
        ys[u * T] = fma(al, p[u], fma(om, r[u], ys[u * T]));
        r[u] = fma(-om, t[u], r[u]);
      }
    }
    if (state == 2) {
      double d2[2] = {0.0, 0.0};
#pragma unroll
      for (int u = 0; u < R; ++u) {
        d2[0] = fma(rhs[u * T], r[u], d2[0]);
        d2[1] = fma(r[u], r[u], d2[1]);
      }
      if (!grid_sum_arrive<2>(g, d2, server)) return;
      if (warp == server) {
        double s[2];
        grid_sum_finish<2>(g, s);
        const double rho = sv[2];
        const double beta = rho != 0.0 && om != 0.0 ? fast_div(s[0], rho) * fast_div(al, om) : 0.0;
        __syncwarp();
        if ((threadIdx.x & 31) == 0) {
          sc[2] = beta;
          sv[1] = s[1];
          sv[2] = s[0];
          state = !(om != 0.0) || !(s[0] != 0.0) || !(s[1] > sv[3] && it < maxit) ? 1 : 0;
        }
      }
      __syncthreads();
    }
    if (state == 1) break;
    const double be = sc[2];
    if (X.K[0] >= 0) {
#pragma unroll
      for (int u = 0; u < R; ++u) {
        p[u] = fma(be, fma(-om, v[u], p[u]), r[u]);
        if (X.K[u] >= 0) {
          pg[X.K[u]] = p[u];
          if (X.staged) X.xl[X.K[u] - X.K0] = p[u];
        }
      }
    }
    if (!grid_barrier(g)) return;
  }
#pragma unroll
  for (int u = 0; u < R; ++u)
    if (X.K[u] >= 0) dx[X.K[u]] = S[X.K[u]] * ys[u * T];
  if (blockIdx.x == 0 && threadIdx.x == 32 * server) {
    res->err = 0;
    res->iters = it;
    res->rr0 = sv[0];
    res->rr = sv[1];
  }
}

// The launch shape of a register-resident kernel: blocks of up to kFWarps slices' warps and the server, four warps a
// block (one per sub-partition) before a second block's worth, then more warps, then more slices a warp.
struct FShape {
  int grid, warps, R;   // R: slices a warp
  bool cluster;
};
FShape fine_shape(const FineDev& F, int sm_cap) {
  FShape s;
  s.grid = std::max(1, std::min(coop_sms(sm_cap), (F.nslice + 3) / 4));
  // up to 64 slices: one cluster (an iteration's 14 FP64 operations of eight slices an SM take 2.1k clocks, its barrier
  // saves more)
  if (F.nslice <= 64) s.grid = std::min(s.grid, kClusterBlocks);
  s.cluster = cluster_grid(s.grid, coop_sms(sm_cap));
  const int per = (F.nslice + s.grid - 1) / s.grid;
  s.warps = std::max(1, std::min(kFWarps, per));
  s.R = (per + s.warps - 1) / s.warps;
  return s;
}
// entries of shared memory, or 0 if the rows do not fit beside `other` bytes
int staged_entries(const FineDev& F, const FShape& s, size_t entry_bytes, size_t other = 0) {
  const size_t cells = (size_t)s.warps * s.R * 32, n = cells * std::max(F.wmax, 1);
  return n * entry_bytes + cells * (entry_bytes - sizeof(int)) + other <= kFDyn ? (int)n : 0;
}

template <class T, int R, bool ST>
cudaError_t launch_cg(cudaStream_t st, const FShape& s, const FineDev& F, const double* Tval, T* Ts, const double* sdiag,
                      const double* b, double bscale, double* dx, const FineCgBufs<T>& B, double* partial, GridSync gs,
                      double tol, int maxit, int replace, PcgResult* res) {
  const void* fn = (const void*)kp_fine_cg_reg<T, R, ST>;
  static DeviceOnce limit;
  if (const cudaError_t e = raise_smem_limit(limit, fn, kFDyn)) return e;
  const size_t eb = sizeof(T) + sizeof(int);
  gs.cluster = s.cluster ? 1 : 0;
  int staged = staged_entries(F, s, eb);
  if (!ST) launch_scale_sell<T>(st, F, Tval, sdiag, Ts);
  void* args[] = {(void*)&F, (void*)&Tval, (void*)&Ts, (void*)&sdiag, (void*)&b, (void*)&bscale, (void*)&dx, (void*)&B,
                  (void*)&partial, (void*)&gs, (void*)&tol, (void*)&maxit, (void*)&replace, (void*)&staged, (void*)&res};
  return launch_persistent(fn, s.grid, 32 * (s.warps + 1), args,
                           staged ? (size_t)staged * eb + (size_t)s.warps * s.R * 32 * sizeof(T) : 0, s.cluster, st);
}

template <int R, bool ST>
cudaError_t launch_bicg(cudaStream_t st, const FShape& s, const FineDev& F, const double* Joff, double* Js,
                        const double* jdiag, const double* D, const double* S, const double* b, double bscale, double* dx,
                        double* work, double* partial, GridSync gs, double tol, int maxit, PcgResult* res) {
  const void* fn = (const void*)kp_fine_bicgstab_reg<R, ST>;
  static DeviceOnce limit;
  if (const cudaError_t e = raise_smem_limit(limit, fn, kFDyn)) return e;
  gs.cluster = s.cluster ? 1 : 0;
  const size_t own = (size_t)3 * R * 32 * (s.warps + 1) * sizeof(double);
  int staged = staged_entries(F, s, sizeof(double) + sizeof(int), own);
  if (!ST) launch_scale_sell<double>(st, F, Joff, S, Js);
  double *pg = work, *sg = work + F.N;
  void* args[] = {(void*)&F, (void*)&Joff, (void*)&Js, (void*)&jdiag, (void*)&D, (void*)&S, (void*)&b, (void*)&bscale,
                  (void*)&dx, (void*)&pg, (void*)&sg, (void*)&partial, (void*)&gs, (void*)&tol, (void*)&maxit,
                  (void*)&staged, (void*)&res};
  return launch_persistent(fn, s.grid, 32 * (s.warps + 1), args,
                           own + (staged ? (size_t)staged * 12 + (size_t)s.warps * s.R * 32 * 8 : 0), s.cluster, st);
}

}  // namespace

template <class T>
cudaError_t launch_fine_cg_reg(cudaStream_t st, const FineDev& F, const double* Tval, T* Ts, const double* sdiag,
                               const double* b, double bscale, double* dx, const FineCgBufs<T>& B, double* partial,
                               GridSync gs, double tol, int maxit, int replace, PcgResult* res) {
  const FShape s = fine_shape(F, gs.sm_cap);
  const bool fits = staged_entries(F, s, sizeof(T) + sizeof(int)) > 0;
  constexpr bool kStream = std::is_same_v<T, float>;
  if (!fits && !kStream) return cudaErrorNotSupported;
#define NLMG_CG(RR)                                                                                                      \
  if (s.R <= RR)                                                                                                         \
  return (fits ? launch_cg<T, RR, true> : launch_cg<T, RR, !kStream>)(st, s, F, Tval, Ts, sdiag, b, bscale, dx, B,       \
                                                                      partial, gs, tol, maxit, replace, res)
  NLMG_CG(1);
  NLMG_CG(2);
  NLMG_CG(3);
  NLMG_CG(4);
  if constexpr (std::is_same_v<T, float>) {
    NLMG_CG(6);
    NLMG_CG(9);
  } else {
    NLMG_CG(5);
  }
#undef NLMG_CG
  return cudaErrorNotSupported;
}
template cudaError_t launch_fine_cg_reg<double>(cudaStream_t, const FineDev&, const double*, double*, const double*,
                                                const double*, double, double*, const FineCgBufs<double>&, double*,
                                                GridSync, double, int, int, PcgResult*);
template cudaError_t launch_fine_cg_reg<float>(cudaStream_t, const FineDev&, const double*, float*, const double*,
                                               const double*, double, double*, const FineCgBufs<float>&, double*,
                                               GridSync, double, int, int, PcgResult*);

cudaError_t launch_fine_bicgstab_reg(cudaStream_t st, const FineDev& F, const double* Joff, double* Js,
                                     const double* jdiag, const double* D, const double* S, const double* b,
                                     double bscale, double* dx, double* work, double* partial, GridSync gs, double tol,
                                     int maxit, PcgResult* res) {
  const FShape s = fine_shape(F, gs.sm_cap);
  const bool fits = staged_entries(F, s, 12, (size_t)3 * s.R * 32 * (s.warps + 1) * sizeof(double)) > 0;
#define NLMG_BICG(RR)                                                                                                    \
  if (s.R <= RR)                                                                                                         \
  return (fits ? launch_bicg<RR, true> : launch_bicg<RR, false>)(st, s, F, Joff, Js, jdiag, D, S, b, bscale, dx, work,   \
                                                                 partial, gs, tol, maxit, res)
  NLMG_BICG(1);
  NLMG_BICG(2);
  NLMG_BICG(3);
  NLMG_BICG(4);
#undef NLMG_BICG
  return cudaErrorNotSupported;
}

}  // namespace nlmg
