// Persistent (cooperative) kernels with their state in memory: one launch runs a whole level-0 linear solve (the Picard
// step's CG, the Newton step's BiCGStab) with device-side scalars, decisions and convergence tests, so the iterations pay
// neither launch gaps nor host round trips. Meshes whose cells fit the registers of the grid run fine_reg.cu instead.
//
// Grid-wide synchronisation uses a counter barrier whose wait is bounded: after ~2 s of polling the kernel records an
// error flag and every block leaves. The launch goes through cudaLaunchCooperativeKernel with at most the co-resident
// number of blocks, so in a correct run every wait ends.
//
// Data written by one block and read by another inside the same launch (CG vectors, per-interface buffers) is read
// with ld.global.cg (L2, bypassing the non-coherent L1), after the barrier that orders the write.
//
// Reductions stay deterministic: each block writes one partial per value; after the barrier every block adds all
// partials (in integers, isum.cuh) and derives the step lengths once, so all blocks take the same
// decisions from bit-identical scalars and a run is bitwise reproducible for a given grid.
#include <atomic>
#include <cmath>

#include "kernels.cuh"
#include "persist.cuh"
#include "psync.cuh"

namespace nlmg {

namespace {

constexpr int kPThreads = 512;                           // threads per block of the persistent kernels

// Cells over the grid, a block's threads side by side (these meshes fill every SM many times over).
#define CSTRIDE(i, n) for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < (n); i += gridDim.x * blockDim.x)

// ---- fine level: A dx = bscale * b with the frozen TPFA matrix --------------------------------------------------
// CG on the symmetrically Jacobi-scaled system (S A S) y = S bscale b, dx = S y, S = diag(A)^-1/2, so the scaled
// matrix has a unit diagonal and only its off-diagonal entries Ts (SELL-32 layout, type T) are read. T = double is
// the FP64 path; T = float runs the Krylov vectors and the matrix in FP32 inside the FP64 nonlinear iteration
// (per-thread partial sums of the dot products in FP32, block and grid sums in FP64). The matrix is applied to the residual r, which every iteration already
// materialises, and A p follows by recurrence (p = r + beta p, q = A r + beta q): no neighbour values have to be
// rebuilt and an iteration needs two grid barriers. The stopping test is on the scaled residual,
// ||S r|| <= tol ||S r_0|| (the r.z of Jacobi-preconditioned CG).
template <class T>
__global__ void __launch_bounds__(kPThreads) kp_fine_cg(FineDev F, const T* __restrict__ Ts,
                                                        const double* __restrict__ sdiag,
                                                        const double* __restrict__ b, double bscale,
                                                        double* __restrict__ dx, T* __restrict__ y,
                                                        T* __restrict__ r, T* __restrict__ p, T* __restrict__ q,
                                                        double* partial, GridSync gs, double tol, int maxit,
                                                        PcgResult* res) {
  __shared__ double sm[kSmDoubles];
  Grid g = grid_start(gs, partial, sm);
  T t1 = (T)0;   // per-thread partial sums in T (a thread holds one or two cells), block and grid sums in FP64
  CSTRIDE(i, F.N) {
    const T ri = (T)(sdiag[i] * bscale * b[i]);
    y[i] = (T)0;
    r[i] = ri;
    t1 = fma(ri, ri, t1);
  }
  double a1[1] = {(double)t1};
  if (!grid_sum<1>(g, a1)) return;
  const double rr0 = a1[0];
  double rr = rr0;
  const double tol2 = tol * tol * rr0;
  T beta = (T)0;
  int it = 0;
  while (rr0 > 0.0 && rr > tol2 && it < maxit) {
    T tpq = (T)0;
    CSTRIDE(K, F.N) {
      const int s = K >> 5, lane = K & 31;
      const T rK = __ldcg(&r[K]);
      T acc = rK;
      const int w = F.sell_w[s];
      int e = F.sell_off[s] + lane;
      int j = 0;
      if (w <= 8) {
        int Ls[8];
        T Tv[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (u < w) {
            Ls[u] = F.nbr[e + 32 * u];
            Tv[u] = Ts[e + 32 * u];
          }
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (u < w) acc -= Tv[u] * __ldcg(&r[Ls[u]]);
        j = w;
      }
      for (e += 32 * j; j < w; ++j, e += 32) acc -= Ts[e] * __ldcg(&r[F.nbr[e]]);
      const T pK = it == 0 ? rK : rK + beta * p[K];
      const T qK = it == 0 ? acc : acc + beta * q[K];
      p[K] = pK;
      q[K] = qK;
      tpq = fma(pK, qK, tpq);
    }
    double pq[2] = {(double)tpq, 0.0};
    if (!grid_sum_x<1, 1>(g, pq, [&](double* o) { o[1] = o[0] != 0.0 ? fast_div(rr, o[0]) : 0.0; }))
      return;
    const double alpha_d = pq[1];
    const T alpha = (T)alpha_d;
    T trn = (T)0;
    CSTRIDE(i, F.N) {
      y[i] = alpha * p[i] + y[i];
      const T ri = r[i] - alpha * q[i];
      r[i] = ri;
      trn = fma(ri, ri, trn);
    }
    double rn[2] = {(double)trn, 0.0};
    if (!grid_sum_x<1, 1>(g, rn, [&](double* o) { o[1] = rr != 0.0 ? fast_div(o[0], rr) : 0.0; }))
      return;
    beta = (T)rn[1];
    rr = rn[0];
    ++it;
    if (!(alpha_d != 0.0)) break;   // breakdown (p.Ap = 0): stop with the current iterate
  }
  CSTRIDE(i, F.N) dx[i] = sdiag[i] * (double)y[i];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    res->err = 0;
    res->iters = it;
    res->rr0 = rr0;
    res->rr = rr;
  }
}

// Pipelined CG (Ghysels and Vanroose) on the same scaled system: the dot products of an iteration are computed from
// vectors updated in the same pass as the matrix product, so one grid barrier per iteration both publishes the
// vector the next matrix product gathers and completes the reduction. Recurrences: n = A w, z = n + beta z,
// s = w + beta s, p = r + beta p, y += alpha p, r -= alpha s, w -= alpha z; gamma = (r, r), delta = (w, r). Used for
// loose tolerances (the recursively updated residual drifts from the true one at the 1e-10 level).
template <class T>
__device__ __forceinline__ T sell_apply(const FineDev& F, const T* __restrict__ Ts, const T* v, int K) {
  const int s = K >> 5, lane = K & 31;
  T acc = __ldcg(&v[K]);
  const int w = F.sell_w[s];
  int e = F.sell_off[s] + lane;
  int j = 0;
  if (w <= 8) {
    int Ls[8];
    T Tv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (u < w) {
        Ls[u] = F.nbr[e + 32 * u];
        Tv[u] = Ts[e + 32 * u];
      }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (u < w) acc -= Tv[u] * __ldcg(&v[Ls[u]]);
    j = w;
  }
  for (e += 32 * j; j < w; ++j, e += 32) acc -= Ts[e] * __ldcg(&v[F.nbr[e]]);
  return acc;
}

template <class T>
__global__ void __launch_bounds__(kPThreads, 2) kp_fine_cg_pipe(FineDev F, const T* __restrict__ Ts,
                                                             const double* __restrict__ sdiag,
                                                             const double* __restrict__ b, double bscale,
                                                             double* __restrict__ dx, T* __restrict__ y,
                                                             T* __restrict__ r, T* wa, T* wb, T* __restrict__ z,
                                                             T* __restrict__ sv, T* __restrict__ p, double* partial,
                                                             GridSync gs, double tol, int maxit, PcgResult* res) {
  __shared__ double sm[kSmDoubles];
  Grid g = grid_start(gs, partial, sm);
  CSTRIDE(i, F.N) {
    r[i] = (T)(sdiag[i] * bscale * b[i]);
    y[i] = z[i] = sv[i] = p[i] = (T)0;
  }
  if (!grid_barrier(g)) return;
  // a4 = {gamma, delta, beta, alpha}: the sums and, from the last block's thread 0, the step lengths of the next
  // iteration (beta = gamma / gamma_old, alpha = gamma / (delta - beta gamma / alpha_old); first: 0, gamma / delta)
  double a4[4] = {0.0, 0.0, 0.0, 0.0};
  CSTRIDE(K, F.N) {
    const T wK = sell_apply<T>(F, Ts, r, K);
    wa[K] = wK;
    const double rK = (double)r[K];
    a4[0] = fma(rK, rK, a4[0]);
    a4[1] = fma((double)wK, rK, a4[1]);
  }
  if (!grid_sum_x<2, 2>(g, a4, [&](double* o) {
        o[2] = 0.0;
        o[3] = o[1] != 0.0 ? fast_div(o[0], o[1]) : 0.0;
      }))
    return;
  double gamma = a4[0], beta_d = a4[2], alpha_d = a4[3];
  const double rr0 = gamma;
  const double tol2 = tol * tol * rr0;
  T* wc = wa;   // current w (read, neighbours gathered)
  T* wn = wb;   // next w (written)
  int it = 0;
  while (rr0 > 0.0 && gamma > tol2 && it < maxit) {
    if (!(alpha_d != 0.0)) break;
    const T alpha = (T)alpha_d, beta = (T)beta_d;
    double n4[4] = {0.0, 0.0, 0.0, 0.0};
    CSTRIDE(K, F.N) {
      const T nK = sell_apply<T>(F, Ts, wc, K);
      const T wK = wc[K];
      const T zK = nK + beta * z[K];
      const T sK = wK + beta * sv[K];
      const T pK = r[K] + beta * p[K];
      z[K] = zK;
      sv[K] = sK;
      p[K] = pK;
      y[K] += alpha * pK;
      const T rK = r[K] - alpha * sK;
      r[K] = rK;
      const T wN = wK - alpha * zK;
      wn[K] = wN;
      n4[0] = fma((double)rK, (double)rK, n4[0]);
      n4[1] = fma((double)wN, (double)rK, n4[1]);
    }
    if (!grid_sum_x<2, 2>(g, n4, [&](double* o) {
          const double g = o[0], d = o[1];
          const double bn = gamma != 0.0 ? fast_div(g, gamma) : 0.0;
          const double den = d - fast_div(bn * g, alpha_d);
          o[2] = bn;
          o[3] = den != 0.0 ? fast_div(g, den) : 0.0;
        }))
      return;
    gamma = n4[0];
    beta_d = n4[2];
    alpha_d = n4[3];
    T* t = wc;
    wc = wn;
    wn = t;
    ++it;
  }
  CSTRIDE(i, F.N) dx[i] = sdiag[i] * (double)y[i];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    res->err = 0;
    res->iters = it;
    res->rr0 = rr0;
    res->rr = gamma;
  }
}

// ---- fine level: Newton update J dx = bscale * b with the exact Jacobian ---------------------------------------
// Row K of the scaled Jacobian applied to v: jd_K v_K + sum_e Js_e v_L(e) (SELL-32 layout; padding entries are 0).
__device__ __forceinline__ double jac_row(const FineDev& F, const double* __restrict__ Js, double jdK, const double* v,
                                          int K) {
  const int s = K >> 5, lane = K & 31;
  double acc = jdK * __ldcg(&v[K]);
  const int w = F.sell_w[s];
  int e = F.sell_off[s] + lane;
  int j = 0;
  if (w <= 8) {
    int Ls[8];
    double Jv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (u < w) {
        Ls[u] = F.nbr[e + 32 * u];
        Jv[u] = Js[e + 32 * u];
      }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (u < w) acc = fma(Jv[u], __ldcg(&v[Ls[u]]), acc);
    j = w;
  }
  for (e += 32 * j; j < w; ++j, e += 32) acc = fma(Js[e], __ldcg(&v[F.nbr[e]]), acc);
  return acc;
}

// BiCGStab (van der Vorst) in FP64 on the symmetrically scaled Newton system (S J S) y = S bscale b, dx = S y, with
// S = D^1/2 and D = 1 / max(J_KK, d_K / 2) the weights of the nonlinear Jacobi smoother (d_K the frozen-coefficient
// diagonal); jd = J_KK D_K and Js = S_K J_KL S_L are formed before the launch. The Jacobian is not symmetric, so CG
// does not apply; BiCGStab's short recurrences keep the whole solve in one persistent launch with a fixed amount of
// memory. One iteration: v = A p and (rh, v) give alpha; s = r - alpha v is published; t = A s, (t, s) and (t, t)
// give omega; y += alpha p + omega s, r = s - omega t, (rh, r) and (r, r) give rho and beta; p = r + beta (p - omega
// v) is published: three reductions and two plain barriers. The stopping test is ||r|| <= tol ||r_0|| on the scaled
// residual, as for the CG; a breakdown (alpha, omega or rho zero) ends the solve with the current y.
__global__ void __launch_bounds__(kPThreads) kp_fine_bicgstab(FineDev F, const double* __restrict__ Js,
                                                              const double* __restrict__ jd,
                                                              const double* __restrict__ sS,
                                                              const double* __restrict__ b, double bscale,
                                                              double* __restrict__ dx, double* __restrict__ y,
                                                              double* __restrict__ r, double* __restrict__ rh,
                                                              double* p, double* __restrict__ v, double* s,
                                                              double* __restrict__ t, double* partial, GridSync gs,
                                                              double tol, int maxit, PcgResult* res) {
  __shared__ double sm[kSmDoubles];
  Grid g = grid_start(gs, partial, sm);
  double a1[1] = {0.0};
  CSTRIDE(i, F.N) {
    const double ri = sS[i] * bscale * b[i];
    y[i] = 0.0;
    r[i] = ri;
    rh[i] = ri;
    p[i] = ri;
    a1[0] = fma(ri, ri, a1[0]);
  }
  if (!grid_sum<1>(g, a1)) return;   // its barrier also publishes p
  const double rr0 = a1[0];
  double rr = rr0, rho = rr0;
  const double tol2 = tol * tol * rr0;
  int it = 0;
  while (rr0 > 0.0 && rr > tol2 && it < maxit) {
    double a2[2] = {0.0, 0.0};
    CSTRIDE(K, F.N) {
      const double vK = jac_row(F, Js, jd[K], p, K);
      v[K] = vK;
      a2[0] = fma(rh[K], vK, a2[0]);
    }
    if (!grid_sum_x<1, 1>(g, a2, [&](double* o) { o[1] = o[0] != 0.0 ? fast_div(rho, o[0]) : 0.0; })) return;
    const double alpha = a2[1];
    if (!(alpha != 0.0)) break;
    CSTRIDE(K, F.N) s[K] = r[K] - alpha * v[K];
    if (!grid_barrier(g)) return;
    double a3[3] = {0.0, 0.0, 0.0};
    CSTRIDE(K, F.N) {
      const double tK = jac_row(F, Js, jd[K], s, K);
      const double sK = s[K];
      t[K] = tK;
      a3[0] = fma(tK, sK, a3[0]);
      a3[1] = fma(tK, tK, a3[1]);
    }
    if (!grid_sum_x<2, 1>(g, a3, [&](double* o) { o[2] = o[1] != 0.0 ? fast_div(o[0], o[1]) : 0.0; })) return;
    const double omega = a3[2];
    double a4[3] = {0.0, 0.0, 0.0};
    CSTRIDE(K, F.N) {
      const double sK = s[K];
      y[K] += alpha * p[K] + omega * sK;
      const double rK = sK - omega * t[K];
      r[K] = rK;
      a4[0] = fma(rh[K], rK, a4[0]);
      a4[1] = fma(rK, rK, a4[1]);
    }
    if (!grid_sum_x<2, 1>(g, a4, [&](double* o) {
          o[2] = rho != 0.0 && omega != 0.0 ? fast_div(o[0], rho) * fast_div(alpha, omega) : 0.0;
        }))
      return;
    ++it;
    rr = a4[1];
    const double beta = a4[2];
    const bool stop = !(omega != 0.0) || !(a4[0] != 0.0);
    rho = a4[0];
    if (stop) break;
    CSTRIDE(K, F.N) p[K] = r[K] + beta * (p[K] - omega * v[K]);
    if (!grid_barrier(g)) return;
  }
  CSTRIDE(i, F.N) dx[i] = sS[i] * y[i];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    res->err = 0;
    res->iters = it;
    res->rr0 = rr0;
    res->rr = rr;
  }
}

int coop_grid(const void* fn, int n_items, int sm_cap) {
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kPThreads, 0);
  if (per_sm < 1) per_sm = 1;
  if (per_sm > 2) per_sm = 2;                   // few, wide blocks: cheap barriers and partial sums
  int maxb = coop_sms(sm_cap) * per_sm;
  int need = (n_items + kPThreads - 1) / kPThreads;
  if (need < 1) need = 1;
  return need < maxb ? need : maxb;
}

}  // namespace

bool cluster_grid(int& grid, int sms) {
  if (grid > kClusterBlocks) return false;
  int g = 1;
  while (g < grid) g *= 2;
  if (g > sms) return false;
  grid = g;
  return true;
}

cudaError_t launch_persistent(const void* fn, int grid, int threads, void** args, size_t smem, bool cluster,
                              cudaStream_t st) {
  if (!cluster) return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(threads), args, smem, st);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = grid;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

cudaError_t raise_smem_limit(DeviceOnce& once, const void* fn, size_t bytes) {
  int dev = -1;
  if (const cudaError_t e = cudaGetDevice(&dev)) return e;
  return once.run(dev, [&] { return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes); });
}

int coop_sms(int sm_cap) {
  static DeviceOnce once;
  static std::atomic<int> count[DeviceOnce::kDevices];
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  const auto ask = [&] {
    const cudaError_t e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (dev < DeviceOnce::kDevices) count[dev].store(n);
    return e;
  };
  if (once.run(dev, ask) == cudaSuccess && dev < DeviceOnce::kDevices) n = count[dev].load();
  return sm_cap > 0 && sm_cap < n ? sm_cap : n;
}

template <class T>
cudaError_t launch_fine_cg(cudaStream_t st, const FineDev& F, const T* Ts, const double* sdiag, const double* b,
                           double bscale, double* dx, T* y, T* r, T* pa, T* pb, T* q, double* partial, GridSync gs,
                           double tol, int maxit, PcgResult* res) {
  (void)pb;
  const void* fn = (const void*)kp_fine_cg<T>;
  int grid = coop_grid(fn, F.N, gs.sm_cap);
  void* args[] = {(void*)&F, (void*)&Ts, (void*)&sdiag, (void*)&b, (void*)&bscale, (void*)&dx, (void*)&y,
                  (void*)&r, (void*)&pa, (void*)&q, (void*)&partial, (void*)&gs, (void*)&tol,
                  (void*)&maxit, (void*)&res};
  return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kPThreads), args, 0, st);
}
template <class T>
cudaError_t launch_fine_cg_pipe(cudaStream_t st, const FineDev& F, const T* Ts, const double* sdiag, const double* b,
                                double bscale, double* dx, T* y, T* r, T* wa, T* wb, T* z, T* sv, T* p,
                                double* partial, GridSync gs, double tol, int maxit, PcgResult* res) {
  const void* fn = (const void*)kp_fine_cg_pipe<T>;
  int grid = coop_grid(fn, F.N, gs.sm_cap);
  void* args[] = {(void*)&F, (void*)&Ts, (void*)&sdiag, (void*)&b, (void*)&bscale, (void*)&dx, (void*)&y,
                  (void*)&r, (void*)&wa, (void*)&wb, (void*)&z, (void*)&sv, (void*)&p, (void*)&partial, (void*)&gs,
                  (void*)&tol, (void*)&maxit, (void*)&res};
  return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kPThreads), args, 0, st);
}
cudaError_t launch_fine_bicgstab(cudaStream_t st, const FineDev& F, const double* Js, const double* jd,
                                 const double* sS, const double* b, double bscale, double* dx, double* work,
                                 double* partial, GridSync gs, double tol, int maxit, PcgResult* res) {
  const void* fn = (const void*)kp_fine_bicgstab;
  const int grid = coop_grid(fn, F.N, gs.sm_cap);
  const size_t n = (size_t)F.N;
  double *y = work, *r = work + n, *rh = work + 2 * n, *p = work + 3 * n, *v = work + 4 * n, *s = work + 5 * n,
         *t = work + 6 * n;
  void* args[] = {(void*)&F, (void*)&Js, (void*)&jd, (void*)&sS, (void*)&b, (void*)&bscale, (void*)&dx,
                  (void*)&y, (void*)&r, (void*)&rh, (void*)&p, (void*)&v, (void*)&s, (void*)&t, (void*)&partial,
                  (void*)&gs, (void*)&tol, (void*)&maxit, (void*)&res};
  return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kPThreads), args, 0, st);
}
template cudaError_t launch_fine_cg_pipe<double>(cudaStream_t, const FineDev&, const double*, const double*,
                                                 const double*, double, double*, double*, double*, double*, double*,
                                                 double*, double*, double*, double*, GridSync, double, int,
                                                 PcgResult*);
template cudaError_t launch_fine_cg<double>(cudaStream_t, const FineDev&, const double*, const double*,
                                            const double*, double, double*, double*, double*, double*, double*,
                                            double*, double*, GridSync, double, int, PcgResult*);
template cudaError_t launch_fine_cg<float>(cudaStream_t, const FineDev&, const float*, const double*, const double*,
                                           double, double*, float*, float*, float*, float*, float*, double*,
                                           GridSync, double, int, PcgResult*);


// ---- failure detection: the bounded grid barrier on its own ---------------------------------------------------
// Every block except `absent` waits at one grid barrier whose spin limit is `spin_limit` (1024-spin granularity);
// the absent block returns without arriving, so the others give up once the limit is spent, set *gs.err and leave.
// With absent < 0 every block arrives and the barrier completes. *passed counts the blocks whose wait completed.
__global__ void __launch_bounds__(kPThreads) kp_barrier_probe(GridSync gs, double* partial, int absent,
                                                              unsigned long long spin_limit, int* passed) {
  __shared__ double sm[kSmDoubles];
  Grid g = grid_start(gs, partial, sm);
  if ((int)blockIdx.x == absent) return;
  const bool ok = grid_barrier(g, spin_limit);
  if (ok && threadIdx.x == 0) atomicAdd(passed, 1);
}

cudaError_t launch_barrier_probe(cudaStream_t st, GridSync gs, double* partial, int blocks, int absent,
                                 unsigned long long spin_limit, int* passed) {
  const void* fn = (const void*)kp_barrier_probe;
  const int grid = coop_grid(fn, blocks * kPThreads, gs.sm_cap);
  void* args[] = {(void*)&gs, (void*)&partial, (void*)&absent, (void*)&spin_limit, (void*)&passed};
  return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kPThreads), args, 0, st);
}

}  // namespace nlmg
