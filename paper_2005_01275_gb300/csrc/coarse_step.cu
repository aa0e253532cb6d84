// The fused coarse Picard step: one cooperative launch runs whole Picard steps on a coarse level (right-hand side,
// hybridized CG, recovery, clamp, Algorithm 1), with device-side scalars and decisions (see psync.cuh for the grid
// synchronisation, and persist.cu for what the persistent kernels share).
#include <algorithm>
#include <cmath>

#include "kernels.cuh"
#include "persist.cuh"
#include "psync.cuh"

namespace nlmg {

namespace {

constexpr int kCWarps = 15;                       // warps that hold lambdas
constexpr int kCThreads = 32 * (kCWarps + 1);     // and one more, the server: it adds up the grid sums
constexpr int kCServer = kCWarps;
constexpr int kMaxU = 2;                          // lambdas a lane owns at most in the register-resident CG

// ---- H lambda = xi ----------------------------------------------------------------------------------------------
// The interface system H over the lambdas is a sparse matrix of about 28 entries a row, fixed during a solve (its
// entries are the two slots' Hc entries times their cells' kappa). One CG iteration is one product with it, ten FP64
// operations a row and one grid sum, and what bounds it here is FP64 issue (28 + 10 warp operations of 19 clocks per
// 32 rows and SM) and the chain product -> dot products -> block sum -> barrier -> grid sum -> step lengths.
//
// Rows of the register-resident form. gsz lanes (1, 2 or 4) share a row, so a small level still gives every SM a warp
// on each of its four sub-partitions: an entry costs a warp one FP64 operation whether 1 or 32 of its lanes have one,
// so more lanes a row only pay until all sub-partitions are busy. The lane that owns a row keeps its CG state in
// registers; the row's entries and columns lie in shared memory (sv, sc: entry j of a warp's rows at 32 (off + j) +
// lane), so that the only loads an iteration waits for are the gathered values. A level whose entries do not fit there
// runs with its state in memory too (hyb_cg_mem), on all sixteen warps: this form with its entries streamed was slower in
// every case measured (an iteration on 107,842 lambdas and 152 SMs 21.0 us instead of 15.7, 78,098 lambdas 18.8 instead
// of 15.6, 27,429 lambdas on 38 SMs 20.3 instead of 15.4, rows of three flux unknowns an interface, 31,229 lambdas, 25.6
// instead of 15.3). Measured, microseconds per iteration before (rows gathered from the per-cell blocks, every sum waited
// for) and after: 27,429 lambdas 13.9 -> 8.1 on 152 SMs, 3,597 lambdas 8.6 -> 5.2.
template <int U>
struct HRows {
  int l[U];        // lambda (< 0: none)
  int n[U];        // entries a lane, the same in the whole warp
  int off[U];      // first entry / 32
  const double* sv;
  const int* sc;
};

// (H v) of the warp's rows, in every lane of a row's group; entries, then the gathered v, eight at a time.
template <int U>
__device__ __forceinline__ void h_product(const HRows<U>& R, int gsz, const double* v, double (&h)[U]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    double a0 = 0.0;
    const int e0 = 32 * R.off[u] + lane;
    for (int j0 = 0; j0 < R.n[u]; j0 += 8) {
      double hv[8], xv[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const bool in = j0 + q < R.n[u];
        const int e = e0 + 32 * (j0 + q);
        hv[q] = in ? R.sv[e] : 0.0;
        xv[q] = in ? __ldcg(&v[R.sc[e]]) : 0.0;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (j0 + q < R.n[u]) a0 = fma(hv[q], xv[q], a0);
    }
    for (int o = gsz >> 1; o > 0; o >>= 1) a0 += __shfl_xor_sync(0xffffffffu, a0, o);
    h[u] = a0;
  }
}

// Pipelined (Ghysels-Vanroose) Jacobi-preconditioned CG on H lambda = xi with the lambdas in registers. On entry u = M r
// (M = diag(H)^-1) of every lambda is published in lu; r and di = M of the owned rows are given. State per row: lam, r,
// u, w = H u, z = H q, q = M s, s = H p, p; the vector m = M w, which the product n = H m gathers, is published
// double-buffered. Per iteration: n = H m; z = n + beta z; q = m + beta q; s = w + beta s; p = u + beta p;
// lam += alpha p; r -= alpha s; u -= alpha q; w -= alpha z; then gamma = (r, u), delta = (w, u), (r, r) in one
// reduction. The barrier that publishes m also publishes the partial sums; while the other warps form n, the server
// warp adds the partials up and derives beta and alpha, so the serial part of the sum hides behind the product (one
// product is spent in vain at the end). lam is stored in every iteration, so that the recovery reads the final values.
template <int U>
__device__ bool hyb_cg_reg(const HRows<U>& R, int gsz, const double (&xi)[U], const double (&di)[U], double* lam,
                           const double* lu, double* ma, double* mb, Grid& g, double tol, int maxit, int& it_out,
                           double& rr0_out, double& rr_out) {
  __shared__ double sc[4];   // beta, alpha, (r, r), (r_0, r_0)
  __shared__ int stop;
  const int warp = threadIdx.x >> 5;
  const bool own = (threadIdx.x & (gsz - 1)) == 0;
  double r[U], u[U], w[U], z[U], s[U], q[U], p[U], lm[U], n[U];
  double d[3] = {0.0, 0.0, 0.0};
  h_product<U>(R, gsz, lu, w);
#pragma unroll
  for (int k = 0; k < U; ++k) {
    r[k] = xi[k];
    u[k] = xi[k] * di[k];
    z[k] = s[k] = q[k] = p[k] = lm[k] = 0.0;
    if (own && R.l[k] >= 0) {
      ma[R.l[k]] = di[k] * w[k];
      d[0] = fma(r[k], u[k], d[0]);
      d[1] = fma(w[k], u[k], d[1]);
      d[2] = fma(r[k], r[k], d[2]);
    }
  }
  if (!grid_sum_arrive<3>(g, d, kCServer)) return false;
  double* mc = ma;   // published m of the current iteration
  double* mn = mb;
  double tol2 = 0.0, ig = 0.0, ia = 0.0;   // the server's: 1 / gamma and 1 / alpha of the last iteration
  int it = 0;
  while (true) {
    if (warp == kCServer) {
      double t[3];
      grid_sum_finish<3>(g, t);
      if (it == 0) tol2 = tol * tol * t[2];
      const double beta = t[0] * ig;                        // gamma / gamma_old (first: 0)
      const double den = fma(-beta, t[0] * ia, t[1]);       // delta - beta gamma / alpha_old
      const double alpha = den != 0.0 ? t[0] * fast_rcp(den) : 0.0;
      if ((threadIdx.x & 31) == 0) {
        if (it == 0) sc[3] = t[2];
        sc[0] = beta;
        sc[1] = alpha;
        sc[2] = t[2];
        stop = !(sc[3] > 0.0 && t[2] > tol2 && it < maxit) || !(alpha != 0.0);
      }
      __syncthreads();
      ig = t[0] != 0.0 ? fast_rcp(t[0]) : 0.0;
      ia = fast_rcp(alpha);
    } else {
      h_product<U>(R, gsz, mc, n);
      __syncthreads();
    }
    if (stop) break;
    d[0] = d[1] = d[2] = 0.0;
    if (own && R.l[0] >= 0) {
      const double b = sc[0], a = sc[1];
#pragma unroll
      for (int k = 0; k < U; ++k)
        if (k == 0 || R.l[k] >= 0) {
          const double m = di[k] * w[k];
          z[k] = fma(b, z[k], n[k]);
          q[k] = fma(b, q[k], m);
          s[k] = fma(b, s[k], w[k]);
          p[k] = fma(b, p[k], u[k]);
          w[k] = fma(-a, z[k], w[k]);
          mn[R.l[k]] = di[k] * w[k];
          u[k] = fma(-a, q[k], u[k]);
          r[k] = fma(-a, s[k], r[k]);
          lm[k] = fma(a, p[k], lm[k]);
          lam[R.l[k]] = lm[k];
          d[0] = fma(r[k], u[k], d[0]);
          d[1] = fma(w[k], u[k], d[1]);
          d[2] = fma(r[k], r[k], d[2]);
        }
    }
    if (!grid_sum_arrive<3>(g, d, kCServer)) return false;
    double* t = mc;
    mc = mn;
    mn = t;
    ++it;
  }
  it_out = it;
  rr0_out = sc[3];
  rr_out = sc[2];
  __syncthreads();   // sc read by all
  return true;
}

// (H v)_l from the assembled SELL form, for the memory-resident forms: one thread per lambda, the 32 lambdas of a slice
// read their entries coalesced; the entries, then the gathered v, are loaded eight at a time before the products. hsv
// was written earlier in the launch, so it is read through L2.
__device__ __forceinline__ double sell_h_product(const LevelDev& L, const double* hsv, const double* v, int l) {
  double h = 0.0;
  const int w = L.hs_w[l >> 5];
  const int e0 = L.hs_off[l >> 5] + (l & 31);
  for (int j0 = 0; j0 < w; j0 += 8) {
    double hv[8], xv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + 32 * (j0 + u);
      const bool in = j0 + u < w;
      hv[u] = in ? __ldcg(&hsv[e]) : 0.0;
      xv[u] = in ? __ldcg(&v[L.hs_col[e]]) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) h = fma(hv[u], xv[u], h);
  }
  return h;
}

// The same pipelined CG with the lambdas' state in memory (levels with more lambdas than the grid has lanes for).
__device__ bool hyb_cg_mem(const LevelDev& L, const double* hsv, double* lam, double* lr, double* lu, double* pp,
                           double* lq, double* ldinv, const HybPipeBufs<double>& P, Grid& g, double tol2, double rr0,
                           int maxit, int& it_out, double& rr_out) {
  // w = H u, m = M w, and the first reduction
  double d3[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  GSTRIDE(l, L.nlam) {
    const double w = sell_h_product(L, hsv, lu, l);
    const double r = lr[l], u = lu[l];
    P.w[l] = w;
    P.ma[l] = ldinv[l] * w;
    P.z[l] = P.s[l] = lq[l] = pp[l] = 0.0;
    d3[0] = fma(r, u, d3[0]);
    d3[1] = fma(w, u, d3[1]);
    d3[2] = fma(r, r, d3[2]);
  }
  if (!grid_sum_x<3, 2>(g, d3, [&](double* o) {
        o[3] = 0.0;
        o[4] = o[1] != 0.0 ? fast_div(o[0], o[1]) : 0.0;
      }))
    return false;
  double gamma = d3[0], rr = d3[2], beta = d3[3], alpha = d3[4];
  double* mc = P.ma;   // published m of the current iteration
  double* mn = P.mb;
  int it = 0;
  while (rr0 > 0.0 && rr > tol2 && it < maxit) {
    if (!(alpha != 0.0)) break;
    double n5[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    GSTRIDE(l, L.nlam) {
      const double n = sell_h_product(L, hsv, mc, l);
      const double w = P.w[l], m = ldinv[l] * w;
      const double z = n + beta * P.z[l];
      const double q = m + beta * lq[l];
      const double sv = w + beta * P.s[l];
      const double p = lu[l] + beta * pp[l];
      P.z[l] = z;
      lq[l] = q;
      P.s[l] = sv;
      pp[l] = p;
      lam[l] = lam[l] + alpha * p;
      const double r = lr[l] - alpha * sv;
      const double u = lu[l] - alpha * q;
      const double wn = w - alpha * z;
      lr[l] = r;
      lu[l] = u;
      P.w[l] = wn;
      mn[l] = ldinv[l] * wn;
      n5[0] = fma(r, u, n5[0]);
      n5[1] = fma(wn, u, n5[1]);
      n5[2] = fma(r, r, n5[2]);
    }
    if (!grid_sum_x<3, 2>(g, n5, [&](double* o) {
          const double gn = o[0], dn = o[1];
          const double bn = gamma != 0.0 ? fast_div(gn, gamma) : 0.0;
          const double den = dn - fast_div(bn * gn, alpha);
          o[3] = bn;
          o[4] = den != 0.0 ? fast_div(gn, den) : 0.0;
        }))
      return false;
    gamma = n5[0];
    rr = n5[2];
    beta = n5[3];
    alpha = n5[4];
    double* tmp = mc;
    mc = mn;
    mn = tmp;
    ++it;
  }
  it_out = it;
  rr_out = rr;
  return true;
}

// CG with two synchronisations an iteration (tight tolerances: its residual tracks the true one more closely): H z, then
// p = z + beta p and q = H z + beta q (= H p) by recurrence; alpha; lam, r and z = M r; beta. z is published by the
// second reduction's barrier.
__device__ bool hyb_cg_two(const LevelDev& L, const double* hsv, double* lam, double* lr, double* lz, double* pp,
                           double* lq, const double* ldinv, Grid& g, double tol2, double rr0, double rz, int maxit,
                           int& it_out, double& rr_out) {
  double rr = rr0, beta = 0.0;
  int it = 0;
  while (rr0 > 0.0 && rr > tol2 && it < maxit) {
    double a1[2] = {0.0, 0.0};
    GSTRIDE(l, L.nlam) {
      const double hz = sell_h_product(L, hsv, lz, l), zl = lz[l];
      const double pl = it == 0 ? zl : zl + beta * pp[l];
      const double ql = it == 0 ? hz : hz + beta * lq[l];
      pp[l] = pl;
      lq[l] = ql;
      a1[0] = fma(pl, ql, a1[0]);
    }
    if (!grid_sum_x<1, 1>(g, a1, [&](double* o) { o[1] = o[0] != 0.0 ? fast_div(rz, o[0]) : 0.0; })) return false;
    const double alpha = a1[1];
    double a3[3] = {0.0, 0.0, 0.0};
    GSTRIDE(l, L.nlam) {
      lam[l] = alpha * pp[l] + lam[l];
      const double ri = lr[l] - alpha * lq[l];
      const double zi = ri * ldinv[l];
      lr[l] = ri;
      lz[l] = zi;
      a3[0] = fma(ri, zi, a3[0]);
      a3[1] = fma(ri, ri, a3[1]);
    }
    if (!grid_sum_x<2, 1>(g, a3, [&](double* o) { o[2] = rz != 0.0 ? fast_div(o[0], rz) : 0.0; })) return false;
    beta = a3[2];
    rz = a3[0];
    rr = a3[1];
    ++it;
    if (!(alpha != 0.0)) break;
  }
  it_out = it;
  rr_out = rr;
  return true;
}

// The rows of the local saddle inverses (right-hand side, recovery) and of the local blocks (linear parts) are read
// four lanes a row (QSTRIDE): one Picard step with a single CG iteration took 223 us on the 64^3 workload's first coarse
// level and 174 us on its second with a thread a row, 164 and 82 us with four lanes.
// A lane's share (entries gi, gi + 4, ...) of ka times the row S of a cell's local saddle inverse on the owned flux data
// plus kb times the row on the pressure data; loc_own gives a slot's flux unknown where the cell owns it, else -1.
__device__ __forceinline__ double saddle_row(const LevelDev& L, const double* __restrict__ S, int lo, int nl, int po,
                                             int mc, const double* bs, const double* bp, double ka, double kb, int gi) {
  double a = 0.0, b = 0.0;
  for (int t0 = gi; t0 < nl; t0 += 16) {
    double sv[4], xv[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int t = t0 + 4 * q, i = t < nl ? L.loc_own[lo + t] : -1;
      sv[q] = i >= 0 ? S[t] : 0.0;
      xv[q] = i >= 0 ? __ldcg(&bs[i]) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (t0 + 4 * q < nl) a = fma(sv[q], xv[q], a);
  }
  for (int q = gi; q < mc; q += 4) b = fma(S[nl + q], __ldcg(&bp[po + q]), b);
  return fma(ka, a, kb * b);
}
// A lane's share of the row S on C^T lambda of cell c (if_lams: a slot's lambda, complemented where its sign is -1).
__device__ __forceinline__ double lambda_row(const LevelDev& L, const double* __restrict__ S, int c, const double* lam,
                                             int gi) {
  double a = 0.0;
  const int k1 = L.if_off[c + 1];
  for (int k0 = L.if_off[c] + gi; k0 < k1; k0 += 16) {
    double sv[4], xv[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = k0 + 4 * q, ls = k < k1 ? L.if_lams[k] : 0, sg = ls < 0;
      sv[q] = k < k1 ? flip(S[L.if_slot[k]], sg) : 0.0;
      xv[q] = k < k1 ? __ldcg(&lam[sg ? ~ls : ls]) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (k0 + 4 * q < k1) a = fma(sv[q], xv[q], a);
  }
  return a;
}

// The solve of one frozen-coefficient coarse saddle (rhs, Jacobi diagonal, CG on H lambda = xi, local recovery) as a
// device function of the persistent grid. kapc, bs and bp may have been written earlier in the same launch, so they
// are read through L2. form: 0 two synchronisations, 1 pipelined in memory, 2 pipelined in registers. Returns false if
// a grid barrier gave up; `iters` and `rr_out` receive the CG iterations and final (r, r).
template <int U>
__device__ bool hyb_solve_dev(const LevelDev& L, const double* __restrict__ Hc, const double* __restrict__ Sinv,
                              const CoarseStepBufs<double>& B, const HRows<U>& R, int form, int gsz, double* sv, int* scol,
                              Grid& g, double tol, int maxit, int& iters, double& rr0_out, double& rr_out) {
  const double *kapc = B.kapc, *bs = B.nb, *bp = B.nb + L.nflux;
  double *ylam = B.ylam, *ydiag = B.ydiag, *lam = B.lam, *dsig = B.dx, *dp = B.dx + L.nflux;
  const int lane = threadIdx.x & 31, gi = threadIdx.x & (gsz - 1);
  // phase 0: per interface slot k of cell c, u_k = kappa A[k,:] bhat + B[k,:] b_p (signed) and kappa Hc[k,k]
  QSTRIDE(k, L.nif) {
    const bool act = k < L.nif;
    double v = 0.0, kp = 0.0;
    int c = 0, sg = 0;
    if (act) {
      c = L.if_cell[k];
      const int mc = L.m[c], lo = L.loc_off[c], nl = L.loc_off[c + 1] - lo, po = L.p_off[c];
      kp = __ldcg(&kapc[c]);
      sg = L.if_lams[k] < 0;
      v = saddle_row(L, Sinv + L.sad_off[c] + (size_t)L.if_slot[k] * (nl + mc), lo, nl, po, mc, bs, bp, kp, 1.0, lane & 3);
    }
    v = quad_sum(v);
    if (act && (lane & 3) == 0) {
      ylam[k] = flip(v, sg);
      const int k0 = L.if_off[c], ni = L.if_off[c + 1] - k0;
      ydiag[k] = kp * Hc[L.hc_off[c] + (k - k0) * ni + (k - k0)];
    }
  }
  if (form == 2) {   // this kappa's H in shared memory
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int l = R.l[u];
      const int w = l >= 0 ? L.hs_w[l >> 5] : 0, e0 = l >= 0 ? L.hs_off[l >> 5] + (l & 31) : 0;
      const double k0 = l >= 0 ? __ldcg(&kapc[L.lam_c0[l]]) : 0.0, k1 = l >= 0 ? __ldcg(&kapc[L.lam_c1[l]]) : 0.0;
      for (int j = 0; j < R.n[u]; ++j) {
        const int je = gi + gsz * j, d = 32 * (R.off[u] + j) + lane;
        double v = 0.0;
        int c = l >= 0 ? l : 0;
        if (je < w) {
          const int e = e0 + 32 * je, i0 = L.hs_i0[e], i1 = L.hs_i1[e];
          c = L.hs_col[e];
          if (i0 >= 0) v = k0 * Hc[i0];
          if (i1 >= 0) v = fma(k1, Hc[i1], v);
        }
        sv[d] = v;
        scol[d] = c;
      }
    }
  } else {   // the SELL form of H at this kappa (padding entries have no contribution: 0)
    GSTRIDE(l, L.nlam) {
      const double k0 = __ldcg(&kapc[L.lam_c0[l]]), k1 = __ldcg(&kapc[L.lam_c1[l]]);
      const int w = L.hs_w[l >> 5];
      int e = L.hs_off[l >> 5] + (l & 31);
      for (int j = 0; j < w; ++j, e += 32) {
        const int i0 = L.hs_i0[e], i1 = L.hs_i1[e];
        double v = 0.0;
        if (i0 >= 0) v = k0 * Hc[i0];
        if (i1 >= 0) v = fma(k1, Hc[i1], v);
        B.hsv[e] = v;
      }
    }
  }
  if (!grid_barrier(g)) return false;
  int it = 0;
  if (form == 2) {
    double xi[U], di[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int l = R.l[u];
      xi[u] = di[u] = 0.0;
      if (l >= 0 && gi == 0) {
        const int y0 = L.lam_y0[l], y1 = L.lam_y1[l];
        xi[u] = __ldcg(&ylam[y0]) + __ldcg(&ylam[y1]);
        di[u] = fast_rcp(__ldcg(&ydiag[y0]) + __ldcg(&ydiag[y1]));
        B.lz[l] = xi[u] * di[u];
        lam[l] = 0.0;
      }
    }
    if (!grid_barrier(g)) return false;
    if (!hyb_cg_reg<U>(R, gsz, xi, di, lam, B.lz, B.pipe.ma, B.pipe.mb, g, tol, maxit, it, rr0_out, rr_out)) return false;
  } else {
    double a2[2] = {0.0, 0.0};
    GSTRIDE(l, L.nlam) {
      const double xi = __ldcg(&ylam[L.lam_y0[l]]) + __ldcg(&ylam[L.lam_y1[l]]);
      const double di = fast_rcp(__ldcg(&ydiag[L.lam_y0[l]]) + __ldcg(&ydiag[L.lam_y1[l]]));
      B.ldinv[l] = di;
      lam[l] = 0.0;
      B.lr[l] = xi;
      const double zi = xi * di;
      B.lz[l] = zi;
      a2[0] = fma(xi, zi, a2[0]);
      a2[1] = fma(xi, xi, a2[1]);
    }
    if (!grid_sum<2>(g, a2)) return false;
    const double rr0 = a2[1], tol2 = tol * tol * rr0;
    rr0_out = rr0;
    if (form == 1) {
      if (!hyb_cg_mem(L, B.hsv, lam, B.lr, B.lz, B.pa, B.lq, B.ldinv, B.pipe, g, tol2, rr0, maxit, it, rr_out)) return false;
    } else {
      if (!hyb_cg_two(L, B.hsv, lam, B.lr, B.lz, B.pa, B.lq, B.ldinv, g, tol2, rr0, a2[0], maxit, it, rr_out)) return false;
    }
  }
  // recovery: sigma^c = kappa A w + B b_p, p_c = B^T w + C b_p / kappa with w = bhat - C^T lambda: four lanes per owned
  // local flux slot (rows y < nyl) and per pressure unknown (the rest)
  QSTRIDE(y, L.nyl + L.np) {
    const bool press = y >= L.nyl;
    const int i = y >= L.nyl + L.np ? -1 : press ? y - L.nyl : L.loc_own[y];
    double v = 0.0;
    if (i >= 0) {
      const int c = press ? L.p_cell[i] : L.slot_cell[y];
      const int mc = L.m[c], lo = L.loc_off[c], nl = L.loc_off[c + 1] - lo, po = L.p_off[c];
      const double* Su = Sinv + L.sad_off[c] + (size_t)(press ? nl + i - po : y - lo) * (nl + mc);
      const double kp = __ldcg(&kapc[c]);
      const double w = lambda_row(L, Su, c, lam, lane & 3);
      v = press ? saddle_row(L, Su, lo, nl, po, mc, bs, bp, 1.0, fast_rcp(kp), lane & 3) - w
                : saddle_row(L, Su, lo, nl, po, mc, bs, bp, kp, 1.0, lane & 3) - kp * w;
    }
    v = quad_sum(v);
    if (i >= 0 && (lane & 3) == 0) (press ? dp : dsig)[i] = v;
  }
  iters = it;
  return true;
}

// ---- fused coarse Picard step -------------------------------------------------------------------------------
// The coarse operator (Prop. 1, eq. structure) is linear in [sigma; p] once kappa is fixed: with kappa_c =
// kappa((Pi~ p)_c), A(x)_sigma,i = sum over the (one or two) owner slots y of flux unknown i of
// (M_c sigma_c)_u / kappa_c + (D_c^T p_c)_u and A(x)_p,i = (D_c sigma_c)_i. Algorithm 1 evaluates A at x + s dx for
// several s; the linear parts of x and of dx (LinParts) are computed once, and each trial is then one pass over the
// flux and pressure unknowns -- (ms_x + s ms_dx) / kappa(pb_x + s pb_dx) + ds_x + s ds_dx -- and one reduction,
// instead of a whole operator evaluation with two synchronisations. On this part the FP64 products of an
// evaluation and its synchronisations are what a coarse step costs, not its bytes.

// Linear parts of v (read through L2: v may have been written earlier in the launch). With shift != 0 the parts
// `acc` first take acc += shift * out (the previous step's accepted trial; the same lane owns both entries).
__device__ void lin_parts_pass(const LevelDev& L, const double* v, LinParts out, LinParts acc, double shift) {
  const bool fold = nonzero(shift);
  const double* vs = v;
  const double* vp = v + L.nflux;
  const int gi = threadIdx.x & 3;
  // a lane's share of a row M of nl entries on the cell's fluxes (four entries in flight)
  auto flux_row = [&](const double* __restrict__ M, int lo, int nl) -> double {
    double m = 0.0;
    for (int t0 = gi; t0 < nl; t0 += 16) {
      double mv[4], xv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int t = t0 + 4 * q;
        mv[q] = t < nl ? M[t] : 0.0;
        xv[q] = t < nl ? __ldcg(&vs[L.loc[lo + t]]) : 0.0;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (t0 + 4 * q < nl) m = fma(mv[q], xv[q], m);
    }
    return m;
  };
  // rows y < nyl: local flux slots; the rest: pressure unknowns
  QSTRIDE(y, L.nyl + L.np) {
    const bool act = y < L.nyl + L.np, press = y >= L.nyl;
    const int i = y - L.nyl;
    double m = 0.0, d = 0.0;
    if (act) {
      const int c = press ? L.p_cell[i] : L.slot_cell[y];
      const int lo = L.loc_off[c], nl = L.loc_off[c + 1] - lo, mc = L.m[c], po = L.p_off[c];
      const int u = press ? i - po : y - lo;
      const double* D = L.Dloc + L.dmat_off[c];
      m = flux_row(press ? D + (size_t)u * nl : L.Mloc + L.mat_off[c] + (size_t)u * nl, lo, nl);
      if (!press)
        for (int q = gi; q < mc; q += 4) d = fma(D[q * nl + u], __ldcg(&vp[po + q]), d);
    }
    m = quad_sum(m);
    d = quad_sum(d);
    if (act && gi == 0) {
      if (press) {
        if (fold) acc.dr[i] = fma(shift, out.dr[i], acc.dr[i]);
        out.dr[i] = m;
      } else {
        if (fold) {
          acc.ms[y] = fma(shift, out.ms[y], acc.ms[y]);
          acc.ds[y] = fma(shift, out.ds[y], acc.ds[y]);
        }
        out.ms[y] = m;
        out.ds[y] = d;
      }
    }
  }
  TSTRIDE(c, L.nc) {
    const int po = L.p_off[c];
    double pb = 0.0;
    for (int q = 0; q < L.m[c]; ++q) pb = fma(L.w[po + q], __ldcg(&vp[po + q]), pb);
    if (fold) acc.pb[c] = fma(shift, out.pb[c], acc.pb[c]);
    out.pb[c] = pb;
  }
}

// A(x + s dx) - b from the linear parts (dir is not read when s == 0), for flux unknown i / pressure unknown i.
__device__ __forceinline__ double trial_flux_row(const LevelDev& L, const LinParts& bx, const LinParts& dx, double s,
                                                 bool nz, const double* b, int kind, double a, int i) {
  double v = 0.0;
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const int y = side == 0 ? L.f_y0[i] : L.f_y1[i];
    if (y < 0) continue;
    const int c = L.slot_cell[y];
    double pb = __ldcg(&bx.pb[c]), m = __ldcg(&bx.ms[y]), d = __ldcg(&bx.ds[y]);
    if (nz) {
      pb = fma(s, __ldcg(&dx.pb[c]), pb);
      m = fma(s, __ldcg(&dx.ms[y]), m);
      d = fma(s, __ldcg(&dx.ds[y]), d);
    }
    v += fma(m, inv_kappa_of(pb, kind, a), d);
  }
  return v - __ldcg(&b[i]);
}
__device__ __forceinline__ double trial_p_row(const LevelDev& L, const LinParts& bx, const LinParts& dx, double s, bool nz,
                                              const double* b, int i) {
  double d = __ldcg(&bx.dr[i]);
  if (nz) d = fma(s, __ldcg(&dx.dr[i]), d);
  return d - __ldcg(&b[L.nflux + i]);
}

// r = A(x + s dx) - b and nb = -r at a trial point; returns this thread's share of ||r||^2.
__device__ double trial_pass(const LevelDev& L, const CoarseStepBufs<double>& B, double s, int kind, double a) {
  const bool nz = nonzero(s);
  double acc = 0.0;
  GSTRIDE(i, L.nflux) {
    const double v = trial_flux_row(L, B.base, B.dir, s, nz, B.b, kind, a, i);
    B.r[i] = v;
    B.nb[i] = flip(v, 1);
    acc = fma(v, v, acc);
  }
  TSTRIDE(i, L.np) {
    const double v = trial_p_row(L, B.base, B.dir, s, nz, B.b, i);
    B.r[L.nflux + i] = v;
    B.nb[L.nflux + i] = flip(v, 1);
    acc = fma(v, v, acc);
  }
  return acc;
}

// Makes x + s dx the iterate: kappa per cell at the new point, x += s dx, and r and nb unless the last trial was there
// (`at_trial`). The linear parts of x are left as they were (the next pass over the step's direction adds s times the
// old direction's).
__device__ void accept_pass(const LevelDev& L, const CoarseStepBufs<double>& B, double s, bool at_trial, int kind,
                            double a) {
  const bool nz = nonzero(s);
  if (!at_trial) (void)trial_pass(L, B, s, kind, a);
  TSTRIDE(c, L.nc) {
    double pb = __ldcg(&B.base.pb[c]);
    if (nz) pb = fma(s, __ldcg(&B.dir.pb[c]), pb);
    B.kapc[c] = kappa_of(pb, kind, a);
  }
  if (nz) {
    const int nx = L.nflux + L.np;
    GSTRIDE(i, nx) B.x[i] = fma(s, __ldcg(&B.dx[i]), B.x[i]);
  }
}

// The scalars of a coarse step. Only warp 0 computes with them (a scalar FP64 operation in all sixteen warps costs the SM
// 300 clocks, a square root 2,800: together a third of a step on a small level); the others follow the outcome it
// publishes with each sum.
struct StepScalars {
  double rn, r0;   // ||A(x) - b||, and at the start of the Picard steps (warp 0)
  double step;     // the accepted scaling (0: every trial was non-finite, x is kept)
  bool at_trial;   // the last trial evaluated is the accepted one
  bool done;       // the coarsest level's stopping test holds at x
};

__device__ __forceinline__ bool step_done(const CoarseStepParams& P, double rn, double r0) {
  return P.coarsest && (rn <= P.tol_rel * r0 || rn <= P.tol_abs);
}

// Algorithm 1 from x (residual norm S.rn) along s0 dx, with trial residuals from the linear parts; a non-finite trial counts
// as +infinity. `first`: S.rn at the accepted point is also the start value of the stopping test.
__device__ bool backtrack_lin(const LevelDev& L, const CoarseStepBufs<double>& B, const CoarseStepParams& P, double s0,
                              bool first, StepScalars& S, int& trials, Grid& g) {
  double s = 1.0, r_s = HUGE_VAL;   // accepted so far (warp 0)
  double s_try = s0;
  int n = -1;                       // halvings accepted (-1: the full step is being tried)
  while (true) {
    // {sum, step to try or accepted, outcome: bit 0 decided, bit 1 the last trial is the accepted one, bit 2 done}
    double v[3] = {trial_pass(L, B, s_try, P.kind, P.a), 0.0, 0.0};
    ++trials;
    if (!grid_sum_x<1, 2>(g, v, [&](double* o) {
          double r = sqrt(o[0]);
          if (!finite_bits(r)) r = HUGE_VAL;
          int code = 0;
          if (n < 0 || !(r > P.bt_theta * r_s)) {   // the full step, or a halving Algorithm 1 keeps
            if (n >= 0) s *= 0.5;
            ++n;
            r_s = r;
            if (!(r_s > S.rn && n < P.bt_nmax)) code = 3;
          } else {
            code = 1;
          }
          double next = 0.5 * s * s0;
          if (code) {
            const bool none = r_s == HUGE_VAL;
            next = none ? 0.0 : s * s0;
            if (none) code = 1;
            else S.rn = r_s;
            if (first) S.r0 = S.rn;
            if (step_done(P, S.rn, S.r0)) code |= 4;
          }
          o[1] = next;
          o[2] = __hiloint2double(0, code);
        }))
      return false;
    s_try = v[1];
    const int code = __double2loint(v[2]);
    if (code) {
      S.step = s_try;
      S.at_trial = (code & 2) != 0;
      S.done = (code & 4) != 0;
      return true;
    }
  }
}

// One launch. On entry x (and, with backtrack_first, the correction in dx and ||A(x) - b|| in rn_in); on exit x, r,
// nb = -r and kappa per cell at the final x.
template <int U>
__global__ void __launch_bounds__(kCThreads, 1) kp_coarse_step(LevelDev L, const double* __restrict__ Hc,
                                                               const double* __restrict__ Sinv, CoarseStepBufs<double> B,
                                                               CoarseStepParams P, double* partial, GridSync gs, int form,
                                                               int gsz, int staged, CoarseStepResult* res) {
  __shared__ double sm[kSmDoubles];
  __shared__ int ew[U * kCWarps];
  extern __shared__ double dyn[];   // the staged entries: values, then columns
  Grid g = grid_start(gs, partial, sm);
  HRows<U> R;
  {
    // rows of this thread: item i = ((warp + kCWarps u) gridDim + block) 32 + lane, gsz consecutive items a lambda
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = (int)(((warp + kCWarps * u) * gridDim.x + blockIdx.x) * 32u) + lane;
      R.l[u] = form == 2 && warp < kCWarps && i < L.nlam * gsz ? i / gsz : -1;
      const int w = R.l[u] >= 0 ? (L.hs_w[R.l[u] >> 5] + gsz - 1) / gsz : 0;
      R.n[u] = __reduce_max_sync(0xffffffffu, w);
      if (lane == 0 && warp < kCWarps) ew[u * kCWarps + warp] = R.n[u];
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < U; ++u) {
      int o = 0;
      for (int k = 0; k < u * kCWarps + min(warp, kCWarps); ++k) o += ew[k];
      R.off[u] = o;
    }
    R.sv = dyn;
    R.sc = (const int*)(dyn + staged);
  }
  int iters = 0, steps = 0, evals = 0, trials = 0, bad = 0;
  StepScalars S{P.rn_in, P.rn_in, 0.0, false, false};
  double pending = 0.0;   // accepted step not yet added to the linear parts of x
  // linear parts of x (and of the given correction)
  lin_parts_pass(L, B.x, B.base, B.base, 0.0);
  ++evals;
  if (P.backtrack_first) {
    lin_parts_pass(L, B.dx, B.dir, B.dir, 0.0);
    ++evals;
  }
  if (!grid_barrier(g)) return;
  if (P.backtrack_first) {
    if (!backtrack_lin(L, B, P, 1.0, true, S, trials, g)) return;
    accept_pass(L, B, S.step, S.at_trial, P.kind, P.a);   // r, nb, kappa at the new x
    pending = S.step;
    if (!grid_barrier(g)) return;
  } else {
    double v[2] = {trial_pass(L, B, 0.0, P.kind, P.a), 0.0};
    accept_pass(L, B, 0.0, true, P.kind, P.a);
    if (!grid_sum_x<1, 1>(g, v, [&](double* o) {
          S.rn = S.r0 = sqrt(o[0]);
          o[1] = __hiloint2double(0, (finite_bits(S.rn) ? 0 : 1) | (step_done(P, S.rn, S.r0) ? 4 : 0));
        }))
      return;
    const int code = __double2loint(v[1]);
    bad = code & 1;
    S.done = (code & 4) != 0;
  }
  for (int k = 0; k < P.nsteps && !bad && !S.done; ++k) {
    int it = 0;
    double rr0 = 0.0, rr = 0.0;
    if (!hyb_solve_dev<U>(L, Hc, Sinv, B, R, form, gsz, dyn, (int*)(dyn + staged), g, P.lin_tol, P.maxit, it, rr0, rr))
      return;
    iters += it;
    if (!finite_bits(rr)) {
      bad = 2;
      break;
    }
    if (!grid_barrier(g)) return;   // dx complete
    // linear parts of dx (after folding the previous accepted step into those of x), and the clamp on Pi~ dp
    lin_parts_pass(L, B.dx, B.dir, B.base, pending);
    ++evals;
    double s0 = 1.0;
    if (P.dp_clamp > 0.0) {
      double m = 0.0;
      TSTRIDE(c, L.nc) m = fmax(m, fabs(B.dir.pb[c]));   // written by this thread just above
      if (!grid_max(g, m, [&](double v) { return v > P.dp_clamp ? fast_div(P.dp_clamp, v) : 1.0; })) return;
      s0 = m;
    } else if (!grid_barrier(g)) {
      return;
    }
    if (!backtrack_lin(L, B, P, s0, false, S, trials, g)) return;
    accept_pass(L, B, S.step, S.at_trial, P.kind, P.a);
    pending = S.step;
    if (!grid_barrier(g)) return;   // r, nb, kappa and x complete
    ++steps;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    res->err = 0;
    res->rn = S.rn;
    res->iters = iters;
    res->steps = steps;
    res->res_evals = evals;
    res->bad = bad;
    res->trials = trials;
  }
}

}  // namespace

cudaError_t launch_coarse_step(cudaStream_t st, const LevelDev& L, const double* Hc, const double* Sinv,
                               const CoarseStepBufs<double>& B, const CoarseStepParams& P, double* partial, GridSync gs,
                               CoarseStepResult* res, bool* sell) {
  constexpr size_t kMaxDyn = 200 * 1024;
  const void* fns[kMaxU] = {(const void*)kp_coarse_step<1>, (const void*)kp_coarse_step<2>};
  static DeviceOnce limits[kMaxU];
  for (int u = 0; u < kMaxU; ++u)
    if (const cudaError_t e = raise_smem_limit(limits[u], fns[u], kMaxDyn)) return e;
  const int sms = coop_sms(gs.sm_cap);
  // A small level runs as one cluster of up to eight blocks, whose barrier costs a quarter of the grid's: worth it while
  // the FP64 work on eight SMs stays small beside it. In row entries and operations a lambda: 163 lambdas of a 2D level
  // (3.7k) gain, 900 (21k: 262 -> 282 us a step) and 482 of a 3D level (28k: 1,046 -> 1,171 us a solve) lose.
  const bool small = (long)L.nlam * (L.hs_wmax + 13) <= 12000;
  const int most = small ? std::min(sms, kClusterBlocks) : sms;
  // lanes per lambda: as many as leave one warp of rows per sub-partition (four per SM)
  int gsz = 4;
  while (gsz > 1 && (long)L.nlam * gsz > 128L * most) gsz /= 2;
  // blocks: four warps' worth of the level's largest item count each
  long items = (long)L.nlam * gsz;
  for (long v : {(long)L.nif, (long)L.nyl, (long)L.np, (long)L.nflux + L.np, (long)L.nc})
    if (v > items) items = v;
  int grid = (int)std::max(1L, std::min((long)most, (items + 127) / 128));
  gs.cluster = cluster_grid(grid, sms) ? 1 : 0;
  // form: registers when every lambda gets lanes in at most kMaxU passes of the grid and the rows' entries fit in shared
  // memory, else memory; two synchronisations when a tight solve is asked for
  int form = B.pipe.ma ? 1 : 0, U = 1, staged = 0;
  if (form == 1 && L.nlam > 0 && (long)L.nlam <= (long)grid * 32 * kCWarps * kMaxU) {
    const long warps = ((long)L.nlam * gsz + 31) / 32;              // of rows
    const long per = (warps + grid - 1) / grid;                     // on one SM
    const long entries = per * 32 * ((L.hs_wmax + gsz - 1) / gsz);
    if ((size_t)entries * 12 <= kMaxDyn) {
      form = 2;
      staged = (int)entries;
      U = per > kCWarps ? 2 : 1;
    }
  }
  if (form != 2) gsz = 1;
  if (sell) *sell = form != 2;
  const void* fn = fns[U - 1];
  void* args[] = {(void*)&L, (void*)&Hc, (void*)&Sinv, (void*)&B, (void*)&P, (void*)&partial, (void*)&gs,
                  (void*)&form, (void*)&gsz, (void*)&staged, (void*)&res};
  return launch_persistent(fn, grid, kCThreads, args, (size_t)staged * 12, gs.cluster != 0, st);
}

}  // namespace nlmg
