// Linear multigrid preconditioner for the level-0 Krylov solves (see mg.cuh), and the preconditioned CG / BiCGStab
// that use it, each captured once per context as CUDA graphs with a device-side conditional while loop.
//
// Every reduction is deterministic: per-block partial sums, then the grid's last block adds the partials, both in
// integers (isum.cuh; the arrival counter is reset by that block, so graphs replay). Maxima are exact.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <set>
#include <string>
#include <type_traits>
#include <vector>

#include "isum.cuh"
#include "mg.cuh"
#include "persist.cuh"

namespace nlmg {

namespace {

static_assert(kMgDegFine <= kMgMaxDeg && kMgDegCoarse <= kMgMaxDeg, "Chebyshev coefficient table too small");
static_assert(kMgMaxLevels * kMgMaxDeg <= 32, "the coefficient table kernel runs one warp");

constexpr int kT = 256;               // threads per block of the preconditioner kernels
constexpr int kMaxRedBlocks = 1024;   // grid cap of the reduction kernels (partials summed by one block)

#define MG_MB_SWITCH(mb, CALL)                                                     \
  switch (mb) {                                                                    \
    case 1: { constexpr int MB = 1; CALL; } break;                                 \
    case 2: { constexpr int MB = 2; CALL; } break;                                 \
    case 3: { constexpr int MB = 3; CALL; } break;                                 \
    case 4: { constexpr int MB = 4; CALL; } break;                                 \
    case 5: { constexpr int MB = 5; CALL; } break;                                 \
    case 6: { constexpr int MB = 6; CALL; } break;                                 \
    case 7: { constexpr int MB = 7; CALL; } break;                                 \
    default: { constexpr int MB = 8; CALL; } break;                                \
  }

inline int blocks_for(long n, int cap = 1 << 20) {
  long b = (n + kT - 1) / kT;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (int)b;
}

// ---------------------------------------------------------------------------------------------------------------
// reductions

// Sums NV values over the grid: block sums to part[block][k]; the last block to arrive adds the partials (at most
// kMaxRedBlocks) and returns true in its warp 0 with the sums in out. The counter is left at zero. On
// the integer pipes (isum.cuh): block trees, 1,024 partials and their trees took 2 us at the end of a kernel.
template <int NV>
__device__ bool reduce_last(double (&v)[NV], double* part, unsigned* cnt, double (&out)[NV]) {
  __shared__ ISum sh[NV * 32];
  __shared__ int last;
  constexpr int M = kMaxRedBlocks / kT;
  const int lane = threadIdx.x & 31;
  double a[NV][1], s[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) a[k][0] = v[k];
  block_sums<NV, 1>(a, s, sh, kT / 32);
  if (threadIdx.x < NV) {
    double mine = s[0];
#pragma unroll
    for (int k = 1; k < NV; ++k) mine = lane == k ? s[k] : mine;
    part[(size_t)blockIdx.x * NV + lane] = mine;
  }
  __syncwarp();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(cnt, 1u) == gridDim.x - 1 ? 1 : 0;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double p[NV][M];
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const int b = (int)threadIdx.x + kT * j;
#pragma unroll
    for (int k = 0; k < NV; ++k) p[k][j] = b < (int)gridDim.x ? __ldcg(&part[(size_t)b * NV + k]) : 0.0;
  }
  block_sums<NV, M>(p, out, sh, kT / 32);
  if (threadIdx.x == 0) *cnt = 0u;
  return threadIdx.x < 32;
}

__device__ __forceinline__ void atomic_max_pos(float* addr, float v) {
  // non-negative floats order like their bit patterns
  atomicMax((unsigned*)addr, __float_as_uint(v));
}

// Chebyshev coefficients of step k on [lam / alpha, lam] (see oracle/precond.py): k = 0 -> (0, 1 / theta);
// k >= 1 -> (rho_k rho_{k-1}, 2 rho_k / delta).
__device__ __forceinline__ void cheb_coef(float lam, int k, float& c1, float& c2) {
  const double lmax = lam, lmin = lam / kMgAlpha;
  const double theta = 0.5 * (lmax + lmin), delta = 0.5 * (lmax - lmin), sigma = theta / delta;
  if (k == 0) {
    c1 = 0.0f;
    c2 = (float)(1.0 / theta);
    return;
  }
  double rho = 1.0 / sigma, rho_prev = rho;
  for (int i = 1; i <= k; ++i) {
    rho_prev = rho;
    rho = 1.0 / (2.0 * sigma - rho);
  }
  c1 = (float)(rho * rho_prev);
  c2 = (float)(2.0 * rho / delta);
}

// The coefficients of every level and step, computed once per setup from the Gershgorin bounds (k_cheb_table):
// tab[(l * kMgMaxDeg + k) * 2 + {0, 1}] = (c1, c2) of cheb_coef.
__device__ __forceinline__ void cheb_tab(const float* __restrict__ tab, int l, int k, float& c1, float& c2) {
  c1 = tab[(l * kMgMaxDeg + k) * 2];
  c2 = tab[(l * kMgMaxDeg + k) * 2 + 1];
}

__device__ __forceinline__ bool stop(const int* done) { return done && *((volatile const int*)done) != 0; }

// Programmatic dependent launch: wait until the preceding kernel of the stream (or graph edge) has finished and its
// writes are visible, then let the next kernel start its launch (it waits the same way before it reads anything).
// Without a programmatic predecessor the wait returns at once.
// What a kernel loads before that (the matrix entries, indices and transfers of its first items) is older than its
// predecessor: a kernel only starts once its predecessor has waited for the one before, and setup and hierarchy are
// several kernels back. So those loads overlap the predecessor, and what is left after the wait is the vectors.
__device__ __forceinline__ void pdl_start() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ float pval(const float* __restrict__ p, size_t i) { return p[i]; }
__device__ __forceinline__ float pval(const __nv_bfloat16* __restrict__ p, size_t i) { return __bfloat162float(p[i]); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// MB consecutive floats from p into v: 16-byte loads when MB % 4 == 0, 8-byte loads when MB is even (the caller
// guarantees p is aligned accordingly: every array here is its own allocation, and a block row or a cell's vector
// segment starts at a multiple of MB floats).
template <int MB>
__device__ __forceinline__ void ld_seg(const float* p, float (&v)[MB]) {
  if constexpr (MB % 4 == 0) {
#pragma unroll
    for (int k = 0; k < MB / 4; ++k) {
      const float4 t = reinterpret_cast<const float4*>(p)[k];
      v[4 * k] = t.x;
      v[4 * k + 1] = t.y;
      v[4 * k + 2] = t.z;
      v[4 * k + 3] = t.w;
    }
  } else if constexpr (MB % 2 == 0) {
#pragma unroll
    for (int k = 0; k < MB / 2; ++k) {
      const float2 t = reinterpret_cast<const float2*>(p)[k];
      v[2 * k] = t.x;
      v[2 * k + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < MB; ++k) v[k] = p[k];
  }
}

// MB consecutive BF16 transfer entries from p, widened to float: 4-byte pair loads when MB is even.
template <int MB>
__device__ __forceinline__ void ld_seg(const __nv_bfloat16* p, float (&v)[MB]) {
  if constexpr (MB % 2 == 0) {
#pragma unroll
    for (int k = 0; k < MB / 2; ++k) {
      const float2 t = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(p)[k]);
      v[2 * k] = t.x;
      v[2 * k + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < MB; ++k) v[k] = __bfloat162float(p[k]);
  }
}

// ---------------------------------------------------------------------------------------------------------------
// setup kernels (once per frozen matrix)

// FP32 copy of the level-0 matrix (off-diagonal entries -T in the SELL layout, diagonal, its inverse) and the
// Gershgorin bound max_K (A_KK + sum_L T_KL) / A_KK of D^-1 A: 2 where a cell has no Dirichlet face, for its diagonal is
// that sum. One pass over the matrix; values are rounded to FP32 on the integer pipe (10^6 cells: conversions, sums and
// two divisions took 60 us, this takes 16).
__global__ void k_fine_vals(FineDev F, const double* __restrict__ Tval, const double* __restrict__ diagT,
                            float* __restrict__ a0off, float* __restrict__ a0diag, float* __restrict__ a0dinv,
                            float* lam) {
  pdl_start();
  float g = 0.0f;
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < F.N; K += gridDim.x * blockDim.x) {
    const int w = F.sell_w[K >> 5], e0 = F.sell_off[K >> 5] + (K & 31);
    for (int j = 0; j < w; ++j) a0off[e0 + 32 * j] = -narrow(Tval[e0 + 32 * j]);
    const double dg = diagT[K], di = fast_rcp(dg);
    a0diag[K] = narrow(dg);
    a0dinv[K] = narrow(di);
    float b = 2.0f;
    if (F.dir_off[K + 1] > F.dir_off[K]) {
      double s = 0.0;
      for (int j = 0; j < w; ++j) s += Tval[e0 + 32 * j];
      b = (float)((dg + s) / dg);
    } else if (!(dg > 0.0)) {
      b = (float)((dg + dg) / dg);
    }
    g = fmaxf(g, b);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) g = fmaxf(g, __shfl_down_sync(0xffffffffu, g, off));
  if ((threadIdx.x & 31) == 0) atomic_max_pos(&lam[0], g);
}

// Sums a whole n-value array over a group of LN = 16 or 32 lanes: after each step a lane keeps the half of the values its
// partner gave up, so 16 values take 15 or 16 shuffles instead of 64 or 80. Entry i = the returned lane index's value:
// lane t of a 16-lane group holds the sum of value t (both halves of a 32-lane group hold it).
template <int LN>
__device__ __forceinline__ float group_sum16(float (&v)[16]) {
  const int lane = threadIdx.x & (LN - 1);
#pragma unroll
  for (int h = 8; h > 0; h >>= 1) {
    const bool up = (lane & h) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float keep = up ? v[i + h] : v[i], give = up ? v[i] : v[i + h];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, h);
    }
  }
  if (LN == 32) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 16);
  return v[0];
}

// Level-1 Galerkin blocks from the fine faces: lane t of a group takes contributions t, t + lanes, ... of the
// block's list and accumulates the whole MB x MB block; a fixed shuffle tree then adds the lanes' blocks. The
// contributions (K, L, e, type): 0 interior face inside the aggregate, T (P_K - P_L)(P_K - P_L)^T; 1 face to another
// aggregate seen from this one's cell K, T P_K P_K^T; 2 the off-diagonal part, -T P_K P_L^T; 3 Dirichlet face (L = its
// entry in the Dirichlet list), h P_K P_K^T with h = Ups_K / r_K, r = 1 / kappa. T is read as the FP32 entry of the level-0
// matrix. With four modes a group is half a warp (an off-diagonal block has about 16 faces) and its 16 lanes end up with
// one entry of the block each; 10^6 cells took 261 us with a warp a block, FP64 entries and a tree per entry.
template <int MB, class PT>
__global__ void k_asm1(int nblk, const int* __restrict__ off, const int4* __restrict__ list,
                       const PT* __restrict__ P0, const float* __restrict__ a0off, const double* __restrict__ r,
                       const double* __restrict__ dir_ups, float* __restrict__ aval) {
  pdl_start();
  constexpr int LN = MB == 4 ? 16 : 32;
  const int lane = threadIdx.x & (LN - 1), per = 32 / LN;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int b0 = warp * per; b0 < nblk; b0 += nw * per) {
    const int b = b0 + (int)((threadIdx.x & 31) / LN);
    float acc[MB * MB];
#pragma unroll
    for (int i = 0; i < MB * MB; ++i) acc[i] = 0.0f;
    const int c1 = b < nblk ? off[b + 1] : 0;
    for (int c = b < nblk ? off[b] + lane : 0; c < c1; c += LN) {
      const int4 t = list[c];
      float pk[MB], pl[MB];
      ld_seg<MB>(P0 + (size_t)t.x * MB, pk);
      float w;
      if (t.w == 3) {
        w = narrow(fast_div(dir_ups[t.y], r[t.x]));
#pragma unroll
        for (int j = 0; j < MB; ++j) pl[j] = pk[j];
      } else {
        w = -a0off[t.z];
        ld_seg<MB>(P0 + (size_t)t.y * MB, pl);
        if (t.w == 0) {
#pragma unroll
          for (int j = 0; j < MB; ++j) {
            pk[j] -= pl[j];
            pl[j] = pk[j];
          }
        } else if (t.w == 1) {
#pragma unroll
          for (int j = 0; j < MB; ++j) pl[j] = pk[j];
        } else {
          w = -w;
        }
      }
#pragma unroll
      for (int u = 0; u < MB; ++u)
#pragma unroll
        for (int v = 0; v < MB; ++v) acc[u * MB + v] = fmaf(w * pk[u], pl[v], acc[u * MB + v]);
    }
    __syncwarp();
    if constexpr (MB == 4) {
      const float s = group_sum16<LN>(acc);
      if (b < nblk) aval[(size_t)b * 16 + lane] = s;
    } else {
#pragma unroll
      for (int i = 0; i < MB * MB; ++i) acc[i] = warp_sum(acc[i]);
#pragma unroll
      for (int i = 0; i < MB * MB; ++i)
        if ((i & 31) == lane) aval[(size_t)b * MB * MB + i] = acc[i];
    }
  }
}

// Unit diagonal on the padded modes of every diagonal block of level l (cells with fewer modes than mb).
__global__ void k_pad_diag(int nc, int mb, const int* __restrict__ dpos, const int* __restrict__ mcnt,
                           float* __restrict__ aval) {
  pdl_start();
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
    float* B = aval + (size_t)dpos[c] * mb * mb;
    for (int u = mcnt[c]; u < mb; ++u) {
      for (int v = 0; v < mb; ++v) B[u * mb + v] = B[v * mb + u] = 0.0f;
      B[u * mb + u] = 1.0f;
    }
  }
}

// Level-l Galerkin blocks (l >= 2) from the level-(l-1) blocks: block (A, B) = sum over (c, d) with agg(c) = A,
// agg(d) = B of P_c^T A_cd P_d, P_c the mbf x MB transfer block of level-(l-1) cell c. One warp per block, lanes
// taking the contributions in turn, then a fixed shuffle tree.
template <int MB, class PT>
__global__ void k_asml(int nblk, int mbf, const int* __restrict__ off, const int4* __restrict__ list,
                       const PT* __restrict__ Pf, const float* __restrict__ afine, float* __restrict__ aval) {
  pdl_start();
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int b = warp; b < nblk; b += nw) {
    float acc[MB * MB];
#pragma unroll
    for (int i = 0; i < MB * MB; ++i) acc[i] = 0.0f;
    for (int c = off[b] + lane; c < off[b + 1]; c += 32) {
      const int4 t = list[c];   // (source block, c, d, -)
      const float* As = afine + (size_t)t.x * mbf * mbf;
      const size_t pc = (size_t)t.y * mbf * MB, pd = (size_t)t.z * mbf * MB;
      for (int i = 0; i < mbf; ++i) {
        float ti[MB];
#pragma unroll
        for (int v = 0; v < MB; ++v) ti[v] = 0.0f;
        for (int j = 0; j < mbf; ++j) {
          const float a = As[i * mbf + j];
#pragma unroll
          for (int v = 0; v < MB; ++v) ti[v] = fmaf(a, pval(Pf, pd + j * MB + v), ti[v]);
        }
#pragma unroll
        for (int u = 0; u < MB; ++u) {
          const float pu = pval(Pf, pc + i * MB + u);
#pragma unroll
          for (int v = 0; v < MB; ++v) acc[u * MB + v] = fmaf(pu, ti[v], acc[u * MB + v]);
        }
      }
    }
    __syncwarp();
    if constexpr (MB == 4) {
      const float s = group_sum16<32>(acc);
      if (lane < 16) aval[(size_t)b * 16 + lane] = s;
    } else {
#pragma unroll
      for (int i = 0; i < MB * MB; ++i) acc[i] = warp_sum(acc[i]);
#pragma unroll
      for (int i = 0; i < MB * MB; ++i)
        if ((i & 31) == lane) aval[(size_t)b * MB * MB + i] = acc[i];
    }
  }
}

// Inverse of each diagonal block of a block level (Gauss-Jordan in FP64 registers, no pivoting: the blocks are
// symmetric positive definite), one thread per cell; conversions on the integer pipe, short reciprocals.
template <int MB>
__global__ void k_block_inv(int nc, const int* __restrict__ dpos, const float* __restrict__ aval,
                            float* __restrict__ dinv) {
  pdl_start();
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
    double A[MB * MB];
    const float* B = aval + (size_t)dpos[c] * MB * MB;
#pragma unroll
    for (int i = 0; i < MB * MB; ++i) A[i] = widen(B[i]);
#pragma unroll
    for (int k = 0; k < MB; ++k) {
      const double dk = fast_rcp(A[k * MB + k]);
      A[k * MB + k] = 1.0;
#pragma unroll
      for (int j = 0; j < MB; ++j) A[k * MB + j] *= dk;
#pragma unroll
      for (int i = 0; i < MB; ++i) {
        if (i == k) continue;
        const double f = A[i * MB + k];
        A[i * MB + k] = 0.0;
#pragma unroll
        for (int j = 0; j < MB; ++j) A[i * MB + j] -= f * A[k * MB + j];
      }
    }
#pragma unroll
    for (int i = 0; i < MB * MB; ++i) dinv[(size_t)c * MB * MB + i] = narrow(A[i]);
  }
}

// The Gershgorin bound max over rows of sum |D^-1 A| of a block level, one warp per cell, a lane per block of its row (a
// thread per cell walked its 27 blocks one memory round trip after another, with the inverse: 37 us on any level).
template <int MB>
__global__ void k_block_bound(int nc, const int* __restrict__ rowptr, const float* __restrict__ aval,
                              const float* __restrict__ dinv, float* lam) {
  pdl_start();
  const int lane = threadIdx.x & 31;
  float g = 0.0f;
  for (int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < nc; c += (gridDim.x * blockDim.x) >> 5) {
    float Di[MB * MB], rs[MB];
#pragma unroll
    for (int u = 0; u < MB; ++u) ld_seg<MB>(dinv + ((size_t)c * MB + u) * MB, *(float(*)[MB])(Di + u * MB));
#pragma unroll
    for (int u = 0; u < MB; ++u) rs[u] = 0.0f;
    const int q1 = rowptr[c + 1];
    for (int q = rowptr[c] + lane; q < q1; q += 32) {
      float Bl[MB * MB];
#pragma unroll
      for (int u = 0; u < MB; ++u) ld_seg<MB>(aval + ((size_t)q * MB + u) * MB, *(float(*)[MB])(Bl + u * MB));
#pragma unroll
      for (int u = 0; u < MB; ++u)
#pragma unroll
        for (int v = 0; v < MB; ++v) {
          float t = 0.0f;
#pragma unroll
          for (int w = 0; w < MB; ++w) t = fmaf(Di[u * MB + w], Bl[w * MB + v], t);
          rs[u] += fabsf(t);
        }
    }
#pragma unroll
    for (int u = 0; u < MB; ++u) g = fmaxf(g, warp_sum(rs[u]));
  }
  if (lane == 0) atomic_max_pos(lam, g);
}

// Chebyshev coefficient table of every level and step from the Gershgorin bounds (one thread per entry).
__global__ void k_cheb_table(const float* __restrict__ lam, float* __restrict__ tab) {
  pdl_start();
  const int t = threadIdx.x;
  if (t >= kMgMaxLevels * kMgMaxDeg) return;
  const int l = t / kMgMaxDeg, k = t % kMgMaxDeg;
  float c1 = 0.0f, c2 = 0.0f;
  if (lam[l] > 0.0f) cheb_coef(lam[l], k, c1, c2);
  tab[2 * t] = c1;
  tab[2 * t + 1] = c2;
}

// Dense inverse of the coarsest level (n = nc * mb <= kMgMaxCoarse) by one cluster of kInvCtas blocks: FP64 Gauss-Jordan
// (symmetric positive definite, no pivoting), column j in block j % kInvCtas. Step k needs column k of its owner; the
// owner updates column k + 1 first, publishes a copy of it with its pivot's reciprocal in its shared memory and arrives
// at the cluster's barrier before the rest of its update, which hides the barrier. n^3 FP64 multiply-adds on one SM take
// 0.5 ms at n = 128 (1.16 ms with a step's serial part), a cluster of eight a tenth of that.
constexpr int kInvCtas = 8;
constexpr int kInvCols = kMgMaxCoarse / kInvCtas;
constexpr int kInvThreads = 256;
__device__ __forceinline__ double ld_cluster(const double* p, unsigned rank) {   // p in block `rank`'s shared memory
  unsigned a;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
  return v;
}
__global__ void __cluster_dims__(kInvCtas, 1, 1) __launch_bounds__(kInvThreads)
    k_coarse_inv(int nc, int mb, const int* __restrict__ rowptr, const int* __restrict__ col,
                 const float* __restrict__ aval, float* __restrict__ cinv) {
  pdl_start();
  __shared__ double S[kInvCols][kMgMaxCoarse];        // own columns
  __shared__ double pub[2][kMgMaxCoarse + 1];         // a published column and its pivot's reciprocal
  __shared__ double f[kMgMaxCoarse + 1], p[kInvCols]; // the step's column, and the pivot row on the own columns
  const int n = nc * mb, rank = (int)blockIdx.x, tid = threadIdx.x;
  for (int i = tid; i < kInvCols * kMgMaxCoarse; i += kInvThreads) S[i / kMgMaxCoarse][i % kMgMaxCoarse] = 0.0;
  __syncthreads();
  for (int c = tid >> 5; c < nc; c += kInvThreads / 32)   // a warp per block row
    for (int q = rowptr[c]; q < rowptr[c + 1]; ++q)
      for (int idx = tid & 31; idx < mb * mb; idx += 32) {
        const int j = col[q] * mb + idx % mb;
        if (j % kInvCtas == rank) S[j / kInvCtas][c * mb + idx / mb] = (double)aval[(size_t)q * mb * mb + idx];
      }
  __syncthreads();
  auto publish = [&](int k) {   // by the owner of column k (none beyond n), whose column is up to date in the whole block
    if (k < n && k % kInvCtas == rank) {
      for (int i = tid; i < n; i += kInvThreads) pub[k & 1][i] = S[k / kInvCtas][i];
      if (tid == 0) pub[k & 1][kMgMaxCoarse] = fast_rcp(S[k / kInvCtas][k]);
    }
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  };
  // one column's update: S_ij -= f_i p_j, row k becomes p, column k -f piv
  auto update = [&](int jl, int k, int i) {
    const int j = jl * kInvCtas + rank;
    const double pj = p[jl];
    if (j == k) S[jl][i] = i == k ? f[kMgMaxCoarse] : -f[i] * f[kMgMaxCoarse];
    else S[jl][i] = i == k ? pj : fma(-f[i], pj, S[jl][i]);
  };
  publish(0);
  for (int k = 0; k < n; ++k) {
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    for (int i = tid; i <= kMgMaxCoarse; i += kInvThreads)
      if (i < n || i == kMgMaxCoarse) f[i] = ld_cluster(&pub[k & 1][i], (unsigned)(k % kInvCtas));
    __syncthreads();
    if (tid < kInvCols) p[tid] = S[tid][k] * f[kMgMaxCoarse];
    __syncthreads();
    const int next = k + 1 < n && (k + 1) % kInvCtas == rank ? (k + 1) / kInvCtas : -1;
    if (next >= 0) {   // the same in the whole block
      for (int i = tid; i < n; i += kInvThreads) update(next, k, i);
      __syncthreads();
    }
    publish(k + 1);
    for (int e = tid; e < kInvCols * kMgMaxCoarse; e += kInvThreads) {
      const int jl = e / kMgMaxCoarse, i = e % kMgMaxCoarse;
      if (i < n && jl * kInvCtas + rank < n && jl != next) update(jl, k, i);
    }
    __syncthreads();
  }
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");   // nobody reads this block's memory any more
  for (int e = tid; e < kInvCols * kMgMaxCoarse; e += kInvThreads) {
    const int jl = e / kMgMaxCoarse, i = e % kMgMaxCoarse, j = jl * kInvCtas + rank;
    if (i < n && j < n) cinv[(size_t)i * n + j] = (float)S[jl][i];
  }
}

// ---------------------------------------------------------------------------------------------------------------
// V-cycle kernels

// The entries of a level-0 row: up to eight in registers (loaded before the wait for the first cell of a thread), the
// rest, if any, read in the product.
struct Row0 {
  int nb[8];
  float a[8];
  int w, e;
};
__device__ __forceinline__ Row0 row0(const FineDev& F, const float* __restrict__ a0off, int K) {
  Row0 R;
  R.w = K < F.N ? F.sell_w[K >> 5] : 0;
  R.e = K < F.N ? F.sell_off[K >> 5] + (K & 31) : 0;
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (j < R.w) {
      R.nb[j] = F.nbr[R.e + 32 * j];
      R.a[j] = a0off[R.e + 32 * j];
    }
  return R;
}
__device__ __forceinline__ float row0_ax(const FineDev& F, const float* __restrict__ a0off, const Row0& R, float ax,
                                         const float* __restrict__ x) {
  float xv[8];
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (j < R.w) xv[j] = x[R.nb[j]];
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (j < R.w) ax = fmaf(R.a[j], xv[j], ax);
  for (int j = 8; j < R.w; ++j) ax = fmaf(a0off[R.e + 32 * j], x[F.nbr[R.e + 32 * j]], ax);
  return ax;
}

// One Chebyshev step on level 0: res = b - A x_in, d = c1 d + c2 D^-1 res, x_out = x_in + d (x_in is gathered by the
// neighbours, so the new iterate goes to the other buffer).
__device__ __forceinline__ float cheb0_cell(const FineDev& F, const float* __restrict__ a0off, const Row0& R, float diag,
                                            float dinv, const float* __restrict__ b, const float* __restrict__ xin,
                                            float* __restrict__ xout, float* __restrict__ d, float c1, float c2, int k,
                                            int K) {
  const float xk = xin[K];
  const float ax = row0_ax(F, a0off, R, diag * xk, xin);
  const float res = b[K] - ax;
  const float dn = (k == 0 ? 0.0f : c1 * d[K]) + c2 * dinv * res;
  d[K] = dn;
  const float xn = xk + dn;
  xout[K] = xn;
  return xn;
}

__global__ void __launch_bounds__(kT, 6) k_cheb0(FineDev F, const float* __restrict__ a0off, const float* __restrict__ a0diag,
                        const float* __restrict__ a0dinv, const float* __restrict__ b, const float* __restrict__ xin,
                        float* __restrict__ xout, float* __restrict__ d, const float* __restrict__ lam, int k,
                        const int* done) {
  int K = blockIdx.x * blockDim.x + threadIdx.x;
  Row0 R = row0(F, a0off, K);
  float dg = K < F.N ? a0diag[K] : 0.0f, di = K < F.N ? a0dinv[K] : 0.0f;
  float c1, c2;
  cheb_tab(lam, 0, k, c1, c2);
  pdl_start();
  if (stop(done)) return;
  while (K < F.N) {
    (void)cheb0_cell(F, a0off, R, dg, di, b, xin, xout, d, c1, c2, k, K);
    K += gridDim.x * blockDim.x;
    if (K < F.N) {
      R = row0(F, a0off, K);
      dg = a0diag[K];
      di = a0dinv[K];
    }
  }
}

// The last Chebyshev step of level 0 (z = xout) fused with the flexible CG step length: rz_new = (r, z),
// beta = (r, z - z_old) / rz (0 on the first step), which equals the plain rz_new / rz for a fixed linear
// preconditioner and tolerates the FP32 rounding of the V-cycle. At most kMaxRedBlocks blocks.
__global__ void __launch_bounds__(kT, 6) k_cheb0_beta(FineDev F, const float* __restrict__ a0off, const float* __restrict__ a0diag,
                             const float* __restrict__ a0dinv, const float* __restrict__ b,
                             const float* __restrict__ xin, float* __restrict__ xout, float* __restrict__ d,
                             const float* __restrict__ lam, int k, const double* __restrict__ r,
                             const float* __restrict__ zold, double* part, MgScal* sc) {
  int K = blockIdx.x * blockDim.x + threadIdx.x;
  Row0 R = row0(F, a0off, K);
  float dg = K < F.N ? a0diag[K] : 0.0f, di = K < F.N ? a0dinv[K] : 0.0f;
  float c1, c2;
  cheb_tab(lam, 0, k, c1, c2);
  pdl_start();
  if (stop(&sc->done)) return;
  const bool first = sc->it == 0;
  double v[2] = {0.0, 0.0};
  while (K < F.N) {
    const float z = cheb0_cell(F, a0off, R, dg, di, b, xin, xout, d, c1, c2, k, K);
    const double rK = r[K];
    v[0] = fma(rK, widen(z), v[0]);
    if (!first) v[1] = fma(rK, widen(zold[K]), v[1]);
    K += gridDim.x * blockDim.x;
    if (K < F.N) {
      R = row0(F, a0off, K);
      dg = a0diag[K];
      di = a0dinv[K];
    }
  }
  double out[2];
  if (reduce_last<2>(v, part, &sc->cnt[1], out) && threadIdx.x == 0) {
    sc->beta = first ? 0.0 : fast_div(out[0] - out[1], sc->rz);
    sc->rz = out[0];
  }
}

// (A x)_u of block-level cell c, one warp per cell: lane = slot * 8 + u, the four slots take every fourth block of
// the row; a shuffle tree adds the slots, so every lane with component u < MB holds (A x)_u. The blocks are taken in
// batches of RB per slot whose column indices, then matrix and vector entries, are all loaded before the first
// product: on the small levels few warps are in flight, and a row costs two dependent memory round trips per batch
// instead of two per block. The products are added in block order either way. A row's first batch can be loaded ahead.
template <int MB>
struct RowBatch {
  static constexpr int RB = MB >= 8 ? 2 : (MB >= 4 ? 4 : 8);
  int cq[RB];
  float bv[RB][MB];
  __device__ __forceinline__ void load(int qb, int q1, int u, const int* __restrict__ col, const float* __restrict__ aval) {
#pragma unroll
    for (int j = 0; j < RB; ++j) cq[j] = u < MB && qb + 4 * j < q1 ? col[qb + 4 * j] : -1;
#pragma unroll
    for (int j = 0; j < RB; ++j) {
      const float* Bq = aval + (size_t)(qb + 4 * j) * MB * MB + u * MB;
#pragma unroll
      for (int v = 0; v < MB; ++v) bv[j][v] = cq[j] >= 0 ? Bq[v] : 0.0f;
    }
  }
};
template <int MB>
__device__ __forceinline__ float row_ax(RowBatch<MB>& A, int q0, int q1, int lane, const int* __restrict__ col,
                                        const float* __restrict__ aval, const float* x) {
  constexpr int RB = RowBatch<MB>::RB;
  const int slot = lane >> 3, u = lane & 7;
  float ax = 0.0f;
  for (int qb = q0 + slot;;) {   // A holds the batch at qb
    float xv[RB][MB];
#pragma unroll
    for (int j = 0; j < RB; ++j) {
      const float* xd = x + (size_t)(A.cq[j] < 0 ? 0 : A.cq[j]) * MB;
#pragma unroll
      for (int v = 0; v < MB; ++v) xv[j][v] = A.cq[j] >= 0 ? xd[v] : 0.0f;
    }
#pragma unroll
    for (int j = 0; j < RB; ++j)
      if (A.cq[j] >= 0) {
#pragma unroll
        for (int v = 0; v < MB; ++v) ax = fmaf(A.bv[j][v], xv[j][v], ax);
      }
    qb += 4 * RB;
    if (u >= MB || qb >= q1) break;
    A.load(qb, q1, u, col, aval);
  }
  __syncwarp();
  ax += __shfl_xor_sync(0xffffffffu, ax, 8);
  ax += __shfl_xor_sync(0xffffffffu, ax, 16);
  return ax;
}
template <int MB>
__device__ __forceinline__ float row_ax(int c, int lane, const int* __restrict__ rowptr, const int* __restrict__ col,
                                        const float* __restrict__ aval, const float* x) {
  RowBatch<MB> A;
  const int q0 = rowptr[c], q1 = rowptr[c + 1];
  A.load(q0 + (lane >> 3), q1, lane & 7, col, aval);
  return row_ax<MB>(A, q0, q1, lane, col, aval, x);
}

// One Chebyshev step on block level l (coefficients c1, c2 of step k): res = b - A x_in, d = c1 d + c2 D^-1 res,
// x_out = x_in + d; warps w0, w0 + nw, ... take one cell each (see row_ax).
template <int MB>
__device__ __forceinline__ void chebl_body(int w0, int nw, int nc, const int* __restrict__ rowptr,
                                           const int* __restrict__ col, const float* __restrict__ aval,
                                           const float* __restrict__ dinv, const float* b, const float* xin,
                                           float* xout, float* d, float c1, float c2, int k) {
  const int lane = threadIdx.x & 31, u = lane & 7;
  for (int c = w0; c < nc; c += nw) {
    const float ax = row_ax<MB>(c, lane, rowptr, col, aval, xin);
    const float res = u < MB ? b[(size_t)c * MB + u] - ax : 0.0f;
    float s = 0.0f;
#pragma unroll
    for (int v = 0; v < MB; ++v) {
      const float rv = __shfl_sync(0xffffffffu, res, v);
      if (u < MB) s = fmaf(dinv[(size_t)c * MB * MB + u * MB + v], rv, s);
    }
    if (lane < MB) {
      const size_t i = (size_t)c * MB + u;
      const float dn = (k == 0 ? 0.0f : c1 * d[i]) + c2 * s;
      d[i] = dn;
      xout[i] = xin[i] + dn;
    }
  }
}

// Residual b - A x of a block level, one warp per cell.
template <int MB>
__device__ __forceinline__ void resl_body(int w0, int nw, int nc, const int* __restrict__ rowptr,
                                          const int* __restrict__ col, const float* __restrict__ aval, const float* b,
                                          const float* x, float* res) {
  const int lane = threadIdx.x & 31;
  for (int c = w0; c < nc; c += nw) {
    const float ax = row_ax<MB>(c, lane, rowptr, col, aval, x);
    if (lane < MB) res[(size_t)c * MB + lane] = b[(size_t)c * MB + lane] - ax;
  }
}

// Restriction of a residual (mbf per cell on level l) to level l+1 (mb per cell), one warp per level-(l+1) cell A:
// lane = k * 8 + u takes component u of children k, k + 4, ...; a shuffle tree adds the lanes. `first` adds the first
// Chebyshev step of level l+1 (x = c2 D^-1 b, d = x).
template <class PT>
__device__ __forceinline__ void restr_body(int w0, int nw, int mbf, const float* res, const PT* __restrict__ Pl,
                                           const int* __restrict__ ch_off, const int* __restrict__ ch, int ncc,
                                           int mb, float* bc, const float* __restrict__ dinvc, float* xc, float* dc,
                                           float c2, int first) {
  const int lane = threadIdx.x & 31, grp = lane >> 3, u = lane & 7;
  // one value per child (level 0): lanes take children one each; else eight lanes per child
  const int cstep = mbf == 1 ? 32 : 4, c0 = mbf == 1 ? lane : grp, uu = mbf == 1 ? 0 : u;
  for (int A = w0; A < ncc; A += nw) {
    float acc[kMaxM];
#pragma unroll
    for (int j = 0; j < kMaxM; ++j) acc[j] = 0.0f;
    if (uu < mbf) {
      // children in pairs, both loaded before the products (see row_ax); products in child order
      const int t1 = ch_off[A + 1];
      for (int t = ch_off[A] + c0; t < t1; t += 2 * cstep) {
        const bool two = t + cstep < t1;
        const int ca = ch[t], cb = two ? ch[t + cstep] : ca;
        const float ra = res[(size_t)ca * mbf + uu], rb = res[(size_t)cb * mbf + uu];
        const size_t pa = ((size_t)ca * mbf + uu) * mb, pb = ((size_t)cb * mbf + uu) * mb;
        float Pa[kMaxM], Pb[kMaxM];
#pragma unroll
        for (int j = 0; j < kMaxM; ++j)
          if (j < mb) {
            Pa[j] = pval(Pl, pa + j);
            Pb[j] = pval(Pl, pb + j);
          }
#pragma unroll
        for (int j = 0; j < kMaxM; ++j)
          if (j < mb) acc[j] = fmaf(Pa[j], ra, acc[j]);
        if (two) {
#pragma unroll
          for (int j = 0; j < kMaxM; ++j)
            if (j < mb) acc[j] = fmaf(Pb[j], rb, acc[j]);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < kMaxM; ++j)
      if (j < mb) acc[j] = warp_sum(acc[j]);
    if (lane < mb) {
      float bj = 0.0f;
#pragma unroll
      for (int j = 0; j < kMaxM; ++j)
        if (j == lane) bj = acc[j];
      bc[(size_t)A * mb + lane] = bj;
      if (first) {
        const float* Dc = dinvc + (size_t)A * mb * mb + lane * mb;
        float s = 0.0f;
#pragma unroll
        for (int v = 0; v < kMaxM; ++v)
          if (v < mb) s = fmaf(Dc[v], acc[v], s);
        const float dn = c2 * s;
        dc[(size_t)A * mb + lane] = dn;
        xc[(size_t)A * mb + lane] = dn;
      }
    }
  }
}

// x += P e on a block level (one thread per cell and component; threads i0, i0 + ni, ...).
template <class PT>
__device__ __forceinline__ void prol_body(long i0, long ni, int nc, int mbf, int mb, const PT* __restrict__ Pl,
                                          const int* __restrict__ agg, const float* e, float* x) {
  const long total = (long)nc * mbf;
  for (long i = i0; i < total; i += ni) {
    const int c = (int)(i / mbf);
    const float* ea = e + (size_t)agg[c] * mb;
    float s = x[i];
    for (int j = 0; j < mb; ++j) s = fmaf(pval(Pl, (size_t)i * mb + j), ea[j], s);
    x[i] = s;
  }
}

// Coarsest level: x = C^-1 b with the dense inverse (threads i0, i0 + ni, ... take one row each).
__device__ __forceinline__ void coarse_solve_body(int i0, int ni, int n, const float* __restrict__ cinv,
                                                  const float* b, float* x) {
  for (int i = i0; i < n; i += ni) {
    float s = 0.0f;
    for (int j = 0; j < n; ++j) s = fmaf(cinv[(size_t)i * n + j], b[j], s);
    x[i] = s;
  }
}

__device__ __forceinline__ int gwarp() { return (blockIdx.x * blockDim.x + threadIdx.x) >> 5; }
__device__ __forceinline__ int nwarps() { return (gridDim.x * blockDim.x) >> 5; }

// One Chebyshev step of a block level, a warp per cell; the row's first batch, its place and the block inverse are loaded
// before the wait.
template <int MB>
__global__ void k_chebl(int nc, const int* __restrict__ rowptr, const int* __restrict__ col,
                        const float* __restrict__ aval, const float* __restrict__ dinv, const float* __restrict__ b,
                        const float* __restrict__ xin, float* __restrict__ xout, float* __restrict__ d,
                        const float* __restrict__ lam, int l, int k, const int* done) {
  const int lane = threadIdx.x & 31, u = lane & 7;
  int c = gwarp();
  RowBatch<MB> A;
  int q0 = 0, q1 = 0;
  float dv[MB];
  auto ahead = [&]() {
    q0 = rowptr[c];
    q1 = rowptr[c + 1];
    A.load(q0 + (lane >> 3), q1, u, col, aval);
#pragma unroll
    for (int v = 0; v < MB; ++v) dv[v] = u < MB ? dinv[(size_t)c * MB * MB + u * MB + v] : 0.0f;
  };
  if (c < nc) ahead();
  float c1, c2;
  cheb_tab(lam, l, k, c1, c2);
  pdl_start();
  if (stop(done)) return;
  while (c < nc) {
    const size_t i = (size_t)c * MB + u;
    const bool own = lane < MB;
    const float bi = u < MB ? b[i] : 0.0f, di = own && k > 0 ? d[i] : 0.0f, xi = own ? xin[i] : 0.0f;
    const float res = bi - row_ax<MB>(A, q0, q1, lane, col, aval, xin);
    float s = 0.0f;
#pragma unroll
    for (int v = 0; v < MB; ++v) {
      const float rv = __shfl_sync(0xffffffffu, res, v);
      if (u < MB) s = fmaf(dv[v], rv, s);
    }
    if (own) {
      const float dn = (k == 0 ? 0.0f : c1 * di) + c2 * s;
      d[i] = dn;
      xout[i] = xi + dn;
    }
    c += nwarps();
    if (c < nc) ahead();
  }
}

template <int MB>
__global__ void k_resl(int nc, const int* __restrict__ rowptr, const int* __restrict__ col,
                       const float* __restrict__ aval, const float* __restrict__ b, const float* __restrict__ x,
                       float* __restrict__ res, const int* done) {
  const int lane = threadIdx.x & 31;
  int c = gwarp();
  RowBatch<MB> A;
  int q0 = 0, q1 = 0;
  auto ahead = [&]() {
    q0 = rowptr[c];
    q1 = rowptr[c + 1];
    A.load(q0 + (lane >> 3), q1, lane & 7, col, aval);
  };
  if (c < nc) ahead();
  pdl_start();
  if (stop(done)) return;
  while (c < nc) {
    const float bi = lane < MB ? b[(size_t)c * MB + lane] : 0.0f;
    const float ax = row_ax<MB>(A, q0, q1, lane, col, aval, x);
    if (lane < MB) res[(size_t)c * MB + lane] = bi - ax;
    c += nwarps();
    if (c < nc) ahead();
  }
}

template <class PT>
__global__ void k_restr(int mbf, const float* __restrict__ res, const PT* __restrict__ Pl,
                        const int* __restrict__ ch_off, const int* __restrict__ ch, int ncc, int mb,
                        float* __restrict__ bc, const float* __restrict__ dinvc, float* __restrict__ xc,
                        float* __restrict__ dc, const float* __restrict__ lam, int lc, int first, const int* done) {
  pdl_start();
  if (stop(done)) return;
  float c1 = 0.0f, c2 = 0.0f;
  if (first) cheb_tab(lam, lc, 0, c1, c2);
  restr_body<PT>(gwarp(), nwarps(), mbf, res, Pl, ch_off, ch, ncc, mb, bc, dinvc, xc, dc, c2, first);
}

// The residual of a block level and its restriction in one pass: a block per cell A of the next level, a warp per child;
// a child's residual stays in the lanes of its components, which take their terms of P^T res, and the warps' sums are
// added in order. `first` adds the first Chebyshev step of the next level. What bounds these levels is the chain of
// dependent kernels of a few microseconds each, so one launch less, and no way through memory for the residual: a CG
// iteration on 229,360 cells 85.1 -> 81.3 us, on 64,000 cells 59.7 -> 56.7 us, of which two such pairs. (The same on
// level 0, whose cells an aggregate reads out of order, loses: 81.3 -> 83.3 us, 10^6 cells 253.9 -> 263.2 us.)
template <class PT, int MB>
__global__ void __launch_bounds__(kT) k_res_restr(const int* __restrict__ rowptr, const int* __restrict__ col,
                                                  const float* __restrict__ aval, const float* __restrict__ b,
                                                  const float* __restrict__ x, const PT* __restrict__ Pl,
                                                  const int* __restrict__ ch_off, const int* __restrict__ ch, int mb,
                                                  float* __restrict__ bc, const float* __restrict__ dinvc,
                                                  float* __restrict__ xc, float* __restrict__ dc,
                                                  const float* __restrict__ lam, int lc, int first, const int* done) {
  constexpr int NW = kT / 32;
  __shared__ float s[NW][kMaxM];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, A = blockIdx.x;
  const int t1 = ch_off[A + 1];
  int t = ch_off[A] + warp, c = 0, q0 = 0, q1 = 0;
  RowBatch<MB> R;
  float P[kMaxM], acc[kMaxM], dv[kMaxM];
  auto ahead = [&]() {
    c = ch[t];
    q0 = rowptr[c];
    q1 = rowptr[c + 1];
    R.load(q0 + (lane >> 3), q1, lane & 7, col, aval);
#pragma unroll
    for (int j = 0; j < kMaxM; ++j) P[j] = j < mb && lane < MB ? pval(Pl, ((size_t)c * MB + lane) * mb + j) : 0.0f;
  };
  if (t < t1) ahead();
#pragma unroll
  for (int j = 0; j < kMaxM; ++j) {
    acc[j] = 0.0f;
    dv[j] = first && warp == 0 && lane < mb && j < mb ? dinvc[((size_t)A * mb + lane) * mb + j] : 0.0f;
  }
  pdl_start();
  if (stop(done)) return;
  while (t < t1) {
    const float bi = lane < MB ? b[(size_t)c * MB + lane] : 0.0f;
    const float ax = row_ax<MB>(R, q0, q1, lane, col, aval, x);
    const float res = lane < MB ? bi - ax : 0.0f;
#pragma unroll
    for (int j = 0; j < kMaxM; ++j) acc[j] = fmaf(P[j], res, acc[j]);
    t += NW;
    if (t < t1) ahead();
  }
#pragma unroll
  for (int j = 0; j < kMaxM; ++j)
    if (j < mb) {
      acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], 1);
      acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], 2);
      acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], 4);
      if (lane == 0) s[warp][j] = acc[j];
    }
  __syncthreads();
  if (warp > 0) return;
  float bj = 0.0f, dn = 0.0f;
  if (lane < mb)
#pragma unroll
    for (int w = 0; w < NW; ++w) bj += s[w][lane];
#pragma unroll
  for (int j = 0; j < kMaxM; ++j) dn = fmaf(dv[j], __shfl_sync(0xffffffffu, bj, j), dn);
  if (lane < mb) {
    const size_t i = (size_t)A * mb + lane;
    bc[i] = bj;
    if (first) {
      float c1, c2;
      cheb_tab(lam, lc, 0, c1, c2);
      xc[i] = dc[i] = c2 * dn;
    }
  }
}

// Level-0 residual b - A x (FP32), one thread per cell.
__global__ void __launch_bounds__(kT, 6) k_res0(FineDev F, const float* __restrict__ a0off, const float* __restrict__ a0diag,
                       const float* __restrict__ b, const float* __restrict__ x, float* __restrict__ res,
                       const int* done) {
  int K = blockIdx.x * blockDim.x + threadIdx.x;
  Row0 R = row0(F, a0off, K);
  float dg = K < F.N ? a0diag[K] : 0.0f;
  pdl_start();
  if (stop(done)) return;
  while (K < F.N) {
    res[K] = b[K] - row0_ax(F, a0off, R, dg * x[K], x);
    K += gridDim.x * blockDim.x;
    if (K < F.N) {
      R = row0(F, a0off, K);
      dg = a0diag[K];
    }
  }
}

__global__ void k_coarse_solve(int n, const float* __restrict__ cinv, const float* __restrict__ b,
                               float* __restrict__ x, const int* done) {
  pdl_start();
  if (stop(done)) return;
  coarse_solve_body(threadIdx.x, blockDim.x, n, cinv, b, x);
}

// x_0 += P e on level 0 (per fine cell) and on a block level (per cell and component); the first item's transfer row and
// aggregate are loaded before the wait.
template <class PT>
__global__ void k_pro0(int N, int mb, const PT* __restrict__ P0, const int* __restrict__ agg,
                       const float* __restrict__ e, float* __restrict__ x, const int* done) {
  int K = blockIdx.x * blockDim.x + threadIdx.x;
  float P[kMaxM];
  int A = 0;
  auto ahead = [&]() {
    A = agg[K];
#pragma unroll
    for (int j = 0; j < kMaxM; ++j)
      if (j < mb) P[j] = pval(P0, (size_t)K * mb + j);
  };
  if (K < N) ahead();
  pdl_start();
  if (stop(done)) return;
  while (K < N) {
    const float* ea = e + (size_t)A * mb;
    float s = x[K];
#pragma unroll
    for (int j = 0; j < kMaxM; ++j)
      if (j < mb) s = fmaf(P[j], ea[j], s);
    x[K] = s;
    K += gridDim.x * blockDim.x;
    if (K < N) ahead();
  }
}
template <class PT>
__global__ void k_prol(int nc, int mbf, int mb, const PT* __restrict__ Pl, const int* __restrict__ agg,
                       const float* __restrict__ e, float* __restrict__ x, const int* done) {
  const long total = (long)nc * mbf;
  long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  float P[kMaxM];
  int A = 0;
  auto ahead = [&]() {
    A = agg[(int)(i / mbf)];
#pragma unroll
    for (int j = 0; j < kMaxM; ++j)
      if (j < mb) P[j] = pval(Pl, (size_t)i * mb + j);
  };
  if (i < total) ahead();
  pdl_start();
  if (stop(done)) return;
  while (i < total) {
    const float* ea = e + (size_t)A * mb;
    float s = x[i];
#pragma unroll
    for (int j = 0; j < kMaxM; ++j)
      if (j < mb) s = fmaf(P[j], ea[j], s);
    x[i] = s;
    i += (long)gridDim.x * blockDim.x;
    if (i < total) ahead();
  }
}

// Row-parallel forms of the block-level smoothing step and residual (the per-level kernels of the V-cycle; the
// small levels' map is formed with the warp-per-cell bodies above): one thread per cell component, cell c = 32 g + t / MB and
// component u = t % MB for thread t of a block of 32 MB threads, so a block holds whole cells; blocks take groups g
// gridDim.x apart. A thread reads row u of each block of the cell's row in block order and the block column's x
// segment, with vector loads, the column indices of kRowBatch blocks before their entries. The warp-per-cell form
// leaves 8 - MB of every 8 lanes idle and runs one cell per warp; here every lane is busy and a warp covers 32 / MB
// cells.
template <int MB>
__device__ __forceinline__ float row_ax_u(int c, int u, const int* __restrict__ rowptr, const int* __restrict__ col,
                                          const float* __restrict__ aval, const float* __restrict__ x) {
  constexpr int RB = MB <= 4 ? 8 : 4;
  float ax = 0.0f;
  const int q1 = rowptr[c + 1];
  for (int qb = rowptr[c]; qb < q1; qb += RB) {
    int cq[RB];
#pragma unroll
    for (int j = 0; j < RB; ++j) cq[j] = qb + j < q1 ? col[qb + j] : -1;
    float a[RB][MB], xv[RB][MB];
#pragma unroll
    for (int j = 0; j < RB; ++j) {
      if (cq[j] >= 0) {
        ld_seg<MB>(aval + ((size_t)(qb + j) * MB + u) * MB, a[j]);
        ld_seg<MB>(x + (size_t)cq[j] * MB, xv[j]);
      } else {
#pragma unroll
        for (int v = 0; v < MB; ++v) a[j][v] = xv[j][v] = 0.0f;
      }
    }
#pragma unroll
    for (int j = 0; j < RB; ++j)
#pragma unroll
      for (int v = 0; v < MB; ++v) ax = fmaf(a[j][v], xv[j][v], ax);
  }
  return ax;
}

template <int MB>
__global__ void __launch_bounds__(32 * MB) k_chebr(int nc, const int* __restrict__ rowptr, const int* __restrict__ col,
                                                   const float* __restrict__ aval, const float* __restrict__ dinv,
                                                   const float* __restrict__ b, const float* __restrict__ xin,
                                                   float* __restrict__ xout, float* __restrict__ d,
                                                   const float* __restrict__ lam, int l, int k, const int* done) {
  pdl_start();
  if (stop(done)) return;
  float c1, c2;
  cheb_tab(lam, l, k, c1, c2);
  __shared__ float rs[32 * MB];
  const int cl = threadIdx.x / MB, u = threadIdx.x - cl * MB;
  const int groups = (nc + 31) / 32;
  for (int g = blockIdx.x; g < groups; g += gridDim.x) {   // the same trip count in every thread of the block
    const int c = g * 32 + cl;
    const bool act = c < nc;
    const size_t i = (size_t)c * MB + u;
    float res = 0.0f, dv[MB];
    if (act) {
      ld_seg<MB>(dinv + i * MB, dv);
      res = b[i] - row_ax_u<MB>(c, u, rowptr, col, aval, xin);
    }
    rs[threadIdx.x] = res;
    __syncthreads();
    if (act) {
      float s = 0.0f;
#pragma unroll
      for (int v = 0; v < MB; ++v) s = fmaf(dv[v], rs[cl * MB + v], s);
      const float dn = (k == 0 ? 0.0f : c1 * d[i]) + c2 * s;
      d[i] = dn;
      xout[i] = xin[i] + dn;
    }
    __syncthreads();
  }
}

template <int MB>
__global__ void __launch_bounds__(32 * MB) k_resr(int nc, const int* __restrict__ rowptr, const int* __restrict__ col,
                                                  const float* __restrict__ aval, const float* __restrict__ b,
                                                  const float* __restrict__ x, float* __restrict__ res,
                                                  const int* done) {
  pdl_start();
  if (stop(done)) return;
  const long rows = (long)nc * MB;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < rows; i += (long)gridDim.x * blockDim.x) {
    const int c = (int)(i / MB), u = (int)(i - (long)c * MB);
    res[i] = b[i] - row_ax_u<MB>(c, u, rowptr, col, aval, x);
  }
}

// Level-0 restriction with MB modes per aggregate (FP32 or BF16 transfers): restr_body's work split and order (one
// warp per aggregate, a lane per child, children t and t + 32 together), with the child's MB transfer entries read
// by vector loads and the aggregate's block-inverse row (for the fused first smoothing step) requested before the
// products. Same sums in the same order, so the same values as the generic kernel.
template <class PT, int MB>
__global__ void k_restr0(const float* __restrict__ res, const PT* __restrict__ P, const int* __restrict__ ch_off,
                         const int* __restrict__ ch, int ncc, float* __restrict__ bc, const float* __restrict__ dinvc,
                         float* __restrict__ xc, float* __restrict__ dc, const float* __restrict__ lam, int first,
                         const int* done) {
  pdl_start();
  if (stop(done)) return;
  float c1 = 0.0f, c2 = 0.0f;
  if (first) cheb_tab(lam, 1, 0, c1, c2);
  const int lane = threadIdx.x & 31;
  for (int A = gwarp(); A < ncc; A += nwarps()) {
    float dv[MB];
    if (first && lane < MB) ld_seg<MB>(dinvc + ((size_t)A * MB + lane) * MB, dv);
    float acc[MB];
#pragma unroll
    for (int j = 0; j < MB; ++j) acc[j] = 0.0f;
    const int t1 = ch_off[A + 1];
    for (int t = ch_off[A] + lane; t < t1; t += 64) {
      const bool two = t + 32 < t1;
      const int ca = ch[t], cb = two ? ch[t + 32] : ca;
      const float ra = res[ca], rb = res[cb];
      float Pa[MB], Pb[MB];
      ld_seg<MB>(P + (size_t)ca * MB, Pa);
      ld_seg<MB>(P + (size_t)cb * MB, Pb);
#pragma unroll
      for (int j = 0; j < MB; ++j) acc[j] = fmaf(Pa[j], ra, acc[j]);
      if (two) {
#pragma unroll
        for (int j = 0; j < MB; ++j) acc[j] = fmaf(Pb[j], rb, acc[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < MB; ++j) acc[j] = warp_sum(acc[j]);
    if (lane < MB) {
      float bj = 0.0f;
#pragma unroll
      for (int j = 0; j < MB; ++j)
        if (j == lane) bj = acc[j];
      bc[(size_t)A * MB + lane] = bj;
      if (first) {
        float s = 0.0f;
#pragma unroll
        for (int v = 0; v < MB; ++v) s = fmaf(dv[v], acc[v], s);
        const float dn = c2 * s;
        dc[(size_t)A * MB + lane] = dn;
        xc[(size_t)A * MB + lane] = dn;
      }
    }
  }
}

// The small levels t .. C of a V-cycle are a linear map of level t's restricted residual, so the setup forms it: block j
// runs their smoothing, residuals, transfers and coarsest solve on the unit vector e_j, out of shared memory (phases
// separated by __syncthreads on copies of the levels' matrices and transfers, with the bodies of the per-level kernels),
// prolongs the result to level t-1 and writes column j of E = P B, n_t x n_(t-1) (column j contiguous). A V-cycle then
// applies E (k_tail_apply) with every SM. Run as phases of one block in every V-cycle instead, the same levels took 25.6 us
// of a 127 us CG iteration on 229,360 cells; forming E takes about as much once per setup.
template <class PT>
__global__ void __launch_bounds__(kTailThreads, 1) k_tail_cols(const MgTailTab* __restrict__ Tg, float* __restrict__ E) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ MgTailTab T_;   // the table itself, read by every phase
  static_assert(sizeof(MgTailTab) % 4 == 0, "table copied in words");
  pdl_start();
  for (int i = threadIdx.x; i < (int)(sizeof(MgTailTab) / 4); i += kTailThreads)
    ((int*)&T_)[i] = __ldg((const int*)Tg + i);
  __syncthreads();
  const MgTailTab* T = &T_;
  constexpr int v = std::is_same_v<PT, float> ? 0 : 1;
  {
    const int nch = T->nchunks[v], ncp = T->ncopies[v];
    for (int i0 = threadIdx.x; i0 < nch; i0 += kTailThreads * 8) {
      float4 buf[8];
      unsigned dst[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = i0 + u * kTailThreads;
        if (i < nch) {
          int lo = 0, hi = ncp - 1;   // last entry whose first chunk is <= i
          while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (T->cp[v][mid].c0 <= (unsigned)i) lo = mid;
            else hi = mid - 1;
          }
          const MgTailCopy& e = T->cp[v][lo];
          buf[u] = __ldg((const float4*)e.src + (i - e.c0));
          dst[u] = e.dst + 16u * (i - e.c0);
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (i0 + u * kTailThreads < nch) *(float4*)(sm + dst[u]) = buf[u];
    }
  }
  __syncthreads();
  const MgDev& M = T->M;
  const int t = T->t, C = M.L - 1;
  const int w0 = threadIdx.x >> 5, nw = kTailThreads / 32;
  const int i0 = threadIdx.x, ni = kTailThreads;
  auto F32 = [&](unsigned off) { return (float*)(sm + off); };
  auto I32 = [&](unsigned off) { return (const int*)(sm + off); };
  auto PL = [&](int l) { return (const PT*)(sm + T->o_P[l]); };
  // buffer of level l's iterate: x[l][0] after the restriction (first step fused), then each Chebyshev step moves
  // it to the other buffer; the coarsest solve writes x[C][0]
  constexpr int kDown = (kMgDegCoarse - 1) & 1, kUp = (2 * kMgDegCoarse - 1) & 1;
  const float* coef = F32(T->o_coef);
  float c1, c2 = 0.0f;
  const int nt = M.nc[t] * M.mb[t], j = blockIdx.x;
  {   // b = e_j and the first smoothing step on it
    if (t < C) cheb_tab(coef, t, 0, c1, c2);
    const int mb = M.mb[t];
    for (int i = i0; i < nt; i += ni) {
      F32(T->o_b[t])[i] = i == j ? 1.0f : 0.0f;
      if (t < C) {
        const float dn = i / mb == j / mb ? c2 * F32(T->o_dinv[t])[(size_t)i * mb + j % mb] : 0.0f;
        F32(T->o_d[t])[i] = dn;
        F32(T->o_x[t][0])[i] = dn;
      }
    }
  }
  __syncthreads();
  for (int l = t; l < C; ++l) {
    const int *rp = I32(T->o_rowptr[l]), *cl = I32(T->o_col[l]);
    const float *av = F32(T->o_aval[l]), *di = F32(T->o_dinv[l]);
    float *xb[2] = {F32(T->o_x[l][0]), F32(T->o_x[l][1])}, *bl = F32(T->o_b[l]), *dl = F32(T->o_d[l]);
    for (int k = 1; k < kMgDegCoarse; ++k) {
      cheb_tab(coef, l, k, c1, c2);
      MG_MB_SWITCH(M.mb[l], (chebl_body<MB>(w0, nw, M.nc[l], rp, cl, av, di, bl, xb[(k - 1) & 1], xb[k & 1],
                                                   dl, c1, c2, k)));
      __syncthreads();
    }
    MG_MB_SWITCH(M.mb[l], (resl_body<MB>(w0, nw, M.nc[l], rp, cl, av, bl, xb[kDown], dl)));
    __syncthreads();
    const int first = l + 1 < C ? 1 : 0;
    c2 = 0.0f;
    if (first) cheb_tab(coef, l + 1, 0, c1, c2);
    restr_body<PT>(w0, nw, M.mb[l], dl, PL(l), I32(T->o_choff[l]), I32(T->o_ch[l]), M.nc[l + 1],
                          M.mb[l + 1], F32(T->o_b[l + 1]), F32(T->o_dinv[l + 1]), F32(T->o_x[l + 1][0]),
                          F32(T->o_d[l + 1]), c2, first);
    __syncthreads();
  }
  coarse_solve_body(i0, ni, M.nc[C] * M.mb[C], F32(T->o_cinv), F32(T->o_b[C]), F32(T->o_x[C][0]));
  __syncthreads();
  for (int l = C - 1; l >= t; --l) {
    const int *rp = I32(T->o_rowptr[l]), *cl = I32(T->o_col[l]);
    const float *av = F32(T->o_aval[l]), *di = F32(T->o_dinv[l]);
    float *xb[2] = {F32(T->o_x[l][0]), F32(T->o_x[l][1])}, *bl = F32(T->o_b[l]), *dl = F32(T->o_d[l]);
    prol_body<PT>(i0, ni, M.nc[l], M.mb[l], M.mb[l + 1], PL(l), I32(T->o_agg[l]),
                         F32(T->o_x[l + 1][l + 1 == C ? 0 : kUp]), xb[kDown]);
    __syncthreads();
    for (int k = 0; k < kMgDegCoarse; ++k) {
      cheb_tab(coef, l, k, c1, c2);
      MG_MB_SWITCH(M.mb[l], (chebl_body<MB>(w0, nw, M.nc[l], rp, cl, av, di, bl, xb[(kDown + k) & 1],
                                                   xb[(kDown + k + 1) & 1], dl, c1, c2, k)));
      __syncthreads();
    }
  }
  const float* xt = F32(T->o_x[t][t == C ? 0 : kUp]);
  const int mbf = M.mb[t - 1], mb = M.mb[t], rows = M.nc[t - 1] * mbf;
  const int* agg = I32(T->o_agg[t - 1]);
  for (int i = i0; i < rows; i += ni) {
    const float* ea = xt + (size_t)agg[i / mbf] * mb;
    float s = 0.0f;
    for (int q = 0; q < mb; ++q) s = fmaf(pval(PL(t - 1), (size_t)i * mb + q), ea[q], s);
    E[(size_t)j * rows + i] = s;
  }
}

// x_(t-1) += E b_t: a block takes 32 rows, each of its kApplyWarps warps an equal run of the columns (coalesced reads, all of
// a lane's entries independent), then the warps' sums are added in order.
constexpr int kApplyWarps = 16;
__global__ void __launch_bounds__(32 * kApplyWarps) k_tail_apply(int rows, int nt, const float* __restrict__ E,
                                                                 const float* __restrict__ b, float* __restrict__ x,
                                                                 const int* done) {
  __shared__ float s[kApplyWarps][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
  const int j0 = nt * warp / kApplyWarps, j1 = nt * (warp + 1) / kApplyWarps;
  float e[16];   // the run's first entries: older than the predecessor
#pragma unroll
  for (int q = 0; q < 16; ++q) e[q] = j0 + q < j1 && i < rows ? E[(size_t)(j0 + q) * rows + i] : 0.0f;
  pdl_start();
  if (stop(done)) return;
  float a = 0.0f;
#pragma unroll
  for (int q = 0; q < 16; ++q)
    if (j0 + q < j1) a = fmaf(e[q], b[j0 + q], a);
#pragma unroll 8
  for (int j = j0 + 16; j < j1; ++j) a = fmaf(i < rows ? E[(size_t)j * rows + i] : 0.0f, b[j], a);
  s[warp][lane] = a;
  __syncthreads();
  if (warp == 0 && i < rows) {
    float t = 0.0f;
#pragma unroll
    for (int w = 0; w < kApplyWarps; ++w) t += s[w][lane];
    x[i] += t;
  }
}

// ---------------------------------------------------------------------------------------------------------------
// Krylov kernels (FP64 outer iteration)

// A v with the frozen FP64 matrix (diagT, Tval) at cell K, v in FP32 (widened on the integer pipe: as conversions the
// seven values cost as much FP64 issue as the products).
__device__ __forceinline__ double amul(const FineDev& F, const double* __restrict__ Tval,
                                       const double* __restrict__ diagT, const float* __restrict__ v, int K) {
  const int w = F.sell_w[K >> 5];
  int e = F.sell_off[K >> 5] + (K & 31);
  double s = diagT[K] * widen(v[K]);
  for (int j = 0; j < w; ++j, e += 32) s = fma(-Tval[e], widen(v[F.nbr[e]]), s);
  return s;
}

// Fused first pre-smoothing step of level 0 for the FP32 right-hand side r32: x0 = D^-1 r32 / theta, d0 = x0.
__device__ __forceinline__ void first_step0(int K, float r32, const float* __restrict__ a0dinv, float c2,
                                            float* __restrict__ x0, float* __restrict__ d0) {
  const float dn = c2 * a0dinv[K] * r32;
  x0[K] = dn;
  d0[K] = dn;
}

// PCG start: x = 0, r = bscale b, r32 = r, first smoothing step, rr0 = ||S r||^2 (S = diag(A)^-1/2).
__global__ void k_pcg_init(int N, const double* __restrict__ b, double bscale, double* __restrict__ x,
                           double* __restrict__ r, float* __restrict__ r32, const float* __restrict__ a0dinv,
                           float* __restrict__ x0, float* __restrict__ d0, const float* __restrict__ lam, double* part,
                           MgScal* sc) {
  pdl_start();
  float c1, c2;
  cheb_tab(lam, 0, 0, c1, c2);
  double v[1] = {0.0};
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < N; K += gridDim.x * blockDim.x) {
    const double ri = bscale * b[K];
    x[K] = 0.0;
    r[K] = ri;
    const float rf = narrow(ri);
    r32[K] = rf;
    first_step0(K, rf, a0dinv, c2, x0, d0);
    v[0] = fma(ri * ri, widen(a0dinv[K]), v[0]);   // ||S r||^2 with S^2 = 1 / A_KK
  }
  double out[1];
  if (reduce_last<1>(v, part, &sc->cnt[0], out) && threadIdx.x == 0) {
    sc->rr0 = out[0];
    sc->rr = out[0];
    sc->it = 0;
    sc->done = !(out[0] > 0.0) ? 1 : 0;
    sc->bad = isfinite(out[0]) ? 0 : 1;
    sc->rz = 0.0;
  }
}

// p = z + beta p, q = A z + beta q (= A p), alpha = rz / (p, q); z is kept as z_old for the next beta.
__global__ void k_pcg_pq(FineDev F, const double* __restrict__ Tval, const double* __restrict__ diagT,
                         const float* __restrict__ z, float* __restrict__ zold, double* __restrict__ p,
                         double* __restrict__ q, double* part, MgScal* sc) {
  pdl_start();
  if (stop(&sc->done)) return;
  const double beta = sc->beta;
  const bool first = sc->it == 0;
  double v[1] = {0.0};
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < F.N; K += gridDim.x * blockDim.x) {
    const double az = amul(F, Tval, diagT, z, K);
    const float zf = z[K];
    const double zk = widen(zf);
    const double pk = first ? zk : fma(beta, p[K], zk);
    const double qk = first ? az : fma(beta, q[K], az);
    p[K] = pk;
    q[K] = qk;
    zold[K] = zf;
    v[0] = fma(pk, qk, v[0]);
  }
  double out[1];
  if (reduce_last<1>(v, part, &sc->cnt[2], out) && threadIdx.x == 0) sc->alpha = fast_div(sc->rz, out[0]);
}

// x += alpha p, r -= alpha q, r32 = r with the first smoothing step of the next V-cycle; ||S r||^2 decides: the
// iteration stops (conditional value 0) at ||S r||^2 <= tol^2 ||S r_0||^2, at maxit, or on a non-finite value.
__global__ void k_pcg_update(int N, const double* __restrict__ p, const double* __restrict__ q,
                             double* __restrict__ x, double* __restrict__ r, float* __restrict__ r32,
                             const float* __restrict__ a0dinv, float* __restrict__ x0, float* __restrict__ d0,
                             const float* __restrict__ lam, double* part, MgScal* sc, cudaGraphConditionalHandle h) {
  pdl_start();
  if (stop(&sc->done)) {
    if (blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(h, 0);
    return;
  }
  const double alpha = sc->alpha;
  float c1, c2;
  cheb_tab(lam, 0, 0, c1, c2);
  double v[1] = {0.0};
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < N; K += gridDim.x * blockDim.x) {
    x[K] = fma(alpha, p[K], x[K]);
    const double ri = fma(-alpha, q[K], r[K]);
    r[K] = ri;
    const float rf = narrow(ri);
    r32[K] = rf;
    first_step0(K, rf, a0dinv, c2, x0, d0);
    v[0] = fma(ri * ri, widen(a0dinv[K]), v[0]);   // ||S r||^2 with S^2 = 1 / A_KK
  }
  double out[1];
  if (reduce_last<1>(v, part, &sc->cnt[3], out) && threadIdx.x == 0) {
    sc->rr = out[0];
    sc->it += 1;
    const bool fin = isfinite(out[0]) && isfinite(alpha);
    if (!fin) sc->bad = 1;
    const int d = (!fin || out[0] <= sc->tol2 * sc->rr0 || sc->it >= sc->maxit) ? 1 : 0;
    sc->done = d;
    cudaGraphSetConditional(h, d ? 0 : 1);
  }
}

// ---- BiCGStab (right-preconditioned) for J dx = bscale b with the Newton Jacobian (jd diagonal, Joff SELL) ------
__device__ __forceinline__ double jmul(const FineDev& F, const double* __restrict__ Joff,
                                       const double* __restrict__ jd, const float* __restrict__ v, int K) {
  const int w = F.sell_w[K >> 5];
  int e = F.sell_off[K >> 5] + (K & 31);
  double s = jd[K] * widen(v[K]);
  for (int j = 0; j < w; ++j, e += 32) s = fma(Joff[e], widen(v[F.nbr[e]]), s);
  return s;
}

// start: x = 0, r = rh = p = bscale b, rho = (rh, r), rr0 = ||W r||^2 (W the Jacobi weights' square roots);
// r32 = p for the first V-cycle (p^ = B p).
__global__ void k_bicg_init(int N, const double* __restrict__ b, double bscale, const double* __restrict__ wgt,
                            double* __restrict__ x, double* __restrict__ r, double* __restrict__ rh,
                            double* __restrict__ p, float* __restrict__ r32, const float* __restrict__ a0dinv,
                            float* __restrict__ x0, float* __restrict__ d0, const float* __restrict__ lam,
                            double* part, MgScal* sc) {
  pdl_start();
  float c1, c2;
  cheb_tab(lam, 0, 0, c1, c2);
  double v[2] = {0.0, 0.0};
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < N; K += gridDim.x * blockDim.x) {
    const double ri = bscale * b[K];
    x[K] = 0.0;
    r[K] = ri;
    rh[K] = ri;
    p[K] = ri;
    const float f32 = narrow(ri);
    r32[K] = f32;
    first_step0(K, f32, a0dinv, c2, x0, d0);
    v[0] = fma(ri, ri, v[0]);
    v[1] = fma(ri * ri, wgt[K], v[1]);
  }
  double out[2];
  if (reduce_last<2>(v, part, &sc->cnt[0], out) && threadIdx.x == 0) {
    sc->rho = out[0];
    sc->rr0 = out[1];
    sc->rr = out[1];
    sc->it = 0;
    sc->done = !(out[1] > 0.0) ? 1 : 0;
    sc->bad = isfinite(out[1]) ? 0 : 1;
  }
}

// v = J p^ (p^ = B p from the V-cycle, kept in FP64 in pp); alpha = rho / (rh, v); s = r - alpha v, r32 = s with the
// first smoothing step of the next V-cycle (s^ = B s).
__global__ void k_bicg_v(FineDev F, const double* __restrict__ Joff, const double* __restrict__ jd,
                         const float* __restrict__ zp, double* __restrict__ pp, double* __restrict__ v,
                         const double* __restrict__ rh, double* part, MgScal* sc) {
  pdl_start();
  if (stop(&sc->done)) return;
  double a[1] = {0.0};
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < F.N; K += gridDim.x * blockDim.x) {
    pp[K] = widen(zp[K]);
    const double vk = jmul(F, Joff, jd, zp, K);
    v[K] = vk;
    a[0] = fma(rh[K], vk, a[0]);
  }
  double out[1];
  if (reduce_last<1>(a, part, &sc->cnt[1], out) && threadIdx.x == 0) sc->alpha = fast_div(sc->rho, out[0]);
}
__global__ void k_bicg_s(int N, const double* __restrict__ r, const double* __restrict__ v, double* __restrict__ s,
                         float* __restrict__ r32, const float* __restrict__ a0dinv, float* __restrict__ x0,
                         float* __restrict__ d0, const float* __restrict__ lam, MgScal* sc) {
  pdl_start();
  if (stop(&sc->done)) return;
  const double alpha = sc->alpha;
  float c1, c2;
  cheb_tab(lam, 0, 0, c1, c2);
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < N; K += gridDim.x * blockDim.x) {
    const double sk = fma(-alpha, v[K], r[K]);
    s[K] = sk;
    const float f32 = narrow(sk);
    r32[K] = f32;
    first_step0(K, f32, a0dinv, c2, x0, d0);
  }
}
// t = J s^ (s^ = B s from the V-cycle), omega = (t, s) / (t, t).
__global__ void k_bicg_t(FineDev F, const double* __restrict__ Joff, const double* __restrict__ jd,
                         const float* __restrict__ zs, const double* __restrict__ s, double* __restrict__ t,
                         double* part, MgScal* sc) {
  pdl_start();
  if (stop(&sc->done)) return;
  double a[2] = {0.0, 0.0};
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < F.N; K += gridDim.x * blockDim.x) {
    const double tk = jmul(F, Joff, jd, zs, K);
    t[K] = tk;
    a[0] = fma(tk, s[K], a[0]);
    a[1] = fma(tk, tk, a[1]);
  }
  double out[2];
  if (reduce_last<2>(a, part, &sc->cnt[2], out) && threadIdx.x == 0) sc->omega = out[1] != 0.0 ? fast_div(out[0], out[1]) : 0.0;
}
// x += alpha p^ + omega s^, r = s - omega t, rho_new = (rh, r), ||W r||^2; beta = (rho_new / rho)(alpha / omega).
__global__ void k_bicg_x(int N, const double* __restrict__ pp, const float* __restrict__ zs,
                         const double* __restrict__ s, const double* __restrict__ t, const double* __restrict__ rh,
                         const double* __restrict__ wgt, double* __restrict__ x, double* __restrict__ r, double* part,
                         MgScal* sc, cudaGraphConditionalHandle h) {
  pdl_start();
  if (stop(&sc->done)) {
    if (blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(h, 0);
    return;
  }
  const double alpha = sc->alpha, omega = sc->omega;
  double a[2] = {0.0, 0.0};
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < N; K += gridDim.x * blockDim.x) {
    x[K] = fma(omega, widen(zs[K]), fma(alpha, pp[K], x[K]));
    const double rk = fma(-omega, t[K], s[K]);
    r[K] = rk;
    a[0] = fma(rh[K], rk, a[0]);
    a[1] = fma(rk * rk, wgt[K], a[1]);
  }
  double out[2];
  if (reduce_last<2>(a, part, &sc->cnt[3], out) && threadIdx.x == 0) {
    sc->rr = out[1];
    sc->it += 1;
    const bool fin = isfinite(out[1]) && isfinite(alpha) && isfinite(omega);
    if (!fin) sc->bad = 1;
    const bool breakdown = omega == 0.0 || sc->rho == 0.0;
    sc->beta = breakdown ? 0.0 : fast_div(out[0], sc->rho) * fast_div(alpha, omega);
    sc->rho = out[0];
    const int d = (!fin || breakdown || out[1] <= sc->tol2 * sc->rr0 || sc->it >= sc->maxit) ? 1 : 0;
    sc->done = d;
    cudaGraphSetConditional(h, d ? 0 : 1);
  }
}
// p = r + beta (p - omega v), r32 = p with the first smoothing step of the next V-cycle; on the first iteration the
// start has set p = r and that step already.
__global__ void k_bicg_p(int N, const double* __restrict__ r, const double* __restrict__ v, double* __restrict__ p,
                         float* __restrict__ r32, const float* __restrict__ a0dinv, float* __restrict__ x0,
                         float* __restrict__ d0, const float* __restrict__ lam, MgScal* sc) {
  pdl_start();
  if (stop(&sc->done) || sc->it == 0) return;
  const double beta = sc->beta, omega = sc->omega;
  float c1, c2;
  cheb_tab(lam, 0, 0, c1, c2);
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < N; K += gridDim.x * blockDim.x) {
    const double pk = fma(beta, fma(-omega, v[K], p[K]), r[K]);
    p[K] = pk;
    const float f32 = narrow(pk);
    r32[K] = f32;
    first_step0(K, f32, a0dinv, c2, x0, d0);
  }
}

// z (FP32) -> out (FP64), and the start of a single application: r32 = b, first smoothing step.
__global__ void k_apply_in(int N, const double* __restrict__ b, float* __restrict__ r32,
                           const float* __restrict__ a0dinv, float* __restrict__ x0, float* __restrict__ d0,
                           const float* __restrict__ lam) {
  pdl_start();
  float c1, c2;
  cheb_tab(lam, 0, 0, c1, c2);
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < N; K += gridDim.x * blockDim.x) {
    const float f32 = narrow(b[K]);
    r32[K] = f32;
    first_step0(K, f32, a0dinv, c2, x0, d0);
  }
}
__global__ void k_apply_out(int N, const float* __restrict__ z, double* __restrict__ out) {
  pdl_start();
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < N; K += gridDim.x * blockDim.x) out[K] = widen(z[K]);
}

}  // namespace

// ---------------------------------------------------------------------------------------------------------------
// host: static structure

int mg_levels_for(const Hierarchy& H) {
  for (int L = 2; L <= (int)H.levels.size() && L <= kMgMaxLevels; ++L) {
    const Level& C = H.levels[L - 1];
    int mb = 0;
    for (int c = 0; c < C.n_cells; ++c) mb = std::max(mb, C.m[c]);
    if ((long)C.n_cells * mb <= kMgMaxCoarse) return L;
  }
  return 0;
}

bool mg_build_host(const FineMesh& fm, const Hierarchy& H, int levels, MgHost& M, std::string& err) {
  if (levels < 2 || levels > (int)H.levels.size() || levels > kMgMaxLevels) {
    err = "multigrid preconditioner: bad number of levels";
    return false;
  }
  const int N = fm.n_cells;
  M.L = levels;
  M.N = N;
  M.nc[0] = N;
  M.mb[0] = 1;
  for (int l = 1; l < levels; ++l) {
    const Level& Lv = H.levels[l];
    M.nc[l] = Lv.n_cells;
    int mb = 1;
    for (int c = 0; c < Lv.n_cells; ++c) mb = std::max(mb, Lv.m[c]);
    if (mb > kMaxM) {
      err = "multigrid preconditioner: more than 8 modes per cell";
      return false;
    }
    M.mb[l] = mb;
    M.mcnt[l] = Lv.m;
    M.padded[l] = std::any_of(Lv.m.begin(), Lv.m.end(), [&](int k) { return k < mb; });
  }
  if ((long)M.nc[levels - 1] * M.mb[levels - 1] > kMgMaxCoarse) {
    err = "multigrid preconditioner: the coarsest level has more than " + std::to_string(kMgMaxCoarse) +
          " unknowns";
    return false;
  }
  // fine SELL positions of each interior face from its first cell (the layout of the residual kernel), and the
  // Dirichlet entry of each Dirichlet face
  std::vector<int> deg(N, 0), dcount(N, 0), face_pos(fm.n_faces, -1), dir_pos(fm.n_faces, -1);
  for (int f = 0; f < fm.n_faces; ++f) {
    if (fm.bc[f] == 0) {
      face_pos[f] = deg[fm.fk[f]];
      ++deg[fm.fk[f]];
      ++deg[fm.fl[f]];
    } else if (fm.bc[f] == 1) {
      dir_pos[f] = dcount[fm.fk[f]]++;
    }
  }
  const int nsl = (N + 31) / 32;
  std::vector<long> soff(nsl + 1, 0);
  for (int s = 0; s < nsl; ++s) {
    int w = 0;
    for (int K = 32 * s; K < std::min(N, 32 * s + 32); ++K) w = std::max(w, deg[K]);
    soff[s + 1] = soff[s] + 32L * w;
  }
  std::vector<int> doff(N + 1, 0);
  for (int K = 0; K < N; ++K) doff[K + 1] = doff[K] + dcount[K];
  // transfers (padded) and children
  for (int l = 0; l + 1 < levels; ++l) {
    const Transfer& T = H.transfers[l];
    const Level& Lc = H.levels[l + 1];
    const int mbf = M.mb[l], mbc = M.mb[l + 1];
    const int ncf = M.nc[l];
    M.agg[l] = T.agg_of;
    M.ch_off[l] = T.agg_off;
    M.ch[l] = T.agg_cells;
    M.P[l].assign((size_t)ncf * mbf * mbc, 0.0f);
    const Level& Lf = H.levels[l];
    for (int a = 0; a < Lc.n_cells; ++a) {
      const int ma = Lc.m[a];
      int t = 0;
      for (int k = T.agg_off[a]; k < T.agg_off[a + 1]; ++k) {
        const int c = T.agg_cells[k];
        const int mc = l == 0 ? 1 : Lf.m[c];
        for (int u = 0; u < mc; ++u, ++t)
          for (int j = 0; j < ma; ++j)
            M.P[l][((size_t)c * mbf + u) * mbc + j] = (float)T.Pblk[T.pblk_off[a] + (size_t)t * ma + j];
      }
    }
  }
  // level 1: block pattern and contributions from the fine faces
  {
    const std::vector<int>& agg = H.transfers[0].agg_of;
    const int nc = M.nc[1];
    std::vector<std::map<int, std::vector<int4>>> rows(nc);
    for (int a = 0; a < nc; ++a) rows[a][a];
    for (int f = 0; f < fm.n_faces; ++f) {
      if (fm.bc[f] == 0) {
        const int K = fm.fk[f], Lc = fm.fl[f];
        const int e = (int)(soff[K >> 5] + 32L * face_pos[f] + (K & 31));
        const int a = agg[K], b = agg[Lc];
        if (a == b) {
          rows[a][a].push_back(make_int4(K, Lc, e, 0));
        } else {
          rows[a][a].push_back(make_int4(K, K, e, 1));
          rows[b][b].push_back(make_int4(Lc, Lc, e, 1));
          rows[a][b].push_back(make_int4(K, Lc, e, 2));
          rows[b][a].push_back(make_int4(Lc, K, e, 2));
        }
      } else if (fm.bc[f] == 1) {
        const int K = fm.fk[f];
        rows[agg[K]][agg[K]].push_back(make_int4(K, doff[K] + dir_pos[f], 0, 3));
      }
    }
    M.rowptr[1].assign(nc + 1, 0);
    M.dpos[1].assign(nc, 0);
    M.asm_off[1].push_back(0);
    for (int a = 0; a < nc; ++a) {
      for (auto& kv : rows[a]) {
        if (kv.first == a) M.dpos[1][a] = (int)M.col[1].size();
        M.col[1].push_back(kv.first);
        for (const int4& t : kv.second) M.asm_list[1].push_back(t);
        M.asm_off[1].push_back((int)M.asm_list[1].size());
      }
      M.rowptr[1][a + 1] = (int)M.col[1].size();
    }
    M.nblk[1] = (int)M.col[1].size();
  }
  // levels l >= 2: from the blocks of level l-1
  for (int l = 2; l < levels; ++l) {
    const std::vector<int>& agg = H.transfers[l - 1].agg_of;
    const int nc = M.nc[l], ncf = M.nc[l - 1];
    std::vector<std::map<int, std::vector<int4>>> rows(nc);
    for (int a = 0; a < nc; ++a) rows[a][a];
    for (int c = 0; c < ncf; ++c)
      for (int q = M.rowptr[l - 1][c]; q < M.rowptr[l - 1][c + 1]; ++q) {
        const int d = M.col[l - 1][q];
        rows[agg[c]][agg[d]].push_back(make_int4(q, c, d, 0));
      }
    M.rowptr[l].assign(nc + 1, 0);
    M.dpos[l].assign(nc, 0);
    M.asm_off[l].push_back(0);
    for (int a = 0; a < nc; ++a) {
      for (auto& kv : rows[a]) {
        if (kv.first == a) M.dpos[l][a] = (int)M.col[l].size();
        M.col[l].push_back(kv.first);
        for (const int4& t : kv.second) M.asm_list[l].push_back(t);
        M.asm_off[l].push_back((int)M.asm_list[l].size());
      }
      M.rowptr[l][a + 1] = (int)M.col[l].size();
    }
    M.nblk[l] = (int)M.col[l].size();
  }
  return true;
}

// ---------------------------------------------------------------------------------------------------------------
// host: enqueueing

namespace {

// Launches with programmatic stream serialization (each kernel starts its launch while its predecessor finishes;
// pdl_start() in every kernel orders the memory accesses). Launch errors surface through cudaGetLastError().
template <class... KArgs, class... Args>
void launchk(cudaStream_t st, int grid, int block, size_t smem, void (*k)(KArgs...), Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, (KArgs)args...);
}

inline int warps_grid(long warps) { return blocks_for(warps * 32, 65535); }
// blocks of the row-parallel block-level kernels: one per group of 32 cells
inline int row_grid(int nc) { return (int)std::min<long>((nc + 31) / 32, 1 << 20); }

// One Chebyshev step k, and the residual, of block level l: row-parallel from W.row_cells cells up, else one warp per
// cell.
void cheb_level(cudaStream_t st, const MgDev& M, const MgWork& W, int l, int k, int cur, const int* flag) {
  if (M.nc[l] >= W.row_cells) {
    MG_MB_SWITCH(M.mb[l], launchk(st, row_grid(M.nc[l]), 32 * MB, 0, k_chebr<MB>, M.nc[l], (const int*)M.rowptr[l],
                                  (const int*)M.col[l], (const float*)W.aval[l], (const float*)W.dinv[l],
                                  (const float*)W.b[l], (const float*)W.x[l][cur], W.x[l][1 - cur], W.d[l],
                                  (const float*)W.coef, l, k, flag));
  } else {
    MG_MB_SWITCH(M.mb[l], launchk(st, warps_grid(M.nc[l]), kT, 0, k_chebl<MB>, M.nc[l], (const int*)M.rowptr[l],
                                  (const int*)M.col[l], (const float*)W.aval[l], (const float*)W.dinv[l],
                                  (const float*)W.b[l], (const float*)W.x[l][cur], W.x[l][1 - cur], W.d[l],
                                  (const float*)W.coef, l, k, flag));
  }
}
void res_level(cudaStream_t st, const MgDev& M, const MgWork& W, int l, int cur, const int* flag) {
  if (M.nc[l] >= W.row_cells) {
    MG_MB_SWITCH(M.mb[l], launchk(st, row_grid(M.nc[l]), 32 * MB, 0, k_resr<MB>, M.nc[l], (const int*)M.rowptr[l],
                                  (const int*)M.col[l], (const float*)W.aval[l], (const float*)W.b[l],
                                  (const float*)W.x[l][cur], W.d[l], flag));
  } else {
    MG_MB_SWITCH(M.mb[l], launchk(st, warps_grid(M.nc[l]), kT, 0, k_resl<MB>, M.nc[l], (const int*)M.rowptr[l],
                                  (const int*)M.col[l], (const float*)W.aval[l], (const float*)W.b[l],
                                  (const float*)W.x[l][cur], W.d[l], flag));
  }
}

// Whether level l's residual and restriction are one kernel: where the residual takes a warp per cell, the blocks (one
// per cell of level l+1) are at most a wave, four an SM, beyond which they lose their early loads and more than they save
// (10^6 cells, 1,935 blocks: the CG iteration 250.8 -> 251.8 us; 64^3, 508 blocks: 98.0 -> 95.5), and aggregates are small
// (with more than two children a warp few blocks walk a long chain).
bool fused_restr(const MgDev& M, const MgWork& W, int l) {
  return M.nc[l] < W.row_cells && M.nc[l + 1] <= W.fused_max && M.nc[l] <= 16L * M.nc[l + 1];
}

// b_(l+1) = P^T (b_l - A x_l), and (first) level l+1's first smoothing step.
template <class PT>
void restrict_level(cudaStream_t st, const MgDev& M, const MgWork& W, int l, int cur, const PT* P, int first,
                    const int* flag) {
  const float* dinv = first ? W.dinv[l + 1] : nullptr;
  float *xc = first ? W.x[l + 1][0] : nullptr, *dc = first ? W.d[l + 1] : nullptr;
  if (fused_restr(M, W, l)) {
    MG_MB_SWITCH(M.mb[l], launchk(st, M.nc[l + 1], kT, 0, k_res_restr<PT, MB>, (const int*)M.rowptr[l],
                                  (const int*)M.col[l], (const float*)W.aval[l], (const float*)W.b[l],
                                  (const float*)W.x[l][cur], P, (const int*)M.ch_off[l], (const int*)M.ch[l],
                                  M.mb[l + 1], W.b[l + 1], dinv, xc, dc, (const float*)W.coef, l + 1, first, flag));
  } else {
    res_level(st, M, W, l, cur, flag);
    launchk(st, warps_grid(M.nc[l + 1]), kT, 0, k_restr<PT>, M.mb[l], (const float*)W.d[l], P,
            (const int*)M.ch_off[l], (const int*)M.ch[l], M.nc[l + 1], M.mb[l + 1], W.b[l + 1], dinv, xc, dc,
            (const float*)W.coef, l + 1, first, flag);
  }
}

}  // namespace

void mg_enqueue_setup(cudaStream_t st, const MgDev& M, const FineDev& F, const MgWork& W, const double* Tval,
                      const double* diagT, const double* r) {
  cudaMemsetAsync(W.lam, 0, kMgMaxLevels * sizeof(float), st);
  launchk(st, blocks_for(M.N, 4096), kT, 0, k_fine_vals, F, Tval, diagT, W.a0off, W.a0diag, W.a0dinv, W.lam);
  int n = 2;
  const int per = M.mb[1] == 4 ? 2 : 1;   // blocks a warp of k_asm1
  if (W.bf16) {
    MG_MB_SWITCH(M.mb[1], launchk(st, warps_grid((M.nblk[1] + per - 1) / per), kT, 0, k_asm1<MB, __nv_bfloat16>, M.nblk[1],
                                  (const int*)M.asm_off[1], (const int4*)M.asm_list[1],
                                  (const __nv_bfloat16*)M.Pb[0], (const float*)W.a0off, r, (const double*)F.dir_ups,
                                  W.aval[1]));
  } else {
    MG_MB_SWITCH(M.mb[1], launchk(st, warps_grid((M.nblk[1] + per - 1) / per), kT, 0, k_asm1<MB, float>, M.nblk[1],
                                  (const int*)M.asm_off[1], (const int4*)M.asm_list[1], (const float*)M.P[0],
                                  (const float*)W.a0off, r, (const double*)F.dir_ups, W.aval[1]));
  }
  auto pad = [&](int l) {
    if (!M.padded[l]) return;
    launchk(st, blocks_for(M.nc[l]), kT, 0, k_pad_diag, M.nc[l], M.mb[l], (const int*)M.dpos[l], (const int*)M.mcnt[l],
            W.aval[l]);
    ++n;
  };
  pad(1);
  for (int l = 2; l < M.L; ++l) {
    if (W.bf16) {
      MG_MB_SWITCH(M.mb[l], launchk(st, warps_grid(M.nblk[l]), kT, 0, k_asml<MB, __nv_bfloat16>, M.nblk[l],
                                    M.mb[l - 1], (const int*)M.asm_off[l], (const int4*)M.asm_list[l],
                                    (const __nv_bfloat16*)M.Pb[l - 1], (const float*)W.aval[l - 1], W.aval[l]));
    } else {
      MG_MB_SWITCH(M.mb[l], launchk(st, warps_grid(M.nblk[l]), kT, 0, k_asml<MB, float>, M.nblk[l], M.mb[l - 1],
                                    (const int*)M.asm_off[l], (const int4*)M.asm_list[l], (const float*)M.P[l - 1],
                                    (const float*)W.aval[l - 1], W.aval[l]));
    }
    ++n;
    pad(l);
  }
  for (int l = 1; l + 1 < M.L; ++l) {
    MG_MB_SWITCH(M.mb[l], launchk(st, (M.nc[l] + 31) / 32, 32, 0, k_block_inv<MB>, M.nc[l], (const int*)M.dpos[l],
                                  (const float*)W.aval[l], W.dinv[l]));
    MG_MB_SWITCH(M.mb[l], launchk(st, warps_grid(M.nc[l]), kT, 0, k_block_bound<MB>, M.nc[l], (const int*)M.rowptr[l],
                                  (const float*)W.aval[l], (const float*)W.dinv[l], W.lam + l));
    n += 2;
  }
  launchk(st, 1, 32, 0, k_cheb_table, (const float*)W.lam, W.coef);
  const int C = M.L - 1;
  launchk(st, kInvCtas, kInvThreads, 0, k_coarse_inv, M.nc[C], M.mb[C], (const int*)M.rowptr[C], (const int*)M.col[C],
          (const float*)W.aval[C], W.cinv);
  const int t = mg_tail_level(M);
  if (t > 0) {
    const int nt = M.nc[t] * M.mb[t];
    if (W.bf16) launchk(st, nt, kTailThreads, W.tail_smem, k_tail_cols<__nv_bfloat16>, (const MgTailTab*)W.tail, W.tailE);
    else launchk(st, nt, kTailThreads, W.tail_smem, k_tail_cols<float>, (const MgTailTab*)W.tail, W.tailE);
    ++n;
  }
  count_launch(n + 2);
}

namespace {

// Shared-memory layout of the small levels from t on (byte offsets, every array in whole 16-byte units); returns the
// total. P slots are sized for FP32 (BF16 transfers use half of theirs).
size_t small_layout(const MgDev& M, int t, MgTailTab* T) {
  const int C = M.L - 1;
  size_t off = 0;
  auto put = [&](unsigned* o, size_t bytes) {
    if (o) *o = (unsigned)off;
    off += (bytes + 15) & ~(size_t)15;
  };
  for (int l = t - 1; l < C; ++l) {   // transfers l -> l+1
    put(T ? &T->o_P[l] : nullptr, (size_t)M.nc[l] * M.mb[l] * M.mb[l + 1] * 4);
    put(T ? &T->o_choff[l] : nullptr, ((size_t)M.nc[l + 1] + 1) * 4);
    put(T ? &T->o_ch[l] : nullptr, (size_t)M.nc[l] * 4);
    put(T ? &T->o_agg[l] : nullptr, (size_t)M.nc[l] * 4);
  }
  for (int l = t; l <= C; ++l) {
    const size_t n = (size_t)M.nc[l] * M.mb[l], mm = (size_t)M.mb[l] * M.mb[l];
    put(T ? &T->o_b[l] : nullptr, n * 4);
    put(T ? &T->o_x[l][0] : nullptr, n * 4);
    if (l == C) break;
    put(T ? &T->o_rowptr[l] : nullptr, ((size_t)M.nc[l] + 1) * 4);
    put(T ? &T->o_col[l] : nullptr, (size_t)M.nblk[l] * 4);
    put(T ? &T->o_aval[l] : nullptr, (size_t)M.nblk[l] * mm * 4);
    put(T ? &T->o_dinv[l] : nullptr, (size_t)M.nc[l] * mm * 4);
    put(T ? &T->o_x[l][1] : nullptr, n * 4);
    put(T ? &T->o_d[l] : nullptr, n * 4);
  }
  const size_t nco = (size_t)M.nc[C] * M.mb[C];
  put(T ? &T->o_cinv : nullptr, nco * nco * 4);
  put(T ? &T->o_coef : nullptr, kMgMaxLevels * kMgMaxDeg * 2 * 4);
  return off;
}

}  // namespace

int mg_tail_level(const MgDev& M) {
  const int C = M.L - 1;
  for (int l = 2; l <= C; ++l)
    if (M.nc[l] * M.mb[l] <= kTailMaxUnknowns && small_layout(M, l, nullptr) <= kTailSmem) return l;
  return 0;
}

void mg_fill_tail(cudaStream_t st, const MgDev& M, MgWork& W) {
  MgTailTab h;
  h.M = M;
  h.t = mg_tail_level(M);
  W.tail_smem = 0;
  if (h.t > 0) {
    const int t = h.t, C = M.L - 1;
    W.tail_smem = small_layout(M, t, &h);
    // copy list: the static structure, the per-setup matrices and transfers (FP32 or BF16 P)
    for (int v = 0; v < 2; ++v) {
      unsigned c0 = 0;
      int n = 0;
      auto add = [&](const void* src, unsigned dst, size_t bytes) {
        const unsigned ch = (unsigned)((bytes + 15) / 16);
        if (ch == 0) return;
        h.cp[v][n++] = MgTailCopy{src, dst, c0};
        c0 += ch;
      };
      for (int l = t - 1; l < C; ++l) {
        const size_t np = (size_t)M.nc[l] * M.mb[l] * M.mb[l + 1];
        if (v == 0) add(M.P[l], h.o_P[l], np * 4);
        else add(M.Pb[l], h.o_P[l], np * 2);
        add(M.ch_off[l], h.o_choff[l], ((size_t)M.nc[l + 1] + 1) * 4);
        add(M.ch[l], h.o_ch[l], (size_t)M.nc[l] * 4);
        add(M.agg[l], h.o_agg[l], (size_t)M.nc[l] * 4);
      }
      for (int l = t; l < C; ++l) {
        const size_t mm = (size_t)M.mb[l] * M.mb[l];
        add(M.rowptr[l], h.o_rowptr[l], ((size_t)M.nc[l] + 1) * 4);
        add(M.col[l], h.o_col[l], (size_t)M.nblk[l] * 4);
        add(W.aval[l], h.o_aval[l], (size_t)M.nblk[l] * mm * 4);
        add(W.dinv[l], h.o_dinv[l], (size_t)M.nc[l] * mm * 4);
      }
      const size_t nco = (size_t)M.nc[C] * M.mb[C];
      add(W.cinv, h.o_cinv, nco * nco * 4);
      add(W.coef, h.o_coef, kMgMaxLevels * kMgMaxDeg * 2 * 4);
      h.ncopies[v] = n;
      h.nchunks[v] = (int)c0;
    }
  }
  // pageable source: the call returns once the table is staged, so h may go out of scope
  cudaMemcpyAsync(W.tail, &h, sizeof(MgTailTab), cudaMemcpyHostToDevice, st);
}

// The V-cycle after the fused first step of level 0 (x[0][0], d[0] set from b[0]); returns the index of the level-0
// buffer that holds z. Levels from mg_tail_level on are one precomputed map (k_tail_cols).
int mg_enqueue_vcycle(cudaStream_t st, const MgDev& M, const FineDev& F, const MgWork& W, const int* flag,
                      bool cg_beta) {
  const int L = M.L, C = L - 1;
  const int tl = mg_tail_level(M);
  const int top = tl > 0 ? tl - 1 : C;   // levels 1 .. top-1 restrict with their own kernels
  int cur[kMgMaxLevels] = {0};
  const int g0 = blocks_for(M.N, W.grid0);
  // down: level-0 smoothing, residual into d[0] (dead until the post-smoothing rewrites it), restriction
  for (int k = 1; k < kMgDegFine; ++k) {
    launchk(st, g0, kT, 0, k_cheb0, F, (const float*)W.a0off, (const float*)W.a0diag, (const float*)W.a0dinv,
            (const float*)W.b[0], (const float*)W.x[0][cur[0]], W.x[0][1 - cur[0]], W.d[0], (const float*)W.coef, k,
            flag);
    cur[0] ^= 1;
  }
  launchk(st, g0, kT, 0, k_res0, F, (const float*)W.a0off, (const float*)W.a0diag, (const float*)W.b[0],
          (const float*)W.x[0][cur[0]], W.d[0], flag);
  if (W.bf16) {
    MG_MB_SWITCH(M.mb[1], launchk(st, warps_grid(M.nc[1]), kT, 0, k_restr0<__nv_bfloat16, MB>, (const float*)W.d[0],
                                  (const __nv_bfloat16*)M.Pb[0], (const int*)M.ch_off[0], (const int*)M.ch[0], M.nc[1],
                                  W.b[1], (const float*)W.dinv[1], W.x[1][0], W.d[1], (const float*)W.coef,
                                  C > 1 ? 1 : 0, flag));
  } else {
    MG_MB_SWITCH(M.mb[1], launchk(st, warps_grid(M.nc[1]), kT, 0, k_restr0<float, MB>, (const float*)W.d[0],
                                  (const float*)M.P[0], (const int*)M.ch_off[0], (const int*)M.ch[0], M.nc[1], W.b[1],
                                  (const float*)W.dinv[1], W.x[1][0], W.d[1], (const float*)W.coef, C > 1 ? 1 : 0,
                                  flag));
  }
  for (int l = 1; l < C && l <= top; ++l) {
    for (int k = 1; k < kMgDegCoarse; ++k) {
      cheb_level(st, M, W, l, k, cur[l], flag);
      cur[l] ^= 1;
    }
    const int first = l != top && l + 1 < C ? 1 : 0;   // (the map holds level top + 1's own)
    if (W.bf16) restrict_level(st, M, W, l, cur[l], (const __nv_bfloat16*)M.Pb[l], first, flag);
    else restrict_level(st, M, W, l, cur[l], (const float*)M.P[l], first, flag);
  }
  if (tl > 0) {   // the small levels' map back to level tl - 1
    const int nt = M.nc[tl] * M.mb[tl], rows = M.nc[tl - 1] * M.mb[tl - 1];
    launchk(st, (rows + 31) / 32, 32 * kApplyWarps, 0, k_tail_apply, rows, nt, (const float*)W.tailE,
            (const float*)W.b[tl], W.x[tl - 1][cur[tl - 1]], flag);
  } else {
    launchk(st, 1, kMgMaxCoarse, 0, k_coarse_solve, M.nc[C] * M.mb[C], (const float*)W.cinv, (const float*)W.b[C],
            W.x[C][0], flag);
  }
  // up
  for (int l = std::min(top, C - 1); l >= 1; --l) {
    if (l != top || tl == 0) {
      if (W.bf16)
        launchk(st, blocks_for((long)M.nc[l] * M.mb[l]), kT, 0, k_prol<__nv_bfloat16>, M.nc[l], M.mb[l],
                M.mb[l + 1], (const __nv_bfloat16*)M.Pb[l], (const int*)M.agg[l],
                (const float*)W.x[l + 1][cur[l + 1]], W.x[l][cur[l]], flag);
      else
        launchk(st, blocks_for((long)M.nc[l] * M.mb[l]), kT, 0, k_prol<float>, M.nc[l], M.mb[l], M.mb[l + 1],
                (const float*)M.P[l], (const int*)M.agg[l], (const float*)W.x[l + 1][cur[l + 1]], W.x[l][cur[l]],
                flag);
    }
    for (int k = 0; k < kMgDegCoarse; ++k) {
      cheb_level(st, M, W, l, k, cur[l], flag);
      cur[l] ^= 1;
    }
  }
  if (W.bf16)
    launchk(st, g0, kT, 0, k_pro0<__nv_bfloat16>, M.N, M.mb[1], (const __nv_bfloat16*)M.Pb[0],
            (const int*)M.agg[0], (const float*)W.x[1][cur[1]], W.x[0][cur[0]], flag);
  else
    launchk(st, g0, kT, 0, k_pro0<float>, M.N, M.mb[1], (const float*)M.P[0], (const int*)M.agg[0],
            (const float*)W.x[1][cur[1]], W.x[0][cur[0]], flag);
  for (int k = 0; k < kMgDegFine; ++k) {
    if (cg_beta && k + 1 == kMgDegFine)
      launchk(st, blocks_for(M.N, kMaxRedBlocks), kT, 0, k_cheb0_beta, F, (const float*)W.a0off,
              (const float*)W.a0diag, (const float*)W.a0dinv, (const float*)W.b[0], (const float*)W.x[0][cur[0]],
              W.x[0][1 - cur[0]], W.d[0], (const float*)W.coef, k, (const double*)W.kr, (const float*)W.z[0], W.part,
              W.sc);
    else
      launchk(st, g0, kT, 0, k_cheb0, F, (const float*)W.a0off, (const float*)W.a0diag, (const float*)W.a0dinv,
              (const float*)W.b[0], (const float*)W.x[0][cur[0]], W.x[0][1 - cur[0]], W.d[0], (const float*)W.coef,
              k, flag);
    cur[0] ^= 1;
  }
  return cur[0];
}

int mg_vcycle_kernels(const MgDev& M, const MgWork& W) {
  const int C = M.L - 1, tl = mg_tail_level(M);
  int n = (kMgDegFine - 1) + 2 + 1 + kMgDegFine;   // level 0: smoothing, residual, restriction, prolongation
  // levels with their own kernels: smoothing, residual and restriction (one or two), and on the way up the prolongations
  // between them; then the map, or the coarsest solve and the prolongation from it
  const int own = tl > 0 ? tl - 1 : C - 1;
  for (int l = 1; l <= own; ++l) n += (kMgDegCoarse - 1) + (fused_restr(M, W, l) ? 1 : 2) + kMgDegCoarse;
  return n + (tl > 0 ? std::max(own - 1, 0) : own) + 1;
}

namespace {

// A graph with one conditional while node whose body is captured from `body(handle)`.
template <class Body>
cudaError_t capture_while(cudaStream_t st, Body&& body, cudaGraphExec_t* out) {
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaGraphCreate(&g, 0);
  if (e != cudaSuccess) return e;
  cudaGraphConditionalHandle h;
  e = cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault);
  if (e == cudaSuccess) {
    cudaGraphNodeParams np = {};
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = h;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    cudaGraphNode_t node;
    e = cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &np);
    if (e == cudaSuccess) {
      cudaGraph_t bg = np.conditional.phGraph_out[0];
      e = cudaStreamBeginCaptureToGraph(st, bg, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
      if (e == cudaSuccess) {
        body(h);
        cudaError_t e2 = cudaStreamEndCapture(st, &bg);
        e = e2 != cudaSuccess ? e2 : cudaGetLastError();
      }
    }
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  return e;
}

template <class Body>
cudaError_t capture_plain(cudaStream_t st, Body&& body, cudaGraphExec_t* out) {
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return e;
  body();
  e = cudaStreamEndCapture(st, &g);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaGraphInstantiate(out, g, 0);
  if (g) cudaGraphDestroy(g);
  return e;
}

}  // namespace

// Preconditioned CG for A dx = -b (b = W.kb, FP64; dx -> W.kx) as two graphs: out[0] the start (x = 0, r = -b with
// the first smoothing step of the first V-cycle), out[1] the conditional while loop over the iterations (V-cycle with
// beta in its last step, p and q, x and r with the convergence test). The tolerance and iteration cap are read from
// W.sc at run time.
cudaError_t mg_capture_pcg(cudaStream_t st, const MgDev& M, const FineDev& F, MgWork& W, const double* Tval,
                           const double* diagT, cudaGraphExec_t* out) {
  const int gr = blocks_for(M.N, kMaxRedBlocks);
  cudaError_t e = capture_plain(st, [&]() {
    launchk(st, gr, kT, 0, k_pcg_init, M.N, (const double*)W.kb, -1.0, W.kx, W.kr, W.b[0],
            (const float*)W.a0dinv, W.x[0][0], W.d[0], (const float*)W.coef, W.part, W.sc);
  }, &out[0]);
  if (e != cudaSuccess) return e;
  // the convergence test is the body's last kernel, so nothing runs after it; the V-cycle kernels need no stop flag
  // (they only write the preconditioner's scratch and z)
  return capture_while(st, [&](cudaGraphConditionalHandle h) {
    const float* z = W.x[0][mg_enqueue_vcycle(st, M, F, W, nullptr, true)];   // its last step gives beta
    launchk(st, gr, kT, 0, k_pcg_pq, F, Tval, diagT, z, W.z[0], W.kp, W.kq, W.part, W.sc);
    launchk(st, gr, kT, 0, k_pcg_update, M.N, (const double*)W.kp, (const double*)W.kq, W.kx, W.kr, W.b[0],
            (const float*)W.a0dinv, W.x[0][0], W.d[0], (const float*)W.coef, W.part, W.sc, h);
  }, &out[1]);
}

// Right-preconditioned BiCGStab for J dx = -b (J: jd diagonal, Joff off-diagonal in the SELL layout; b = W.kb;
// dx -> W.kx; stopping on ||W r|| with W^2 = wgt). out[0] the start (r, r^, p = r with the first smoothing step of
// p^ = B p), out[1] the loop: p (from the second iteration on), p^ = B p, v = J p^, s, s^ = B s, t = J s^, then x
// and r with the convergence test as the last kernel.
cudaError_t mg_capture_bicgstab(cudaStream_t st, const MgDev& M, const FineDev& F, MgWork& W, const double* jd,
                                const double* Joff, const double* wgt, cudaGraphExec_t* out) {
  const int gr = blocks_for(M.N, kMaxRedBlocks);
  cudaError_t e = capture_plain(st, [&]() {
    launchk(st, gr, kT, 0, k_bicg_init, M.N, (const double*)W.kb, -1.0, wgt, W.kx, W.kr, W.krh, W.kp, W.b[0],
            (const float*)W.a0dinv, W.x[0][0], W.d[0], (const float*)W.coef, W.part, W.sc);
  }, &out[0]);
  if (e != cudaSuccess) return e;
  return capture_while(st, [&](cudaGraphConditionalHandle h) {
    launchk(st, gr, kT, 0, k_bicg_p, M.N, (const double*)W.kr, (const double*)W.kv, W.kp, W.b[0],
            (const float*)W.a0dinv, W.x[0][0], W.d[0], (const float*)W.coef, W.sc);
    const int zp = mg_enqueue_vcycle(st, M, F, W, nullptr, false);
    launchk(st, gr, kT, 0, k_bicg_v, F, Joff, jd, (const float*)W.x[0][zp], W.kpp, W.kv, (const double*)W.krh,
            W.part, W.sc);
    launchk(st, gr, kT, 0, k_bicg_s, M.N, (const double*)W.kr, (const double*)W.kv, W.ks, W.b[0],
            (const float*)W.a0dinv, W.x[0][0], W.d[0], (const float*)W.coef, W.sc);
    const int zs = mg_enqueue_vcycle(st, M, F, W, nullptr, false);
    launchk(st, gr, kT, 0, k_bicg_t, F, Joff, jd, (const float*)W.x[0][zs], (const double*)W.ks, W.kt, W.part,
            W.sc);
    launchk(st, gr, kT, 0, k_bicg_x, M.N, (const double*)W.kpp, (const float*)W.x[0][zs], (const double*)W.ks,
            (const double*)W.kt, (const double*)W.krh, wgt, W.kx, W.kr, W.part, W.sc, h);
  }, &out[1]);
}

// One V-cycle z = B b for parity tests: b = W.kb (FP64) -> W.kx (FP64).
cudaError_t mg_capture_apply(cudaStream_t st, const MgDev& M, const FineDev& F, MgWork& W, cudaGraphExec_t* out) {
  return capture_plain(st, [&]() {
    const int g0 = blocks_for(M.N, W.grid0);
    launchk(st, g0, kT, 0, k_apply_in, M.N, (const double*)W.kb, W.b[0], (const float*)W.a0dinv, W.x[0][0], W.d[0],
            (const float*)W.coef);
    const int zi = mg_enqueue_vcycle(st, M, F, W, nullptr, false);
    launchk(st, g0, kT, 0, k_apply_out, M.N, (const float*)W.x[0][zi], W.kx);
  }, out);
}

cudaError_t mg_set_smem_limits() {
  static DeviceOnce f32, bf16;
  if (const cudaError_t e = raise_smem_limit(f32, (const void*)k_tail_cols<float>, kTailSmem)) return e;
  return raise_smem_limit(bf16, (const void*)k_tail_cols<__nv_bfloat16>, kTailSmem);
}

}  // namespace nlmg
