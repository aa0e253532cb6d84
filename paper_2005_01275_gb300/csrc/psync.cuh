// Synchronisation and sums of the persistent (cooperative) kernels: the bounded grid barrier, deterministic grid sums
// and the division that derives step lengths from them.
//
// What the sums cost, and why they run on the integer pipes, stands in isum.cuh.
#pragma once
#include <cuda_runtime.h>

#include "isum.cuh"
#include "persist.cuh"

namespace nlmg {

constexpr unsigned long long kSpinLimit = 1ull << 23;   // x ~0.2 us polls ~ 2 s
constexpr int kMaxNV = 6;                                // values per grid sum at most
constexpr int kMaxPWarps = 32;                           // warps of a persistent block at most
constexpr int kSmDoubles = 2 * kMaxNV * kMaxPWarps;      // block-reduction scratch: one integer sum per warp and value

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void red_add_release_gpu(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// The synchronisation state one thread of a persistent kernel carries: the launch's barrier words, the two
// buffers of per-block partial sums (used alternately by consecutive reductions), kSmDoubles doubles of shared
// memory, the number of reductions so far and the barrier phase (both the same in every block).
struct Grid {
  GridSync gs;
  double* partial;
  double* sm;
  unsigned seq;
  unsigned phase;   // the counter's top bit after the last barrier
};

// A grid of at most kClusterBlocks blocks is launched as one thread-block cluster (gs.cluster), whose hardware barrier takes
// the place of the counter: it orders the same writes at cluster scope, needs no polling and cannot be left waiting by a
// block that was never scheduled.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// The state at the start of a launch. The counter's top bit is wherever the last launch left it; no block can have
// completed a barrier of this launch before this block's first arrival, so every block reads the same bit.
__device__ __forceinline__ Grid grid_start(const GridSync& gs, double* partial, double* sm) {
  __shared__ unsigned phase;
  if (threadIdx.x == 0) phase = gs.cluster ? 0u : ld_acquire_gpu(gs.count) & 0x80000000u;
  __syncthreads();
  return Grid{gs, partial, sm, 0u, phase};
}

// One arrival and the bounded wait for all others, by one thread: every block adds 1 to gs.count except block 0, which
// adds 2^31 - (gridDim.x - 1), so the counter's top bit flips exactly when the last block arrives and its low bits
// return to 0 (barriers follow one another without a reset). The arrival is a release without a return value, the
// polls are acquire loads without a sleep (a sleep of 20 ns was measured to cost 2 us). Returns false (and sets *err)
// if the wait gave up after ~2 s or another block's did.
__device__ __forceinline__ void grid_arrive(Grid& g) {
  red_add_release_gpu(g.gs.count, blockIdx.x == 0 ? 0x80000000u - (gridDim.x - 1u) : 1u);
}
__device__ __forceinline__ bool grid_wait(Grid& g, unsigned long long spin_limit) {
  unsigned long long spins = 0;
  while (((ld_acquire_gpu(g.gs.count) ^ g.phase) & 0x80000000u) == 0u) {
    if ((++spins & 1023u) == 0 && (spins > spin_limit || *((volatile int*)g.gs.err) != 0)) {
      atomicExch(g.gs.err, 1);
      return false;
    }
  }
  return true;
}

// Bounded grid barrier: thread 0 arrives after __syncthreads (its release covers the block's earlier writes).
__device__ __forceinline__ bool grid_barrier(Grid& g, unsigned long long spin_limit = kSpinLimit) {
  if (g.gs.cluster) {
    cluster_arrive();
    cluster_wait();
    return true;
  }
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    grid_arrive(g);
    ok = grid_wait(g, spin_limit) ? 1 : 0;
  }
  g.phase ^= 0x80000000u;
  __syncthreads();
  return ok != 0;
}

// Grid sums of NV values, in two halves, for a block whose warp `server` does the serial part (it may hold values too).
// grid_sum_arrive: warp sums, the block's sums to the partial buffer, then the grid barrier; on return every block's
// earlier writes and partials are visible. The other warps run `meanwhile` (on registers) while the server waits.
// grid_sum_finish, by the server warp alone: every block's partials added (all blocks get bit-identical sums, so they take
// the same decisions); every lane of that warp returns the sums.
// Consecutive reductions use the two partial buffers in turn: a block can only overwrite a buffer after every block
// has passed the next barrier, i.e. has finished reading it.
template <int NV>
__device__ __forceinline__ constexpr int part_stride() {   // doubles of a block's partials: whole double2
  return NV <= 2 ? 2 : NV <= 4 ? 4 : 8;
}
template <int NV, class Work>
__device__ __forceinline__ bool grid_sum_arrive(Grid& g, const double (&v)[NV], int server, Work&& meanwhile) {
  static_assert(NV >= 1 && NV <= kMaxNV, "grid sums: the shared scratch holds kMaxNV values per warp");
  __shared__ int ok;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  ISum* sm = (ISum*)g.sm;
  {
    double a[NV][1];
    ISum s[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) a[k][0] = v[k];
    warp_sums<NV, 1>(a, s);
    if (lane < NV) {
      ISum mine = s[0];
#pragma unroll
      for (int k = 1; k < NV; ++k)
        if (lane == k) mine = s[k];
      sm[lane * kMaxPWarps + warp] = mine;
    }
  }
  __syncthreads();
  ++g.seq;
  if (warp == server) {
    ISum a[NV];
    double s[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) a[k] = lane < nw ? sm[k * kMaxPWarps + lane] : ISum{0ll, 0};
    warp_sums_i<NV>(a, s);
    if (lane < NV) {
      double mine = s[0];
#pragma unroll
      for (int k = 1; k < NV; ++k) mine = lane == k ? s[k] : mine;
      g.partial[((g.seq - 1u) & 1u) * kPartStride + blockIdx.x * part_stride<NV>() + lane] = mine;
    }
    __syncwarp();
    if (lane == 0 && !g.gs.cluster) {
      grid_arrive(g);
      ok = grid_wait(g, kSpinLimit) ? 1 : 0;
    }
    __syncwarp();
  }
  if (g.gs.cluster) {
    cluster_arrive();
    if (warp != server) meanwhile();
    cluster_wait();
    return true;
  }
  if (warp != server) meanwhile();
  g.phase ^= 0x80000000u;
  __syncthreads();
  return ok != 0;
}
template <int NV>
__device__ __forceinline__ bool grid_sum_arrive(Grid& g, const double (&v)[NV], int server) {
  return grid_sum_arrive<NV>(g, v, server, [] {});
}
template <int NV>
__device__ __forceinline__ void grid_sum_finish(const Grid& g, double (&s)[NV]) {
  constexpr int M = 5, ST = part_stride<NV>();   // partials per lane: up to 160 blocks in one step
  const double2* part = (const double2*)(g.partial + ((g.seq - 1u) & 1u) * kPartStride);
  const int lane = threadIdx.x & 31, G = (int)gridDim.x;
  double a[NV][M];
  ISum t[NV];
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const int b = lane + 32 * j;
#pragma unroll
    for (int k = 0; k < NV; k += 2) {
      const double2 x = b < G ? __ldcg(&part[(b * ST + k) / 2]) : make_double2(0.0, 0.0);
      a[k][j] = x.x;
      if (k + 1 < NV) a[k + 1][j] = x.y;
    }
  }
  // larger grids (the memory-resident kernels put two blocks on an SM): the rest onto the lane's first value in double, in
  // block order
  for (int b = 32 * M + lane; b < G; b += 32)
#pragma unroll
    for (int k = 0; k < NV; ++k) a[k][0] += __ldcg((const double*)part + b * ST + k);
  warp_sums<NV, M>(a, t);
#pragma unroll
  for (int k = 0; k < NV; ++k) s[k] = isum_value(t[k]);
}

// Grid sums that every thread needs at once, followed by `post(o)` on the NV sums, which derives NX scalars from them
// (the CG step lengths) into o[NV..NV+NX-1]: it runs once per block, in warp 0.
template <int NV, int NX = 0, class PostFn>
__device__ __forceinline__ bool grid_sum_x(Grid& g, double (&v)[NV + NX], PostFn&& post) {
  __shared__ double o[NV + NX];
  double in[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) in[k] = v[k];
  if (!grid_sum_arrive<NV>(g, in, 0)) return false;
  if (threadIdx.x < 32) {
    double s[NV];
    grid_sum_finish<NV>(g, s);
    double x[NV + NX];
#pragma unroll
    for (int k = 0; k < NV; ++k) x[k] = s[k];
    post(x);
    if (threadIdx.x == 0)
#pragma unroll
      for (int k = 0; k < NV + NX; ++k) o[k] = x[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV + NX; ++k) v[k] = o[k];
  return true;
}

template <int NV>
__device__ __forceinline__ bool grid_sum(Grid& g, double (&v)[NV]) {
  return grid_sum_x<NV, 0>(g, v, [](double*) {});
}

// Max over the warp of a non-negative value (their bits order like unsigned integers), in every lane.
__device__ __forceinline__ double warp_max(double m) {
  const unsigned hi = (unsigned)__double2hiint(m), mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)__double2loint(m) : 0u);
  return __hiloint2double((int)mh, (int)ml);
}

// post(max over the grid of one non-negative value per thread) (exact, hence deterministic), by the same protocol; post
// runs in warp 0.
template <class PostFn>
__device__ __forceinline__ bool grid_max(Grid& g, double& v, PostFn&& post) {
  __shared__ double o;
  double* part = g.partial + (g.seq & 1u) * kPartStride;
  ++g.seq;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double m = warp_max(v);
  if (lane == 0) g.sm[warp] = m;
  __syncthreads();
  if (warp == 0) {
    m = warp_max(lane < nw ? g.sm[lane] : 0.0);
    if (lane == 0) part[blockIdx.x] = m;
  }
  if (!grid_barrier(g)) return false;
  if (warp == 0) {
    m = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) m = fmax(m, __ldcg(&part[b]));
    m = post(warp_max(m));
    if (lane == 0) o = m;
  }
  __syncthreads();
  v = o;
  return true;
}

// Items 0 .. n-1 over the warps of the grid: consecutive groups of 32 go to consecutive blocks, so a level with few
// items is spread over all SMs (an SM issues one FP64 warp operation every 19 clocks: 16 warps on one SM take 16 times
// as long as one warp on each of 16; equal runs of groups per block were measured slower: level-0 BiCGStab on 48^3
// cells 9.85 ms against 9.27). The item of a thread is the same in every pass over the same n.
#define GSTRIDE(i, n)                                                                                     \
  for (int i = (int)(((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32u + (threadIdx.x & 31u)); i < (n); \
       i += (int)(gridDim.x * blockDim.x))

// The same from the last warp down: for a second set of items in the same pass, on the warps the first set leaves idle.
#define TSTRIDE(i, n)                                                                                         \
  for (int i = (int)((((blockDim.x - 1u - threadIdx.x) >> 5) * gridDim.x + blockIdx.x) * 32u + (threadIdx.x & 31u)); \
       i < (n); i += (int)(gridDim.x * blockDim.x))

// Rows 0 .. n-1 of short sums, four lanes (part of a warp) a row: lane gi = 0 .. 3 of a row's group takes its entries gi,
// gi + 4, ..., and quad_sum adds the four. A thread a row walks one chain of dependent loads and 64-clock FP64
// operations as long as the row; four lanes a row cut it to a quarter, read the row's entries side by side, and still
// leave a warp's operations mostly busy. The loop is the same for all lanes of a warp (row >= n: no row).
#define QSTRIDE(row, n)                                                                                           \
  for (int qb_ = (int)(((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 8u), row = qb_ + (int)((threadIdx.x & 31u) >> 2); \
       qb_ < (n); qb_ += (int)(gridDim.x * (blockDim.x >> 2)), row = qb_ + (int)((threadIdx.x & 31u) >> 2))
__device__ __forceinline__ double quad_sum(double v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v;
}

// Tests and signs of a double on the integer pipe.
__device__ __forceinline__ bool nonzero(double v) { return ((__double2hiint(v) << 1) | __double2loint(v)) != 0; }
__device__ __forceinline__ bool finite_bits(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
// v, or -v when neg is 1
__device__ __forceinline__ double flip(double v, int neg) {
  return __hiloint2double(__double2hiint(v) ^ (neg << 31), __double2loint(v));
}

}  // namespace nlmg
