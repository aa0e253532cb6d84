// Calls the library's device arithmetic (sums over warps, blocks and grids) on host arrays, for the tests that
// compare it with exact arithmetic.
#include <cuda_runtime.h>

#include "../paper_2005_01275_gb300/csrc/isum.cuh"
#include "../paper_2005_01275_gb300/csrc/psync.cuh"

using namespace nlmg;

namespace {

// v: [block][NV][M][threads]; out: [block][NV]
template <int NV, int M>
__global__ void k_block(const double* v, double* out) {
  __shared__ ISum sm[NV * 32];
  double a[NV][M], s[NV];
  for (int k = 0; k < NV; ++k)
    for (int j = 0; j < M; ++j) a[k][j] = v[((size_t)(blockIdx.x * NV + k) * M + j) * blockDim.x + threadIdx.x];
  block_sums<NV, M>(a, s, sm, blockDim.x / 32);
  if (threadIdx.x == 0)
    for (int k = 0; k < NV; ++k) out[blockIdx.x * NV + k] = s[k];
}

// v: [NV][block][threads]; out: [block][NV] (every block reports what it got)
template <int NV>
__global__ void __launch_bounds__(512) k_grid(const double* v, double* out, double* partial, GridSync gs) {
  __shared__ double sm[kSmDoubles];
  Grid g = grid_start(gs, partial, sm);
  double a[NV];
  for (int k = 0; k < NV; ++k) a[k] = v[((size_t)k * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x];
  if (!grid_sum<NV>(g, a)) return;
  if (threadIdx.x == 0)
    for (int k = 0; k < NV; ++k) out[blockIdx.x * NV + k] = a[k];
}

// Copies n doubles in, runs `launch` on device buffers and copies m doubles out.
template <class F>
int with_buffers(const double* v, size_t n, double* out, size_t m, F&& launch) {
  double *dv = nullptr, *dout = nullptr;
  cudaError_t e = cudaMalloc(&dv, n * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&dout, m * sizeof(double));
  if (e == cudaSuccess) e = cudaMemcpy(dv, v, n * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = launch(dv, dout);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpy(out, dout, m * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFree(dv);
  cudaFree(dout);
  return (int)e;
}

}  // namespace

extern "C" int block_sums_host(const double* v, double* out, int blocks, int threads, int nv, int m) {
  return with_buffers(v, (size_t)blocks * threads * nv * m, out, (size_t)blocks * nv, [&](double* d, double* o) {
    if (nv == 1 && m == 1) k_block<1, 1><<<blocks, threads>>>(d, o);
    else if (nv == 3 && m == 1) k_block<3, 1><<<blocks, threads>>>(d, o);
    else if (nv == 1 && m == 4) k_block<1, 4><<<blocks, threads>>>(d, o);
    else if (nv == 2 && m == 5) k_block<2, 5><<<blocks, threads>>>(d, o);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
  });
}

// Sums of two values over a cooperative grid (cluster: over one cluster of `blocks` <= 8 blocks).
extern "C" int grid_sums_host(const double* v, double* out, int blocks, int threads, int cluster) {
  double* partial = nullptr;
  unsigned* words = nullptr;
  cudaError_t e = cudaMalloc(&partial, 2 * kPartStride * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&words, 64 * sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemset(words, 0, 64 * sizeof(unsigned));
  int r = (int)e;
  if (e == cudaSuccess)
    r = with_buffers(v, (size_t)2 * blocks * threads, out, (size_t)blocks * 2, [&](double* d, double* o) {
      GridSync gs{words, (int*)(words + 32), 0, cluster};
      const double* dv = d;
      void* args[] = {(void*)&dv, (void*)&o, (void*)&partial, (void*)&gs};
      if (!cluster) return cudaLaunchCooperativeKernel((const void*)k_grid<2>, dim3(blocks), dim3(threads), args, 0, 0);
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(blocks);
      cfg.blockDim = dim3(threads);
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = blocks;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      return cudaLaunchKernelExC(&cfg, (const void*)k_grid<2>, args);
    });
  cudaFree(partial);
  cudaFree(words);
  return r;
}

namespace {
__global__ void k_scalar(const double* v, double* out, int n, int op) {   // v: a, then b
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double a = v[i], b = v[n + i];
  out[i] = op == 0 ? fast_rcp(a) : op == 1 ? fast_div(a, b) : op == 2 ? (double)narrow(a) : widen((float)a);
}
}  // namespace

// op: 0 1 / a, 1 a / b, 2 the float next to a, 3 the double of a (a float)
extern "C" int scalar_host(const double* v, double* out, int n, int op) {
  return with_buffers(v, (size_t)2 * n, out, (size_t)n, [&](double* d, double* o) {
    k_scalar<<<(n + 127) / 128, 128>>>(d, o, n, op);
    return cudaGetLastError();
  });
}
