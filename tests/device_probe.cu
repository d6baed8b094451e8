// Device routines of the library behind plain C calls, for the tests that look at one routine alone, and
// the words in which a context's kernels report a wait that gave up.
#include <cuda_runtime.h>

#include "dev_state.cuh"
#include "device.cuh"

using namespace nls;

namespace {

template <typename FT>
__global__ void k_ring(int n, int b, const FT* P, FT* x, int stages, int* ok) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int BS = dev::SolveBlock<FT>::BS;
  FT* y = (FT*)smem;
  unsigned char* ring = smem + ((n + BS - 1) / BS * BS * sizeof(FT) + 127) / 128 * 128;
  for (int a = threadIdx.x; a < n; a += blockDim.x) y[a] = x[a];
  __syncthreads();
  const bool r = dev::band_solve_ring<FT>(n, b, P, y, ring, stages);
  if (threadIdx.x == 0) *ok = r ? 1 : 0;
  for (int a = threadIdx.x; a < n; a += blockDim.x) x[a] = y[a];
}

__global__ void k_log_inv(int n, const double* x, const double2* tab, double* log, double* inv) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const dev::LogInv r = dev::log_inv(x[i], tab);
  log[i] = r.log;
  inv[i] = r.inv;
}

template <typename FT>
__global__ void k_recip(int n, const FT* x, FT* y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = dev::recip<FT>(x[i]);
}
template <typename FT>
int recip_of(int n, const FT* x, FT* y) {
  FT *dx = nullptr, *dy = nullptr;
  cudaMalloc(&dx, n * sizeof(FT));
  cudaMalloc(&dy, n * sizeof(FT));
  cudaMemcpy(dx, x, n * sizeof(FT), cudaMemcpyHostToDevice);
  k_recip<FT><<<(n + 255) / 256, 256>>>(n, dx, dy);
  cudaMemcpy(y, dy, n * sizeof(FT), cudaMemcpyDeviceToHost);
  cudaFree(dx);
  cudaFree(dy);
  return (int)cudaGetLastError();
}

// x = (packed operands P)^-1 x in one CTA, `host` arrays in and out; without_copies: the CTA comes
// without its copying warp, so that no operand ever arrives.  Returns a CUDA error code.
template <typename FT>
int ring(int n, int b, const FT* P, FT* x, int stages, int without_copies, int* ok) {
  constexpr int BS = dev::SolveBlock<FT>::BS;
  const size_t nblk = (n + BS - 1) / BS, np = nblk * dev::packed_block_entries<FT>(b);
  const size_t sm = (nblk * BS * sizeof(FT) + 127) / 128 * 128 + dev::kRingHead + stages * dev::ring_stage_bytes<FT>(b);
  FT *dP = nullptr, *dx = nullptr;
  int* dok = nullptr;
  cudaMalloc(&dP, np * sizeof(FT));
  cudaMalloc(&dx, n * sizeof(FT));
  cudaMalloc(&dok, sizeof(int));
  cudaMemcpy(dP, P, np * sizeof(FT), cudaMemcpyHostToDevice);
  cudaMemcpy(dx, x, n * sizeof(FT), cudaMemcpyHostToDevice);
  cudaFuncSetAttribute(k_ring<FT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_ring<FT><<<1, dev::ring_threads<FT>(b) - (without_copies ? 32 : 0), sm>>>(n, b, dP, dx, stages, dok);
  cudaMemcpy(x, dx, n * sizeof(FT), cudaMemcpyDeviceToHost);
  cudaMemcpy(ok, dok, sizeof(int), cudaMemcpyDeviceToHost);
  cudaFree(dP);
  cudaFree(dx);
  cudaFree(dok);
  return (int)cudaGetLastError();
}

}  // namespace

extern "C" {

int probe_ring_f32(int n, int b, const float* P, float* x, int stages, int without_copies, int* ok) {
  return ring<float>(n, b, P, x, stages, without_copies, ok);
}
int probe_ring_f64(int n, int b, const double* P, double* x, int stages, int without_copies, int* ok) {
  return ring<double>(n, b, P, x, stages, without_copies, ok);
}

// log x[i] and 1 / x[i] as the element routines of Eq. 2 take them.
int probe_log_inv(int n, const double* x, double* log, double* inv) {
  const std::vector<double2> tab = dev::log_table();
  double2* dt = nullptr;
  double* d = nullptr;
  cudaMalloc(&dt, tab.size() * sizeof(double2));
  cudaMalloc(&d, 3 * (size_t)n * sizeof(double));
  cudaMemcpy(dt, tab.data(), tab.size() * sizeof(double2), cudaMemcpyHostToDevice);
  cudaMemcpy(d, x, n * sizeof(double), cudaMemcpyHostToDevice);
  k_log_inv<<<(n + 255) / 256, 256>>>(n, d, dt, d + n, d + 2 * (size_t)n);
  cudaMemcpy(log, d + n, n * sizeof(double), cudaMemcpyDeviceToHost);
  cudaMemcpy(inv, d + 2 * (size_t)n, n * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFree(dt);
  cudaFree(d);
  return (int)cudaGetLastError();
}

// 1 / x[i] as the band factorizations take it of a pivot.
int probe_recip_f32(int n, const float* x, float* y) { return recip_of<float>(n, x, y); }
int probe_recip_f64(int n, const double* x, double* y) { return recip_of<double>(n, x, y); }

// What a wait that gave up leaves behind: the flag of the triangular solves and, with a tiled coarse
// factorization, the status of the coarse cluster solves.  Returns whether there is such a status.
int probe_report_wait(void* ctx) {
  Dev& D = *((Context*)ctx)->dev;  // an nls_ctx holds its Context and nothing else
  *(volatile int*)D.err_host = 1;
  if (!D.tlu || !D.tlu->solve_status) return 0;
  const int32_t st = ST_TIMEOUT;
  cudaMemcpy(D.tlu->solve_status, &st, sizeof(st), cudaMemcpyHostToDevice);
  return 1;
}

}  // extern "C"
