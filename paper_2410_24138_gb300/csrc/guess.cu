// Learned initial guess for the local Newton solves (not part of the paper's method; see
// include/nls.h for the definition of inputs, outputs and the acceptance rule).  Two kinds of
// network: scalar (Eq. 1 on P1 triangles) and displacement (Eq. 2 on Q1 quadrilaterals, two
// components per node).
//
// Kernels:
//   k_guess_features   per subdomain: the 4 x 33 side samples of each component of x on the
//                      box one node beyond the local unknowns (clamped to the mesh); Eq. 1:
//                      log k on 16 x 16 points and the load factor times f; Eq. 2: the load
//                      factor; box width and height (raw values).
//   k_normalise        raw features -> network inputs ((x - mean) / scale).
//   k_gemm_bf16        C = A B with BF16 operands on the tensor cores (mma.sync m16n8k16,
//                      FP32 accumulation); operands are read as FP32 and rounded to BF16 when
//                      staged, so master weights and activations stay FP32.
//   k_gemm_f32         the same product in FP32 (inference and the FP32 gradient check).
//   k_guess_decode     guess at every local unknown = Coons patch of its component's side
//                      samples + bilinear interpolation of that component's 32 x 32 correction.
//   k_guess_harvest    training pair: raw features + correction (w - Coons) of the converged
//                      local state, per component, sampled bilinearly on the canonical grid.
//   k_adam             one Adam step on the FP32 master parameters.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <vector>

#include "dev_state.cuh"
#include "device.cuh"
#include "nls_internal.h"

namespace nls {

constexpr int kSide = 33, kKS = 16, kGrid = 32;
constexpr int kNF = NLS_GUESS_FEATURES, kNO = NLS_GUESS_OUTPUTS, kG2 = kGrid * kGrid;
constexpr int kNF2 = NLS_GUESS_FEATURES_DISP, kNO2 = NLS_GUESS_OUTPUTS_DISP;
static_assert(4 * kSide + kKS * kKS + 3 == kNF, "feature layout (Eq. 1)");
static_assert(kG2 == kNO, "output layout (Eq. 1)");
static_assert(2 * 4 * kSide + 3 == kNF2, "feature layout (Eq. 2)");
static_assert(2 * kG2 == kNO2, "output layout (Eq. 2)");

// ------------------------------------------------------------------------------------------
// network state
// ------------------------------------------------------------------------------------------
struct GuessNet {
  int device = 0;
  int kind = NLS_GUESS_KIND_SCALAR, nf = kNF, no = kNO;  // inputs and outputs per subdomain
  int h1 = 0, h2 = 0;
  int64_t capacity = 0, npairs = 0, nparam = 0;
  int64_t off[6] = {0};  // W1, b1, W2, b2, W3, b3
  int adam_t = 0;
  float *p = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;
  float *mean = nullptr, *scale = nullptr;
  float tscale = 1.f;
  float *dX = nullptr, *dT = nullptr;  // raw dataset
  // work buffers for batches of up to bmax rows
  int bmax = 0;
  float *X = nullptr, *T = nullptr, *Z1 = nullptr, *A1 = nullptr, *Z2 = nullptr, *A2 = nullptr, *Y = nullptr;
  float *dA = nullptr, *dZ = nullptr, *lossbuf = nullptr;
  // training: minibatch indices and partial losses of a chunk of steps, sums of squares of the targets
  int64_t chunk_indices = 0;
  int32_t* idx_chunk = nullptr;
  float* loss_chunk = nullptr;
  double* sq = nullptr;
  std::vector<void*> allocs;
  template <typename T>
  T* alloc(size_t n) {
    void* q = nullptr;
    const cudaError_t e = cudaMalloc(&q, std::max<size_t>(n, 1) * sizeof(T));
    if (e != cudaSuccess) {
      cudaGetLastError();  // reported here, not by the next launch
      throw CudaFailure(std::string("network buffers: ") + cudaGetErrorString(e));
    }
    allocs.push_back(q);
    return (T*)q;
  }
  void release(void* q) {
    const auto it = std::find(allocs.begin(), allocs.end(), q);
    if (!q || it == allocs.end()) return;
    allocs.erase(it);
    cudaFree(q);
  }
  void ensure_batch(int B);
  void ensure_chunk(int64_t indices);
};

// per-context attachment: geometry maps and buffers
struct GuessCtx {
  GuessNet* net = nullptr;
  int mode = 0;
  int nsub = 0;
  int ndof = 1;  // components per node (the network's kind)
  // per subdomain: side sample maps (node0, node1, weight), k sample elements and f element
  // (Eq. 1), box
  int32_t *side_n0 = nullptr, *side_n1 = nullptr, *kelem = nullptr, *felem = nullptr;
  float *side_w = nullptr, *box = nullptr;  // box: Lx, Ly
  // per local unknown (concatenated as the local states): (s, t) of its node in the box
  double2* st = nullptr;
  // per canonical point of every subdomain: 4 local-unknown positions (-1 = ring) and weights
  int4* cidx = nullptr;
  float2* cw = nullptr;
  // buffers
  float *raw = nullptr, *xin = nullptr, *yout = nullptr;
  double* side = nullptr;  // side samples [nsub][ndof x 132] of the last feature pass
  double* guess = nullptr; // proposed local states (total local unknowns)
  int32_t* accepted = nullptr;
  double* fcell_dev = nullptr;
  double* diag = nullptr;  // per local unknown: the Jacobi smoothing's diagonal
  int sweeps = 6;  // smoothing defaults: 6 sweeps for the scalar kind, 2 for the displacement kind
  double omega = 0.8;
  int64_t proposed_total = 0, accepted_total = 0;
  std::vector<void*> allocs;
  template <typename T>
  T* upload(Dev& D, const std::vector<T>& h) {
    void* q = nullptr;
    CK(cudaMalloc(&q, std::max<size_t>(h.size(), 1) * sizeof(T)));
    allocs.push_back(q);
    if (!h.empty()) CK(cudaMemcpyAsync(q, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice, D.s));
    return (T*)q;
  }
  template <typename T>
  T* alloc(size_t n) {
    void* q = nullptr;
    CK(cudaMalloc(&q, std::max<size_t>(n, 1) * sizeof(T)));
    allocs.push_back(q);
    return (T*)q;
  }
  ~GuessCtx() {
    for (void* q : allocs) cudaFree(q);
  }
};

namespace {

// ------------------------------------------------------------------------------------------
// splitmix64 on the host (weights and minibatch indices)
// ------------------------------------------------------------------------------------------
struct SplitMix {
  uint64_t s;
  uint64_t next() {
    s += 0x9E3779B97F4A7C15ull;
    uint64_t z = s;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
  }
  double uniform() { return (double)(next() >> 11) * (1.0 / 9007199254740992.0); }
  double normal() {
    const double u1 = std::max(uniform(), 1e-300), u2 = uniform();
    return std::sqrt(-2.0 * std::log(u1)) * std::cos(2.0 * M_PI * u2);
  }
};

// ------------------------------------------------------------------------------------------
// GEMM: C(i, j) = sum_k A(i, k) B(k, j), with what follows the product in its epilogue
// ------------------------------------------------------------------------------------------
__device__ inline float gelu_f(float z) {
  const float u = 0.7978845608028654f * (z + 0.044715f * z * z * z);
  return 0.5f * z * (1.f + tanhf(u));
}
__device__ inline float gelu_grad_f(float z) {
  const float u = 0.7978845608028654f * (z + 0.044715f * z * z * z);
  const float th = tanhf(u);
  const float du = 0.7978845608028654f * (1.f + 3.f * 0.044715f * z * z);
  return 0.5f * (1.f + th) + 0.5f * z * (1.f - th * th) * du;
}

// What a GEMM does with its sums on the way out:
//   kPlain     C = sum
//   kBiasAct   z = sum + bias (per column) into C, gelu(z) into `act` (if given)
//   kGeluBack  C = sum gelu'(z), z read from `z` (same shape)
enum Epilogue { kPlain, kBiasAct, kGeluBack };
struct GemmOut {
  float* C;
  int64_t ld;
  Epilogue mode;
  const float* bias;
  float* act;
  const float* z;
};
__device__ __forceinline__ void gemm_out(const GemmOut& o, int i, int j, float sum) {
  const int64_t e = i * o.ld + j;
  float v = 0.f + sum;
  if (o.mode == kBiasAct) v += o.bias[j];
  else if (o.mode == kGeluBack) v *= gelu_grad_f(o.z[e]);
  o.C[e] = v;
  if (o.mode == kBiasAct && o.act) o.act[e] = gelu_f(v);
}

// BF16 GEMM on the tensor cores.  The shapes are a few hundred wide (batch 64 .. 1024): bound by the
// latency of the chunks of K, so a CTA takes a 32 x 32 tile (64 to 256 of them per product) in chunks
// of 64 of K, loaded into registers one chunk ahead; AK, BK say which operand is contiguous along K
// (the loads of a warp follow the contiguous index).  Each warp owns 16 x 16 of the tile and
// accumulates K in steps of 16 in order, as the 64 x 64 kernel with chunks of 16 did (20 us per
// product; the same bits).
template <bool AK, bool BK>
__global__ void __launch_bounds__(128) k_gemm_bf16(int M, int N, int K, const float* __restrict__ A, int64_t lda,
                                                   const float* __restrict__ B, int64_t ldb, GemmOut out) {
  constexpr int KC = 64, LD = KC + 8, Q = 32 * KC / 128;
  __shared__ __nv_bfloat16 As[2][32][LD], Bs[2][32][LD];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int wm = (wid >> 1) * 16, wn = (wid & 1) * 16;
  const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  const int g = lane >> 2, t = lane & 3;
  float acc[2][4] = {};
  float ra[Q], rb[Q];
  auto at = [&](bool kfast, int q, int& r, int& k) {  // element q of this thread within a 32 x KC chunk
    const int e = tid + 128 * q;
    r = kfast ? e / KC : e % 32;
    k = kfast ? e % KC : e / 32;
  };
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      int r, k;
      at(AK, q, r, k);
      ra[q] = (i0 + r < M && k0 + k < K) ? A[AK ? (i0 + r) * lda + k0 + k : (k0 + k) * lda + i0 + r] : 0.f;
      at(BK, q, r, k);
      rb[q] = (j0 + r < N && k0 + k < K) ? B[BK ? (j0 + r) * ldb + k0 + k : (k0 + k) * ldb + j0 + r] : 0.f;
    }
  };
  auto store = [&](int s) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      int r, k;
      at(AK, q, r, k);
      As[s][r][k] = __float2bfloat16_rn(ra[q]);
      at(BK, q, r, k);
      Bs[s][r][k] = __float2bfloat16_rn(rb[q]);
    }
  };
  fetch(0);
  store(0);
  __syncthreads();
  for (int k0 = 0, s = 0; k0 < K; k0 += KC, s ^= 1) {
    const bool more = k0 + KC < K;
    if (more) fetch(k0 + KC);
    const int steps = min(KC, K - k0 + 15) / 16;
    for (int kk = 0; kk < steps; ++kk) {
      const uint32_t* ar0 = reinterpret_cast<const uint32_t*>(&As[s][wm + g][16 * kk + 2 * t]);
      const uint32_t* ar1 = reinterpret_cast<const uint32_t*>(&As[s][wm + g + 8][16 * kk + 2 * t]);
#pragma unroll
      for (int ni = 0; ni < 2; ++ni) {
        const uint32_t* br = reinterpret_cast<const uint32_t*>(&Bs[s][wn + 8 * ni + g][16 * kk + 2 * t]);
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
            "{%0,%1,%2,%3};\n"
            : "+f"(acc[ni][0]), "+f"(acc[ni][1]), "+f"(acc[ni][2]), "+f"(acc[ni][3])
            : "r"(ar0[0]), "r"(ar1[0]), "r"(ar0[4]), "r"(ar1[4]), "r"(br[0]), "r"(br[4]));
      }
    }
    if (more) store(s ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int ni = 0; ni < 2; ++ni)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int i = i0 + wm + g + (c >= 2 ? 8 : 0), j = j0 + wn + ni * 8 + 2 * t + (c & 1);
      if (i < M && j < N) gemm_out(out, i, j, acc[ni][c]);
    }
}

// FP32 GEMM (inference, the FP32 gradient check): a 16 R x 16 R tile per CTA, R x R sums per thread,
// chunks of 16 of K loaded one ahead.  Every sum runs over K in order in one accumulator, as in a
// 16 x 16 tile with one sum per thread (3.8 TFLOP/s over the three products of a batch of 1024).
template <bool AK, bool BK, int R>
__global__ void __launch_bounds__(256) k_gemm_f32(int M, int N, int K, const float* __restrict__ A, int64_t lda,
                                                  const float* __restrict__ B, int64_t ldb, GemmOut out) {
  constexpr int KC = 16, T = 16 * R, LD = T + 4;
  __shared__ __align__(16) float As[2][KC][LD], Bs[2][KC][LD];
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  const int i0 = blockIdx.y * T, j0 = blockIdx.x * T;
  float acc[R][R] = {}, ra[R], rb[R];
  auto at = [&](bool kfast, int q, int& r, int& k) {
    const int e = tid + 256 * q;
    r = kfast ? e / KC : e % T;
    k = kfast ? e % KC : e / T;
  };
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < R; ++q) {
      int r, k;
      at(AK, q, r, k);
      ra[q] = (i0 + r < M && k0 + k < K) ? A[AK ? (i0 + r) * lda + k0 + k : (k0 + k) * lda + i0 + r] : 0.f;
      at(BK, q, r, k);
      rb[q] = (j0 + r < N && k0 + k < K) ? B[BK ? (j0 + r) * ldb + k0 + k : (k0 + k) * ldb + j0 + r] : 0.f;
    }
  };
  auto store = [&](int s) {
#pragma unroll
    for (int q = 0; q < R; ++q) {
      int r, k;
      at(AK, q, r, k);
      As[s][k][r] = ra[q];
      at(BK, q, r, k);
      Bs[s][k][r] = rb[q];
    }
  };
  fetch(0);
  store(0);
  __syncthreads();
  for (int k0 = 0, s = 0; k0 < K; k0 += KC, s ^= 1) {
    const bool more = k0 + KC < K;
    if (more) fetch(k0 + KC);
#pragma unroll
    for (int kk = 0; kk < KC; ++kk) {
      float a[R], b[R];
      if constexpr (R == 4) {
        *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(&As[s][kk][ty * 4]);
        *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(&Bs[s][kk][tx * 4]);
      } else {
#pragma unroll
        for (int i = 0; i < R; ++i) a[i] = As[s][kk][ty * R + i], b[i] = Bs[s][kk][tx * R + i];
      }
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[i][j] += a[i] * b[j];
    }
    if (more) store(s ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int ii = i0 + ty * R + i, jj = j0 + tx * R + j;
      if (ii < M && jj < N) gemm_out(out, ii, jj, acc[i][j]);
    }
}

template <bool AK, bool BK>
void gemm_t(cudaStream_t s, bool bf16, int M, int N, int K, const float* A, int64_t lda, const float* B, int64_t ldb,
            const GemmOut& out) {
  // One launch has at most 65,535 tile rows: more rows (batches of over two million) go out in slabs.  (A
  // third grid dimension made 40 training steps of 256 rows 8 % slower, 6.28 -> 6.85 ms; tiles numbered along
  // one dimension 2 %.)
  auto slabs = [&](int t, auto kernel, int threads) {
    const int64_t most = (int64_t)t * 65535;
    for (int64_t m = 0; m < M; m += most) {
      const int rows = (int)std::min<int64_t>(most, M - m);
      GemmOut o = out;
      o.C += m * o.ld;
      if (o.act) o.act += m * o.ld;
      if (o.z) o.z += m * o.ld;
      kernel<<<dim3((N + t - 1) / t, (rows + t - 1) / t), threads, 0, s>>>(rows, N, K, A + (AK ? m * lda : m), lda, B, ldb, o);
      CK(cudaGetLastError());
    }
  };
  if (bf16) {
    slabs(32, k_gemm_bf16<AK, BK>, 128);
  } else {
    // 64 x 64 tiles (4 x 4 sums per thread, half the reads) once they give most SMs a CTA, else 32 x 32.  A
    // layer of 512 x 512 with 64 / 32: 28.7 / 16.4 us at 32 tiles of 64 (256 rows), 28.7 / 22.7 at 64, 28.8 / 30.8
    // at 80, 96 and 104, 28.8 / 41.0 at 128, 82 / 125 at 512 (4096 rows): level from 80 to the line.
    if (((int64_t)N + 63) / 64 * (((int64_t)M + 63) / 64) >= 100) slabs(64, k_gemm_f32<AK, BK, 4>, 256);
    else slabs(32, k_gemm_f32<AK, BK, 2>, 256);
  }
}

// C(i, j) = sum_k A(i, k) B(k, j).  ak (bk): A (B) is stored with K contiguous, row i (column j) lda
// (ldb) apart; otherwise with i (j) contiguous, the rows of K lda (ldb) apart.
void gemm(cudaStream_t s, bool bf16, int M, int N, int K, const float* A, bool ak, int64_t lda, const float* B, bool bk,
          int64_t ldb, const GemmOut& out) {
  if (ak && bk) gemm_t<true, true>(s, bf16, M, N, K, A, lda, B, ldb, out);
  else if (ak) gemm_t<true, false>(s, bf16, M, N, K, A, lda, B, ldb, out);
  else if (bk) gemm_t<false, true>(s, bf16, M, N, K, A, lda, B, ldb, out);
  else gemm_t<false, false>(s, bf16, M, N, K, A, lda, B, ldb, out);
}

// ------------------------------------------------------------------------------------------
// elementwise pieces
// ------------------------------------------------------------------------------------------
// dY = (Y - T) / B; per-block partial losses (fixed order) into part
__global__ void k_loss_grad(int64_t total, int B, const float* Y, const float* T, float* dY, float* part) {
  __shared__ float red[256];
  float acc = 0.f;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const float d = Y[e] - T[e];
    dY[e] = d / (float)B;
    acc += d * d;
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0] / (2.f * (float)B);
}

// Column sums over the batch, one thread per column, rows in order, 16 of them in flight.
__global__ void __launch_bounds__(32) k_colsum(int B, int n, const float* __restrict__ dZ, float* db) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  float acc = 0.f;
  int i = 0;
  for (; i + 16 <= B; i += 16) {
    float v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = dZ[(int64_t)(i + q) * n + j];
#pragma unroll
    for (int q = 0; q < 16; ++q) acc += v[q];
  }
  for (; i < B; ++i) acc += dZ[(int64_t)i * n + j];
  db[j] = acc;
}

__global__ void k_adam(int64_t n, float* p, const float* g, float* m, float* v, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[e];
    const float mi = b1 * m[e] + (1.f - b1) * gi;
    const float vi = b2 * v[e] + (1.f - b2) * gi * gi;
    m[e] = mi;
    v[e] = vi;
    p[e] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// minibatch: X = normalised raw features, T = raw targets / tscale
__global__ void k_gather_batch(int B, int nf, int no, const int32_t* idx, const float* dX, const float* dT,
                               const float* mean, const float* scale, float tscale, float* X, float* T) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)B * (nf + no);
       e += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(e / (nf + no)), c = (int)(e % (nf + no));
    const int64_t src = idx[r];
    if (c < nf) X[(int64_t)r * nf + c] = (dX[src * nf + c] - mean[c]) / scale[c];
    else T[(int64_t)r * no + (c - nf)] = dT[src * no + (c - nf)] / tscale;
  }
}

__global__ void k_normalise(int B, int nf, const float* raw, const float* mean, const float* scale, float* X) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)B * nf; e += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(e % nf);
    X[e] = (raw[e] - mean[c]) / scale[c];
  }
}

// per-feature mean and standard deviation over the first n pairs (fixed-order sums)
__global__ void k_feature_stats(int64_t n, int nf, const float* dX, float* mean, float* scale) {
  const int c = blockIdx.x;
  __shared__ double red[256];
  double s = 0.0;
  for (int64_t r = threadIdx.x; r < n; r += blockDim.x) s += dX[r * nf + c];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  const double mu = red[0] / (double)n;
  __syncthreads();
  double q = 0.0;
  for (int64_t r = threadIdx.x; r < n; r += blockDim.x) {
    const double d = dX[r * nf + c] - mu;
    q += d * d;
  }
  red[threadIdx.x] = q;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    mean[c] = (float)mu;
    const double sd = sqrt(red[0] / (double)n);
    scale[c] = (float)(sd > 1e-12 ? sd : 1.0);
  }
}

// Sums of squares of the targets, one per CTA (added on the host in CTA order).
constexpr int kRmsBlocks = 256;
__global__ void k_target_squares(int64_t total, const float* dT, double* out) {
  __shared__ double red[256];
  double s = 0.0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x)
    s += (double)dT[e] * dT[e];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = red[0];
}

// ------------------------------------------------------------------------------------------
// geometry kernels (one CTA per subdomain)
// ------------------------------------------------------------------------------------------
struct GeoArgs {
  const SubMeta* meta;
  const int32_t *side_n0, *side_n1, *kelem, *felem;
  const float *side_w, *box;
  const double2* st;
  const int4* cidx;
  const float2* cw;
  const double* kcoef;
  const double* fcell;
  const double* x;
  double load;
  float* raw;
  double* side;
  int ndof, nf;  // components per node, inputs per subdomain
};

__device__ inline double side_value(const double* S, int side, double u) {
  // linear interpolation among the kSide samples of one side, u in [0, 1]
  const double q = u * (kSide - 1);
  int i0 = (int)floor(q);
  i0 = max(0, min(kSide - 2, i0));
  const double w = q - i0;
  return (1.0 - w) * S[side * kSide + i0] + w * S[side * kSide + i0 + 1];
}

__device__ inline double coons_eval(const double* S, double s, double t) {
  // sides: 0 bottom (t = 0), 1 top (t = 1), 2 left (s = 0), 3 right (s = 1)
  const double P00 = S[0], P10 = S[kSide - 1], P01 = S[kSide], P11 = S[2 * kSide - 1];
  return (1 - t) * side_value(S, 0, s) + t * side_value(S, 1, s) + (1 - s) * side_value(S, 2, t) +
         s * side_value(S, 3, t) - ((1 - s) * (1 - t) * P00 + s * (1 - t) * P10 + (1 - s) * t * P01 + s * t * P11);
}

__device__ inline double corr_eval(const float* Y, double s, double t, float tscale) {
  // bilinear interpolation of the kGrid x kGrid correction at (s, t); grid points at (a + 0.5) / kGrid
  double gx = s * kGrid - 0.5, gy = t * kGrid - 0.5;
  gx = fmin(fmax(gx, 0.0), kGrid - 1.0);
  gy = fmin(fmax(gy, 0.0), kGrid - 1.0);
  int a0 = min((int)gx, kGrid - 2), b0 = min((int)gy, kGrid - 2);
  const double wa = gx - a0, wb = gy - b0;
  const double v = (1 - wa) * (1 - wb) * Y[b0 * kGrid + a0] + wa * (1 - wb) * Y[b0 * kGrid + a0 + 1] +
                   (1 - wa) * wb * Y[(b0 + 1) * kGrid + a0] + wa * wb * Y[(b0 + 1) * kGrid + a0 + 1];
  return v * tscale;
}

// Eq. 1: [side samples (132), log k (256), load f, box width, box height]; Eq. 2: [side samples of
// component 0 (132), of component 1 (132), load, box width, box height].
__global__ void k_guess_features(GeoArgs G, int nsub) {
  const int sub = blockIdx.x;
  if (sub >= nsub) return;
  constexpr int NS = 4 * kSide;
  const int nd = G.ndof;
  float* out = G.raw + (int64_t)sub * G.nf;
  double* S = G.side + (int64_t)sub * nd * NS;
  for (int e = threadIdx.x; e < nd * NS; e += blockDim.x) {
    const int c = e / NS, q = e % NS;
    const int64_t k = (int64_t)sub * NS + q;
    const double w = G.side_w[k];
    const double v = (1.0 - w) * G.x[(int64_t)G.side_n0[k] * nd + c] + w * G.x[(int64_t)G.side_n1[k] * nd + c];
    S[e] = v;
    out[e] = (float)v;
  }
  if (nd == 1) {
    for (int q = threadIdx.x; q < kKS * kKS; q += blockDim.x)
      out[NS + q] = (float)log(G.kcoef[G.kelem[(int64_t)sub * kKS * kKS + q]]);
    if (threadIdx.x == 0) {
      out[NS + kKS * kKS] = (float)(G.load * G.fcell[G.felem[sub]]);
      out[NS + kKS * kKS + 1] = G.box[2 * sub];
      out[NS + kKS * kKS + 2] = G.box[2 * sub + 1];
    }
  } else if (threadIdx.x == 0) {
    out[nd * NS] = (float)G.load;
    out[nd * NS + 1] = G.box[2 * sub];
    out[nd * NS + 2] = G.box[2 * sub + 1];
  }
}

// local unknown a is component a % ndof of its node (node-major, component-interleaved)
__global__ void k_guess_decode(GeoArgs G, int nsub, const float* Y, float tscale, double* guess) {
  const int sub = blockIdx.x;
  if (sub >= nsub) return;
  const SubMeta m = G.meta[sub];
  const int nd = G.ndof;
  const double* S = G.side + (int64_t)sub * nd * 4 * kSide;
  const float* Ys = Y + (int64_t)sub * nd * kG2;
  for (int a = threadIdx.x; a < m.n; a += blockDim.x) {
    const int c = a % nd;
    const double2 p = G.st[m.vec_off + a];
    guess[m.vec_off + a] = coons_eval(S + c * 4 * kSide, p.x, p.y) + corr_eval(Ys + c * kG2, p.x, p.y, tscale);
  }
}

// Harvest: raw features (already in G.raw) and the correction of the converged local state w
// sampled on the canonical grid.
__global__ void k_guess_harvest(GeoArgs G, int nsub, const double* w, float* dX, float* dT, int64_t slot0) {
  const int sub = blockIdx.x;
  if (sub >= nsub) return;
  const SubMeta m = G.meta[sub];
  const int nd = G.ndof;
  const double* S = G.side + (int64_t)sub * nd * 4 * kSide;
  float* X = dX + (slot0 + sub) * G.nf;
  float* T = dT + (slot0 + sub) * nd * kG2;
  for (int q = threadIdx.x; q < G.nf; q += blockDim.x) X[q] = G.raw[(int64_t)sub * G.nf + q];
  for (int e = threadIdx.x; e < nd * kG2; e += blockDim.x) {
    const int comp = e / kG2, q = e % kG2;
    const int4 id = G.cidx[(int64_t)sub * kG2 + q];
    const float2 wt = G.cw[(int64_t)sub * kG2 + q];
    const int ids[4] = {id.x, id.y, id.z, id.w};
    const double wts[4] = {(1.0 - wt.x) * (1.0 - wt.y), wt.x * (1.0 - wt.y), (1.0 - wt.x) * wt.y, wt.x * wt.y};
    double v = 0.0;
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (ids[c] >= 0) {
        const int64_t l = m.vec_off + (int64_t)ids[c] * nd + comp;
        const double2 p = G.st[l];
        v += wts[c] * (w[l] - coons_eval(S + comp * 4 * kSide, p.x, p.y));
      }
    T[e] = (float)v;
  }
}

}  // namespace

// The work buffers grow as a whole: a failed allocation leaves the network with those it had.
void GuessNet::ensure_batch(int B) {
  if (B <= bmax) return;
  const int wide = std::max({h1, h2, no});
  float** const buf[9] = {&X, &T, &Z1, &A1, &Z2, &A2, &Y, &dA, &dZ};
  const int width[9] = {nf, no, h1, h1, h2, h2, no, wide, wide};
  float* grown[9] = {};
  try {
    if (!lossbuf) lossbuf = alloc<float>(1024);
    for (int k = 0; k < 9; ++k) grown[k] = alloc<float>((size_t)B * width[k]);
  } catch (...) {
    for (float* q : grown) release(q);
    throw;
  }
  for (int k = 0; k < 9; ++k) {
    release(*buf[k]);
    *buf[k] = grown[k];
  }
  bmax = B;
}

// Training steps issued between two reads of their losses: kTrainChunk, or as many (one at least) as have
// kTrainIndices minibatch indices together (16 MB; from 16,384 rows on a step outlasts the read).
constexpr int kTrainChunk = 256;
constexpr int64_t kTrainIndices = int64_t(1) << 22;

namespace {

// forward pass of B rows of normalised inputs in net.X (or `X` if given) into net.Y
void net_forward(GuessNet& N, cudaStream_t s, int B, const float* X, bool bf16) {
  auto layer = [&](const float* in, int k, int l, int n, float* Z, float* act) {
    gemm(s, bf16, B, n, k, in, true, k, N.p + N.off[2 * l], true, k, {Z, n, kBiasAct, N.p + N.off[2 * l + 1], act, nullptr});
  };
  layer(X, N.nf, 0, N.h1, N.Z1, N.A1);
  layer(N.A1, N.h1, 1, N.h2, N.Z2, N.A2);
  layer(N.A2, N.h2, 2, N.no, N.Y, nullptr);
}

constexpr int kLossParts = 256;

// gradient (into N.g) and partial losses (into `parts`, kLossParts of them) of the batch in N.X / N.T
void net_gradient(GuessNet& N, cudaStream_t s, int B, bool bf16, float* parts) {
  net_forward(N, s, B, N.X, bf16);
  k_loss_grad<<<kLossParts, 256, 0, s>>>((int64_t)B * N.no, B, N.Y, N.T, N.dZ, parts);
  // layer l from its dZ: dW = dZ^T (inputs), db = column sums, and dZ of the layer below
  auto layer = [&](int l, const float* dZ, int n, const float* in, int k, float* below, const float* Zbelow) {
    gemm(s, bf16, n, k, B, dZ, false, n, in, false, k, {N.g + N.off[2 * l], k, kPlain, nullptr, nullptr, nullptr});
    k_colsum<<<(n + 31) / 32, 32, 0, s>>>(B, n, dZ, N.g + N.off[2 * l + 1]);
    if (below)
      gemm(s, bf16, B, k, n, dZ, true, n, N.p + N.off[2 * l], false, k, {below, k, kGeluBack, nullptr, nullptr, Zbelow});
  };
  layer(2, N.dZ, N.no, N.A2, N.h2, N.dA, N.Z2);
  layer(1, N.dA, N.h2, N.A1, N.h1, N.dZ, N.Z1);
  layer(0, N.dZ, N.h1, N.X, N.nf, nullptr, nullptr);
  CK(cudaGetLastError());
}

float loss_of(const float* parts) {
  double L = 0.0;
  for (int q = 0; q < kLossParts; ++q) L += parts[q];
  return (float)L;
}

}  // namespace

void GuessNet::ensure_chunk(int64_t indices) {
  if (!loss_chunk) loss_chunk = alloc<float>((size_t)kTrainChunk * kLossParts);
  if (indices <= chunk_indices) return;
  int32_t* const grown = alloc<int32_t>((size_t)indices);
  release(idx_chunk);
  idx_chunk = grown;
  chunk_indices = indices;
}

namespace {

// ------------------------------------------------------------------------------------------
// host geometry of the attachment (structured P1 or Q1 meshes of the unit square)
// ------------------------------------------------------------------------------------------
// Leading-term Jacobian diagonal of every local unknown: sum over the subdomain's elements of
// k_e |grad phi_a|^2 |e| (the smoothing of proposed starts divides by it times (1 + w_a^2)).
std::vector<double> jacobi_diagonal(const Context& c) {
  const LocalSet& s = c.ov;
  std::vector<double> diag(s.total_n, 0.0);
  for (int sb = 0; sb < s.count; ++sb) {
    const SubMeta& m = s.meta[sb];
    for (int e = 0; e < m.ne; ++e) {
      const int64_t ge = s.elem_gid[m.elem_off + e];
      const double* g = &c.geom[ge * c.geom_stride];
      const double ke = c.k_elem.empty() ? 1.0 : c.k_elem[ge];
      for (int a = 0; a < 3; ++a) {
        const int t = s.lconn[(m.elem_off + e) * 3 + a];
        if (t < m.n) diag[m.vec_off + t] += ke * g[6] * (g[2 * a] * g[2 * a] + g[2 * a + 1] * g[2 * a + 1]);
      }
    }
    for (int a = 0; a < m.n; ++a)
      if (!(diag[m.vec_off + a] > 0.0)) throw std::runtime_error("learned guess: zero Jacobi diagonal");
  }
  return diag;
}

// Eq. 2: diagonal of the linear-elastic Q1 stiffness (the tangent at zero displacement) at every
// local unknown, sum over elements and Gauss points of w det(J) ((lambda + 2 mu) (dN_a/dX_c)^2 +
// mu (dN_a/dX_c')^2) for component c (c' the other one).
std::vector<double> elasticity_diagonal(const Context& c) {
  const LocalSet& s = c.ov;
  double mu = 0.0, lam = 0.0;
  lame(c, mu, lam);
  std::vector<double> diag(s.total_n, 0.0);
  for (int sb = 0; sb < s.count; ++sb) {
    const SubMeta& m = s.meta[sb];
    for (int e = 0; e < m.ne; ++e) {
      const int64_t ge = s.elem_gid[m.elem_off + e];
      for (int q = 0; q < 4; ++q) {
        const double* g = &c.geom[ge * c.geom_stride + q * 10];
        for (int a = 0; a < 4; ++a) {
          const int t = s.lconn[(m.elem_off + e) * 4 + a];
          if (t >= m.nV) continue;
          const double gx = g[2 * a], gy = g[2 * a + 1];
          diag[m.vec_off + 2 * t] += g[8] * ((lam + 2.0 * mu) * gx * gx + mu * gy * gy);
          diag[m.vec_off + 2 * t + 1] += g[8] * ((lam + 2.0 * mu) * gy * gy + mu * gx * gx);
        }
      }
    }
    for (int a = 0; a < m.n; ++a)
      if (!(diag[m.vec_off + a] > 0.0)) throw std::runtime_error("learned guess: zero Jacobi diagonal");
  }
  return diag;
}

// The scalar kind needs Eq. 1 on P1 triangles, the displacement kind Eq. 2 on Q1 quadrilaterals.
bool guess_kind_matches(const Context& c, int kind) {
  if (kind == NLS_GUESS_KIND_SCALAR) return c.elem_type == NLS_P1_TRI && c.ndof == 1;
  return kind == NLS_GUESS_KIND_DISPLACEMENT && c.elem_type == NLS_Q1_QUAD && c.ndof == 2 &&
         c.law == NLS_LAW_NEOHOOKE;
}

void build_geometry(Context& c, GuessCtx& G) {
  const int nd = c.ndof;
  G.ndof = nd;
  // grid indices from coordinates
  double xmin = 1e300, xmax = -1e300, ymin = 1e300, ymax = -1e300;
  for (int64_t v = 0; v < c.n_nodes; ++v) {
    xmin = std::min(xmin, c.xy[2 * v]);
    xmax = std::max(xmax, c.xy[2 * v]);
    ymin = std::min(ymin, c.xy[2 * v + 1]);
    ymax = std::max(ymax, c.xy[2 * v + 1]);
  }
  const int64_t side = (int64_t)std::llround(std::sqrt((double)c.n_nodes));
  if (side * side != c.n_nodes) throw std::runtime_error("learned guess: mesh is not a square structured grid");
  const int nn = (int)side - 1;  // cells per side
  const double hx = (xmax - xmin) / nn, hy = (ymax - ymin) / nn;
  std::vector<int32_t> gi(c.n_nodes), gj(c.n_nodes);
  for (int64_t v = 0; v < c.n_nodes; ++v) {
    const double fx = (c.xy[2 * v] - xmin) / hx, fy = (c.xy[2 * v + 1] - ymin) / hy;
    gi[v] = (int32_t)std::llround(fx);
    gj[v] = (int32_t)std::llround(fy);
    if (std::abs(fx - gi[v]) > 1e-6 || std::abs(fy - gj[v]) > 1e-6 || gj[v] * side + gi[v] != v)
      throw std::runtime_error("learned guess: nodes are not numbered as a lexicographic structured grid");
  }
  auto node = [&](int i, int j) { return (int32_t)(j * side + i); };
  const LocalSet& s = c.ov;
  const int nsub = s.count;
  const bool scalar = nd == 1;
  std::vector<int32_t> n0((size_t)nsub * 4 * kSide), n1((size_t)nsub * 4 * kSide),
      kel(scalar ? (size_t)nsub * kKS * kKS : 0), fel(scalar ? nsub : 0);
  std::vector<float> sw((size_t)nsub * 4 * kSide), box(2 * (size_t)nsub);
  std::vector<double2> st(s.total_n);
  const std::vector<double> diag = scalar ? jacobi_diagonal(c) : elasticity_diagonal(c);
  std::vector<int4> cidx((size_t)nsub * kG2);
  std::vector<float2> cw((size_t)nsub * kG2);
  for (int sb = 0; sb < nsub; ++sb) {
    const SubMeta& m = s.meta[sb];
    int ia = INT32_MAX, ib = -1, ja = INT32_MAX, jb = -1;
    std::map<int64_t, int> local;  // node -> local unknown index
    for (int a = 0; a < m.nV; ++a) {
      const int32_t v = s.tnode_gid[m.tnode_off + a];
      ia = std::min(ia, gi[v]);
      ib = std::max(ib, gi[v]);
      ja = std::min(ja, gj[v]);
      jb = std::max(jb, gj[v]);
      local[v] = a;
    }
    // box [ia-1, ib+1] x [ja-1, jb+1] clamped to the mesh (the clamp acts only where local
    // unknowns reach a Neumann edge)
    const int i0 = std::max(ia - 1, 0), i1 = std::min(ib + 1, nn), j0 = std::max(ja - 1, 0), j1 = std::min(jb + 1, nn);
    const double Lx = (i1 - i0) * hx, Ly = (j1 - j0) * hy;
    box[2 * sb] = (float)Lx;
    box[2 * sb + 1] = (float)Ly;
    for (int q = 0; q < kSide; ++q) {
      const double u = (double)q / (kSide - 1);
      // bottom / top: along i at j0 / j1; left / right: along j at i0 / i1
      const double fi = i0 + u * (i1 - i0), fj = j0 + u * (j1 - j0);
      int ii = std::min((int)std::floor(fi), i1 - 1), jj = std::min((int)std::floor(fj), j1 - 1);
      const double wi = fi - ii, wj = fj - jj;
      const size_t base = (size_t)sb * 4 * kSide;
      n0[base + q] = node(ii, j0);
      n1[base + q] = node(ii + 1, j0);
      sw[base + q] = (float)wi;
      n0[base + kSide + q] = node(ii, j1);
      n1[base + kSide + q] = node(ii + 1, j1);
      sw[base + kSide + q] = (float)wi;
      n0[base + 2 * kSide + q] = node(i0, jj);
      n1[base + 2 * kSide + q] = node(i0, jj + 1);
      sw[base + 2 * kSide + q] = (float)wj;
      n0[base + 3 * kSide + q] = node(i1, jj);
      n1[base + 3 * kSide + q] = node(i1, jj + 1);
      sw[base + 3 * kSide + q] = (float)wj;
    }
    for (int b = 0; b < (scalar ? kKS : 0); ++b)
      for (int a = 0; a < kKS; ++a) {
        const double fx = i0 + (a + 0.5) / kKS * (i1 - i0), fy = j0 + (b + 0.5) / kKS * (j1 - j0);
        const int ci = std::min((int)fx, nn - 1), cj = std::min((int)fy, nn - 1);
        // SW-NE diagonal: the lower triangle (2c) when the point is below the diagonal
        const bool lower = (fx - ci) >= (fy - cj);
        kel[(size_t)sb * kKS * kKS + b * kKS + a] = 2 * (cj * nn + ci) + (lower ? 0 : 1);
      }
    if (scalar) {
      const int ci = std::min((i0 + i1) / 2, nn - 1), cj = std::min((j0 + j1) / 2, nn - 1);
      fel[sb] = 2 * (cj * nn + ci);
    }
    for (int a = 0; a < m.n; ++a) {
      const int32_t v = s.tnode_gid[m.tnode_off + a / nd];
      st[m.vec_off + a] = make_double2((gi[v] - i0) / (double)(i1 - i0), (gj[v] - j0) / (double)(j1 - j0));
    }
    for (int b = 0; b < kGrid; ++b)
      for (int a = 0; a < kGrid; ++a) {
        const double fx = i0 + (a + 0.5) / kGrid * (i1 - i0), fy = j0 + (b + 0.5) / kGrid * (j1 - j0);
        const int ii = std::min((int)std::floor(fx), i1 - 1), jj = std::min((int)std::floor(fy), j1 - 1);
        auto lid = [&](int i, int j) {
          auto it = local.find(node(i, j));
          return it == local.end() ? -1 : it->second;
        };
        cidx[(size_t)sb * kG2 + b * kGrid + a] = make_int4(lid(ii, jj), lid(ii + 1, jj), lid(ii, jj + 1), lid(ii + 1, jj + 1));
        cw[(size_t)sb * kG2 + b * kGrid + a] = make_float2((float)(fx - ii), (float)(fy - jj));
      }
  }
  Dev& D = *c.dev;
  G.nsub = nsub;
  G.side_n0 = G.upload(D, n0);
  G.side_n1 = G.upload(D, n1);
  G.side_w = G.upload(D, sw);
  G.kelem = G.upload(D, kel);
  G.felem = G.upload(D, fel);
  G.box = G.upload(D, box);
  G.st = G.upload(D, st);
  G.cidx = G.upload(D, cidx);
  G.cw = G.upload(D, cw);
  G.diag = G.upload(D, diag);
  G.raw = G.alloc<float>((size_t)nsub * G.net->nf);
  G.xin = G.alloc<float>((size_t)nsub * G.net->nf);
  G.side = G.alloc<double>((size_t)nsub * nd * 4 * kSide);
  G.guess = G.alloc<double>(s.total_n);
  G.accepted = G.alloc<int32_t>(nsub);
  std::vector<double> fcell(c.n_elems, 1.0);
  if (!c.f_elem.empty()) fcell = c.f_elem;
  G.fcell_dev = G.upload(D, fcell);
  CK(cudaStreamSynchronize(D.s));
}

GeoArgs geo_args(Context& c, GuessCtx& G, const double* x, double load) {
  GeoArgs a;
  std::memset(&a, 0, sizeof(a));
  Dev& D = *c.dev;
  a.meta = D.ov.meta;
  a.side_n0 = G.side_n0;
  a.side_n1 = G.side_n1;
  a.kelem = G.kelem;
  a.felem = G.felem;
  a.side_w = G.side_w;
  a.box = G.box;
  a.st = G.st;
  a.cidx = G.cidx;
  a.cw = G.cw;
  a.kcoef = D.kcoef;
  a.fcell = G.fcell_dev;
  a.x = x;
  a.load = load;
  a.raw = G.raw;
  a.side = G.side;
  a.ndof = G.ndof;
  a.nf = G.net->nf;
  return a;
}

}  // namespace

// ------------------------------------------------------------------------------------------
// hooks used by the solver
// ------------------------------------------------------------------------------------------
GuessProposal guess_propose(Context& c, const double* x, double load) {
  Dev& D = *c.dev;
  GuessCtx* G = (GuessCtx*)D.guess;
  GuessProposal out;
  if (!G || !(G->mode & NLS_GUESS_USE) || !G->net) return out;
  if ((G->mode & NLS_GUESS_FIRST_OUTER) && D.outer_k > 0) return out;
  GuessNet& N = *G->net;
  N.ensure_batch(G->nsub);
  GeoArgs a = geo_args(c, *G, x, load);
  LAUNCH(D, k_guess_features, G->nsub, 128, 0, a, G->nsub);
  LAUNCH(D, k_normalise, 1216, 256, 0, G->nsub, N.nf, G->raw, N.mean, N.scale, G->xin);
  net_forward(N, D.s, G->nsub, G->xin, false);
  D.launches += 3;
  LAUNCH(D, k_guess_decode, G->nsub, 128, 0, a, G->nsub, N.Y, N.tscale, G->guess);
  CK(cudaMemsetAsync(G->accepted, 0, sizeof(int32_t) * G->nsub, D.s));
  G->proposed_total += G->nsub;
  out.x = G->guess;
  out.accepted = G->accepted;
  out.diag = G->diag;
  out.sweeps = G->sweeps;
  out.omega = G->omega;
  return out;
}

// Smoothing parameters of the attached guess (diagonal, sweeps, omega) without a proposal.
GuessProposal guess_smoothing(Context& c) {
  GuessProposal out;
  GuessCtx* G = c.dev ? (GuessCtx*)c.dev->guess : nullptr;
  if (!G) return out;
  out.diag = G->diag;
  out.sweeps = G->sweeps;
  out.omega = G->omega;
  return out;
}

// Test hooks: the raw features at x (host) into out [nsub x nf], and the decode of given network
// outputs Y [nsub x no] (normalised units) at x into out [total local unknowns].
int guess_features(Context& c, const double* x, double load, float* out) {
  GuessCtx* G = c.dev ? (GuessCtx*)c.dev->guess : nullptr;
  if (!G) {
    c.last_error = "the learned-guess hooks need an attached network";
    return NLS_E_ARG;
  }
  Dev& D = *c.dev;
  try {
    CK(cudaMemcpyAsync(D.x, x, sizeof(double) * c.N, cudaMemcpyHostToDevice, D.s));
    GeoArgs a = geo_args(c, *G, D.x, load);
    LAUNCH(D, k_guess_features, G->nsub, 128, 0, a, G->nsub);
    CK(cudaMemcpyAsync(out, G->raw, sizeof(float) * (size_t)G->nsub * G->net->nf, cudaMemcpyDeviceToHost, D.s));
    CK(cudaStreamSynchronize(D.s));
  } catch (const std::exception& ex) {
    c.last_error = ex.what();
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

int guess_decode(Context& c, const double* x, double load, const float* Y, double* out) {
  GuessCtx* G = c.dev ? (GuessCtx*)c.dev->guess : nullptr;
  if (!G || !G->net) {
    c.last_error = "the learned-guess hooks need an attached network";
    return NLS_E_ARG;
  }
  Dev& D = *c.dev;
  GuessNet& N = *G->net;
  try {
    N.ensure_batch(G->nsub);
    CK(cudaMemcpyAsync(D.x, x, sizeof(double) * c.N, cudaMemcpyHostToDevice, D.s));
    CK(cudaMemcpyAsync(N.Y, Y, sizeof(float) * (size_t)G->nsub * N.no, cudaMemcpyHostToDevice, D.s));
    GeoArgs a = geo_args(c, *G, D.x, load);
    LAUNCH(D, k_guess_features, G->nsub, 128, 0, a, G->nsub);
    LAUNCH(D, k_guess_decode, G->nsub, 128, 0, a, G->nsub, N.Y, N.tscale, G->guess);
    CK(cudaMemcpyAsync(out, G->guess, sizeof(double) * c.ov.total_n, cudaMemcpyDeviceToHost, D.s));
    CK(cudaStreamSynchronize(D.s));
  } catch (const std::exception& ex) {
    c.last_error = ex.what();
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

int guess_set_smoothing(Context& c, int32_t sweeps, double omega) {
  GuessCtx* G = c.dev ? (GuessCtx*)c.dev->guess : nullptr;
  if (!G) {
    c.last_error = "nls_guess_set_smoothing needs an attached network";
    return NLS_E_ARG;
  }
  if (sweeps < 0 || sweeps > 64 || !(omega > 0.0 && omega <= 1.0)) {
    c.last_error = "smoothing needs sweeps in [0, 64] and omega in (0, 1]";
    return NLS_E_ARG;
  }
  G->sweeps = sweeps;
  G->omega = omega;
  return NLS_OK;
}

void guess_after_local(Context& c, const double* x, double load, bool proposed) {
  Dev& D = *c.dev;
  GuessCtx* G = (GuessCtx*)D.guess;
  if (!G) return;
  if (proposed) {
    std::vector<int32_t> acc(G->nsub);
    CK(cudaMemcpyAsync(acc.data(), G->accepted, sizeof(int32_t) * G->nsub, cudaMemcpyDeviceToHost, D.s));
    CK(cudaStreamSynchronize(D.s));
    for (int32_t v : acc) G->accepted_total += v;
  }
  if ((G->mode & NLS_GUESS_HARVEST) && G->net) {
    GuessNet& N = *G->net;
    if (N.npairs + G->nsub > N.capacity) return;  // dataset full: stop recording
    GeoArgs a = geo_args(c, *G, x, load);
    if (!proposed) LAUNCH(D, k_guess_features, G->nsub, 128, 0, a, G->nsub);
    LAUNCH(D, k_guess_harvest, G->nsub, 128, 0, a, G->nsub, D.ov.w, N.dX, N.dT, N.npairs);
    N.npairs += G->nsub;
  }
}

// New k / f on an attached context: the per-element f copy and the Jacobi diagonal follow.
void guess_coefficients_changed(Context& c) {
  GuessCtx* G = (c.dev && c.dev->guess) ? (GuessCtx*)c.dev->guess : nullptr;
  if (!G) return;
  Dev& D = *c.dev;
  const std::vector<double> diag = jacobi_diagonal(c);
  CK(cudaMemcpyAsync(G->diag, diag.data(), sizeof(double) * diag.size(), cudaMemcpyHostToDevice, D.s));
  std::vector<double> fcell(c.n_elems, 1.0);
  if (!c.f_elem.empty()) fcell = c.f_elem;
  CK(cudaMemcpyAsync(G->fcell_dev, fcell.data(), sizeof(double) * fcell.size(), cudaMemcpyHostToDevice, D.s));
  CK(cudaStreamSynchronize(D.s));
}

void guess_free(Context& c) {
  if (c.dev && c.dev->guess) {
    delete (GuessCtx*)c.dev->guess;
    c.dev->guess = nullptr;
  }
}

}  // namespace nls

// ------------------------------------------------------------------------------------------
// C ABI
// ------------------------------------------------------------------------------------------
using nls::GuessNet;

struct nls_guess_net {
  GuessNet n;
};

extern "C" {

int nls_guess_create(nls_guess_net** out, int device, int32_t h1, int32_t h2, uint64_t seed, int64_t capacity) {
  return nls_guess_create_kind(out, device, NLS_GUESS_KIND_SCALAR, h1, h2, seed, capacity);
}

int nls_guess_create_kind(nls_guess_net** out, int device, int32_t kind, int32_t h1, int32_t h2, uint64_t seed,
                          int64_t capacity) {
  if (!out || h1 <= 0 || h2 <= 0 || h1 % 16 || h2 % 16 || capacity < 0) return NLS_E_ARG;
  if (kind != NLS_GUESS_KIND_SCALAR && kind != NLS_GUESS_KIND_DISPLACEMENT) return NLS_E_ARG;
  nls_guess_net* w = new (std::nothrow) nls_guess_net();
  if (!w) return NLS_E_NOMEM;
  GuessNet& N = w->n;
  try {
    CK(cudaSetDevice(device));
    N.device = device;
    N.kind = kind;
    N.nf = kind == NLS_GUESS_KIND_SCALAR ? nls::kNF : nls::kNF2;
    N.no = kind == NLS_GUESS_KIND_SCALAR ? nls::kNO : nls::kNO2;
    N.h1 = h1;
    N.h2 = h2;
    N.capacity = capacity;
    const int64_t sz[6] = {(int64_t)h1 * N.nf, h1, (int64_t)h2 * h1, h2, (int64_t)N.no * h2, N.no};
    int64_t o = 0;
    for (int k = 0; k < 6; ++k) {
      N.off[k] = o;
      o += sz[k];
    }
    N.nparam = o;
    std::vector<float> p(o, 0.f);
    nls::SplitMix rng{seed};
    const int fan_in[3] = {N.nf, h1, h2};
    for (int l = 0; l < 3; ++l) {
      const double sd = 1.0 / std::sqrt((double)fan_in[l]);
      for (int64_t e = 0; e < sz[2 * l]; ++e) p[N.off[2 * l] + e] = (float)(sd * rng.normal());
    }
    N.p = N.alloc<float>(o);
    N.m = N.alloc<float>(o);
    N.v = N.alloc<float>(o);
    N.g = N.alloc<float>(o);
    CK(cudaMemcpy(N.p, p.data(), o * sizeof(float), cudaMemcpyHostToDevice));
    CK(cudaMemset(N.m, 0, o * sizeof(float)));
    CK(cudaMemset(N.v, 0, o * sizeof(float)));
    N.mean = N.alloc<float>(N.nf);
    N.scale = N.alloc<float>(N.nf);
    std::vector<float> zero(N.nf, 0.f), one(N.nf, 1.f);
    CK(cudaMemcpy(N.mean, zero.data(), N.nf * sizeof(float), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(N.scale, one.data(), N.nf * sizeof(float), cudaMemcpyHostToDevice));
    N.dX = N.alloc<float>((size_t)capacity * N.nf);
    N.dT = N.alloc<float>((size_t)capacity * N.no);
  } catch (const std::exception&) {
    for (void* q : N.allocs) cudaFree(q);
    delete w;
    return NLS_E_CUDA;
  }
  *out = w;
  return NLS_OK;
}

void nls_guess_destroy(nls_guess_net* w) {
  if (!w) return;
  cudaSetDevice(w->n.device);
  cudaDeviceSynchronize();
  for (void* q : w->n.allocs) cudaFree(q);
  delete w;
}

int nls_guess_dims(const nls_guess_net* w, int32_t* kind, int32_t* n_in, int32_t* n_out) {
  if (!w) return NLS_E_ARG;
  if (kind) *kind = w->n.kind;
  if (n_in) *n_in = w->n.nf;
  if (n_out) *n_out = w->n.no;
  return NLS_OK;
}

int nls_guess_pairs(const nls_guess_net* w, int64_t* n) {
  if (!w || !n) return NLS_E_ARG;
  *n = w->n.npairs;
  return NLS_OK;
}

int nls_guess_get_params(const nls_guess_net* w, float* params, int64_t* count) {
  if (!w || !count) return NLS_E_ARG;
  *count = w->n.nparam;
  if (!params) return NLS_OK;
  if (cudaSetDevice(w->n.device) != cudaSuccess) return NLS_E_CUDA;
  return cudaMemcpy(params, w->n.p, w->n.nparam * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess ? NLS_OK
                                                                                                        : NLS_E_CUDA;
}

int nls_guess_set_params(nls_guess_net* w, const float* params, int64_t count) {
  if (!w || !params || count != w->n.nparam) return NLS_E_ARG;
  GuessNet& N = w->n;
  if (cudaSetDevice(N.device) != cudaSuccess) return NLS_E_CUDA;
  if (cudaMemcpy(N.p, params, count * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) return NLS_E_CUDA;
  cudaMemset(N.m, 0, count * sizeof(float));
  cudaMemset(N.v, 0, count * sizeof(float));
  N.adam_t = 0;
  return cudaDeviceSynchronize() == cudaSuccess ? NLS_OK : NLS_E_CUDA;
}

int nls_guess_get_normalisation(const nls_guess_net* w, float* mean, float* scale, float* tscale) {
  if (!w) return NLS_E_ARG;
  const GuessNet& N = w->n;
  if (cudaSetDevice(N.device) != cudaSuccess) return NLS_E_CUDA;
  if (mean) cudaMemcpy(mean, N.mean, N.nf * sizeof(float), cudaMemcpyDeviceToHost);
  if (scale) cudaMemcpy(scale, N.scale, N.nf * sizeof(float), cudaMemcpyDeviceToHost);
  if (tscale) *tscale = N.tscale;
  return cudaDeviceSynchronize() == cudaSuccess ? NLS_OK : NLS_E_CUDA;
}

int nls_guess_set_normalisation(nls_guess_net* w, const float* mean, const float* scale, float tscale) {
  if (!w || !mean || !scale || !(tscale > 0.f)) return NLS_E_ARG;
  GuessNet& N = w->n;
  if (cudaSetDevice(N.device) != cudaSuccess) return NLS_E_CUDA;
  cudaMemcpy(N.mean, mean, N.nf * sizeof(float), cudaMemcpyHostToDevice);
  cudaMemcpy(N.scale, scale, N.nf * sizeof(float), cudaMemcpyHostToDevice);
  N.tscale = tscale;
  return cudaDeviceSynchronize() == cudaSuccess ? NLS_OK : NLS_E_CUDA;
}

int nls_guess_gradient(nls_guess_net* w, int32_t B, const float* X, const float* T, int32_t precision, float* grad,
                       float* loss) {
  if (!w || B <= 0 || !X || !T || !grad) return NLS_E_ARG;
  GuessNet& N = w->n;
  try {
    CK(cudaSetDevice(N.device));
    N.ensure_batch(B);
    CK(cudaMemcpy(N.X, X, (size_t)B * N.nf * sizeof(float), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(N.T, T, (size_t)B * N.no * sizeof(float), cudaMemcpyHostToDevice));
    nls::net_gradient(N, 0, B, precision == 1, N.lossbuf);
    CK(cudaMemcpy(grad, N.g, N.nparam * sizeof(float), cudaMemcpyDeviceToHost));
    float parts[nls::kLossParts];
    CK(cudaMemcpy(parts, N.lossbuf, sizeof(parts), cudaMemcpyDeviceToHost));
    if (loss) *loss = nls::loss_of(parts);
  } catch (const std::exception&) {
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

int nls_guess_forward(nls_guess_net* w, int32_t B, const float* X, float* Y) {
  if (!w || B <= 0 || !X || !Y) return NLS_E_ARG;
  GuessNet& N = w->n;
  try {
    CK(cudaSetDevice(N.device));
    N.ensure_batch(B);
    CK(cudaMemcpy(N.X, X, (size_t)B * N.nf * sizeof(float), cudaMemcpyHostToDevice));
    nls::net_forward(N, 0, B, N.X, false);
    CK(cudaMemcpy(Y, N.Y, (size_t)B * N.no * sizeof(float), cudaMemcpyDeviceToHost));
  } catch (const std::exception&) {
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

int nls_guess_train(nls_guess_net* w, int32_t steps, int32_t batch, double lr, uint64_t seed, float* loss_out) {
  if (!w || steps < 0 || batch <= 0) return NLS_E_ARG;
  GuessNet& N = w->n;
  if (N.npairs <= 0) return NLS_E_ARG;
  try {
    CK(cudaSetDevice(N.device));
    N.ensure_batch(batch);
    // normalisation from the harvested pairs (inputs per feature, targets by their rms)
    nls::k_feature_stats<<<N.nf, 256>>>(N.npairs, N.nf, N.dX, N.mean, N.scale);
    if (!N.sq) N.sq = N.alloc<double>(nls::kRmsBlocks);
    nls::k_target_squares<<<nls::kRmsBlocks, 256>>>(N.npairs * N.no, N.dT, N.sq);
    std::vector<double> sq(nls::kRmsBlocks);
    CK(cudaMemcpy(sq.data(), N.sq, sizeof(double) * sq.size(), cudaMemcpyDeviceToHost));
    double sum = 0.0;
    for (double v : sq) sum += v;
    const double hr = std::sqrt(sum / (double)std::max<int64_t>(N.npairs * N.no, 1));
    N.tscale = (float)(hr > 1e-30 ? hr : 1.0);
    // The steps go out without waiting for one another: the minibatches of a chunk of steps are drawn and
    // copied ahead, their partial losses stay on the device until the chunk is done.
    nls::SplitMix rng{seed};
    const int chunk = (int)std::max<int64_t>(
        1, std::min<int64_t>(nls::kTrainIndices / batch, std::min(nls::kTrainChunk, (int)steps)));
    N.ensure_chunk((int64_t)chunk * batch);
    std::vector<int32_t> idx;
    std::vector<float> parts;
    for (int s0 = 0; s0 < steps; s0 += chunk) {
      const int ns = std::min(chunk, steps - s0);
      idx.resize((size_t)ns * batch);
      for (auto& r : idx) r = (int32_t)(rng.next() % (uint64_t)N.npairs);
      CK(cudaMemcpy(N.idx_chunk, idx.data(), idx.size() * sizeof(int32_t), cudaMemcpyHostToDevice));
      for (int st = 0; st < ns; ++st) {
        nls::k_gather_batch<<<1216, 256>>>(batch, N.nf, N.no, N.idx_chunk + (size_t)st * batch, N.dX, N.dT, N.mean, N.scale,
                                           N.tscale, N.X, N.T);
        nls::net_gradient(N, 0, batch, true, N.loss_chunk + (size_t)st * nls::kLossParts);
        N.adam_t += 1;
        const float b1 = 0.9f, b2 = 0.999f;
        nls::k_adam<<<1216, 256>>>(N.nparam, N.p, N.g, N.m, N.v, (float)lr, b1, b2, 1e-8f,
                                   1.f - std::pow(b1, (float)N.adam_t), 1.f - std::pow(b2, (float)N.adam_t));
        CK(cudaGetLastError());
      }
      parts.resize((size_t)ns * nls::kLossParts);
      CK(cudaMemcpy(parts.data(), N.loss_chunk, parts.size() * sizeof(float), cudaMemcpyDeviceToHost));
      if (loss_out)
        for (int st = 0; st < ns; ++st) loss_out[s0 + st] = nls::loss_of(&parts[(size_t)st * nls::kLossParts]);
    }
    CK(cudaDeviceSynchronize());
  } catch (const std::exception&) {
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

int nls_guess_attach(nls_ctx* ctx, nls_guess_net* w, int32_t mode);  // defined in api.cpp (needs the context)

}  // extern "C"

namespace nls {

int guess_attach(Context& c, nls_guess_net* w, int32_t mode) {
  if (!c.is_setup || !c.dev) {
    c.last_error = "nls_guess_attach needs a context after nls_setup";
    return NLS_E_ARG;
  }
  try {
    CK(cudaSetDevice(c.device));
    guess_free(c);
    if (!w || mode == 0) return NLS_OK;
    if (w->n.device != c.device) {
      c.last_error = "network and context live on different devices";
      return NLS_E_ARG;
    }
    if (!guess_kind_matches(c, w->n.kind)) {
      c.last_error = "the network's kind does not match the problem (scalar: Eq. 1 on P1 triangles; "
                     "displacement: Eq. 2 on Q1 quadrilaterals)";
      return NLS_E_ARG;
    }
    GuessCtx* G = new GuessCtx();
    G->net = &w->n;
    G->mode = mode;
    if (w->n.kind == NLS_GUESS_KIND_DISPLACEMENT) G->sweeps = 2;
    build_geometry(c, *G);
    c.dev->guess = G;
  } catch (const std::exception& ex) {
    c.last_error = ex.what();
    guess_free(c);
    return NLS_E_UNSUPPORTED;
  }
  return NLS_OK;
}

int guess_counts(Context& c, int64_t* proposed, int64_t* accepted) {
  GuessCtx* G = c.dev ? (GuessCtx*)c.dev->guess : nullptr;
  if (proposed) *proposed = G ? G->proposed_total : 0;
  if (accepted) *accepted = G ? G->accepted_total : 0;
  if (G) G->proposed_total = G->accepted_total = 0;
  return NLS_OK;
}

}  // namespace nls
