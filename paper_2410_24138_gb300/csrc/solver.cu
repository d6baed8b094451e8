// Device solver of the two-level nonlinear Schwarz method (sm_103a).
//
// Kernels:
//   k_local_newton   one persistent launch per F_x evaluation: every overlapping subdomain
//                    (longest first, pulled from a device work counter) runs its local
//                    Newton loop for Eq. 4 -- colour-ordered element assembly of the FP64
//                    residual and of the local Jacobian (rows in slices of 32), tiled band LU
//                    in FP32 or FP64, triangular solves with FP64 iterative refinement, Armijo
//                    line search -- and refactors the Jacobian at the converged state for the
//                    exact tangent (Eq. 6 / Eq. 12).  It writes P~_i T_i straight into F_x.
//   k_local_apply    one CTA per subdomain: sum_i P~_i (R_i DF(v_i) P_i)^-1 R_i DF(v_i) y.
//   k_harmonic       energy-minimising extension of the RGDSW interface values (setup).
//   k_galerkin       per non-overlapping subdomain: Phi_j^T K^(j)(x) Phi_j (coarse matrix).
//   k_local_factor   the refactorisation at the converged states, where it is a launch of its own.
//   k_coarse_*       band LU / solve of A_0 = P_0^T DF P_0 in one CTA (Eq. 9), its explicit inverse;
//                    k_dense_gemv_t applies that.
//   k_elem_residual, k_node_residual   global residual F(u): element contributions, then fixed-order
//                    sums per node.
//   k_global_jacobian  colour-ordered global Jacobian DF(u) (Eq. 3).
//   k_dots, k_gmres_*  GMRES vector kernels with fixed-order (deterministic) reductions.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <numeric>
#include <stdexcept>
#include <string>
#include <type_traits>
#include <mutex>
#include <vector>

#include "dev_state.cuh"
#include "device.cuh"
#include "nls_internal.h"

namespace nls {

// coarse_tlu.cu
void tlu_prepare(Context& c, bool f32);
void tlu_factor(Context& c);
void tlu_free(Context& c);
bool tlu_solve(Context& c, const double* rhs, double* z, int accumulate, const int* skip, int* reset);
void tlu_check_solves(Context& c);

namespace {



constexpr int kVecBlocks = 1216;  // 8 per SM on 152 SMs
constexpr int kMaxGmresVecs = 128;


// ------------------------------------------------------------------------------------------
// argument blocks
// ------------------------------------------------------------------------------------------
struct LocalArgs {
  const SubMeta* meta;
  const int32_t *tnode_gid, *elem_gid, *lconn, *color_ptr, *rowptr, *colidx, *epos;
  const uint8_t* owned;
  double* csr;
  void* factor;
  void* dinv;  // packed triangular-solve operands (diagonal-block inverses + couplings)
  double* wbuf;
  double* work;        // two per-subdomain FP64 vectors (vec_off), `work_stride` apart
  int64_t work_stride;
  int32_t *its, *status;
  int32_t* chord;  // per subdomain: steps of the last launch taken with the stored factors
  int reuse;       // 1: a subdomain whose previous status is OK may start with chord steps
  const int32_t* order;
  int32_t* queue;
  const double *geom, *kcoef, *fext;
  dev::NHLaw nh;  // Eq. 2
  double load;
  int ndof, nen, count, max_n, max_nt, max_b;
  double rtol, atol, armijo, ir_rtol;
  int maxit, ls_trials, ir_max;
  int l2_dist;            // L2 prefetch distance of the triangular solves (blocks; 0 = off)
  int gal_rows;           // coarse blocks: rows of Phi and K Phi in shared memory
  int ring;               // tangent application: stages of the operand ring (0: operands in registers)
  int* err;               // host-mapped: set when a bounded wait gave up
  const double* x;        // evaluation point (global)
  double* out;            // F_x: owned entries receive x - w
  const double* guess;    // optional start states (concatenated local vectors)
  const double* guess_diag;  // Jacobi diagonal (leading term) of the smoothing of the start
  int guess_sweeps;
  double guess_omega;
  int want_tangent;
  int split_factor;           // 1: the tangent's band LU and packing run in k_local_factor
  int32_t* accepted;          // per subdomain: 1 where the proposed start was taken
  unsigned long long* phase;  // optional per-phase clock counters (profiling), see kPhaseNames
  // tangent application
  const double* v;
  const double* add;
  // coarse (harmonic extension / Galerkin)
  const double* phi;
  const int64_t* phi_off;
  const int32_t* cj_ptr;
  double* Y;
  double* blk;
  const int64_t* blk_off;
};

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// shared-memory plan (bytes) of the local kernels
struct SmemPlan {
  size_t xt, r, rt, s, red, yv, win, rp, flag, total;
};

// Shared memory of the batched local kernels.  Only what the inner loops hit per entry stays in
// shared memory -- the table state (gathered by every element), the residual being assembled,
// the band-LU window and the solve vector (which lives in the window once the factors are
// packed); the current residual, the Newton step and the refinement residual are per-subdomain
// vectors in global memory (read and written O(n) times per phase, coalesced).
struct LocalPlan {
  size_t xt, racc, red, win, flag, total;
};

// Shared memory a CTA can opt in to (227 KB), less one unit of its alignment.
constexpr size_t kSmemFull = 227 * 1024 - 128;

// Shared memory of the harmonic extension (k_harmonic): the table state, the solve vector and
// the window of dev::band_lu ((b + 2) rows of 2b + 1 entries, reciprocal pivots, flag), FP64.
__host__ __device__ inline SmemPlan harmonic_plan(int max_n, int max_nt, int max_b) {
  SmemPlan p;
  size_t o = 0;
  p.xt = o; o += align_up(sizeof(double) * max_nt, 16);
  p.r = p.rt = p.s = p.red = 0;  // unused
  p.yv = o; o += align_up(sizeof(double) * max_n, 16);
  p.win = o; o += align_up(sizeof(double) * (size_t)(max_b + 2) * (2 * max_b + 1), 16);
  p.rp = o; o += align_up(sizeof(double) * (max_b + 2), 16);
  p.flag = o; o += 16;
  p.total = o;
  return p;
}

template <typename FT>
__host__ __device__ inline LocalPlan newton_plan(int max_n, int max_nt, int max_b) {
  LocalPlan p;
  const size_t inv = 4 * (size_t)dev::SolveBlock<FT>::BS * (dev::SolveBlock<FT>::BS + 1);
  size_t o = 0;
  p.xt = o; o += sizeof(double) * max_nt;
  p.racc = o; o += sizeof(double) * max_n;
  p.red = o; o += sizeof(double) * 40;
  // the size the limit on the subdomains is stated for: a window of (b + 10) rows of the band
  size_t lim = (size_t)dev::band_limit_rows(max_b) * dev::band_limit_stride(max_b);
  lim = lim > inv ? lim : inv;
  lim = lim > (size_t)max_n ? lim : (size_t)max_n;
  lim = o + align_up(sizeof(FT) * lim, 16) + align_up(sizeof(FT) * dev::band_limit_rows(max_b), 16) + 16;
  // the tiled window, with room for the next panel's tiles where that fits
  o = align_up(o, 16);
  p.win = o;
  size_t w = dev::band_lu_window<FT>(max_b, 0);
  w = w > inv ? w : inv;
  w = w > (size_t)max_n ? w : (size_t)max_n;
  const size_t full = dev::band_lu_window<FT>(max_b, 1);
  if (full > w && o + sizeof(FT) * full + 16 <= kSmemFull) w = full;
  o += align_up(sizeof(FT) * w, 16);
  p.flag = o; o += 16;
  p.total = o > lim ? o : lim;
  return p;
}

// Tangent application: the table vector (later the refined solution), the reductions, the solve
// vector and `stages` stages of the ring.
template <typename FT>
__host__ __device__ inline LocalPlan apply_plan(int max_n, int max_nt, int max_b, int stages) {
  LocalPlan p;
  size_t o = 0;
  p.xt = o; o += sizeof(double) * max_nt;
  p.racc = 0;
  p.red = o; o += sizeof(double) * 40;
  o = align_up(o, 16);
  p.win = o; o += sizeof(FT) * align_up(max_n, dev::SolveBlock<FT>::BS);
  if (stages) o = align_up(o, 128);  // the bulk copies write whole 128-byte lines
  p.flag = o;
  if (stages) o += dev::kRingHead + stages * dev::ring_stage_bytes<FT>(max_b);
  p.total = o;
  return p;
}

// ------------------------------------------------------------------------------------------
// local assembly (colour-ordered, deterministic)
// ------------------------------------------------------------------------------------------
template <int LAW>
__device__ bool local_residual(const LocalArgs& A, const SubMeta& m, const double* xt, double* r) {
  const int nd = A.ndof, nen = A.nen;
  for (int a = threadIdx.x; a < m.n; a += blockDim.x) {
    const int64_t g = (int64_t)A.tnode_gid[m.tnode_off + a / nd] * nd + a % nd;
    r[a] = -A.load * A.fext[g];
  }
  __syncthreads();
  bool ok = true;
  const int32_t* cp = A.color_ptr + m.color_off;
  for (int c = 0; c < m.ncolor; ++c) {
    for (int e = cp[c] + threadIdx.x; e < cp[c + 1]; e += blockDim.x) {
      const int64_t le = m.elem_off + e;
      const int32_t gid = A.elem_gid[le];
      const int32_t* lc = A.lconn + le * nen;
      if (LAW == NLS_LAW_DIFFUSION) {
        const double* geo = A.geom + (int64_t)gid * 8;
        const dev::P1State st = dev::p1_state(geo, A.kcoef[gid], xt[lc[0]], xt[lc[1]], xt[lc[2]]);
        double re[3];
        dev::p1_residual(geo, st, re);
#pragma unroll
        for (int a = 0; a < 3; ++a)
          if (lc[a] < m.nV) r[lc[a]] += re[a];
      } else {
        const double* geo = A.geom + (int64_t)gid * 40;
        double ue[8], re[8];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          ue[2 * a] = xt[2 * lc[a]];
          ue[2 * a + 1] = xt[2 * lc[a] + 1];
        }
        bool eok = true;
        dev::nh_residual(geo, ue, A.nh, re, eok);
        ok = ok && eok;
#pragma unroll
        for (int a = 0; a < 4; ++a)
          if (lc[a] < m.nV) {
            r[2 * lc[a]] += re[2 * a];
            r[2 * lc[a] + 1] += re[2 * a + 1];
          }
      }
    }
    __syncthreads();
  }
  return __syncthreads_and(ok ? 1 : 0) != 0;
}

// Local Jacobian into the CSR block of the subdomain (rows per m.nrows) and, when `band` is
// given, also into the band rows of the local matrix (row-major, 2 b + 1 per row, local
// unknowns only) that the in-place band LU then factors.  Element tangents are formed in FP64
// for both forms: the CSR block, against which the FP32 factors are refined, is the exact
// Jacobian; only the band copy that is factored is rounded to the factors' precision.
template <int LAW, typename FT = double>
__device__ void local_jacobian(const LocalArgs& A, const SubMeta& m, const double* xt, double* csr,
                               FT* band = nullptr) {
  const int nen = A.nen, nd = A.ndof, ned = nen * nd, ned2 = ned * ned;
  const int W = 2 * m.b + 1, n = m.n;
  for (int64_t k = threadIdx.x; k < m.nnz; k += blockDim.x) csr[k] = 0.0;
  if (band)
    for (int64_t k = threadIdx.x; k < (int64_t)n * W; k += blockDim.x) band[k] = (FT)0;
  __syncthreads();
  const int32_t* cp = A.color_ptr + m.color_off;
  for (int c = 0; c < m.ncolor; ++c) {
    for (int e = cp[c] + threadIdx.x; e < cp[c + 1]; e += blockDim.x) {
      const int64_t le = m.elem_off + e;
      const int32_t gid = A.elem_gid[le];
      const int32_t* lc = A.lconn + le * nen;
      const int32_t* ep = A.epos + m.epos_off + (int64_t)e * ned2;
      if (LAW == NLS_LAW_DIFFUSION) {
        const double* geo = A.geom + (int64_t)gid * 8;
        const dev::P1State st = dev::p1_state(geo, A.kcoef[gid], xt[lc[0]], xt[lc[1]], xt[lc[2]]);
        double K[9];
        dev::p1_jacobian<double>(geo, st, K);
        // the nine (row, col) targets of one element are distinct: issue every load before any
        // store so that one memory latency is paid per element, not one per entry
        double oc[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) oc[q] = (ep[q] >= 0) ? csr[ep[q]] : 0.0;
#pragma unroll
        for (int q = 0; q < 9; ++q)
          if (ep[q] >= 0) csr[ep[q]] = oc[q] + K[q];
        if (band) {
          FT ob[9];
          int64_t bp[9];
#pragma unroll
          for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
              const bool in = lc[a] < n && lc[b] < n;
              bp[a * 3 + b] = in ? (int64_t)lc[a] * W + (lc[b] - lc[a] + m.b) : -1;
              ob[a * 3 + b] = in ? band[bp[a * 3 + b]] : (FT)0;
            }
#pragma unroll
          for (int q = 0; q < 9; ++q)
            if (bp[q] >= 0) band[bp[q]] = ob[q] + (FT)K[q];
        }
      } else {
        const double* geo = A.geom + (int64_t)gid * 40;
        double ue[8];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          ue[2 * a] = xt[2 * lc[a]];
          ue[2 * a + 1] = xt[2 * lc[a] + 1];
        }
        dev::NHTangent K;
        dev::nh_tangent(geo, ue, A.nh, K);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const int32_t* epa = ep + 16 * a;  // rows (a, 0) and (a, 1): 16 consecutive targets
          double oc[16];
#pragma unroll
          for (int q = 0; q < 16; ++q) oc[q] = (epa[q] >= 0) ? csr[epa[q]] : 0.0;
#pragma unroll
          for (int q = 0; q < 16; ++q)
            if (epa[q] >= 0) csr[epa[q]] = oc[q] + K(a, q >> 3, (q & 7) >> 1, q & 1);
          if (band && lc[a] < m.nV) {
#pragma unroll
            for (int b = 0; b < 4; ++b)
              if (lc[b] < m.nV) {
#pragma unroll
                for (int da = 0; da < 2; ++da)
#pragma unroll
                  for (int db = 0; db < 2; ++db) {
                    const int row = 2 * lc[a] + da, col = 2 * lc[b] + db;
                    band[(int64_t)row * W + (col - row + m.b)] += (FT)K(a, da, b, db);
                  }
              }
          }
        }
      }
    }
    __syncthreads();
  }
}

// f(value, column) over the entries of local row a, in ascending column order
template <typename F>
__device__ __forceinline__ void for_row(const LocalArgs& A, const SubMeta& m, int a, F&& f) {
  const int q = m.slice == 32 ? a >> 5 : a, h = m.slice == 32 ? min(32, m.n - (a & ~31)) : 1;
  const int2 bw = *(const int2*)(A.rowptr + m.rowptr_off + 2 * q);
  const int64_t first = m.nnz_off + bw.x + (m.slice == 32 ? a & 31 : 0);
  const double* v = A.csr + first;
  const int32_t* c = A.colidx + first;
  int k = 0;
  for (; k + 6 <= bw.y; k += 6) {  // six entries in flight
    double val[6];
    int32_t col[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) val[i] = v[(k + i) * h], col[i] = c[(k + i) * h];
#pragma unroll
    for (int i = 0; i < 6; ++i) f(val[i], col[i]);
  }
  for (; k < bw.y; ++k) f(v[k * h], c[k * h]);
}

// y = (packed operands)^-1 y through the ring where it has two stages (none without unknowns) and the CTA
// the threads, else with the operands in registers.  Returns false if a bounded wait gave up.
struct Ring {
  unsigned char* mem;
  int stages;
};
template <typename FT, bool PF>
__device__ bool triangular_solves(const LocalArgs& A, const SubMeta& m, const FT* Dv, FT* yv, const Ring& ring) {
  if (ring.stages >= 2 && (int)blockDim.x >= dev::ring_threads<FT>(m.b))
    return dev::band_solve_ring<FT>(m.n, m.b, Dv, yv, ring.mem, ring.stages);
  dev::band_solve_packed<FT, PF>(m.n, m.b, Dv, yv, A.l2_dist);
  return true;
}

// s = J^-1 rhs with the band factors, then FP64 iterative refinement against the local matrix
// (columns < n) when the factors are FP32.  s and yv are in shared memory (s may be rhs's copy).
// Returns false if a bounded wait gave up.
template <typename FT, bool PF>
__device__ __forceinline__ bool local_solve(const LocalArgs& A, const SubMeta& m, const FT* Dv, const double* rhs,
                                            double rhs_norm, double* s, FT* yv, double* red, const Ring& ring) {
  const int n = m.n;
  for (int a = threadIdx.x; a < n; a += blockDim.x) yv[a] = (FT)rhs[a];
  __syncthreads();
  for (int sw = 0;; ++sw) {
    if (!triangular_solves<FT, PF>(A, m, Dv, yv, ring)) return false;
    for (int a = threadIdx.x; a < n; a += blockDim.x) s[a] = (sw ? s[a] : 0.0) + (double)yv[a];
    __syncthreads();
    if (sizeof(FT) == 8 || sw >= A.ir_max) return true;
    double loc = 0.0;
    for (int a = threadIdx.x; a < n; a += blockDim.x) {
      double acc = rhs[a];
      for_row(A, m, a, [&](double v, int32_t col) {
        if (col < n) acc -= v * s[col];
      });
      yv[a] = (FT)acc;
      loc += acc * acc;
    }
    const double rn = sqrt(dev::block_sum(loc, red));
    if (!(rn > A.ir_rtol * rhs_norm)) return true;
  }
}

// Damped Jacobi sweeps on a proposed local start (in xt's local unknowns): they remove the
// pointwise part of the proposal's error, w <- w - omega r(w) / (d (1 + w^2)) on all entries at
// once, d the diagonal of the Jacobian's leading term.  Leaves the residual of the result in racc
// and returns false if an evaluation was not finite.
template <int LAW>
__device__ bool smooth_proposal(const LocalArgs& A, const SubMeta& m, double* xt, double* racc) {
  bool okg = local_residual<LAW>(A, m, xt, racc);
  for (int sw = 0; sw < A.guess_sweeps && okg; ++sw) {
    for (int a = threadIdx.x; a < m.n; a += blockDim.x) {
      const double q = (LAW == NLS_LAW_DIFFUSION) ? 1.0 + xt[a] * xt[a] : 1.0;
      xt[a] -= A.guess_omega * racc[a] / (A.guess_diag[m.vec_off + a] * q);
    }
    __syncthreads();
    okg = local_residual<LAW>(A, m, xt, racc);
  }
  return okg;
}

// Test hook: the smoothing of given starts (A.guess, concatenated local vectors) at the point A.x,
// one CTA per subdomain, into A.out (concatenated local vectors).
template <int LAW>
__global__ void __launch_bounds__(256) k_guess_smooth(LocalArgs A) {
  extern __shared__ __align__(128) unsigned char smem[];
  double* xt = (double*)smem;
  double* racc = xt + A.max_nt;
  const int sub = blockIdx.x, nd = A.ndof;
  const SubMeta m = A.meta[sub];
  for (int t = threadIdx.x; t < m.nt; t += blockDim.x)
    xt[t] = A.x[(int64_t)A.tnode_gid[m.tnode_off + t / nd] * nd + t % nd];
  __syncthreads();
  for (int a = threadIdx.x; a < m.n; a += blockDim.x) xt[a] = A.guess[m.vec_off + a];
  __syncthreads();
  smooth_proposal<LAW>(A, m, xt, racc);
  for (int a = threadIdx.x; a < m.n; a += blockDim.x) A.out[m.vec_off + a] = xt[a];
}

// ------------------------------------------------------------------------------------------
// k_local_newton: the batched local corrections T_i of Eq. 4
// ------------------------------------------------------------------------------------------
// MAXT is the largest CTA the instantiation is compiled for: 128-thread CTAs keep four CTAs per SM
// within the register file; 256-thread CTAs two (Eq. 1), or one with the whole register budget per
// thread (Eq. 2, whose element tangents need it).
template <int LAW, typename FT, int MAXT>
__global__ void __launch_bounds__(MAXT, (MAXT <= 128 ? 4 : LAW == NLS_LAW_DIFFUSION ? 2 : 1))
    k_local_newton(LocalArgs A) {
  extern __shared__ __align__(128) unsigned char smem[];
  const LocalPlan P = newton_plan<FT>(A.max_n, A.max_nt, A.max_b);
  double* xt = (double*)(smem + P.xt);
  double* racc = (double*)(smem + P.racc);  // residual being assembled
  double* red = (double*)(smem + P.red);
  FT* win = (FT*)(smem + P.win);
  FT* yv = win;  // the solve vector lives in the LU window once the factors are packed
  int* flag = (int*)(smem + P.flag);
  // no static shared memory: in front of an array aligned to 128 bytes it would take as many of the limit
  int* const s_item = flag + 3;
  const int tid = threadIdx.x, nd = A.ndof;
  const size_t win_cap = (P.flag - P.win) / sizeof(FT);
  const int inv_warps = min((int)(blockDim.x >> 5), (int)(win_cap / dev::pack_scratch<FT>()));
  long long tp = clock64();
  // thread 0 charges the cycles since the last mark to phase `id` (profiling only)
  auto mark = [&](int id) {
    if (A.phase && tid == 0) {
      const long long t = clock64();
      atomicAdd(A.phase + id, (unsigned long long)(t - tp));
      tp = t;
    }
  };
  for (;;) {
    if (tid == 0) *s_item = atomicAdd(A.queue, 1);
    __syncthreads();
    const int item = *s_item;
    __syncthreads();
    if (item >= A.count) break;
    const int sub = A.order[item];
    const SubMeta m = A.meta[sub];
    const int n = m.n;
    double* csr = A.csr + m.nnz_off;
    FT* F = (FT*)A.factor + m.factor_off;
    FT* Dv = (FT*)A.dinv + m.dinv_off;
    double* wb = A.wbuf + m.vec_off;
    double* r = A.work + m.vec_off;                  // current residual
    double* s = A.work + A.work_stride + m.vec_off;  // Newton step
    // the LU window serves the solves: the solve vector, then the ring of operands
    const size_t ring_at = align_up(P.win + sizeof(FT) * align_up(n, dev::SolveBlock<FT>::BS), 128);
    const Ring ring{smem + ring_at, n > 0 && ring_at < P.flag ? dev::ring_stages<FT>(m.b, P.flag - ring_at) : 0};
    for (int t = tid; t < m.nt; t += blockDim.x)
      xt[t] = A.x[(int64_t)A.tnode_gid[m.tnode_off + t / nd] * nd + t % nd];
    __syncthreads();
    bool ok = local_residual<LAW>(A, m, xt, racc);
    double loc = 0.0;
    for (int a = tid; a < n; a += blockDim.x) {
      r[a] = racc[a];
      loc += racc[a] * racc[a];
    }
    double rn = sqrt(dev::block_sum(loc, red));
    if (!ok) rn = INFINITY;
    // the stopping test is relative to the residual of the method's own start R_i x, with or
    // without a proposed start, so the proposal cannot change the accuracy of T_i
    const double tol = fmax(A.atol, A.rtol * rn);
    if (A.guess) {
      // acceptance test: take the proposed start only if its local residual is smaller
      for (int a = tid; a < n; a += blockDim.x) {
        wb[a] = xt[a];
        xt[a] = A.guess[m.vec_off + a];
      }
      __syncthreads();
      bool okg = smooth_proposal<LAW>(A, m, xt, racc);
      double lg = 0.0;
      for (int a = tid; a < n; a += blockDim.x) lg += racc[a] * racc[a];
      double rng = sqrt(dev::block_sum(lg, red));
      if (!okg) rng = INFINITY;
      const bool take = isfinite(rng) && rng < rn;
      if (take) {
        for (int a = tid; a < n; a += blockDim.x) r[a] = racc[a];
        rn = rng;
      } else {
        for (int a = tid; a < n; a += blockDim.x) xt[a] = wb[a];
      }
      __syncthreads();
      if (tid == 0 && A.accepted) A.accepted[sub] = take ? 1 : 0;
    }
    int its = 0, status = ST_OK, chord = 0;
    if (!isfinite(rn)) status = ST_NONFINITE;
    // the stored factors (and local Jacobian) are those of this subdomain's converged state of
    // the previous F_x evaluation when that evaluation succeeded here: chord steps with them
    // until one contracts the residual by less than a factor 10 or fails the line search
    bool stored = A.reuse && A.status[sub] == ST_OK;
    mark(0);
    while (status == ST_OK && rn > tol) {
      if (its >= A.maxit) {
        status = ST_MAXIT;
        break;
      }
      if (!stored) {
        local_jacobian<LAW, FT>(A, m, xt, csr, F);
        mark(1);
        if (dev::band_lu_inplace<FT>(n, m.b, F, win, win_cap, flag)) {
          status = ST_PIVOT;
          break;
        }
        dev::band_pack_solve<FT>(n, m.b, F, Dv, win, inv_warps);
        mark(2);
      }
      if (!local_solve<FT, false>(A, m, Dv, r, rn, racc, yv, red, ring)) {
        status = ST_TIMEOUT;
        if (tid == 0) *A.err = 1;
        break;
      }
      mark(3);
      for (int a = tid; a < n; a += blockDim.x) {
        s[a] = racc[a];
        wb[a] = xt[a];
      }
      __syncthreads();
      double alpha = 1.0, rtn = INFINITY;
      bool accepted = false;
      for (int trial = 0; trial < A.ls_trials; ++trial) {
        for (int a = tid; a < n; a += blockDim.x) xt[a] = wb[a] - alpha * s[a];
        __syncthreads();
        const bool tok = local_residual<LAW>(A, m, xt, racc);
        double l2 = 0.0;
        for (int a = tid; a < n; a += blockDim.x) l2 += racc[a] * racc[a];
        rtn = sqrt(dev::block_sum(l2, red));
        if (!tok) rtn = INFINITY;
        if (isfinite(rtn) && rtn <= (1.0 - A.armijo * alpha) * rn) {
          accepted = true;
          break;
        }
        alpha *= 0.5;
      }
      mark(4);
      if (!accepted) {
        for (int a = tid; a < n; a += blockDim.x) xt[a] = wb[a];
        __syncthreads();
        if (stored) {  // retry the step with the Jacobian at the current state
          stored = false;
          continue;
        }
        ++its;
        status = ST_LS;
        break;
      }
      ++its;
      if (stored) {
        ++chord;
        if (rtn > 0.1 * rn) stored = false;
      }
      for (int a = tid; a < n; a += blockDim.x) r[a] = racc[a];
      __syncthreads();
      rn = rtn;
    }
    if (A.want_tangent && status != ST_NONFINITE && status != ST_PIVOT && status != ST_TIMEOUT) {
      local_jacobian<LAW, FT>(A, m, xt, csr, F);
      mark(5);
      if (!A.split_factor) {
        if (dev::band_lu_inplace<FT>(n, m.b, F, win, win_cap, flag)) status = ST_PIVOT;
        else dev::band_pack_solve<FT>(n, m.b, F, Dv, win, inv_warps);
      }
      mark(6);
    }
    for (int a = tid; a < n; a += blockDim.x) {
      wb[a] = xt[a];
      if (A.owned[m.vec_off + a]) {
        const int64_t g = (int64_t)A.tnode_gid[m.tnode_off + a / nd] * nd + a % nd;
        A.out[g] = A.x[g] - xt[a];
      }
    }
    if (tid == 0) {
      A.its[sub] = its;
      if (A.chord) A.chord[sub] = chord;
      A.status[sub] = status;
    }
    __syncthreads();
    mark(7);
  }
}

// ------------------------------------------------------------------------------------------
// k_local_factor: the tangent's refactorisation at the converged states -- band LU of the band
// that k_local_newton assembled and the packed solve operands -- as its own launch.  The Newton
// kernel's FP64 element tangents of Eq. 2 hold all of an SM's registers for one CTA; this kernel
// needs few registers and (FP32) about 65 KB of shared memory, so three CTAs share an SM and hide
// each other's per-step barrier latency.  One CTA per subdomain, longest first; subdomains whose
// local solve failed are skipped, a zero pivot marks the subdomain ST_PIVOT.
// ------------------------------------------------------------------------------------------
template <typename FT>
__host__ __device__ inline LocalPlan factor_plan(int max_b) {
  LocalPlan p{};
  size_t o = 0;
  const size_t lu = dev::band_lu_window<FT>(max_b, 1);
  const size_t inv = 4 * dev::pack_scratch<FT>();
  p.win = o; o += align_up(sizeof(FT) * (lu > inv ? lu : inv), 16);
  p.flag = o; o += 16;
  p.total = o;
  return p;
}

// MAXT = 256: three CTAs per SM; MAXT = 512: one, for at most one subdomain per SM.
template <typename FT, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT <= 256 ? 3 : 1) k_local_factor(LocalArgs A) {
  extern __shared__ __align__(128) unsigned char smem[];
  const LocalPlan P = factor_plan<FT>(A.max_b);
  FT* win = (FT*)(smem + P.win);
  int* flag = (int*)(smem + P.flag);
  const size_t win_cap = (P.flag - P.win) / sizeof(FT);
  const int inv_warps = min((int)(blockDim.x >> 5), (int)(win_cap / dev::pack_scratch<FT>()));
  const int sub = A.order[blockIdx.x];
  const int st = A.status[sub];
  if (st == ST_NONFINITE || st == ST_PIVOT || st == ST_TIMEOUT) return;
  const SubMeta m = A.meta[sub];
  FT* F = (FT*)A.factor + m.factor_off;
  FT* Dv = (FT*)A.dinv + m.dinv_off;
  if (dev::band_lu_inplace<FT>(m.n, m.b, F, win, win_cap, flag)) {
    if (threadIdx.x == 0) A.status[sub] = ST_PIVOT;
  } else {
    dev::band_pack_solve<FT>(m.n, m.b, F, Dv, win, inv_warps);
  }
}

// ------------------------------------------------------------------------------------------
// k_local_apply: out[owned] = (R_i DF(v_i) P_i)^-1 R_i DF(v_i) v  (+ add[owned])
// ------------------------------------------------------------------------------------------
// MAXT = 256: the whole register budget; 128: three CTAs per SM.
template <typename FT, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT <= 128 ? 3 : 1) k_local_apply(LocalArgs A) {
  extern __shared__ __align__(128) unsigned char smem[];
  const LocalPlan P = apply_plan<FT>(A.max_n, A.max_nt, A.max_b, A.ring);
  double* yt = (double*)(smem + P.xt);
  double* red = (double*)(smem + P.red);
  FT* yv = (FT*)(smem + P.win);
  const int sub = A.order[blockIdx.x], tid = threadIdx.x, nd = A.ndof;
  const SubMeta m = A.meta[sub];
  const int n = m.n;
  const Ring ring{smem + P.flag, A.ring && n > 0 ? dev::ring_stages<FT>(m.b, P.total - P.flag) : 0};
  const FT* Dv = (const FT*)A.dinv + m.dinv_off;
  double* q = A.work + m.vec_off;
  for (int t = tid; t < m.nt; t += blockDim.x) yt[t] = A.v[(int64_t)A.tnode_gid[m.tnode_off + t / nd] * nd + t % nd];
  __syncthreads();
  double loc = 0.0;
  for (int a = tid; a < n; a += blockDim.x) {
    double acc = 0.0;
    for_row(A, m, a, [&](double v, int32_t col) { acc += v * yt[col]; });
    q[a] = acc;
    loc += acc * acc;
  }
  const double qn = sqrt(dev::block_sum(loc, red));
  double* z = yt;  // the table vector has been used
  if (!local_solve<FT, true>(A, m, Dv, q, qn, z, yv, red, ring) && tid == 0) *A.err = 1;
  for (int a = tid; a < n; a += blockDim.x)
    if (A.owned[m.vec_off + a]) {
      const int64_t g = (int64_t)A.tnode_gid[m.tnode_off + a / nd] * nd + a % nd;
      A.out[g] = z[a] + (A.add ? A.add[g] : 0.0);
    }
}

// ------------------------------------------------------------------------------------------
// coarse space: harmonic extension (setup) and Galerkin blocks
// ------------------------------------------------------------------------------------------
template <int LAW>
__global__ void __launch_bounds__(256) k_harmonic(LocalArgs A) {
  extern __shared__ __align__(128) unsigned char smem[];
  const SmemPlan P = harmonic_plan(A.max_n, A.max_nt, A.max_b);
  double* xt = (double*)(smem + P.xt);
  double* yv = (double*)(smem + P.yv);
  double* win = (double*)(smem + P.win);
  double* rp = (double*)(smem + P.rp);
  int* flag = (int*)(smem + P.flag);
  const int j = blockIdx.x, tid = threadIdx.x, nd = A.ndof;
  const SubMeta m = A.meta[j];
  const int n = m.n;
  const int nc = A.cj_ptr[j + 1] - A.cj_ptr[j];
  double* phi = const_cast<double*>(A.phi) + A.phi_off[j];
  if (tid == 0) A.status[j] = ST_OK;
  const int32_t* rowptr = A.rowptr + m.rowptr_off;
  const int32_t* colidx = A.colidx + m.nnz_off;
  double* csr = A.csr + m.nnz_off;
  double* F = (double*)A.factor + m.factor_off;
  for (int t = tid; t < m.nt; t += blockDim.x) xt[t] = A.x[(int64_t)A.tnode_gid[m.tnode_off + t / nd] * nd + t % nd];
  __syncthreads();
  local_jacobian<LAW>(A, m, xt, csr);
  if (n == 0 || nc == 0) return;
  dev::RowSource src{rowptr, colidx, csr};
  if (dev::band_lu<double>(n, m.b, src, F, win, rp, flag)) {
    if (tid == 0) A.status[j] = ST_PIVOT;
    return;
  }
  for (int lc = 0; lc < nc; ++lc) {
    for (int a = tid; a < n; a += blockDim.x) {
      double acc = 0.0;
      for (int k = rowptr[a]; k < rowptr[a + 1]; ++k) {
        const int col = colidx[k];
        if (col >= n) acc -= csr[k] * phi[(int64_t)col * nc + lc];
      }
      yv[a] = acc;
    }
    __syncthreads();
    dev::band_solve<double>(n, m.b, F, yv);
    for (int a = tid; a < n; a += blockDim.x) phi[(int64_t)a * nc + lc] = yv[a];
    __syncthreads();
  }
}

// Rows of Phi_j and K^(j) Phi_j that the Galerkin kernel keeps in shared memory at a time: kGalRows, or as
// many (one at least) as leave room for two CTAs per SM where a subdomain has more than 226 coarse dofs (a
// long one beside many small ones).  The sums run over the rows in order, however many are kept.
constexpr int kGalRows = 32;
int galerkin_rows(size_t smem_optin, int max_nc) {
  const size_t half = (smem_optin + 1024) / 2 - 1024;  // 1 KB of every CTA is the system's
  return (int)std::min<size_t>(kGalRows, std::max<size_t>(1, half / (2 * sizeof(double) * std::max(max_nc, 1))));
}
size_t galerkin_smem(size_t smem_optin, int max_nt, int max_nc) {
  return sizeof(double) * std::max((size_t)max_nt, (size_t)2 * galerkin_rows(smem_optin, max_nc) * max_nc);
}

template <int LAW>
__global__ void __launch_bounds__(256, 2) k_galerkin(LocalArgs A) {
  extern __shared__ __align__(128) unsigned char smem[];
  double* xt = (double*)smem;
  const int j = blockIdx.x, tid = threadIdx.x, nd = A.ndof;
  const SubMeta m = A.meta[j];
  const int nc = A.cj_ptr[j + 1] - A.cj_ptr[j];
  const double* phi = A.phi + A.phi_off[j];
  double* Y = A.Y + A.phi_off[j];
  const int32_t* rowptr = A.rowptr + m.rowptr_off;
  const int32_t* colidx = A.colidx + m.nnz_off;
  double* csr = A.csr + m.nnz_off;
  for (int t = tid; t < m.nt; t += blockDim.x) xt[t] = A.x[(int64_t)A.tnode_gid[m.tnode_off + t / nd] * nd + t % nd];
  __syncthreads();
  local_jacobian<LAW>(A, m, xt, csr);
  if (nc == 0) return;
  // Y = K^(j) Phi_j
  for (int64_t idx = tid; idx < (int64_t)m.nt * nc; idx += blockDim.x) {
    const int t = (int)(idx / nc), lc = (int)(idx % nc);
    double acc = 0.0;
    for (int k = rowptr[t]; k < rowptr[t + 1]; ++k) acc += csr[k] * phi[(int64_t)colidx[k] * nc + lc];
    Y[idx] = acc;
  }
  __syncthreads();
  // block = Phi_j^T Y: rows of Phi and Y through shared memory, A.gal_rows at a time, one thread per entry
  // (a warp per entry read both arrays 8 bytes at a time, nc entries apart).  Eq. 2's tangent is
  // symmetric: the entries c <= d are formed, and mirrored.
  double* ps = xt;  // the table vector has been used; A.gal_rows x nc of Phi, then of Y
  double* ys = ps + A.gal_rows * nc;
  double* blk = A.blk + A.blk_off[j];
  const bool sym = LAW == NLS_LAW_NEOHOOKE;
  const int pairs = sym ? nc * (nc + 1) / 2 : nc * nc;
  for (int e0 = 0; e0 < pairs; e0 += blockDim.x) {
    const int e = e0 + tid;
    int c = 0, d = 0;
    if (sym) {  // e-th pair of the rows 0 .. c of the lower triangle
      c = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
      while ((c + 1) * (c + 2) / 2 <= e) ++c;
      while (c * (c + 1) / 2 > e) --c;
      d = e - c * (c + 1) / 2;
    } else {
      c = e / nc;
      d = e % nc;
    }
    double acc = 0.0;
    for (int t0 = 0; t0 < m.nt; t0 += A.gal_rows) {
      const int rows = min(A.gal_rows, m.nt - t0);
      __syncthreads();
      for (int q = tid; q < rows * nc; q += blockDim.x) {
        ps[q] = phi[(int64_t)t0 * nc + q];
        ys[q] = Y[(int64_t)t0 * nc + q];
      }
      __syncthreads();
      if (e < pairs)
        for (int t = 0; t < rows; ++t) acc += ps[t * nc + d] * ys[t * nc + c];
    }
    if (e < pairs) {
      if (sym) blk[c * nc + d] = blk[d * nc + c] = acc;
      else blk[d * nc + c] = acc;
    }
  }
}

__global__ void k_a0_gather(int64_t nentries, const int32_t* ptr, const int64_t* src, const double* blk, double* A0) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nentries; e += (int64_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int32_t k = ptr[e]; k < ptr[e + 1]; ++k) acc += blk[src[k]];
    A0[e] = acc;
  }
}

// to[k] = from[src[k]], 0 where src[k] is negative (padding of a sliced matrix)
__global__ void k_gather_values(int64_t n, const int64_t* src, const double* from, double* to) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    to[k] = src[k] >= 0 ? from[src[k]] : 0.0;
}

// the same for positions kept by position32
__global__ void k_gather_values32(int64_t n, const int32_t* src, const double* from, double* to) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    to[k] = from[(uint32_t)src[k]];
}

// coarse band factorization (one CTA); the window also holds the packing scratch of at least four
// warps
template <typename FT>
__host__ __device__ constexpr size_t coarse_window(int b0) {
  const size_t lu = dev::band_lu_window<FT>(b0, 1), inv = 4 * dev::pack_scratch<FT>();
  return lu > inv ? lu : inv;
}
template <typename FT>
__global__ void __launch_bounds__(1024) k_coarse_factor(int N0, int b0, const double* A0, FT* F, FT* Dinv, int* status) {
  extern __shared__ __align__(128) unsigned char smem[];
  FT* win = (FT*)smem;
  int* flag = (int*)(smem + align_up(sizeof(FT) * coarse_window<FT>(b0), 16));
  const int64_t total = (int64_t)N0 * (2 * b0 + 1);
  // entries left of the matrix count as zero, whatever the caller's band holds there
  for (int64_t k = threadIdx.x; k < total; k += blockDim.x) {
    const int d = (int)(k % (2 * b0 + 1));
    F[k] = (k / (2 * b0 + 1) - b0 + d >= 0) ? (FT)A0[k] : (FT)0;
  }
  __syncthreads();
  const int bad = dev::band_lu_inplace<FT>(N0, b0, F, win, coarse_window<FT>(b0), flag);
  // the LU window is free again: it holds the packing scratch
  const int pw = min((int)(blockDim.x >> 5), (int)(coarse_window<FT>(b0) / dev::pack_scratch<FT>()));
  if (!bad) dev::band_pack_solve<FT>(N0, b0, F, Dinv, win, pw);
  if (threadIdx.x == 0) *status = bad ? ST_PIVOT : ST_OK;
}

// Bytes of the solve vector before the operand ring.
template <typename FT>
__host__ __device__ constexpr size_t coarse_solve_vector(int N0) {
  return (sizeof(FT) * (size_t)((N0 + dev::SolveBlock<FT>::BS - 1) / dev::SolveBlock<FT>::BS * dev::SolveBlock<FT>::BS) + 127) /
         128 * 128;
}

// Columns of A_0^-1 from the band factors: the solves A_0 z = e_col in the factors' precision, stored in
// that precision and transposed (AinvT[col][row]) so that the GEMV below reads it coalesced.  FP32
// columns are refined where they are applied (coarse_solve): the FP64 residual of one vector costs
// N0 (2 b0 + 1) multiply-adds, that of every column of the inverse N0 times as many.  The forward
// sweep starts at the block of the column, above which e_col and z vanish.
//
// k_coarse_inverse: one CTA per column, through the operand ring.
template <typename FT>
__global__ void __launch_bounds__(256) k_coarse_inverse(int N0, int b0, const FT* Dinv, FT* AinvT, int stages, int* err) {
  extern __shared__ __align__(128) unsigned char smem[];
  FT* y = (FT*)smem;
  for (int col = blockIdx.x; col < N0; col += gridDim.x) {
    for (int a = threadIdx.x; a < N0; a += blockDim.x) y[a] = (a == col) ? (FT)1 : (FT)0;
    __syncthreads();
    if (!dev::band_solve_ring<FT>(N0, b0, Dinv, y, smem + coarse_solve_vector<FT>(N0), stages,
                                  col / dev::SolveBlock<FT>::BS) &&
        threadIdx.x == 0)
      *err = 1;
    for (int a = threadIdx.x; a < N0; a += blockDim.x) AinvT[(int64_t)col * N0 + a] = y[a];
    __syncthreads();
  }
}

// k_coarse_inverse_blocks: 32 columns per CTA.  With one column per CTA every column streams all packed
// operands from L2 (N_0 = 5235, b_0 = 197: 38 GB, 3.5 ms).  Here a step's operands are staged once in
// shared memory for 32 columns.  Rows of the operands as broadcast 16-byte groups against one column per
// lane took a shared-memory word per multiply-add (2.4 ms); a warp now takes 32 rows (FP64: 16) by 32
// columns, a lane 8 x 4 (4 x 4) of them, for 12 words per 32 multiply-adds (1.4 ms).  The rows that
// a block couples to are kept in a window of shared memory; the forward result of a
// block goes through AinvT.  A column's sums are those of band_solve_packed: even and odd terms
// apart, blocks in order.
template <typename FT>
__host__ __device__ constexpr int inverse_blocks(int b0) {  // blocks of the window
  constexpr int BS = dev::SolveBlock<FT>::BS;
  return 1 + (b0 + BS - 1) / BS;
}
template <typename FT>
__host__ __device__ constexpr size_t inverse_smem(int b0, int buffers) {
  constexpr size_t BS = dev::SolveBlock<FT>::BS;
  return sizeof(FT) * (buffers * BS * (BS + (b0 + 3) / 4 * 4) + inverse_blocks<FT>(b0) * BS * 33);
}
// R consecutive rows of the operands, from row r, times the block held in v
template <int R, typename FT>
__device__ __forceinline__ void inverse_dots(const FT* rows, int r, const FT* v, FT* out) {
  constexpr int BS = dev::SolveBlock<FT>::BS, G = dev::LuTile<FT>::G;
  using Vec = dev::LuVec<FT>;
  FT a0[R], a1[R];
#pragma unroll
  for (int i = 0; i < R; ++i) a0[i] = a1[i] = 0;
#pragma unroll
  for (int j = 0; j < BS; j += G) {
    Vec w[R];
#pragma unroll
    for (int i = 0; i < R; ++i) w[i] = *(const Vec*)(rows + (r + i) * BS + dev::packed_at<FT>(r + i, j));
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int q = 0; q < G; q += 2) {
        a0[i] += w[i].v[q] * v[j + q];
        a1[i] += w[i].v[q + 1] * v[j + q + 1];
      }
  }
#pragma unroll
  for (int i = 0; i < R; ++i) out[i] = a0[i] + a1[i];
}
// Rows r0 + TR (lane / 8) + i (i < TR; rows past `rows` read the last one) of the operands times columns
// lane % 8 + 8 c of the BS x 32 block `v`, even and odd terms apart as above.
template <int TR, typename FT>
__device__ __forceinline__ void inverse_tile(const FT* ops, int r0, int rows, const FT* v, int ld, FT (&out)[TR][4]) {
  constexpr int BS = dev::SolveBlock<FT>::BS, G = dev::LuTile<FT>::G;
  using Vec = dev::LuVec<FT>;
  const int lane = threadIdx.x & 31;
  int r[TR];
#pragma unroll
  for (int i = 0; i < TR; ++i) r[i] = min(r0 + TR * (lane >> 3) + i, rows - 1);
  v += lane & 7;
  FT odd[TR][4];
#pragma unroll
  for (int i = 0; i < TR; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) out[i][c] = odd[i][c] = 0;
#pragma unroll 2
  for (int j = 0; j < BS; j += G) {
    Vec w[TR];
#pragma unroll
    for (int i = 0; i < TR; ++i) w[i] = *(const Vec*)(ops + r[i] * BS + dev::packed_at<FT>(r[i], j));
#pragma unroll
    for (int q = 0; q < G; q += 2) {
      FT a[4], b[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) a[c] = v[(j + q) * ld + 8 * c], b[c] = v[(j + q + 1) * ld + 8 * c];
#pragma unroll
      for (int i = 0; i < TR; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          out[i][c] += w[i].v[q] * a[c];
          odd[i][c] += w[i].v[q + 1] * b[c];
        }
    }
  }
#pragma unroll
  for (int i = 0; i < TR; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) out[i][c] += odd[i][c];
}
template <typename FT>
__global__ void __launch_bounds__(256) k_coarse_inverse_blocks(int N0, int b0, const FT* __restrict__ Dinv,
                                                                FT* AinvT, int buffers) {
  constexpr int BS = dev::SolveBlock<FT>::BS, G = dev::LuTile<FT>::G, LD = 33;
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int SE = BS * (BS + b0), SP = BS * (BS + (b0 + 3) / 4 * 4);  // operands of one step, and their room
  FT* ops = (FT*)smem;
  FT* win = ops + buffers * SP;  // row i of the matrix at (i mod WR) LD, a column per lane
  const int WB = inverse_blocks<FT>(b0), WR = WB * BS;
  const int nblk = (N0 + BS - 1) / BS, c0 = blockIdx.x * 32, t0 = c0 / BS;
  const int64_t PB = dev::packed_block_entries<FT>(b0);
  const int steps = (nblk - t0) + nblk;
  auto block_of = [&](int s) { return s < nblk - t0 ? t0 + s : steps - 1 - s; };
  auto stage = [&](int s, FT* dst) {  // operands of step s
    if (s < steps) {
      const bool fwd = s < nblk - t0;
      const FT* P = Dinv + (int64_t)block_of(s) * PB;
      const FT *d = P + (fwd ? 0 : BS * BS), *c = P + 2 * BS * BS + (fwd ? 0 : (int64_t)b0 * BS);
      for (int e = tid; e < SE / G; e += blockDim.x) {
        const FT* src = e < BS * BS / G ? d + e * G : c + (e - BS * BS / G) * G;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(tc::smem_u32(dst + e * G)), "l"(src)
                     : "memory");
      }
    }
    dev::cp_async_commit();
  };
  // the rows of block u enter the window: unit columns (forward) or the forward result
  auto enter = [&](int u, bool fwd) {
    if (u < 0 || u >= nblk) return;
    FT* w = win + (u % WB) * BS * LD;
#pragma unroll
    for (int q = 0; q < BS * 32 / 256; ++q) {
      const int e = tid + 256 * q, r = e % BS, c = e / BS, i = u * BS + r, col = c0 + c;
      FT v = 0;
      if (fwd) v = (i == col && i < N0) ? (FT)1 : (FT)0;
      else if (u >= t0 && i < N0 && col < N0) v = AinvT[(int64_t)col * N0 + i];
      w[r * LD + c] = v;
    }
  };
  stage(0, ops);
  for (int q = 0; q < WB; ++q) enter(t0 + q, true);
  for (int s = 0; s < steps; ++s) {
    const bool fwd = s < nblk - t0;
    const int t = block_of(s), k0 = t * BS;
    if (s == nblk - t0) {  // turn: the last blocks, all written out by this CTA
      __syncthreads();
      for (int q = 0; q < WB; ++q) enter(nblk - 1 - q, false);
    }
    FT* cur = ops + (buffers > 1 ? (s & 1) * SP : 0);
    if (buffers == 1 && s > 0) stage(s, ops);
    dev::cp_async_wait<0>();
    __syncthreads();
    if (buffers > 1) stage(s + 1, ops + ((s + 1) & 1) * SP);
    constexpr int RW = BS / 8;  // rows of the diagonal block per warp (eight warps)
    const int slot = (t % WB) * BS;
    FT v[BS], x[RW];
    FT* blk = win + slot * LD + lane;
#pragma unroll
    for (int j = 0; j < BS; ++j) v[j] = blk[j * LD];
    inverse_dots<RW, FT>(cur, wid * RW, v, x);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RW; ++i) blk[(wid * RW + i) * LD] = (k0 + wid * RW + i < N0) ? x[i] : (FT)0;
    __syncthreads();
    // the solved block to global memory, rows along the lanes
#pragma unroll
    for (int q = 0; q < BS * 32 / 256; ++q) {
      const int r = (tid + 256 * q) % BS, c = (tid + 256 * q) / BS;
      if (k0 + r < N0 && c0 + c < N0) AinvT[(int64_t)(c0 + c) * N0 + k0 + r] = win[(slot + r) * LD + c];
    }
    constexpr int TR = 2 * G;  // rows per lane
    for (int r0 = wid * 4 * TR; r0 < b0; r0 += 32 * TR) {
      FT y[TR][4];
      inverse_tile<TR, FT>(cur + BS * BS, r0, b0, win + slot * LD, LD, y);
      const int r = r0 + TR * (lane >> 3);
#pragma unroll
      for (int i = 0; i < TR; ++i) {
        const int row = fwd ? k0 + BS + r + i : k0 - 1 - r - i;
        int at = fwd ? slot + BS + r + i : slot - 1 - r - i;  // row mod WR
        at = at >= WR ? at - WR : at < 0 ? at + WR : at;
        if (r + i < b0 && row >= 0 && row < N0) {
#pragma unroll
          for (int c = 0; c < 4; ++c) win[at * LD + (lane & 7) + 8 * c] -= y[i][c];
        }
      }
    }
    __syncthreads();
    // block t leaves the window; the block beyond it on the other side takes its place
    if (fwd) enter(t + WB, true);
    else enter(t - WB, false);
  }
}

// z = A_0^-1 g with the explicit inverse (stored transposed).  Grid (row tiles of 32, column
// chunks): lane = row, the 8 warps of a CTA stride over the chunk's columns (coalesced rows of
// AinvT), warp partials are summed in shared memory in warp order, chunk partials go to `part`, and the
// last CTA of a row tile (a ticket per tile) adds them in chunk order, so the result is reproducible
// (a launch of its own for that sum: 3 to 6 us per application).  z = the sum (accumulate = 0) or z +=
// it (accumulate = 1); `reset`, if given, is cleared (the refinement flag of the solve that starts
// here).  With `skip` set (a refinement that has converged) the kernel returns at once.
//
// What bounds it is the FP64 unit: N_0^2 multiply-adds, and as long again for widening FP32 entries with
// the conversion instruction, which runs there too (N_0 = 5235: 115 us, of which the 110 MB take 17).  So
// an entry is widened with integer instructions (59 us), which is exact but for zeros, subnormal numbers,
// infinities and NaN: a warp lane that meets one among its next entries converts those the usual way.
constexpr int kGemvChunks = 16;
// Largest coarse dimension with an explicit inverse (N0^2 entries in the factors' precision:
// 1 GB in FP32 at the limit); larger coarse problems use the one-CTA band solve.
constexpr int kMaxInverseN0 = 16384;
// Coarse dofs up to which the inverse is formed column by column.  FP32 launches beside the local solves, by
// columns and 32 columns per CTA: 27 / 81 us at N_0 = 402, 207 / 232 at 1149, 407 / 527 at 1428, 402 / 539 at 2268,
// 1046 / 860 at 3600 (b_0 = 59 .. 167); FP64, whose CTAs end at b_0 = 112: 86 / 695 us at 402, 967 / 3425 at
// 1428.  The line lies below the crossing, where the two are within a third of each other.
constexpr int kInverseColumns = 2048;
// acc += sum_i AinvT[i * stride] * g[8 i], i < U, in order
template <int U>
__device__ __forceinline__ double gemv_terms(const float* A, int64_t stride, const double* g, double acc) {
  float a[U];
  double b[U];
  bool special = false;
#pragma unroll
  for (int i = 0; i < U; ++i) a[i] = A[i * stride], b[i] = g[8 * i];
#pragma unroll
  for (int i = 0; i < U; ++i) special |= (__float_as_uint(a[i]) << 1) - 0x01000000u >= 0xfe000000u;
  if (!special) {
    // sign, exponent re-biased by 1023 - 127, 23 bits of mantissa on top of the 52
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int q = __float_as_int(a[i]);
      acc += __hiloint2double(((q >> 3) & (int)0x8fffffff) + (896 << 20), q << 29) * b[i];
    }
  } else {
#pragma unroll
    for (int i = 0; i < U; ++i) acc += (double)a[i] * b[i];
  }
  return acc;
}
template <int U>
__device__ __forceinline__ double gemv_terms(const double* A, int64_t stride, const double* g, double acc) {
#pragma unroll
  for (int i = 0; i < U; ++i) acc += A[i * stride] * g[8 * i];
  return acc;
}
template <typename FT>
__global__ void __launch_bounds__(256) k_dense_gemv_t(int N0, const FT* AinvT, const double* g, double* part,
                                                       unsigned* tickets, double* z, int accumulate, const int* skip,
                                                       int* reset) {
  if (skip && *skip) return;
  __shared__ double acc_s[8][33];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int row = blockIdx.x * 32 + lane;
  const int per = (N0 + gridDim.y - 1) / gridDim.y;
  const int c0 = blockIdx.y * per, c1 = min(N0, c0 + per);
  double acc = 0.0;
  if (row < N0) {
    int col = c0 + wid;
    const int64_t stride = 8 * (int64_t)N0;
    for (; col + 56 < c1; col += 64) acc = gemv_terms<8>(AinvT + (int64_t)col * N0 + row, stride, g + col, acc);
    for (; col + 8 < c1; col += 16) acc = gemv_terms<2>(AinvT + (int64_t)col * N0 + row, stride, g + col, acc);
    if (col < c1) acc = gemv_terms<1>(AinvT + (int64_t)col * N0 + row, stride, g + col, acc);
  }
  acc_s[wid][lane] = acc;
  __syncthreads();
  if (wid != 0) return;
  if (row < N0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += acc_s[w][lane];
    part[(int64_t)blockIdx.y * N0 + row] = t;
  }
  __threadfence();
  __syncwarp();
  unsigned n = 0;
  if (lane == 0) n = atomicAdd(tickets + blockIdx.x, 1u);
  if (__shfl_sync(0xffffffffu, n, 0) != kGemvChunks - 1) return;
  __threadfence();
  if (lane == 0) {
    tickets[blockIdx.x] = 0;
    if (reset && blockIdx.x == 0) *reset = 0;
  }
  if (row >= N0) return;
  double p[kGemvChunks], t = 0.0;
#pragma unroll
  for (int c = 0; c < kGemvChunks; ++c) p[c] = __ldcg(part + (int64_t)c * N0 + row);
#pragma unroll
  for (int c = 0; c < kGemvChunks; ++c) t += p[c];
  z[row] = accumulate ? z[row] + t : t;
}

// One step of the refinement of an explicit-inverse coarse solve: r = g - A_0 z (FP64 band
// A_0, one warp per row, 8 rows per CTA) and its test.  Every CTA stores its partial sums of
// r^2 and g^2; the last CTA to finish (atomic ticket) adds them in CTA order and sets *done
// when ||r|| <= ir_rtol ||g|| (or the norms are not finite), then returns the ticket counter
// to 0.  With *done already set the kernel does nothing.
__global__ void __launch_bounds__(256) k_coarse_residual(int N0, int b0, const double* A0, const double* g,
                                                          const double* z, double* r, double* part,
                                                          unsigned* ticket, int* done, double ir_rtol) {
  if (*done) return;
  __shared__ double s_r[8], s_g[8];
  __shared__ int s_last;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int a = blockIdx.x * 8 + wid, W = 2 * b0 + 1;
  double rr = 0.0, gg = 0.0;
  if (a < N0) {
    double acc = 0.0;
    for (int d = lane; d < W; d += 32) {
      const int cc = a - b0 + d;
      if (cc >= 0 && cc < N0) acc += A0[(int64_t)a * W + d] * z[cc];
    }
    acc = dev::warp_sum(acc);
    const double ra = g[a] - acc;
    if (lane == 0) r[a] = ra;
    rr = ra * ra;
    gg = g[a] * g[a];
  }
  if (lane == 0) s_r[wid] = rr, s_g[wid] = gg;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tr = 0.0, tg = 0.0;
    for (int w = 0; w < 8; ++w) tr += s_r[w], tg += s_g[w];
    part[2 * blockIdx.x] = tr;
    part[2 * blockIdx.x + 1] = tg;
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (s_last && wid == 0) {
    __threadfence();
    double tr = 0.0, tg = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) tr += __ldcg(part + 2 * b), tg += __ldcg(part + 2 * b + 1);
    tr = dev::warp_sum(tr);
    tg = dev::warp_sum(tg);
    if (lane == 0) {
      *done = !(sqrt(tr) > ir_rtol * sqrt(tg)) ? 1 : 0;
      *ticket = 0;
    }
  }
}

// One coarse solve with the packed band factors in one CTA (the solve vector in shared memory):
// z = (accumulate ? z : 0) + A_0^-1 rhs in the factors' precision.  With *skip set (a refinement
// that has converged) the kernel does nothing; `reset`, if given, is cleared (the refinement flag
// of the solve that starts here).  Needs blockDim.x >= 32 + b0.  `stages`: stages of the operand ring
// behind the solve vector (at least two, and ring_threads threads), or 0: operands in registers.
template <typename FT>
__global__ void __launch_bounds__(512) k_coarse_band_solve(int N0, int b0, const FT* Dinv, const double* rhs,
                                                             double* z, int accumulate, const int* skip, int* reset,
                                                             int l2d, int stages, int* err) {
  if (skip && *skip) return;
  extern __shared__ __align__(128) unsigned char smem[];
  FT* y = (FT*)smem;
  if (reset && threadIdx.x == 0) *reset = 0;
  for (int a = threadIdx.x; a < N0; a += blockDim.x) y[a] = (FT)rhs[a];
  __syncthreads();
  if (stages) {
    if (!dev::band_solve_ring<FT>(N0, b0, Dinv, y, smem + coarse_solve_vector<FT>(N0), stages) && threadIdx.x == 0)
      *err = 1;
  } else {
    dev::band_solve_packed<FT, true>(N0, b0, Dinv, y, l2d);
  }
  for (int a = threadIdx.x; a < N0; a += blockDim.x) z[a] = (accumulate ? z[a] : 0.0) + (double)y[a];
}

// ------------------------------------------------------------------------------------------
// global assembly: the residual by element contributions and node sums, the Jacobian in colour
// passes (elements of one colour share no node)
// ------------------------------------------------------------------------------------------
// Element residuals (the weak forms of Eqs. 1 and 2) of every element, one thread per element,
// into Re[(e nen + a) ndof + d]; k_node_residual adds them up per node.
template <int LAW>
__global__ void k_elem_residual(int64_t ne, const int32_t* conn, const double* geom, const double* kcoef,
                                const double* x, double* Re, dev::NHLaw nh, int* bad) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ne; e += (int64_t)gridDim.x * blockDim.x) {
    if (LAW == NLS_LAW_DIFFUSION) {
      const int32_t* c = conn + e * 3;
      const double* geo = geom + e * 8;
      const dev::P1State st = dev::p1_state(geo, kcoef[e], x[c[0]], x[c[1]], x[c[2]]);
      double re[3];
      dev::p1_residual(geo, st, re);
#pragma unroll
      for (int a = 0; a < 3; ++a) Re[e * 3 + a] = re[a];
    } else {
      const int32_t* c = conn + e * 4;
      const double* geo = geom + e * 40;
      double ue[8], re[8];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        ue[2 * a] = x[2 * (int64_t)c[a]];
        ue[2 * a + 1] = x[2 * (int64_t)c[a] + 1];
      }
      bool ok = true;
      dev::nh_residual(geo, ue, nh, re, ok);
      if (!ok) *bad = 1;
#pragma unroll
      for (int q = 0; q < 8; ++q) Re[e * 8 + q] = re[q];
    }
  }
}

// F = -load fext + the contributions of the elements around every node, added in ascending
// element order (star_ref[k] = e nen + a: element e, where the node is e's a-th); 0 on the
// Dirichlet dofs.
__global__ void k_node_residual(int64_t n_nodes, int nd, const int64_t* star_ptr, const int32_t* star_ref,
                                const double* Re, double load, const double* fext, const uint8_t* free_dof,
                                double* F) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n_nodes;
       v += (int64_t)gridDim.x * blockDim.x) {
    double acc0 = 0.0, acc1 = 0.0;
    for (int64_t k = star_ptr[v]; k < star_ptr[v + 1]; ++k) {
      const int64_t r = (int64_t)star_ref[k] * nd;
      acc0 += Re[r];
      if (nd == 2) acc1 += Re[r + 1];
    }
    for (int d = 0; d < nd; ++d) {
      const int64_t i = v * nd + d;
      F[i] = free_dof[i] ? -load * fext[i] + (d == 0 ? acc0 : acc1) : 0.0;
    }
  }
}

template <int LAW>
__global__ void k_global_jacobian(const int32_t* elems, int e0, int e1, const int32_t* conn, const double* geom,
                                  const double* kcoef, const double* x, const int32_t* epos, double* val,
                                  dev::NHLaw nh) {
  for (int i = e0 + blockIdx.x * blockDim.x + threadIdx.x; i < e1; i += gridDim.x * blockDim.x) {
    const int32_t e = elems[i];
    if (LAW == NLS_LAW_DIFFUSION) {
      const int32_t* c = conn + (int64_t)e * 3;
      const double* geo = geom + (int64_t)e * 8;
      const dev::P1State st = dev::p1_state(geo, kcoef[e], x[c[0]], x[c[1]], x[c[2]]);
      double K[9];
      dev::p1_jacobian<double>(geo, st, K);
      const int32_t* ep = epos + (int64_t)e * 9;
#pragma unroll
      for (int q = 0; q < 9; ++q) val[(uint32_t)ep[q]] += K[q];
    } else {
      const int32_t* c = conn + (int64_t)e * 4;
      const double* geo = geom + (int64_t)e * 40;
      double ue[8];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        ue[2 * a] = x[2 * (int64_t)c[a]];
        ue[2 * a + 1] = x[2 * (int64_t)c[a] + 1];
      }
      dev::NHTangent K;
      dev::nh_tangent(geo, ue, nh, K);
      const int32_t* ep = epos + (int64_t)e * 64;
#pragma unroll
      for (int q = 0; q < 64; ++q) val[(uint32_t)ep[q]] += K(q >> 4, (q >> 3) & 1, (q & 7) >> 1, q & 1);
    }
  }
}

// ------------------------------------------------------------------------------------------
// vector kernels
// ------------------------------------------------------------------------------------------
__global__ void k_axpby(int64_t n, double a, const double* x, double b, const double* y, double* z) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    z[i] = a * x[i] + (y ? b * y[i] : 0.0);
}

__global__ void k_mask(int64_t n, const uint8_t* free_dof, double* x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (!free_dof[i]) x[i] = 0.0;
}

// x = v on the free dofs, 0 elsewhere; y = 0 (y may be v's memory)
__global__ void k_masked_copy(int64_t n, const uint8_t* free_dof, const double* v, double* x, double* y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    x[i] = free_dof[i] ? v[i] : 0.0;
    y[i] = 0.0;
  }
}

__global__ void k_set_dirichlet(int64_t n, const uint8_t* free_dof, const double* ubc, double* x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (!free_dof[i]) x[i] = ubc[i];
}

// Row i of a global matrix in slices of 32 rows (one warp's rows read consecutive entries; see
// Context::g_slice): sum over its entries, eight of them in flight, padding included (value 0).  Bound
// by the entries' bytes; with CSR rows, one thread each, a warp touched 32 lines per entry (384^2
// Neo-Hooke: DF v 27.6 -> 18.5 us, P_0 c 24.5 -> 18.4 us, and P_0^T v, whose rows were coalesced but read
// one entry at a time, 31.6 -> 21 us).
__device__ __forceinline__ double sliced_row(int64_t i, const int64_t* __restrict__ slice, const int32_t* __restrict__ col,
                                             const double* __restrict__ val, const double* __restrict__ x) {
  const int64_t q = i >> 5, first = slice[q] + (i & 31);
  const int width = (int)((slice[q + 1] - slice[q]) >> 5);
  double acc = 0.0;
  int k = 0;
  for (; k + 8 <= width; k += 8) {
    double v[8];
    int32_t c[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = val[first + 32 * (k + e)], c[e] = col[first + 32 * (k + e)];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc += v[e] * x[c[e]];
  }
  for (; k < width; ++k) acc += val[first + 32 * k] * x[col[first + 32 * k]];
  return acc;
}

// y = J x on free rows (0 on Dirichlet rows)
__global__ void __launch_bounds__(256) k_spmv_free(int64_t n, const int64_t* slice, const int32_t* col, const double* val,
                                                   const uint8_t* free_dof, const double* x, double* y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = free_dof[i] ? sliced_row(i, slice, col, val, x) : 0.0;
}

// p = P0 c; y = a * x + s * p (x may be null), and p itself into `plain` where given
__global__ void __launch_bounds__(256) k_p0_apply(int64_t n, const int64_t* slice, const int32_t* col, const double* val,
                                                  const double* c, double a, const double* x, double s, double* y,
                                                  double* plain) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double p = sliced_row(i, slice, col, val, c);
    if (plain) plain[i] = p;
    if (y) y[i] = (x ? a * x[i] : 0.0) + s * p;
  }
}

// g = P0^T v, one CTA per coarse row (the rows are long: every fine dof in the support of the
// coarse function); fixed-order warp and CTA sums.
__global__ void __launch_bounds__(256) k_p0t_apply(int n0, const int32_t* rowptr, const int32_t* col,
                                                    const double* val, const double* v, double* g) {
  __shared__ double red[40];
  for (int r = blockIdx.x; r < n0; r += gridDim.x) {
    double acc = 0.0;
    const int32_t k1 = rowptr[r + 1];
    int32_t k = rowptr[r] + threadIdx.x;
    for (; k + 7 * 256 < k1; k += 8 * 256) {  // eight entries in flight
      double w[8];
      int32_t c[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) w[e] = val[k + 256 * e], c[e] = col[k + 256 * e];
#pragma unroll
      for (int e = 0; e < 8; ++e) acc += w[e] * v[c[e]];
    }
    for (; k < k1; k += 256) acc += val[k] * v[col[k]];
    acc = dev::block_sum(acc, red);
    if (threadIdx.x == 0) g[r] = acc;
  }
}

// ---- products of several vectors ------------------------------------------------------------------
// What bounds these kernels is FP64 issue and, at the smaller sizes, the launches: a warp's FP64
// instruction takes 64 cycles, so five additions per vector and warp for a shuffle reduction cost
// more than the products.  A CTA takes a tile of 256 E elements, w held in registers, eight vectors at
// a time; the eight sums of a warp are reduced together (nine additions instead of forty); the
// last CTA to finish adds the partial sums in CTA order, so results do not depend on scheduling.  One
// Gram-Schmidt pass with its update and the next pass's products is one launch: an iteration's
// orthogonalisation takes four launches instead of eleven (N = 296,450, 240 iterations: 43 -> 18 ms).
constexpr int kTile = 256;  // threads per CTA

// Sums of acc[0..7] over the warp; lane l returns the one of index 4 (l >> 4) + 2 ((l >> 3) & 1) +
// ((l >> 2) & 1).
__device__ __forceinline__ double warp_sum8(const double (&acc)[8]) {
  const int lane = threadIdx.x & 31;
  double a[4], b[2];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const bool up = lane & 16;
    a[q] = (up ? acc[q + 4] : acc[q]) + __shfl_xor_sync(0xffffffffu, up ? acc[q] : acc[q + 4], 16);
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const bool up = lane & 8;
    b[q] = (up ? a[q + 2] : a[q]) + __shfl_xor_sync(0xffffffffu, up ? a[q] : a[q + 2], 8);
  }
  const bool up = lane & 4;
  double s = (up ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, up ? b[0] : b[1], 4);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  return s;
}

// Partial sums of this CTA's tile: partial[i gridDim.x + blockIdx.x] = sum over the tile of V_i w.
template <int E>
__device__ void tile_dots(int64_t n, int nv, const double* __restrict__ V, int64_t ld, const double (&w)[E],
                          double* partial) {
  __shared__ double red[2][8][8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t k0 = (int64_t)blockIdx.x * kTile * E + threadIdx.x;
  for (int i0 = 0, s = 0; i0 < nv; i0 += 8, s ^= 1) {
    double acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      acc[q] = 0.0;
      if (i0 + q < nv) {
        const double* v = V + (int64_t)(i0 + q) * ld + k0;
#pragma unroll
        for (int e = 0; e < E; ++e)
          if (k0 + e * kTile < n) acc[q] += v[e * kTile] * w[e];
      }
    }
    const double t = warp_sum8(acc);
    if ((lane & 3) == 0) red[s][wid][4 * (lane >> 4) + 2 * ((lane >> 3) & 1) + ((lane >> 2) & 1)] = t;
    __syncthreads();
    if (threadIdx.x < 8 && i0 + (int)threadIdx.x < nv) {
      double sum = 0.0;
#pragma unroll
      for (int q = 0; q < kTile / 32; ++q) sum += red[s][q][threadIdx.x];
      partial[(int64_t)(i0 + threadIdx.x) * gridDim.x + blockIdx.x] = sum;
    }
  }
}

// True in every thread of the last CTA to get here (the ticket counter is returned to 0).
__device__ bool last_cta(unsigned* ticket) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    if (s_last) *ticket = 0;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last != 0;
}

// Sum of the CTAs' partial sums of vector i, by one warp; every lane receives it.
__device__ __forceinline__ double warp_total(int i, const double* partial) {
  double t = 0.0;
  for (int k = threadIdx.x & 31; k < (int)gridDim.x; k += 32) t += __ldcg(partial + (int64_t)i * gridDim.x + k);
  return dev::warp_sum(t);
}

template <int E>
__device__ __forceinline__ void tile_load(int64_t n, const double* w, double (&r)[E]) {
  const int64_t k0 = (int64_t)blockIdx.x * kTile * E + threadIdx.x;
#pragma unroll
  for (int e = 0; e < E; ++e) r[e] = k0 + e * kTile < n ? w[k0 + e * kTile] : 0.0;
}

// w -= sum_i coef[i] V_i on the tile, in place and in r
template <int E>
__device__ __forceinline__ void tile_update(int64_t n, int nv, const double* __restrict__ V, int64_t ld,
                                            const double* coef, double* w, double (&r)[E]) {
  const int64_t k0 = (int64_t)blockIdx.x * kTile * E + threadIdx.x;
  double s[E];
#pragma unroll
  for (int e = 0; e < E; ++e) s[e] = 0.0;
#pragma unroll 4
  for (int i = 0; i < nv; ++i) {
    const double c = coef[i];
    const double* v = V + (int64_t)i * ld + k0;
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (k0 + e * kTile < n) s[e] += c * v[e * kTile];
  }
#pragma unroll
  for (int e = 0; e < E; ++e) {
    r[e] -= s[e];
    if (k0 + e * kTile < n) w[k0 + e * kTile] = r[e];
  }
}

// out[i] = V_i . w, i < nv; with `coef` given, w -= sum_i coef[i] V_i first.
template <int E>
__global__ void __launch_bounds__(kTile) k_dots(int64_t n, int nv, const double* __restrict__ V, int64_t ld,
                                                const double* coef, double* w, double* partial, unsigned* ticket,
                                                double* out) {
  double r[E];
  tile_load<E>(n, w, r);
  if (coef) tile_update<E>(n, nv, V, ld, coef, w, r);
  tile_dots<E>(n, nv, V, ld, r, partial);
  if (!last_cta(ticket)) return;
  for (int i = threadIdx.x >> 5; i < nv; i += kTile / 32) {
    const double t = warp_total(i, partial);
    if ((threadIdx.x & 31) == 0) out[i] = t;
  }
}

// y = x / *nrm
__global__ void k_scale_inv(int64_t n, const double* x, const double* nrm, double* y) {
  const double s = 1.0 / *nrm;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = x[i] * s;
}

// ---- GMRES least-squares state on the device (GmresState) --------------------------------------

// A new cycle: g = (rn, 0, ..., 0).
__global__ void k_gmres_start(int m, double rn, double target, int limit, double* g, GmresState* st) {
  for (int i = threadIdx.x; i <= m; i += blockDim.x) g[i] = (i == 0) ? rn : 0.0;
  if (threadIdx.x == 0) {
    st->j = 0;
    st->done = 0;
    st->limit = limit;
    st->target = target;
    st->res = rn;
  }
}

// After iteration j (one thread): the Hessenberg column h_i = scal[i] + scal[half + i] (the two
// Gram-Schmidt passes, i <= j) and h_{j+1} = scal[kMaxGmresVecs]; apply the earlier rotations to it,
// form the rotation that annihilates h_{j+1}, rotate g, keep the column of R (row-major, m x m); then
// decide whether the cycle goes on, and (inside a graph) set `h`, the condition of the next
// iteration's IF node.
__device__ void gmres_givens(int j, int m, const double* scal, double* Rm, double* cs, double* sn, double* g,
                             GmresState* st, cudaGraphConditionalHandle h, int use_handle) {
  double lo = scal[0] + scal[kMaxGmresVecs / 2];
  const double hn = scal[kMaxGmresVecs];
  for (int i = 0; i < j; ++i) {
    const double hi = scal[i + 1] + scal[kMaxGmresVecs / 2 + i + 1];
    Rm[(size_t)i * m + j] = cs[i] * lo + sn[i] * hi;
    lo = -sn[i] * lo + cs[i] * hi;
  }
  const double d = hypot(lo, hn);
  cs[j] = lo / d;
  sn[j] = hn / d;
  Rm[(size_t)j * m + j] = d;
  g[j + 1] = -sn[j] * g[j];
  g[j] = cs[j] * g[j];
  const double res = fabs(g[j + 1]);
  const int done = (!isfinite(hn) || res <= st->target || hn == 0.0) ? 1 : 0;
  st->j = j + 1;
  st->res = res;
  st->done = done;
  if (use_handle) cudaGraphSetConditional(h, (!done && j + 1 < st->limit) ? 1u : 0u);
}

// The second Gram-Schmidt update of iteration j, w -= sum_i coef[i] V_i, its norm into
// scal[kMaxGmresVecs], and the Givens step.
template <int E>
__global__ void __launch_bounds__(kTile) k_gmres_update(int64_t n, int j, const double* __restrict__ V, int64_t ld,
                                                        const double* coef, double* w, double* partial,
                                                        unsigned* ticket, int m, double* scal, double* Rm, double* cs,
                                                        double* sn, double* g, GmresState* st,
                                                        cudaGraphConditionalHandle h, int use_handle) {
  __shared__ double red[40];
  double r[E], acc = 0.0;
  tile_load<E>(n, w, r);
  tile_update<E>(n, j + 1, V, ld, coef, w, r);
#pragma unroll
  for (int e = 0; e < E; ++e) acc += r[e] * r[e];
  acc = dev::block_sum(acc, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = acc;
  if (!last_cta(ticket) || threadIdx.x >= 32) return;
  const double t = warp_total(0, partial);
  if (threadIdx.x == 0) {
    scal[kMaxGmresVecs] = sqrt(t);
    gmres_givens(j, m, scal, Rm, cs, sn, g, st, h, use_handle);
  }
}

// y = R^-1 g over the cycle's st->j iterations (back substitution) into coef.
__global__ void k_gmres_lsq(int m, const double* Rm, const double* g, const GmresState* st, double* coef) {
  if (threadIdx.x != 0) return;
  const int n = st->j;
  for (int i = n - 1; i >= 0; --i) {
    double acc = g[i];
    for (int k = i + 1; k < n; ++k) acc -= Rm[(size_t)i * m + k] * coef[k];
    coef[i] = acc / Rm[(size_t)i * m + i];
  }
}

// w += sign sum_{i < st->j} coef[i] V_i (the number of vectors read from the device)
__global__ void k_multiaxpy_dev(int64_t n, const GmresState* st, const double* V, int64_t ld, const double* coef,
                                double sign, double* w) {
  const int nv = st->j;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int i = 0; i < nv; ++i) acc += coef[i] * V[(int64_t)i * ld + k];
    w[k] += sign * acc;
  }
}

}  // namespace


namespace {

inline int grid_for(int64_t n, int threads = 256) {
  int64_t b = (n + threads - 1) / threads;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, kVecBlocks));
}


// The triangular solves need warp 0 plus one thread per coupled row (32 + b threads).
int min_local_threads(const Context& c) { return ((32 + c.ov.max_b + 31) / 32) * 32; }

// 256 threads for Eq. 2, and for Eq. 1 while all subdomains are resident at two CTAs per SM: the
// kernel is bound by latency, and a subdomain's factorization takes 0.39 ms with 256 threads against
// 0.50 ms with 128 (n = 1598, b = 42, one CTA per SM).  With more subdomains than that, four CTAs of
// 128 threads per SM.
int local_threads(const Context& c) {
  int pick = c.opt.threads_per_block ? c.opt.threads_per_block
             : (c.ndof == 1 && c.dev && c.ov.count > 2 * c.dev->nsm) ? 128 : 256;
  if (!c.opt.threads_per_block && c.dev && c.dev->newton_T) pick = c.dev->newton_T;
  return std::max(pick, min_local_threads(c));
}

// Threads of the operand ring at the largest half bandwidth, and the largest CTA of the tangent application:
// in FP64 half bandwidths from 113 on need more, and keep the operands in registers (32 + b threads).
constexpr int kApplyMax = 256;
int apply_ring_threads(const Context& c) {
  return c.opt.local_precision == NLS_PREC_FP32_IR ? dev::ring_threads<float>(c.ov.max_b)
                                                   : dev::ring_threads<double>(c.ov.max_b);
}

// CTA size of the tangent application: the solving warps and the copying one, and enough threads for
// the matrix products -- 256 while every subdomain has an SM to itself, else 128, three CTAs of which
// share an SM.  (A kernel for 512 threads is held to 128 registers, and a solve step took 1900 cycles
// instead of 750.)
int apply_threads(const Context& c) {
  const int ring = apply_ring_threads(c);
  const int need = std::max(64, std::max(ring <= kApplyMax ? ring : 0, min_local_threads(c)));
  if (c.dev && c.dev->apply_T) return std::max(c.dev->apply_T, need);
  const int nsm = c.dev ? c.dev->nsm : 152;
  return std::max(need, c.ov.count <= nsm ? 256 : 128);
}

bool fp32_local(const Context& c) { return c.opt.local_precision == NLS_PREC_FP32_IR; }
bool fp32_coarse(const Context& c) { return c.opt.coarse_precision == NLS_PREC_FP32_IR; }

// Largest half bandwidth of A_0 the one-CTA band LU takes (its window sits in shared memory) and
// that the coarse band solves take (warp 0 plus one thread per coupled row in a CTA of at most
// 512 threads, which keeps 128 registers per thread for the double-buffered operands).
constexpr int kMaxBandB0 = 128;
constexpr int kMaxSolveB0 = 512 - 32;

bool coarse_tiles(const Context& c) {
  return c.opt.coarse_factor == NLS_COARSE_FACTOR_TILES ||
         (c.opt.coarse_factor == NLS_COARSE_FACTOR_AUTO && c.cs.b0 > kMaxBandB0);
}

// CTA size of the one-CTA coarse band solves: warp 0 plus one thread per coupled row.
int coarse_solve_threads(const Context& c) { return std::max(256, (32 + c.cs.b0 + 31) / 32 * 32); }

dev::NHLaw nh_law(const Context& c) {
  dev::NHLaw law;
  lame(c, law.mu, law.lam);
  law.tab = c.dev->logtab;  // null for Eq. 1, which does not read it
  return law;
}

LocalArgs make_args(const Context& c, const LocalSet& hs, const DeviceLocalSet& ds) {
  LocalArgs A;
  std::memset(&A, 0, sizeof(A));
  Dev& D = *c.dev;
  A.meta = ds.meta;
  A.tnode_gid = ds.tnode_gid;
  A.elem_gid = ds.elem_gid;
  A.lconn = ds.lconn;
  A.color_ptr = ds.color_ptr;
  A.rowptr = ds.rowptr;
  A.colidx = ds.colidx;
  A.epos = ds.epos;
  A.owned = ds.owned;
  A.csr = ds.csr_val;
  A.factor = ds.factor;
  A.dinv = ds.dinv;
  A.wbuf = ds.w;
  A.work = ds.work;
  A.work_stride = hs.total_n;
  A.its = ds.its;
  A.status = ds.status;
  A.chord = ds.chord;
  A.reuse = 0;
  A.order = ds.order;
  A.queue = ds.queue;
  A.geom = D.geom;
  A.kcoef = D.kcoef;
  A.fext = D.fext;
  A.nh = nh_law(c);
  A.load = 1.0;
  A.ndof = c.ndof;
  A.nen = c.nen;
  A.count = hs.count;
  A.max_n = hs.max_n;
  A.max_nt = hs.max_nt;
  A.max_b = hs.max_b;
  A.rtol = c.opt.inner_rtol;
  A.atol = c.opt.inner_atol;
  A.armijo = c.opt.armijo;
  A.ir_rtol = c.opt.ir_rtol;
  A.maxit = c.opt.inner_maxit;
  A.ls_trials = c.opt.ls_trials;
  A.ir_max = c.opt.ir_max_sweeps;
  A.l2_dist = c.opt.l2_prefetch;
  A.err = D.err_dev;
  return A;
}

// Allow the kernel the whole opt-in shared memory minus its static shared memory.
template <typename K>
void set_smem(K kernel, size_t optin) {
  cudaFuncAttributes fa;
  CK(cudaFuncGetAttributes(&fa, kernel));
  const size_t dyn = optin > fa.sharedSizeBytes ? optin - fa.sharedSizeBytes : 0;
  CK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
}

void sync(Dev& D) { CK(cudaStreamSynchronize(D.s)); }

// Elements per thread of the tiled vector kernels: one while the tiles then fill the SMs at most once, four
// beyond.  An iteration's orthogonalisation against 10 vectors (four launches) with 1 / 4 / 16 elements:
// 35 / 44 / 81 us at n = 4,225, 46 / 47 / 84 at 50,000, 100 / 66 / 88 at 296,450, 259 / 152 / 151 at 1,050,625,
// 1902 / 959 / 1136 at 8,396,802; against 40 vectors at the last size 5256 / 3033 / 4377 (sixteen elements
// of w and of the sums leave a thread too few registers for several vectors in flight).
int tile_elems(const Dev& D, int64_t n) { return n <= (int64_t)kTile * D.nsm ? 1 : 4; }
int tile_grid(const Dev& D, int64_t n) {
  const int64_t t = (int64_t)kTile * tile_elems(D, n);
  return (int)std::max<int64_t>(1, (n + t - 1) / t);
}

void dots(Dev& D, int64_t n, int nv, const double* V, int64_t ld, const double* coef, double* w, double* out) {
  const int E = tile_elems(D, n), grid = tile_grid(D, n);
  if (E == 1) LAUNCH_NAMED(D, "k_dots", k_dots<1>, grid, kTile, 0, n, nv, V, ld, coef, w, D.partial, D.ticket, out);
  else LAUNCH_NAMED(D, "k_dots", k_dots<4>, grid, kTile, 0, n, nv, V, ld, coef, w, D.partial, D.ticket, out);
}

// ---- reductions with a host read-back ---------------------------------------------------------
double dot(Dev& D, int64_t n, const double* x, const double* y) {
  dots(D, n, 1, x, (int64_t)0, nullptr, const_cast<double*>(y), D.scal);
  CK(cudaMemcpyAsync(D.h_scal, D.scal, sizeof(double), cudaMemcpyDeviceToHost, D.s));
  sync(D);
  return D.h_scal[0];
}

// A NaN or infinite sum of squares stays non-finite (std::max(0.0, NaN) would give 0: a NaN state
// must never read as converged).
double norm2(Dev& D, int64_t n, const double* x) {
  const double d = dot(D, n, x, x);
  return std::isfinite(d) ? std::sqrt(std::max(0.0, d)) : d;
}

// ---- global residual / Jacobian ------------------------------------------------------------
void global_residual(Context& c, const double* x, double* F, double load) {
  Dev& D = *c.dev;
  const dev::NHLaw nh = nh_law(c);
  if (c.law == NLS_LAW_DIFFUSION)
    LAUNCH(D, k_elem_residual<NLS_LAW_DIFFUSION>, grid_for(c.n_elems), 256, 0, c.n_elems, D.conn, D.geom, D.kcoef, x,
           D.Re, nh, D.bad);
  else
    LAUNCH(D, k_elem_residual<NLS_LAW_NEOHOOKE>, grid_for(c.n_elems), 256, 0, c.n_elems, D.conn, D.geom, D.kcoef, x,
           D.Re, nh, D.bad);
  LAUNCH(D, k_node_residual, grid_for(c.n_nodes), 256, 0, c.n_nodes, c.ndof, D.star_ptr, D.star_ref, D.Re, load,
         D.fext, D.free_dof, F);
}

void global_jacobian(Context& c, const double* x) {
  Dev& D = *c.dev;
  const dev::NHLaw nh = nh_law(c);
  CK(cudaMemsetAsync(D.g_val, 0, sizeof(double) * c.g_col.size(), D.s));
  for (size_t k = 0; k + 1 < c.g_color_ptr.size(); ++k) {
    const int e0 = c.g_color_ptr[k], e1 = c.g_color_ptr[k + 1];
    if (c.law == NLS_LAW_DIFFUSION)
      LAUNCH(D, (k_global_jacobian<NLS_LAW_DIFFUSION>), grid_for(e1 - e0), 256, 0, D.g_elem, e0, e1, D.conn, D.geom,
             D.kcoef, x, D.g_epos, D.g_val, nh);
    else
      LAUNCH(D, (k_global_jacobian<NLS_LAW_NEOHOOKE>), grid_for(e1 - e0), 256, 0, D.g_elem, e0, e1, D.conn, D.geom,
             D.kcoef, x, D.g_epos, D.g_val, nh);
  }
}

// ---- batched local kernels ---------------------------------------------------------------------
template <typename FT>
size_t local_newton_smem(const LocalSet& s) {
  return newton_plan<FT>(s.max_n, s.max_nt, s.max_b).total;
}

// Persistent grid: as many CTAs as fit on the device at once (registers and shared memory), at
// most one per subdomain; the work counter hands out the subdomains.
const char* newton_kernel_name(int law, bool f32, int maxt) {
  static const char* names[8] = {
      "k_local_newton<diffusion, double, 128>", "k_local_newton<diffusion, float, 128>",
      "k_local_newton<diffusion, double, 256>", "k_local_newton<diffusion, float, 256>",
      "k_local_newton<neohooke, double, 128>",  "k_local_newton<neohooke, float, 128>",
      "k_local_newton<neohooke, double, 256>",  "k_local_newton<neohooke, float, 256>"};
  return names[(law == NLS_LAW_DIFFUSION ? 0 : 4) + (maxt > 128 ? 2 : 0) + (f32 ? 1 : 0)];
}

template <int LAW, typename FT, int MAXT>
void launch_newton_t(Dev& D, int count, int T, size_t sm, const LocalArgs& A) {
  int occ = 0;
  CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_local_newton<LAW, FT, MAXT>, T, sm));
  occ = std::max(1, occ);
  // With one CTA per SM a concurrent one-CTA coarse factorization could never share an SM with
  // this persistent grid: leave it one (the CTAs pull subdomains from the work counter, so one
  // fewer CTA only means more subdomains for the others).
  const int spare = (D.coarse_beside && occ == 1 && D.nsm > 1) ? 1 : 0;
  const int grid = std::min(count, (D.nsm - spare) * occ);
  LAUNCH_NAMED(D, newton_kernel_name(LAW, sizeof(FT) == 4, MAXT), (k_local_newton<LAW, FT, MAXT>), grid, T, sm, A);
}

template <int LAW, typename FT>
void launch_newton_law(Dev& D, int count, int T, size_t sm, const LocalArgs& A) {
  if (T <= 128) launch_newton_t<LAW, FT, 128>(D, count, T, sm, A);
  else launch_newton_t<LAW, FT, 256>(D, count, T, sm, A);
}

// CTAs of the batched local Newton kernel resident per SM at the current CTA size.
int newton_ctas_per_sm(Context& c) {
  const int T = local_threads(c);
  const bool f32 = fp32_local(c);
  const size_t sm = f32 ? local_newton_smem<float>(c.ov) : local_newton_smem<double>(c.ov);
  int occ = 0;
  auto q = [&](auto kernel) { CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, T, sm)); };
  const bool big = T > 128;
  if (c.law == NLS_LAW_DIFFUSION) {
    if (f32) big ? q(k_local_newton<NLS_LAW_DIFFUSION, float, 256>) : q(k_local_newton<NLS_LAW_DIFFUSION, float, 128>);
    else big ? q(k_local_newton<NLS_LAW_DIFFUSION, double, 256>) : q(k_local_newton<NLS_LAW_DIFFUSION, double, 128>);
  } else {
    if (f32) big ? q(k_local_newton<NLS_LAW_NEOHOOKE, float, 256>) : q(k_local_newton<NLS_LAW_NEOHOOKE, float, 128>);
    else big ? q(k_local_newton<NLS_LAW_NEOHOOKE, double, 256>) : q(k_local_newton<NLS_LAW_NEOHOOKE, double, 128>);
  }
  return std::max(1, occ);
}

// The tangent's refactorisation goes to k_local_factor when the Newton kernel, at its current
// CTA size, holds one CTA per SM and the factor kernel fits at least two.
bool split_local_factor(Context& c) {
  int occ = 0;
  if (fp32_local(c))
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_local_factor<float, 256>, 256, factor_plan<float>(c.ov.max_b).total));
  else
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_local_factor<double, 256>, 256, factor_plan<double>(c.ov.max_b).total));
  return newton_ctas_per_sm(c) == 1 && occ >= 2;
}

void dispatch_local_newton(Context& c, const LocalSet& s, const LocalArgs& A, int T) {
  Dev& D = *c.dev;
  const bool f32 = fp32_local(c);
  const size_t sm = f32 ? local_newton_smem<float>(s) : local_newton_smem<double>(s);
  if (c.law == NLS_LAW_DIFFUSION) {
    if (f32) launch_newton_law<NLS_LAW_DIFFUSION, float>(D, s.count, T, sm, A);
    else launch_newton_law<NLS_LAW_DIFFUSION, double>(D, s.count, T, sm, A);
  } else {
    if (f32) launch_newton_law<NLS_LAW_NEOHOOKE, float>(D, s.count, T, sm, A);
    else launch_newton_law<NLS_LAW_NEOHOOKE, double>(D, s.count, T, sm, A);
  }
}

void launch_local_newton(Context& c, const double* x, double* out, double load, const GuessProposal& g,
                         bool want_tangent) {
  Dev& D = *c.dev;
  LocalArgs A = make_args(c, c.ov, D.ov);
  A.x = x;
  A.out = out;
  A.load = load;
  A.guess = g.x;
  A.accepted = g.accepted;
  A.guess_diag = g.diag;
  A.guess_sweeps = g.x ? g.sweeps : 0;
  A.guess_omega = g.omega;
  A.want_tangent = want_tangent ? 1 : 0;
  A.split_factor = (want_tangent && split_local_factor(c)) ? 1 : 0;
  A.phase = D.prof ? D.phase : nullptr;
  A.reuse = (D.local_reuse_active && D.local_factors_valid) ? 1 : 0;
  CK(cudaMemsetAsync(D.ov.queue, 0, sizeof(int32_t), D.s));
  dispatch_local_newton(c, c.ov, A, local_threads(c));
  if (A.split_factor) {
    // 512 threads shorten one factorization (1.01 against 1.15 ms at n = 3120, b = 83), three CTAs of
    // 256 threads per SM finish more of them: the larger CTA while every subdomain has an SM
    const bool big = c.ov.count <= D.nsm;
    auto run = [&](auto kernel, const char* name, size_t sm) {
      LAUNCH_NAMED(D, name, kernel, c.ov.count, big ? 512 : 256, sm, A);
    };
    if (fp32_local(c)) {
      const size_t sm = factor_plan<float>(c.ov.max_b).total;
      big ? run(k_local_factor<float, 512>, "k_local_factor<float>", sm)
          : run(k_local_factor<float, 256>, "k_local_factor<float>", sm);
    } else {
      const size_t sm = factor_plan<double>(c.ov.max_b).total;
      big ? run(k_local_factor<double, 512>, "k_local_factor<double>", sm)
          : run(k_local_factor<double, 256>, "k_local_factor<double>", sm);
    }
  }
}

// Stages of the tangent application's operand ring: as many as leave room for the CTAs per SM that the
// subdomains fill (three at most), at least two.  (4096 solves of n = 3120, b = 83 in one launch are
// bound by HBM with three stages at three CTAs per SM or six at one.)
template <typename FT>
int apply_ring_stages(const Context& c) {
  const Dev& D = *c.dev;
  if (apply_ring_threads(c) > kApplyMax) return 0;
  const size_t per_sm = D.smem_optin + 1024, want = std::min(3, (c.ov.count + D.nsm - 1) / D.nsm);
  for (int st = dev::kRingMax; st >= 2; --st) {
    const size_t sm = apply_plan<FT>(c.ov.max_n, c.ov.max_nt, c.ov.max_b, st).total;
    if (sm <= D.smem_optin - 128 && ((sm + 1024) * want <= per_sm || st == 2)) return st;
  }
  return 0;
}

template <typename FT>
void launch_apply_t(Context& c, LocalArgs& A, int T) {
  Dev& D = *c.dev;
  A.ring = apply_ring_stages<FT>(c);
  const size_t sm = apply_plan<FT>(c.ov.max_n, c.ov.max_nt, c.ov.max_b, A.ring).total;
  const char* name = sizeof(FT) == 4 ? "k_local_apply<float>" : "k_local_apply<double>";
  if (T <= 128) LAUNCH_NAMED(D, name, (k_local_apply<FT, 128>), c.ov.count, T, sm, A);
  else LAUNCH_NAMED(D, name, (k_local_apply<FT, 256>), c.ov.count, T, sm, A);
}

void launch_local_apply(Context& c, const double* v, const double* add, double* out) {
  LocalArgs A = make_args(c, c.ov, c.dev->ov);
  A.v = v;
  A.add = add;
  A.out = out;
  if (fp32_local(c)) launch_apply_t<float>(c, A, apply_threads(c));
  else launch_apply_t<double>(c, A, apply_threads(c));
}

// ---- autotuner (nls_options.autotune) -------------------------------------------------------
// Candidates are timed with CUDA events on the context's own data and the fastest is kept for
// the life of the context.  Every candidate computes the same quantities (only the order of
// the reductions inside a subdomain differs), so the timed launches double as warm-up.
template <typename F>
float time_on_stream(Dev& D, F&& f) {
  cudaEvent_t a, b;
  CK(cudaEventCreate(&a));
  CK(cudaEventCreate(&b));
  CK(cudaEventRecord(a, D.s));
  f();
  CK(cudaEventRecord(b, D.s));
  CK(cudaEventSynchronize(b));
  float ms = 0.f;
  CK(cudaEventElapsedTime(&ms, a, b));
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  return ms;
}

void tune_local_newton(Context& c, const double* x, double* out, double load, const GuessProposal& guess) {
  Dev& D = *c.dev;
  if (D.newton_tuned || !c.opt.autotune || c.opt.threads_per_block) return;
  const int need = min_local_threads(c);
  const int cand[2] = {128, 256};
  // warm-up with the fixed choice (first touch of the factor storage and the caches)
  launch_local_newton(c, x, out, load, guess, true);
  double best = INFINITY;
  int bestT = 0;
  for (int i = 0; i < 2; ++i) {
    if (cand[i] < need) continue;
    D.newton_T = cand[i];
    const float ms = time_on_stream(D, [&] { launch_local_newton(c, x, out, load, guess, true); });
    D.newton_ms[i] = ms;
    if (ms < best) {
      best = ms;
      bestT = cand[i];
    }
  }
  D.newton_T = bestT;
  D.newton_tuned = true;
}

void tune_local_apply(Context& c, const double* v, double* out) {
  Dev& D = *c.dev;
  if (D.apply_tuned || !c.opt.autotune) return;
  D.apply_T = 32;  // the smallest CTA that the kernel takes
  const int need = apply_threads(c);
  std::vector<int> cand;
  for (int T : {need, need + 32, need + 64, 128, 192, 256})
    if (T >= need && T <= 256 && std::find(cand.begin(), cand.end(), T) == cand.end()) cand.push_back(T);
  D.apply_T = need;
  launch_local_apply(c, v, nullptr, out);  // warm-up
  double best = INFINITY;
  int bestT = need;
  for (int T : cand) {
    D.apply_T = T;
    float ms = INFINITY;
    for (int rep = 0; rep < 2; ++rep)
      ms = std::min(ms, time_on_stream(D, [&] { launch_local_apply(c, v, nullptr, out); }));
    if (ms < best) {
      best = ms;
      bestT = T;
    }
  }
  D.apply_T = bestT;
  D.apply_tuned = true;
}

// ---- coarse ---------------------------------------------------------------------------------
LocalArgs coarse_args(Context& c) {
  Dev& D = *c.dev;
  LocalArgs A = make_args(c, c.nov, D.nov);
  A.phi = D.phi;
  A.phi_off = D.phi_off;
  A.cj_ptr = D.cj_ptr;
  A.Y = D.Y;
  A.blk = D.blk;
  A.blk_off = D.blk_off;
  return A;
}

// Shared memory of the one-CTA band factorization; never less than the window of (b + 10) band
// rows that the limit on its half bandwidth is stated for.
size_t coarse_factor_smem(const Context& c, bool f32) {
  const size_t fs = f32 ? sizeof(float) : sizeof(double);
  const size_t BS = f32 ? dev::SolveBlock<float>::BS : dev::SolveBlock<double>::BS;
  const size_t R = (size_t)dev::band_limit_rows(c.cs.b0);
  const size_t lim = fs * (R * dev::band_limit_stride(c.cs.b0) + R + 4 * BS * (BS + 1)) + 16;
  const size_t need = align_up(fs * (f32 ? coarse_window<float>(c.cs.b0) : coarse_window<double>(c.cs.b0)), 16) + 16;
  return std::max(lim, need);
}

// A_0(x) = P_0^T DF(x) P_0 -> band -> factor.  Returns false on a bad pivot.
void coarse_matrix_launch(Context& c, const double* x);
void coarse_inverse_launch(Context& c);

// Raises DeviceTimeout if a local triangular solve has given up waiting since the last check (its
// stream synchronised by the caller).
void check_local_waits(Dev& D) {
  volatile int* e = D.err_host;
  if (!*e) return;
  *e = 0;
  throw DeviceTimeout("a triangular solve gave up waiting for its operands");
}

// Ends a call that failed: its work is awaited and what its waits reported is dropped, so that it is not
// taken for a later call's.
void forget_waits(Dev& D) {
  if (D.tlu && D.tlu->solve_status) cudaMemsetAsync(D.tlu->solve_status, 0, sizeof(int32_t), D.s);
  cudaStreamSynchronize(D.s);
  if (D.s2) cudaStreamSynchronize(D.s2);
  if (D.err_host) *(volatile int*)D.err_host = 0;
}

// Reads the coarse factorization's status word (synchronises the stream).
bool coarse_status_ok(Dev& D) {
  int32_t st = 0;
  CK(cudaMemcpyAsync(&st, D.cstatus, sizeof(int32_t), cudaMemcpyDeviceToHost, D.s));
  sync(D);
  if (st == ST_TIMEOUT) throw DeviceTimeout("a tile of the coarse factorization gave up waiting for its operands");
  return st == ST_OK;
}
// The same, after checking that no coarse cluster solve gave up waiting.
bool coarse_status_ok(Context& c) {
  tlu_check_solves(c);
  return coarse_status_ok(*c.dev);
}

bool coarse_matrix(Context& c, const double* x) {
  coarse_matrix_launch(c, x);
  return coarse_status_ok(c);
}

// A_0(x) = P_0^T DF(x) P_0 in band storage (D.A0): Galerkin blocks per non-overlapping subdomain
// and their gather.
void coarse_assemble_launch(Context& c, const double* x) {
  Dev& D = *c.dev;
  LocalArgs A = coarse_args(c);
  A.x = x;
  const int T = 256;
  A.gal_rows = galerkin_rows(D.smem_optin, c.cs.max_nc);
  const size_t sm = galerkin_smem(D.smem_optin, c.nov.max_nt, c.cs.max_nc);
  if (c.law == NLS_LAW_DIFFUSION) LAUNCH(D, (k_galerkin<NLS_LAW_DIFFUSION>), c.nov.count, T, sm, A);
  else LAUNCH(D, (k_galerkin<NLS_LAW_NEOHOOKE>), c.nov.count, T, sm, A);
  const int64_t ne = (int64_t)c.cs.N0 * (2 * c.cs.b0 + 1);
  LAUNCH(D, k_a0_gather, grid_for(ne), 256, 0, ne, D.a0_ptr, D.a0_src, D.blk, D.A0);
}

// Band factorization of D.A0 (one CTA; its size autotuned at the first call) into the packed
// solve operands; the status word is read by coarse_status_ok.
void coarse_factor_launch(Context& c) {
  Dev& D = *c.dev;
  if (D.tlu) {
    tlu_factor(c);
    return;
  }
  const bool f32 = fp32_coarse(c);
  const size_t fsm = coarse_factor_smem(c, f32);
  auto factor = [&](int T) {
    if (f32)
      LAUNCH(D, k_coarse_factor<float>, 1, T, fsm, c.cs.N0, c.cs.b0, D.A0, (float*)D.A0f, (float*)D.A0dinv,
             D.cstatus);
    else
      LAUNCH(D, k_coarse_factor<double>, 1, T, fsm, c.cs.N0, c.cs.b0, D.A0, (double*)D.A0f, (double*)D.A0dinv,
             D.cstatus);
  };
  if (c.opt.autotune && !D.coarse_tuned) {
    // the factorization reads A_0 and overwrites its own outputs: every candidate is a full,
    // valid factorization; the fastest CTA size is kept
    double best = INFINITY;
    int bestT = 1024;
    for (int T : {256, 512, 1024}) {
      const float ms = time_on_stream(D, [&] { factor(T); });
      if (ms < best) {
        best = ms;
        bestT = T;
      }
    }
    D.coarse_T = bestT;
    D.coarse_tuned = true;
  }
  factor(D.coarse_T);
}

void coarse_matrix_launch(Context& c, const double* x) {
  coarse_assemble_launch(c, x);
  coarse_factor_launch(c);
}

void coarse_solve(Context& c, const double* g, double* z) {
  Dev& D = *c.dev;
  if (D.ainv_valid) {
    // z = A_0^-1 g, then (FP32 inverse) up to min(ir_max_sweeps, 3) refinement steps
    // z += A_0^-1 (g - A_0 z) until ||g - A_0 z|| <= ir_rtol ||g||: a fixed sequence of launches
    // (graph-capturable) whose steps after convergence return at once
    const int N0 = c.cs.N0;
    const dim3 gg((N0 + 31) / 32, kGemvChunks);
    const bool f32 = fp32_coarse(c);
    auto apply_inverse = [&](const double* rhs, int accumulate, const int* skip, int* reset) {
      if (f32)
        LAUNCH(D, k_dense_gemv_t<float>, gg, 256, 0, N0, (const float*)D.ainv, rhs, D.gpart, D.gticket, z, accumulate,
               skip, reset);
      else
        LAUNCH(D, k_dense_gemv_t<double>, gg, 256, 0, N0, (const double*)D.ainv, rhs, D.gpart, D.gticket, z, accumulate,
               skip, reset);
    };
    apply_inverse(g, 0, nullptr, D.cflag);
    const int sweeps = f32 ? std::min(c.opt.ir_max_sweeps, 3) : 0;
    for (int sw = 0; sw < sweeps; ++sw) {
      LAUNCH(D, k_coarse_residual, (N0 + 7) / 8, 256, 0, N0, c.cs.b0, D.A0, g, z, D.cres, D.cpart,
             (unsigned*)(D.cflag + 1), D.cflag, c.opt.ir_rtol);
      apply_inverse(D.cres, 1, D.cflag, nullptr);
    }
    return;
  }
  // band factors: one solve in one CTA, then (FP32 factors) up to ir_max_sweeps refinement steps
  // z += A_0^-1 (g - A_0 z) with the FP64 residual on every SM; the same fixed launch sequence
  // as above, the steps after convergence returning at once
  const int N0 = c.cs.N0;
  const bool f32 = fp32_coarse(c);
  const int b0 = c.cs.b0;
  const int T = std::max(coarse_solve_threads(c), std::min(512, f32 ? dev::ring_threads<float>(b0) : dev::ring_threads<double>(b0)));
  // the operand ring behind the solve vector, where two stages of it fit (15 against 18 us per solve at
  // N_0 = 699, b_0 = 77)
  auto ring = [&](size_t vec, size_t stage, int threads) {
    const size_t room = D.smem_optin - 128;
    if (T < threads || vec + dev::kRingHead + 2 * stage > room) return 0;
    return (int)std::min<size_t>(dev::kRingMax, (room - vec - dev::kRingHead) / stage);
  };
  auto band_solve = [&](const double* rhs, int accumulate, const int* skip, int* reset) {
    if (tlu_solve(c, rhs, z, accumulate, skip, reset)) return;  // tiled factors: the cluster solve
    if (f32) {
      const size_t vec = coarse_solve_vector<float>(N0), stage = dev::ring_stage_bytes<float>(b0);
      const int st = ring(vec, stage, dev::ring_threads<float>(b0));
      LAUNCH(D, k_coarse_band_solve<float>, 1, T, st ? vec + dev::kRingHead + st * stage : sizeof(float) * N0, N0, b0,
             (const float*)D.A0dinv, rhs, z, accumulate, skip, reset, c.opt.l2_prefetch, st, D.err_dev);
    } else {
      const size_t vec = coarse_solve_vector<double>(N0), stage = dev::ring_stage_bytes<double>(b0);
      const int st = ring(vec, stage, dev::ring_threads<double>(b0));
      LAUNCH(D, k_coarse_band_solve<double>, 1, T, st ? vec + dev::kRingHead + st * stage : sizeof(double) * N0, N0, b0,
             (const double*)D.A0dinv, rhs, z, accumulate, skip, reset, c.opt.l2_prefetch, st, D.err_dev);
    }
  };
  band_solve(g, 0, nullptr, D.cflag);
  const int sweeps = f32 ? c.opt.ir_max_sweeps : 0;
  for (int sw = 0; sw < sweeps; ++sw) {
    LAUNCH(D, k_coarse_residual, (N0 + 7) / 8, 256, 0, N0, c.cs.b0, D.A0, g, z, D.cres, D.cpart,
           (unsigned*)(D.cflag + 1), D.cflag, c.opt.ir_rtol);
    band_solve(D.cres, 1, D.cflag, nullptr);
  }
}

// x = u - P0 c
void p0_update(Context& c, const double* u, const double* cv, double* x) {
  Dev& D = *c.dev;
  LAUNCH(D, k_p0_apply, grid_for(c.N), 256, 0, c.N, D.p0_slice, D.p0_col, D.p0_val, cv, 1.0, u, -1.0, x,
         (double*)nullptr);
}

void p0t(Context& c, const double* v, double* g) {
  Dev& D = *c.dev;
  LAUNCH(D, k_p0t_apply, c.cs.N0, 256, 0, c.cs.N0, D.p0t_rowptr, D.p0t_col, D.p0t_val, v, g);
}

struct CoarseResult {
  int its = 0;
  int status = ST_OK;
};

// Coarse Newton for Eq. 9: g(c) = P0^T F(u - P0 c) = 0, c <- c + alpha A0^-1 g.  Leaves
// D.c = T_0(u) and D.u0 = u - P0 T_0(u).
CoarseResult coarse_newton(Context& c, const double* u, double load) {
  Dev& D = *c.dev;
  CoarseResult R;
  const int N0 = c.cs.N0;
  CK(cudaMemsetAsync(D.c, 0, sizeof(double) * N0, D.s));
  CK(cudaMemcpyAsync(D.u0, u, sizeof(double) * c.N, cudaMemcpyDeviceToDevice, D.s));
  global_residual(c, D.u0, D.F, load);
  p0t(c, D.F, D.g);
  double gn = norm2(D, N0, D.g);
  if (!std::isfinite(gn)) {
    R.status = ST_NONFINITE;
    return R;
  }
  const double tol = std::max(c.opt.inner_atol, c.opt.inner_rtol * gn);
  // With coarse_reuse the iteration starts from the factorization of the previous tangent
  // phase's A_0 (chord steps, solved with its explicit inverse) and forms A_0 at the current
  // point only when a step contracts ||g|| by less than half or fails the line search; the
  // stopping test is the same either way.
  bool refresh = !(c.opt.coarse_reuse && D.coarse_fact_valid);
  while (gn > tol) {
    if (R.its >= c.opt.inner_maxit) {
      R.status = ST_MAXIT;
      break;
    }
    const bool chord = !refresh;
    if (!chord) {
      D.ainv_valid = false;  // the explicit inverse belongs to an older A_0
      D.coarse_fact_valid = coarse_matrix(c, D.u0);
      if (!D.coarse_fact_valid) {
        R.status = ST_PIVOT;
        break;
      }
      // the explicit inverse costs about a third of one band solve, and every solve with it
      // (GEMV + FP64 refinement) a tenth
      if (D.ainv) {
        coarse_inverse_launch(c);
        D.ainv_valid = true;
      }
    }
    coarse_solve(c, D.g, D.dc);
    double alpha = 1.0, gtn = INFINITY;
    bool accepted = false;
    for (int trial = 0; trial < c.opt.ls_trials; ++trial) {
      LAUNCH(D, k_axpby, grid_for(N0), 256, 0, (int64_t)N0, 1.0, D.c, alpha, D.dc, D.ct);
      p0_update(c, u, D.ct, D.x);
      global_residual(c, D.x, D.F, load);
      p0t(c, D.F, D.gt);
      gtn = norm2(D, N0, D.gt);
      if (std::isfinite(gtn) && gtn <= (1.0 - c.opt.armijo * alpha) * gn) {
        accepted = true;
        break;
      }
      alpha *= 0.5;
    }
    if (!accepted && chord) {
      refresh = true;  // retry the step with A_0 at the current point
      continue;
    }
    R.its += 1;
    if (!accepted) {
      R.status = ST_LS;
      break;
    }
    refresh = !c.opt.coarse_reuse || gtn > 0.5 * gn;
    std::swap(D.c, D.ct);
    std::swap(D.u0, D.x);
    std::swap(D.g, D.gt);
    gn = gtn;
  }
  return R;
}

}  // namespace

// ------------------------------------------------------------------------------------------
// setup on the device
// ------------------------------------------------------------------------------------------
namespace {

// The flags that a kernel whose bounded wait gave up sets (host memory, mapped): [0] is read at the end of
// the call that launched it; [1] takes those of the allocation-free corrections, which report it in the
// subdomains' status words and return before their work is done.
void alloc_err(Dev& D) {
  CK(cudaHostAlloc(&D.err_host, 2 * sizeof(int), cudaHostAllocMapped));
  D.err_host[0] = D.err_host[1] = 0;
  CK(cudaHostGetDevicePointer((void**)&D.err_dev, D.err_host, 0));
}

void upload_set(Dev& D, const LocalSet& h, DeviceLocalSet& d, bool fp32_factor, bool with_dinv = true) {
  d.count = h.count;
  d.meta = D.upload(h.meta);
  d.tnode_gid = D.upload(h.tnode_gid);
  d.elem_gid = D.upload(h.elem_gid);
  d.lconn = D.upload(h.lconn);
  d.color_ptr = D.upload(h.color_ptr);
  d.rowptr = D.upload(h.rowptr);
  d.colidx = D.upload(h.colidx);
  d.epos = D.upload(h.epos);
  d.owned = D.upload(h.owned);
  d.csr_val = D.alloc<double>(h.total_nnz);
  if (fp32_factor) {
    d.factor = D.alloc<float>(h.total_factor);
    if (with_dinv) d.dinv = D.alloc<float>(h.total_dinv);
  } else {
    d.factor = D.alloc<double>(h.total_factor);
    if (with_dinv) d.dinv = D.alloc<double>(h.total_dinv);
  }
  d.w = D.alloc<double>(h.total_n);
  d.work = D.alloc<double>(2 * (size_t)h.total_n);
  d.its = D.alloc<int32_t>(h.count);
  d.chord = D.alloc<int32_t>(h.count);
  d.status = D.alloc<int32_t>(h.count);
  // longest first: cost ~ n b^2
  std::vector<int32_t> order(h.count);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    const double ca = (double)h.meta[a].n * h.meta[a].b * h.meta[a].b, cb = (double)h.meta[b].n * h.meta[b].b * h.meta[b].b;
    return ca > cb;
  });
  d.order = D.upload(order);
  d.queue = D.alloc<int32_t>(1);
}

}  // namespace

// Energy-minimising extension of the interface values of the coarse basis (RGDSW, Section 2)
// with K = DF(u^(0)), u^(0) = Dirichlet data and zero elsewhere, then the values of P_0 and
// P_0^T.  The factors of the non-overlapping problems are needed for the extension only.
// RGDSW coarse basis: the interface values (host) extended into every non-overlapping
// subdomain by the energy-minimising (harmonic) extension with DF(x) (k_harmonic), then P_0 and
// P_0^T gathered.  x = nullptr: the Dirichlet data u^(0) (the basis built once, at setup);
// otherwise the current outer iterate (coarse_rebuild).
void coarse_extension(Context& c, const double* x = nullptr) {
  Dev& D = *c.dev;
  Coarse& cs = c.cs;
  const int64_t N = c.N;
  const size_t lim = D.smem_optin;
  auto need = [&](size_t b, const char* what) {
    if (b > lim) throw std::runtime_error(std::string(what) + " needs more shared memory than the device offers");
  };
  if (!D.nov.factor) D.nov.factor = D.alloc<double>(c.nov.total_factor);
  CK(cudaMemcpyAsync(D.phi, cs.phi_host.data(), sizeof(double) * cs.phi_host.size(), cudaMemcpyHostToDevice, D.s));
  CK(cudaMemcpyAsync(D.x, x ? x : D.ubc, sizeof(double) * N, cudaMemcpyDeviceToDevice, D.s));
  LocalArgs A = coarse_args(c);
  A.x = D.x;
  const size_t sm = harmonic_plan(c.nov.max_n, c.nov.max_nt, c.nov.max_b).total;
  need(sm, "coarse harmonic extension");
  if (c.law == NLS_LAW_DIFFUSION) LAUNCH(D, k_harmonic<NLS_LAW_DIFFUSION>, c.nov.count, 256, sm, A);
  else LAUNCH(D, k_harmonic<NLS_LAW_NEOHOOKE>, c.nov.count, 256, sm, A);
  std::vector<int32_t> st(c.nov.count);
  CK(cudaMemcpyAsync(st.data(), D.nov.status, sizeof(int32_t) * st.size(), cudaMemcpyDeviceToHost, D.s));
  sync(D);
  for (int32_t s : st)
    if (s != ST_OK) throw std::runtime_error("coarse harmonic extension hit a zero pivot");
  const int64_t np = (int64_t)cs.p0_col.size(), nt = (int64_t)cs.p0t_col.size();
  LAUNCH(D, k_gather_values, grid_for(np), 256, 0, np, D.p0_src, D.phi, D.p0_val);
  LAUNCH(D, k_gather_values32, grid_for(nt), 256, 0, nt, D.p0t_src, D.p0_val, D.p0t_val);
  if (!c.opt.coarse_rebuild) {  // rebuilt every outer iteration otherwise: keep the factor storage
    D.release(D.nov.factor);
    D.nov.factor = nullptr;
  }
}

int device_setup(Context& c) {
  try {
    CK(cudaSetDevice(c.device));
    Dev* Dp = new Dev();
    c.dev = Dp;
    Dev& D = *Dp;
    // NULL selects the legacy default stream, which orders against every blocking stream of
    // the caller (a torch tensor filled on the default stream is complete before we read it).
    D.s = (cudaStream_t)c.stream;
    c.own_stream = false;
    cudaDeviceProp prop;
    CK(cudaGetDeviceProperties(&prop, c.device));
    D.nsm = prop.multiProcessorCount;
    D.smem_optin = prop.sharedMemPerBlockOptin;
    D.conn = D.upload(c.conn);
    D.geom = D.upload(c.geom);
    if (c.law == NLS_LAW_NEOHOOKE) D.logtab = D.upload(dev::log_table());
    std::vector<double> k = c.k_elem;
    if (k.empty()) k.assign(c.n_elems, 1.0);
    D.kcoef = D.upload(k);
    D.fext = D.upload(c.fext);
    D.ubc = D.upload(c.ubc);
    D.free_dof = D.upload(c.free_dof);
    D.g_elem = D.upload(c.g_elem);
    {
      // node stars as element-local references (e nen + a), ascending element ids
      std::vector<int32_t> ref(c.star_el.size());
      for (int64_t v = 0; v < c.n_nodes; ++v)
        for (int64_t k = c.star_ptr[v]; k < c.star_ptr[v + 1]; ++k) {
          const int32_t e = c.star_el[k];
          int a = 0;
          while (a < c.nen - 1 && c.conn[(int64_t)e * c.nen + a] != v) ++a;
          ref[k] = e * c.nen + a;
        }
      D.star_ptr = D.upload(c.star_ptr);
      D.star_ref = D.upload(ref);
      D.Re = D.alloc<double>((size_t)c.n_elems * c.nen * c.ndof);
    }
    D.g_slice = D.upload(c.g_slice);
    D.g_col = D.upload(c.g_col);
    D.g_epos = D.upload(c.g_epos);
    D.g_val = D.alloc<double>(c.g_col.size());
    upload_set(D, c.ov, D.ov, fp32_local(c));
    const int N = (int)c.N;
    D.u = D.alloc<double>(N);
    D.ut = D.alloc<double>(N);
    D.x = D.alloc<double>(N);
    D.u0 = D.alloc<double>(N);
    D.Fx = D.alloc<double>(N);
    D.F = D.alloc<double>(N);
    D.t1 = D.alloc<double>(N);
    D.t2 = D.alloc<double>(N);
    D.w0 = D.alloc<double>(N);
    D.gx = D.alloc<double>(N);
    D.m = std::max(1, std::min(c.opt.gmres_restart, kMaxGmresVecs / 2 - 2));
    D.V = D.alloc<double>((size_t)(D.m + 1) * N);
    CK(cudaMemsetAsync(D.V, 0, sizeof(double) * (size_t)(D.m + 1) * N, D.s));
    D.partial = D.alloc<double>((size_t)tile_grid(D, N) * (D.m + 2) + 1024);
    D.ticket = D.alloc<unsigned>(1);
    CK(cudaMemsetAsync(D.ticket, 0, sizeof(unsigned), D.s));
    D.scal = D.alloc<double>(kMaxGmresVecs + 8);
    D.coef = D.alloc<double>(kMaxGmresVecs + 8);
    D.gR = D.alloc<double>((size_t)D.m * D.m);
    D.gcs = D.alloc<double>(D.m);
    D.gsn = D.alloc<double>(D.m);
    D.gg = D.alloc<double>(D.m + 1);
    D.gst = (GmresState*)D.alloc<double>(4);
    D.bad = D.alloc<int>(4);
    D.phase = D.alloc<unsigned long long>(8);
    CK(cudaMemsetAsync(D.phase, 0, sizeof(unsigned long long) * 8, D.s));
    CK(cudaDeviceGetAttribute(&D.clock_khz, cudaDevAttrClockRate, c.device));
    CK(cudaMallocHost(&D.h_scal, sizeof(double) * (kMaxGmresVecs + 8)));
    alloc_err(D);
    // kernel attributes for large dynamic shared memory
    const size_t lim = D.smem_optin;
    auto need = [&](size_t b, const char* what) {
      if (b > lim) throw std::runtime_error(std::string(what) + " needs more shared memory than the device offers");
    };
    if (c.ov.max_b > 128)
      throw std::runtime_error("a local band matrix has a half bandwidth above 128 (" + std::to_string(c.ov.max_b) +
                               "); the local band factorisation supports 128");
    if (c.coarse_kind == NLS_COARSE_RGDSW && !coarse_tiles(c) && c.cs.b0 > kMaxBandB0)
      throw std::runtime_error("the coarse matrix has a half bandwidth of " + std::to_string(c.cs.b0) +
                               "; the one-CTA band factorisation supports " + std::to_string(kMaxBandB0) +
                               " (the tiled one, coarse_factor = NLS_COARSE_FACTOR_TILES, up to " +
                               std::to_string(kMaxSolveB0) + ")");
    if (c.coarse_kind == NLS_COARSE_RGDSW && c.cs.b0 > kMaxSolveB0)
      throw std::runtime_error("the coarse matrix has a half bandwidth of " + std::to_string(c.cs.b0) +
                               "; the coarse solves support " + std::to_string(kMaxSolveB0));
    need(local_newton_smem<float>(c.ov), "local Newton (FP32 factors)");
    if (!fp32_local(c)) need(local_newton_smem<double>(c.ov), "local Newton (FP64 factors)");
    set_smem(k_local_newton<NLS_LAW_DIFFUSION, float, 128>, lim);
    set_smem(k_local_newton<NLS_LAW_DIFFUSION, double, 128>, lim);
    set_smem(k_local_newton<NLS_LAW_NEOHOOKE, float, 128>, lim);
    set_smem(k_local_newton<NLS_LAW_NEOHOOKE, double, 128>, lim);
    set_smem(k_local_newton<NLS_LAW_DIFFUSION, float, 256>, lim);
    set_smem(k_local_newton<NLS_LAW_DIFFUSION, double, 256>, lim);
    set_smem(k_local_newton<NLS_LAW_NEOHOOKE, float, 256>, lim);
    set_smem(k_local_newton<NLS_LAW_NEOHOOKE, double, 256>, lim);
    set_smem(k_local_apply<float, 128>, lim);
    set_smem(k_local_apply<float, 256>, lim);
    set_smem(k_local_apply<double, 128>, lim);
    set_smem(k_local_apply<double, 256>, lim);
    set_smem(k_local_factor<float, 256>, lim);
    set_smem(k_local_factor<double, 256>, lim);
    set_smem(k_local_factor<float, 512>, lim);
    set_smem(k_local_factor<double, 512>, lim);
    set_smem(k_guess_smooth<NLS_LAW_DIFFUSION>, lim);
    set_smem(k_guess_smooth<NLS_LAW_NEOHOOKE>, lim);
    set_smem(k_harmonic<NLS_LAW_DIFFUSION>, lim);
    set_smem(k_harmonic<NLS_LAW_NEOHOOKE>, lim);
    set_smem(k_galerkin<NLS_LAW_DIFFUSION>, lim);
    set_smem(k_galerkin<NLS_LAW_NEOHOOKE>, lim);
    set_smem(k_coarse_factor<float>, lim);
    set_smem(k_coarse_factor<double>, lim);
    if (c.coarse_kind == NLS_COARSE_RGDSW) {
      Coarse& cs = c.cs;
      if (cs.N0 == 0) throw std::runtime_error("the partition has no coarse nodes (one subdomain?)");
      if (!coarse_tiles(c)) need(coarse_factor_smem(c, fp32_coarse(c)), "coarse band factorization");
      need(galerkin_smem(lim, c.nov.max_nt, cs.max_nc), "coarse blocks");
      need((fp32_coarse(c) ? sizeof(float) : sizeof(double)) * (size_t)cs.N0, "coarse band solve");
      upload_set(D, c.nov, D.nov, false, false);
      D.phi = D.upload(cs.phi_host);
      D.phi_off = D.upload(cs.phi_off);
      D.cj_ptr = D.upload(cs.cj_ptr);
      D.Y = D.alloc<double>(cs.phi_total);
      D.blk = D.alloc<double>(cs.blk_total);
      D.blk_off = D.upload(cs.blk_off);
      D.a0_ptr = D.upload(cs.a0_ptr);
      D.a0_src = D.upload(cs.a0_src);
      D.A0 = D.alloc<double>((size_t)cs.N0 * (2 * cs.b0 + 1));
      const size_t ndinv = (size_t)packed_solve_entries(cs.N0, cs.b0);
      if (fp32_coarse(c)) {
        D.A0f = D.alloc<float>((size_t)cs.N0 * (2 * cs.b0 + 1));
        D.A0dinv = D.alloc<float>(ndinv);
      } else {
        D.A0f = D.alloc<double>((size_t)cs.N0 * (2 * cs.b0 + 1));
        D.A0dinv = D.alloc<double>(ndinv);
      }
      D.cstatus = D.alloc<int32_t>(1);
      // refinement of the coarse solves: per-CTA partial norms, converged flag and ticket counter
      D.cpart = D.alloc<double>(2 * (size_t)((cs.N0 + 7) / 8));
      D.cflag = D.alloc<int>(2);
      CK(cudaMemsetAsync(D.cflag, 0, 2 * sizeof(int), D.s));
      set_smem(k_coarse_band_solve<float>, lim);
      set_smem(k_coarse_band_solve<double>, lim);
      if (coarse_tiles(c)) tlu_prepare(c, fp32_coarse(c));
      if (cs.N0 <= kMaxInverseN0) {
        if (fp32_coarse(c)) D.ainv = D.alloc<float>((size_t)cs.N0 * cs.N0);
        else D.ainv = D.alloc<double>((size_t)cs.N0 * cs.N0);
        D.gpart = D.alloc<double>((size_t)cs.N0 * kGemvChunks);
        D.gticket = D.alloc<unsigned>((cs.N0 + 31) / 32);
        CK(cudaMemsetAsync(D.gticket, 0, (cs.N0 + 31) / 32 * sizeof(unsigned), D.s));
        set_smem(k_coarse_inverse<float>, lim);
        set_smem(k_coarse_inverse<double>, lim);
        set_smem(k_coarse_inverse_blocks<float>, lim);
        set_smem(k_coarse_inverse_blocks<double>, lim);
      }
      D.p0_slice = D.upload(cs.p0_slice);
      D.p0_col = D.upload(cs.p0_col);
      D.p0_src = D.upload(cs.p0_src);
      D.p0_val = D.alloc<double>(cs.p0_col.size());
      D.p0t_rowptr = D.upload(cs.p0t_rowptr);
      D.p0t_col = D.upload(cs.p0t_col);
      D.p0t_src = D.upload(cs.p0t_src);
      D.p0t_val = D.alloc<double>(cs.p0t_col.size());
      D.c = D.alloc<double>(cs.N0);
      D.ct = D.alloc<double>(cs.N0);
      D.dc = D.alloc<double>(cs.N0);
      D.g = D.alloc<double>(cs.N0);
      D.gt = D.alloc<double>(cs.N0);
      D.tg = D.alloc<double>(cs.N0);  // the tangent's coarse right-hand side (never swapped)
      D.cres = D.alloc<double>(cs.N0);
      coarse_extension(c);
    }
    sync(D);
    c.device_bytes = D.bytes;
  } catch (const DeviceTimeout& ex) {
    c.last_error = ex.what();
    return NLS_E_DEVICE_TIMEOUT;
  } catch (const CudaFailure& ex) {
    c.last_error = ex.what();
    return NLS_E_CUDA;
  } catch (const std::bad_alloc&) {
    c.last_error = "host allocation failed";
    return NLS_E_NOMEM;
  } catch (const std::exception& ex) {
    c.last_error = ex.what();
    return NLS_E_ARG;
  }
  return NLS_OK;
}

int device_set_coefficients(Context& c) {
  try {
    Dev& D = *c.dev;
    CK(cudaSetDevice(c.device));
    std::vector<double> k = c.k_elem;
    if (k.empty()) k.assign(c.n_elems, 1.0);
    CK(cudaMemcpyAsync(D.kcoef, k.data(), sizeof(double) * k.size(), cudaMemcpyHostToDevice, D.s));
    CK(cudaMemcpyAsync(D.fext, c.fext.data(), sizeof(double) * c.fext.size(), cudaMemcpyHostToDevice, D.s));
    if (c.coarse_kind == NLS_COARSE_RGDSW) coarse_extension(c);
    D.coarse_fact_valid = false;
    D.ainv_valid = false;
    D.tangent_ready = false;
    guess_coefficients_changed(c);
    sync(D);
  } catch (const CudaFailure& ex) {
    c.last_error = ex.what();
    return NLS_E_CUDA;
  } catch (const std::exception& ex) {
    c.last_error = ex.what();
    return NLS_E_ARG;
  }
  return NLS_OK;
}

int device_upload_fext(Context& c) {
  try {
    Dev& D = *c.dev;
    CK(cudaSetDevice(c.device));
    CK(cudaMemcpyAsync(D.fext, c.fext.data(), sizeof(double) * c.fext.size(), cudaMemcpyHostToDevice, D.s));
    sync(D);
  } catch (const CudaFailure& ex) {
    c.last_error = ex.what();
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

void device_free(Context& c) {
  if (!c.dev) return;
  Dev& D = *c.dev;
  cudaSetDevice(c.device);
  if (D.s) cudaStreamSynchronize(D.s);
  guess_free(c);
  tlu_free(c);
  D.reset_graphs();
  if (D.cap) cudaStreamDestroy(D.cap);
  if (D.s2) cudaStreamSynchronize(D.s2), cudaStreamDestroy(D.s2);
  if (D.ev_u0) cudaEventDestroy(D.ev_u0);
  if (D.ev_coarse) cudaEventDestroy(D.ev_coarse);
  for (void* p : D.allocs)
    if (p) cudaFree(p);
  if (D.h_scal) cudaFreeHost(D.h_scal);
  if (D.err_host) cudaFreeHost(D.err_host);
  for (auto& r : D.evs) {
    cudaEventDestroy(r.a);
    cudaEventDestroy(r.b);
  }
  if (c.own_stream && D.s) cudaStreamDestroy(D.s);
  c.own_stream = false;
  delete c.dev;
  c.dev = nullptr;
}

// ------------------------------------------------------------------------------------------
// F_x, tangent, GMRES, outer Newton
// ------------------------------------------------------------------------------------------
namespace {

struct FxInfo {
  int coarse_its = 0;
  int coarse_status = ST_OK;
  int64_t local_its = 0;
  int64_t local_chord = 0;
  int local_failures = 0;
  int first_failed = -1;
  bool pivot_failure = false;
};

// Explicit A_0^-1 from the current coarse factors (N0 <= kMaxInverseN0), issued on D.s; coarse solves use
// it (refined in FP64 against A_0 where it is applied) once ainv_valid is set.
void coarse_inverse_launch(Context& c) {
  Dev& D = *c.dev;
  if (!D.ainv) return;
  const int N0 = c.cs.N0;
  const int b0 = c.cs.b0;
  // one CTA per column while that is bound by the latency of a column's steps: up to kInverseColumns
  // columns and the half bandwidth of a 256-thread CTA, then 32 columns per CTA, which read the operands 32
  // times less often
  auto run = [&](auto columns, auto blocks, const char* name, int threads, size_t vec, size_t stage, size_t two,
                 size_t one, auto* Dinv, auto* Ainv) {
    const size_t ring = vec + dev::kRingHead + 3 * stage;
    if (N0 <= kInverseColumns && threads <= 256 && ring <= D.smem_optin - 128) {
      LAUNCH_NAMED(D, name, columns, std::min(N0, D.nsm * 16), threads, ring, N0, b0, Dinv, Ainv, 3, D.err_dev);
    } else {
      const int buffers = two <= D.smem_optin ? 2 : 1;  // half bandwidths past about 400 in FP64: one
      LAUNCH_NAMED(D, name, blocks, (N0 + 31) / 32, 256, buffers == 2 ? two : one, N0, b0, Dinv, Ainv, buffers);
    }
  };
  if (fp32_coarse(c))
    run(k_coarse_inverse<float>, k_coarse_inverse_blocks<float>, "k_coarse_inverse<float>", dev::ring_threads<float>(b0),
        coarse_solve_vector<float>(N0), dev::ring_stage_bytes<float>(b0), inverse_smem<float>(b0, 2),
        inverse_smem<float>(b0, 1), (const float*)D.A0dinv, (float*)D.ainv);
  else
    run(k_coarse_inverse<double>, k_coarse_inverse_blocks<double>, "k_coarse_inverse<double>",
        dev::ring_threads<double>(b0), coarse_solve_vector<double>(N0), dev::ring_stage_bytes<double>(b0),
        inverse_smem<double>(b0, 2), inverse_smem<double>(b0, 1), (const double*)D.A0dinv, (double*)D.ainv);
}

// The tangent phase's coarse work at u_0, first part (issued on D.s): DF(u_0) for the coarse term
// of Eq. 12 and A_0(u_0).  These kernels use many CTAs and run before the persistent local
// Newton launch, which then holds every SM.
void tangent_coarse_assemble(Context& c) {
  Dev& D = *c.dev;
  global_jacobian(c, D.u0);
  D.ainv_valid = false;
  coarse_assemble_launch(c, D.u0);
}

// Second part (issued on the high-priority second stream): the one-CTA factorization of A_0(u_0),
// placed beside the local Newton CTAs, and (N_0 <= kMaxInverseN0) the explicit inverse the GMRES
// iterations' coarse solves use.  The factorization's status is read by the caller.
void tangent_coarse_factor(Context& c) {
  coarse_factor_launch(c);
  coarse_inverse_launch(c);
}

// F_x(u) into D.Fx; prepares everything the tangent needs.
FxInfo evaluate_Fx(Context& c, const double* u, double load, double* t_inner, double* t_coarse) {
  Dev& D = *c.dev;
  FxInfo info;
  const int cp = c.opt.coupling;
  CK(cudaMemsetAsync(D.Fx, 0, sizeof(double) * c.N, D.s));
  auto t0 = std::chrono::steady_clock::now();
  const double* point = u;
  if (cp != NLS_COUPLING_ONE) {
    CoarseResult cr = coarse_newton(c, u, load);
    info.coarse_its = cr.its;
    info.coarse_status = cr.status;
    if (cp == NLS_COUPLING_HYBRID) point = D.u0;
  }
  sync(D);
  auto t1 = std::chrono::steady_clock::now();
  // The tangent phase's coarse work depends on u_0 only.  DF(u_0) and A_0(u_0) (many CTAs, FP64) go
  // first on this stream; the single-CTA factorization of A_0 and the explicit inverse go on a second
  // stream of the highest priority, beside the batched local solves, whose persistent grid leaves them
  // one SM where it holds one CTA per SM (it pulls subdomains from a work counter: a CTA less, or one
  // that starts late, only takes fewer of them).  Beside a local grid that fills the registers of every
  // SM the assembly itself starved: 4.8 instead of 1.2 ms a launch for Eq. 2's Galerkin blocks (384^2 cells).
  // The tiled factorization spreads every step over many CTAs: it cannot live in the corner of the
  // machine the local grid leaves, so it runs alone on the main stream, before the local solves.
  const bool two_level = cp != NLS_COUPLING_ONE;
  const bool serial_coarse = two_level && D.tlu != nullptr;
  const bool spare_sm = two_level && !serial_coarse && newton_ctas_per_sm(c) == 1;
  if (serial_coarse) {
    tangent_coarse_assemble(c);
    tangent_coarse_factor(c);
  } else if (two_level) {
    tangent_coarse_assemble(c);
    if (!D.s2) {
      int least = 0, greatest = 0;
      CK(cudaDeviceGetStreamPriorityRange(&least, &greatest));
      CK(cudaStreamCreateWithPriority(&D.s2, cudaStreamNonBlocking, greatest));
      CK(cudaEventCreateWithFlags(&D.ev_u0, cudaEventDisableTiming));
      CK(cudaEventCreateWithFlags(&D.ev_coarse, cudaEventDisableTiming));
    }
    CK(cudaEventRecord(D.ev_u0, D.s));
    CK(cudaStreamWaitEvent(D.s2, D.ev_u0, 0));
    std::swap(D.s, D.s2);
    try {
      tangent_coarse_factor(c);
    } catch (...) {
      std::swap(D.s, D.s2);
      throw;
    }
    CK(cudaEventRecord(D.ev_coarse, D.s));
    std::swap(D.s, D.s2);
  }
  const GuessProposal proposal = guess_propose(c, point, load);
  tune_local_newton(c, point, D.Fx, load, proposal);
  D.coarse_beside = spare_sm;
  launch_local_newton(c, point, D.Fx, load, proposal, true);
  D.coarse_beside = false;
  D.local_factors_valid = true;  // every subdomain with status OK now holds its tangent factors
  guess_after_local(c, point, load, proposal.x != nullptr);
  std::vector<int32_t> its(c.ov.count), st(c.ov.count), ch(c.ov.count);
  CK(cudaMemcpyAsync(its.data(), D.ov.its, sizeof(int32_t) * its.size(), cudaMemcpyDeviceToHost, D.s));
  CK(cudaMemcpyAsync(st.data(), D.ov.status, sizeof(int32_t) * st.size(), cudaMemcpyDeviceToHost, D.s));
  CK(cudaMemcpyAsync(ch.data(), D.ov.chord, sizeof(int32_t) * ch.size(), cudaMemcpyDeviceToHost, D.s));
  sync(D);
  auto t2 = std::chrono::steady_clock::now();
  for (int i = 0; i < c.ov.count; ++i) {
    info.local_its += its[i];
    info.local_chord += ch[i];
    if (st[i] != ST_OK) {
      info.local_failures += 1;
      if (info.first_failed < 0) info.first_failed = i;
      if (st[i] == ST_PIVOT) info.pivot_failure = true;
    }
  }
  if (two_level) {
    // F_x += P0 T_0(u); the coarse part of the tangent at u_0 = u - P0 T_0(u) comes from the
    // second stream
    LAUNCH(D, k_p0_apply, grid_for(c.N), 256, 0, c.N, D.p0_slice, D.p0_col, D.p0_val, D.c, 1.0, D.Fx, 1.0, D.Fx,
           (double*)nullptr);
    if (!serial_coarse) CK(cudaStreamWaitEvent(D.s, D.ev_coarse, 0));
    D.coarse_fact_valid = coarse_status_ok(c);
    if (!D.coarse_fact_valid) info.pivot_failure = true;
    D.ainv_valid = D.coarse_fact_valid && D.ainv != nullptr;
  }
  sync(D);
  auto t3 = std::chrono::steady_clock::now();
  if (t_inner) *t_inner += std::chrono::duration<double>(t2 - t1).count();
  if (t_coarse) *t_coarse += std::chrono::duration<double>(t1 - t0).count() + std::chrono::duration<double>(t3 - t2).count();
  c.dev->tangent_ready = true;
  return info;
}

// y = DF_x v (Eq. 6 / Eq. 12)
void tangent(Context& c, const double* v, double* y) {
  Dev& D = *c.dev;
  const int cp = c.opt.coupling;
  if (cp == NLS_COUPLING_ONE) {
    launch_local_apply(c, v, nullptr, y);
    return;
  }
  // w0 = P0 A0^-1 P0^T DF(u0) v
  LAUNCH(D, k_spmv_free, grid_for(c.N), 256, 0, c.N, D.g_slice, D.g_col, D.g_val, D.free_dof, v, D.t1);
  p0t(c, D.t1, D.tg);
  coarse_solve(c, D.tg, D.dc);
  // hybrid: t2 = v - w0 in the same pass
  const bool hybrid = cp == NLS_COUPLING_HYBRID;
  LAUNCH(D, k_p0_apply, grid_for(c.N), 256, 0, c.N, D.p0_slice, D.p0_col, D.p0_val, D.dc, 1.0, v, -1.0,
         hybrid ? D.t2 : (double*)nullptr, D.w0);
  launch_local_apply(c, hybrid ? D.t2 : v, D.w0, y);
}

struct GmresResult {
  int its = 0;
  double relres = 0.0;
  bool converged = false;
};

// GMRES(m), zero initial guess, classical Gram-Schmidt with one re-orthogonalisation (device
// multi-dots), Givens rotations and the least-squares update on the device.  Solution into D.gx.
//
// A cycle of up to m iterations runs without the host: with CUDA graphs it is one graph of m
// conditional (IF) nodes in a chain, node j holding iteration j's body (tangent application,
// two Gram-Schmidt passes, norm, scaling, Givens step); the Givens kernel of iteration j sets the
// shared condition to "continue" or "stop" (converged, breakdown, or the cycle's iteration limit),
// so no body after the last useful one is launched.  The host reads the cycle's state once, then
// the least-squares solve and the update run on the device.  The cycle graph holds device pointers
// and kernel arguments, so it is keyed by everything those depend on: the options, the
// coarse-solve form (explicit inverse or band factors), the tangent CTA size and the scratch
// vectors.  Without graphs (profiling, or cuda_graphs = 0) the same kernels run on the stream and
// the host reads the state after every iteration.
std::string cycle_graph_key(Context& c) {
  Dev& D = *c.dev;
  std::string key((const char*)&c.opt, sizeof(c.opt));
  key += D.ainv_valid ? 'i' : 'b';
  key += std::to_string(apply_threads(c)) + "," + std::to_string(D.m) + ",";
  // scratch vectors the tangent writes (some are swapped by the coarse Newton iteration)
  for (const void* p : {(const void*)D.t1, (const void*)D.t2, (const void*)D.w0, (const void*)D.tg,
                        (const void*)D.dc, (const void*)D.gpart, (const void*)D.cres,
                        (const void*)D.cpart, (const void*)D.cflag})
    key += std::to_string((uintptr_t)p) + ",";
  return key;
}

// Captures (first use) and launches the cycle graph; body(j, next, use) issues iteration j, whose
// Givens step sets `next` (the condition of node j + 1) when `use` is set.  The kernels of every
// body are counted apart, for the launch count once the cycle's length is known.
template <typename F>
void run_cycle_graph(Context& c, F&& body) {
  Dev& D = *c.dev;
  const std::string key = cycle_graph_key(c);
  if (key != D.graph_key || D.it_exec.empty()) {
    D.reset_graphs();
    D.graph_key = key;
    if (!D.cap) CK(cudaStreamCreateWithFlags(&D.cap, cudaStreamNonBlocking));
    cudaGraph_t G = nullptr;
    CK(cudaGraphCreate(&G, 0));
    const cudaStream_t saved = D.s;
    const int64_t l0 = D.launches;
    try {
      // one condition per node (a handle belongs to one conditional node): node 0 runs by default,
      // node j + 1 only when iteration j's Givens step sets its handle; all are reset at launch
      std::vector<cudaGraphConditionalHandle> h(D.m);
      for (int j = 0; j < D.m; ++j)
        CK(cudaGraphConditionalHandleCreate(&h[j], G, j == 0 ? 1u : 0u, cudaGraphCondAssignDefault));
      cudaGraphNode_t prev = nullptr;
      D.it_launches.assign(D.m, 0);
      for (int j = 0; j < D.m; ++j) {
        cudaGraphNodeParams p = {};
        p.type = cudaGraphNodeTypeConditional;
        p.conditional.handle = h[j];
        p.conditional.type = cudaGraphCondTypeIf;
        p.conditional.size = 1;
        cudaGraphNode_t node = nullptr;
        CK(cudaGraphAddNode(&node, G, prev ? &prev : nullptr, nullptr, prev ? 1 : 0, &p));
        cudaGraph_t bg = p.conditional.phGraph_out[0];
        const int64_t lj = D.launches;
        CK(cudaStreamBeginCaptureToGraph(D.cap, bg, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
        D.s = D.cap;
        try {
          body(j, j + 1 < D.m ? h[j + 1] : cudaGraphConditionalHandle{}, j + 1 < D.m ? 1 : 0);
        } catch (...) {
          cudaGraph_t tmp = nullptr;
          cudaStreamEndCapture(D.cap, &tmp);
          throw;
        }
        D.s = saved;
        CK(cudaStreamEndCapture(D.cap, &bg));
        D.it_launches[j] = D.launches - lj;
        prev = node;
      }
      cudaGraphExec_t ex = nullptr;
      CK(cudaGraphInstantiate(&ex, G, 0));
      D.it_exec.assign(1, ex);
    } catch (...) {
      D.s = saved;
      D.launches = l0;
      cudaGraphDestroy(G);
      D.reset_graphs();
      throw;
    }
    cudaGraphDestroy(G);
    D.launches = l0;
  }
  CK(cudaGraphLaunch(D.it_exec[0], D.s));
}

GmresResult gmres(Context& c, const double* b) {
  Dev& D = *c.dev;
  const int64_t N = c.N;
  const int m = D.m;
  GmresResult R;
  tune_local_apply(c, b, D.t1);
  const bool graphs = c.opt.cuda_graphs && !D.prof;
  CK(cudaMemsetAsync(D.gx, 0, sizeof(double) * N, D.s));
  const double bn = norm2(D, N, b);
  if (bn == 0.0) {
    R.converged = true;
    return R;
  }
  double* r = D.t2;
  CK(cudaMemcpyAsync(r, b, sizeof(double) * N, cudaMemcpyDeviceToDevice, D.s));
  double rn = bn;
  const double target = c.opt.gmres_rtol * bn;
  // iteration j of a cycle: w = DF_x v_j, CGS2 against v_0 .. v_j, h_{j+1,j} = ||w||, v_{j+1} =
  // w / h_{j+1,j}, Givens step (sets the graph condition when `use_handle`)
  auto body = [&](int j, cudaGraphConditionalHandle h, int use_handle) {
    double* vj = D.V + (size_t)j * N;
    double* w = D.V + (size_t)(j + 1) * N;
    tangent(c, vj, w);
    // h = V^T w; w -= V h, h' = V^T w; w -= V h', ||w|| and the Givens step; v_{j+1} = w / ||w||
    double* second = D.scal + kMaxGmresVecs / 2;
    dots(D, N, j + 1, D.V, N, nullptr, w, D.scal);
    dots(D, N, j + 1, D.V, N, D.scal, w, second);
    const int E = tile_elems(D, N), grid = tile_grid(D, N);
    auto update = [&](auto kernel) {
      LAUNCH_NAMED(D, "k_gmres_update", kernel, grid, kTile, 0, N, j, D.V, N, second, w, D.partial, D.ticket, m, D.scal,
                   D.gR, D.gcs, D.gsn, D.gg, D.gst, h, use_handle);
    };
    if (E == 1) update(k_gmres_update<1>);
    else update(k_gmres_update<4>);
    LAUNCH(D, k_scale_inv, grid_for(N), 256, 0, N, w, D.scal + kMaxGmresVecs, w);
  };
  GmresState st;
  while (R.its < c.opt.gmres_maxit) {
    LAUNCH(D, k_axpby, grid_for(N), 256, 0, N, 1.0 / rn, r, 0.0, nullptr, D.V);
    const int limit = std::min(m, c.opt.gmres_maxit - R.its);
    LAUNCH(D, k_gmres_start, 1, 32, 0, m, rn, target, limit, D.gg, D.gst);
    if (graphs) {
      run_cycle_graph(c, body);
      CK(cudaMemcpyAsync(&st, D.gst, sizeof(st), cudaMemcpyDeviceToHost, D.s));
      sync(D);
      for (int j = 0; j < st.j; ++j) D.launches += D.it_launches[j];
    } else {
      for (int j = 0; j < limit; ++j) {
        body(j, cudaGraphConditionalHandle{}, 0);
        CK(cudaMemcpyAsync(&st, D.gst, sizeof(st), cudaMemcpyDeviceToHost, D.s));
        sync(D);
        if (st.done || st.j >= limit) break;
      }
    }
    // y = R^-1 g (back substitution) and x += V y, on the device
    LAUNCH(D, k_gmres_lsq, 1, 32, 0, m, D.gR, D.gg, D.gst, D.coef);
    LAUNCH(D, k_multiaxpy_dev, grid_for(N), 256, 0, N, D.gst, D.V, N, D.coef, 1.0, D.gx);
    R.its += st.j;
    R.relres = st.res / bn;
    if (st.done && st.res <= target) {
      R.converged = true;
      break;
    }
    // restart: r = b - A x
    tangent(c, D.gx, D.t1);
    LAUNCH(D, k_axpby, grid_for(N), 256, 0, N, 1.0, b, -1.0, D.t1, r);
    rn = norm2(D, N, r);
    R.relres = rn / bn;
    if (rn <= target) {
      R.converged = true;
      break;
    }
    if (st.done) break;
  }
  return R;
}

}  // namespace

int solve(Context& c, double* u_user, int u_dev, nls_report* rep) {
  Dev& D = *c.dev;
  nls_report rp;
  std::memset(&rp, 0, sizeof(rp));
  rp.first_failed_subdomain = -1;
  int status = NLS_OK;
  const int64_t N = c.N;
  const int64_t launches0 = D.launches;
  try {
    CK(cudaSetDevice(c.device));
    D.prof = c.opt.profile_kernels != 0;
    // a solve depends on its inputs only: the coarse factorization is reused across the outer
    // iterations of this call, never from an earlier one
    D.coarse_fact_valid = false;
    D.ainv_valid = false;
    D.local_factors_valid = false;
    D.local_reuse_active = c.opt.local_reuse != 0;
    struct ReuseScope {  // chord steps only inside this solve, never in a later nls_eval_Fx
      Dev& d;
      ~ReuseScope() { d.local_reuse_active = false; }
    } reuse_scope{D};
    cudaEvent_t e0, e1;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    CK(cudaEventRecord(e0, D.s));
    auto w0 = std::chrono::steady_clock::now();
    CK(cudaMemcpyAsync(D.u, u_user, sizeof(double) * N, u_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, D.s));
    LAUNCH(D, k_set_dirichlet, grid_for(N), 256, 0, N, D.free_dof, D.ubc, D.u);
    double t_inner = 0, t_coarse = 0, t_gmres = 0;
    const int L = std::max(1, c.opt.load_steps);
    double nF = INFINITY;
    // F_x at a point, with the statistics of its local and coarse solves
    auto eval_fx = [&](const double* x, double load) {
      FxInfo f = evaluate_Fx(c, x, load, &t_inner, &t_coarse);
      rp.subdomain_newton_steps += f.local_its;
      rp.local_chord_steps += f.local_chord;
      rp.coarse_newton_steps += f.coarse_its;
      rp.local_failures += f.local_failures;
      if (rp.first_failed_subdomain < 0) rp.first_failed_subdomain = f.first_failed;
      return f;
    };
    for (int step = 1; step <= L && status == NLS_OK; ++step) {
      const double load = (double)step / L;
      bool have_fx = false;  // D.Fx and the tangent data belong to D.u (from the backtracking)
      FxInfo fi;
      for (int k = 0;; ++k) {
        global_residual(c, D.u, D.F, load);
        nF = norm2(D, N, D.F);
        if (c.opt.verbose) std::fprintf(stderr, "[nls] load %.3f outer %d ||F|| = %.3e\n", load, k, nF);
        if (!std::isfinite(nF)) {
          status = NLS_E_DIVERGED;
          break;
        }
        if (nF < c.opt.outer_atol) break;
        if (k >= c.opt.outer_maxit) {
          status = NLS_W_NOT_CONVERGED;
          break;
        }
        if (!have_fx) {
          if (c.opt.coarse_rebuild && c.opt.coupling != NLS_COUPLING_ONE && c.coarse_kind == NLS_COARSE_RGDSW) {
            // the coarse basis from the current tangent: P_0 changes, so does every A_0
            coarse_extension(c, D.u);
            D.coarse_fact_valid = false;
            D.ainv_valid = false;
          }
          D.outer_k = k;
          fi = eval_fx(D.u, load);
          D.outer_k = -1;
        }
        have_fx = false;
        if (fi.pivot_failure) {
          status = NLS_E_PIVOT;
          break;
        }
        const double fxn = norm2(D, N, D.Fx);
        if (fxn == 0.0) {
          // Every correction vanished.  With all local and coarse solves converged, ||F|| is below
          // what their stopping tests resolve: the outer iteration has converged as far as it can.
          // With failed solves (their corrections are dropped) it cannot progress: not converged.
          if (fi.local_failures > 0 || fi.coarse_status != ST_OK) status = NLS_W_NOT_CONVERGED;
          break;
        }
        auto g0 = std::chrono::steady_clock::now();
        GmresResult gr = gmres(c, D.Fx);
        sync(D);
        t_gmres += std::chrono::duration<double>(std::chrono::steady_clock::now() - g0).count();
        rp.gmres_iterations += gr.its;
        rp.outer_iterations += 1;
        if (c.opt.verbose)
          std::fprintf(stderr, "[nls]   ||Fx|| = %.3e gmres %d (rel %.2e) local its %lld coarse its %d\n", fxn, gr.its,
                       gr.relres, (long long)fi.local_its, fi.coarse_its);
        if (!c.opt.outer_backtrack) {
          LAUNCH(D, k_axpby, grid_for(N), 256, 0, N, 1.0, D.u, -1.0, D.gx, D.u);
          continue;
        }
        // Backtracking on ||F_x||: the first of alpha = 1, 1/2, ... (at most min(ls_trials, 5))
        // with ||F(u')|| < outer_atol or ||F_x(u')|| <= (1 - armijo alpha) ||F_x(u)||, u' = u - alpha
        // du; the last trial is taken otherwise.  An accepted trial's F_x and tangent data serve
        // the next outer iteration, so a full step costs nothing extra.
        const int trials = std::max(1, std::min(c.opt.ls_trials, 5));
        double alpha = 1.0;
        for (int t = 0; t < trials; ++t) {
          LAUNCH(D, k_axpby, grid_for(N), 256, 0, N, 1.0, D.u, -alpha, D.gx, D.ut);
          global_residual(c, D.ut, D.F, load);
          const double nFt = norm2(D, N, D.F);
          if (nFt < c.opt.outer_atol) break;
          D.outer_k = k + 1;  // a trial point: the next outer iterate
          const FxInfo ft = eval_fx(D.ut, load);
          D.outer_k = -1;
          const double fxt = norm2(D, N, D.Fx);
          if ((std::isfinite(fxt) && fxt <= (1.0 - c.opt.armijo * alpha) * fxn) || t + 1 == trials ||
              ft.pivot_failure) {
            fi = ft;
            have_fx = true;
            break;
          }
          alpha *= 0.5;
        }
        if (c.opt.verbose && alpha < 1.0) std::fprintf(stderr, "[nls]   outer step alpha = %.4g\n", alpha);
        std::swap(D.u, D.ut);
      }
    }
    rp.final_residual = nF;
    CK(cudaMemcpyAsync(u_user, D.u, sizeof(double) * N, u_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, D.s));
    CK(cudaEventRecord(e1, D.s));
    CK(cudaEventSynchronize(e1));
    tlu_check_solves(c);
    check_local_waits(D);
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, e0, e1));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    const double wall = std::chrono::duration<double>(std::chrono::steady_clock::now() - w0).count();
    rp.time_total_s = ms * 1e-3;
    rp.time_inner_s = t_inner;
    rp.time_coarse_s = t_coarse;
    rp.time_gmres_s = t_gmres;
    rp.time_other_s = std::max(0.0, wall - t_inner - t_coarse - t_gmres);
    D.prof_flush();
  } catch (const DeviceTimeout& ex) {
    c.last_error = ex.what();
    status = NLS_E_DEVICE_TIMEOUT;
    forget_waits(D);
  } catch (const CudaFailure& ex) {
    c.last_error = ex.what();
    status = NLS_E_CUDA;
    forget_waits(D);
  } catch (const std::exception& ex) {
    c.last_error = ex.what();
    status = NLS_E_ARG;
    forget_waits(D);
  }
  rp.kernel_launches = D.launches - launches0;
  rp.status = status;
  if (rep) *rep = rp;
  return status;
}

int eval_F(Context& c, const double* u, double* F, int is_dev, double load) {
  Dev& D = *c.dev;
  try {
    if (is_dev) {  // read and written in place: the element pass has read u before F is written
      global_residual(c, u, F, load);
    } else {
      CK(cudaMemcpyAsync(D.x, u, sizeof(double) * c.N, cudaMemcpyHostToDevice, D.s));
      global_residual(c, D.x, D.F, load);
      CK(cudaMemcpyAsync(F, D.F, sizeof(double) * c.N, cudaMemcpyDeviceToHost, D.s));
    }
    sync(D);
  } catch (const std::exception& ex) {
    c.last_error = ex.what();
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

int eval_Fx(Context& c, const double* u, double* Fx, int is_dev, double load, int32_t* its, int32_t* st) {
  Dev& D = *c.dev;
  D.prof = c.opt.profile_kernels != 0;
  try {
    CK(cudaMemcpyAsync(D.u, u, sizeof(double) * c.N, is_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, D.s));
    FxInfo fi = evaluate_Fx(c, D.u, load, nullptr, nullptr);
    CK(cudaMemcpyAsync(Fx, D.Fx, sizeof(double) * c.N, is_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, D.s));
    if (its) CK(cudaMemcpyAsync(its, D.ov.its, sizeof(int32_t) * c.ov.count, cudaMemcpyDeviceToHost, D.s));
    if (st) CK(cudaMemcpyAsync(st, D.ov.status, sizeof(int32_t) * c.ov.count, cudaMemcpyDeviceToHost, D.s));
    sync(D);
    check_local_waits(D);
    if (fi.pivot_failure) return NLS_E_PIVOT;
  } catch (const DeviceTimeout& ex) {
    c.last_error = ex.what();
    forget_waits(D);
    return NLS_E_DEVICE_TIMEOUT;
  } catch (const std::exception& ex) {
    c.last_error = ex.what();
    forget_waits(D);
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

int apply_tangent(Context& c, const double* v, double* y, int is_dev) {
  Dev& D = *c.dev;
  if (!D.tangent_ready) {
    c.last_error = "nls_apply_tangent needs a preceding nls_eval_Fx";
    return NLS_E_ARG;
  }
  D.prof = c.opt.profile_kernels != 0;
  try {
    // device arrays are used in place; where y overlaps v at an offset, it would be cleared over parts of v
    // not read yet
    const uintptr_t pv = (uintptr_t)v, py = (uintptr_t)y, bytes = sizeof(double) * c.N;
    const bool staged = !is_dev || (pv != py && pv < py + bytes && py < pv + bytes);
    if (staged) CK(cudaMemcpyAsync(D.t1, v, bytes, is_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, D.s));
    double* out = is_dev ? y : D.gx;
    LAUNCH(D, k_masked_copy, grid_for(c.N), 256, 0, c.N, D.free_dof, staged ? D.t1 : v, D.x, out);
    tangent(c, D.x, out);
    if (!is_dev) CK(cudaMemcpyAsync(y, D.gx, sizeof(double) * c.N, cudaMemcpyDeviceToHost, D.s));
    sync(D);
    check_local_waits(D);
  } catch (const DeviceTimeout& ex) {
    c.last_error = ex.what();
    forget_waits(D);
    return NLS_E_DEVICE_TIMEOUT;
  } catch (const std::exception& ex) {
    c.last_error = ex.what();
    forget_waits(D);
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

int get_local_states(Context& c, double* w, int is_dev) {
  Dev& D = *c.dev;
  try {
    CK(cudaMemcpyAsync(w, D.ov.w, sizeof(double) * c.ov.total_n, is_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, D.s));
    sync(D);
  } catch (const std::exception& ex) {
    c.last_error = ex.what();
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

int kernel_stats(const Context& c, int32_t cap, nls_kernel_stat* out, int32_t* n_out) {
  if (!c.dev) {
    *n_out = 0;
    return NLS_OK;
  }
  Dev& D = *c.dev;
  try {
    D.prof_flush();
  } catch (const std::exception&) {
    return NLS_E_CUDA;
  }
  int32_t n = 0;
  for (auto& st : D.stats) {
    if (out && n < cap) {
      out[n].name = st.name.c_str();
      out[n].launches = st.launches;
      out[n].total_ms = st.ms;
    }
    ++n;
  }
  // k_local_newton phases: CTA-milliseconds (sum over CTAs of thread 0's clock64 deltas)
  static const char* kPhaseNames[8] = {"phase:gather+residual", "phase:jacobian", "phase:band_lu",
                                       "phase:solve+refine",   "phase:line_search", "phase:tangent_jacobian",
                                       "phase:tangent_band_lu", "phase:output"};
  unsigned long long ph[8] = {0};
  try {
    CK(cudaMemcpy(ph, D.phase, sizeof(ph), cudaMemcpyDeviceToHost));
  } catch (const std::exception&) {
    return NLS_E_CUDA;
  }
  for (int k = 0; k < 8; ++k) {
    if (!ph[k]) continue;
    if (out && n < cap) {
      out[n].name = kPhaseNames[k];
      out[n].launches = 0;
      out[n].total_ms = (double)ph[k] / (double)D.clock_khz;
    }
    ++n;
  }
  *n_out = std::min(n, cap);
  return NLS_OK;
}

void reset_kernel_stats(Context& c) {
  if (!c.dev) return;
  try {
    c.dev->prof_flush();
    CK(cudaMemsetAsync(c.dev->phase, 0, sizeof(unsigned long long) * 8, c.dev->s));
  } catch (const std::exception&) {
  }
  c.dev->stats.clear();
}

int get_coarse_basis(const Context& c, double* P0) {
  if (c.coarse_kind != NLS_COARSE_RGDSW || !c.dev) return NLS_E_ARG;
  Dev& D = *c.dev;
  try {
    std::vector<double> vals(c.cs.p0_col.size());
    CK(cudaMemcpyAsync(vals.data(), D.p0_val, sizeof(double) * vals.size(), cudaMemcpyDeviceToHost, D.s));
    CK(cudaStreamSynchronize(D.s));
    std::memset(P0, 0, sizeof(double) * c.N * c.cs.N0);
    for (int64_t g = 0; g < c.N; ++g)
      for (int64_t k = c.cs.p0_slice[g >> 5] + (g & 31); k < c.cs.p0_slice[(g >> 5) + 1]; k += 32)
        if (c.cs.p0_src[k] >= 0) P0[(int64_t)c.cs.p0_col[k] * c.N + g] = vals[k];
  } catch (const std::exception&) {
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

int guess_smooth(Context& c, const double* x, double load, const double* w, double* out) {
  if (!c.dev || !c.dev->guess) {
    c.last_error = "the learned-guess hooks need an attached network";
    return NLS_E_ARG;
  }
  Dev& D = *c.dev;
  try {
    const GuessProposal g = guess_smoothing(c);
    CK(cudaMemcpyAsync(D.x, x, sizeof(double) * c.N, cudaMemcpyHostToDevice, D.s));
    CK(cudaMemcpyAsync(D.ov.w, w, sizeof(double) * c.ov.total_n, cudaMemcpyHostToDevice, D.s));
    LocalArgs A = make_args(c, c.ov, D.ov);
    A.x = D.x;
    A.load = load;
    A.guess = D.ov.w;
    A.guess_diag = g.diag;
    A.guess_sweeps = g.sweeps;
    A.guess_omega = g.omega;
    A.out = D.ov.work;  // concatenated local vectors
    const size_t sm = sizeof(double) * ((size_t)c.ov.max_nt + c.ov.max_n) + 16;
    if (c.law == NLS_LAW_DIFFUSION) LAUNCH(D, k_guess_smooth<NLS_LAW_DIFFUSION>, c.ov.count, 128, sm, A);
    else LAUNCH(D, k_guess_smooth<NLS_LAW_NEOHOOKE>, c.ov.count, 128, sm, A);
    CK(cudaMemcpyAsync(out, D.ov.work, sizeof(double) * c.ov.total_n, cudaMemcpyDeviceToHost, D.s));
    sync(D);
  } catch (const std::exception& ex) {
    c.last_error = ex.what();
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

int get_coarse_matrix(const Context& c, double* A0) {
  if (c.coarse_kind != NLS_COARSE_RGDSW || !c.dev || !c.dev->A0) return NLS_E_ARG;
  Dev& D = *c.dev;
  try {
    CK(cudaMemcpyAsync(A0, D.A0, sizeof(double) * (size_t)c.cs.N0 * (2 * c.cs.b0 + 1), cudaMemcpyDeviceToHost, D.s));
    CK(cudaStreamSynchronize(D.s));
  } catch (const std::exception&) {
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

// The coarse factorization and solve on a given band matrix (parity hook and utility): a context
// with only the coarse problem, run on the legacy default stream and freed on return.
int band_solve(int device, int32_t n, int32_t b, const double* band, const double* rhs, double* x, int32_t precision,
               int32_t method, double* factors_out) {
  if (n < 1 || b < 0 || !band || !rhs || !x) return NLS_E_ARG;
  if ((precision != NLS_PREC_FP64 && precision != NLS_PREC_FP32_IR) || method < NLS_COARSE_FACTOR_AUTO ||
      method > NLS_COARSE_FACTOR_TILES)
    return NLS_E_ARG;
  Context c;
  c.device = device;
  c.stream = nullptr;
  nls_options_default(&c.opt);
  c.opt.coarse_precision = precision;
  c.opt.coarse_factor = method;
  c.coarse_kind = NLS_COARSE_RGDSW;
  c.cs.N0 = n;
  c.cs.b0 = b;
  int status = NLS_OK;
  try {
    if (b > kMaxSolveB0 || (!coarse_tiles(c) && b > kMaxBandB0)) return NLS_E_UNSUPPORTED;
    CK(cudaSetDevice(device));
    c.dev = new Dev();
    Dev& D = *c.dev;
    D.s = nullptr;
    cudaDeviceProp prop;
    CK(cudaGetDeviceProperties(&prop, device));
    D.nsm = prop.multiProcessorCount;
    D.smem_optin = prop.sharedMemPerBlockOptin;
    const bool f32 = fp32_coarse(c);
    const size_t fs = f32 ? sizeof(float) : sizeof(double);
    if (fs * (size_t)n > D.smem_optin || (!coarse_tiles(c) && coarse_factor_smem(c, f32) > D.smem_optin)) {
      device_free(c);
      return NLS_E_UNSUPPORTED;  // the one-CTA window or the solve vector exceeds shared memory
    }
    alloc_err(D);
    const size_t nw = (size_t)n * (2 * b + 1);
    D.A0 = D.alloc<double>(nw);
    CK(cudaMemcpyAsync(D.A0, band, sizeof(double) * nw, cudaMemcpyHostToDevice, D.s));
    const size_t ndinv = (size_t)packed_solve_entries(n, b);
    if (f32) {
      D.A0f = D.alloc<float>(nw);
      D.A0dinv = D.alloc<float>(ndinv);
    } else {
      D.A0f = D.alloc<double>(nw);
      D.A0dinv = D.alloc<double>(ndinv);
    }
    D.cstatus = D.alloc<int32_t>(1);
    D.cpart = D.alloc<double>(2 * (size_t)((n + 7) / 8));
    D.cflag = D.alloc<int>(2);
    CK(cudaMemsetAsync(D.cflag, 0, 2 * sizeof(int), D.s));
    D.cres = D.alloc<double>(n);
    D.g = D.alloc<double>(n);
    D.dc = D.alloc<double>(n);
    CK(cudaMemcpyAsync(D.g, rhs, sizeof(double) * n, cudaMemcpyHostToDevice, D.s));
    set_smem(k_coarse_factor<float>, D.smem_optin);
    set_smem(k_coarse_factor<double>, D.smem_optin);
    set_smem(k_coarse_band_solve<float>, D.smem_optin);
    set_smem(k_coarse_band_solve<double>, D.smem_optin);
    if (coarse_tiles(c)) tlu_prepare(c, f32);
    coarse_factor_launch(c);
    if (!coarse_status_ok(D)) {
      status = NLS_E_PIVOT;
    } else {
      coarse_solve(c, D.g, D.dc);
      CK(cudaMemcpyAsync(x, D.dc, sizeof(double) * n, cudaMemcpyDeviceToHost, D.s));
    }
    if (factors_out) {
      std::vector<float> f(f32 ? nw : 0);
      if (f32) CK(cudaMemcpyAsync(f.data(), D.A0f, sizeof(float) * nw, cudaMemcpyDeviceToHost, D.s));
      else CK(cudaMemcpyAsync(factors_out, D.A0f, sizeof(double) * nw, cudaMemcpyDeviceToHost, D.s));
      sync(D);
      if (f32)
        for (size_t k = 0; k < nw; ++k) factors_out[k] = (double)f[k];
    }
    sync(D);
    tlu_check_solves(c);
    check_local_waits(D);
  } catch (const DeviceTimeout&) {
    status = NLS_E_DEVICE_TIMEOUT;
  } catch (const CudaFailure&) {
    status = NLS_E_CUDA;
  } catch (const std::bad_alloc&) {
    status = NLS_E_NOMEM;
  } catch (const std::exception&) {
    status = NLS_E_ARG;
  }
  device_free(c);
  return status;
}

// ------------------------------------------------------------------------------------------
// Local corrections without any allocation.
//
// Some callers cannot allocate device memory when they need the corrections: a solver step
// being recorded into a CUDA graph (cudaMalloc is not allowed while a stream is capturing),
// a host application whose memory manager owns every byte of the GPU, or a time-critical loop
// that must not risk the device-wide synchronisation cudaMalloc / cudaFree can cause.  For
// them the batched local-Newton kernel also runs on a fixed scratch area compiled into this
// library: a file-scope device array of kNoAllocScratchBytes that every GPU which loads the
// library keeps until the process exits.  Host code cannot use the array's name as a device
// address, so the address is looked up once per device with cudaGetSymbolAddress (on the
// first call on that device, which should therefore come before any stream capture) and then
// passed to the kernel.  All calls share the area and leave their contents in it; calls
// whose work overlaps on the GPU (different streams, or different contexts on one device)
// race on it.
// ------------------------------------------------------------------------------------------
namespace {

constexpr size_t kNoAllocScratchBytes = size_t(32) << 20;
__device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mutex;
void* g_noalloc_addr[kNoAllocMaxDevices] = {nullptr};

// Device address of the scratch array for the current device (looked up once per device).
cudaError_t noalloc_scratch_address(int device, void** out) {
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (device < 0 || device >= kNoAllocMaxDevices) return cudaErrorInvalidDevice;
  if (!g_noalloc_addr[device]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_addr[device] = p;
  }
  *out = g_noalloc_addr[device];
  return cudaSuccess;
}

}  // namespace

int local_corrections_noalloc(Context& c, const double* x, double* Fx, int32_t* its_out, int32_t* status_out,
                              double load) {
  if (!c.is_setup || !c.dev) {
    c.last_error = "nls_local_corrections_noalloc needs a context after nls_setup";
    return NLS_E_ARG;
  }
  Dev& D = *c.dev;
  const LocalSet& s = c.ov;
  const bool f32 = fp32_local(c);
  // scratch plan: matrix values and work vectors, band factors, packed solve operands, local states,
  // its, status, work counter.  The limit is stated for the entries of the matrices and three work
  // vectors; the padded values and two vectors (at most one value of padding per row) never need more.
  const size_t fbytes = f32 ? sizeof(float) : sizeof(double);
  size_t off = 0;
  const size_t o_csr = off, o_work = sizeof(double) * (size_t)s.total_nnz;
  off = align_up(off + sizeof(double) * (size_t)s.total_entries, 256);
  off = align_up(off + 3 * sizeof(double) * (size_t)s.total_n, 256);
  const size_t o_fac = off;
  off = align_up(off + fbytes * (size_t)s.total_factor, 256);
  const size_t o_dinv = off;
  off = align_up(off + fbytes * (size_t)s.total_dinv, 256);
  const size_t o_w = off;
  off = align_up(off + sizeof(double) * (size_t)s.total_n, 256);
  const size_t o_its = off;
  off = align_up(off + sizeof(int32_t) * (size_t)s.count, 256);
  const size_t o_st = off;
  off = align_up(off + sizeof(int32_t) * (size_t)s.count, 256);
  const size_t o_q = off;
  off = align_up(off + sizeof(int32_t), 256);
  if (off > kNoAllocScratchBytes) {
    c.last_error = "problem needs " + std::to_string(off) + " bytes of scratch; the allocation-free entry point has " +
                   std::to_string(kNoAllocScratchBytes);
    return NLS_E_ARG;
  }
  try {
    CK(cudaSetDevice(c.device));
    // per-launch event timing would create events: keep this path allocation free (the flag is
    // restored on return, so the context's profiling option is untouched)
    struct ProfScope {
      Dev& d;
      bool saved;
      ~ProfScope() { d.prof = saved; }
    } prof_scope{D, D.prof};
    D.prof = false;
    void* base = nullptr;
    CK(noalloc_scratch_address(c.device, &base));
    unsigned char* sc = (unsigned char*)base;
    LocalArgs A = make_args(c, s, D.ov);
    A.csr = (double*)(sc + o_csr);
    A.factor = sc + o_fac;
    A.dinv = sc + o_dinv;
    A.wbuf = (double*)(sc + o_w);
    A.work = (double*)(sc + o_work);
    A.work_stride = s.total_n;
    A.its = its_out ? its_out : (int32_t*)(sc + o_its);
    A.status = status_out ? status_out : (int32_t*)(sc + o_st);
    A.queue = (int32_t*)(sc + o_q);
    A.chord = nullptr;  // no chord steps here: the context's counters stay as they are
    A.reuse = 0;
    A.x = x;
    A.out = Fx;
    A.load = load;
    A.guess = nullptr;
    A.want_tangent = 0;
    A.err = D.err_dev + 1;
    // the work counter must start at zero; the rest of the area is written before it is read
    CK(cudaMemsetAsync(A.queue, 0, sizeof(int32_t), D.s));
    LAUNCH(D, k_mask, grid_for(c.N), 256, 0, c.N, D.free_dof, Fx);
    dispatch_local_newton(c, s, A, local_threads(c));
  } catch (const std::exception& ex) {
    c.last_error = ex.what();
    return NLS_E_CUDA;
  }
  return NLS_OK;
}

void options_changed(Context& c) {
  if (!c.dev) return;
  c.dev->coarse_fact_valid = false;
  c.dev->ainv_valid = false;
  c.dev->reset_graphs();
}

int get_tuning(const Context& c, nls_tuning* out) {
  std::memset(out, 0, sizeof(*out));
  out->newton_threads = local_threads(c);
  out->apply_threads = c.dev ? apply_threads(c) : std::max(64, min_local_threads(c));
  if (c.dev) {
    out->newton_tuned = c.dev->newton_tuned ? 1 : 0;
    out->apply_tuned = c.dev->apply_tuned ? 1 : 0;
    out->newton_ms[0] = c.dev->newton_ms[0];
    out->newton_ms[1] = c.dev->newton_ms[1];
    for (auto g : c.dev->it_exec) out->graphs_captured += g ? 1 : 0;
    out->coarse_threads = c.dev->coarse_T;
  }
  return NLS_OK;
}

}  // namespace nls
