// Device building blocks of the nonlinear Schwarz solver (sm_103a).
//
// * element routines of Eq. 1 (P1 nonlinear diffusion) and Eq. 2 (Q1 compressible Neo-Hooke),
// * block reductions with a fixed summation order (results do not depend on scheduling),
// * the no-pivoting band LU: in place by square tiles in a shared-memory window (the local and
//   coarse matrices), and row by row from CSR rows (the harmonic extension),
// * blocked forward / backward substitution with the band factors (one warp solves each
//   32-row diagonal block, the whole CTA applies its coupling to the next b rows).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "nls_internal.h"
#include "tcgen05.cuh"

namespace nls {
namespace dev {

constexpr int kWarp = 32;

// The dynamic shared memory of the kernel.  The large routines below are real calls (their code would
// otherwise be in every kernel twice, and their registers with it); they take their arrays as offsets
// into it, because through a pointer argument the compiler could only use generic loads, which take
// about twice as long as shared-memory ones.
extern __shared__ __align__(128) unsigned char dyn_smem[];
__device__ __forceinline__ uint32_t dyn_offset(const void* p) { return tc::smem_u32(p) - tc::smem_u32(dyn_smem); }

// ------------------------------------------------------------------------------------------
// reductions (deterministic for a fixed block size)
// ------------------------------------------------------------------------------------------
__device__ inline double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the block; every thread receives the result.  `red` holds >= 33 doubles.
__device__ inline double block_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  if (wid == 0) {
    double t = (lane < nw) ? red[lane] : 0.0;
    t = warp_sum(t);
    if (lane == 0) red[32] = t;
  }
  __syncthreads();
  return red[32];
}

// ------------------------------------------------------------------------------------------
// Eq. 1 on P1 triangles.  geo = {dphi_0/dx, dphi_0/dy, dphi_1/dx, ..., area, pad}.
// Residual of the element:  r_a = k Q (grad u . grad phi_a), Q = int_T (1 + u^2) by the
// exact edge-midpoint rule; the source term is handled through the external load vector.
// ------------------------------------------------------------------------------------------
struct P1State {
  double gx, gy, m01, m12, m20, kq, k, area;
};

__device__ inline P1State p1_state(const double* geo, double k, double u0, double u1, double u2) {
  P1State s;
  s.gx = u0 * geo[0] + u1 * geo[2] + u2 * geo[4];
  s.gy = u0 * geo[1] + u1 * geo[3] + u2 * geo[5];
  s.m01 = 0.5 * (u0 + u1);
  s.m12 = 0.5 * (u1 + u2);
  s.m20 = 0.5 * (u2 + u0);
  s.area = geo[6];
  s.k = k;
  const double Q = s.area * (1.0 / 3.0) * (3.0 + s.m01 * s.m01 + s.m12 * s.m12 + s.m20 * s.m20);
  s.kq = k * Q;
  return s;
}

__device__ inline void p1_residual(const double* geo, const P1State& s, double r[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) r[a] = s.kq * (s.gx * geo[2 * a] + s.gy * geo[2 * a + 1]);
}

// K[a][b] = d r_a / d u_b = k Q grad phi_a . grad phi_b + k (grad u . grad phi_a) dQ/du_b
template <typename T>
__device__ inline void p1_jacobian(const double* geo, const P1State& s, T K[9]) {
  const double a3 = s.area * (1.0 / 3.0);
  const double dQ[3] = {a3 * (s.m01 + s.m20), a3 * (s.m01 + s.m12), a3 * (s.m12 + s.m20)};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double flux = s.gx * geo[2 * a] + s.gy * geo[2 * a + 1];
#pragma unroll
    for (int b = 0; b < 3; ++b)
      K[a * 3 + b] = (T)(s.kq * (geo[2 * a] * geo[2 * b] + geo[2 * a + 1] * geo[2 * b + 1]) + s.k * flux * dQ[b]);
  }
}

// ------------------------------------------------------------------------------------------
// Eq. 2 on Q1 quadrilaterals, 2x2 Gauss.  geo per Gauss point q (stride 10): dN_a/dX (4 x 2)
// then weight * det(dX/dxi).  P = mu F - (mu - lambda ln J) F^-T.
// With p_a = F^-1 applied from the left to grad N_a (p_a[i] = sum_J gradN_a[J] Finv[J][i]):
//   r_{a,i}      = w [ mu (F gradN_a)_i - (mu - lambda ln J) p_a[i] ]
//   K_{ai, bk}   = w [ mu delta_ik gradN_a . gradN_b + lambda p_a[i] p_b[k] + (mu - lambda ln J) p_a[k] p_b[i] ]
//
// What bounds these routines is the FP64 rate of the part (1.9 multiply-adds per clock and SM): every
// form below is chosen for its number of FP64 instructions.  The gradients of the four shape
// functions sum to zero, so F takes the displacements relative to node 0, and node 0's rows and
// columns are minus the sums of the others; the tangent is symmetric; the residual goes through w P
// once per Gauss point; log J and 1 / J share one table step.  Per element: residual 218 FP64
// instructions (551 before), tangent 458 (about 1500 before).  Residuals of 147,456 elements: 135 ->
// 72 us.
// ------------------------------------------------------------------------------------------

// log and reciprocal of one positive normal double.  Table-driven logarithm (Tang, "Table-driven
// implementation of the logarithm function in IEEE floating-point arithmetic", 1990): x = 2^e m with
// m in [0.75, 1.5), r the tabulated reciprocal of the middle of m's bin (1 next to 1), t = m r - 1
// exact to one rounding, |t| <= 2^-7, log x = e log 2 - log r + log(1 + t) with the series of
// log(1 + t) to t^7 / 7 (the next term is below 2^-58).  The reciprocal starts from r (1 - t)(1 + t^2)
// = (1 / m)(1 - t^4) and takes one Newton step, which squares the relative error 2^-28.  Largest errors on
// 1.2e7 arguments against quadruple precision: 1.5e-16 absolute for |log x| < 1 (2.5 ulp in the bins next to
// 1, where that is below 5e-18), 0.81 ulp beyond, 0.63 ulp for the reciprocal; log() and a division
// have 1 and 0.5 ulp.  What enters the stress is c = mu - lambda log J, whose own rounding is as large.
// Anything outside [2^-1007, 2^1007) (zero, negative, NaN and infinite among it) goes to log() and a
// division.
constexpr int kLogBins = 128;  // tab[i] = {r, -log r}, see log_table()
// The table of log_inv: per bin of m in [0.75, 1.5) the reciprocal r of its middle (1 for the two
// bins next to 1, where log must keep its relative accuracy) and -log r.
inline std::vector<double2> log_table() {
  auto from_hi = [](uint32_t hi) {
    const uint64_t bits = (uint64_t)hi << 32;
    double x;
    std::memcpy(&x, &bits, sizeof(x));
    return x;
  };
  std::vector<double2> t(kLogBins);
  for (int i = 0; i < kLogBins; ++i) {
    const double a = from_hi(0x3fe80000u + ((uint32_t)i << 13)), b = from_hi(0x3fe80000u + ((uint32_t)(i + 1) << 13));
    const double r = (a == 1.0 || b == 1.0) ? 1.0 : (double)(2.0L / ((long double)a + (long double)b));
    t[i].x = r;
    t[i].y = (double)-std::log((long double)r);
  }
  return t;
}

struct LogInv {
  double log, inv;
};
__device__ __forceinline__ LogInv log_inv(double x, const double2* __restrict__ tab) {
  const int hi = __double2hiint(x);
  if ((unsigned)(hi - 0x01000000) >= 0x7de00000u) return {x > 0.0 ? log(x) : 0.0, 1.0 / x};
  const int q = hi - 0x3fe80000, e = q >> 20;
  const double2 c = __ldg(tab + ((q >> 13) & (kLogBins - 1)));
  const double m = __hiloint2double(hi - (e << 20), __double2loint(x));
  const double t = fma(m, c.x, -1.0), t2 = t * t;
  double p = fma(t, 1.0 / 7.0, -1.0 / 6.0);
  p = fma(t, p, 1.0 / 5.0);
  p = fma(t, p, -1.0 / 4.0);
  p = fma(t, p, 1.0 / 3.0);
  p = fma(t, p, -1.0 / 2.0);
  double l = fma(t2, p, t) + c.y;
  double r = c.x;
  if (e != 0) {
    l = fma((double)e, 0.69314718055994530942, l);
    r = __hiloint2double(__double2hiint(r) - (e << 20), __double2loint(r));  // r 2^-e, normal
  }
  const double a = 1.0 - t, y = fma(t2, a, a) * r;
  return {l, fma(y, fma(-x, y, 1.0), y)};
}

// Lame parameters of Eq. 2 and the logarithm's table.
struct NHLaw {
  double mu, lam;
  const double2* tab;
};

// F - I at a Gauss point from the displacements relative to node 0 (d[a - 1] of node a).
struct NHPoint {
  double F00, F01, F10, F11, inv, c;  // inv = 1 / J, c = mu - lambda ln J (mu where J <= 0)
  bool ok;
};
__device__ __forceinline__ NHPoint nh_point(const double* g, const double (&dx)[3], const double (&dy)[3],
                                            const NHLaw& law) {
  NHPoint p;
  p.F00 = 1.0;
  p.F01 = 0.0;
  p.F10 = 0.0;
  p.F11 = 1.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double bx = g[2 * a + 2], by = g[2 * a + 3];
    p.F00 += dx[a] * bx;
    p.F01 += dx[a] * by;
    p.F10 += dy[a] * bx;
    p.F11 += dy[a] * by;
  }
  const double det = p.F00 * p.F11 - p.F01 * p.F10;
  p.ok = det > 0.0;
  const LogInv li = log_inv(det, law.tab);
  p.inv = li.inv;
  p.c = law.mu - law.lam * li.log;
  return p;
}

__device__ __forceinline__ void nh_relative(const double u[8], double (&dx)[3], double (&dy)[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    dx[a] = u[2 * a + 2] - u[0];
    dy[a] = u[2 * a + 3] - u[1];
  }
}

// r_a = sum_q w P grad N_a with P = mu F - c F^-T
__device__ inline void nh_residual(const double* geo, const double u[8], const NHLaw& law, double r[8], bool& ok) {
  double dx[3], dy[3];
  nh_relative(u, dx, dy);
#pragma unroll
  for (int k = 0; k < 8; ++k) r[k] = 0.0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const double* g = geo + q * 10;
    const NHPoint p = nh_point(g, dx, dy, law);
    ok = ok && p.ok;
    const double mw = law.mu * g[8], cw = p.c * (p.inv * g[8]);
    const double P00 = mw * p.F00 - cw * p.F11, P01 = mw * p.F01 + cw * p.F10;
    const double P10 = mw * p.F10 + cw * p.F01, P11 = mw * p.F11 - cw * p.F00;
#pragma unroll
    for (int a = 1; a < 4; ++a) {
      const double bx = g[2 * a], by = g[2 * a + 1];
      r[2 * a] += P00 * bx;
      r[2 * a] += P01 * by;
      r[2 * a + 1] += P10 * bx;
      r[2 * a + 1] += P11 * by;
    }
  }
  r[0] = -(r[2] + r[4] + r[6]);
  r[1] = -(r[3] + r[5] + r[7]);
}

// The element tangent of Eq. 2, K[a][b] the 2 x 2 block of nodes a <= b, row-major (K[b][a] is its
// transpose): blocks of nodes 1 .. 3 from the Gauss points, those of node 0 from the sums.
struct NHTangent {
  double K[10][4];  // (0,0) (0,1) (0,2) (0,3) (1,1) (1,2) (1,3) (2,2) (2,3) (3,3)
  static __host__ __device__ constexpr int at(int a, int b) { return a * 4 - a * (a - 1) / 2 + (b - a); }
  // entry (a, i), (b, k) for any order of the nodes
  __device__ __forceinline__ double operator()(int a, int i, int b, int k) const {
    return a <= b ? K[at(a, b)][2 * i + k] : K[at(b, a)][2 * k + i];
  }
};

__device__ inline void nh_tangent(const double* geo, const double u[8], const NHLaw& law, NHTangent& T) {
  double dx[3], dy[3];
  nh_relative(u, dx, dy);
  double gg[3][3];  // sum_q w mu grad N_a . grad N_b, on the diagonal of the blocks
#pragma unroll
  for (int a = 1; a < 4; ++a)
#pragma unroll
    for (int b = a; b < 4; ++b) {
      gg[a - 1][b - 1] = 0.0;
#pragma unroll
      for (int k = 0; k < 4; ++k) T.K[NHTangent::at(a, b)][k] = 0.0;
    }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const double* g = geo + q * 10;
    const NHPoint p = nh_point(g, dx, dy, law);
    const double w = g[8], mw = law.mu * w, lw = law.lam * w, cw = p.c * w, sw = lw + cw;
    const double i00 = p.F11 * p.inv, i01 = -p.F01 * p.inv, i10 = -p.F10 * p.inv, i11 = p.F00 * p.inv;
    double p0[3], p1[3];  // F^-1 from the left on grad N_a
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      p0[a] = g[2 * a + 2] * i00 + g[2 * a + 3] * i10;
      p1[a] = g[2 * a + 2] * i01 + g[2 * a + 3] * i11;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double s0 = sw * p0[a], s1 = sw * p1[a], l0 = lw * p0[a], l1 = lw * p1[a], c0 = cw * p0[a], c1 = cw * p1[a];
      const double mx = mw * g[2 * a + 2], my = mw * g[2 * a + 3];
#pragma unroll
      for (int b = a; b < 3; ++b) {
        double(&K)[4] = T.K[NHTangent::at(a + 1, b + 1)];
        gg[a][b] += mx * g[2 * b + 2];
        gg[a][b] += my * g[2 * b + 3];
        K[0] += s0 * p0[b];
        K[3] += s1 * p1[b];
        if (a == b) {
          K[1] += s0 * p1[b];
        } else {
          K[1] += l0 * p1[b];
          K[1] += c1 * p0[b];
          K[2] += l1 * p0[b];
          K[2] += c0 * p1[b];
        }
      }
    }
  }
#pragma unroll
  for (int a = 1; a < 4; ++a)
#pragma unroll
    for (int b = a; b < 4; ++b) {
      double(&K)[4] = T.K[NHTangent::at(a, b)];
      K[0] += gg[a - 1][b - 1];
      K[3] += gg[a - 1][b - 1];
      if (a == b) K[2] = K[1];
    }
#pragma unroll
  for (int b = 1; b < 4; ++b)
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int k = 0; k < 2; ++k) T.K[NHTangent::at(0, b)][2 * i + k] = -(T(1, i, b, k) + T(2, i, b, k) + T(3, i, b, k));
  T.K[0][0] = -(T(0, 0, 1, 0) + T(0, 0, 2, 0) + T(0, 0, 3, 0));
  T.K[0][1] = T.K[0][2] = -(T(0, 0, 1, 1) + T(0, 0, 2, 1) + T(0, 0, 3, 1));
  T.K[0][3] = -(T(0, 1, 1, 1) + T(0, 1, 2, 1) + T(0, 1, 3, 1));
}

// ------------------------------------------------------------------------------------------
// Band LU without pivoting.  Rows of the matrix come from a CSR block (columns are table dof
// indices; only columns < n belong to the local matrix) or from a dense band array.
// Factor layout (row-major band, W = 2b + 1 entries per row): d < b holds L[i][i-b+d],
// d = b holds 1 / U[i][i], d > b holds U[i][i+d-b].
// ------------------------------------------------------------------------------------------
struct RowSource {
  const int32_t* rowptr;  // nullptr: dense band rows in `val` (W entries per row)
  const int32_t* colidx;
  const double* val;
};

template <typename FT>
__device__ inline void load_band_row_warp(int row, int n, int b, const RowSource& src, FT* dst) {
  const int W = 2 * b + 1, lane = threadIdx.x & 31;
  if (src.rowptr == nullptr) {
    for (int d = lane; d < W; d += 32) dst[d] = (row < n) ? (FT)src.val[(int64_t)row * W + d] : (FT)0;
    __syncwarp();
    return;
  }
  for (int d = lane; d < W; d += 32) dst[d] = (FT)0;
  __syncwarp();
  if (row < n) {
    const int k1 = src.rowptr[row + 1];
    for (int k = src.rowptr[row] + lane; k < k1; k += 32) {
      const int col = src.colidx[k];
      if (col < n) dst[col - row + b] = (FT)src.val[k];
    }
  }
  __syncwarp();
}

// Returns (to every thread) 0 on success, 1 if a pivot was zero or not finite.
// smem: win [(b + 2) * (2b + 1)], rp [b + 2], flag [1].
template <typename FT>
__device__ int band_lu(int n, int b, const RowSource& src, FT* __restrict__ F, FT* win, FT* rp, int* flag) {
  const int W = 2 * b + 1, R = b + 2;
  const int tid = threadIdx.x, T = blockDim.x, wid = tid >> 5, nw = T >> 5;
  if (n <= 0) return 0;
  if (tid == 0) *flag = 0;
  // rows 0..b into slots 0..b
  for (int i = wid; i <= b; i += nw) load_band_row_warp<FT>(i, n, b, src, win + (i % R) * W);
  __syncthreads();
  if (tid == 0) {
    const FT p = win[b];
    if (!(p != (FT)0) || !isfinite((double)p)) *flag = 1;
    rp[0] = (FT)1 / p;
  }
  __syncthreads();
  const int bb = b * b;
  const int dq = (b > 0) ? T / b : 0, dr = (b > 0) ? T % b : 0;
  const int ri0 = (b > 0) ? tid / b : 0, cj0 = (b > 0) ? tid % b : 0;
  for (int k = 0; k < n; ++k) {
    const int sk = k % R;
    const FT* rowk = win + sk * W;
    const FT rpk = rp[sk];
    const int lim = min(b, n - 1 - k);
    // warp 0: write back row k (scaled L part, reciprocal pivot) and stage row k + b + 1
    if (wid == 0) {
      FT* out = F + (int64_t)k * W;
      for (int d = tid; d < W; d += 32) {
        const int j = k - b + d;
        FT v = rowk[d];
        if (d < b) v = (j >= 0) ? v * rp[j % R] : (FT)0;
        else if (d == b) v = rpk;
        out[d] = v;
      }
      load_band_row_warp<FT>(k + b + 1, n, b, src, win + ((k + b + 1) % R) * W);
    }
    // rank-1 update of rows k+1..k+lim, columns k+1..k+lim
    if (lim > 0) {
      const int base = (k + 1) % R;
      int ri = ri0, cj = cj0;
      for (int idx = tid; idx < bb; idx += T) {
        if (ri < lim && cj < lim) {
          int slot = base + ri;
          if (slot >= R) slot -= R;
          FT* rowi = win + slot * W;
          const FT l = rowi[b - 1 - ri] * rpk;
          const FT nv = rowi[cj - ri + b] - l * rowk[b + 1 + cj];
          rowi[cj - ri + b] = nv;
          if (idx == 0) {
            if (!(nv != (FT)0) || !isfinite((double)nv)) *flag = 1;
            rp[(k + 1) % R] = (FT)1 / nv;
          }
        }
        cj += dr;
        ri += dq;
        if (cj >= b) {
          cj -= b;
          ri += 1;
        }
      }
    } else if (tid == 0 && k + 1 < n) {
      const FT nv = win[((k + 1) % R) * W + b];
      if (!(nv != (FT)0) || !isfinite((double)nv)) *flag = 1;
      rp[(k + 1) % R] = (FT)1 / nv;
    }
    __syncthreads();
  }
  return *flag;
}

// ------------------------------------------------------------------------------------------
// In-place band LU by square tiles.  F holds the assembled band rows on entry (row-major,
// W = 2b + 1) and the factors on exit (layout as above).
//
// What bounds it: the chain of pivots (a reciprocal, a product and an update per pivot), and what
// every elimination step costs besides.  One step per pivot with a CTA barrier, a shared-memory
// load and a store per updated entry costs 1400 (b = 42) to 2600 cycles (b = 83) in FP32.  Here NB
// pivots are eliminated per panel with two barriers:
//   A  one thread per row (column) finishes the panel's L (U) tiles in registers;
//   B  warp 0 updates the next diagonal tile and factors it, while the other warps fetch the tiles
//      that enter with the next panel (cp.async), apply the NB rank-1 updates to the trailing
//      tiles with one load and one store per entry (G x G entries per lane, 16-byte loads), and
//      write the finished tiles out.
// Every entry still receives its updates one pivot after the other in ascending order, each one
// fused multiply-add with the multiplier rounded before it, so the FP32 factors are bit for bit
// those of the step-by-step elimination.  Factorization with packing, one CTA per SM, before and
// now: n = 1598, b = 42, FP32 1.06 ms (128 threads) -> 0.39 ms (256 threads); n = 3120, b = 83, FP32
// 3.9 -> 1.0 ms (512 threads); n = 2520, b = 75, FP64 8.8 -> 5.9 ms (4.6 ms of it FP64 instructions at
// the part's rate).
//
// The window holds the active tiles: tile (I, J) of the matrix sits in slot (I mod RT, J mod RT),
// RT = tb + 2 with tb = ceil(b / NB) -- the tb + 1 tile rows and columns a panel touches, and the
// ones entering with the next panel (RT = tb + 1 and no copy ahead where that does not fit).  Tile
// entries outside the band are exact zeros and stay zero; rows past n hold the identity.  A tile
// row is 64 bytes: its 16-byte groups are permuted by the row pair, and the rows of a pair swapped
// in odd slot columns, so that the vector loads of rows and of columns across two neighbouring
// tiles hit distinct banks.
// ------------------------------------------------------------------------------------------
template <typename FT>
__device__ inline void cp_async_elem(FT* sdst, const FT* gsrc) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(sdst);
  if (sizeof(FT) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gsrc) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gsrc) : "memory");
}
__device__ inline void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ inline void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Entries per 16-byte group, and rows of a tile: 16 in FP32, 8 in FP64 (64-byte tile rows).
template <typename FT>
struct LuTile {
  static constexpr int G = 16 / (int)sizeof(FT);
  static constexpr int NB = 4 * G;
  static constexpr int TE = NB * NB;
};

// Tiles of half a band, and window entries of the tiled band LU (the tiles, with the next panel's
// for ahead = 1, and the transposed multipliers of one diagonal tile).
template <typename FT>
__host__ __device__ constexpr int band_lu_half(int b) {
  return b > 0 ? (b + LuTile<FT>::NB - 1) / LuTile<FT>::NB : 1;
}
template <typename FT>
__host__ __device__ constexpr size_t band_lu_window(int b, int ahead) {
  const size_t rt = (size_t)(band_lu_half<FT>(b) + 1 + ahead);
  return (rt * rt + 1) * LuTile<FT>::TE;
}

// Rows and row stride of a (b + 10)-row window: the size that the limits on the half bandwidth and
// on the subdomain size are stated for (no tiled window that such a window allows is larger).
__host__ __device__ constexpr int band_limit_rows(int b) { return b + 10; }
__host__ __device__ constexpr int band_limit_stride(int b) {
  int w = 2 * b + 1;
  while (((w - 1) & 31) != 8 && ((w - 1) & 31) != 24) ++w;
  return w;
}

// 1 / p.  FP64: from the FP32 reciprocal (relative error e < 2^-23) by r (1 + e + e^2), three FP64
// instructions at about 70 cycles each instead of a division; the next term of the series is below
// 2^-69, so that only the last rounding is left (0.50 ulp on the arguments above).
template <typename FT>
__device__ inline FT recip(FT p) {
  if constexpr (sizeof(FT) == 4) {
    return __frcp_rn(p);
  } else {
    const unsigned e = ((unsigned)__double2hiint(p) >> 20) & 0x7ff;
    if (e - 923u >= 200u) return (FT)1 / p;  // outside [2^-100, 2^100): no FP32 value to start from
    const double r = (double)__frcp_rn((float)p), err = fma(-p, r, 1.0);
    return fma(r, fma(err, err, err), r);
  }
}
// Zero, infinite or NaN, without floating-point instructions.
__device__ inline bool bad_pivot(float p) {
  const unsigned u = __float_as_uint(p) & 0x7fffffffu;
  return u == 0 || u >= 0x7f800000u;
}
__device__ inline bool bad_pivot(double p) {
  const unsigned h = (unsigned)__double2hiint(p) & 0x7fffffffu;
  return (h | (unsigned)__double2loint(p)) == 0 || h >= 0x7ff00000u;
}

// f(integral_constant<int, I>) for I = I0 .. N - 1: a loop whose index is a constant in its body
template <int I, int N, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

template <typename FT>
struct alignas(16) LuVec {
  FT v[LuTile<FT>::G];
};

// Returns (to every thread) 0 on success, 1 if a pivot was zero or not finite.  `flag`: three ints
// of shared memory.  `win`: at least
// band_lu_window<FT>(b, 0) entries, 16-byte aligned, win_cap of them usable.  blockDim.x: a
// multiple of 32, at least 64.
template <typename FT>
__device__ __noinline__ int band_lu_at(int n, int b, FT* __restrict__ F, uint32_t win_off, size_t win_cap,
                                        uint32_t flag_off) {
  FT* const win = (FT*)(dyn_smem + win_off);
  int* const flag = (int*)(dyn_smem + flag_off);
  constexpr int G = LuTile<FT>::G, NB = LuTile<FT>::NB, TE = LuTile<FT>::TE;
  constexpr int RH = 32 / NB;       // tile rows a warp covers with one entry per lane
  constexpr int C = NB * NB / 32;   // entries per lane of a tile spread over a warp
  using Vec = LuVec<FT>;
  if (n <= 0) return 0;
  int* const s_task = flag + 1;  // two task counters, used in turn
  const int W = 2 * b + 1, tb = band_lu_half<FT>(b), NP = (n + NB - 1) / NB;
  const bool ahead = band_lu_window<FT>(b, 1) <= win_cap;
  const int RT = tb + 1 + (ahead ? 1 : 0);
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = T >> 5;
  FT* const dt = win + RT * RT * TE;  // dt[k NB + i]: multiplier l_ik of the current diagonal tile
  auto tile = [&](int si, int sj) { return win + (si * RT + sj) * TE; };
  // entry (r, c) of a tile in slot column sj; c a multiple of G for vector access
  auto at = [](int r, int c, int sj) {
    return ((r ^ (sj & 1)) * 4 + (((c / G) ^ (r >> 1)) & 3)) * G + c % G;
  };
  auto wrap = [&](int s) { return s >= RT ? s - RT : s; };  // slot index < 2 RT into the ring
  // one warp copies tile (I, J) into slots (si, sj): lane (r0, c) rows r0, r0 + RH, ..
  const int lr = lane / NB, lc = lane % NB;
  auto fetch = [&](int I, int J, int si, int sj) {
    FT* t = tile(si, sj);
    const int i0 = I * NB + lr, j = J * NB + lc, d0 = j - i0 + b;
    const FT* src = F + ((int64_t)i0 * W + d0);
    const bool jn = j < n;
#pragma unroll
    for (int q = 0; q < NB / RH; ++q) {
      FT* dst = t + at(lr + q * RH, lc, sj);
      const int i = i0 + q * RH;
      if (jn && i < n && (unsigned)(d0 - q * RH) < (unsigned)W) cp_async_elem<FT>(dst, src + q * RH * (int64_t)(W - 1));
      else *dst = (i == j) ? (FT)1 : (FT)0;
    }
  };
  // the q-th of the 2 tb + 1 tiles that enter with tile row and column h (in slot sh): (h, h - tb ..
  // h), then (h - tb .. h - 1, h)
  auto enter = [&](int q, int h, int sh) {
    const int back = q <= tb ? tb - q : 2 * tb + 1 - q;
    if (back > h) return;
    const int so = sh - back < 0 ? sh - back + RT : sh - back;
    if (q <= tb) fetch(h, h - back, sh, so);
    else fetch(h - back, h, so, sh);
  };
  // one warp writes the tile (I, J) of slots (si, sj) out
  auto emit = [&](int I, int J, int si, int sj) {
    const FT* t = tile(si, sj);
    const int i0 = I * NB + lr, j = J * NB + lc, d0 = j - i0 + b;
    FT* dst = F + ((int64_t)i0 * W + d0);
    const bool jn = j < n;
    FT v[NB / RH];
#pragma unroll
    for (int q = 0; q < NB / RH; ++q) v[q] = t[at(lr + q * RH, lc, sj)];
#pragma unroll
    for (int q = 0; q < NB / RH; ++q)
      if (jn && i0 + q * RH < n && (unsigned)(d0 - q * RH) < (unsigned)W) dst[q * RH * (int64_t)(W - 1)] = v[q];
  };
  // warp 0 factors the diagonal tile in slot s: lane (r, h) = (lane % NB, lane / NB) holds row r,
  // columns h C .. h C + C - 1; pivot rows and columns by shuffles
  auto factor = [&](int s) {
    FT* D = tile(s, s);
    const int r = lane % NB, h = lane / NB;
    FT a[C];
#pragma unroll
    for (int g = 0; g < C; g += G) {
      const Vec v = *(const Vec*)(D + at(r, h * C + g, s));
#pragma unroll
      for (int q = 0; q < G; ++q) a[g + q] = v.v[q];
    }
    bool bad = false;
    static_for<0, NB>([&](auto kc) {
      constexpr int k = decltype(kc)::value, hk = k / C, kj = k % C, j0 = hk == NB / C - 1 ? kj + 1 : 0;
      const FT p = __shfl_sync(0xffffffffu, a[kj], k + NB * hk);
      const FT x = __shfl_sync(0xffffffffu, a[kj], r + NB * hk);
      FT u[C];
#pragma unroll
      for (int j = j0; j < C; ++j) u[j] = __shfl_sync(0xffffffffu, a[j], k + NB * h);
      const FT rp = recip<FT>(p);
      bad |= bad_pivot(p);
      const FT l = x * rp;
#pragma unroll
      for (int j = j0; j < C; ++j) {
        const FT y = a[j] - l * u[j];
        a[j] = (r > k && h * C + j > k) ? y : a[j];
      }
      if (h == hk) a[kj] = r > k ? l : (r == k ? rp : a[kj]);
    });
#pragma unroll
    for (int g = 0; g < C; g += G) {
      Vec v;
#pragma unroll
      for (int q = 0; q < G; ++q) v.v[q] = a[g + q];
      *(Vec*)(D + at(r, h * C + g, s)) = v;
    }
#pragma unroll
    for (int j = 0; j < C; ++j) dt[(h * C + j) * NB + r] = a[j];
    if (bad && lane == 0) *flag = 1;
  };
  if (tid == 0) *flag = 0, s_task[0] = s_task[1] = 0;
  for (int h = 0; h <= tb && h < NP; ++h)
    for (int q = wid; q < 2 * tb + 1; q += nw) enter(q, h, h);
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  if (wid == 0) factor(0);
  __syncthreads();
  int sK = 0;
  for (int K = 0; K < NP; ++K) {
    FT* D = tile(sK, sK);
    const int s1 = wrap(sK + 1);
    // A: L tiles (I, K) row by row, U tiles (K, J) column by column
    const int half = (tb * NB + 31) & ~31;  // a warp takes rows or columns, not both
    for (int idx = tid; idx < 2 * half; idx += T) {
      const bool lower = idx < half;
      const int q = lower ? idx : idx - half;
      const int o = q / NB, x = q % NB;  // tile K + 1 + o, row or column x
      if (o >= tb || K + 1 + o >= NP) continue;
      const int so = wrap(s1 + o);
      FT a[NB];
      if (lower) {
        FT* L = tile(so, sK);
#pragma unroll
        for (int g = 0; g < NB; g += G) {
          const Vec v = *(const Vec*)(L + at(x, g, sK));
#pragma unroll
          for (int i = 0; i < G; ++i) a[g + i] = v.v[i];
        }
#pragma unroll
        for (int k = 0; k < NB; ++k) {
#pragma unroll
          for (int g = k / G * G; g < NB; g += G) {
            const Vec v = *(const Vec*)(D + at(k, g, sK));
#pragma unroll
            for (int i = 0; i < G; ++i) {
              if (g + i == k) a[k] *= v.v[i];
              else if (g + i > k) a[g + i] -= a[k] * v.v[i];
            }
          }
        }
#pragma unroll
        for (int g = 0; g < NB; g += G) {
          Vec v;
#pragma unroll
          for (int i = 0; i < G; ++i) v.v[i] = a[g + i];
          *(Vec*)(L + at(x, g, sK)) = v;
        }
      } else {
        FT* U = tile(sK, so);
#pragma unroll
        for (int k = 0; k < NB; ++k) a[k] = U[at(k, x, so)];
#pragma unroll
        for (int k = 0; k < NB; ++k) {
#pragma unroll
          for (int g = (k + 1) / G * G; g < NB; g += G) {
            const Vec v = *(const Vec*)(dt + k * NB + g);
#pragma unroll
            for (int i = 0; i < G; ++i)
              if (g + i > k) a[g + i] -= v.v[i] * a[k];
          }
        }
#pragma unroll
        for (int k = 1; k < NB; ++k) U[at(k, x, so)] = a[k];
      }
    }
    if (tid == 0) s_task[(K + 1) & 1] = 0;
    __syncthreads();
    // B
    if (wid == 0 && K + 1 < NP) {
      // the next diagonal tile: C entries per lane
      constexpr int RL = C / G;  // rows per lane
      FT* O = tile(s1, s1);
      const FT *L = tile(s1, sK), *U = tile(sK, s1);
      const int r0 = (lane >> 2) * RL, c0 = (lane & 3) * G;
      Vec acc[RL];
#pragma unroll
      for (int i = 0; i < RL; ++i) acc[i] = *(const Vec*)(O + at(r0 + i, c0, s1));
#pragma unroll
      for (int k = 0; k < NB; k += G) {
        Vec l[RL], v[G];
#pragma unroll
        for (int i = 0; i < RL; ++i) l[i] = *(const Vec*)(L + at(r0 + i, k, sK));
#pragma unroll
        for (int i = 0; i < G; ++i) v[i] = *(const Vec*)(U + at(k + i, c0, s1));
#pragma unroll
        for (int q = 0; q < G; ++q)
#pragma unroll
          for (int i = 0; i < RL; ++i)
#pragma unroll
            for (int j = 0; j < G; ++j) acc[i].v[j] -= l[i].v[q] * v[q].v[j];
      }
#pragma unroll
      for (int i = 0; i < RL; ++i) *(Vec*)(O + at(r0 + i, c0, s1)) = acc[i];
      __syncwarp();
      factor(s1);
    }
    // tiles that enter, trailing updates, finished tiles out: handed out to the warps in that order
    const int n_in = (ahead && K + tb + 1 < NP) ? 2 * tb + 1 : 0, pairs = (tb + 1) / 2;
    const int n_up = K + 1 < NP ? tb * pairs : 0, n_task = n_in + n_up + 2 * tb + 1;
    for (;;) {
      int task = 0;
      if (lane == 0) task = atomicAdd(&s_task[K & 1], 1);
      task = __shfl_sync(0xffffffffu, task, 0);
      if (task >= n_task) break;
      if (task < n_in) {
        enter(task, K + tb + 1, sK == 0 ? RT - 1 : sK - 1);
      } else if (task < n_in + n_up) {
        // one tile row by two tile columns, G x G entries per lane
        const int u = task - n_in, oi = u / pairs, oj = 2 * (u % pairs) + ((lane & 7) >> 2);
        if (oj >= tb || K + 1 + oi >= NP || K + 1 + oj >= NP || (oi == 0 && oj == 0)) continue;
        const int si = wrap(s1 + oi), sj = wrap(s1 + oj);
        const int r0 = (lane >> 3) * G, c0 = (lane & 3) * G;
        FT* O = tile(si, sj);
        const FT *L = tile(si, sK), *U = tile(sK, sj);
        Vec acc[G];
#pragma unroll
        for (int i = 0; i < G; ++i) acc[i] = *(const Vec*)(O + at(r0 + i, c0, sj));
        // pivots before the first one whose row or column reaches this tile contribute zeros
        const int kb = max(0, (max(oi, 2 * (u % pairs)) + 1) * NB - b) / G * G;
#pragma unroll
        for (int k = 0; k < NB; k += G) {
          if (k < kb) continue;
          Vec l[G], v[G];
#pragma unroll
          for (int i = 0; i < G; ++i) l[i] = *(const Vec*)(L + at(r0 + i, k, sK));
#pragma unroll
          for (int i = 0; i < G; ++i) v[i] = *(const Vec*)(U + at(k + i, c0, sj));
#pragma unroll
          for (int q = 0; q < G; ++q)
#pragma unroll
            for (int i = 0; i < G; ++i)
#pragma unroll
              for (int j = 0; j < G; ++j) acc[i].v[j] -= l[i].v[q] * v[q].v[j];
        }
#pragma unroll
        for (int i = 0; i < G; ++i) *(Vec*)(O + at(r0 + i, c0, sj)) = acc[i];
      } else {
        const int q = task - n_in - n_up, o = q <= tb ? q : q - tb;  // (K + o, K), then (K, K + o)
        if (K + o >= NP) continue;
        if (q <= tb) emit(K + o, K, wrap(sK + o), sK);
        else emit(K, K + o, sK, wrap(sK + o));
      }
    }
    if (!ahead) {
      __syncthreads();  // slot K is free: the next panel's last row and column take it
      if (K + tb + 1 < NP)
        for (int q = wid; q < 2 * tb + 1; q += nw) enter(q, K + tb + 1, sK);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    sK = s1;
  }
  return *flag;
}
template <typename FT>
__device__ __forceinline__ int band_lu_inplace(int n, int b, FT* F, FT* win, size_t win_cap, int* flag) {
  return band_lu_at<FT>(n, b, F, dyn_offset(win), win_cap, dyn_offset(flag));
}

// ------------------------------------------------------------------------------------------
// Triangular solves with the band factors, in place on y[0..n) (shared memory).
// ------------------------------------------------------------------------------------------
// Block size of the triangular solves: 32 rows (one warp) for FP32 factors, 16 for FP64
// (two register sets of BS values per thread stay within the register budget).
template <typename FT>
struct SolveBlock {
  static constexpr int BS = sizeof(FT) == 4 ? 32 : 16;
};

// The factor values of block k0 + BS are loaded into registers while block k0 is solved, so
// the global-memory latency of the next block overlaps the current one.
//
// Roles: warp 0 solves the BS x BS diagonal block; threads 32 .. 32 + b - 1 each own one of the
// b rows coupled to the block.  Both roles keep their current and next values in the same two
// register arrays (Dcur/Dnxt), so a thread holds 2 BS values.  Needs blockDim.x >= 32 + b.
template <typename FT>
__device__ void band_solve(int n, int b, const FT* __restrict__ F, FT* y) {
  constexpr int BS = SolveBlock<FT>::BS;
  const int W = 2 * b + 1, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const bool diag = wid == 0;
  const bool offd = tid >= 32 && tid < 32 + b;
  const int r = tid - 32;
  FT cur[BS], nxt[BS];
  // forward (unit lower L): block k0 = rows [k0, k0 + kb)
#define NLS_LOAD_FWD(k0_, R_)                                                             \
  {                                                                                       \
    const int kb_ = min(BS, n - (k0_));                                                   \
    if (diag) {                                                                           \
      _Pragma("unroll") for (int j = 0; j < BS; ++j) {                                    \
        const int d = j - lane + b;                                                       \
        R_[j] = (j < lane && lane < kb_ && d >= 0) ? F[(int64_t)((k0_) + lane) * W + d] : (FT)0; \
      }                                                                                   \
    } else if (offd) {                                                                    \
      const int i_ = (k0_) + kb_ + r;                                                     \
      _Pragma("unroll") for (int j = 0; j < BS; ++j) {                                    \
        const int d = j + b - kb_ - r;                                                    \
        R_[j] = (i_ < n && j < kb_ && d >= 0) ? F[(int64_t)i_ * W + d] : (FT)0;           \
      }                                                                                   \
    }                                                                                     \
  }
  if (n > 0) NLS_LOAD_FWD(0, cur);
  for (int k0 = 0; k0 < n; k0 += BS) {
    const int kb = min(BS, n - k0);
    if (k0 + BS < n) NLS_LOAD_FWD(k0 + BS, nxt);
    if (diag) {
      FT yl = (lane < kb) ? y[k0 + lane] : (FT)0;
#pragma unroll
      for (int j = 0; j < BS; ++j) {
        const FT yj = __shfl_sync(0xffffffffu, yl, j);
        if (j < kb) yl -= cur[j] * yj;
      }
      if (lane < kb) y[k0 + lane] = yl;
    }
    __syncthreads();
    if (offd) {
      const int i = k0 + kb + r;
      if (i < n) {
        FT acc = 0;
#pragma unroll
        for (int j = 0; j < BS; ++j)
          if (j < kb) acc += cur[j] * y[k0 + j];
        y[i] -= acc;
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < BS; ++j) cur[j] = nxt[j];
  }
#undef NLS_LOAD_FWD
  // backward (U, diagonal stored inverted): block rows [k0, k1)
#define NLS_LOAD_BWD(k1_, R_)                                                             \
  {                                                                                       \
    const int k0_ = max(0, (k1_) - BS), kb_ = (k1_) - k0_;                                \
    if (diag) {                                                                           \
      _Pragma("unroll") for (int j = 0; j < BS; ++j) {                                    \
        const int d = j - lane + b;                                                       \
        R_[j] = (j >= lane && lane < kb_ && j < kb_ && d <= 2 * b) ? F[(int64_t)(k0_ + lane) * W + d] : (FT)0; \
      }                                                                                   \
    } else if (offd) {                                                                    \
      const int i_ = k0_ - 1 - r;                                                         \
      _Pragma("unroll") for (int j = 0; j < BS; ++j) {                                    \
        R_[j] = (i_ >= 0 && j < kb_ && j + 1 + r <= b) ? F[(int64_t)i_ * W + (j + 1 + r + b)] : (FT)0; \
      }                                                                                   \
    }                                                                                     \
  }
  if (n > 0) NLS_LOAD_BWD(n, cur);
  for (int k1 = n; k1 > 0; k1 -= BS) {
    const int k0 = max(0, k1 - BS), kb = k1 - k0;
    if (k0 > 0) NLS_LOAD_BWD(k0, nxt);
    if (diag) {
      FT yl = (lane < kb) ? y[k0 + lane] : (FT)0;
#pragma unroll
      for (int j = BS - 1; j >= 0; --j) {
        if (j < kb) {
          FT xj = (lane == j) ? yl * cur[j] : (FT)0;
          xj = __shfl_sync(0xffffffffu, xj, j);
          if (lane == j) yl = xj;
          else if (lane < j) yl -= cur[j] * xj;
        }
      }
      if (lane < kb) y[k0 + lane] = yl;
    }
    __syncthreads();
    if (offd) {
      const int i = k0 - 1 - r;
      if (i >= 0) {
        FT acc = 0;
#pragma unroll
        for (int j = 0; j < BS; ++j)
          if (j < kb) acc += cur[j] * y[k0 + j];
        y[i] -= acc;
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < BS; ++j) cur[j] = nxt[j];
  }
#undef NLS_LOAD_BWD
}

// ------------------------------------------------------------------------------------------
// Packed solve operands.  After a factorization the operands of the two triangular solves are
// copied, block by block (BS rows), into rows of BS entries = 128 bytes, one per row that the block
// solves or couples to:
//
//   block t (rows k0 = t BS .. k0 + bs - 1), PB = 2 BS^2 + 2 b BS entries:
//     [0, BS^2)               inv(L_tt): row r holds inv(L_tt)[r][j], j < BS (identity padded)
//     [BS^2, 2 BS^2)          inv(U_tt) likewise (U's diagonal is stored inverted)
//     [2 BS^2, + b BS)        CL: row r holds L[k0 + BS + r][k0 + j]
//     [2 BS^2 + b BS, + b BS) CU: row r holds U[k0 - 1 - r][k0 + j]
//
// The thread that owns a row reads it as eight 16-byte groups; group g of row r is stored at position
// g ^ (r mod 8), so that eight threads reading their rows from shared memory touch all banks.  (With
// the rows along the threads instead, one 4-byte load per term, a solve step issued 64 loads on its
// critical warp, and packing had to transpose everything.)
//
// The explicit diagonal-block inverses replace the BS-step dependent shuffle chain of a
// diagonal block by one short dot product per row.  One warp per block; `tmp` (16-byte aligned)
// holds pack_scratch<FT>() entries per warp that takes part (`nwarps`).
// ------------------------------------------------------------------------------------------
template <typename FT>
__host__ __device__ constexpr int64_t packed_block_entries(int b) {
  return 2 * (int64_t)SolveBlock<FT>::BS * SolveBlock<FT>::BS + 2 * (int64_t)b * SolveBlock<FT>::BS;
}
// Position of entry j of row r within the row.
template <typename FT>
__host__ __device__ constexpr int packed_at(int r, int j) {
  return (((j / LuTile<FT>::G) ^ (r & 7)) * LuTile<FT>::G) + j % LuTile<FT>::G;
}

// Rows of the scratch: padded to whole 16-byte groups, with the column writes of a warp spread over
// the banks.
template <typename FT>
__host__ __device__ constexpr int pack_stride() {
  return SolveBlock<FT>::BS + LuTile<FT>::G;
}
template <typename FT>
__host__ __device__ constexpr size_t pack_scratch() {
  return (size_t)SolveBlock<FT>::BS * pack_stride<FT>();
}

// Blocks t = first + wid, first + wid + stride, ... are packed by warp `wid` (< nwarps); one CTA
// packing everything passes first = 0, stride = nwarps, several CTAs pass their own offsets.
template <typename FT>
__device__ void band_pack_solve_range(int n, int b, const FT* __restrict__ F, FT* __restrict__ P, FT* tmp, int nwarps,
                                      int first, int stride) {
  constexpr int BS = SolveBlock<FT>::BS, G = LuTile<FT>::G, LD = pack_stride<FT>(), E = BS * BS / 32, H = 32 / BS;
  using Vec = LuVec<FT>;
  const int W = 2 * b + 1, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nblk = (n + BS - 1) / BS;
  const int64_t PB = packed_block_entries<FT>(b);
  if (wid < nwarps) {
    FT* M = tmp + wid * BS * LD;
    const int hi = lane / BS, lo = lane % BS;  // a warp covers H rows of BS entries at once
    for (int t = first + wid; t < nblk; t += stride) {
      const int k0 = t * BS, bs = min(BS, n - k0);
      FT* out = P + (int64_t)t * PB;
      FT vu[E];  // U_tt (its diagonal stored inverted), entry (i, j) = (q H + hi, lo)
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const int i = q * H + hi, j = lo;
        const bool in = i < bs && j < bs && i - j <= b && j - i <= b;
        const FT v = in ? F[(int64_t)(k0 + i) * W + (j - i + b)] : (i == j) ? (FT)1 : (FT)0;
        M[lo * LD + i] = (j < i) ? v : (FT)0;  // L_tt, transposed
        vu[q] = (j < i) ? (FT)0 : v;
      }
      __syncwarp();
      FT x[BS];
      // column `lane` of inv(L) (lanes past BS repeat one): forward substitution with e_lane, each
      // unknown taken out of all later rows at once
#pragma unroll
      for (int i = 0; i < BS; ++i) x[i] = (i == lo) ? (FT)1 : (FT)0;
#pragma unroll
      for (int j = 0; j < BS - 1; ++j)
#pragma unroll
        for (int g = (j + 1) / G * G; g < BS; g += G) {
          const Vec v = *(const Vec*)(M + j * LD + g);
#pragma unroll
          for (int i = 0; i < G; ++i)
            if (g + i > j) x[g + i] -= v.v[i] * x[j];
        }
      __syncwarp();
      if (lane < BS) {
#pragma unroll
        for (int i = 0; i < BS; ++i) out[i * BS + packed_at<FT>(i, lane)] = x[i];
      }
#pragma unroll
      for (int q = 0; q < E; ++q) M[(q * H + hi) * LD + lo] = vu[q];
      __syncwarp();
      // column `lane` of inv(U): backward substitution with e_lane, row by row
#pragma unroll
      for (int i = BS - 1; i >= 0; --i) {
        FT acc = (i == lo) ? (FT)1 : (FT)0, diag = (FT)0;
#pragma unroll
        for (int g = i / G * G; g < BS; g += G) {
          const Vec v = *(const Vec*)(M + i * LD + g);
#pragma unroll
          for (int j = 0; j < G; ++j) {
            if (g + j == i) diag = v.v[j];
            else if (g + j > i) acc -= v.v[j] * x[g + j];
          }
        }
        x[i] = acc * diag;
      }
      __syncwarp();
      if (lane < BS) {
#pragma unroll
        for (int i = 0; i < BS; ++i) out[BS * BS + i * BS + packed_at<FT>(i, lane)] = x[i];
      }
      // couplings: rows of the band become rows of the operands
      FT* cl = out + 2 * BS * BS;
      FT* cu = cl + (int64_t)b * BS;
      const bool jn = lo < bs;
      for (int r0 = 0; r0 < b; r0 += 8 * H) {
        FT vl[8], vc[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int r = r0 + q * H + hi, j = lo;
          const int il = k0 + BS + r, dl = j - BS - r + b, iu = k0 - 1 - r, du = j + 1 + r + b;
          vl[q] = (jn && r < b && il < n && dl >= 0) ? F[(int64_t)il * W + dl] : (FT)0;
          vc[q] = (jn && r < b && iu >= 0 && du <= 2 * b) ? F[(int64_t)iu * W + du] : (FT)0;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int r = r0 + q * H + hi;
          if (r < b) {
            cl[(int64_t)r * BS + packed_at<FT>(r, lo)] = vl[q];
            cu[(int64_t)r * BS + packed_at<FT>(r, lo)] = vc[q];
          }
        }
      }
    }
  }
  __syncthreads();
}

template <typename FT>
__device__ __noinline__ void band_pack_at(int n, int b, const FT* __restrict__ F, FT* __restrict__ P, uint32_t tmp_off,
                                          int nwarps) {
  band_pack_solve_range<FT>(n, b, F, P, (FT*)(dyn_smem + tmp_off), nwarps, 0, nwarps);
}
template <typename FT>
__device__ __forceinline__ void band_pack_solve(int n, int b, const FT* F, FT* P, FT* tmp, int nwarps) {
  band_pack_at<FT>(n, b, F, P, dyn_offset(tmp), nwarps);
}

// Triangular solves with the packed operands, in place on y[0..n) (shared memory): warp 0
// applies the block inverse (lane r: row r of inv(L_tt) or inv(U_tt) dotted with the block of
// y), threads 32 .. 32 + b - 1 apply the coupling to the next b rows.  With PF the operands of
// the next block are loaded into registers while the current one is applied (2 BS operand
// registers per thread: for kernels with few CTAs per SM, where nothing else hides the load
// latency); without PF each block's operands are loaded at the top of its step (BS registers,
// for kernels that keep enough CTAs resident).  With l2d > 0 the operands of the block l2d steps
// ahead are prefetched into L2 (one 128-byte line per thread: the diagonal-block inverse by the
// first BS^2 sizeof(FT) / 128 threads, the b coupling lines by the coupling threads), so that
// the register loads of the current and next block wait for L2 rather than HBM.  Needs blockDim.x >=
// 32 + b.
template <typename FT, bool PF>
__device__ void band_solve_packed(int n, int b, const FT* __restrict__ P, FT* y, int l2d = 0) {
  constexpr int BS = SolveBlock<FT>::BS;
  constexpr int NB = PF ? 2 : 1;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const bool diag = wid == 0 && lane < BS;
  const bool offd = tid >= 32 && tid < 32 + b;
  const int r = tid - 32;
  const int64_t PB = packed_block_entries<FT>(b);
  const int nblk = (n + BS - 1) / BS;
  const int64_t oL = 0, oU = BS * BS, oCL = 2 * BS * BS, oCU = 2 * BS * BS + (int64_t)b * BS;
  FT buf[NB][BS];
  auto load = [&](int t, int which, int64_t od, int64_t oc) {
    const FT* Pt = P + (int64_t)t * PB;
    if (diag || offd) {
      const int row = diag ? lane : r;
      const FT* R = Pt + (diag ? od : oc) + (int64_t)row * BS;
#pragma unroll
      for (int j = 0; j < BS; j += LuTile<FT>::G) {
        const LuVec<FT> v = *(const LuVec<FT>*)(R + packed_at<FT>(row, j));
#pragma unroll
        for (int i = 0; i < LuTile<FT>::G; ++i) buf[which][j + i] = v.v[i];
      }
    }
  };
  constexpr int LINE = 128 / (int)sizeof(FT);            // entries per 128-byte line
  constexpr int DLINES = BS * BS * (int)sizeof(FT) / 128;  // lines of one diagonal-block inverse
  auto l2pf = [&](int t, int64_t od, int64_t oc) {
    const FT* Pt = P + (int64_t)t * PB;
    const FT* a = nullptr;
    if (tid < DLINES) a = Pt + od + (int64_t)tid * LINE;
    else if (offd) a = Pt + oc + (int64_t)r * LINE;
    if (a) asm volatile("prefetch.global.L2 [%0];" ::"l"(__cvta_generic_to_global(a)));
  };
  // forward: diag lanes read inv(L_tt), coupling threads read CL
  if (PF && nblk > 0) load(0, 0, oL, oCL);
  for (int q = 1; q < l2d && q < nblk; ++q) l2pf(q, oL, oCL);
  for (int t = 0; t < nblk; ++t) {
    const int k0 = t * BS, kb = min(BS, n - k0);
    if (l2d > 0 && t + l2d < nblk) l2pf(t + l2d, oL, oCL);
    if (PF) {
      if (t + 1 < nblk) load(t + 1, NB - 1, oL, oCL);
    } else {
      load(t, 0, oL, oCL);
    }
    const FT* cur = buf[0];
    if (wid == 0) {  // the whole warp reaches __syncwarp; only lanes < BS hold a block row
      FT a0 = 0, a1 = 0;
      if (diag) {
#pragma unroll
        for (int j = 0; j < BS; j += 2) {
          a0 += cur[j] * ((j < kb) ? y[k0 + j] : (FT)0);
          a1 += cur[j + 1] * ((j + 1 < kb) ? y[k0 + j + 1] : (FT)0);
        }
      }
      __syncwarp();
      if (lane < kb) y[k0 + lane] = a0 + a1;
    }
    __syncthreads();
    if (offd) {
      const int i = k0 + BS + r;
      if (i < n) {
        FT a0 = 0, a1 = 0;
#pragma unroll
        for (int j = 0; j < BS; j += 2) {
          a0 += cur[j] * y[k0 + j];
          a1 += cur[j + 1] * y[k0 + j + 1];
        }
        y[i] -= a0 + a1;
      }
    }
    __syncthreads();
    if (PF) {
#pragma unroll
      for (int j = 0; j < BS; ++j) buf[0][j] = buf[NB - 1][j];
    }
  }
  // backward: diag lanes read inv(U_tt), coupling threads read CU
  if (PF && nblk > 0) load(nblk - 1, 0, oU, oCU);
  for (int q = 1; q < l2d && nblk - 1 - q >= 0; ++q) l2pf(nblk - 1 - q, oU, oCU);
  for (int t = nblk - 1; t >= 0; --t) {
    const int k0 = t * BS, kb = min(BS, n - k0);
    if (l2d > 0 && t - l2d >= 0) l2pf(t - l2d, oU, oCU);
    if (PF) {
      if (t > 0) load(t - 1, NB - 1, oU, oCU);
    } else {
      load(t, 0, oU, oCU);
    }
    const FT* cur = buf[0];
    if (wid == 0) {
      FT a0 = 0, a1 = 0;
      if (diag) {
#pragma unroll
        for (int j = 0; j < BS; j += 2) {
          a0 += cur[j] * ((j < kb) ? y[k0 + j] : (FT)0);
          a1 += cur[j + 1] * ((j + 1 < kb) ? y[k0 + j + 1] : (FT)0);
        }
      }
      __syncwarp();
      if (lane < kb) y[k0 + lane] = a0 + a1;
    }
    __syncthreads();
    if (offd) {
      const int i = k0 - 1 - r;
      if (i >= 0) {
        FT a0 = 0, a1 = 0;
#pragma unroll
        for (int j = 0; j < BS; j += 2) {
          if (j < kb) a0 += cur[j] * y[k0 + j];
          if (j + 1 < kb) a1 += cur[j + 1] * y[k0 + j + 1];
        }
        y[i] -= a0 + a1;
      }
    }
    __syncthreads();
    if (PF) {
#pragma unroll
      for (int j = 0; j < BS; ++j) buf[0][j] = buf[NB - 1][j];
    }
  }
}

// ------------------------------------------------------------------------------------------
// The same triangular solves with the operands streamed through shared memory.
//
// What bounds them: 2 ceil(n / BS) dependent block steps, each reading BS (BS + b) operand entries
// once (15 KB in FP32 at b = 85).  One thread of an extra warp keeps `stages` blocks in flight by bulk
// copies (cp.async.bulk on mbarriers), and the chain of a step is warp 0's alone: it applies the
// diagonal inverse, takes the coupling to the next block's rows itself and goes on, while the other
// warps add the coupling to the rows beyond; one named barrier of the solving warps per step keeps
// the order of the additions to every row, so the results are bit for bit those of
// band_solve_packed.  Every warp reads its operands of the next step into registers as soon as the
// current ones are used, so that only the exchange of the solved block is on the chain.  FP64: two
// lanes per row, the even and the odd terms, because a warp's FP64 instruction takes 64 cycles.
//
// Ring in shared memory (16-byte aligned): 128 bytes of mbarriers and a flag, then the stages, each
// the diagonal inverse and the coupling of one block and direction.  y: nblk BS entries, 16-byte
// aligned.  Needs ring_threads(b) threads and two stages; every thread of the CTA calls it, after a
// barrier that follows the writes of y and P.  n > 0: without unknowns there are no operands, and the
// first wait would be for one.  The forward sweep starts at block t0: y must vanish in the rows before
// it.  Returns false if a bounded wait gave up.
// ------------------------------------------------------------------------------------------
constexpr int kRingMax = 6;
constexpr int kRingHead = 128;
// Lanes per row (SP), and the warps that solve: warp 0 and those of the rows past the next block.
template <typename FT>
__host__ __device__ constexpr int ring_split() {
  return 32 / SolveBlock<FT>::BS;
}
template <typename FT>
__host__ __device__ constexpr int ring_warps(int b) {
  return 1 + (b > SolveBlock<FT>::BS ? (ring_split<FT>() * (b - SolveBlock<FT>::BS) + 31) / 32 : 0);
}
template <typename FT>
__host__ __device__ constexpr int ring_threads(int b) {
  return 32 * (ring_warps<FT>(b) + 1);
}
template <typename FT>
__host__ __device__ constexpr size_t ring_stage_bytes(int b) {
  return sizeof(FT) * SolveBlock<FT>::BS * (size_t)(SolveBlock<FT>::BS + b);
}
template <typename FT>
__host__ __device__ constexpr int ring_stages(int b, size_t bytes) {
  const size_t s = bytes < kRingHead ? 0 : (bytes - kRingHead) / ring_stage_bytes<FT>(b);
  return s < kRingMax ? (int)s : kRingMax;
}

// sum_j c[j] x[j] over a block in the order of band_solve_packed (even and odd j apart): one lane per
// row, or two lanes 16 apart that hold the even (lane < 16) and the odd terms.
template <typename FT>
__device__ __forceinline__ FT block_dot(const FT (&c)[SolveBlock<FT>::BS / ring_split<FT>()], const FT* x) {
  constexpr int BS = SolveBlock<FT>::BS, G = LuTile<FT>::G;
  if constexpr (ring_split<FT>() == 1) {
    FT a0 = 0, a1 = 0;
#pragma unroll
    for (int j = 0; j < BS; j += G) {
      const LuVec<FT> v = *(const LuVec<FT>*)(x + j);
#pragma unroll
      for (int q = 0; q < G; q += 2) {
        a0 += c[j + q] * v.v[q];
        a1 += c[j + q + 1] * v.v[q + 1];
      }
    }
    return a0 + a1;
  } else {
    const int h = (threadIdx.x & 31) >> 4;
    FT a = 0;
#pragma unroll
    for (int j = 0; j < BS / 2; ++j) a += c[j] * x[2 * j + h];
    return a + __shfl_xor_sync(0xffffffffu, a, 16);
  }
}

template <typename FT>
__device__ __forceinline__ bool band_solve_ring(int n, int b, const FT* __restrict__ P, FT* y, unsigned char* ring,
                                                int stages, int t0 = 0) {
  constexpr int BS = SolveBlock<FT>::BS;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int cw = ring_warps<FT>(b), nblk = (n + BS - 1) / BS, nf = nblk - t0, steps = nf + nblk;
  const int64_t PB = packed_block_entries<FT>(b);
  uint64_t* full = (uint64_t*)ring;
  uint64_t* empty = full + kRingMax;
  volatile int* dead = (volatile int*)(empty + kRingMax);
  if (tid == 0) {
    for (int q = 0; q < stages; ++q) {
      tc::mbar_init(full + q, 1);
      tc::mbar_init(empty + q, cw);
    }
    *dead = 0;
    tc::mbar_init_fence();
  }
  for (int a = n + tid; a < nblk * BS; a += blockDim.x) y[a] = (FT)0;
  // the packed operands and whatever the ring's memory held were written by ordinary stores; the
  // copies below go through the asynchronous proxy
  asm volatile("fence.proxy.async;" ::: "memory");
  __syncthreads();
  const size_t sb = ring_stage_bytes<FT>(b);
  int issued = steps;  // steps whose copies the copying thread has sent out
  if (wid == cw) {
    if (lane == 0) {
      const uint32_t dbytes = sizeof(FT) * BS * BS, cbytes = (uint32_t)(sizeof(FT) * BS * b);
      int st = 0;
      uint32_t par = 1;  // parity of the previous use of the stage
      for (int s = 0; s < steps; ++s) {
        if (s >= stages && !tc::mbar_wait(empty + st, par)) {
          *dead = 1;
          issued = s;
          break;
        }
        const bool fwd = s < nf;
        const FT* Pt = P + (int64_t)(fwd ? t0 + s : steps - 1 - s) * PB;
        const FT* d = Pt + (fwd ? 0 : BS * BS);
        const FT* c = Pt + 2 * BS * BS + (fwd ? 0 : (int64_t)b * BS);
        unsigned char* dst = ring + kRingHead + st * sb;
        tc::mbar_arrive_expect_tx(full + st, dbytes + cbytes);
        tc::bulk_load(dst, d, dbytes, full + st);
        if (cbytes) tc::bulk_load(dst + dbytes, c, cbytes, full + st);
        if (++st == stages) {
          st = 0;
          par ^= 1;
        }
      }
    }
    __syncwarp();
  } else if (wid < cw) {
    constexpr int SP = ring_split<FT>(), J = BS / SP;  // lanes per row, terms per lane
    const int h = SP == 1 ? 0 : lane >> 4, rl = lane % BS;
    const int r = wid == 0 ? rl : BS + (wid - 1) * BS + rl;  // coupled row of this lane
    const bool mine = r < b;
    FT d[J], c[J];  // this lane's terms of the diagonal inverse (warp 0) and of the coupling
    int st = 0;      // stage and parity of the next operands
    uint32_t par = 0;
    bool live = true;
    auto arrived = [&] { return tc::mbar_test(full + st, par); };
    auto settle = [&](bool there) {  // the next operands are there, or the wait has given up
      if (!there && live && !tc::mbar_wait(full + st, par)) {
        live = false;
        *dead = 1;
      }
      __syncwarp();
    };
    auto load = [&](FT (&v)[J], int row, const FT* rows) {
      constexpr int G = LuTile<FT>::G;
      const FT* R = rows + row * BS;
      if constexpr (SP == 1) {
#pragma unroll
        for (int j = 0; j < BS; j += G) {
          const LuVec<FT> w = *(const LuVec<FT>*)(R + packed_at<FT>(row, j));
#pragma unroll
          for (int i = 0; i < G; ++i) v[j + i] = w.v[i];
        }
      } else {
#pragma unroll
        for (int j = 0; j < J; ++j) v[j] = R[packed_at<FT>(row, SP * j + h)];
      }
    };
    auto load_d = [&] { load(d, rl, (const FT*)(ring + kRingHead + st * sb)); };
    auto load_c = [&] {
      if (mine) load(c, r, (const FT*)(ring + kRingHead + st * sb) + BS * BS);
    };
#pragma unroll
    for (int j = 0; j < J; ++j) c[j] = (FT)0;
    settle(arrived());
    if (wid == 0) load_d();
    load_c();
    for (int s = 0; s < steps; ++s) {
      const bool fwd = s < nf, more = s + 1 < steps;
      const int k0 = (fwd ? t0 + s : steps - 1 - s) * BS, i = fwd ? k0 + BS + r : k0 - 1 - r;
      const bool add = mine && i >= 0 && i < n;
      const int used = st;
      if (++st == stages) {
        st = 0;
        par ^= 1;
      }
      const bool there = more && arrived();  // asked for early, used after the diagonal block
      if (wid == 0) {
        const FT x = block_dot<FT>(d, y + k0);
        __syncwarp();
        if (h == 0 && k0 + rl < n) y[k0 + rl] = x;
      }
      if (cw > 1) asm volatile("bar.sync 1, %0;" ::"r"(32 * cw) : "memory");
      else __syncwarp();
      const FT yi = add ? y[i] : (FT)0;
      const FT t = block_dot<FT>(c, y + k0);
      if (add && h == 0) y[i] = yi - t;
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(empty + used);
      if (more) {
        settle(there);
        if (wid == 0) load_d();
        load_c();
      }
    }
  }
  __syncthreads();
  const bool ok = *dead == 0;
  // some wait gave up (on either side): see the copies in flight land before the memory is used again
  if (!ok && wid == cw && lane == 0)
    for (int s = issued > stages ? issued - stages : 0; s < issued; ++s)
      tc::mbar_wait(full + s % stages, (uint32_t)(s / stages) & 1u);
  __syncthreads();
  if (tid == 0)
    for (int q = 0; q < stages; ++q) {
      tc::mbar_inval(full + q);
      tc::mbar_inval(empty + q);
    }
  return ok;
}

}  // namespace dev
}  // namespace nls
