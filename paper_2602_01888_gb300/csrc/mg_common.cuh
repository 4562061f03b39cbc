// Internal definitions shared by the CUDA translation units of libmg.
//
// Grid/operator layout on the device (every level, both precisions):
//   node (i, j) of a level with nx x ny vertices is stored at i + pitch * j,
//   rows j = 0 .. nyr-1 (nyr = ny - 1 when periodic in y, else ny), pitch a multiple of
//   32 elements so every row starts on a 256-byte (FP64) / 128-byte (FP32) boundary.
//   The operator of a level is the symmetric 9-point matrix A = -L_h of the generalized
//   Poisson equation (Eqs. 16-18 in conservative form) or its Galerkin coarsening; per
//   node we keep its E, N, NE, NW couplings and the diagonal (plus 1/diagonal).  The
//   W, S, SW, SE couplings of node (i, j) are the E, N, NE, NW couplings of its
//   neighbours (i-1, j), (i, j-1), (i-1, j-1), (i+1, j-1): the matrix is symmetric.
//   Dirichlet nodes keep their value in the solution array (boundary data on the finest
//   level, 0 on coarse levels) and are never updated.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace mg {

template <typename T>
struct Lvl {
  int nx, ny, nyr, periodic, pitch;
  const T *cE, *cN, *cNE, *cNW, *diag, *dinv;
  // 1: the NE / NW couplings are zero at every node (a map without cross term, Eq. 13 = 0)
  // and are neither read nor multiplied; adding a zero product changes no sum, so the
  // results equal the 9-point form's.
  int five_point;
};

__host__ __device__ inline int rows_stored(int ny, int periodic) { return periodic ? ny - 1 : ny; }

__device__ __forceinline__ int row_dn(int j, int nyr) { return j == 0 ? nyr - 1 : j - 1; }
__device__ __forceinline__ int row_up(int j, int nyr) { return j == nyr - 1 ? 0 : j + 1; }

template <typename T>
__device__ __forceinline__ bool is_unknown(const Lvl<T>& L, int i, int j) {
  if (i < 1 || i > L.nx - 2 || j < 0 || j >= L.nyr) return false;
  return L.periodic || (j >= 1 && j <= L.ny - 2);
}

// Sum of the eight off-diagonal couplings times x at unknown (i, j) (four for a 5-point
// operator: the diagonal terms are zero and skipped).
template <typename T>
__device__ __forceinline__ T offdiag(const Lvl<T>& L, const T* __restrict__ x, int i, int j) {
  const int p = L.pitch;
  const int jd = row_dn(j, L.nyr), ju = row_up(j, L.nyr);
  const size_t r0 = (size_t)j * p, rd = (size_t)jd * p, ru = (size_t)ju * p;
  T s = L.cE[r0 + i] * x[r0 + i + 1];
  s = fma(L.cE[r0 + i - 1], x[r0 + i - 1], s);
  s = fma(L.cN[r0 + i], x[ru + i], s);
  s = fma(L.cN[rd + i], x[rd + i], s);
  if (L.five_point) return s;
  s = fma(L.cNE[r0 + i], x[ru + i + 1], s);
  s = fma(L.cNE[rd + i - 1], x[rd + i - 1], s);
  s = fma(L.cNW[r0 + i], x[ru + i - 1], s);
  s = fma(L.cNW[rd + i + 1], x[rd + i + 1], s);
  return s;
}

// Forward colour order (i mod 2, j mod 2): (0,0), (1,1), (1,0), (0,1).
__host__ __device__ inline int colour_ci(int c) { return (c == 1 || c == 2) ? 1 : 0; }
__host__ __device__ inline int colour_cj(int c) { return (c == 0 || c == 2) ? 0 : 1; }

// Device-side solve state (one per solve in flight).  Scalars are produced by the
// "last block" of a reducing kernel from per-block partial sums in a fixed order, so
// every result is bitwise reproducible run to run.
struct SolveState {
  double r0;          // reference norm ||r_0||_2
  double rr;          // ||r||_2^2 of the current iterate
  double rel;         // sqrt(rr) / r0
  double rz;          // previous-direction quantities of flexible CG
  double pq, pr, zq, pq_old;
  double alpha, beta;
  double scale;       // power-of-two scaling of r before the FP32 cycle (mixed)
  double inv_scale;
  double inv_scale_r32;  // 1/scale of the r32 the current FP32 cycle started from
  double rtol;
  int it;             // iterations done
  int max_iters;
  int done;           // 1 once converged / exhausted / diverged: later kernels exit at once
  int status;         // 0 running/converged, 6 not converged, 7 diverged
  int hist_n;
  int verify;         // recursive residual met rtol: recompute the true one next
  int guard;          // body passes; bounds the device-driven loop whatever happens
  int verify_fail;    // true-residual checks that did not meet rtol
  int x_zero;         // the initial iterate is zero everywhere (cold start, no Dirichlet data)
  int pad_;
  long long n_unknowns;  // for the rms used by the FP32 scaling
  unsigned int ticket[8];  // arrival counters of the last-block reductions
  double hist[256];
};

static_assert(sizeof(SolveState) % 8 == 0, "SolveState is copied as 8-byte words");

// ---- FP32 <-> FP64 on the integer pipe ---------------------------------------------
// GB300 converts between FP32 and FP64 on its FP64 pipe, which takes some 60 cycles an instruction
// and warp; the same values from the bits of the two IEEE 754 formats take about ten instructions of
// two cycles.  Every value but a NaN converts as the cast does (to nearest, ties to even); a NaN
// stays one.
struct Bits64 {
  unsigned hi, lo;
};

__host__ __device__ __forceinline__ Bits64 widen_bits(unsigned mag, unsigned sign, bool tiny) {
  // mag: exponent and fraction bits, of the value times 2^64 if tiny (below the normal range)
  const unsigned rebias = tiny ? 0x34000000u : (mag >= 0x7f800000u ? 0x70000000u : 0x38000000u);
  return {(mag ? (mag >> 3) + rebias : 0u) | sign, mag << 29};
}

__device__ __forceinline__ double widen(float v) {
  const bool tiny = (__float_as_uint(v) & 0x7f800000u) == 0;
  const unsigned u = __float_as_uint(tiny ? v * 0x1p64f : v);
  const Bits64 b = widen_bits(u & 0x7fffffffu, u & 0x80000000u, tiny);
  return __hiloint2double((int)b.hi, (int)b.lo);
}

// Magnitude bits of the nearest float outside its normal range: overflow, infinity, NaN, or a
// multiple of 2^-149 below 2^-126.
__host__ __device__ __forceinline__ unsigned narrow_far(unsigned mag, unsigned lo) {
  if (mag >= 0x47f00000u) return mag > 0x7ff00000u || (mag == 0x7ff00000u && lo) ? 0x7fffffffu : 0x7f800000u;
  const unsigned sh = 926u - (mag >> 20);  // from units of 2^(e - 1075) to 2^-149; at least 30
  if (sh >= 54u) return 0u;
  const unsigned long long m = ((unsigned long long)((mag & 0xfffffu) | 0x100000u) << 32) | lo;
  const unsigned long long q = m >> sh, rem = m & ((1ull << sh) - 1);
  return (unsigned)(q + (rem + (q & 1) > (1ull << (sh - 1)) ? 1 : 0));
}

__host__ __device__ __forceinline__ unsigned narrow_bits(unsigned hi, unsigned lo) {
  const unsigned mag = hi & 0x7fffffffu;
  unsigned f = ((mag - 0x38000000u) << 3) | (lo >> 29);
  f += (lo & 0x1fffffffu) + (f & 1u) > 0x10000000u ? 1u : 0u;
  if (mag - 0x38100000u >= 0x0fe00000u) f = narrow_far(mag, lo);
  return f | (hi & 0x80000000u);
}

__device__ __forceinline__ float narrow(double v) {
  return __uint_as_float(narrow_bits((unsigned)__double2hiint(v), (unsigned)__double2loint(v)));
}

// ---- deterministic block reduction -------------------------------------------------
// Sums each of the K values of v over the block in a fixed order (warp q adds value q's NT / 32
// columns of shared memory, then its lanes in a shuffle tree); valid in thread 0.  A tree in every
// warp first would take 40 FP64 instructions a value where this takes 12: they are the scarce ones.
template <int NT, int K>
constexpr int kSumsShared = K * NT + K;

template <int NT, int K>
__device__ __forceinline__ void block_sums(double (&v)[K], double* sh /* kSumsShared<NT, K> */) {
  constexpr int NW = NT / 32;
  static_assert(K <= NW && (NW & (NW - 1)) == 0, "one warp per value, a power of two of columns");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < K; ++q) sh[q * NT + threadIdx.x] = v[q];
  __syncthreads();
  if (warp < K) {
    double t[NW];
#pragma unroll
    for (int w = 0; w < NW; ++w) t[w] = sh[warp * NT + w * 32 + lane];
#pragma unroll
    for (int n = NW / 2; n > 0; n >>= 1)
#pragma unroll
      for (int w = 0; w < n; ++w) t[w] += t[w + n];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t[0] += __shfl_down_sync(0xffffffffu, t[0], o);
    if (lane == 0) sh[K * NT + warp] = t[0];
  }
  __syncthreads();
  if (threadIdx.x == 0)
#pragma unroll
    for (int q = 0; q < K; ++q) v[q] = sh[K * NT + q];
}

// After thread 0 of each block has written the block's partial sums, the block that arrives last
// (counted with an atomic ticket) returns true in all its threads; it then owns the
// final fixed-order reduction.  The ticket is reset for the next use.
__device__ __forceinline__ bool last_block_arrival(unsigned int* ticket, unsigned int nblocks,
                                                   int* sh_flag) {
  if (threadIdx.x == 0) {
    __threadfence();  // the partial sums (written by this thread) before the ticket
    const unsigned int t = atomicAdd(ticket, 1u);
    *sh_flag = (t == nblocks - 1);
    if (t == nblocks - 1) *ticket = 0u;
    __threadfence();
  }
  __syncthreads();
  return *sh_flag;
}

// Fixed-order sums of K rows of n partials (row q at part + q n) by one block (tree over a strided
// split; the order depends only on n and the block size); valid in thread 0.  A thread's loads are
// issued together: one at a time, each waits a round trip to L2.
template <int NT, int K>
__device__ __forceinline__ void reduce_partials(const double* part, int n, double (&v)[K], double* sh) {
  constexpr int B = 8;
#pragma unroll
  for (int q = 0; q < K; ++q) v[q] = 0.0;
  for (int base = 0; base < n; base += B * NT) {
    const int k0 = base + threadIdx.x;
    double w[K][B];
#pragma unroll
    for (int q = 0; q < K; ++q)
#pragma unroll
      for (int u = 0; u < B; ++u) w[q][u] = k0 + u * NT < n ? __ldcg(part + (size_t)q * n + k0 + u * NT) : 0.0;
#pragma unroll
    for (int u = 0; u < B; ++u) {
      if (base + u * NT >= n) break;  // uniform: no FP64 issue slots for rows past the end
#pragma unroll
      for (int q = 0; q < K; ++q) v[q] += w[q][u];
    }
  }
  block_sums<NT, K>(v, sh);
}

}  // namespace mg
