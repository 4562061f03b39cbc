// Setup kernels: coefficient build (Eqs. 1, 10-15, 39-42), fine-level operator,
// right-hand side (Eq. 11), Galerkin coarse operators (Sec. 3) and the coarsest-level
// inverse.  They run once per problem (or per geometry update); everything is FP64
// except the Galerkin products of the mixed-precision hierarchy, which are FP32.
#include "mg_common.cuh"
#include "mg_kernels.h"
#include "mg_launch.h"

namespace mg {

static const double kPi = 3.14159265358979323846;

// Whether det J is zero, negative or NaN, from the bits: a comparison would run on the FP64 pipe.
__device__ __forceinline__ bool folds(double det) {
  return (unsigned long long)__double_as_longlong(det) - 1u >= 0x7ff0000000000000ull;
}

// eps = det(J) J^-1 (s I) J^-T for J = [[a, b], [c, d]] (Eqs. 10, 12-15); unit: s is 1.
__device__ __forceinline__ void store_eps(double a, double b, double c, double d, double s,
                                          size_t k, double* D, double* exx, double* exy,
                                          double* eyy, int* folded, bool unit) {
  const double det = a * d - b * c;
  if (folds(det)) atomicOr(folded, 1);
  D[k] = det;
  const double sd = unit ? 1.0 / det : s / det;  // one division per node, cheaper as a reciprocal
  exx[k] = sd * (d * d + b * b);     // Eq. 12
  exy[k] = sd * (-d * c - b * a);    // Eq. 13 = Eq. 14
  eyy[k] = sd * (c * c + a * a);     // Eq. 15
}

// One CTA per 32 x 32 tile of nodes (32 x 8 threads, four rows each).  The sine warp's Jacobian is
// built from transcendental factors of x alone and of y alone, so they are evaluated once per column
// and once per row of the tile, in shared memory, rather than once per node: FP64 transcendentals,
// not memory traffic, bound this kernel otherwise.
constexpr int kEpsTile = 32;

__global__ void __launch_bounds__(256) k_eps_sine_warp(double p0, int nx, int nyr, double x0, double y0,
                                                       double hx, double hy,
                                                       const double* __restrict__ eps, int pitch,
                                                       double* D, double* exx, double* exy, double* eyy,
                                                       int* folded) {
  __shared__ double colv[4][kEpsTile], rowv[2][kEpsTile];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int i0 = blockIdx.x * kEpsTile, j0 = blockIdx.y * kEpsTile;
  if (ty == 0) {  // factors of x
    const double x = x0 + (i0 + tx) * hx;
    sincos(kPi * x, &colv[0][tx], &colv[1][tx]);
    sincos(2.0 * kPi * x, &colv[2][tx], &colv[3][tx]);
  } else if (ty == 1) {  // factors of y
    const double y = y0 + (j0 + tx) * hy;
    sincos(kPi * y, &rowv[0][tx], &rowv[1][tx]);
  }
  __syncthreads();
  const int i = i0 + tx;
  if (i >= nx) return;
  const double sx = colv[0][tx], cx = colv[1][tx], s2x = colv[2][tx], c2x = colv[3][tx];
#pragma unroll
  for (int r = 0; r < kEpsTile / 8; ++r) {
    const int ly = ty + 8 * r, j = j0 + ly;
    if (j >= nyr) break;
    const double sy = rowv[0][ly], cy = rowv[1][ly];
    const double a = 1.0 + p0 * kPi * cx * sy;  // Jxx
    const double b = p0 * kPi * sx * cy;        // Jxy
    const double c = p0 * 2.0 * kPi * c2x * sy;  // Jyx
    const double d = 1.0 + p0 * kPi * s2x * cy;  // Jyy
    const size_t k = (size_t)j * pitch + i;
    if (eps) store_eps(a, b, c, d, eps[k], k, D, exx, exy, eyy, folded, false);
    else store_eps(a, b, c, d, 1.0, k, D, exx, exy, eyy, folded, true);
  }
}

// Polar map (Eq. 29), the general formula with what depends on one coordinate taken out of the node:
// the row's sum of squares, and 1 / x for the division.  det J = x (cos^2 + sin^2) is x but for
// rounding, so the quotient eps' / x corrected by its residual against det J is eps' / det J to one
// rounding.  The closed form (D = x, eps_xx = s x, eps_yy = s / x) would be cheaper still, but its
// rounding is the same at every node of a circle and adds up in the row sums of the operator: at
// 8193^2 it moves the solution by 3e-10.  Ten FP64 operations a node bound it: 8193 x 8192 1.43 ms (1.54
// with a material), 2.60 ms with the division and the sums at every node.
__global__ void __launch_bounds__(256) k_eps_polar(int nx, int nyr, double x0, double y0, double hx, double hy,
                                                   const double* __restrict__ eps, int pitch,
                                                   double* __restrict__ D, double* __restrict__ exx,
                                                   double* __restrict__ exy, double* __restrict__ eyy, int* folded) {
  __shared__ double colv[kEpsTile], rowv[3][kEpsTile];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int i0 = blockIdx.x * kEpsTile, j0 = blockIdx.y * kEpsTile;
  if (ty == 0) colv[tx] = 1.0 / (x0 + (i0 + tx) * hx);
  if (ty == 1) {
    double c, a;
    sincos(y0 + (j0 + tx) * hy, &c, &a);
    rowv[0][tx] = c;
    rowv[1][tx] = a;
    rowv[2][tx] = c * c + a * a;
  }
  __syncthreads();
  const int i = i0 + tx;
  if (i >= nx) return;
  const double x = x0 + i * hx, rx = colv[tx];
#pragma unroll
  for (int r = 0; r < kEpsTile / 8; ++r) {
    const int ly = ty + 8 * r, j = j0 + ly;
    if (j >= nyr) break;
    const double c = rowv[0][ly], a = rowv[1][ly];  // Jyx, Jxx
    const double b = -x * c, d = x * a;             // Jxy, Jyy
    const double det = a * d - b * c;
    if (folds(det)) atomicOr(folded, 1);
    const size_t k = (size_t)j * pitch + i;
    D[k] = det;
    const double m = eps ? eps[k] : 1.0, q = m * rx;
    const double sd = fma(rx, fma(-det, q, m), q);
    exx[k] = sd * (d * d + b * b);  // Eq. 12
    exy[k] = 0.0;                   // Eq. 13 vanishes identically
    eyy[k] = sd * rowv[2][ly];      // Eq. 15
  }
}

// The other analytic maps, whose Eqs. 10, 12-15 are a factor of x times a factor of y:
//   sinh (Eq. 52)    D = a(x) d(y)             eps_xx = s (1 / a) d          eps_yy = s a (1 / d)
//   affine, identity D, eps_xx / s, eps_xy / s and eps_yy / s constant (cD, cxx, cxy, cyy)
// with a = p0 p1 cosh(p1 x), d = p0 p1 cosh(p1 y).  The factors are evaluated once per column and row
// of a tile of 32 x 32 nodes; a node costs two products and no division (SINH: five), so the 32 or 40
// bytes it moves bound the kernel.  Through the general formula the FP64 pipe did, with a division a
// node.  cross = 0: Eq. 13 vanishes identically, eps_xy is zero.
template <bool SINH>
__global__ void __launch_bounds__(256) k_eps_separable(double p0, double p1, double cD, double cxx,
                                                       double cxy, double cyy, int nx, int nyr, double x0, double y0,
                                                       double hx, double hy, const double* __restrict__ eps, int pitch,
                                                       double* __restrict__ D, double* __restrict__ exx,
                                                       double* __restrict__ exy, double* __restrict__ eyy, int* folded,
                                                       int cross) {
  __shared__ double colv[2][kEpsTile], rowv[2][kEpsTile];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int i0 = blockIdx.x * kEpsTile, j0 = blockIdx.y * kEpsTile;
  double fD = cD, fx = cxx, fy = cyy;
  if (SINH) {
    if (ty < 2) {
      const double f = p0 * p1 * cosh(p1 * (ty == 0 ? x0 + (i0 + tx) * hx : y0 + (j0 + tx) * hy));
      (ty == 0 ? colv : rowv)[0][tx] = f;
      (ty == 0 ? colv : rowv)[1][tx] = 1.0 / f;
    }
    __syncthreads();
    fD = fy = colv[0][tx];
    fx = colv[1][tx];
  }
  const int i = i0 + tx;
  if (i >= nx) return;
#pragma unroll
  for (int r = 0; r < kEpsTile / 8; ++r) {
    const int ly = ty + 8 * r, j = j0 + ly;
    if (j >= nyr) break;
    const size_t k = (size_t)j * pitch + i;
    double det = fD, gx = fx, gy = fy;
    if (SINH) {
      det *= rowv[0][ly];
      gx *= rowv[0][ly];
      gy *= rowv[1][ly];
    }
    if (folds(det)) atomicOr(folded, 1);
    D[k] = det;
    const double s = eps ? eps[k] : 1.0;
    exx[k] = s * gx;                   // Eq. 12
    exy[k] = cross ? s * cxy : 0.0;    // Eq. 13 = Eq. 14
    eyy[k] = s * gy;                   // Eq. 15
  }
}

// Even reflection of a grid with Neumann y sides into the periodic grid of twice the height
// (2n rows, n = ny - 1): row j' of the doubled grid copies row j' - n (j' >= n) or n - j'
// (j' < n) of the source, with eps_xy negated in the mirrored half and zero on the two
// Neumann rows (j' = 0, n), where an odd function vanishes.
__global__ void k_mirror_eps(int nx, int n, int ps, const double* __restrict__ D0,
                             const double* __restrict__ exx0, const double* __restrict__ exy0,
                             const double* __restrict__ eyy0, int pd, double* D, double* exx,
                             double* exy, double* eyy) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int jd = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= nx || jd >= 2 * n) return;
  const int js = jd >= n ? jd - n : n - jd;
  const double sg = (jd == 0 || jd == n) ? 0.0 : (jd > n ? 1.0 : -1.0);
  const size_t s = (size_t)js * ps + i, d = (size_t)jd * pd + i;
  D[d] = D0[s];
  exx[d] = exx0[s];
  exy[d] = sg * exy0[s];
  eyy[d] = eyy0[s];
}

// d/dx: central difference (Eqs. 39, 41), one-sided second order at the line ends;
// i2h = 1 / (2 hx).
__device__ __forceinline__ double ddx(const double* __restrict__ f, size_t r, int i, int nx,
                                      double i2h) {
  if (i == 0) return (-3.0 * f[r] + 4.0 * f[r + 1] - f[r + 2]) * i2h;
  if (i == nx - 1) return (3.0 * f[r + nx - 1] - 4.0 * f[r + nx - 2] + f[r + nx - 3]) * i2h;
  return (f[r + i + 1] - f[r + i - 1]) * i2h;
}

// d/dy (Eqs. 40, 42); a periodic line wraps and adds `jump` across the seam; i2h = 1 / (2 hy).
__device__ __forceinline__ double ddy(const double* __restrict__ f, int i, int j, int ny, int nyr,
                                      int periodic, int pitch, double i2h, double jump) {
  if (periodic) {
    const double fp = (j + 1 >= nyr) ? f[(size_t)(j + 1 - nyr) * pitch + i] + jump
                                     : f[(size_t)(j + 1) * pitch + i];
    const double fm = (j - 1 < 0) ? f[(size_t)(j - 1 + nyr) * pitch + i] - jump
                                  : f[(size_t)(j - 1) * pitch + i];
    return (fp - fm) * i2h;
  }
  if (j == 0)
    return (-3.0 * f[i] + 4.0 * f[(size_t)pitch + i] - f[2 * (size_t)pitch + i]) * i2h;
  if (j == ny - 1)
    return (3.0 * f[(size_t)(ny - 1) * pitch + i] - 4.0 * f[(size_t)(ny - 2) * pitch + i] +
            f[(size_t)(ny - 3) * pitch + i]) * i2h;
  return (f[(size_t)(j + 1) * pitch + i] - f[(size_t)(j - 1) * pitch + i]) * i2h;
}

// The inner nodes' four central differences stand in a branch of their own: inlined together, ddx and
// ddy become predicated code, whose one-sided formulas take FP64 issue slots at every node (2049^2:
// 294 -> 217 us; 27 FP64 operations a node, the pipe is the bound).
__global__ void k_eps_grid(int nx, int ny, int nyr, int periodic, double i2hx, double i2hy,
                           const double* __restrict__ xp, const double* __restrict__ yp,
                           double jump_x, double jump_y, const double* __restrict__ eps,
                           int pitch, double* D, double* exx, double* exy, double* eyy,
                           int* folded) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= nx || j >= nyr) return;
  const size_t r = (size_t)j * pitch, k = r + i;
  double a, b, c, d;
  if (i > 0 && i < nx - 1 && j > 0 && j < nyr - 1) {  // the inner case of ddx and ddy
    a = (xp[k + 1] - xp[k - 1]) * i2hx;          // Eq. 39
    b = (xp[k + pitch] - xp[k - pitch]) * i2hy;  // Eq. 40
    c = (yp[k + 1] - yp[k - 1]) * i2hx;          // Eq. 41
    d = (yp[k + pitch] - yp[k - pitch]) * i2hy;  // Eq. 42
  } else {
    a = ddx(xp, r, i, nx, i2hx);
    b = ddy(xp, i, j, ny, nyr, periodic, pitch, i2hy, jump_x);
    c = ddx(yp, r, i, nx, i2hx);
    d = ddy(yp, i, j, ny, nyr, periodic, pitch, i2hy, jump_y);
  }
  if (eps) store_eps(a, b, c, d, eps[k], k, D, exx, exy, eyy, folded, false);
  else store_eps(a, b, c, d, 1.0, k, D, exx, exy, eyy, folded, true);
}

// Couplings of the symmetric conservative 9-point operator A = -L_h.  five: eps_xy is zero
// everywhere, so the NE / NW couplings are zero and written without reading it.
template <typename T>
__global__ void k_assemble_couplings(int nx, int ny, int nyr, int periodic, int pitch, T ihx2,
                                     T ihy2, T ixy4, const T* __restrict__ exx,
                                     const T* __restrict__ exy,
                                     const T* __restrict__ eyy, T* cE, T* cN,
                                     T* cNE, T* cNW, int five) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= nx || j >= nyr) return;
  const size_t k = (size_t)j * pitch + i;
  const bool has_up = periodic || (j + 1 <= ny - 1);
  const int ju = (j + 1 == nyr) ? 0 : j + 1;
  const size_t ku = (size_t)ju * pitch + i;
  T e = T(0), n = T(0), ne = T(0), nw = T(0);
  if (i + 1 <= nx - 1) e = T(-0.5) * (exx[k] + exx[k + 1]) * ihx2;
  if (has_up) {
    n = T(-0.5) * (eyy[k] + eyy[ku]) * ihy2;
    if (!five) {
      if (i + 1 <= nx - 1) ne = -(exy[k + 1] + exy[ku]) * ixy4;  // to (i+1, j+1)
      if (i >= 1) nw = (exy[k - 1] + exy[ku]) * ixy4;             // to (i-1, j+1)
    }
  }
  cE[k] = e;
  cN[k] = n;
  cNE[k] = ne;
  cNW[k] = nw;
}

// diag = -(sum of the 8 couplings) at unknowns (zero row sums), 1 at Dirichlet nodes; the
// zero NE / NW terms of a 5-point operator are left out of the sum (which they do not change).
// dinv = 1 / diag unless dinv is null (a mixed-precision hierarchy takes its FP32 reciprocal
// from the FP32 diagonal instead and never reads an FP64 one).
template <typename T>
__global__ void k_assemble_diag(int nx, int ny, int nyr, int periodic, int pitch,
                                const T* __restrict__ cE, const T* __restrict__ cN,
                                const T* __restrict__ cNE, const T* __restrict__ cNW,
                                T* diag, T* dinv, int five) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= nx || j >= nyr) return;
  const size_t k = (size_t)j * pitch + i;
  const bool unk = (i >= 1 && i <= nx - 2) && (periodic || (j >= 1 && j <= ny - 2));
  if (!unk) {
    diag[k] = T(1);
    if (dinv) dinv[k] = T(1);
    return;
  }
  const int jd = (j == 0) ? nyr - 1 : j - 1;
  const size_t ks = (size_t)jd * pitch + i;
  T s = cE[k] + cE[k - 1] + cN[k] + cN[ks];
  if (!five) s = s + cNE[k] + cNE[ks - 1] + cNW[k] + cNW[ks + 1];
  diag[k] = -s;
  if (dinv) dinv[k] = T(1) / (-s);
}

// One pass over the finest level: the couplings of k_assemble_couplings, the diagonal, its reciprocal
// (dinv when given) and, when fE is given, the FP32 copy of k_op_to_f32 with the reciprocal of the FP32
// diagonal (pitch pf).  A warp covers 32 columns, of which it owns the inner 30, and marches down
// a strip of rows: every tensor value is loaded once (shuffles and the row before give the
// neighbours').  A coupling is rounded like the separate kernel's: -(1/2)(a + b) / h^2 is the sum times
// the exact constant -(1/2) / h^2 (halving is exact), one rounding per operation (__dadd_rn,
// __dmul_rn: no contracted multiply-add), so the couplings are bitwise those of the separate kernels.
// The cross couplings of a node cancel in the row sum, -q(i+1,j) - q(i,j+1) + q(i-1,j) + q(i,j+1) -
// q(i,j-1) - q(i-1,j) + q(i,j-1) + q(i+1,j) = 0, so the diagonal is minus the sum of the E, W, N and S
// ones (three roundings instead of seven).  FIVE: eps_xy is zero everywhere; NE / NW get zeros, for
// the kernels that have no 5-point form.  Bound by the FP64 pipe: 11 operations a node (FIVE: 7) and
// the five of dinv's reciprocal.  9-point 2049^2 157 us, 197 us with the two separate kernels; 5-point
// 8193^2 with the FP32 copy 1.33 -> 1.22 ms (every first lane computed its W coupling, predicated).
constexpr int kAsmCols = 30;

template <bool FIVE>
__global__ void __launch_bounds__(256) k_assemble_pass(int nx, int ny, int nyr, int periodic, int pitch, double mx,
                                                       double my, double mxy, const double* __restrict__ exx,
                                                       const double* __restrict__ exy,
                                                       const double* __restrict__ eyy, int rows, double* cE, double* cN,
                                                       double* cNE, double* cNW, double* diag, double* dinv, int pf,
                                                       float* fE, float* fN, float* fNE, float* fNW, float* fdiag,
                                                       float* fdinv) {
  const int lane = threadIdx.x;
  const int i = blockIdx.x * kAsmCols + lane - 1;
  const int jb = (blockIdx.y * blockDim.y + threadIdx.y) * rows;
  if (jb >= nyr) return;  // one strip per warp
  const bool col = i >= 0 && i < nx, own = col && lane >= 1 && lane <= kAsmCols, has_e = i + 1 <= nx - 1;
  auto get = [&](const double* __restrict__ f, int j) { return col ? f[(size_t)j * pitch + i] : 0.0; };
  auto left = [](double v) { return __shfl_up_sync(0xffffffffu, v, 1); };
  auto right = [](double v) { return __shfl_down_sync(0xffffffffu, v, 1); };
  // couplings of row j to row j + 1 from the tensor values of the two rows
  auto ups = [&](int j, double q, double y, double qu, double yu, double& n, double& ne, double& nw) {
    const bool up = col && (periodic || j + 1 <= ny - 1);
    n = up ? __dmul_rn(__dadd_rn(y, yu), my) : 0.0;
    ne = nw = 0.0;
    if (FIVE) return;
    const double ql = left(q), qr = right(q);
    ne = up && has_e ? __dmul_rn(__dadd_rn(qr, qu), -mxy) : 0.0;
    nw = up && i >= 1 ? __dmul_rn(__dadd_rn(ql, qu), mxy) : 0.0;
  };
  double q = FIVE ? 0.0 : get(exy, jb), y = get(eyy, jb);
  double ns = 0.0;  // coupling of the row below to this one
  if (jb > 0 || periodic) {
    const int jm = jb == 0 ? nyr - 1 : jb - 1;
    ns = __dmul_rn(__dadd_rn(get(eyy, jm), y), my);
  }
  for (int r = 0; r < rows; ++r) {
    const int j = jb + r;
    if (j >= nyr) break;
    const int ju = (j + 1 == nyr) ? 0 : j + 1;
    const double x = get(exx, j), qu = FIVE ? 0.0 : get(exy, ju), yu = get(eyy, ju);
    const double xr = right(x);
    const double e = col && has_e ? __dmul_rn(__dadd_rn(x, xr), mx) : 0.0;
    double n, ne, nw;
    ups(j, q, y, qu, yu, n, ne, nw);
    const double ew = left(e);
    if (own) {
      const size_t k = (size_t)j * pitch + i;
      const bool unk = (i >= 1 && i <= nx - 2) && (periodic || (j >= 1 && j <= ny - 2));
      double d = 1.0;
      if (unk) {
        d = -__dadd_rn(__dadd_rn(__dadd_rn(e, ew), n), ns);
      }
      cE[k] = e;
      cN[k] = n;
      cNE[k] = ne;
      cNW[k] = nw;
      diag[k] = d;
      if (dinv) dinv[k] = unk ? 1.0 / d : 1.0;
      if (fE) {
        const size_t kf = (size_t)j * pf + i;
        fE[kf] = narrow(e);
        fN[kf] = narrow(n);
        fNE[kf] = narrow(ne);
        fNW[kf] = narrow(nw);
        const float dg = narrow(d);
        fdiag[kf] = dg;
        fdinv[kf] = 1.0f / dg;
      }
    }
    q = qu;
    y = yu;
    ns = n;
  }
}

__global__ void k_rhs(int nx, int ny, int nyr, int periodic, int pitch,
                      const double* __restrict__ rho, int rho_pitch, const double* __restrict__ D,
                      double* b) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= nx || j >= nyr) return;
  const bool unk = (i >= 1 && i <= nx - 2) && (periodic || (j >= 1 && j <= ny - 2));
  const size_t k = (size_t)j * pitch + i;
  b[k] = unk ? rho[(size_t)j * rho_pitch + i] * D[k] : 0.0;  // Eq. 11
}

// Tensor of the next coarser level of a rediscretized hierarchy: each of the three nodal
// fields at coarse node (I, J), full weighting (1/16)[1 2 1; 2 4 2; 1 2 1] about fine node
// (2I, 2J) where all eight fine neighbours exist (rows wrap when periodic), the coincident
// fine value on the coarse boundary ring.
// TS / TD: precision of the fine and of the coarse fields (the mixed path coarsens in FP32).
// five: the cross term is zero on the fine level, so on the coarse one (written, not computed).
template <typename TS, typename TD>
__global__ void k_coarsen_eps(int nxf, int nyrf, int pf, int nxc, int nyc, int nyrc, int pc, int periodic,
                              const TS* __restrict__ f0, const TS* __restrict__ f1,
                              const TS* __restrict__ f2, TD* c0, TD* c1, TD* c2, int five) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int J = blockIdx.y * blockDim.y + threadIdx.y;
  if (I >= nxc || J >= nyrc) return;
  const int fi = 2 * I, fj = 2 * J;
  const bool inner = (I >= 1 && I <= nxc - 2) && (periodic || (J >= 1 && J <= nyc - 2));
  const int jd = fj == 0 ? nyrf - 1 : fj - 1, ju = fj + 1 == nyrf ? 0 : fj + 1;
  const size_t r0 = (size_t)fj * pf, rd = (size_t)jd * pf, ru = (size_t)ju * pf, K = (size_t)J * pc + I;
  const TS* const f[3] = {f0, f1, f2};
  TD* const c[3] = {c0, c1, c2};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (a == 1 && five) {
      c[a][K] = TD(0);
      continue;
    }
    const TS* g = f[a];
    TD v;
    if (inner)
      v = (TD(4) * TD(g[r0 + fi]) +
           TD(2) * (TD(g[r0 + fi - 1]) + TD(g[r0 + fi + 1]) + TD(g[rd + fi]) + TD(g[ru + fi])) +
           (TD(g[rd + fi - 1]) + TD(g[rd + fi + 1]) + TD(g[ru + fi - 1]) + TD(g[ru + fi + 1]))) / TD(16);
    else
      v = TD(g[r0 + fi]);
    c[a][K] = v;
  }
}

// Bilinear weight of a fine offset d from a coarse node (in fine units).
__host__ __device__ constexpr double pw(int d) { return d == 0 ? 1.0 : ((d == 1 || d == -1) ? 0.5 : 0.0); }

// A[(fi,fj),(fi+di,fj+dj)] through the symmetric storage of a level.
template <typename T>
__device__ __forceinline__ T fine_entry(const Lvl<T>& F, int fi, int fj, int di, int dj) {
  const size_t r0 = (size_t)fj * F.pitch, rd = (size_t)row_dn(fj, F.nyr) * F.pitch;
  if (dj == 0) {
    if (di == 0) return F.diag[r0 + fi];
    return di > 0 ? F.cE[r0 + fi] : F.cE[r0 + fi - 1];
  }
  if (dj > 0) {
    if (di == 0) return F.cN[r0 + fi];
    return di > 0 ? F.cNE[r0 + fi] : F.cNW[r0 + fi];
  }
  if (di == 0) return F.cN[rd + fi];
  return di < 0 ? F.cNE[rd + fi - 1] : F.cNW[rd + fi + 1];
}

// A_H = (1/4) P^T A_h P: for each coarse unknown I, row(I, I+o) = (1/4) sum_k sum_l
// P(k, I) A(k, l) P(l, I+o) over fine k in the 3x3 support of I and the 9 stencil
// neighbours l of k, for the five entries stored (o = centre, E, N, NE, NW; the others are
// the symmetric partners' entries).  Every loop is unrolled so the bilinear weights are
// constants and only the (k, l, o) triples with non-zero weight remain (109 multiply-adds).
// FIVE: the fine operator is 5-point (F.five_point): its diagonal entries are zero and their
// products, which would add zeros, are skipped (69 multiply-adds, the same sums).
template <typename T, bool FIVE>
__global__ void k_galerkin(Lvl<T> F, int nxc, int nyc, int nyrc, int pitchc, T* cE, T* cN, T* cNE,
                           T* cNW, T* diag, T* dinv) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int J = blockIdx.y * blockDim.y + threadIdx.y;
  if (I >= nxc || J >= nyrc) return;
  const size_t K = (size_t)J * pitchc + I;
  const bool unk = (I >= 1 && I <= nxc - 2) && (F.periodic || (J >= 1 && J <= nyc - 2));
  if (!unk) {
    cE[K] = cN[K] = cNE[K] = cNW[K] = T(0);
    diag[K] = dinv[K] = T(1);
    return;
  }
  T row[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) row[a][b] = T(0);
#pragma unroll
  for (int kj = -1; kj <= 1; ++kj) {
    int fj = 2 * J + kj;
    if (fj < 0) fj += F.nyr;
    if (fj >= F.nyr) fj -= F.nyr;
#pragma unroll
    for (int ki = -1; ki <= 1; ++ki) {
      const int fi = 2 * I + ki;
#pragma unroll
      for (int lj = -1; lj <= 1; ++lj)
#pragma unroll
        for (int li = -1; li <= 1; ++li) {
          if (FIVE && li != 0 && lj != 0) continue;
          const T a = fine_entry(F, fi, fj, li, lj);
#pragma unroll
          for (int oj = 0; oj <= 1; ++oj)
#pragma unroll
            for (int oi = -1; oi <= 1; ++oi) {
              if (oj == 0 && oi < 0) continue;  // W: not stored
              const double w = 0.25 * pw(ki) * pw(kj) * pw(ki + li - 2 * oi) * pw(kj + lj - 2 * oj);
              if (w != 0.0) row[oi + 1][oj + 1] = fma((T)w, a, row[oi + 1][oj + 1]);
            }
        }
    }
  }
  diag[K] = row[1][1];
  dinv[K] = T(1) / row[1][1];
  cE[K] = row[2][1];
  cN[K] = row[1][2];
  cNE[K] = row[2][2];
  cNW[K] = row[0][2];
}

// The same product in FP64 collapsed first along x, then along y (P is the tensor product of the
// one-dimensional interpolations): 62 FP64 operations a coarse node instead of 118.  Per fine row j
// and coarse column I the first step gives h0, h1 (coupling of column I to itself and to I + 1
// within the row) and u0, u1, um (to columns I, I + 1, I - 1 of the row above):
//   h0 = d(2I) + (d(2I-1) + d(2I+1)) / 4 + E(2I-1) + E(2I)
//   h1 = (E(2I) + E(2I+1)) / 2 + d(2I+1) / 4
//   u0 = N(2I) + (N(2I-1) + N(2I+1)) / 4 + (NE(2I-1) + NE(2I) + NW(2I) + NW(2I+1)) / 2
//   u1 = (NE(2I) + NE(2I+1)) / 2 + N(2I+1) / 4,   um = (NW(2I) + NW(2I-1)) / 2 + N(2I-1) / 4
// and the second combines the rows 2J - 1, 2J, 2J + 1 the same way.  A warp holds 32 coarse columns,
// of which it owns the inner 30 (the lanes beside supply E's and NW's missing halves), and marches
// up a strip of coarse rows, so each fine row is collapsed once.  Pairs of columns are loaded as one
// vector.  FIVE: zero NE / NW, whose terms vanish exactly (42 operations).  Bound by the FP64 pipe
// (81% busy): 2049^2 -> 1025^2 -> 513^2 220 us, 292 us with k_galerkin.  The sums are ordered so that
// large terms cancel before small ones are added.  Rms errors against exact sums as fractions of the
// direct product's (which stay below 8e-17 of the largest coupling off the diagonal and 2.3e-16 on it),
// for operators of smooth, rough, tenfold jumping and 30 : 1 stretched tensors, two levels: E 0.44-0.81,
// N 0.65-0.95, NE 0.66-0.86, NW 0.66-0.92, diagonal 0.35-0.68.  Not below it: E at y couplings 30 times
// the x ones (1.2, the diagonal 0.9), N of the 5-point polar operator at equal couplings (1.2, 0.7).
constexpr int kGalCols = 30;

struct GalRow {
  double h0, h1, u0, u1, um;
};

template <bool FIVE>
__global__ void __launch_bounds__(128, 5) k_galerkin_rows(Lvl<double> F, int nxc, int nyc, int nyrc, int pitchc, int rows,
                                                       double* __restrict__ cE, double* __restrict__ cN,
                                                       double* __restrict__ cNE, double* __restrict__ cNW,
                                                       double* __restrict__ diag, double* __restrict__ dinv) {
  const int lane = threadIdx.x & 31;
  const int I = blockIdx.x * kGalCols + lane - 1;
  const int Jb = (blockIdx.y * (blockDim.x / 32) + (threadIdx.x >> 5)) * rows, Je = min(Jb + rows, nyrc);
  if (Jb >= nyrc) return;  // one strip per warp
  const bool col = I >= 0 && I < nxc, own = col && lane >= 1 && lane <= kGalCols;
  auto left = [](double v) { return __shfl_up_sync(0xffffffffu, v, 1); };
  auto right = [](double v) { return __shfl_down_sync(0xffffffffu, v, 1); };
  constexpr double hu = FIVE ? 0.125 : 0.5;
  auto row = [&](int j) -> GalRow {  // j wrapped or clamped into the grid by the caller
    const size_t k = (size_t)j * F.pitch + 2 * I;
    const double2 z = make_double2(0.0, 0.0);
    auto get = [&](const double* a) { return col ? __ldg(reinterpret_cast<const double2*>(a + k)) : z; };
    const double2 d = get(F.diag), e = get(F.cE), n = get(F.cN);
    const double dl = left(d.y), el = left(e.y), nl = left(n.y);
    GalRow g;
    g.h0 = fma(0.25, dl + d.y, (d.x + e.x) + el);
    g.h1 = fma(0.5, e.x, fma(0.5, e.y, 0.25 * d.y));
    g.u0 = fma(0.25, nl + n.y, n.x);
    if (FIVE) {  // four times u1 and um: hu takes the factor
      g.u1 = n.y;
      g.um = nl;
    } else {
      const double2 ne = get(F.cNE), nw = get(F.cNW);
      const double nel = left(ne.y), nwl = left(nw.y);
      g.u0 = fma(0.5, (nel + ne.x) + (nw.x + nw.y), g.u0);
      g.u1 = fma(0.5, ne.x + ne.y, 0.25 * n.y);
      g.um = fma(0.5, nw.x + nwl, 0.25 * nl);
    }
    return g;
  };
  auto fine = [&](int j) { return F.periodic ? (j < 0 ? j + F.nyr : (j >= F.nyr ? j - F.nyr : j)) : min(max(j, 0), F.nyr - 1); };
  GalRow p = row(fine(2 * Jb - 1));
  for (int J = Jb; J < Je; ++J) {
    const GalRow c = row(fine(2 * J)), n = row(fine(2 * J + 1));
    const double s_um = right(p.um + c.um);  // um of column I + 1
    const double h1l = left(n.h1);           // h1 of column I - 1
    if (own) {
      const size_t K = (size_t)J * pitchc + I;
      const bool unk = I >= 1 && I <= nxc - 2 && (F.periodic || (J >= 1 && J <= nyc - 2));
      double vE = 0.0, vN = 0.0, vNE = 0.0, vNW = 0.0, vd = 1.0;
      if (unk) {
        vd = 0.25 * fma(0.25, p.h0, fma(0.25, n.h0, c.h0 + (p.u0 + c.u0)));
        vE = 0.25 * fma(0.25, p.h1 + n.h1, fma(hu, s_um, fma(hu, c.u1, fma(hu, p.u1, c.h1))));
        vN = 0.25 * fma(0.5, c.u0, fma(0.5, n.u0, 0.25 * n.h0));
        vNE = 0.25 * fma(hu, c.u1, fma(hu, n.u1, 0.25 * n.h1));
        vNW = 0.25 * fma(hu, c.um, fma(hu, n.um, 0.25 * h1l));
      }
      diag[K] = vd;
      dinv[K] = unk ? 1.0 / vd : 1.0;
      cE[K] = vE;
      cN[K] = vN;
      cNE[K] = vNE;
      cNW[K] = vNW;
    }
    p = n;
  }
}

// INT: conversions on the integer pipe (mg_common.cuh) instead of the conversion instruction, whose time
// on the FP64 pipe is about that of the copy in HBM: faster where the arrays stay in L2 (us, INT against
// the instruction: 513^2 3.5, 4.7; 1025^2 9.4, 12.6), slower on smaller and larger ones (129^2 2.5, 1.95;
// 2049^2 63.8, 47.4).
template <bool INT>
__global__ void k_op_to_f32(int nx, int nyr, int ps, int pd, const double* __restrict__ a0,
                            const double* __restrict__ a1, const double* __restrict__ a2,
                            const double* __restrict__ a3, const double* __restrict__ a4,
                            const double* __restrict__ a5, float* b0, float* b1, float* b2,
                            float* b3, float* b4, float* b5, int five, int dinv_f32) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= nx || j >= nyr) return;
  const size_t s = (size_t)j * ps + i, d = (size_t)j * pd + i;
  auto f32 = [](double v) { return INT ? narrow(v) : (float)v; };
  b0[d] = f32(a0[s]);
  b1[d] = f32(a1[s]);
  b2[d] = five ? 0.0f : f32(a2[s]);  // a 5-point operator's NE / NW are zero: not read
  b3[d] = five ? 0.0f : f32(a3[s]);
  const float dg = f32(a4[s]);
  b4[d] = dg;
  b5[d] = dinv_f32 ? 1.0f / dg : f32(a5[s]);  // dinv_f32: reciprocal of the FP32 diagonal
}

// Dense matrix of the coarsest level's unknowns, inverted by Gauss-Jordan elimination
// (SPD: no pivoting) in one CTA.  The matrix lives in shared memory when it fits
// (m <= kCoarseSmemM), else in the output array.  At step k one warp scales the pivot row (one
// division) while another copies the pivot column, then every thread updates its elements, spread
// over all 32 warps: a step is bound by one SM's FP64 rate (m^2 multiply-adds at two a clock).
// With a thread per row (serial over its m elements, each thread dividing for itself) the 7 x 7
// coarsest level of a square grid took 207 us; so it takes 93 us (both ncu, cold caches), the same
// values bit for bit.
__global__ void __launch_bounds__(kCoarseFactorThreads) k_coarse_factor(Lvl<double> L, double* out, int* status) {
  extern __shared__ __align__(16) double smat[];
  __shared__ double rowk[kCoarseMax], colk[kCoarseMax];
  __shared__ int bad;
  const int ux = L.nx - 2;
  const int uy = L.periodic ? L.nyr : L.ny - 2;
  const int m = ux * uy;
  const int j0 = L.periodic ? 0 : 1;
  double* M = (m <= kCoarseSmemM) ? smat : out;
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) M[e] = 0.0;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  for (int p = threadIdx.x; p < m; p += blockDim.x) {
    const int i = 1 + p % ux, j = j0 + p / ux;
    for (int dj = -1; dj <= 1; ++dj)
      for (int di = -1; di <= 1; ++di) {
        const int ni = i + di;
        int nj = j + dj;
        if (L.periodic) nj = (nj + L.nyr) % L.nyr;
        const bool unk = (ni >= 1 && ni <= L.nx - 2) &&
                         (L.periodic || (nj >= 1 && nj <= L.ny - 2));
        if (!unk) continue;
        const int q = (ni - 1) + ux * (nj - j0);
        M[(size_t)p * m + q] += fine_entry(L, i, j, di, dj);
      }
  }
  __syncthreads();
  constexpr int KE = 4;  // elements a thread keeps indices of (m <= 64); larger m: recomputed
  const int nt = blockDim.x, t = threadIdx.x;
  int ei[KE], ej[KE];
#pragma unroll
  for (int r = 0; r < KE; ++r) {
    ei[r] = (t + r * nt) / m;
    ej[r] = (t + r * nt) - ei[r] * m;
  }
  for (int k = 0; k < m; ++k) {
    if (t < 32) {  // scaled pivot row, its reciprocal pivot at k
      const double piv = M[(size_t)k * m + k];
      if (!(piv > 0.0)) bad = 1;
      const double ip = 1.0 / piv;
      for (int jj = t; jj < m; jj += 32) rowk[jj] = (jj == k) ? ip : M[(size_t)k * m + jj] * ip;
    } else {
      for (int i = t - 32; i < m; i += nt - 32) colk[i] = M[(size_t)i * m + k];
    }
    __syncthreads();
    if (bad) {
      if (t == 0) *status = 11;
      return;  // uniform
    }
    const double ip = rowk[k];
    auto update = [&](int e, int i, int jj) {
      const double f = colk[i];
      M[e] = i == k ? rowk[jj] : (jj == k ? -f * ip : fma(-f, rowk[jj], M[e]));
    };
    if (m * m <= KE * nt) {
#pragma unroll
      for (int r = 0; r < KE; ++r)
        if (t + r * nt < m * m) update(t + r * nt, ei[r], ej[r]);
    } else {
      for (int e = t; e < m * m; e += nt) update(e, e / m, e - (e / m) * m);
    }
    __syncthreads();
  }
  if (M != out)
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) out[e] = M[e];
  if (threadIdx.x == 0) *status = 0;
}

// ------------------------------------------------------------------ host launchers
static dim3 grid2(int nx, int ny, dim3 b) { return dim3((nx + b.x - 1) / b.x, (ny + b.y - 1) / b.y); }

cudaError_t launch_eps_analytic(int kind, const double* prm, int nx, int ny, int periodic,
                                double x0, double y0, double hx, double hy, const double* eps,
                                int pitch, double* D, double* exx, double* exy, double* eyy,
                                int* folded, cudaStream_t s) {
  const int nyr = rows_stored(ny, periodic);
  dim3 b(32, 8), g((nx + kEpsTile - 1) / kEpsTile, (nyr + kEpsTile - 1) / kEpsTile);
  if (kind == 1) {
    k_eps_sine_warp<<<g, b, 0, s>>>(prm[0], nx, nyr, x0, y0, hx, hy, eps, pitch, D, exx, exy, eyy, folded);
    return cudaGetLastError();
  }
  if (kind == 2) {
    k_eps_polar<<<g, b, 0, s>>>(nx, nyr, x0, y0, hx, hy, eps, pitch, D, exx, exy, eyy, folded);
    return cudaGetLastError();
  }
  const double ja = kind == 4 ? prm[0] : 1.0, jb = kind == 4 ? prm[1] : 0.0, jc = kind == 4 ? prm[2] : 0.0,
               jd = kind == 4 ? prm[3] : 1.0, det = ja * jd - jb * jc;
  const auto f = kind == 3 ? k_eps_separable<true> : k_eps_separable<false>;
  f<<<g, b, 0, s>>>(prm[0], prm[1], det, (jd * jd + jb * jb) / det, (-jd * jc - jb * ja) / det,
                    (jc * jc + ja * ja) / det, nx, nyr, x0, y0, hx, hy, eps, pitch, D, exx, exy, eyy, folded,
                    map_kind_five_point(kind, prm) ? 0 : 1);
  return cudaGetLastError();
}

cudaError_t launch_mirror_eps(int nx, int n, int ps, const double* D0, const double* exx0,
                              const double* exy0, const double* eyy0, int pd, double* D, double* exx,
                              double* exy, double* eyy, cudaStream_t s) {
  dim3 b(32, 8);
  k_mirror_eps<<<grid2(nx, 2 * n, b), b, 0, s>>>(nx, n, ps, D0, exx0, exy0, eyy0, pd, D, exx, exy, eyy);
  return cudaGetLastError();
}

cudaError_t launch_eps_grid(int nx, int ny, int periodic, double hx, double hy, const double* xp,
                            const double* yp, double jx, double jy, const double* eps, int pitch,
                            double* D, double* exx, double* exy, double* eyy, int* folded,
                            cudaStream_t s) {
  const int nyr = rows_stored(ny, periodic);
  dim3 b(32, 8);
  k_eps_grid<<<grid2(nx, nyr, b), b, 0, s>>>(nx, ny, nyr, periodic, 0.5 / hx, 0.5 / hy, xp, yp, jx, jy, eps,
                                             pitch, D, exx, exy, eyy, folded);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_assemble(const Op<T>& A, double hx, double hy, const T* exx, const T* exy, const T* eyy,
                            cudaStream_t s, bool dinv) {
  if constexpr (sizeof(T) == 8) {
    if (!A.five_point) return launch_assemble_nine(A, nullptr, hx, hy, exx, exy, eyy, s, dinv);
  }
  const int nyr = rows_stored(A.ny, A.periodic);
  dim3 b(32, 8);
  k_assemble_couplings<T><<<grid2(A.nx, nyr, b), b, 0, s>>>(
      A.nx, A.ny, nyr, A.periodic, A.pitch, T(1.0 / (hx * hx)), T(1.0 / (hy * hy)), T(1.0 / (4.0 * hx * hy)),
      exx, exy, eyy, A.cE, A.cN, A.cNE, A.cNW, A.five_point);
  k_assemble_diag<T><<<grid2(A.nx, nyr, b), b, 0, s>>>(A.nx, A.ny, nyr, A.periodic, A.pitch, A.cE,
                                                       A.cN, A.cNE, A.cNW, A.diag, dinv ? A.dinv : nullptr,
                                                       A.five_point);
  return cudaGetLastError();
}
template cudaError_t launch_assemble<double>(const OpF64&, double, double, const double*, const double*,
                                             const double*, cudaStream_t, bool);
template cudaError_t launch_assemble<float>(const OpF32&, double, double, const float*, const float*,
                                            const float*, cudaStream_t, bool);

// -(1/2) / h^2 exactly (halving is exact), as k_assemble_couplings rounds its couplings
template <bool FIVE>
static cudaError_t assemble_pass(const OpF64& A, const OpF32* B, double hx, double hy, const double* exx,
                                 const double* exy, const double* eyy, cudaStream_t s, bool dinv) {
  const int nyr = rows_stored(A.ny, A.periodic);
  // strips of eight rows (one row is read twice a strip); shorter ones on grids too small to hide a
  // strip's chain of loads (9-point, us by rows 1 / 2 / 8, two separate kernels: 129^2 3.0 / 4.4 / 12.7,
  // 4.7; 385^2 8.5 / 9.5 / 12.9, 11.5; 769^2 25.4 / 25.4 / 32.0, 31.0; 1025^2 43.5 / 41.4 / 42.8, 51.3;
  // 2049^2 165 / 158 / 154, 195)
  const int gx = (A.nx + kAsmCols - 1) / kAsmCols;
  const long long warps = (long long)gx * nyr;  // of one row each
  const int rows = warps <= 40 * kSMs ? 1 : warps <= 240 * kSMs ? 2 : 8;
  dim3 b(32, 8), g(gx, (nyr + 8 * rows - 1) / (8 * rows));
  k_assemble_pass<FIVE><<<g, b, 0, s>>>(
      A.nx, A.ny, nyr, A.periodic, A.pitch, -0.5 * (1.0 / (hx * hx)), -0.5 * (1.0 / (hy * hy)), 1.0 / (4.0 * hx * hy), exx,
      exy, eyy, rows, A.cE, A.cN, A.cNE, A.cNW, A.diag, dinv ? A.dinv : nullptr, B ? B->pitch : 0, B ? B->cE : nullptr,
      B ? B->cN : nullptr, B ? B->cNE : nullptr, B ? B->cNW : nullptr, B ? B->diag : nullptr, B ? B->dinv : nullptr);
  return cudaGetLastError();
}

cudaError_t launch_assemble_nine(const OpF64& A, const OpF32* B, double hx, double hy, const double* exx,
                                 const double* exy, const double* eyy, cudaStream_t s, bool dinv) {
  return assemble_pass<false>(A, B, hx, hy, exx, exy, eyy, s, dinv);
}

cudaError_t launch_assemble_five(const OpF64& A, const OpF32* B, double hx, double hy, const double* exx,
                                 const double* eyy, cudaStream_t s, bool dinv) {
  return assemble_pass<true>(A, B, hx, hy, exx, nullptr, eyy, s, dinv);
}

cudaError_t launch_rhs(const OpF64& A, const double* rho, int rho_pitch, const double* D, double* b,
                       cudaStream_t s) {
  const int nyr = rows_stored(A.ny, A.periodic);
  dim3 bl(32, 8);
  k_rhs<<<grid2(A.nx, nyr, bl), bl, 0, s>>>(A.nx, A.ny, nyr, A.periodic, A.pitch, rho, rho_pitch, D,
                                            b);
  return cudaGetLastError();
}

template <typename TS, typename TD>
cudaError_t launch_coarsen_eps(const Op<TS>& F, const Op<TD>& C, const TS* const* e, TD* const* c,
                               cudaStream_t s) {
  const int nyrc = rows_stored(C.ny, C.periodic);
  dim3 b(32, 8);
  k_coarsen_eps<TS, TD><<<grid2(C.nx, nyrc, b), b, 0, s>>>(F.nx, rows_stored(F.ny, F.periodic), F.pitch, C.nx,
                                                            C.ny, nyrc, C.pitch, C.periodic, e[0], e[1], e[2],
                                                            c[0], c[1], c[2], C.five_point);
  return cudaGetLastError();
}
template cudaError_t launch_coarsen_eps<double, double>(const OpF64&, const OpF64&, const double* const*,
                                                        double* const*, cudaStream_t);
template cudaError_t launch_coarsen_eps<double, float>(const OpF64&, const OpF32&, const double* const*,
                                                       float* const*, cudaStream_t);
template cudaError_t launch_coarsen_eps<float, float>(const OpF32&, const OpF32&, const float* const*,
                                                      float* const*, cudaStream_t);

template <typename T>
cudaError_t launch_galerkin(const Op<T>& F, const Op<T>& C, cudaStream_t s) {
  const int nyrc = rows_stored(C.ny, C.periodic);
  if constexpr (sizeof(T) == 8) {
    const uintptr_t all = (uintptr_t)F.cE | (uintptr_t)F.cN | (uintptr_t)F.cNE | (uintptr_t)F.cNW | (uintptr_t)F.diag;
    if (F.pitch % 2 == 0 && all % 16 == 0) {  // rows readable in pairs of columns
      // strips of eight coarse rows (one more fine row collapsed per strip: 6%), shorter on small levels,
      // whose few warps would leave SMs idle and wait for a strip's chain of loads (9-point, us by rows 1 / 2
      // / 8, k_galerkin: 129^2 -> 65^2 5.1 / 8.1 / 25.9, 6.0; 385^2 11.2 / 13.3 / 26.2, 14.3; 513^2 14.5 / 13.4
      // / 26.2, 18.6; 1025^2 52.6 / 47.1 / 63.3, 60.3; 4097^2 742 / 662 / 618, 906)
      const int gx = (C.nx + kGalCols - 1) / kGalCols;
      const long long warps = (long long)gx * nyrc;  // of one row each
      const int rows = warps <= 12 * kSMs ? 1 : warps <= 128 * kSMs ? 2 : 8;
      const dim3 g(gx, (nyrc + 4 * rows - 1) / (4 * rows));
      if (F.five_point)
        k_galerkin_rows<true><<<g, 128, 0, s>>>(lvl_of(F), C.nx, C.ny, nyrc, C.pitch, rows, C.cE, C.cN, C.cNE, C.cNW,
                                                C.diag, C.dinv);
      else
        k_galerkin_rows<false><<<g, 128, 0, s>>>(lvl_of(F), C.nx, C.ny, nyrc, C.pitch, rows, C.cE, C.cN, C.cNE, C.cNW,
                                                 C.diag, C.dinv);
      return cudaGetLastError();
    }
  }
  dim3 b(32, 4);
  if (F.five_point)
    k_galerkin<T, true><<<grid2(C.nx, nyrc, b), b, 0, s>>>(lvl_of(F), C.nx, C.ny, nyrc, C.pitch, C.cE,
                                                           C.cN, C.cNE, C.cNW, C.diag, C.dinv);
  else
    k_galerkin<T, false><<<grid2(C.nx, nyrc, b), b, 0, s>>>(lvl_of(F), C.nx, C.ny, nyrc, C.pitch, C.cE,
                                                            C.cN, C.cNE, C.cNW, C.diag, C.dinv);
  return cudaGetLastError();
}
template cudaError_t launch_galerkin<double>(const OpF64&, const OpF64&, cudaStream_t);
template cudaError_t launch_galerkin<float>(const OpF32&, const OpF32&, cudaStream_t);

// Coarsest operator in FP64 from an FP32 level (mixed path: its hierarchy is FP32).
__global__ void k_op_to_f64(int nx, int nyr, int ps, int pd, const float* __restrict__ a0,
                            const float* __restrict__ a1, const float* __restrict__ a2,
                            const float* __restrict__ a3, const float* __restrict__ a4, double* b0,
                            double* b1, double* b2, double* b3, double* b4, double* b5) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= nx || j >= nyr) return;
  const size_t s = (size_t)j * ps + i, d = (size_t)j * pd + i;
  b0[d] = a0[s];
  b1[d] = a1[s];
  b2[d] = a2[s];
  b3[d] = a3[s];
  b4[d] = a4[s];
  b5[d] = 1.0 / (double)a4[s];
}

cudaError_t launch_op_to_f64(const OpF32& A, const OpF64& B, cudaStream_t s) {
  const int nyr = rows_stored(A.ny, A.periodic);
  dim3 b(32, 8);
  k_op_to_f64<<<grid2(A.nx, nyr, b), b, 0, s>>>(A.nx, nyr, A.pitch, B.pitch, A.cE, A.cN, A.cNE, A.cNW,
                                                A.diag, B.cE, B.cN, B.cNE, B.cNW, B.diag, B.dinv);
  return cudaGetLastError();
}

cudaError_t launch_op_to_f32(const OpF64& A, const OpF32& B, cudaStream_t s, bool dinv_f32) {
  const int nyr = rows_stored(A.ny, A.periodic);
  dim3 b(32, 8);
  const long long nodes = (long long)A.nx * nyr;
  const auto f = nodes >= 100000 && nodes <= 2000000 ? k_op_to_f32<true> : k_op_to_f32<false>;
  f<<<grid2(A.nx, nyr, b), b, 0, s>>>(A.nx, nyr, A.pitch, B.pitch, A.cE, A.cN, A.cNE,
                                                A.cNW, A.diag, A.dinv, B.cE, B.cN, B.cNE, B.cNW,
                                                B.diag, B.dinv, A.five_point, dinv_f32 ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_coarse_factor(const OpF64& A, double* inv, int* status, cudaStream_t s) {
  const int m = coarse_unknowns(A.nx, A.ny, A.periodic);
  const size_t sm = (m <= kCoarseSmemM) ? (size_t)m * m * sizeof(double) : 0;
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(k_coarse_factor, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(kCoarseSmemM * kCoarseSmemM * sizeof(double)));
    if (e != cudaSuccess) return e;
    attr = true;
  }
  k_coarse_factor<<<1, kCoarseFactorThreads, sm, s>>>(lvl_of(A), inv, status);
  return cudaGetLastError();
}

}  // namespace mg

// ------------------------------------------------------------------ C ABI (mg_kernels.h)
using namespace mg;

static bool op_ok(const mgk_op_f64* A) {
  return A && A->nx >= 3 && A->ny >= 3 && A->pitch >= A->nx && A->cE && A->cN && A->cNE && A->cNW &&
         A->diag && A->dinv && (!A->periodic || A->ny >= 3);
}

extern "C" int mgk_eps_analytic(int kind, const double* params4, int nx, int ny, int periodic,
                                double x0, double y0, double hx, double hy, const double* eps_phys,
                                int pitch, double* D, double* exx, double* exy, double* eyy,
                                int* folded, void* stream) {
  if (kind < 0 || kind > 4 || !params4 || nx < 3 || ny < 3 || pitch < nx || !D || !exx || !exy ||
      !eyy || !folded)
    return 1;
  return launch_eps_analytic(kind, params4, nx, ny, periodic, x0, y0, hx, hy, eps_phys, pitch, D,
                             exx, exy, eyy, folded, (cudaStream_t)stream) == cudaSuccess ? 0 : 4;
}

extern "C" int mgk_eps_grid(int nx, int ny, int periodic, double hx, double hy, const double* xp,
                            const double* yp, double jump_x, double jump_y, const double* eps_phys,
                            int pitch, double* D, double* exx, double* exy, double* eyy,
                            int* folded, void* stream) {
  if (nx < 3 || ny < 3 || (periodic ? ny - 1 : ny) < 3 || pitch < nx || !xp || !yp || !D || !exx ||
      !exy || !eyy || !folded)
    return 1;
  return launch_eps_grid(nx, ny, periodic, hx, hy, xp, yp, jump_x, jump_y, eps_phys, pitch, D, exx,
                         exy, eyy, folded, (cudaStream_t)stream) == cudaSuccess ? 0 : 4;
}

extern "C" int mgk_assemble(const mgk_op_f64* A, double hx, double hy, const double* exx,
                            const double* exy, const double* eyy, void* stream) {
  if (!op_ok(A) || !exx || !exy || !eyy || !(hx > 0) || !(hy > 0)) return 1;
  return launch_assemble(op_from(*A), hx, hy, exx, exy, eyy, (cudaStream_t)stream) == cudaSuccess
             ? 0 : 4;
}

extern "C" int mgk_assemble_five(const mgk_op_f64* A, const mgk_op_f32* B, double hx, double hy,
                                 const double* exx, const double* eyy, void* stream) {
  if (!op_ok(A) || !A->five_point || !exx || !eyy || !(hx > 0) || !(hy > 0)) return 1;
  if (B && (B->nx != A->nx || B->ny != A->ny || B->periodic != A->periodic || B->pitch < B->nx || !B->cE ||
            !B->cN || !B->cNE || !B->cNW || !B->diag || !B->dinv))
    return 1;
  const OpF32 b = B ? op_from(*B) : OpF32();
  return launch_assemble_five(op_from(*A), B ? &b : nullptr, hx, hy, exx, eyy, (cudaStream_t)stream, true) ==
                 cudaSuccess
             ? 0 : 4;
}

extern "C" int mgk_rhs(const mgk_op_f64* A, const double* rho_phys, const double* D, double* b,
                       void* stream) {
  if (!A || A->nx < 3 || A->ny < 3 || A->pitch < A->nx || !rho_phys || !D || !b) return 1;
  return launch_rhs(op_from(*A), rho_phys, A->pitch, D, b, (cudaStream_t)stream) == cudaSuccess
             ? 0 : 4;
}

extern "C" int mgk_coarsen_eps(const mgk_op_f64* fine, const mgk_op_f64* coarse, const double* e0,
                               const double* e1, const double* e2, double* c0, double* c1, double* c2,
                               void* stream) {
  if (!fine || !coarse || !e0 || !e1 || !e2 || !c0 || !c1 || !c2 || fine->nx < 3 || fine->ny < 3 ||
      fine->pitch < fine->nx || coarse->pitch < coarse->nx || (fine->nx - 1) % 2 || (fine->ny - 1) % 2 ||
      coarse->nx != (fine->nx - 1) / 2 + 1 || coarse->ny != (fine->ny - 1) / 2 + 1 ||
      coarse->periodic != fine->periodic)
    return 1;
  const double* e[3] = {e0, e1, e2};
  double* c[3] = {c0, c1, c2};
  return launch_coarsen_eps(op_from(*fine), op_from(*coarse), e, c, (cudaStream_t)stream) == cudaSuccess ? 0
                                                                                                        : 4;
}

extern "C" int mgk_galerkin(const mgk_op_f64* fine, const mgk_op_f64* coarse, void* stream) {
  if (!op_ok(fine) || !op_ok(coarse) || (fine->nx - 1) % 2 || (fine->ny - 1) % 2 ||
      coarse->nx != (fine->nx - 1) / 2 + 1 || coarse->ny != (fine->ny - 1) / 2 + 1 ||
      coarse->periodic != fine->periodic)
    return 1;
  return launch_galerkin<double>(op_from(*fine), op_from(*coarse), (cudaStream_t)stream) ==
                 cudaSuccess ? 0 : 4;
}

extern "C" int mgk_op_to_f32(const mgk_op_f64* src, const mgk_op_f32* dst, void* stream) {
  if (!op_ok(src) || !dst || dst->nx != src->nx || dst->ny != src->ny || dst->pitch < dst->nx ||
      !dst->cE || !dst->cN || !dst->cNE || !dst->cNW || !dst->diag || !dst->dinv)
    return 1;
  return launch_op_to_f32(op_from(*src), op_from(*dst), (cudaStream_t)stream) == cudaSuccess ? 0
                                                                                                : 4;
}

extern "C" int mgk_coarse_factor(const mgk_op_f64* A, double* inv, int* status, void* stream) {
  if (!op_ok(A) || !inv || !status) return 1;
  const int uy = A->periodic ? A->ny - 1 : A->ny - 2;
  if ((A->nx - 2) * uy > kCoarseMax || uy < 1) return 1;
  return launch_coarse_factor(op_from(*A), inv, status, (cudaStream_t)stream) == cudaSuccess ? 0
                                                                                               : 4;
}
