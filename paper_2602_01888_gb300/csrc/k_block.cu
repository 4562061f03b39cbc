// Register-block smoother: ns four-colour Gauss-Seidel sweeps (Sec. 2.1, omega = 1) of a tile in
// one pass, optionally after the coarse correction (Eq. 24), optionally followed by the residual
// and its full weighting (Eqs. 20-23).
//
// A thread owns a 2 x 2 block of nodes, one of each colour: a (0,0), b (1,0), c (0,1), d (1,1), and
// keeps its right-hand sides, reciprocal diagonals and the 26 couplings that touch the block in
// registers for all 4 ns phases.  Of a node's eight neighbours three are the thread's own, so a
// phase takes five shared-memory loads, nine multiply-adds and one store per node; the iterate
// lies in four planes, one per colour, in which every access is unit-stride.  (The tile kernels
// that keep the couplings in shared memory take seventeen loads a node.)  A warp is one row of
// blocks (64 columns x 2 rows); phases skip the block rows that no longer matter.
//
// Halo, recomputed around the owned nodes: successive phases of a sweep step one row, and one
// column unless their colours share it, so an owned tile that starts on an even row and column and
// ends on odd ones needs ns = 1: 3 columns to its left, 2 to its right, 4 rows; ns = 2: 5, 4 and 8;
// with the residual and its weighting (coarse nodes of the tile) 2 more to the left and below, and
// two more to the right.  CTAs are persistent: once
// a tile's couplings are in registers its staging area is refilled by 16-byte asynchronous
// copies of the next tile, which land behind the phases.
//
// What bounds it: on small levels the latency of one tile (copies, then 4 ns phases of a barrier and
// a dependent chain each); from 1025^2 up the shared-memory pipe (LSU wavefronts 44%, issue slots 44%
// of peak at 4097^2) of one 1024-thread CTA per SM, not HBM (DRAM bytes equal the algorithmic 32 a
// node).  Two FP32 sweeps, against the kernel each size used before (CUDA events, launches from the
// host): 129^2 15.5 -> 5.3 us, 513^2 14.4 -> 6.2 us, 1025^2 36.9 -> 16.7 us (tile kernels), 4097^2
// 203 -> 164 us (row marching).  Marching a strip with everything in one warp's registers, without
// any barrier, was slower (177 us at 4097^2, 18 us at 1025^2: two warps a scheduler cannot hide the
// chain of a step).  FP64 (32 x 32 regions, two CTAs an SM) is bound by a phase's chain of ten FP64
// operations: two sweeps with the restriction or the correction take about 11 us at 65^2 and 129^2,
// where the fused tile kernel took 18 us without either.
//
// Operations per node and their order are those of the per-colour kernels and of
// k_resid_restrict, so the results are the same bit for bit.
#include <cstdint>
#include <type_traits>

#include "mg_block.h"
#include "mg_common.cuh"
#include "mg_launch.h"

namespace mg {

template <typename T, int NS, int TX_, int TY, bool RR>
struct BlockGeom {
  static constexpr int TX = TX_;                     // blocks a row (a warp or half a warp)
  static constexpr int RX = 2 * TX, RY = 2 * TY;     // nodes of the staged region
  static constexpr int VEC = 16 / (int)sizeof(T);    // elements of a 16-byte chunk
  // halo columns (left, right) and rows (below, above): see the reach in the head of this file; left
  // and below rounded up to whole chunks and blocks, the owned width to whole chunks
  static constexpr int HL = VEC == 4 ? (NS == 2 || RR ? 8 : 4) : (NS == 2 ? (RR ? 8 : 6) : (RR ? 6 : 4));
  static constexpr int HR = VEC == 4 ? (NS == 2 && RR ? 8 : 4) : (NS == 2 ? (RR ? 6 : 4) : (RR ? 4 : 2));
  static constexpr int HB = 4 * NS + (RR ? 2 : 0), HT = 4 * NS;
  static constexpr int OX = RX - HL - HR, OY = RY - HB - HT;
  static constexpr int THREADS = TX * TY;
  static constexpr int CTAS = sizeof(T) == 8 ? 2 : 1;  // resident CTAs a SM
  static constexpr int PLANE = TX * TY;
  static constexpr int CHX = RX / VEC, CHUNKS = CHX * RY;  // chunks of a row, of an array
  static constexpr int CW = TX + 1, CH = TY + 1;     // coarse nodes under the region
  // elements: 7 staged arrays, the iterate's planes, the coarse correction; with RR two buffers of
  // the diagonal (the next tile's arrives while this one's is needed) and three residual planes
  static constexpr int ARR = RX * RY;
  static constexpr int ELEMS = 7 * ARR + 4 * PLANE + CW * CH + (RR ? 2 * ARR + 3 * PLANE : 0);
  static constexpr int SMEM = ((ELEMS * (int)sizeof(T) + 15) / 16) * 16;
  static_assert(OX > 0 && OY > 0, "no owned nodes");
  static_assert(HL % VEC == 0 && OX % VEC == 0 && OX % 2 == 0 && OY % 2 == 0, "region starts on a chunk and a block");
  static_assert(CTAS * (SMEM + 1024 + 32) <= 228 * 1024, "resident CTAs must fit in shared memory");
};

template <int BYTES>
__device__ __forceinline__ void blk_copy(void* dst, const void* src, bool on) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = on ? BYTES : 0;  // 0: zero fill
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(BYTES), "r"(n) : "memory");
}

template <typename T>
struct T2;
template <>
struct T2<float> {
  using type = float2;
};
template <>
struct T2<double> {
  using type = double2;
};

template <typename T, int NS, int TX, int TY, bool REV, bool RR, bool FIVE>
__global__ void __launch_bounds__(TX * TY, BlockGeom<T, NS, TX, TY, RR>::CTAS)
    k_smooth_block(Lvl<T> L, const T* __restrict__ xin, T* __restrict__ xout, const T* __restrict__ b,
                   const T* __restrict__ eH, T* __restrict__ bH, int pitchc, int nxc, int nyc, int nyrc, int tiles_x,
                   int ntiles, const int* __restrict__ skip) {
  if (skip && *skip) return;
  using G = BlockGeom<T, NS, TX, TY, RR>;
  using P2 = typename T2<T>::type;
  constexpr int RX = G::RX, RY = G::RY, PL = G::PLANE, ARR = G::ARR;
  extern __shared__ __align__(16) unsigned char blk_smem[];
  T* const stage = reinterpret_cast<T*>(blk_smem);  // E N NE NW 1/diag b x
  T* const plane = stage + 7 * ARR;
  T* const es = plane + 4 * PL;
  T* const dg = es + ((G::CW * G::CH + 3) & ~3);  // 2 x ARR (RR)
  T* const rp = dg + 2 * ARR;                     // residual planes b, c, d (RR)
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX, t = threadIdx.x;
  const int p = L.pitch;

  auto request = [&](int tile, int buf) {
    const int X0 = (tile % tiles_x) * G::OX - G::HL, Y0 = (tile / tiles_x) * G::OY - G::HB;
    for (int q = t; q < G::CHUNKS; q += G::THREADS) {
      const int ly = q / G::CHX, lx = (q - ly * G::CHX) * G::VEC;
      const int i = X0 + lx;
      int j = Y0 + ly;
      bool on = i >= 0 && i + G::VEC <= p;
      if (L.periodic) {
        j %= L.nyr;
        if (j < 0) j += L.nyr;
      } else {
        on = on && j >= 0 && j < L.nyr;
      }
      const size_t k = on ? (size_t)j * p + i : 0;
      T* const d = stage + ly * RX + lx;
      blk_copy<16>(d, L.cE + k, on);
      blk_copy<16>(d + ARR, L.cN + k, on);
      if (!FIVE) {
        blk_copy<16>(d + 2 * ARR, L.cNE + k, on);
        blk_copy<16>(d + 3 * ARR, L.cNW + k, on);
      }
      blk_copy<16>(d + 4 * ARR, L.dinv + k, on);
      blk_copy<16>(d + 5 * ARR, b + k, on);
      if (xin) blk_copy<16>(d + 6 * ARR, xin + k, on);
      if (RR) blk_copy<16>(dg + buf * ARR + ly * RX + lx, L.diag + k, on);
    }
    if (!RR && eH) {
      const int I0 = X0 / 2, J0 = Y0 / 2;  // even starts
      for (int q = t; q < G::CW * G::CH; q += G::THREADS) {
        const int cy = q / G::CW, I = I0 + (q - cy * G::CW);
        int J = J0 + cy;
        bool on = I >= 0 && I < nxc;
        if (L.periodic) {
          J %= nyrc;
          if (J < 0) J += nyrc;
        } else {
          on = on && J >= 0 && J < nyrc;
        }
        blk_copy<(int)sizeof(T)>(es + q, eH + (on ? (size_t)J * pitchc + I : 0), on);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  int tile = blockIdx.x, buf = 0;
  if (tile >= ntiles) return;
  request(tile, 0);
  for (; tile < ntiles; tile += gridDim.x, buf ^= 1) {
    const int X0 = (tile % tiles_x) * G::OX - G::HL, Y0 = (tile / tiles_x) * G::OY - G::HB;
    const int i0 = X0 + 2 * tx, j0 = Y0 + 2 * ty;
    const bool u0 = i0 >= 1 && i0 <= L.nx - 2, u1 = i0 + 1 >= 1 && i0 + 1 <= L.nx - 2;
    const bool v0 = L.periodic || (j0 >= 1 && j0 <= L.ny - 2), v1 = L.periodic || (j0 + 1 >= 1 && j0 + 1 <= L.ny - 2);
    const bool ma = u0 && v0, mb = u1 && v0, mc = u0 && v1, md = u1 && v1;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    // couplings, right-hand side and reciprocal diagonal of the block into registers
    const int o0 = (2 * ty) * RX + 2 * tx, o1 = o0 + RX, om = ty > 0 ? o0 - RX : o0;  // rows j0, j0 + 1, j0 - 1
    auto pair = [&](int arr, int o) { return *reinterpret_cast<const P2*>(stage + arr * ARR + o); };
    const P2 E0 = pair(0, o0), E1 = pair(0, o1);
    const T E0l = __shfl_up_sync(0xffffffffu, E0.y, 1), E1l = __shfl_up_sync(0xffffffffu, E1.y, 1);
    const P2 Nm = pair(1, om), N0 = pair(1, o0), N1 = pair(1, o1);
    P2 NEm{}, NE0{}, NE1{}, NWm{}, NW0{}, NW1{};
    T NEml = T(0), NE0l = T(0), NWmr = T(0), NW0r = T(0);
    if (!FIVE) {
      NEm = pair(2, om), NE0 = pair(2, o0), NE1 = pair(2, o1);
      NWm = pair(3, om), NW0 = pair(3, o0), NW1 = pair(3, o1);
      NEml = __shfl_up_sync(0xffffffffu, NEm.y, 1);
      NE0l = __shfl_up_sync(0xffffffffu, NE0.y, 1);
      NWmr = __shfl_down_sync(0xffffffffu, NWm.x, 1);
      NW0r = __shfl_down_sync(0xffffffffu, NW0.x, 1);
    }
    const P2 D0 = pair(4, o0), D1 = pair(4, o1), b0 = pair(5, o0), b1 = pair(5, o1);
    T xa = T(0), xb = T(0), xc = T(0), xd = T(0);
    if (xin) {
      const P2 r0 = pair(6, o0), r1 = pair(6, o1);
      xa = r0.x, xb = r0.y, xc = r1.x, xd = r1.y;
    }
    if (!RR && eH) {  // bilinear coarse correction at the unknowns
      const T ea = es[ty * G::CW + tx], eb = es[ty * G::CW + tx + 1], ec = es[(ty + 1) * G::CW + tx],
              ed = es[(ty + 1) * G::CW + tx + 1];
      if (ma) xa += ea;
      if (mb) xb += T(0.5) * (ea + eb);
      if (mc) xc += T(0.5) * (ea + ec);
      if (md) xd += T(0.25) * ((ea + eb) + (ec + ed));
    }
    T* const A = plane + ty * TX + tx;
    T* const B = A + PL;
    T* const C = B + PL;
    T* const D = C + PL;
    *A = xa;
    *B = xb;
    *C = xc;
    *D = xd;
    __syncthreads();
    if (tile + (int)gridDim.x < ntiles) request(tile + gridDim.x, buf ^ 1);

    // off-diagonal sums, terms in the order of offdiag().  The planes are indexed past a block row's
    // ends at the region's edges: still inside the planes, values unused.
    auto sum_a = [&]() {
      T s = E0.x * xb;
      s = fma(E0l, B[-1], s);
      s = fma(N0.x, xc, s);
      s = fma(Nm.x, C[-TX], s);
      if (!FIVE) {
        s = fma(NE0.x, xd, s);
        s = fma(NEml, D[-TX - 1], s);
        s = fma(NW0.x, D[-1], s);
        s = fma(NWm.y, D[-TX], s);
      }
      return s;
    };
    auto sum_b = [&]() {
      T s = E0.y * A[1];
      s = fma(E0.x, xa, s);
      s = fma(N0.y, xd, s);
      s = fma(Nm.y, D[-TX], s);
      if (!FIVE) {
        s = fma(NE0.y, C[1], s);
        s = fma(NEm.x, C[-TX], s);
        s = fma(NW0.y, xc, s);
        s = fma(NWmr, C[-TX + 1], s);
      }
      return s;
    };
    auto sum_c = [&]() {
      T s = E1.x * xd;
      s = fma(E1l, D[-1], s);
      s = fma(N1.x, A[TX], s);
      s = fma(N0.x, xa, s);
      if (!FIVE) {
        s = fma(NE1.x, B[TX], s);
        s = fma(NE0l, B[-1], s);
        s = fma(NW1.x, B[TX - 1], s);
        s = fma(NW0.y, xb, s);
      }
      return s;
    };
    auto sum_d = [&]() {
      T s = E1.y * C[1];
      s = fma(E1.x, xc, s);
      s = fma(N1.y, B[TX], s);
      s = fma(N0.y, xb, s);
      if (!FIVE) {
        s = fma(NE1.y, A[TX + 1], s);
        s = fma(NE0.x, xa, s);
        s = fma(NW1.y, A[TX], s);
        s = fma(NW0r, A[1], s);
      }
      return s;
    };
#pragma unroll
    for (int ph = 0; ph < 4 * NS; ++ph) {
      const int c = REV ? 3 - (ph & 3) : (ph & 3);  // colours a, d, b, c
      const int row = 2 * ty + ((c == 1 || c == 3) ? 1 : 0);
      if (row > ph && row < RY - 1 - ph) {
        if (c == 0) {
          const T v = (b0.x - sum_a()) * D0.x;
          if (ma) *A = xa = v;
        } else if (c == 1) {
          const T v = (b1.y - sum_d()) * D1.y;
          if (md) *D = xd = v;
        } else if (c == 2) {
          const T v = (b0.y - sum_b()) * D0.y;
          if (mb) *B = xb = v;
        } else {
          const T v = (b1.x - sum_c()) * D1.x;
          if (mc) *C = xc = v;
        }
      }
      if (ph + 1 < 4 * NS || RR) __syncthreads();
    }
    const bool own = 2 * tx >= G::HL && 2 * tx < RX - G::HR && 2 * ty >= G::HB && 2 * ty < RY - G::HT;
    if (own && i0 < L.nx) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        if (j0 + r >= L.nyr) continue;
        T* const o = xout + (size_t)(j0 + r) * p + i0;
        if (i0 + 1 < L.nx) {
          P2 v;
          v.x = r ? xc : xa;
          v.y = r ? xd : xb;
          *reinterpret_cast<P2*>(o) = v;
        } else {
          o[0] = r ? xc : xa;
        }
      }
    }
    if constexpr (RR) {
      const T* const d = dg + buf * ARR;
      const P2 g0 = *reinterpret_cast<const P2*>(d + o0), g1 = *reinterpret_cast<const P2*>(d + o1);
      // at the owned nodes and one block row and column before them
      const bool used = 2 * ty >= G::HB - 2 && 2 * ty < RY - G::HT;
      T ra = T(0), rb = T(0), rc = T(0), rd = T(0);
      if (used) {
        if (ma) ra = b0.x - fma(g0.x, xa, sum_a());
        if (mb) rb = b0.y - fma(g0.y, xb, sum_b());
        if (mc) rc = b1.x - fma(g1.x, xc, sum_c());
        if (md) rd = b1.y - fma(g1.y, xd, sum_d());
      }
      T* const Rb = rp + ty * TX + tx;
      T* const Rc = Rb + PL;
      T* const Rd = Rc + PL;
      *Rb = rb;
      *Rc = rc;
      *Rd = rd;
      __syncthreads();
      const int I = i0 >> 1, J = j0 >> 1;
      if (own && I < nxc && J < nyrc) {
        const bool unk = (I >= 1 && I <= nxc - 2) && (L.periodic || (J >= 1 && J <= nyc - 2));
        T v = T(0);
        if (unk) {
          const T edge = Rb[-1] + rb + Rc[-TX] + rc;
          const T corner = Rd[-TX - 1] + Rd[-TX] + Rd[-1] + rd;
          v = (T(4) * ra + T(2) * edge + corner) * T(0.0625);
        }
        bH[(size_t)J * pitchc + I] = v;
      }
    }
  }
}

// ------------------------------------------------------------------ launcher
static int blk_sms() {
  static const int n = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 148;
  }();
  return n;
}

template <typename T>
bool block_can(const Op<T>& A, const T* xin, const T* xout, const T* b) {
  const uintptr_t all = (uintptr_t)xin | (uintptr_t)xout | (uintptr_t)b | (uintptr_t)A.cE | (uintptr_t)A.cN |
                        (uintptr_t)A.cNE | (uintptr_t)A.cNW | (uintptr_t)A.dinv;
  return A.pitch % (16 / (int)sizeof(T)) == 0 && all % 16 == 0 && !(A.periodic && (A.ny - 1) % 2);
}

template <typename T>
bool block_can_restrict(const Op<T>& A) {
  return (uintptr_t)A.diag % 16 == 0 && (A.nx - 1) % 2 == 0 && (A.ny - 1) % 2 == 0;
}

template <typename T, int NS, int TX, int TY, bool RR>
static cudaError_t block_impl(const Op<T>& A, const T* xin, T* xout, const T* b, int rev, const T* eH, T* bH,
                              int pitch_c, const int* skip, cudaStream_t s) {
  using G = BlockGeom<T, NS, TX, TY, RR>;
  auto raise = [](auto kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM + 32);
  };
  static const cudaError_t attr = [&] {
    cudaError_t e = raise(k_smooth_block<T, NS, TX, TY, false, RR, false>);
    if (!e) e = raise(k_smooth_block<T, NS, TX, TY, false, RR, true>);
    if constexpr (!RR) {
      if (!e) e = raise(k_smooth_block<T, NS, TX, TY, true, RR, false>);
      if (!e) e = raise(k_smooth_block<T, NS, TX, TY, true, RR, true>);
    }
    return e;
  }();
  if (attr != cudaSuccess) return attr;
  const Lvl<T> L = lvl_of(A);
  const int nxc = (A.nx - 1) / 2 + 1, nyc = (A.ny - 1) / 2 + 1, nyrc = rows_stored(nyc, A.periodic);
  const int tx = (L.nx + G::OX - 1) / G::OX, ty = (L.nyr + G::OY - 1) / G::OY, ntiles = tx * ty;
  const int slots = blk_sms() * G::CTAS, grid = ntiles < slots ? ntiles : slots;
  auto go = [&](auto kern) {
    kern<<<grid, G::THREADS, G::SMEM + 32, s>>>(L, xin, xout, b, eH, bH, pitch_c, nxc, nyc, nyrc, tx, ntiles, skip);
    return cudaGetLastError();
  };
  if constexpr (!RR) {
    if (rev)
      return L.five_point ? go(k_smooth_block<T, NS, TX, TY, true, RR, true>) : go(k_smooth_block<T, NS, TX, TY, true, RR, false>);
  }
  return L.five_point ? go(k_smooth_block<T, NS, TX, TY, false, RR, true>) : go(k_smooth_block<T, NS, TX, TY, false, RR, false>);
}

template <typename T>
cudaError_t launch_smooth_block(const Op<T>& A, const T* xin, T* xout, const T* b, int ns, int rev, const T* eH, T* bH,
                                int pitch_c, const int* skip, cudaStream_t s) {
  if (xin == xout || !block_can(A, xin, xout, b) || (bH && (rev || eH || !block_can_restrict(A))))
    return cudaErrorInvalidValue;
  if (ns != 1 && ns != 2) return cudaErrorInvalidValue;
  const int nyr = rows_stored(A.ny, A.periodic);
  auto go = [&](auto ns_c, auto tx_c, auto ty_c) {
    constexpr int NS = decltype(ns_c)::value, TX = decltype(tx_c)::value, TY = decltype(ty_c)::value;
    return bH ? block_impl<T, NS, TX, TY, true>(A, xin, xout, b, rev, eH, bH, pitch_c, skip, s)
              : block_impl<T, NS, TX, TY, false>(A, xin, xout, b, rev, eH, bH, pitch_c, skip, s);
  };
  using One = std::integral_constant<int, 1>;
  using Two = std::integral_constant<int, 2>;
  using N16 = std::integral_constant<int, 16>;
  using N32 = std::integral_constant<int, 32>;
  if constexpr (sizeof(T) == 4) {
    // tall tiles (64 rows) where they fill the GPU, half as tall ones on small levels
    const bool tall = (long long)A.nx * nyr > 48LL * 16 * kSMs;
    if (ns == 2) return tall ? go(Two(), N32(), N32()) : go(Two(), N32(), N16());
    return tall ? go(One(), N32(), N32()) : go(One(), N32(), N16());
  } else {
    // 32 x 32 regions: a phase is a chain of ten FP64 operations whatever the tile, so small tiles on
    // many SMs (the levels this kernel is chosen for have few)
    return ns == 2 ? go(Two(), N16(), N16()) : go(One(), N16(), N16());
  }
}

#define MG_BLOCK_INST(T)                                                                                             \
  template bool block_can<T>(const Op<T>&, const T*, const T*, const T*);                                            \
  template bool block_can_restrict<T>(const Op<T>&);                                                                 \
  template cudaError_t launch_smooth_block<T>(const Op<T>&, const T*, T*, const T*, int, int, const T*, T*, int,     \
                                              const int*, cudaStream_t);
MG_BLOCK_INST(float)
MG_BLOCK_INST(double)
#undef MG_BLOCK_INST

}  // namespace mg
