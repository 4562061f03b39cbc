// The small levels of a point-smoothed V-cycle and the coarsest dense solve in one CTA, each level
// held in registers: a thread owns a 2 x 2 block of nodes of one level (one node per colour) with
// its couplings, diagonal and right-hand sides, all levels' threads side by side.  The iterate of a
// level lies in four shared-memory planes, one per colour, with a border; a colour phase is five
// shared-memory loads, nine multiply-adds and one barrier among the level's own warps.  What is
// left is a chain of about a dozen phases a level, each one barrier and one dependent sum long;
// the kernel that keeps the levels' arrays in shared memory (k_tail) took seventeen loads and the
// index arithmetic of a strided loop per node in each of them: 33^2 and below, V(2,2), FP32 30 us
// -> 14.4 us, FP64 50 -> 34 us (ncu, cold caches); there the FP64 pipe's latency is the chain.
//
// Values: per node the operations of k_tail in the same order; the dense solve sums a row of the
// inverse in a few interleaved partial sums instead of one chain.
#include <cstdint>

#include "mg_common.cuh"
#include "mg_fused.h"
#include "mg_launch.h"

namespace mg {

constexpr int kTBThreads = 512;
constexpr int kTBInvM = 128;  // inverses up to this order are brought into shared memory

// Blocks of a level, its threads (whole warps) and its shared memory in elements.
struct TailGeom {
  int nbx, nby, thr, pl;  // pl: elements of one plane
};
__host__ __device__ inline TailGeom tail_geom(int nx, int nyr) {
  TailGeom g;
  g.nbx = (nx + 1) / 2;
  g.nby = (nyr + 1) / 2;
  g.thr = (g.nbx * g.nby + 31) / 32 * 32;
  g.pl = (g.nbx + 2) * (g.nby + 2);
  return g;
}

template <typename T>
__global__ void __launch_bounds__(kTBThreads) k_tail_block(TailArgs<T> a, int inv_smem, const int* __restrict__ skip) {
  if (skip && *skip) return;
  extern __shared__ __align__(16) unsigned char tb_smem[];
  __shared__ double bs[kCoarseMax], part[kTBThreads];
  __shared__ T* s_x[kMaxTail];  // planes a b c d, then residual planes b c d
  __shared__ T* s_b[kMaxTail];  // right-hand side, row-major (levels above 0)
  const int nl = a.nlev, t = threadIdx.x;
  const Lvl<T>& Lc = a.lv[nl - 1].L;
  const int ux = Lc.nx - 2, m = ux * (Lc.periodic ? Lc.nyr : Lc.ny - 2), jc0 = Lc.periodic ? 0 : 1;
  double* const sinv = reinterpret_cast<double*>(tb_smem);
  if (inv_smem) {
    for (int e = t; e < m * m; e += kTBThreads)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(sinv + e)),
                   "l"(a.inv + e)
                   : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // this thread's level and block; every thread walks the same layout
  int ml = -1, bx = 0, by = 0, nth = 0;
  TailGeom mg_{};
  T *X = nullptr, *mb = nullptr;
  {
    T* p = reinterpret_cast<T*>(tb_smem + (inv_smem ? (size_t)m * m * sizeof(double) : 0));
    int off = 0;
    for (int l = 0; l < nl; ++l) {
      const Lvl<T>& L = a.lv[l].L;
      if (l < nl - 1) {
        const TailGeom g = tail_geom(L.nx, L.nyr);
        if (t >= off && t < off + g.thr) {
          ml = l;
          mg_ = g;
          nth = g.thr;
          by = (t - off) / g.nbx;
          bx = (t - off) - by * g.nbx;
          X = p;
        }
        if (t == 0) s_x[l] = p;
        off += g.thr;
        for (int e = t; e < 7 * g.pl; e += kTBThreads) p[e] = T(0);
        p += 7 * g.pl;
      } else {
        if (t == 0) s_x[l] = p;  // the coarsest iterate, row-major
        for (int e = t; e < L.nx * L.nyr; e += kTBThreads) p[e] = T(0);
        p += L.nx * L.nyr;
      }
      if (l > 0) {
        if (ml == l) mb = p;
        if (t == 0) s_b[l] = p;
        p += L.nx * L.nyr;
      }
    }
  }
  const bool on = ml >= 0 && by < mg_.nby;
  // couplings, diagonal, reciprocal diagonal, right-hand side and iterate of the block
  Lvl<T> L = a.lv[ml < 0 ? 0 : ml].L;
  const int i0 = 2 * bx, j0 = 2 * by, pw = mg_.nbx + 2, PL = mg_.pl;
  auto at = [&](const T* arr, int i, int j) -> T {
    if (!on || i < 0 || i >= L.nx) return T(0);
    if (L.periodic) j = j < 0 ? j + L.nyr : (j >= L.nyr ? j - L.nyr : j);
    else if (j < 0 || j >= L.nyr) return T(0);
    return __ldg(arr + (size_t)j * L.pitch + i);
  };
  auto pair = [&](const T* arr, int j, T& u, T& v) {
    u = at(arr, i0, j);
    v = at(arr, i0 + 1, j);
  };
  T E0l, E0x, E0y, E1l, E1x, E1y, Nmx, Nmy, N0x, N0y, N1x, N1y;
  T NEml, NEmx, NE0l, NE0x, NE0y, NE1x, NE1y, NWmy, NWmr, NW0x, NW0y, NW0r, NW1x, NW1y;
  E0l = at(L.cE, i0 - 1, j0);
  E1l = at(L.cE, i0 - 1, j0 + 1);
  pair(L.cE, j0, E0x, E0y);
  pair(L.cE, j0 + 1, E1x, E1y);
  pair(L.cN, j0 - 1, Nmx, Nmy);
  pair(L.cN, j0, N0x, N0y);
  pair(L.cN, j0 + 1, N1x, N1y);
  NEml = at(L.cNE, i0 - 1, j0 - 1);
  NEmx = at(L.cNE, i0, j0 - 1);
  NE0l = at(L.cNE, i0 - 1, j0);
  pair(L.cNE, j0, NE0x, NE0y);
  pair(L.cNE, j0 + 1, NE1x, NE1y);
  NWmy = at(L.cNW, i0 + 1, j0 - 1);
  NWmr = at(L.cNW, i0 + 2, j0 - 1);
  pair(L.cNW, j0, NW0x, NW0y);
  NW0r = at(L.cNW, i0 + 2, j0);
  pair(L.cNW, j0 + 1, NW1x, NW1y);
  T sa, sb, sc, sd, ga, gb, gc, gd;
  pair(L.dinv, j0, sa, sb);
  pair(L.dinv, j0 + 1, sc, sd);
  pair(L.diag, j0, ga, gb);
  pair(L.diag, j0 + 1, gc, gd);
  const bool u0 = i0 >= 1 && i0 <= L.nx - 2, u1 = i0 + 1 <= L.nx - 2;
  const bool v0 = L.periodic || (j0 >= 1 && j0 <= L.ny - 2), v1 = L.periodic || j0 + 1 <= L.ny - 2;
  const bool ma = on && u0 && v0, mbb = on && u1 && v0, mc = on && u0 && v1, md = on && u1 && v1;
  T ba = T(0), bb = T(0), bc = T(0), bd = T(0), xa = T(0), xb = T(0), xc = T(0), xd = T(0);
  if (ml == 0) {
    pair(a.lv[0].b, j0, ba, bb);
    pair(a.lv[0].b, j0 + 1, bc, bd);
    if (!a.zero) {
      pair(a.lv[0].x, j0, xa, xb);
      pair(a.lv[0].x, j0 + 1, xc, xd);
    }
  }
  // plane positions: own block, the block rows below and above (wrapped on a periodic level)
  const int ro = by + 1, rd = L.periodic && by == 0 ? mg_.nby : by, ru = L.periodic && by == mg_.nby - 1 ? 1 : by + 2;
  const int o = ro * pw + bx + 1, od = rd * pw + bx + 1, ou = ru * pw + bx + 1;
  T *A = X, *B = X + PL, *C = X + 2 * PL, *D = X + 3 * PL, *Rb = X + 4 * PL, *Rc = X + 5 * PL, *Rd = X + 6 * PL;
  auto barrier = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(ml + 1), "r"(nth) : "memory"); };  // the level's warps
  auto put = [&]() {
    if (on) A[o] = xa, B[o] = xb, C[o] = xc, D[o] = xd;
  };
  auto sum_a = [&]() {
    T s = E0x * xb;
    s = fma(E0l, B[o - 1], s);
    s = fma(N0x, xc, s);
    s = fma(Nmx, C[od], s);
    s = fma(NE0x, xd, s);
    s = fma(NEml, D[od - 1], s);
    s = fma(NW0x, D[o - 1], s);
    return fma(NWmy, D[od], s);
  };
  auto sum_b = [&]() {
    T s = E0y * A[o + 1];
    s = fma(E0x, xa, s);
    s = fma(N0y, xd, s);
    s = fma(Nmy, D[od], s);
    s = fma(NE0y, C[o + 1], s);
    s = fma(NEmx, C[od], s);
    s = fma(NW0y, xc, s);
    return fma(NWmr, C[od + 1], s);
  };
  auto sum_c = [&]() {
    T s = E1x * xd;
    s = fma(E1l, D[o - 1], s);
    s = fma(N1x, A[ou], s);
    s = fma(N0x, xa, s);
    s = fma(NE1x, B[ou], s);
    s = fma(NE0l, B[o - 1], s);
    s = fma(NW1x, B[ou - 1], s);
    return fma(NW0y, xb, s);
  };
  auto sum_d = [&]() {
    T s = E1y * C[o + 1];
    s = fma(E1x, xc, s);
    s = fma(N1y, B[ou], s);
    s = fma(N0y, xb, s);
    s = fma(NE1y, A[ou + 1], s);
    s = fma(NE0x, xa, s);
    s = fma(NW1y, A[ou], s);
    return fma(NW0r, A[o + 1], s);
  };
  auto colour = [&](int c) {  // order (0,0), (1,1), (1,0), (0,1)
    if (c == 0) {
      if (ma) A[o] = xa = (ba - sum_a()) * sa;
    } else if (c == 1) {
      if (md) D[o] = xd = (bd - sum_d()) * sd;
    } else if (c == 2) {
      if (mbb) B[o] = xb = (bb - sum_b()) * sb;
    } else {
      if (mc) C[o] = xc = (bc - sum_c()) * sc;
    }
    barrier();
  };
  __syncthreads();
  for (int l = 0; l < nl - 1; ++l) {
    if (ml == l) {
      if (l > 0 && on) {  // right-hand side left by the level above
        auto bat = [&](int i, int j) -> T { return i < L.nx && j < L.nyr ? mb[j * L.nx + i] : T(0); };
        ba = bat(i0, j0);
        bb = bat(i0 + 1, j0);
        bc = bat(i0, j0 + 1);
        bd = bat(i0 + 1, j0 + 1);
      }
      put();
      barrier();
      for (int s = 0; s < a.nu1; ++s)
        for (int c = 0; c < 4; ++c) colour(c);
      T ra = T(0), rb = T(0), rc = T(0), rdv = T(0);
      if (ma) ra = ba - fma(ga, xa, sum_a());
      if (mbb) rb = bb - fma(gb, xb, sum_b());
      if (mc) rc = bc - fma(gc, xc, sum_c());
      if (md) rdv = bd - fma(gd, xd, sum_d());
      if (on) Rb[o] = rb, Rc[o] = rc, Rd[o] = rdv;
      barrier();
      const Lvl<T>& H = a.lv[l + 1].L;
      if (on && bx < H.nx && by < H.nyr) {  // coarse node (bx, by)
        const bool unk = bx >= 1 && bx <= H.nx - 2 && (H.periodic || (by >= 1 && by <= H.ny - 2));
        T v = T(0);
        if (unk) {
          const T edge = Rb[o - 1] + rb + Rc[od] + rc;
          const T corner = Rd[od - 1] + Rd[od] + Rd[o - 1] + rdv;
          v = (T(4) * ra + T(2) * edge + corner) * T(0.0625);
        }
        s_b[l + 1][by * H.nx + bx] = v;
      }
    }
    __syncthreads();
  }
  {  // coarsest level: x = inv b
    const T* cb = s_b[nl - 1];
    for (int q = t; q < m; q += kTBThreads) bs[q] = (double)cb[(jc0 + q / ux) * Lc.nx + 1 + q % ux];
    if (inv_smem) asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const int mp = (m + 31) / 32 * 32, P = kTBThreads / mp;  // P threads share a row (m <= 256: P >= 2)
    const int q = t % mp, h = t / mp;
    const double* const iv = inv_smem ? sinv : a.inv;
    double s = 0.0;
    if (h < P && q < m)
      for (int k = h; k < m; k += P) s = fma(iv[(size_t)k * m + q], bs[k], s);
    part[t] = s;
    __syncthreads();
    if (t < m) {
      double v = part[t];
      for (int k = 1; k < P; ++k) v += part[t + k * mp];
      s_x[nl - 1][(jc0 + t / ux) * Lc.nx + 1 + t % ux] = (T)v;
    }
    __syncthreads();
  }
  for (int l = nl - 2; l >= 0; --l) {
    if (ml == l) {
      const Lvl<T>& H = a.lv[l + 1].L;
      const T* const hx = s_x[l + 1];
      const TailGeom hg = tail_geom(H.nx, H.nyr);
      auto e = [&](int I, int J) -> T {  // coarse correction at (I, J)
        if (l + 1 == nl - 1) return hx[J * H.nx + I];
        return hx[((J & 1) * 2 + (I & 1)) * hg.pl + (J / 2 + 1) * (hg.nbx + 2) + I / 2 + 1];
      };
      if (on) {
        const int I = bx, J = by, Jp = J + 1 == H.nyr ? 0 : J + 1;
        if (ma) xa += e(I, J);
        if (mbb) xb += T(0.5) * (e(I, J) + e(I + 1, J));
        if (mc) xc += T(0.5) * (e(I, J) + e(I, Jp));
        if (md) xd += T(0.25) * ((e(I, J) + e(I + 1, J)) + (e(I, Jp) + e(I + 1, Jp)));
      }
      put();
      barrier();
      for (int s = 0; s < a.nu2; ++s)
        for (int c = 3; c >= 0; --c) colour(c);
    }
    __syncthreads();
  }
  if (ml == 0 && on) {
    T* const gx = a.lv[0].x;
    auto st = [&](int i, int j, T v) {
      if (i < L.nx && j < L.nyr) gx[(size_t)j * L.pitch + i] = v;
    };
    st(i0, j0, xa);
    st(i0 + 1, j0, xb);
    st(i0, j0 + 1, xc);
    st(i0 + 1, j0 + 1, xd);
  }
}

// Dynamic shared memory the kernel needs for these levels, 0 when they do not fit it: point
// smoothing, at least one level above the coarsest, all levels' blocks on one CTA's threads, and an
// even row count on a periodic level.
template <typename T>
static size_t tail_block_smem(const TailArgs<T>& a, int* inv_smem) {
  if (a.line || a.nlev < 2) return 0;
  size_t n = 0;
  int thr = 0;
  for (int l = 0; l < a.nlev; ++l) {
    const Lvl<T>& L = a.lv[l].L;
    if (l < a.nlev - 1) {
      if (L.periodic && L.nyr % 2) return 0;
      const TailGeom g = tail_geom(L.nx, L.nyr);
      thr += g.thr;
      n += (size_t)7 * g.pl;
    } else {
      n += (size_t)L.nx * L.nyr;
    }
    if (l > 0) n += (size_t)L.nx * L.nyr;
  }
  if (thr > kTBThreads) return 0;
  const Lvl<T>& C = a.lv[a.nlev - 1].L;
  const int m = coarse_unknowns(C.nx, C.ny, C.periodic);
  *inv_smem = m <= kTBInvM;
  const size_t bytes = n * sizeof(T) + (*inv_smem ? (size_t)m * m * sizeof(double) : 0);
  return bytes <= kTailSmemMax ? bytes : 0;
}

template <typename T>
bool tail_block_can(const TailArgs<T>& a) {
  int s;
  return tail_block_smem(a, &s) > 0;
}

template <typename T>
cudaError_t launch_tail_block(const TailArgs<T>& a, const int* skip, cudaStream_t s) {
  int inv_smem = 0;
  const size_t sm = tail_block_smem(a, &inv_smem);
  if (sm == 0) return cudaErrorInvalidValue;
  static const cudaError_t attr =
      cudaFuncSetAttribute(k_tail_block<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTailSmemMax);
  if (attr != cudaSuccess) return attr;
  k_tail_block<T><<<1, kTBThreads, sm, s>>>(a, inv_smem, skip);
  return cudaGetLastError();
}

template bool tail_block_can<double>(const TailArgs<double>&);
template bool tail_block_can<float>(const TailArgs<float>&);
template cudaError_t launch_tail_block<double>(const TailArgs<double>&, const int*, cudaStream_t);
template cudaError_t launch_tail_block<float>(const TailArgs<float>&, const int*, cudaStream_t);

}  // namespace mg
