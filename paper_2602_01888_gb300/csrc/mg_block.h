// Register-block smoother, optionally with the residual and its restriction (k_block.cu).
#pragma once
#include <cuda_runtime.h>

#include "mg_launch.h"

namespace mg {

// Owned columns of a tile of two sweeps a pass, without the residual.
template <typename T>
constexpr int block_tile_width() {
  return sizeof(T) == 4 ? 52 : 22;
}

// Whether the kernel can run on these arrays: 16-byte aligned, a pitch that keeps rows 16-byte
// aligned, and an even row count on a periodic level.
template <typename T>
bool block_can(const Op<T>& A, const T* xin, const T* xout, const T* b);
// Whether it can also restrict the residual: sides of 2 m + 1, as in every exact hierarchy, and the
// diagonal (which smoothing alone does not read) 16-byte aligned.
template <typename T>
bool block_can_restrict(const Op<T>& A);

// xout = ns four-colour Gauss-Seidel sweeps of (xin [+ P eH]) in forward (rev = 0) or reversed
// colour order; xin != xout.  xin == nullptr: a zero iterate.  bH (nullable; rev = 0, eH
// nullptr, block_can_restrict): also the full weighting of b - A xout at the coarse nodes (0
// on the coarse boundary ring; row pitch pitch_c).  pitch_c is eH's row pitch otherwise.
template <typename T>
cudaError_t launch_smooth_block(const Op<T>& A, const T* xin, T* xout, const T* b, int ns, int rev, const T* eH, T* bH,
                                int pitch_c, const int* skip, cudaStream_t s);

}  // namespace mg
