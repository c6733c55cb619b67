// SELL-32 row product shared by the FP64 Krylov kernels.
#pragma once
#include "avip_internal.h"

namespace avip {

// One row of y = A v over the SELL-32 structure (diagonal first, then ascending columns).
// Slots are fetched in groups of 8 so that the column loads, the value loads and the
// dependent gathers of a group are all in flight together.
__device__ __forceinline__ double sell_row_dot(const SellView& A, int slice, int lane, int row,
                                               const double* __restrict__ v) {
  constexpr int U = 8;
  const int base = __ldg(A.sl_ptr + slice) + lane;
  const int w = __ldg(A.sl_w + slice);
  const int rl = __ldg(A.rlen + row);
  double acc = 0.0;
  for (int k0 = 0; k0 < w; k0 += U) {
    int c[U];
    double av[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = k0 + u;
      c[u] = row;
      av[u] = 0.0;
      if (k < rl) {
        c[u] = __ldg(A.col + base + k * kSlice);
        av[u] = __ldg(A.aval + base + k * kSlice);
      }
    }
    double xv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) xv[u] = (k0 + u < rl) ? __ldcg(v + c[u]) : 0.0;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k0 + u < rl) acc = fma(av[u], xv[u], acc);
  }
  return acc;
}

// Fused multiply-add in the accumulation type.
__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fma_t(float a, float b, float c) { return fmaf(a, b, c); }

// Contiguous share [sa, sb) of nsl slices for warp w of nw (equal slice counts).
__device__ __forceinline__ void warp_slices(int nsl, int w, int nw, int& sa, int& sb) {
  sa = (int)((long long)nsl * w / nw);
  sb = (int)((long long)nsl * (w + 1) / nw);
}

// Gathered vectors are written by other blocks in an earlier phase of the same launch and read
// after a grid (or cluster) barrier: release increment, acquire wait, then bar.sync, which orders
// every later weak load of the block after the other blocks' writes.  They are read with
// ld.global.ca (__ldca: cached in L1 and L2), never through the read-only .nc path, whose
// contents may go stale within a launch; neighbouring rows of a warp's contiguous share gather
// mostly the same entries, so L1 serves most of them.

}  // namespace avip
