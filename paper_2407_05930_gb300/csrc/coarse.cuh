// Dense coarsest-level solve (Sec. 5: a direct method on the coarsest level)
// shared by the stand-alone kernel and the persistent coarse-cycle kernel, so
// both give the same bits: Z = A_c^{-1} Y with the precomputed FP64 inverse,
// FP64 arithmetic.
#pragma once

#include <cstdint>

namespace amgsym {

// Units of work of the dense solve: one row times 8 columns.
__host__ __device__ inline int64_t coarse_units(int32_t n, int32_t C) { return (int64_t)n * ((C + 7) / 8); }

// Units warp, warp + nwarps, ... of Z (n x C) by whole warps: lane l sums the
// terms j = l, l + 32, ... in ascending order for 8 columns (the inverse's row
// read once per 8 columns, coalesced across the lanes; the lanes' rows of Y
// contiguous), then the lanes swap halves of their columns (xor 16, 8, 4) and
// add the rest (xor 2, 1): 9 FP64 adds a lane instead of 40, FP64 issue (16
// cycles a warp instruction) being what bounds this kernel.  LD(p) loads one Y
// value or one 16-byte vector of them (through L2 when Y was written in the
// same launch).
template <typename T, typename LD>
__device__ __forceinline__ void coarse_rows_warp(int32_t n, int32_t C, const double* __restrict__ Ainv,
                                                 const T* Y, T* Z, int64_t warp, int64_t nwarps, LD ld) {
  constexpr int NV = 16 / (int)sizeof(T);  // values of a 16-byte vector
  struct alignas(16) V16 {
    T v[NV];
  };
  const int lane = threadIdx.x & 31;
  const int groups = (C + 7) / 8;
  const bool vec = C % 8 == 0 && ((uintptr_t)Y & 15) == 0;
  for (int64_t u0 = warp; u0 < coarse_units(n, C); u0 += nwarps) {
    const int i = (int)(u0 / groups), c0 = (int)(u0 - (int64_t)i * groups) * 8;
    const double* a = Ainv + (int64_t)i * n;
    const int nc = C - c0 < 8 ? C - c0 : 8;
    double acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = 0.0;
    auto row = [&](int j, T (&yv)[8]) {
      const T* y = Y + (int64_t)j * C + c0;
      if (vec) {
#pragma unroll
        for (int h = 0; h < 8 / NV; ++h) {
          const uint4 w = ld(reinterpret_cast<const uint4*>(y) + h);
          const V16 t = *reinterpret_cast<const V16*>(&w);
#pragma unroll
          for (int q = 0; q < NV; ++q) yv[h * NV + q] = t.v[q];
        }
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) yv[q] = q < nc ? ld(y + q) : (T)0;
      }
    };
    // two terms per lane in flight (all loads first, then the fmas in
    // ascending j: the same sum as one term at a time)
    int j = lane;
    for (; j + 32 < n; j += 64) {
      double av[2];
      T yv[2][8];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        av[u] = a[j + 32 * u];
        row(j + 32 * u, yv[u]);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q < nc) acc[q] = fma(av[u], (double)yv[u][q], acc[q]);
      }
    }
    if (j < n) {
      const double av = a[j];
      T yv[8];
      row(j, yv);
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q < nc) acc[q] = fma(av, (double)yv[q], acc[q]);
    }
    int col = 0;
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1) {
      const int off = 4 * h;
      const bool up = (lane & off) != 0;
#pragma unroll
      for (int q = 0; q < h; ++q) {
        const double send = up ? acc[q] : acc[q + h];
        const double keep = up ? acc[q + h] : acc[q];
        acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, off);
      }
      if (up) col += h;
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
    if ((lane & 3) == 0 && col < nc) Z[(int64_t)i * C + c0 + col] = (T)acc[0];
  }
}

}  // namespace amgsym
