// Multi-vector kernels of the GMRES solve and of the low-rank correction
// (LRCAMG, Sec. 2.2): dots of one vector with many, sums of many vectors with
// per-column coefficients, per-column scaling.  FP64, interleaved [rows][C]
// layouts.  A "vector set" V holds J vectors of rows x Cv values, vector j at
// V + j * vstride; column c of a [rows][C] vector pairs with column c % Cv of
// the set (Cv = C for GMRES bases, Cv = 2^s for per-block correction vectors
// shared by every right-hand side).  Sums run in a fixed order (per-thread
// rows, then a fixed combination across threads and blocks): results are
// bit-reproducible run to run.
#include <cuda_runtime.h>

#include <algorithm>

#include "device.h"
#include "dot.cuh"

namespace amgsym {

namespace {

constexpr int kJChunk = 8;  // vectors of a set per pass over W

// part[(blk * J + j) * C + c] = sum over this block's rows of V_j[row][c % Cv] * W[row][c].
// A thread keeps kJChunk sums of one column.  With C dividing a warp the lanes
// of a column combine by the halving exchange of dot.cuh (they swap half of
// their kJChunk sums), and one barrier per chunk hands the warps' lines to
// the threads that add them; otherwise every row slot leaves its line.
__global__ void __launch_bounds__(kBlock) mdot_partial_kernel(const double* V, int64_t vstride,
                                                              int32_t Cv, int32_t J, const double* W,
                                                              int64_t rows, int32_t C, double* __restrict__ part) {
  pdl_wait();
  __shared__ double sm[kJChunk * kBlock];  // [line][u][column]
  const int rpb = kBlock / C;  // rows per block step
  const int col = threadIdx.x % C, rl = threadIdx.x / C;
  const bool act = rl < rpb;
  const int vc = col % Cv;
  const bool shuffles = dot_shuffles(C);
  const int lines = dot_lines(C, rpb);
  for (int j0 = 0; j0 < J; j0 += kJChunk) {
    double acc[kJChunk];
#pragma unroll
    for (int u = 0; u < kJChunk; ++u) acc[u] = 0.0;
    if (act) {
      for (int64_t row = blockIdx.x * (int64_t)rpb + rl; row < rows; row += (int64_t)gridDim.x * rpb) {
        const double w = W[row * C + col];
#pragma unroll
        for (int u = 0; u < kJChunk; ++u)
          if (j0 + u < J) acc[u] = fma(V[(int64_t)(j0 + u) * vstride + row * Cv + vc], w, acc[u]);
      }
    }
    __syncthreads();  // the previous chunk's lines have been read
    if (shuffles) {
      int sub = 0;
      bool dup = false;
      dot_exchange<kJChunk, kJChunk>(acc, C, threadIdx.x & 31, sub, dup);
      const int left = kJChunk * C > 32 ? kJChunk * C / 32 : 1;
      double* line = sm + (threadIdx.x >> 5) * kJChunk * C + sub * C + col;
#pragma unroll
      for (int u = 0; u < kJChunk; ++u)
        if (!dup && u < left) line[u * C] = acc[u];
    } else if (act) {
#pragma unroll
      for (int u = 0; u < kJChunk; ++u) sm[rl * kJChunk * C + u * C + col] = acc[u];
    }
    __syncthreads();
    const int nu = min(kJChunk, J - j0) * C;
    for (int t = threadIdx.x; t < nu; t += kBlock) {
      double s[4] = {0.0, 0.0, 0.0, 0.0};
      int r = 0;
      for (; r + 4 <= lines; r += 4) {
#pragma unroll
        for (int q = 0; q < 4; ++q) s[q] += sm[(r + q) * kJChunk * C + t];
      }
      for (; r < lines; ++r) s[0] += sm[r * kJChunk * C + t];
      part[((int64_t)blockIdx.x * J + j0) * C + t] = (s[0] + s[1]) + (s[2] + s[3]);
    }
  }
}

// H[t] = sum over blocks of part[b * n + t], n = J * C.  A block serves
// kFinalCols consecutive sums with kBlock / kFinalCols threads each (their
// terms strided, then halved in shared memory).  One thread per sum walked up
// to 608 dependent adds, 110 us a call and two thirds of a GMRES step at 64^3,
// s = 3; with the exchanges above the solve to 1e-12 went from 22.0 to 12.8 ms.
constexpr int kFinalCols = 8;
__global__ void __launch_bounds__(kBlock) mdot_final_kernel(const double* part, int32_t nblk, int32_t n,
                                                            double* __restrict__ H) {
  pdl_wait();
  __shared__ double sm[kBlock];
  constexpr int kSlices = kBlock / kFinalCols;
  const int t = blockIdx.x * kFinalCols + threadIdx.x % kFinalCols;
  const int sl = threadIdx.x / kFinalCols;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  if (t < n) {
    int b = sl;
    for (; b + 3 * kSlices < nblk; b += 4 * kSlices) {
#pragma unroll
      for (int q = 0; q < 4; ++q) s[q] += part[(int64_t)(b + q * kSlices) * n + t];
    }
#pragma unroll
    for (int q = 0; q < 3; ++q)
      if (b + q * kSlices < nblk) s[q] += part[(int64_t)(b + q * kSlices) * n + t];
  }
  sm[threadIdx.x] = (s[0] + s[1]) + (s[2] + s[3]);
  for (int h = kSlices / 2; h >= 1; h >>= 1) {
    __syncthreads();
    if (sl < h) sm[threadIdx.x] += sm[threadIdx.x + h * kFinalCols];
  }
  if (sl == 0 && t < n) H[t] = sm[threadIdx.x];
}

// W[row][c] += sign * sum_j V_j[row][c % Cv] * H[j * C + c]  (j in order).
__global__ void __launch_bounds__(kBlock) maxpy_kernel(const double* V, int64_t vstride, int32_t Cv,
                                                       int32_t J, const double* H, double sign,
                                                       double* __restrict__ W, int64_t rows, int32_t C) {
  pdl_wait();
  const int64_t total = rows * C;
  for (int64_t e = blockIdx.x * (int64_t)kBlock + threadIdx.x; e < total; e += (int64_t)gridDim.x * kBlock) {
    const int64_t row = e / C;
    const int c = (int)(e - row * C);
    const int64_t vo = row * Cv + c % Cv;
    double acc = 0.0;
    for (int j = 0; j < J; ++j) acc = fma(V[(int64_t)j * vstride + vo], H[j * C + c], acc);
    W[e] = fma(sign, acc, W[e]);
  }
}

// Out[row][c] = W[row][c] * s[c].
__global__ void __launch_bounds__(kBlock) colscale_kernel(const double* W, const double* s,
                                                          double* out, int64_t rows, int32_t C) {
  pdl_wait();
  const int64_t total = rows * C;
  for (int64_t e = blockIdx.x * (int64_t)kBlock + threadIdx.x; e < total; e += (int64_t)gridDim.x * kBlock)
    out[e] = W[e] * s[e % C];
}

// out[row][c] = W[row][c] * (1 / sqrt(n2[c])), 0 where n2[c] <= 0: the factors
// once per block (C <= kBlock).
__global__ void __launch_bounds__(kBlock) colnormalize_kernel(const double* W,
                                                              const double* n2, double* out,
                                                              int64_t rows, int32_t C) {
  pdl_wait();
  __shared__ double s[kBlock];
  if ((int)threadIdx.x < C) {
    const double n = sqrt(fmax(0.0, n2[threadIdx.x]));
    s[threadIdx.x] = n > 0.0 ? 1.0 / n : 0.0;
  }
  __syncthreads();
  const int64_t total = rows * C;
  for (int64_t e = blockIdx.x * (int64_t)kBlock + threadIdx.x; e < total; e += (int64_t)gridDim.x * kBlock)
    out[e] = W[e] * s[e % C];
}

int grid_elems(int64_t total) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((total + kBlock - 1) / kBlock, max_grid_blocks()));
}

}  // namespace

int mdot_blocks(int64_t rows, int32_t C) {
  const int rpb = kBlock / C;
  return (int)std::max<int64_t>(1, std::min<int64_t>((rows + rpb - 1) / rpb, num_sms() * 4));
}

void launch_mdot(const double* V, int64_t vstride, int32_t Cv, int32_t J, const double* W, int64_t rows, int32_t C,
                 double* part, double* H, cudaStream_t st) {
  if (J <= 0) return;
  const int g = mdot_blocks(rows, C);
  count_launch(2);
  launch_pdl(mdot_partial_kernel, g, kBlock, 0, st, V, vstride, Cv, J, W, rows, C, part);
  launch_pdl(mdot_final_kernel, (J * C + kFinalCols - 1) / kFinalCols, kBlock, 0, st, part, g, J * C, H);
}

void launch_maxpy(const double* V, int64_t vstride, int32_t Cv, int32_t J, const double* H, double sign, double* W,
                  int64_t rows, int32_t C, cudaStream_t st) {
  if (J <= 0) return;
  count_launch();
  launch_pdl(maxpy_kernel, grid_elems(rows * C), kBlock, 0, st, V, vstride, Cv, J, H, sign, W, rows, C);
}

void launch_colnormalize(const double* W, const double* n2, double* out, int64_t rows, int32_t C, cudaStream_t st) {
  count_launch();
  launch_pdl(colnormalize_kernel, grid_elems(rows * C), kBlock, 0, st, W, n2, out, rows, C);
}

void launch_colscale(const double* W, const double* s, double* out, int64_t rows, int32_t C, cudaStream_t st) {
  count_launch();
  launch_pdl(colscale_kernel, grid_elems(rows * C), kBlock, 0, st, W, s, out, rows, C);
}

}  // namespace amgsym
