// Deterministic per-column dot products fused into kernel epilogues.
//
// Every participating kernel uses 256-thread blocks in which thread t owns
// the CPT consecutive columns c0 = (t % TPR) * CPT of row slot t / TPR.  A
// block reduces its threads' partials in shared memory in a fixed order,
// writes one partial per column to global memory, and the last block to
// finish (integer ticket) sums the block partials in a fixed order and runs
// the finalisation (CG scalars, convergence test).  No floating-point
// atomics: results are bit-reproducible run to run.
#pragma once

#include "device.h"

namespace amgsym {

constexpr int kBlock = 256;

__device__ __forceinline__ void dot_finalize_column(const DotArgs& d, int c, double sum) {
  DevScalars s = d.sc;
  switch (d.final) {
    case FIN_STORE_RZ:
      s.rz[c] = sum;
      break;
    case FIN_ALPHA: {
      const double rz = s.rz[c];
      double a = 0.0;
      if (s.active[c] && rz != 0.0) {
        if (sum > 0.0 && isfinite(sum)) a = rz / sum;
        else s.status[1] = 1;  // breakdown: p^T A p <= 0 or NaN
      }
      s.alpha[c] = a;
      break;
    }
    case FIN_BETA: {
      const double rz = s.rz[c];
      s.beta[c] = (s.active[c] && rz != 0.0) ? sum / rz : 0.0;
      s.rz[c] = sum;
      break;
    }
    case FIN_CONV:
      s.rr[c] = sum;
      break;
    default:
      break;
  }
}

// Per-RHS stage of FIN_CONV / FIN_STORE_BN; colsum in shared memory [C].
__device__ __forceinline__ void dot_finalize_rhs(const DotArgs& d, const double* colsum) {
  DevScalars s = d.sc;
  const int nrhs = d.cp.nrhs, nb = d.cp.nb;
  if (d.final == FIN_STORE_BN) {
    for (int r = threadIdx.x; r < nrhs; r += blockDim.x) {
      double t = 0.0;
      for (int i = 0; i < nb; ++i) t += colsum[r * nb + i];
      s.bnorm2[r] = t;
    }
    return;
  }
  if (d.final != FIN_CONV) return;
  __shared__ int n_active;
  if (threadIdx.x == 0) n_active = 0;
  __syncthreads();
  for (int r = threadIdx.x; r < nrhs; r += blockDim.x) {
    double t = 0.0;
    for (int i = 0; i < nb; ++i) t += colsum[r * nb + i];
    const double bn = s.bnorm2[r];
    const double rel2 = bn > 0.0 ? t / bn : 0.0;
    s.relres[r] = sqrt(rel2);
    bool act = s.active[r * nb] != 0;
    if (act && !(rel2 > *s.tol2)) {  // converged (NaN keeps it active)
      act = false;
      for (int i = 0; i < nb; ++i) s.active[r * nb + i] = 0;
    }
    if (act) atomicAdd(&n_active, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    s.status[0] = n_active;
    if (d.cp.count_iter) s.status[2] += 1;
  }
}

// Block + grid reduction.  part[q] is this thread's partial for column
// c0 + q (zero when !has_cols).  Every sum runs in a fixed assignment of
// threads to terms, so the order of additions, and the result, never varies
// from run to run.  Shared scratch (dynamic): dot_smem_doubles(...).
//
// What bounds it: FP64 adds issue at 2 lanes per clock per SM here (16 cycles
// a warp instruction) and one dependent add takes longer than a shared load,
// so the tail of a fused dot is the number of FP64 add instructions per warp
// plus the chains of dependent adds, not the bytes.  Hence: a warp combines
// its row slots by halving exchanges (lane pairs swap half of their columns,
// so 8 columns over 32 lanes take 4 + 2 + 1 + 1 + 1 = 9 adds a lane, not
// 8 x 5 = 40), and every later stage sums a few interleaved chains.
// Measured on whole solves to 1e-12: FP64 2D 64x64 (C = 2, three dots an
// iteration) 4.05 -> 2.96 ms, mixed 256^3 (C = 8) 107.1 -> 103.9 ms, against
// full butterflies of every column and one thread per column summing up to 128
// slices.
__host__ __device__ inline bool dot_shuffles(int S) { return S > 0 && (S & (S - 1)) == 0 && S <= 32; }

// Lines of per-column partials a block leaves in shared memory: one per warp
// when the S lanes of a row slot divide a warp, else one per row slot.
__host__ __device__ inline int dot_lines(int S, int rows_pb) { return dot_shuffles(S) ? kBlock / 32 : rows_pb; }

__host__ __device__ inline int dot_smem_doubles(int S, int rows_pb, int C) {
  return dot_lines(S, rows_pb) * C + kBlock + C;
}

// Steps K.. of the halving exchange over the lanes lane ^ (S << K): v[0 .. NV)
// holds columns sub .. sub + NV - 1 of the thread's CPT.  `dup`: this lane's
// last value is also held by a lower lane.
template <int NV, int CPT>
__device__ __forceinline__ void dot_exchange(double (&v)[CPT], int off, int lane, int& sub, bool& dup) {
  if constexpr (NV > 1) {
    if (off >= 32) return;
    constexpr int H = NV / 2;
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int q = 0; q < H; ++q) {
      const double send = up ? v[q] : v[q + H];
      const double keep = up ? v[q + H] : v[q];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
    if (up) sub += H;
    dot_exchange<H, CPT>(v, off << 1, lane, sub, dup);
  } else {
    for (; off < 32; off <<= 1) {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
      if (lane & off) dup = true;
    }
  }
}

// The block's threads' partials as lines of C columns in sm (unsynchronised).
template <int CPT>
__device__ __forceinline__ void dot_block_lines(double (&part)[CPT], int c0, bool has_cols, int rloc, int S, int C,
                                                double* sm) {
  if (dot_shuffles(S)) {
    const int lane = threadIdx.x & 31;
    int sub = 0;
    bool dup = false;
    dot_exchange<CPT, CPT>(part, S, lane, sub, dup);
    // log2(32 / S) halvings leave max(1, CPT S / 32) columns per lane
    const int left = CPT * S > 32 ? CPT * S / 32 : 1;
    if (has_cols && !dup) {
      double* line = sm + (threadIdx.x >> 5) * C + c0 + sub;
#pragma unroll
      for (int q = 0; q < CPT; ++q)
        if (q < left) line[q] = part[q];
    }
  } else if (has_cols) {
#pragma unroll
    for (int q = 0; q < CPT; ++q) sm[rloc * C + c0 + q] = part[q];
  }
}

// out[c] = sum of `count` lines of src (stride C; GLOBAL: written by other
// blocks, read through L2), for the whole block: thread t sums the lines
// t / C, t / C + slices, ... of column t % C in four chains, then the slices
// are added in shared memory (red: kBlock doubles) by four chains again.
// Synchronises before out may be read.
template <bool GLOBAL>
__device__ __forceinline__ void dot_sum_lines(const double* src, int count, int C, double* red, double* out) {
  const int c = threadIdx.x % C, sl = threadIdx.x / C;
  auto ld = [&](int r) { return GLOBAL ? __ldcg(src + (int64_t)r * C + c) : src[r * C + c]; };
  // few lines: one thread per column, no second stage
  const int slices = count <= 8 ? 1 : min((int)blockDim.x / C, count);
  if (sl < slices) {
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    int r = sl;
    for (; r + 3 * slices < count; r += 4 * slices) {
#pragma unroll
      for (int u = 0; u < 4; ++u) t[u] += ld(r + u * slices);
    }
#pragma unroll
    for (int u = 0; u < 3; ++u)
      if (r + u * slices < count) t[u] += ld(r + u * slices);
    const double v = (t[0] + t[1]) + (t[2] + t[3]);
    if (slices == 1)
      out[c] = v;
    else
      red[sl * C + c] = v;
  }
  // halve the slices until one is left: log2(slices) dependent adds
  for (int n = slices; n > 1;) {
    const int h = (n + 1) >> 1;
    __syncthreads();
    if (sl < n - h) red[sl * C + c] += red[(sl + h) * C + c];
    n = h;
  }
  if (slices > 1) {
    if (sl == 0) out[c] = red[c];
  }
  __syncthreads();
}

// The CG scalars of every column, then of every right-hand side.
__device__ __forceinline__ void dot_finalize(const DotArgs& d, const double* colsum, int C) {
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    double t = colsum[c];
    if (d.coupled) {  // one CG per RHS: the sum over its blocks, in block order
      const int nb = d.cp.nb, c0 = (c / nb) * nb;
      t = 0.0;
      for (int i = 0; i < nb; ++i) t += colsum[c0 + i];
    }
    dot_finalize_column(d, c, t);
  }
  if (d.final == FIN_CONV || d.final == FIN_STORE_BN) {
    __syncthreads();
    dot_finalize_rhs(d, colsum);
  }
}

template <int CPT>
__device__ __forceinline__ void block_dot(const DotArgs& d, double (&part)[CPT], int c0, bool has_cols,
                                          int rloc, int rows_pb, int S, int C, double* sm, int slot, int nslots,
                                          double* partials, unsigned* ticket) {
  const int lines = dot_lines(S, rows_pb);
  double* red = sm + lines * C;
  dot_block_lines<CPT>(part, c0, has_cols, rloc, S, C, sm);
  __syncthreads();
  dot_sum_lines<false>(sm, lines, C, red, partials + (int64_t)slot * C);
  __shared__ unsigned is_last;
  if (threadIdx.x == 0) {
    // the block's stores, made visible to this thread by the barrier, are
    // released with its arrival (cumulativity), and acquired by the last block
    __threadfence();
    is_last = (atomicAdd(ticket, 1u) == (unsigned)nslots - 1u) ? 1u : 0u;
    __threadfence();
  }
  __syncthreads();
  if (!is_last) return;
  double* colsum = sm;  // [C] (the line area is free now)
  dot_sum_lines<true>(partials, nslots, C, red, colsum);
  dot_finalize(d, colsum, C);
  if (threadIdx.x == 0) *ticket = 0u;
  __syncthreads();  // the block may go on to reuse the shared scratch
}

// Two-level variant for the batched kernels (see BDot): any number of items
// per problem, each reduction stage reading at most 32 lines per column.
template <int CPT>
__device__ __forceinline__ void block_dot2(const DotArgs& d, double (&part)[CPT], int c0, bool has_cols, int rloc,
                                           int rows_pb, int S, int C, double* sm, int slot, const BDot& bd) {
  const int lines = dot_lines(S, rows_pb);
  double* red = sm + lines * C;
  dot_block_lines<CPT>(part, c0, has_cols, rloc, S, C, sm);
  __syncthreads();
  dot_sum_lines<false>(sm, lines, C, red, bd.partials + (int64_t)slot * C);
  __shared__ unsigned last_chunk, last_all;
  const int chunk = slot >> 5;
  const int nch = (bd.nslots + 31) >> 5;
  const int in_chunk = min(32, bd.nslots - chunk * 32);
  if (threadIdx.x == 0) {
    __threadfence();
    last_chunk = (atomicAdd(bd.chunk_tickets + chunk, 1u) == (unsigned)in_chunk - 1u) ? 1u : 0u;
    __threadfence();
  }
  __syncthreads();
  if (!last_chunk) return;
  dot_sum_lines<true>(bd.partials + (int64_t)chunk * 32 * C, in_chunk, C, red, bd.chunk_partials + (int64_t)chunk * C);
  if (threadIdx.x == 0) {
    bd.chunk_tickets[chunk] = 0u;
    __threadfence();
    last_all = (atomicAdd(bd.ticket, 1u) == (unsigned)nch - 1u) ? 1u : 0u;
    __threadfence();
  }
  __syncthreads();
  if (!last_all) return;
  double* colsum = sm;
  dot_sum_lines<true>(bd.chunk_partials, nch, C, red, colsum);
  dot_finalize(d, colsum, C);
  if (threadIdx.x == 0) *bd.ticket = 0u;
  __syncthreads();
}

}  // namespace amgsym
