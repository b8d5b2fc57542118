// Deterministic per-column dot products fused into kernel epilogues.
//
// Every participating kernel uses 256-thread blocks in which a thread owns some
// consecutive columns of a row slot: slot t / TPR for thread t where TPR = C / CPT
// threads serve a row alone, the place in TileLayout (spmm_common.cuh) in the
// products.  A block reduces its threads' partials in shared memory in a fixed order,
// writes one partial per column to global memory, and the last block to
// finish (integer ticket) sums the block partials in a fixed order and runs
// the finalisation (CG scalars, convergence test).  No floating-point
// atomics: results are bit-reproducible run to run.
#pragma once

#include "device.h"
#include "fp32_sum.h"

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
        else if (atomicExch(s.status + 1, 1) == 0) {  // breakdown: p^T A p <= 0 or NaN
          s.fault[0] = c;
          s.fault[1] = s.status[2];
          s.fault[2] = sum;
          s.fault[3] = rz;
        }
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
    if (act && !(rel2 > *s.tol2)) {  // converged (or NaN: the breakdown flag was set at p^T A p)
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
// What bounds it: FP64 adds and conversions issue at 2 lanes per clock per SM
// here (16 cycles a warp instruction), so the tail of a fused dot is the number
// of FP64 instructions per SM plus the chains of dependent adds and of L2 round
// trips, not the bytes.  Hence:
//  * FP64 partials: a warp combines its row slots by halving exchanges (lane
//    pairs swap half of their columns: 4 + 2 + 1 + 1 + 1 = 9 adds a lane for 8
//    columns, not 8 x 5 = 40).
//  * FP32 partials go to shared memory as they are; kBlock threads sum up to 16
//    of them each with error-free FP32 additions (fp32_sum.h: nearer to the exact
//    sum than additions in FP64) and convert once, instead of a conversion and an
//    FP64 add for every partial.
//  * The block partials: eight loads in flight per thread; many of them in two
//    levels, so that the last block does not add nslots x C values alone.
// Before, from a block's last product to the end of the kernel (456 blocks, FP32):
// 6.2 us at 8 columns, 12.5 at 24, 10.0 at 32, of which the last block's sum of
// the block partials 3.0, 6.3 and 7.5; a mixed solve runs three of these an
// iteration (128^3 at 32 columns, to 1e-12: 31.8 -> 30.9 ms; 256^3: 100.5 -> 99.9).
__host__ __device__ inline bool dot_shuffles(int S) { return S > 0 && (S & (S - 1)) == 0 && S <= 32; }

// Lines of per-column FP64 partials a block leaves in shared memory: one per
// warp when the S lanes of a row slot divide a warp, else one per row slot.
__host__ __device__ inline int dot_lines(int S, int rows_pb) { return dot_shuffles(S) ? kBlock / 32 : rows_pb; }

// Shared scratch: the lines (FP64), or the FP32 partials column by column (an
// odd pitch spreads the columns of a row slot over the banks); then the sums.
__host__ __device__ inline int dot_pitch(int rows_pb) { return rows_pb | 1; }
__host__ __device__ inline int dot_area(int S, int rows_pb, int C) {
  const int f64 = dot_lines(S, rows_pb) * C, f32 = (C * dot_pitch(rows_pb) + 1) / 2;
  return (f64 > f32 ? f64 : f32) + C;
}
__host__ __device__ inline int dot_smem_doubles(int S, int rows_pb, int C) { return dot_area(S, rows_pb, C) + kBlock; }

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

// out[c] = sum over sl < n of red[sl * C + c], halving n: log2(n) dependent
// adds.  Starts and ends with a barrier.
__device__ __forceinline__ void dot_fold(int n, int C, double* red, double* out) {
  const int c = threadIdx.x % C, sl = threadIdx.x / C;
  while (n > 1) {
    const int h = (n + 1) >> 1;
    __syncthreads();
    if (sl < n - h) red[sl * C + c] += red[(sl + h) * C + c];
    n = h;
  }
  __syncthreads();
  if (sl == 0) out[c] = red[c];
  __syncthreads();
}

// out[c] = sum of `count` lines of src (stride C; GLOBAL: written by other
// blocks, read through L2), for the whole block: thread t sums the lines
// t / C, t / C + slices, ... of column t % C in four chains, eight loads in
// flight; the slices are folded in red (kBlock doubles).
template <bool GLOBAL>
__device__ __forceinline__ void dot_sum_lines(const double* src, int count, int C, double* red, double* out) {
  const int c = threadIdx.x % C, sl = threadIdx.x / C;
  auto ld = [&](int r) { return GLOBAL ? __ldcg(src + (int64_t)r * C + c) : src[r * C + c]; };
  constexpr int U = GLOBAL ? 8 : 4;
  // few lines in shared memory: one thread per column, nothing to fold
  const int slices = !GLOBAL && count <= 8 ? 1 : min((int)blockDim.x / C, count);
  if (sl < slices) {
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    for (int r = sl; r < count; r += U * slices) {
      double v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) v[u] = r + u * slices < count ? ld(r + u * slices) : 0.0;
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (r + u * slices < count) t[u & 3] += v[u];
    }
    red[sl * C + c] = (t[0] + t[1]) + (t[2] + t[3]);
  }
  dot_fold(slices, C, red, out);
}

// The block's sum per column of FP64 partials.
template <int CPT>
__device__ __forceinline__ void dot_block_sum(double (&part)[CPT], int c0, bool has_cols, int rloc, int rows_pb, int S,
                                              int C, double* sm, double* red, double* out) {
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
  __syncthreads();
  dot_sum_lines<false>(sm, dot_lines(S, rows_pb), C, red, out);
}

// The same of FP32 partials (fp32_sum.h).
template <int CPT>
__device__ __forceinline__ void dot_block_sum(float (&part)[CPT], int c0, bool has_cols, int rloc, int rows_pb, int S,
                                              int C, double* sm, double* red, double* out) {
  float* f = reinterpret_cast<float*>(sm);
  const int pitch = dot_pitch(rows_pb);
  if (has_cols) {
#pragma unroll
    for (int q = 0; q < CPT; ++q) f[(c0 + q) * pitch + rloc] = part[q];
  }
  __syncthreads();
  const int nsl = min(kBlock / C, rows_pb);
  const int c = threadIdx.x / nsl, sl = threadIdx.x - c * nsl;
  if (c < C) red[sl * C + c] = fp32_sum(f + c * pitch, sl, nsl, rows_pb);
  dot_fold(nsl, C, red, out);
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

// One of n arrivals at a ticket: whether this block is the last.  The block's
// stores, made visible to thread 0 by the barrier before, are released with its
// arrival (cumulativity) and acquired by the last block.
__device__ __forceinline__ bool dot_arrive(unsigned* ticket, int n) {
  __shared__ unsigned last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = (atomicAdd(ticket, 1u) == (unsigned)n - 1u) ? 1u : 0u;
    __threadfence();
  }
  __syncthreads();
  const bool l = last != 0u;
  __syncthreads();  // before another arrival writes it
  return l;
}

// Two levels: blocks (slots) leave partials[slot]; the last of each chunk of 32
// slots sums them into chunk_partials[chunk]; the last chunk sums those and
// finalises.  Any number of slots, each stage reading at most 32 lines a column
// (up to 1024 slots).
template <int CPT, typename DT>
__device__ __forceinline__ void block_dot2(const DotArgs& d, DT (&part)[CPT], int c0, bool has_cols, int rloc,
                                           int rows_pb, int S, int C, double* sm, int slot, const BDot& bd) {
  double* red = sm + dot_area(S, rows_pb, C);
  dot_block_sum<CPT>(part, c0, has_cols, rloc, rows_pb, S, C, sm, red, bd.partials + (int64_t)slot * C);
  const int chunk = slot >> 5;
  const int nch = (bd.nslots + 31) >> 5;
  const int in_chunk = min(32, bd.nslots - chunk * 32);
  if (!dot_arrive(bd.chunk_tickets + chunk, in_chunk)) return;
  dot_sum_lines<true>(bd.partials + (int64_t)chunk * 32 * C, in_chunk, C, red, bd.chunk_partials + (int64_t)chunk * C);
  if (threadIdx.x == 0) bd.chunk_tickets[chunk] = 0u;
  if (!dot_arrive(bd.ticket, nch)) return;
  double* colsum = sm;  // [C] (the partials' area is free now)
  dot_sum_lines<true>(bd.chunk_partials, nch, C, red, colsum);
  dot_finalize(d, colsum, C);
  if (threadIdx.x == 0) *bd.ticket = 0u;
  __syncthreads();  // the block may go on to reuse the shared scratch
}

// The grid's dot of one problem (slot = block): one level up to 4096 block
// partials (2 us of FP64 adds in the last block), where a second arrival costs
// as much as it saves.
template <int CPT, typename DT>
__device__ __forceinline__ void block_dot(const DotArgs& d, DT (&part)[CPT], int c0, bool has_cols, int rloc,
                                          int rows_pb, int S, int C, double* sm) {
  const DevScalars& sc = d.sc;
  const int slot = blockIdx.x, nslots = gridDim.x;
  if (nslots * C > 4096 && nslots > 32) {
    BDot bd;
    bd.partials = sc.partials;
    bd.chunk_partials = sc.partials + sc.partial_cap;
    bd.ticket = sc.ticket;
    bd.chunk_tickets = sc.ticket + 1;
    bd.nslots = nslots;
    block_dot2<CPT, DT>(d, part, c0, has_cols, rloc, rows_pb, S, C, sm, slot, bd);
    return;
  }
  double* red = sm + dot_area(S, rows_pb, C);
  dot_block_sum<CPT>(part, c0, has_cols, rloc, rows_pb, S, C, sm, red, sc.partials + (int64_t)slot * C);
  if (!dot_arrive(sc.ticket, nslots)) return;
  double* colsum = sm;  // [C] (the partials' area is free now)
  dot_sum_lines<true>(sc.partials, nslots, C, red, colsum);
  dot_finalize(d, colsum, C);
  if (threadIdx.x == 0) *sc.ticket = 0u;
  __syncthreads();
}

}  // namespace amgsym
