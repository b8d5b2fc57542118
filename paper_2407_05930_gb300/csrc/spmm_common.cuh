// Device code shared by the single-problem and batched SpMM kernels.
#pragma once

#include <cuda_bf16.h>

#include "device.h"
#include "dot.cuh"

namespace amgsym {

template <typename T>
struct AccOf {
  using type = float;
};
template <>
struct AccOf<double> {
  using type = double;
};

template <typename T>
__device__ __forceinline__ float to_f(T v) {
  return (float)v;
}
template <>
__device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}

template <typename A, typename T>
__device__ __forceinline__ A cvt(T v) {
  return (A)v;
}
template <>
__device__ __forceinline__ float cvt<float, __nv_bfloat16>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}
template <>
__device__ __forceinline__ double cvt<double, __nv_bfloat16>(__nv_bfloat16 v) {
  return (double)__bfloat162float(v);
}

// Vector of N consecutive T, aligned to its size up to 32 bytes (a 32-byte
// vector is one 256-bit access where the hardware has it, else two 16-byte ones).
template <typename T, int N>
struct alignas(sizeof(T) * N <= 32 ? sizeof(T) * N : 32) Vec {
  T v[N];
};

template <typename T, int N>
__device__ __forceinline__ Vec<T, N> ldv(const T* p) {
  return *reinterpret_cast<const Vec<T, N>*>(p);
}
// 32-byte vectors as one 256-bit load (ld.global.v8.f32 / .v4.f64, sm_100 and
// later): one request per warp instruction instead of two 128-bit ones.
template <>
__device__ __forceinline__ Vec<float, 8> ldv<float, 8>(const float* p) {
  Vec<float, 8> r;
  asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3]), "=f"(r.v[4]), "=f"(r.v[5]), "=f"(r.v[6]),
                 "=f"(r.v[7])
               : "l"(p));
  return r;
}
template <>
__device__ __forceinline__ Vec<double, 4> ldv<double, 4>(const double* p) {
  Vec<double, 4> r;
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(r.v[0]), "=d"(r.v[1]), "=d"(r.v[2]), "=d"(r.v[3])
               : "l"(p));
  return r;
}
// The same load through L2 only (ld.global.cg): coherent with what other
// blocks of the same launch wrote before a grid barrier (the persistent
// coarse-cycle kernel), unlike the read-only data path.
template <typename T, int N>
__device__ __forceinline__ Vec<T, N> ldv_cg(const T* p) {
  Vec<T, N> r;
  constexpr int B = (int)sizeof(T) * N;
  if constexpr (B % 16 == 0) {
#pragma unroll
    for (int i = 0; i < B / 16; ++i) reinterpret_cast<uint4*>(&r)[i] = __ldcg(reinterpret_cast<const uint4*>(p) + i);
  } else if constexpr (B % 8 == 0) {
#pragma unroll
    for (int i = 0; i < B / 8; ++i) reinterpret_cast<uint2*>(&r)[i] = __ldcg(reinterpret_cast<const uint2*>(p) + i);
  } else {
    static_assert(B % 4 == 0, "vector of 4-byte multiples");
#pragma unroll
    for (int i = 0; i < B / 4; ++i)
      reinterpret_cast<unsigned*>(&r)[i] = __ldcg(reinterpret_cast<const unsigned*>(p) + i);
  }
  return r;
}
template <typename T, int N, bool COH>
__device__ __forceinline__ Vec<T, N> ldx(const T* p) {
  if constexpr (COH)
    return ldv_cg<T, N>(p);
  else
    return ldv<T, N>(p);
}
template <typename T, int N>
__device__ __forceinline__ void stv(T* p, const Vec<T, N>& v) {
  *reinterpret_cast<Vec<T, N>*>(p) = v;
}

// The compute type: FP64 if either operand is FP64, else FP32.
template <typename MT, typename XT>
struct ComputeOf {
  using type = float;
};
template <typename XT>
struct ComputeOf<double, XT> {
  using type = double;
};
template <typename MT>
struct ComputeOf<MT, double> {
  using type = double;
};
template <>
struct ComputeOf<double, double> {
  using type = double;
};

// The entries of one row in the diagonal-offset form: every value load and
// gather of a batch of diagonals issued before its FMAs (no dependent index
// loads: the columns are row + offset); one batch holds all diagonals with
// 16-byte column vectors and four with 32-byte ones (registers).  The sum
// runs over the diagonals in ascending offset, i.e. column, order -- the
// order of the CSR loop -- and skips columns outside [0, rows); padded
// positions inside hold 0 and add fma(0, x, acc) = acc.
template <typename MT, typename XT, typename CT, int CPT, bool COH>
__device__ __forceinline__ void dia_row(const SpmmArgs& a, int row, int c0, CT (&acc)[CPT]) {
  const MT* __restrict__ dv = static_cast<const MT*>(a.dval);
  const XT* X = static_cast<const XT*>(a.X);
  const int64_t n = a.dstride;
  constexpr int UB = CPT * sizeof(XT) >= 32 ? 4 : kMaxDiag;
#pragma unroll
  for (int d0 = 0; d0 < kMaxDiag; d0 += UB) {
    if (d0 < a.ndiag) {
      CT m[UB];
      Vec<XT, CPT> x[UB];
#pragma unroll
      for (int u = 0; u < UB; ++u) {
        const int d = d0 + u;
        const int j = row + a.doff[d];
        const bool ok = d < a.ndiag && (unsigned)j < (unsigned)a.rows;
        m[u] = ok ? cvt<CT>(dv[(int64_t)a.dsrc[d] * n + row + a.dshift[d]]) : (CT)0;
        if (ok) {
          x[u] = ldx<XT, CPT, COH>(X + (int64_t)j * a.C + c0);
        } else {
#pragma unroll
          for (int q = 0; q < CPT; ++q) x[u].v[q] = (XT)0;
        }
      }
#pragma unroll
      for (int u = 0; u < UB; ++u) {
        if (sizeof(CT) == 8 && d0 + u >= a.ndiag) continue;  // uniform
#pragma unroll
        for (int q = 0; q < CPT; ++q) acc[q] = fma(m[u], (CT)x[u].v[q], acc[q]);
      }
    }
  }
}

// The CSR entries kb + e, kb + e + KL, ... < ke of one row, U per step,
// predicated: all index/value loads first, then all gathers, so a row of up
// to U * KL entries costs one round trip and a 7-point row (U = 4) two, with
// every gather of a step in flight at once.  FP64 sums skip the masked fmas: an
// FP64 instruction takes 16 issue cycles whatever its lanes hold (2 lanes per
// clock per SM), so a 19-entry row at KL = 4 costs 5 fmas per column, not 8.
template <typename MT, typename XT, typename CT, int CPT, int KL, bool COH>
__device__ __forceinline__ void csr_row(const SpmmArgs& a, int kb, int ke, int e, int c0, CT (&acc)[CPT]) {
  const MT* __restrict__ val = static_cast<const MT*>(a.val);
  const XT* X = static_cast<const XT*>(a.X);
  const int32_t* __restrict__ idx = a.idx;
  const int C = a.C;
  constexpr int U = CPT >= 8 ? 2 : 4;
  for (int k = kb + e; k < ke; k += U * KL) {
    int j[U];
    CT m[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool ok = k + u * KL < ke;
      j[u] = ok ? __ldg(idx + k + u * KL) : 0;
      m[u] = ok ? cvt<CT>(val[k + u * KL]) : (CT)0;
    }
    Vec<XT, CPT> x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (k + u * KL < ke) {
        x[u] = ldx<XT, CPT, COH>(X + (int64_t)j[u] * C + c0);
      } else {
#pragma unroll
        for (int q = 0; q < CPT; ++q) x[u].v[q] = (XT)0;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (sizeof(CT) == 8 && k + u * KL >= ke) continue;
#pragma unroll
      for (int q = 0; q < CPT; ++q) acc[q] = fma(m[u], (CT)x[u].v[q], acc[q]);
    }
  }
}

// The entries kb + e, kb + e + KL, ... < ke of one row of a halo-staged
// matrix: the same batches, masking and fma sequence as csr_row (so the same
// sums), with 16-bit column indices into the tile's halo and the gathered
// rows read from shared memory (xs: [halo][C], staged by the caller).
template <typename MT, typename XT, typename CT, int CPT, int KL>
__device__ __forceinline__ void halo_row(const SpmmArgs& a, const XT* xs, int kb, int ke, int e, int c0,
                                         CT (&acc)[CPT]) {
  const MT* __restrict__ val = static_cast<const MT*>(a.val);
  const uint16_t* __restrict__ li = a.lidx;
  const int C = a.C;
  // 8 entries per lane per batch (one global round trip for the index and
  // value loads of rows up to 8 * KL entries); each gathered row comes from
  // shared memory right before its fmas.  The fma sequence of every lane is
  // that of csr_row (entries in order, a masked entry adds fma(0, 0, acc)).
  constexpr int U = 8;
  for (int k = kb + e; k < ke; k += U * KL) {
    int j[U];
    CT m[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool ok = k + u * KL < ke;
      j[u] = ok ? (int)__ldg(li + k + u * KL) : 0;
      m[u] = ok ? cvt<CT>(val[k + u * KL]) : (CT)0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      Vec<XT, CPT> x;
      if (k + u * KL < ke) {
        x = *reinterpret_cast<const Vec<XT, CPT>*>(xs + j[u] * C + c0);
      } else {
#pragma unroll
        for (int q = 0; q < CPT; ++q) x.v[q] = (XT)0;
      }
#pragma unroll
      for (int q = 0; q < CPT; ++q) acc[q] = fma(m[u], (CT)x.v[q], acc[q]);
    }
  }
}

// The interface couplings of flagged row number f (A_out,i of eq.
// "hL_splitting"; one value per block column).
template <typename XT, typename CT, int CPT, bool COH>
__device__ __forceinline__ void iface_row(const SpmmArgs& a, int f, int c0, CT (&acc)[CPT]) {
  const CT* __restrict__ iv = static_cast<const CT*>(a.ival);
  const XT* X = static_cast<const XT*>(a.X);
  for (int ee = __ldg(a.iptr + f); ee < __ldg(a.iptr + f + 1); ++ee) {
    const int j = __ldg(a.icol + ee);
    const Vec<XT, CPT> xv = ldx<XT, CPT, COH>(X + (int64_t)j * a.C + c0);
#pragma unroll
    for (int q = 0; q < CPT; ++q) {
      const int blk = (c0 + q) % a.nb;
      acc[q] = fma(iv[(int64_t)ee * a.nb + blk], (CT)xv.v[q], acc[q]);
    }
  }
}

// Number of flagged rows before `row` (row <= rows).
__device__ __forceinline__ int flag_index(const SpmmArgs& a, int row) {
  if (row >= a.rows) return a.nflag;
  const uint32_t wd = __ldg(a.imask + (row >> 5));
  return __ldg(a.iprefix + (row >> 5)) + __popc(wd & ((1u << (row & 31)) - 1u));
}

// Epilogue of CPT columns of one row: Y = alpha acc + beta Z, the optional dot.
template <typename XT, typename OT, typename CT, typename DT, int CPT, bool HAS_DOT, bool COH>
__device__ __forceinline__ void row_epilogue(const SpmmArgs& a, int row, int c0, CT (&acc)[CPT],
                                             const Vec<XT, CPT>& zpre, bool use_zpre, const Vec<XT, CPT>& wpre,
                                             bool use_wpre, DT (&dpart)[CPT]) {
  const int C = a.C;
  CT alpha, beta;
  if constexpr (sizeof(CT) == 8) {
    alpha = a.alpha;
    beta = a.beta;
  } else {
    alpha = a.alpha_f;
    beta = a.beta_f;
  }
  // Y may alias Z (in-place update z += ...); each row reads Z before writing Y.
  OT* Y = static_cast<OT*>(a.Y);
  Vec<OT, CPT> out;
  if (a.epi >= EPI_RESIDUAL) {
    // the epilogue operand as loaded early by the caller (use_zpre), else now;
    // passed by value so that it stays in registers
    const Vec<XT, CPT> zv = use_zpre ? zpre : ldx<XT, CPT, COH>(static_cast<const XT*>(a.Z) + (int64_t)row * C + c0);
    // the factors +-1 of residuals and updates take no multiply (the same
    // rounding: z - acc = fma(-1, acc, 1 * z))
    if (a.epi == EPI_RESIDUAL) {
#pragma unroll
      for (int q = 0; q < CPT; ++q) acc[q] = (CT)zv.v[q] - acc[q];
    } else if (a.epi == EPI_UPDATE) {
#pragma unroll
      for (int q = 0; q < CPT; ++q) acc[q] = fma(alpha, acc[q], (CT)zv.v[q]);
    } else {
#pragma unroll
      for (int q = 0; q < CPT; ++q) acc[q] = fma(alpha, acc[q], beta * (CT)zv.v[q]);
    }
  } else if (a.epi == EPI_SCALE) {
#pragma unroll
    for (int q = 0; q < CPT; ++q) acc[q] = alpha * acc[q];
  }
#pragma unroll
  for (int q = 0; q < CPT; ++q) out.v[q] = (OT)acc[q];
  if (a.jmode == 1) {
    // presmoothing of the next level from zero: Y2 = jd o Y, the arithmetic
    // of the stand-alone diagonal step (one product of the stored values)
    const XT d = static_cast<const XT*>(a.jd)[row];
    Vec<OT, CPT> o2;
#pragma unroll
    for (int q = 0; q < CPT; ++q) o2.v[q] = (OT)(d * (XT)out.v[q]);
    stv<OT, CPT>(static_cast<OT*>(a.Y2) + (int64_t)row * C + c0, o2);
  } else if (a.jmode == 2) {
    // postsmoothing: X + jd o r with r the stored residual value
    const XT d = static_cast<const XT*>(a.jd)[row];
    const Vec<XT, CPT> xr = ldx<XT, CPT, COH>(static_cast<const XT*>(a.X) + (int64_t)row * C + c0);
#pragma unroll
    for (int q = 0; q < CPT; ++q) out.v[q] = (OT)fma(d, (XT)out.v[q], xr.v[q]);
  }
  stv<OT, CPT>(Y + (int64_t)row * C + c0, out);
  if (HAS_DOT) {
    if (a.dot.mode == DOT_WY) {
      // the dot partner as loaded early by the caller (use_wpre), else now
      const Vec<XT, CPT> wv =
          use_wpre ? wpre : ldx<XT, CPT, COH>(static_cast<const XT*>(a.dot.W) + (int64_t)row * C + c0);
#pragma unroll
      for (int q = 0; q < CPT; ++q) dpart[q] = fma((DT)wv.v[q], (DT)acc[q], dpart[q]);
    } else {
#pragma unroll
      for (int q = 0; q < CPT; ++q) dpart[q] = fma((DT)acc[q], (DT)acc[q], dpart[q]);
    }
  }
}

// Resident blocks per SM asked of the compiler.  FP64 with two vectors of
// columns keeps 3 (80 registers: at 8 blocks the CSR kernels spilled 48 to 132
// bytes a thread); its bound is FP64 issue, which a few warps saturate.  The plain
// reduced product keeps 4 (256^3, 16 columns: 573 us, 586 with 3; 2000 x 1600 the
// same: 221 against 230).
template <typename XT, int CPT, bool HAS_DOT, bool HAS_IFACE, bool DIA>
constexpr int spmm_min_blocks() {
  return (DIA && HAS_DOT)                  ? 3
         : DIA && HAS_IFACE                ? 4
         : sizeof(XT) == 8 && CPT >= 4     ? 3
         : (DIA || CPT >= 8)               ? 4
         : sizeof(XT) == 8 && CPT >= 2     ? 4
         : (HAS_DOT || HAS_IFACE)          ? 6
                                           : 8;
}

// The thread's place in the tile layout of one SpMM.  A row is served by
// S = TPC * KL threads: TPC column threads (each owning CPT consecutive
// columns, TPC = C / CPT) times KL entry lanes (lane e takes the row's entries
// e, e + KL, ...).  When S divides a warp the row slots fill the block; else,
// with KL > 1, each warp holds 32 / S slots and idles the rest of its lanes
// (the lanes of a slot exchange by shuffles).
//
// The KL partial sums of a column combine by halving exchanges: the entry
// lanes e and e ^ (KL / 2) swap half of their columns and add, then e and
// e ^ (KL / 4), so a lane ends with E = max(1, CPT / KL) columns from ec0 and
// runs the epilogue of those (`own`: no lower lane holds them too).  Against a full
// exchange with the epilogue in lane 0 that is CPT - 1 instead of
// CPT log2(KL) shuffles and adds, and an epilogue of E instead of CPT columns.
// Each column's sum is the same tree.  Measured on whole solves to 1e-12 with
// the skipped FP64 fmas: FP64 192^3 (C = 8, two solves) 302 -> 270 ms, FP64
// ragged 87k rows at C = 12 (three column threads a row: one entry lane before)
// 24.7 -> 18.4 ms, mixed 128^3 at C = 32 34.5 -> 32.0 ms.
struct TileLayout {
  int TPC, S, rows_pb, g, e, c0, ec0;
  bool slot_ok, own;
};

template <int CPT, int KL>
__host__ __device__ constexpr int tile_cols() {  // columns of a thread in the epilogue
  return CPT / KL > 0 ? CPT / KL : 1;
}

template <int CPT, int KL>
__device__ __forceinline__ TileLayout tile_layout(int C) {
  TileLayout t;
  t.TPC = C / CPT;
  t.S = t.TPC * KL;
  t.rows_pb = tile_rows_pb(t.TPC, KL);
  int w;
  if (KL > 1 && 32 % t.S) {
    const int lane = threadIdx.x & 31, rpw = 32 / t.S, sl = lane / t.S;
    t.g = (threadIdx.x >> 5) * rpw + sl;
    t.slot_ok = sl < rpw;
    w = lane - sl * t.S;
  } else {
    t.g = threadIdx.x / t.S;
    t.slot_ok = t.g < t.rows_pb;
    w = threadIdx.x - t.g * t.S;
  }
  t.e = KL > 1 ? w / t.TPC : 0;
  t.c0 = (w - t.e * t.TPC) * CPT;
  t.ec0 = t.c0;
  t.own = t.slot_ok;
#pragma unroll
  for (int off = KL / 2, h = CPT / 2; off >= 1; off >>= 1, h >>= 1) {
    if (t.e & off) {
      if (h >= 1)
        t.ec0 += h;
      else
        t.own = false;
    }
  }
  return t;
}

// Combines the entry lanes' sums; the thread's columns are left in acc[0 .. E).
template <int CPT, int KL, typename CT>
__device__ __forceinline__ void combine_lanes(const TileLayout& t, CT (&acc)[CPT]) {
#pragma unroll
  for (int off = KL / 2, h = CPT / 2; off >= 1; off >>= 1, h >>= 1) {
    const bool up = (t.e & off) != 0;
    const int src = (threadIdx.x & 31) + (up ? -off : off) * t.TPC;  // (outside a slot: any lane)
    if (h >= 1) {
#pragma unroll
      for (int q = 0; q < CPT / 2; ++q) {
        if (q < h) {
          const CT send = up ? acc[q] : acc[q + h];
          const CT keep = up ? acc[q + h] : acc[q];
          acc[q] = keep + __shfl_sync(0xffffffffu, send, src);
        }
      }
    } else {
      acc[0] += __shfl_sync(0xffffffffu, acc[0], src);
    }
  }
}

// Rows [first_slot * rows_pb + k * slot_step * rows_pb, ...) below row_end
// of one SpMM, for the whole block; this thread's dot partial (its epilogue
// columns) is added to dpart.  KL > 1 keeps several gathers of one row in
// flight (the ptr -> idx -> X latency chain) and spreads the long rows of the
// coarse levels over many lanes.  DIA: the matrix is in the diagonal-offset
// form (one lane per row, no row pointers).  COH: vector operands are loaded
// through L2 only (written earlier in the same launch).
//
// Interface rows (HAS_IFACE) take a second pass: the main pass computes
// every row but stores none of the flagged ones, so no row waits on the
// flag -> prefix -> pointer -> coupling chain; then the flagged rows (about
// 2 % of them at 256^3) are recomputed with their couplings, from the
// compact list of flagged rows.  whole: the block's share of the whole
// matrix, and of its flagged rows the slots f_slot, f_slot + f_step, ... (none
// with f_step = 0); otherwise the block owns rows [first_slot * rows_pb,
// row_end) alone and takes their flagged rows.
// A flagged row's sum is the same in both designs: its entries, then its
// couplings (entry lane 0), then the lane combination.
template <typename MT, typename XT, typename OT, int CPT, int KL, bool HAS_DOT, bool HAS_IFACE, bool DIA = false,
          bool COH = false>
__device__ __forceinline__ void spmm_tile(const SpmmArgs& a, int first_slot, int slot_step, int row_end,
                                          typename AccOf<XT>::type (&dpart)[tile_cols<CPT, KL>()], bool whole = true,
                                          int f_slot = 0, int f_step = 0) {
  static_assert(!DIA || KL == 1, "the diagonal-offset form runs one entry lane per row");
  using CT = typename ComputeOf<MT, XT>::type;
  using DT = typename AccOf<XT>::type;  // per-thread dot partial type
  constexpr int E = tile_cols<CPT, KL>();
  // Early epilogue-operand loads, issued with the row's matrix and X loads so
  // that the epilogue adds no dependent round trip: Z (beta != 0) in the CSR
  // variants launched at 6 blocks per SM, Z and the dot partner W in the
  // diagonal-form dot variants (3 blocks per SM, registers to spare).
  constexpr bool ZPF = (HAS_DOT || HAS_IFACE) && !DIA;
  constexpr bool DPF = HAS_DOT && DIA;
  constexpr bool PTR_PF = ZPF && !DIA;
  const int C = a.C;
  const TileLayout t = tile_layout<CPT, KL>(C);
  const int rows_pb = t.rows_pb, g = t.g, e = t.e, c0 = t.c0, ec0 = t.ec0;
  const bool slot_ok = t.slot_ok;
  const XT* Z = static_cast<const XT*>(a.Z);
  const int32_t* __restrict__ ptr = a.ptr;
  auto epilogue = [&](int row, CT (&acc)[CPT], const Vec<XT, E>& zpre, bool use_z, const Vec<XT, E>& wpre, bool use_w) {
    CT out[E];
#pragma unroll
    for (int q = 0; q < E; ++q) out[q] = acc[q];
    row_epilogue<XT, OT, CT, DT, E, HAS_DOT, COH>(a, row, ec0, out, zpre, use_z, wpre, use_w, dpart);
  };

  // The trip count is block-uniform (the shuffles need every lane of the warp).
  // In the variants with registers to spare (ZPF), the row pointers of a
  // thread's next row are loaded one iteration ahead, which takes one
  // dependent load off each row's chain.
  const int step_rows = slot_step * rows_pb;
  int kb_next = 0, ke_next = 0;
  if (PTR_PF) {
    const int row0 = first_slot * rows_pb + g;
    if (slot_ok && row0 < row_end) {
      kb_next = __ldg(ptr + row0);
      ke_next = __ldg(ptr + row0 + 1);
    }
  }
  for (int base = first_slot * rows_pb; base < row_end; base += step_rows) {
    const int row = base + g;
    const bool live = slot_ok && row < row_end;
    const bool own = t.own && live;  // this thread runs an epilogue
    CT acc[CPT];
#pragma unroll
    for (int q = 0; q < CPT; ++q) acc[q] = (CT)0;
    Vec<XT, E> zpre, wpre;
    int kb = kb_next, ke = ke_next;
    if (PTR_PF) {
      if (slot_ok && row + step_rows < row_end) {
        kb_next = __ldg(ptr + row + step_rows);
        ke_next = __ldg(ptr + row + step_rows + 1);
      }
    } else if (!DIA && live) {
      kb = __ldg(ptr + row);
      ke = __ldg(ptr + row + 1);
    }
    bool flagged = false;
    if (live) {
      // interface flag word and epilogue operand loaded with the row pointers,
      // off the critical path of the gathers
      const uint32_t iface_word = (HAS_IFACE && own) ? __ldg(a.imask + (row >> 5)) : 0u;
      if ((ZPF || DPF) && own && a.epi >= EPI_RESIDUAL) zpre = ldx<XT, E, COH>(Z + (int64_t)row * C + ec0);
      if (DPF && own && a.dot.mode == DOT_WY)
        wpre = ldx<XT, E, COH>(static_cast<const XT*>(a.dot.W) + (int64_t)row * C + ec0);
      if (DIA)
        dia_row<MT, XT, CT, CPT, COH>(a, row, c0, acc);
      else
        csr_row<MT, XT, CT, CPT, KL, COH>(a, kb, ke, e, c0, acc);
      flagged = HAS_IFACE && (iface_word >> (row & 31)) & 1u;
    }
    combine_lanes<CPT, KL, CT>(t, acc);
    if (own && !flagged)
      epilogue(row, acc, zpre, (ZPF || DPF) && a.epi >= EPI_RESIDUAL, wpre, DPF && a.dot.mode == DOT_WY);
  }
  if (HAS_IFACE && (!whole || f_step > 0)) {
    // the flagged rows, with their couplings
    const int f_begin = whole ? 0 : flag_index(a, first_slot * rows_pb);
    const int f_end = whole ? a.nflag : flag_index(a, row_end);
    const int fs0 = whole ? f_slot : 0, fstep = whole ? f_step : 1;
    for (int fb = f_begin + fs0 * rows_pb; fb < f_end; fb += fstep * rows_pb) {
      const int f = fb + g;
      const bool live = slot_ok && f < f_end;
      const int row = live ? __ldg(a.irows + f) : 0;
      CT acc[CPT];
#pragma unroll
      for (int q = 0; q < CPT; ++q) acc[q] = (CT)0;
      if (live) {
        if (DIA) {
          dia_row<MT, XT, CT, CPT, COH>(a, row, c0, acc);
        } else {
          csr_row<MT, XT, CT, CPT, KL, COH>(a, __ldg(ptr + row), __ldg(ptr + row + 1), e, c0, acc);
        }
        if (e == 0) iface_row<XT, CT, CPT, COH>(a, f, c0, acc);
      }
      combine_lanes<CPT, KL, CT>(t, acc);
      if (t.own && live) epilogue(row, acc, Vec<XT, E>{}, false, Vec<XT, E>{}, false);
    }
  }
}

}  // namespace amgsym
