// Programmatic dependent launch of the solve's kernels on an ordinary stream.
//
// A V-cycle is a chain of some 30 dependent launches, and below the finest
// level most of them run for a few microseconds: the drain of one grid and the
// launch of the next cost as much as the work.  A kernel launched here may
// start while its predecessor on the stream drains; it calls pdl_wait() before
// it touches anything another kernel writes or reads, which returns when the
// predecessor has completed and its stores are visible, and only then lets its
// own successor start (so at most one grid waits behind the running one, and
// completion stays transitive along the stream).  Every kernel launched by
// launch_pdl calls pdl_wait() first, in every thread.
//
// The read-only data path (__ldg, or a pointer that is both const and
// __restrict__) is for data that nothing writes while the kernel lives, and
// here that life overlaps the predecessor's: it holds for matrices, index lists
// and the coarsest inverse only.  What another kernel of the solve writes
// (vectors, dot results, the CG scalars) comes by ordinary loads or through L2,
// which the wait orders; their pointers carry no __restrict__.
//
// The attribute goes only to a kernel whose predecessor on the stream is known:
// a launch_pdl kernel of the same call, with nothing between the two.  A call
// that is a chain of launches opens a PdlScope on its stream; the first kernel of
// the scope, and the first after a copy, a memset or a kernel launched otherwise
// (pdl_break()), starts in the ordinary way, behind whatever the stream holds,
// and so does the last kernel of a chain, so that what follows the call (a copy, a
// graph, a caller's kernel) is behind an ordinary launch.  How an early start is
// ordered before and after work that is not a kernel is not documented; nothing
// rests on it.
// Outside a scope every launch is an ordinary one: a setup (its damping decides
// every later cycle of the handle), a solve (copies between its steps, its
// iterations in a graph), a batch, and a call of one launch (back-to-back reduced
// products at 256^3 took 38.6 us with the attribute, 37.0 without).
//
// Nor while a stream is captured: between the kernel nodes of a graph the
// programmatic edges cost more than they hide (mixed solves 0-2 %, an FP64
// solve of 87k rows 4 % slower).  Eager V-cycles: 57k rows 131 -> 85 us, 256^3
// 665 -> 612 us; GMRES at 64^3 12.1 -> 11.1 ms.
#pragma once

#include <cuda_runtime.h>

namespace amgsym {

__device__ __forceinline__ void pdl_wait() {
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
}

// The calling thread's open scope.
struct PdlState {
  bool on = false;            // an eager stream's scope is open
  bool after_kernel = false;  // the last operation of the scope was a launch_pdl kernel
  cudaStream_t st = nullptr;
};
extern thread_local PdlState t_pdl;

class PdlScope {
 public:
  explicit PdlScope(cudaStream_t st) : outer_(t_pdl) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const bool eager = cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone;
    t_pdl = PdlState{eager, false, st};
  }
  ~PdlScope() { t_pdl = outer_; }
  PdlScope(const PdlScope&) = delete;
  PdlScope& operator=(const PdlScope&) = delete;

 private:
  PdlState outer_;
};

// After an operation of the scope's stream that is not a launch_pdl kernel.
inline void pdl_break() { t_pdl.after_kernel = false; }

template <typename T>
struct Same {
  using type = T;
};

// The arguments have the kernel's own parameter types: what is passed converts
// to them by the language's implicit conversions, checked by the compiler.
template <typename... P>
inline void launch_pdl(void (*kern)(P...), dim3 grid, int block, size_t smem, cudaStream_t st,
                       typename Same<P>::type... args) {
  const bool in_scope = t_pdl.on && t_pdl.st == st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = in_scope && t_pdl.after_kernel ? 1 : 0;
  (void)cudaLaunchKernelEx(&cfg, kern, args...);  // errors: cudaGetLastError (check_launch)
  if (in_scope) t_pdl.after_kernel = true;
}

}  // namespace amgsym
