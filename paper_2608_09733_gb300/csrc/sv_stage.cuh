// sv_stage.cuh -- a pass program in shared memory, for kernels that run a
// program over one tile or a few: each op's descriptor is then read once, and
// read in place (device memory or the constant bank) its miss is waited for
// before the op.  Copied up front, the misses of all ops overlap.  (k_sweep
// over 16 tiles and more keeps the constant bank: with a copy its 14- to
// 17-qubit passes were 3 to 5 % slower.)
#pragma once

#include <cstddef>

#include "sv_prog_layout.h"

namespace sv {

// Bytes of a staged program (a multiple of 16).
template <typename R>
__host__ __device__ constexpr int staged_bytes(int ncoef) {
  return (int)offsetof(SweepProgram<R>, coef) + (ncoef * (int)sizeof(Cx<R>) + 15) / 16 * 16;
}

#ifdef __CUDACC__
// Copies what the program uses of its header, ops, phases and coefficients to
// `dst` (16-byte aligned, staged_bytes), all threads of the CTA taking part;
// the caller synchronizes before it reads the copy.  GLOBAL: the program is in
// device memory (not a kernel parameter) and read through L2, since the host
// may have written it while the kernel runs.
template <bool GLOBAL, typename R>
__device__ __forceinline__ const SweepProgram<R>& stage_program(const SweepProgram<R>& P, void* dst) {
  const uint4* s = reinterpret_cast<const uint4*>(&P);
  uint4* d = reinterpret_cast<uint4*>(dst);
  const int ops = (int)offsetof(SweepProgram<R>, ops) / 16, ph = (int)offsetof(SweepProgram<R>, ph) / 16,
            coef = (int)offsetof(SweepProgram<R>, coef) / 16;
  static_assert(offsetof(SweepProgram<R>, ops) % 16 == 0 && offsetof(SweepProgram<R>, ph) % 16 == 0 &&
                    offsetof(SweepProgram<R>, coef) % 16 == 0 && sizeof(DevOp) % 16 == 0,
                "16-byte parts");
  auto load = [&](int i) {
    if constexpr (GLOBAL)
      return __ldcg(s + i);
    else
      return s[i];
  };
  int nops, ncoef, nphases;
  if constexpr (GLOBAL) {
    nops = __ldcg(&P.h.nops);
    ncoef = __ldcg(&P.h.ncoef);
    nphases = __ldcg(&P.h.nphases);
  } else {
    nops = P.h.nops;
    ncoef = P.h.ncoef;
    nphases = P.h.nphases;
  }
  const int ops_end = ops + nops * ((int)sizeof(DevOp) / 16);
  const int ph_end = ph + (nphases * (int)sizeof(Phase) + 15) / 16;
  const int coef_end = coef + (ncoef * (int)sizeof(Cx<R>) + 15) / 16;
  for (int i = threadIdx.x; i < ops_end; i += blockDim.x) d[i] = load(i);
  for (int i = ph + threadIdx.x; i < ph_end; i += blockDim.x) d[i] = load(i);
  for (int i = coef + threadIdx.x; i < coef_end; i += blockDim.x) d[i] = load(i);
  return *reinterpret_cast<const SweepProgram<R>*>(dst);
}
#endif

}  // namespace sv
