// Dispatch of one local function on the register strips over storage type,
// depth and scheme; each k_strip_*.cu instantiates it for some of the builtins.
#pragma once

#include "strip_kernels.cuh"

namespace lope {

namespace {

template <class Op, class T> cudaError_t strip_t(const StepArgs& a, const Op& op) {
  constexpr int KMAX = strip_kmax(Op::NF, Op::R, Op::STAR);
  if (a.s.stages == 2) return StripRunner<Op, T, 2, 2>::run_vec(a, op);
  if (a.s.stages == 3) return StripRunner<Op, T, 3, 3>::run_vec(a, op);
  if (a.s.stages != 1) return cudaErrorNotSupported;
  if constexpr (KMAX > 4) {
    if (a.ksteps == KMAX) return StripRunner<Op, T, KMAX, 1>::run(a, op);
  }
  switch (a.ksteps) {
    case 4: return StripRunner<Op, T, 4, 1>::run(a, op);
    case 2: return StripRunner<Op, T, 2, 1>::run(a, op);
    case 1: return StripRunner<Op, T, 1, 1>::run(a, op);
    default: return cudaErrorNotSupported;
  }
}

template <class Op> cudaError_t strip_op(const StepArgs& a, const Op& op) {
  switch (a.g.dtype) {
    case kF32: return strip_t<Op, float>(a, op);
    case kBF16: return strip_t<Op, __nv_bfloat16>(a, op);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace
}  // namespace lope
