// Register strips of the three-field shallow-water builtins.
#include "k_strip.cuh"

namespace lope {

cudaError_t launch_strip_swe(const StepArgs& a) {
  const double* p = a.s.prm;
  if (a.s.kind == kSwe) return strip_op(a, OpSwe{-p[0] * p[2], -p[0] * p[1]});
  return strip_op(a, OpSweFlux::make(p));
}

}  // namespace lope
