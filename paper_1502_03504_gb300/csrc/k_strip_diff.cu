// Register strips of the single-field diffusion builtins, and the support
// check and dispatch of the path.
#include "k_strip.cuh"

namespace lope {

int strip_kmax_of(const StepArgs& a) {
  if (a.g.ndim == 3) return kBrickK;
  if (a.s.kind == kUser) return kStripUserK;
  return strip_kmax(a.g.nf, a.s.radius, a.s.star);
}

bool strip_supported(const StepArgs& a) {
  const Geom& g = a.g;
  if (g.ndim == 3) return brick_supported(a);
  if (g.ndim != 2 || a.adjoint || a.stage >= 2 || g.dtype == kF64 || has_external(g)) return false;
  if (a.s.radius < 1 || a.s.radius > 2 || g.n[1] > (int64_t(1) << 30) || g.n[2] > (int64_t(1) << 30))
    return false;
  for (int ax = 1; ax < 3; ++ax)
    if (g.bc[ax][0] == kPeriodic && g.n[ax] < a.s.radius) return false;
  const bool vec = strip_vec(a);
  // BF16 rows that are not whole 8-byte vectors have no asynchronous element
  // copy; steps of several stages and run-time compiled functions are built for
  // aligned rows only.
  if (!vec && (g.dtype == kBF16 || a.s.stages != 1 || a.s.kind == kUser)) return false;
  if (a.s.stages != 1) return a.ksteps == 1 && a.s.kind != kUser;
  if (a.s.kind == kUser && !a.s.star) return false;
  return a.ksteps == strip_kmax_of(a) || a.ksteps == 4 || a.ksteps == 2 || a.ksteps == 1;
}

cudaError_t launch_strip(const StepArgs& a) {
  if (a.g.ndim == 3) return launch_brick(a);
  switch (a.s.kind) {
    case kUser: return jit_launch(a, kPathStrip);
    case kJacobi5: return strip_op(a, OpJacobi5{a.s.prm[0]});
    case kStar9r2: return strip_op(a, OpStar9r2{a.s.prm[0]});
    case kSwe: case kSweFlux: return launch_strip_swe(a);
    case kLinear: return launch_strip_linear(a);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace lope
