// Register strips of the 2D weight tables (star and box, radius 1 and 2).
#include "k_strip.cuh"

namespace lope {

namespace {

template <int RR> cudaError_t star(const StepArgs& a) {
  OpStarLinear<2, RR> op;
  for (int ax = 0; ax < 3; ++ax)
    for (int d = 0; d < 2 * RR + 1; ++d) op.w[ax][d] = a.s.star_w[ax][d];
  return strip_op(a, op);
}
template <int RR> cudaError_t box(const StepArgs& a) {
  OpBoxLinear<2, RR> op;
  for (int i = 0; i < (2 * RR + 1) * (2 * RR + 1); ++i) op.w[i] = a.s.box[i];
  return strip_op(a, op);
}

}  // namespace

cudaError_t launch_strip_linear(const StepArgs& a) {
  if (a.s.star) return a.s.radius == 1 ? star<1>(a) : star<2>(a);
  return a.s.radius == 1 ? box<1>(a) : box<2>(a);
}

}  // namespace lope
