// Register bricks (brick_device.cuh): support check, the cut of the grid and
// the launch, for the 7-point diffusion and radius-1 star tables.
#include <algorithm>
#include <cstring>

#include "brick_device.cuh"
#include "strip_kernels.cuh"

namespace lope {

namespace {

constexpr int kRY = 4, kWY = 16;  // rows per thread, half-warps per block

// z chunks: among the counts that keep a chunk at least as long as its
// pipeline's fill, the one that maximises the busy fraction of the last wave
// times the share of planes that are not fill.
template <int K> int brick_chunk(int nz, int tiles, int slots, double* share = nullptr) {
  double best = -1.0;
  int bzc = nz;
  const int most = std::max(1, std::min(nz / (2 * K), 4 * slots / tiles + 1));
  for (int n = 1; n <= most; ++n) {
    const int zc = (nz + n - 1) / n, m = (nz + zc - 1) / zc, b = tiles * m, waves = (b + slots - 1) / slots;
    const double score = double(b) / (double(waves) * slots) * nz / (double(m) * (zc + 2 * K));
    if (score > best + 1e-9) {
      best = score;
      bzc = zc;
    }
  }
  if (share) *share = best;
  return bzc;
}

template <class Op, class T, int K, int MODE = kBrickPlain> struct BrickRunner {
  using G = BrickGeom<T, K, kRY, kWY>;
  // outs: the output of every level (kBrickStates), else out[K-1] alone is used
  template <bool VEC>
  static cudaError_t go(const StepArgs& a, const Op& op, void* const* outs, const void* const* uts, int* blocks_out) {
    auto kern = &brick3d_kernel<Op, T, K, kRY, kWY, MODE, VEC>;
    static PerDevice memo;
    int occ = 0;
    const cudaError_t e = blocks_per_sm(memo, kern, G::THREADS, G::SMEM, &occ);
    if (e != cudaSuccess) return e;
    BrickParams<Op, T> p;
    std::memset(static_cast<void*>(&p), 0, sizeof(p));
    p.op = op;
    p.in = static_cast<const T*>(a.in[0]);
    for (int l = 0; l < K; ++l) {
      p.out[l] = static_cast<T*>(outs ? outs[l] : a.out[0]);
      if (uts) p.ut[l] = static_cast<const T*>(uts[l]);
    }
    p.partials = a.partials;
    p.g.nx = int(a.g.n[2]);
    p.g.ny = int(a.g.n[1]);
    p.g.nz = int(a.g.n[0]);
    for (int ax = 0; ax < 3; ++ax)
      for (int sd = 0; sd < 2; ++sd) {
        p.g.bc[ax][sd] = a.g.bc[ax][sd];
        p.g.bval[ax][sd] = float(a.g.bval[ax][sd]);
      }
    p.tiles_x = brick_count(p.g.nx, G::BX, G::HL * kStripV, p.g.bc[2][0] == kDirichlet, p.g.bc[2][1] == kDirichlet);
    p.tiles_y = brick_count(p.g.ny, G::BY, K, p.g.bc[1][0] == kDirichlet, p.g.bc[1][1] == kDirichlet);
    const int tiles = p.tiles_x * p.tiles_y;
    p.zchunk = brick_chunk<K>(p.g.nz, tiles, device_sms());
    const int blocks = tiles * ((p.g.nz + p.zchunk - 1) / p.zchunk);
    if (blocks_out) *blocks_out = blocks;
    if (MODE == kBrickAdjoint && (!a.partials || blocks > a.partial_count)) return cudaErrorInvalidValue;
    kern<<<blocks, G::THREADS, G::SMEM, a.stream>>>(p);
    count_launches(1);
    return cudaGetLastError();
  }
  static cudaError_t run(const StepArgs& a, const Op& op) {
    if (strip_vec(a)) return go<true>(a, op, nullptr, nullptr, nullptr);
    if constexpr (sizeof(T) == 4) return go<false>(a, op, nullptr, nullptr, nullptr);
    return cudaErrorNotSupported;
  }
};

template <class Op, class T> cudaError_t brick_t(const StepArgs& a, const Op& op) {
  if (a.ksteps == kBrickK) return BrickRunner<Op, T, kBrickK>::run(a, op);
  if (a.ksteps == 2) return BrickRunner<Op, T, 2>::run(a, op);
  return cudaErrorNotSupported;
}
template <class Op> cudaError_t brick_op(const StepArgs& a, const Op& op) {
  return a.g.dtype == kF32 ? brick_t<Op, float>(a, op) : brick_t<Op, __nv_bfloat16>(a, op);
}

template <class T> cudaError_t states_t(const StepArgs& a, void* const* outs) {
  const OpDiff7 op{a.s.prm[0]};
  if (a.ksteps == 4) return BrickRunner<OpDiff7, T, 4, kBrickStates>::template go<true>(a, op, outs, nullptr, nullptr);
  if (a.ksteps == 2) return BrickRunner<OpDiff7, T, 2, kBrickStates>::template go<true>(a, op, outs, nullptr, nullptr);
  return cudaErrorNotSupported;
}
template <class T> cudaError_t adjoint_t(const StepArgs& a, const void* const* uts, int* blocks) {
  const OpBrickAdjoint op{a.s.prm[0]};
  if (a.ksteps == 2) return BrickRunner<OpBrickAdjoint, T, 2, kBrickAdjoint>::template go<true>(a, op, nullptr, uts, blocks);
  return cudaErrorNotSupported;
}

}  // namespace

cudaError_t launch_brick_states(const StepArgs& a, void* const* outs) {
  return a.g.dtype == kF32 ? states_t<float>(a, outs) : states_t<__nv_bfloat16>(a, outs);
}
cudaError_t launch_brick_adjoint(const StepArgs& a, const void* const* uts, int* blocks) {
  return a.g.dtype == kF32 ? adjoint_t<float>(a, uts, blocks) : adjoint_t<__nv_bfloat16>(a, uts, blocks);
}
bool brick_adjoint_supported(const StepArgs& a) {
  StepArgs b = a;
  b.adjoint = false;
  b.ksteps = 2;
  return a.s.kind == kDiff7 && strip_vec(a) && brick_supported(b);
}

bool brick_supported(const StepArgs& a) {
  const Geom& g = a.g;
  if (g.ndim != 3 || g.nf != 1 || a.adjoint || a.stage >= 2 || a.s.stages != 1 || has_external(g)) return false;
  if (a.s.radius != 1 || !a.s.star || (a.s.kind != kDiff7 && a.s.kind != kLinear)) return false;
  if (g.dtype == kF64 || (g.dtype == kBF16 && !strip_vec(a))) return false;
  // the first and last block of a Dirichlet axis lie inside it; offsets within
  // a plane are 32-bit
  if (g.n[2] < 64 || g.n[1] < kRY * kWY || g.n[0] > (int64_t(1) << 30) ||
      g.n[1] * g.n[2] >= (int64_t(1) << 31))
    return false;
  return a.ksteps == kBrickK || a.ksteps == 2;
}

int64_t brick_cells(const StepArgs& a) {
  using G = BrickGeom<float, kBrickK, kRY, kWY>;
  const Geom& g = a.g;
  return int64_t(G::BX) * brick_count(int(g.n[2]), G::BX, G::HL * kStripV, g.bc[2][0] == kDirichlet, g.bc[2][1] == kDirichlet) *
         G::BY * brick_count(int(g.n[1]), G::BY, kBrickK, g.bc[1][0] == kDirichlet, g.bc[1][1] == kDirichlet);
}

double brick_share(const StepArgs& a, int slots) {
  using G = BrickGeom<float, kBrickK, kRY, kWY>;
  const Geom& g = a.g;
  const int tx = brick_count(int(g.n[2]), G::BX, G::HL * kStripV, g.bc[2][0] == kDirichlet, g.bc[2][1] == kDirichlet);
  const int ty = brick_count(int(g.n[1]), G::BY, kBrickK, g.bc[1][0] == kDirichlet, g.bc[1][1] == kDirichlet);
  if (tx == 1 || ty == 1) return 1.0;
  double share = 0.0;
  brick_chunk<kBrickK>(int(g.n[0]), tx * ty, slots, &share);
  return share;
}

cudaError_t launch_brick(const StepArgs& a) {
  if (a.s.kind == kDiff7) return brick_op(a, OpDiff7{a.s.prm[0]});
  OpStarLinear<3, 1> op;
  for (int ax = 0; ax < 3; ++ax)
    for (int d = 0; d < 3; ++d) op.w[ax][d] = a.s.star_w[ax][d];
  return brick_op(a, op);
}

}  // namespace lope
