// Host-side runner of the register strips (strip_device.cuh): depths and block
// shape per function shape, the cut of the grid into strips and chunks, and
// the launch.  Shared by k_strip_*.cu (builtins) and jit.cu (run-time compiled
// local functions).
#pragma once

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "per_device.h"
#include "strip_device.cuh"

namespace lope {

namespace {

// Depth of a pass (the most sweeps one launch fuses): while the registers of a
// lane's queues last, deeper is faster.  One field, radius 1: 8 (jacobi5 FP32
// 8192^2, per sweep: 25 us at depth 4, 18.5 at 6, 17.2 at 8); three-field star
// functions: 6 (linear shallow water FP32 4096^2: 19.0 us at 4, 12.9 at 6);
// radius 2 and box functions: 4 (star9r2 FP32 8192^2: 33.9 us at 4, 41 at
// 6, where it spills; nonlinear shallow water 30.8 and 41).  Radius-2 box tables and
// run-time compiled radius-2 functions of three fields spill at 4 already and run at 2
// by default (api.cu, strip_depth).  What is left of the sweep count runs at depths 4, 2 and 1.
constexpr int strip_kmax(int nf, int radius, bool star) {
  if (radius > 1 || !star) return 4;
  return nf == 1 ? 8 : nf == 3 ? 6 : 4;
}

// Block shape.  One field: blocks of 4 warps, 16 warps of 128 registers per SM;
// several: as many as their registers allow (three rows of every field and
// level stay live; held to 168 registers the nonlinear shallow water spills:
// 44 against 31 us per sweep at 4096^2 FP32).
template <class T, int R, int NF, int K, int STG> struct StripCfg {
  static constexpr int NWB = 4;
  static constexpr int D = STG >= 2 ? 16 : 8;
  static constexpr int MINB = NF == 1 ? 4 : 2;
  static constexpr size_t SMEM = size_t(NWB) * NF * D * StripGeom<T, R, K>::ROWB;
  // Which marches compute on packed pairs (PM of Strip).  A pair takes half the
  // issue slots and twice the FMA pipe's time, and costs moves for the taps along
  // x: BF16 gains everywhere, having moves for its conversions anyway (4096^2,
  // 24 sweeps: linear shallow water 319 -> 290 us, nonlinear 804 -> 777, with
  // Dirichlet sides 1306 -> 998), FP32 only with masks (nonlinear shallow water
  // with Dirichlet sides 1171 -> 1073 us, star9r2 298 -> 278; without masks
  // star9r2 8192^2 x50 1.70 -> 1.97 ms).  Element copies at depth 8 spill
  // on scalars already (with masks a 72-byte frame) and stay on them.
  static constexpr int pm(bool vec, bool dirichlet) {
    return sizeof(T) == 2 ? 2 : !dirichlet || (!vec && K == 8) ? 0 : 1;
  }
  // Whether the kernel holds the masked march.  Without it one field gains (fewer
  // registers: jacobi5 4096^2 x24 143 -> 138 us, BF16 star9r2 300^2 50 -> 39);
  // three fields lose 2 to 3 % and keep it.
  static constexpr bool masks(bool dirichlet) { return dirichlet || NF > 1; }
};

// Cut a grid into units for `slots` resident warps: as many chunks as fill
// them once, but none shorter than the 2 K R rows it stages again, unless the
// grid is so small that some SMs would have no warp for each of their four
// schedulers: then chunks of down to two rows (a launch's time is its longest
// chunk's).
inline StripCut strip_cut(const StripGrid& g, int valid, int kr, int slots) {
  StripCut c;
  c.strips = (g.nx + valid - 1) / valid;
  c.el = g.bc[1][0] == kDirichlet;
  c.er = g.bc[1][1] == kDirichlet && c.strips > c.el;
  const int ne = c.el + c.er, ni = c.strips - ne;
  const bool ylo = g.bc[0][0] == kDirichlet;
  constexpr int kNum = 2, kDen = 3;  // an edge chunk's share of an inner chunk's rows
  const int spread = std::min(g.ny / 2, 4 * device_sms() / c.strips);
  const int most = std::max(1, std::max(g.ny / (2 * kr), spread));
  // n chunks per inner strip, n * kDen / kNum per edge strip
  int n = int((int64_t(slots) * kNum) / (int64_t(ni) * kNum + int64_t(ne) * kDen));
  n = n < 1 ? 1 : n > most ? most : n;
  c.hc = (g.ny + n - 1) / n;
  c.top = ylo && n > 2 ? c.hc - c.hc * kNum / kDen : 0;
  c.hc = (g.ny + c.top + n - 1) / n;
  c.nc = (g.ny + c.top + c.hc - 1) / c.hc;
  int m = n * kDen / kNum;
  m = m < 1 ? 1 : m > most ? most : m;
  c.hce = (g.ny + c.top + m - 1) / m;
  if (c.hce <= c.top) c.hce = c.top + 1;
  c.nce = (g.ny + c.top + c.hce - 1) / c.hce;
  return c;
}

// Rows in whole vectors, every field pointer aligned for them (the outputs are
// checked to be 16-byte aligned by the caller).
inline bool strip_vec(const StepArgs& a) {
  if (a.g.n[2] % kStripV != 0) return false;
  for (int f = 0; f < a.g.nf; ++f)
    if (reinterpret_cast<uintptr_t>(a.in[f]) & 15) return false;
  return true;
}

inline bool strip_dirichlet(const StepArgs& a) {
  for (int ax = 1; ax < 3; ++ax)
    for (int sd = 0; sd < 2; ++sd)
      if (a.g.bc[ax][sd] == kDirichlet) return true;
  return false;
}

inline void strip_grid(const StepArgs& a, StripGrid* g) {
  g->nx = int(a.g.n[2]);
  g->ny = int(a.g.n[1]);
  for (int sd = 0; sd < 2; ++sd) {
    g->bc[0][sd] = a.g.bc[1][sd];
    g->bval[0][sd] = a.g.bval[1][sd];
    g->bc[1][sd] = a.g.bc[2][sd];
    g->bval[1][sd] = a.g.bval[2][sd];
  }
}

template <class Op, class T, int K, int STG>
struct StripRunner {
  using Cfg = StripCfg<T, Op::R, Op::NF, K, STG>;
  using G = StripGeom<T, Op::R, K>;
  static constexpr size_t SMEM = Cfg::SMEM;
  template <bool VEC, bool DIR> static auto kernel() {
    return &strip2d_kernel<Op, T, K, STG, Cfg::D, Cfg::NWB, Cfg::MINB, VEC,
                           Cfg::pm(VEC, DIR), Cfg::masks(DIR)>;
  }
  template <bool VEC, bool DIR> static cudaError_t occupancy(int* occ) {
    static PerDevice memo;
    return blocks_per_sm(memo, kernel<VEC, DIR>(), 32 * Cfg::NWB, SMEM, occ);
  }
  static void params(const StepArgs& a, int occ, StripParams<Op, T>* p) {
    for (int f = 0; f < Op::NF; ++f) {
      p->in[f] = static_cast<const T*>(a.in[f]);
      p->out[f] = static_cast<T*>(a.out[f]);
    }
    for (int s = 2; s <= STG; ++s) {
      double ca, cb;
      rk_coeffs(STG, s, &ca, &cb);
      p->rk[2 * (s - 2)] = ca;
      p->rk[2 * (s - 2) + 1] = cb;
    }
    strip_grid(a, &p->g);
    p->cut = strip_cut(p->g, G::VALID, K * Op::R, occ * device_sms() * Cfg::NWB);
    p->units = strip_units(p->cut);
  }
  template <bool VEC, bool DIR> static cudaError_t go(const StepArgs& a, const Op& op) {
    int occ = 1;
    cudaError_t e = occupancy<VEC, DIR>(&occ);
    if (e != cudaSuccess) return e;
    StripParams<Op, T> p;
    std::memset(static_cast<void*>(&p), 0, sizeof(p));
    p.op = op;
    params(a, occ, &p);
    kernel<VEC, DIR>()<<<(p.units + Cfg::NWB - 1) / Cfg::NWB, 32 * Cfg::NWB, SMEM, a.stream>>>(p);
    count_launches(1);
    return cudaGetLastError();
  }
  static cudaError_t run_vec(const StepArgs& a, const Op& op) {
    if (!strip_vec(a)) return cudaErrorNotSupported;
    return strip_dirichlet(a) ? go<true, true>(a, op) : go<true, false>(a, op);
  }
  static cudaError_t run(const StepArgs& a, const Op& op) {
    if (strip_vec(a)) return run_vec(a, op);
    if constexpr (sizeof(T) == 4) return strip_dirichlet(a) ? go<false, true>(a, op) : go<false, false>(a, op);
    return cudaErrorNotSupported;
  }
};

}  // namespace
}  // namespace lope
