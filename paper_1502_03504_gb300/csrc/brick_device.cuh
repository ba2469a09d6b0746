// Register bricks: K sweeps of a 3D radius-1 star function per pass, every
// intermediate state in registers (device templates; compiles under nvcc and
// NVRTC alike).  The 3D form of the register strips (strip_device.cuh).
//
// A block of WY half-warps owns a column of the grid, 64 columns (16 lanes of 4)
// by WY x RY rows, and marches a chunk of planes along z.  At step t it takes plane
// t of the input and computes plane t-l of every level l = 1 .. K (the state
// after l sweeps) from the last three planes of level l-1 in registers; level K
// is stored.  Taps along z come from that queue, along x from the lane's own
// columns and by shuffle from its neighbours, along y from the thread's own
// rows and, past them, from the first and last rows of the neighbouring
// half-warps, which each leaves in shared memory once per plane and level.  All
// levels of a step read rows that were left one step before, so one block
// barrier per plane is enough.  The outer K rows and 4 columns of the column
// are computed again by the neighbouring blocks.  Planes arrive in a private
// ring of shared memory per warp through cp.async, PF planes ahead, from
// source rows and columns fixed for the whole march (periodic sides already
// wrapped).
//
// Dirichlet sides: the first and last column of blocks start and end at the
// grid's side, so the values past it are what the outermost lanes see instead
// of a shuffle and the outermost half-warps instead of an exchanged row; neither
// needs a mask in the steady loop (masking the cells past a side level by level
// cost 1.6x at 512^3).  Only the planes past a z side are set, in loops of their
// own over the first and last steps.  Each level is rounded to the storage
// precision: bitwise the result of K one-sweep launches.
//
// What bounds it: latency, with 8 warps per SM: issue is busy 65 % of the time at
// 512^3, and a warp waits on exchange rows and planes in shared memory (0.53 per
// issue) and on staged planes (0.29), hardly on the barrier (0.06).
// One block of 16 half-warps x 4 rows and up to 255 registers measured best
// (diff7 FP32, us per sweep, 512^3 Dirichlet / 256^3 periodic / 130 x 500 x 510):
//   K = 4: 73.5 / 13.4 / 33.9 (244 registers)
//   K = 3: 77.2 / 15.1 / 37.3 (197); 12 half-warps, two blocks of 168: 95 / 18 / 51
//   K = 2: 95.5 / 17.5 / 52; 5 or 6 rows per thread were no better
// against 109 (two sweeps per launch) / 25.4 / 75.7 (one) on the z-marches.  The
// blocks cover 1.56 times the points of a periodic 256^3 grid (five blocks of 64 along
// x and y) and 1.27 times those of a Dirichlet 512^3; 128 columns (a warp per row)
// would cover 1.88 times the former.
#pragma once

#include "strip_device.cuh"

namespace lope {

namespace {

__device__ __forceinline__ void brick_store_n(float* d, const float (&w)[4], int j0, int j1) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (i >= j0 && i < j1) d[i] = w[i];
}

// Taps of column p of row r of a level: center plane c (rows of this thread),
// the rows beyond them, the columns beyond the lane's, the planes below and above.
template <int RY>
struct BrickAcc {
  const float (&c)[RY][kStripV];
  const float (&zm)[RY][kStripV];
  const float (&zp)[RY][kStripV];
  const float (&up)[kStripV];  // row -1
  const float (&dn)[kStripV];  // row RY
  float xl, xr;                // columns -1 and V of row r
  int r, p;
  __device__ __forceinline__ float operator()(int, int dx, int dy, int dz) const {
    if (dz != 0) return dz < 0 ? zm[r][p] : zp[r][p];
    if (dy != 0) return r + dy < 0 ? up[p] : r + dy >= RY ? dn[p] : c[r + dy][p];
    return p + dx < 0 ? xl : p + dx >= kStripV ? xr : c[r][p + dx];
  }
  __device__ __forceinline__ int64_t gidx() const { return 0; }
};

}  // namespace

struct BrickGrid {
  int nx, ny, nz;
  int bc[3][2];        // z, y, x
  float bval[3][2];
};

// What a brick pass computes besides the state K sweeps on.
enum : int {
  kBrickPlain = 0,
  kBrickStates = 1,  // every level's state is stored (a checkpoint segment's recomputation)
  kBrickAdjoint = 2  // K steps of the transposed diffusion backward in time, each with its
                     // sum of (L^T lambda) u_t over the grid (dL/dc)
};
// 256^3 FP32, us per launch: four states stored 75 (320 MB; four sweeps one at a
// time 98); two adjoint steps 63 (256 MB; one at a time 2 x 41).  The states u_t go
// to registers one step ahead of their use: staged two planes deep in shared
// memory that cost 6 more, and three steps per pass 43.
// dL/dc is summed in FP64, whose pipe runs one warp instruction in about 19 cycles:
// a conversion and an addition for each row of four cells made the launch 90 us.
// So a thread gathers the row sums of three planes in a pair of floats without
// loss (two-sum) before FP64 takes them; rows too large for a pair go to FP64 alone.

// One step of lambda' = lambda + c L^T lambda; the second result is L^T lambda
// (the operations of OpAdjDiffusion in the same order).
struct OpBrickAdjoint {
  static constexpr int R = 1, NF = 1;
  static constexpr bool REDUCES = false, STAR = true;
  Coef c;
  template <class C, class A>
  __device__ __forceinline__ void operator()(const A& U, C (&o)[1], C& lt) const {
    const C l = U(0, 0, 0, 0);
    const C nb = add(add(add(U(0, 1, 0, 0), U(0, -1, 0, 0)), add(U(0, 0, 1, 0), U(0, 0, -1, 0))),
                     add(U(0, 0, 0, 1), U(0, 0, 0, -1)));
    lt = fma_(C(-6), l, nb);
    o[0] = fma_(c.get(C()), lt, l);
  }
};

template <class Op, class T> struct BrickParams {
  Op op;
  const T* in;
  T* out[4];           // out[K-1]: the state K sweeps on; kBrickStates: out[l-1] level l
  const T* ut[4];      // kBrickAdjoint: u_t of level l in ut[l-1]
  double* partials;    // kBrickAdjoint: per-block sums, added to
  BrickGrid g;
  int tiles_x, tiles_y, zchunk;
};

template <class T, int K, int RY, int WY> struct BrickGeom {
  static constexpr int LX = 16;                            // lanes along x
  static constexpr int HL = 1;                             // halo lanes per side (K <= 4 columns)
  static constexpr int BX = LX * kStripV, BY = WY * RY;    // cells of a block
  static constexpr int THREADS = WY * LX;
  static constexpr int ROWB = LX * kStripV * int(sizeof(T));
  static constexpr int D = 4;                              // ring planes
  static constexpr int RING = D * RY * ROWB;               // bytes per half-warp
  static constexpr int EXROW = LX * kStripV * 4;           // an exchanged row (FP32)
  static constexpr int EXL = (WY + 2) * 2 * EXROW;         // a level's rows: half-warps -1 .. WY
  static constexpr int EX = K * EXL;                       // one of two exchange buffers
  static constexpr int SMEM = WY * RING + 2 * EX;
};

// Block i of n along an axis of extent m, blocks of b cells whose outer h are
// halo: first cell c and outputs [o0, o1).  A Dirichlet side needs no halo: the
// first block then starts at cell 0, the last ends at cell m - 1 (m >= b).
struct BrickSpan { int c, o0, o1; };
__host__ __device__ inline BrickSpan brick_span(int i, int n, int m, int b, int h, bool dlo, bool dhi) {
  const int v = b - 2 * h;
  BrickSpan s;
  s.c = i * v - (dlo ? 0 : h);
  s.o0 = i == 0 ? 0 : s.c + h;
  s.o1 = s.c + b - h < m ? s.c + b - h : m;
  if (dhi && i == n - 1) {
    s.c = m - b;
    s.o1 = m;
  }
  return s;
}
__host__ __device__ inline int brick_count(int m, int b, int h, bool dlo, bool dhi) {
  const int v = b - 2 * h, r = m - (dlo ? h : 0) - (dhi ? h : 0);
  return r <= v ? 1 : (r + v - 1) / v;
}

namespace {

template <class Op, class T, int K, int RY, int WY, int MODE, bool VEC>
struct Brick {
  using G = BrickGeom<T, K, RY, WY>;
  static_assert(MODE == kBrickPlain || VEC, "the adjoint's forms stage whole vectors");
  static_assert(Op::R == 1 && Op::NF == 1 && Op::STAR && K <= 4, "radius-1 star function of one field");
  static constexpr int V = kStripV, VB = V * int(sizeof(T)), D = G::D, PF = D - 1;

  static __device__ __forceinline__ void march(const BrickParams<Op, T>& p, unsigned char* smem,
                                               const BrickSpan& sx, const BrickSpan& sy, int z0, int z1) {
    const BrickGrid& g = p.g;
    const int lane = threadIdx.x % G::LX, wy = threadIdx.x / G::LX;
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    const int x = sx.c + lane * V;
    const int yw = sy.c + wy * RY;  // first row of this half-warp
    const int nsteps = (z1 - z0) + 2 * K;
    int gx[VEC ? 1 : V];
    if constexpr (VEC) {
      gx[0] = wrap(x, nx);
    } else {
#pragma unroll
      for (int j = 0; j < V; ++j) gx[j] = wrap(sx.c + lane + G::LX * j, nx);
    }
    int roff[RY];  // source rows, wrapped
#pragma unroll
    for (int r = 0; r < RY; ++r) roff[r] = wrap(yw + r, ny) * nx + (VEC ? gx[0] : 0);
    // What the outermost lanes see past their columns: the value of the
    // Dirichlet side the block ends at (elsewhere they are halo lanes, whose
    // results nothing reads).
    const float vxl = g.bval[2][0], vxr = g.bval[2][1];
    const bool first = lane == 0, last = lane == G::LX - 1;
    constexpr int kFar = 1 << 30;
    const int zlo = g.bc[0][0] == kDirichlet ? 0 : -kFar, zhi = g.bc[0][1] == kDirichlet ? nz : kFar;

    unsigned char* ring = smem + wy * G::RING;
    const uint32_t rbase = smem_u32(ring);
    // Exchanged rows (two buffers, used in turn): per level and half-warp its
    // first and last row.  Own rows, and the neighbours' rows beside them.
    // The rows of half-warps -1 and WY hold the Dirichlet y sides' values.
    constexpr int EXR = G::EXROW / 4, EXL = G::EXL / 4;  // floats per row, per level
    float* ex = reinterpret_cast<float*>(smem + WY * G::RING) + 2 * EXR + lane * V;
    for (int i = threadIdx.x; i < 2 * K * 2 * EXR; i += G::THREADS) {
      const int lv = i / (2 * EXR), j = i % (2 * EXR);  // buffer and level, row and column
      float* e = reinterpret_cast<float*>(smem + WY * G::RING) + lv * EXL;
      if (j < EXR) e[EXR + j] = g.bval[1][0];
      else e[(WY + 1) * 2 * EXR + j - EXR] = g.bval[1][1];
    }
    float* exw = ex + wy * 2 * EXR;
    const float* exu = exw - EXR;
    const float* exd = exw + 2 * EXR;
    const int64_t plane = int64_t(nx) * ny;
    int lz = wrap(z0 - K, nz);
    const T* src = p.in + int64_t(lz) * plane;
    // output columns [jv0, jv1) of this lane (aligned rows: all or none)
    const int jv0 = max(0, sx.o0 - x), jv1 = min(V, sx.o1 - x);
    const int64_t rowoff = int64_t(yw) * nx + x;  // row 0 of this thread in a plane
    T* dst = p.out[K - 1] + int64_t(z0 - 2 * K) * plane + rowoff;  // of step t's stored plane
    uint32_t rd = 0;
    // bit r: row r is an output row of this lane
    unsigned ok = 0;
#pragma unroll
    for (int r = 0; r < RY; ++r) {
      if (jv0 < jv1 && yw + r >= sy.o0 && yw + r < sy.o1) ok |= 1u << r;
    }
    // Planes of this pass's z range: out and ut hold plane z at z * plane.
    int64_t zoff = int64_t(z0 - K) * plane;  // of step t's newest plane
    // kBrickAdjoint: u_t of every level for the coming step, loaded to registers
    // right after the level's last use of the step before.
    float ut[MODE == kBrickAdjoint ? K : 1][RY][V];
    auto load_state = [&](int l, int t) {  // the plane level l computes at step t, if in the chunk
      if (unsigned(t - K - l) < unsigned(z1 - z0)) {
        const T* s = p.ut[l - 1] + (int64_t(z0 - K + t - l) * plane);
#pragma unroll
        for (int r = 0; r < RY; ++r)
          if (ok >> r & 1) strip_load(s + roff[r], ut[l - 1][r]);
      }
    };
    auto copy_plane = [&](uint32_t slot) {
#pragma unroll
      for (int r = 0; r < RY; ++r) {
        const uint32_t d = rbase + slot + r * (D * G::ROWB);
        const T* row = src + roff[r];
        if constexpr (VEC) {
          cp_async_vec<VB>(d + lane * VB, row);
        } else {
#pragma unroll
          for (int j = 0; j < V; ++j)
            cp_async_elem<int(sizeof(T))>(d + (lane + G::LX * j) * int(sizeof(T)), row + gx[j]);
        }
      }
      src += plane;
      if (++lz == nz) {
        lz = 0;
        src -= int64_t(nz) * plane;
      }
    };
#pragma unroll 1
    for (int t = 0; t < PF; ++t) {
      if (t < nsteps) copy_plane(t * G::ROWB);
      cp_async_commit();
    }

    // kBrickAdjoint: this thread's sum; the row sums not yet in it, and the
    // rounding errors of their sum
    double red = 0.0;
    float sum = 0.f, low = 0.f;
    float q[K][3][RY][V];
    auto put_row = [&](float* d, const float (&w)[V]) {
      *reinterpret_cast<float4*>(d) = make_float4(w[0], w[1], w[2], w[3]);
    };
    __syncthreads();
    auto step = [&](auto ph_tag, auto z_tag, int t) {
      constexpr bool ZEDGE = decltype(z_tag)::value != 0;  // levels may lie past a z side
      // a level's plane past a Dirichlet z side holds its value
      auto mask = [&](float (&w)[RY][V], int z) {
        if (z < zlo || z >= zhi) {
#pragma unroll
          for (int r = 0; r < RY; ++r)
#pragma unroll
            for (int j = 0; j < V; ++j) w[r][j] = z < zlo ? g.bval[0][0] : g.bval[0][1];
        }
      };
      constexpr int PH = decltype(ph_tag)::value;  // t mod 3
      const int nb = (t & 1) * (G::EX / 4), ob = G::EX / 4 - nb;
      float* const wrow = exw + nb;
      const float* const urow = exu + ob;
      const float* const drow = exd + ob;
      cp_async_wait<PF - 1>();
      if constexpr (!VEC) __syncwarp();
#pragma unroll
      for (int r = 0; r < RY; ++r)
        strip_load(reinterpret_cast<const T*>(ring + rd + r * (D * G::ROWB)) + lane * V, q[0][PH][r]);
      if constexpr (!VEC) __syncwarp();
      if (t + PF < nsteps) copy_plane((rd + PF * G::ROWB) & (D * G::ROWB - 1));
      cp_async_commit();
      if constexpr (ZEDGE) mask(q[0][PH], z0 - K + t);
      put_row(wrow, q[0][PH][0]);
      put_row(wrow + EXR, q[0][PH][RY - 1]);
      auto level = [&](auto l_tag) {
        constexpr int L = decltype(l_tag)::value;
        // slots of level L-1: newest plane, the center one before it, the one below
        constexpr int ZP = ((PH - (L - 1)) % 3 + 3) % 3, CC = (ZP + 2) % 3, ZM = (ZP + 1) % 3;
        float up[V], dn[V];
        strip_load(urow + (L - 1) * EXL, up);
        strip_load(drow + (L - 1) * EXL, dn);
        float o[RY][V];
        // kBrickAdjoint: a chain of FMAs over each row's cells
        float rsum[MODE == kBrickAdjoint ? RY : 1];
        const bool inside = MODE == kBrickAdjoint && unsigned(t - K - L) < unsigned(z1 - z0);
#pragma unroll
        for (int r = 0; r < RY; ++r) {
          float chain = 0.f;
          float xl = shfl_left(q[L - 1][CC][r][V - 1]), xr = shfl_right(q[L - 1][CC][r][0]);
          if (first) xl = vxl;
          if (last) xr = vxr;
#pragma unroll
          for (int j = 0; j < V; ++j) {
            BrickAcc<RY> acc{q[L - 1][CC], q[L - 1][ZM], q[L - 1][ZP], up, dn, xl, xr, r, j};
            float res[1], second = 0.f;
            p.op(acc, res, second);
            o[r][j] = res[0];
            if constexpr (MODE == kBrickAdjoint) chain = fma_(second, ut[L - 1][r][j], chain);
          }
          if constexpr (MODE == kBrickAdjoint) rsum[r] = inside && (ok >> r & 1) ? chain : 0.f;
        }
        if constexpr (MODE == kBrickAdjoint) {
          float most = 0.f;
#pragma unroll
          for (int r = 0; r < RY; ++r) most = fmaxf(most, fabsf(rsum[r]));
          if (most < 1.2676506e30f) {  // 2^100: no sum of a period's rows overflows
#pragma unroll
            for (int r = 0; r < RY; ++r) {
              const float n = add(sum, rsum[r]), d = sub(n, sum);
              low = add(low, add(sub(sum, sub(n, d)), sub(rsum[r], d)));
              sum = n;
            }
          } else {
#pragma unroll
            for (int r = 0; r < RY; ++r) red += double(rsum[r]);
          }
        }
        if constexpr (MODE == kBrickAdjoint) load_state(L, t + 1);
        if constexpr (MODE == kBrickStates && L < K) {
          if (unsigned(t - K - L) < unsigned(z1 - z0)) {
            T* d = p.out[L - 1] + (zoff - L * plane + rowoff);
#pragma unroll
            for (int r = 0; r < RY; ++r)
              if (ok >> r & 1) strip_store(d + int64_t(r) * nx, o[r]);
          }
        }
        if constexpr (L == K) {
          if (t >= 2 * K && t < nsteps) {
#pragma unroll
            for (int r = 0; r < RY; ++r)
              if (ok >> r & 1) {
                if constexpr (VEC) strip_store(dst + int64_t(r) * nx, o[r]);
                else brick_store_n(dst + int64_t(r) * nx, o[r], jv0, jv1);
              }
          }
        } else {
          constexpr int W = ((PH - L) % 3 + 3) % 3;  // slot of plane t - L
#pragma unroll
          for (int r = 0; r < RY; ++r) strip_round<T>(o[r]);
          if constexpr (ZEDGE) mask(o, z0 - K + t - L);
#pragma unroll
          for (int r = 0; r < RY; ++r)
#pragma unroll
            for (int j = 0; j < V; ++j) q[L][W][r][j] = o[r][j];
          put_row(wrow + L * EXL, o[0]);
          put_row(wrow + L * EXL + EXR, o[RY - 1]);
        }
      };
      level(StripTag<1>());
      if constexpr (K >= 2) level(StripTag<2>());
      if constexpr (K >= 3) level(StripTag<3>());
      if constexpr (K >= 4) level(StripTag<4>());
      dst += plane;
      zoff += plane;
      rd = (rd + G::ROWB) & (D * G::ROWB - 1);
      __syncthreads();
    };
    // Steps run in threes (the queue's period); planes whose level is not
    // complete yet, and those past z1, are computed and dropped.
    int t = 0;
    auto run_to = [&](auto z_tag, int end) {
#pragma unroll 1
      for (; t < end; t += 3) {
        step(StripTag<0>(), z_tag, t);
        step(StripTag<1>(), z_tag, t + 1);
        step(StripTag<2>(), z_tag, t + 2);
        if constexpr (MODE == kBrickAdjoint) {
          red += double(sum) + double(low);
          sum = low = 0.f;
        }
      }
    };
    run_to(StripTag<1>(), z0 - K < zlo ? 2 * K : 0);
    run_to(StripTag<0>(), z1 + K > zhi ? nsteps - 2 * K - 2 : nsteps);
    run_to(StripTag<1>(), nsteps);
    cp_async_wait<0>();
    if constexpr (MODE == kBrickAdjoint) {
      // the block's sum in a fixed order
      __shared__ double ws[G::THREADS / 32];
      double total = red;
      for (int o = 16; o > 0; o >>= 1) total += __shfl_down_sync(0xffffffffu, total, o);
      if (threadIdx.x % 32 == 0) ws[threadIdx.x / 32] = total;
      __syncthreads();
      if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < G::THREADS / 32; ++w) s += ws[w];
        p.partials[blockIdx.x] += s;
      }
    }
  }
};

template <class Op, class T, int K, int RY, int WY, int MODE, bool VEC>
__global__ void __launch_bounds__(BrickGeom<T, K, RY, WY>::THREADS, 1) brick3d_kernel(const __grid_constant__ BrickParams<Op, T> p) {
  using B = Brick<Op, T, K, RY, WY, MODE, VEC>;
  using G = typename B::G;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ntiles = p.tiles_x * p.tiles_y;
  const int tile = blockIdx.x % ntiles, zc = blockIdx.x / ntiles;
  const int z0 = zc * p.zchunk, z1 = min(p.g.nz, z0 + p.zchunk);
  if (z0 >= z1) return;
  const BrickGrid& g = p.g;
  const BrickSpan sx = brick_span(tile % p.tiles_x, p.tiles_x, g.nx, G::BX, G::HL * kStripV,
                                  g.bc[2][0] == kDirichlet, g.bc[2][1] == kDirichlet);
  const BrickSpan sy = brick_span(tile / p.tiles_x, p.tiles_y, g.ny, G::BY, K,
                                  g.bc[1][0] == kDirichlet, g.bc[1][1] == kDirichlet);
  B::march(p, smem_raw, sx, sy, z0, z1);
}

}  // namespace
}  // namespace lope
