// Register strips: K sweeps of a 2D local function per pass over the grid,
// every intermediate state in registers (device templates; compiles under
// nvcc and NVRTC alike).
//
// FP32 and BF16 storage.  A warp owns a strip of 32 x V = 128 consecutive
// columns (V = 4 per lane) and marches along y over a chunk of rows.  At each
// step it takes one staged row of the input state and advances a pipeline
// of levels: level l (the state after l sweeps) is computed R rows behind level
// l-1 from a queue of that level's last 2R+1 rows in registers, and level K is
// stored.  Taps along y come from the queue; taps along x from the lane's own
// registers or, past its V columns, from the neighbouring lanes by warp
// shuffles.  The sweeps use no shared memory and no barrier.  The outer h >= K R
// columns of a strip (h a whole number of lanes) are computed again by the
// neighbouring strip, and the first 2 K R steps of a chunk fill the pipeline.
// Every level is rounded to the storage precision, so the result is bitwise
// that of K one-sweep launches.
//
// What bounds it: HBM reads and writes each value once per K sweeps; from K = 4
// (three fields) or K = 8 (one) on, instruction issue does.  So the steady loop
// has no branch around a level: conditional levels (which would skip the rows
// that only fill the pipeline) made the compiler keep the queue in place with
// moves, 17 of the 52 instructions per level and row.  jacobi5 FP32 8192^2, per
// sweep: 31 us with conditional levels on pairs of columns (packed f32x2
// arithmetic), 25 us branch-free on scalars at K = 4, 17.7 us at K = 8, against
// 56.8 us on the two-sweep shared-memory tiles.  Packed arithmetic halves its issue
// slots but not its time on the FMA pipe (K = 8: 138.5M -> 121.1M warp instructions,
// 148 -> 162 us), so only marches with many other instructions use it (StripCfg::pm).
//
// The rows arrive in a private ring of shared memory per warp through
// asynchronous copies (cp.async), PF rows ahead.  A lane's source column is
// fixed for the whole march, with a periodic side already wrapped, so periodic
// grids cost nothing extra.  Past a Dirichlet side every level holds the side's
// value (rows first, then columns: the slowest axis decides); only strips and
// chunks whose window crosses such a side run the instance with those masks.
#pragma once

#include "device_common.cuh"

namespace lope {

namespace {

constexpr int kStripV = 4;  // columns per lane

__device__ __forceinline__ float shfl_left(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float shfl_right(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }

// A lane's V columns of a row.  Packed: two register pairs for the f32x2
// instructions, pair j holding columns j and j + 2, so that a tap one column to
// the side is the other pair for half of the columns and takes one move and a
// shuffled value for the rest.
template <bool PK> struct StripVal { using type = float; };
template <> struct StripVal<true> { using type = F2; };
template <bool PK> struct StripRow {
  float w[kStripV];
  __device__ __forceinline__ float get(int i) const { return w[i]; }
  __device__ __forceinline__ void set(const float (&x)[kStripV]) {
#pragma unroll
    for (int i = 0; i < kStripV; ++i) w[i] = x[i];
  }
};
template <> struct StripRow<true> {
  F2 w[2];
  __device__ __forceinline__ float get(int i) const { return i < 2 ? w[i].lo() : w[i - 2].hi(); }
  __device__ __forceinline__ void set(const float (&x)[kStripV]) {
    w[0] = F2::make(x[0], x[2]);
    w[1] = F2::make(x[1], x[3]);
  }
};

// Accessor of column p (packed: columns p and p + 2) of a lane's row: q holds
// the 2R+1 rows of the level below, row n in slot n mod (2R+1); C0 is the slot of
// the row being computed.  EAGER: the neighbouring lanes' columns of that row
// were fetched once (xl[i]: column -1-i, xr[i]: column V+i); otherwise each tap
// that needs one shuffles it.
template <int NF, int NQ, int C0, bool EAGER, bool PK>
struct StripAcc {
  static constexpr int V = kStripV;
  const StripRow<PK> (&q)[NQ][NF];
  const float (&xl)[NF][NQ / 2];
  const float (&xr)[NF][NQ / 2];
  int p;
  __device__ __forceinline__ float at(const StripRow<PK>& w, int f, int i) const {
    if (i < 0) return EAGER ? xl[f][-1 - i] : shfl_left(w.get(V + i));
    if (i >= V) return EAGER ? xr[f][i - V] : shfl_right(w.get(i - V));
    return w.get(i);
  }
  __device__ __forceinline__ auto operator()(int f, int dx, int dy, int) const {
    const StripRow<PK>& w = q[(C0 + dy + NQ) % NQ][f];
    const int i = p + dx;
    if constexpr (PK) {
      if (i == 0 || i == 1) return w.w[i];
      return F2::make(at(w, f, i), at(w, f, i + 2));
    } else {
      return at(w, f, i);
    }
  }
  __device__ __forceinline__ int64_t gidx() const { return 0; }
};

// Round a lane's row to what storage would hold.
template <class T> __device__ __forceinline__ void strip_round(float (&w)[kStripV]) {
  if constexpr (sizeof(T) == 2) {
#pragma unroll
    for (int p = 0; p < kStripV; p += 2) {
      const __nv_bfloat162 b = __floats2bfloat162_rn(w[p], w[p + 1]);
      const uint32_t v = *reinterpret_cast<const uint32_t*>(&b);
      w[p] = __uint_as_float(v << 16);
      w[p + 1] = __uint_as_float(v & 0xffff0000u);
    }
  }
}

// A row's columns in order.
__device__ __forceinline__ StripRow<false> strip_flat(const float (&o)[kStripV]) {
  return {{o[0], o[1], o[2], o[3]}};
}
__device__ __forceinline__ StripRow<false> strip_flat(const F2 (&o)[2]) {
  return {{o[0].lo(), o[1].lo(), o[0].hi(), o[1].hi()}};
}

// A lane's V values of a staged row (16 or 8 bytes of shared memory).
__device__ __forceinline__ void strip_load(const float* s, float (&w)[4]) {
  const float4 v = *reinterpret_cast<const float4*>(s);
  w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
}
__device__ __forceinline__ void strip_load(const __nv_bfloat16* s, float (&w)[4]) {
  const uint2 v = *reinterpret_cast<const uint2*>(s);
  w[0] = __uint_as_float(v.x << 16);
  w[1] = __uint_as_float(v.x & 0xffff0000u);
  w[2] = __uint_as_float(v.y << 16);
  w[3] = __uint_as_float(v.y & 0xffff0000u);
}

// A lane's V values to memory: one vector store, or element by element (the
// first nv of them) where rows are not aligned for it.
__device__ __forceinline__ void strip_store(float* d, const float (&w)[4]) {
  *reinterpret_cast<float4*>(d) = make_float4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ void strip_store(__nv_bfloat16* d, const float (&w)[4]) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(w[0], w[1]);
  const __nv_bfloat162 b = __floats2bfloat162_rn(w[2], w[3]);
  *reinterpret_cast<uint2*>(d) = make_uint2(*reinterpret_cast<const uint32_t*>(&a),
                                            *reinterpret_cast<const uint32_t*>(&b));
}
__device__ __forceinline__ void strip_store_n(float* d, const float (&w)[4], int nv) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (i < nv) d[i] = w[i];
}

template <int B>
__device__ __forceinline__ void cp_async_vec(uint32_t dst, const void* src) {
  if constexpr (B == 16) cp_async_16(dst, src);
  else cp_async_elem<B>(dst, src);
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <int V> struct StripTag { static constexpr int value = V; };

// Whether a local function is a run-time compiled one (Op::USER).
template <class Op> constexpr auto strip_user(int) -> decltype(Op::USER) { return Op::USER; }
template <class Op> constexpr bool strip_user(long) { return false; }

}  // namespace

// One grid as a strip pass sees it.
struct StripGrid {
  int nx, ny;
  int bc[2][2];        // [0 = y axis, 1 = x axis][side]
  double bval[2][2];
};

// Strip geometry of a function of radius R at depth K: HL halo lanes on each
// side, VALID output columns per strip.
template <class T, int R, int K> struct StripGeom {
  static constexpr int V = kStripV;
  static constexpr int HL = (K * R + V - 1) / V;
  static constexpr int VALID = (32 - 2 * HL) * V;
  static constexpr int ROWB = 32 * V * int(sizeof(T));  // bytes of a staged row
};

// One unit of work: K sweeps of the strip whose first output column is x0 over
// rows [y0, y1).  ring: this warp's NF x D staged rows.  VEC: rows are a whole
// number of vectors and every pointer is aligned for them; otherwise (FP32) lane
// l stages columns l, l + 32, ... element by element.
// STG >= 2: the K = STG levels are the stages of one Runge-Kutta step: level l
// >= 2 is a_l u + b_l E(level l-1), u read again from the ring, which keeps
// STG R rows behind the newest for it.
// PM: which marches compute on packed pairs of columns, 0 none, 1 those with
// masks, 2 all.
template <class Op, class T, int K, int STG, int D, bool VEC, int PM>
struct Strip {
  using C = float;
  using G = StripGeom<T, Op::R, K>;
  static constexpr int R = Op::R, NF = Op::NF, NQ = 2 * R + 1, V = G::V, VB = V * int(sizeof(T));
  static constexpr int ROWB = G::ROWB, RING = D * ROWB, BYTES = NF * RING;
  static constexpr int PF = D - 1 - (STG >= 2 ? STG * R : 0);  // rows staged ahead
  static_assert((D & (D - 1)) == 0 && PF >= 2, "ring depth");
  static_assert(STG == 1 || K == STG, "the levels are the stages of one step");
  static_assert(VEC || sizeof(T) == 4, "element copies of 4 bytes");
  // Star functions of one field read both x neighbours of the row: fetch them
  // once per row.  The builtins of several fields read a few of theirs only.  A
  // run-time compiled function never shuffles inside its own body, whose
  // control flow is the user's.
  // The builtins are plain arithmetic: what they compute from rows that have not
  // come yet is dropped.  A run-time compiled function may loop or index by the
  // values it reads, so its queues start out as copies of the first row and its
  // last steps repeat the last one: it sees states and boundary values only.
  // (Steps that leave out the incomplete levels instead doubled the code: 7.3 s
  // to compile Gray-Scott, 4.3 this way.)
  static constexpr bool USER = strip_user<Op>(0);
  static constexpr bool EAGER = Op::STAR && (NF == 1 || USER);

  template <bool MASK>
  static __device__ __forceinline__ void march(const Op& op, const T* const* in, T* const* out,
                                               const StripGrid& g, int x0, int y0, int y1,
                                               unsigned char* ring, const Coef* rk) {
    // Run-time compiled functions stay on scalars: their bodies may need them, and
    // a packed product that feeds a sum may be contracted.
    constexpr bool PK = !USER && (PM == 2 || (PM == 1 && MASK));
    constexpr int NP = PK ? 2 : V;  // values of type W per row
    using W = typename StripVal<PK>::type;
    const int lane = threadIdx.x & 31;
    const int nx = g.nx, ny = g.ny;
    const int x = x0 + (lane - G::HL) * V;  // this lane's first column
    const int yb = y0 - K * R;              // row of step 0
    const int nsteps = (y1 - y0) + 2 * K * R;
    // Source columns, wrapped (a column past a Dirichlet side stages a cell of
    // the row, which the mask replaces).
    int gx[VEC ? 1 : V];
    if constexpr (VEC) {
      gx[0] = wrap(x, nx);
    } else {
#pragma unroll
      for (int j = 0; j < V; ++j) gx[j] = wrap(x0 - G::HL * V + lane + 32 * j, nx);
    }
    // Past a Dirichlet x side: bit j of cmask, and the side's value (a lane's
    // columns are all left of the grid or none is, so it sees one side).
    unsigned cmask = 0;
    const C cval = x < 0 ? C(g.bval[1][0]) : C(g.bval[1][1]);
    const C vy0 = C(g.bval[0][0]), vy1 = C(g.bval[0][1]);
    constexpr int kFar = 1 << 30;
    int ylo = -kFar, yhi = kFar;
    if constexpr (MASK) {
      const bool l = g.bc[1][0] == kDirichlet, h = g.bc[1][1] == kDirichlet;
#pragma unroll
      for (int j = 0; j < V; ++j)
        if ((l && x + j < 0) || (h && x + j >= nx)) cmask |= 1u << j;
      if (g.bc[0][0] == kDirichlet) ylo = 0;
      if (g.bc[0][1] == kDirichlet) yhi = ny;
    }
    auto mask = [&](C (&w)[V], int y) {
      const bool o0 = y < ylo, o1 = y >= yhi;
      const C vy = o0 ? vy0 : vy1;
#pragma unroll
      for (int j = 0; j < V; ++j) {
        if (cmask >> j & 1) w[j] = cval;
        if (o0 || o1) w[j] = vy;
      }
    };

    const uint32_t rbase = smem_u32(ring);
    int lw = wrap(yb, ny);  // row of the next copy
    // One field: a running source pointer; several: the kernel's pointers (in
    // constant memory) plus one running offset.
    int64_t lrow = int64_t(lw) * nx + (VEC ? gx[0] : 0);
    const T* src = in[0] + lrow;
    auto copy_row = [&](uint32_t slot) {
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        const T* row = NF == 1 ? src : in[f] + lrow;
        const uint32_t d = rbase + f * RING + slot;
        if constexpr (VEC) {
          cp_async_vec<VB>(d + lane * VB, row);
        } else {
#pragma unroll
          for (int j = 0; j < V; ++j)
            cp_async_elem<int(sizeof(T))>(d + (lane + 32 * j) * int(sizeof(T)), row + gx[j]);
        }
      }
      const bool end = ++lw == ny;
      if constexpr (NF == 1) {
        src += nx;
        if (end) src -= int64_t(ny) * nx;
      } else {
        lrow += nx;
        if (end) lrow -= int64_t(ny) * nx;
      }
      if (end) lw = 0;
    };
    if constexpr (!VEC) __syncwarp();
#pragma unroll 1
    for (int t = 0; t < PF; ++t) {
      if (t < nsteps) copy_row(t * ROWB);
      cp_async_commit();
    }

    StripRow<PK> q[K][NQ][NF];
    if constexpr (USER) {
      cp_async_wait<PF - 1>();
      if constexpr (!VEC) __syncwarp();
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        C w[V];
        strip_load(reinterpret_cast<const T*>(ring + f * RING) + lane * V, w);
        if constexpr (MASK) mask(w, yb);
#pragma unroll
        for (int l = 0; l < K; ++l)
#pragma unroll
          for (int n = 0; n < NQ; ++n) q[l][n][f].set(w);
      }
    }
    const int nv = lane < G::HL || lane >= 32 - G::HL ? 0 : max(0, min(V, nx - x));
    int64_t orow = int64_t(y0 - 2 * K * R) * nx + x;  // output offset of step t's stored row
    T* dst = out[0] + orow;
    uint32_t rd = 0;                                  // ring slot of row t
    auto step = [&](auto ph_tag, int t) {
      constexpr int PH = decltype(ph_tag)::value;  // t mod NQ
      cp_async_wait<PF - 1>();
      if constexpr (!VEC) __syncwarp();
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        C w[V];
        strip_load(reinterpret_cast<const T*>(ring + f * RING + rd) + lane * V, w);
        if constexpr (MASK && PK) mask(w, yb + t);
        q[0][PH][f].set(w);
      }
      if constexpr (!VEC) __syncwarp();
      if (t + PF < nsteps) copy_row((rd + PF * ROWB) & (RING - 1));
      cp_async_commit();
      if constexpr (MASK && !PK) {
#pragma unroll
        for (int f = 0; f < NF; ++f) mask(q[0][PH][f].w, yb + t);
      }
      auto level = [&](auto l_tag) {
        constexpr int L = decltype(l_tag)::value;
        constexpr int C0 = ((PH - L * R) % NQ + NQ) % NQ;
        W o[NF][NP];
        C xl[NF][R], xr[NF][R];
        if constexpr (EAGER) {
#pragma unroll
          for (int f = 0; f < NF; ++f)
#pragma unroll
            for (int i = 0; i < R; ++i) {
              xl[f][i] = shfl_left(q[L - 1][C0][f].get(V - 1 - i));
              xr[f][i] = shfl_right(q[L - 1][C0][f].get(i));
            }
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          StripAcc<NF, NQ, C0, EAGER, PK> acc{q[L - 1], xl, xr, p};
          W r[NF];
          W unused = W(0.f);
          op(acc, r, unused);
#pragma unroll
          for (int f = 0; f < NF; ++f) o[f][p] = r[f];
        }
        if constexpr (STG >= 2 && L >= 2) {
          const Coef ca = rk[2 * (L - 2)], cb = rk[2 * (L - 2) + 1];
#pragma unroll
          for (int f = 0; f < NF; ++f) {
            C b[V];
            strip_load(reinterpret_cast<const T*>(ring + f * RING + ((rd - L * R * ROWB) & (RING - 1))) + lane * V, b);
            if constexpr (MASK) mask(b, yb + t - L * R);
            StripRow<PK> u;
            u.set(b);
#pragma unroll
            for (int p = 0; p < NP; ++p) o[f][p] = fma_(cb.get(W()), o[f][p], mul(ca.get(W()), u.w[p]));
          }
        }
        if constexpr (L == K) {
          if (t >= 2 * K * R && t < nsteps) {
#pragma unroll
            for (int f = 0; f < NF; ++f) {
              T* d = NF == 1 ? dst : out[f] + orow;
              if constexpr (VEC) {
                if (nv > 0) strip_store(d, strip_flat(o[f]).w);
              } else {
                strip_store_n(d, strip_flat(o[f]).w, nv);
              }
            }
          }
        } else {
#pragma unroll
          for (int f = 0; f < NF; ++f) {
            if constexpr (MASK || sizeof(T) == 2) {
              StripRow<false> w = strip_flat(o[f]);
              strip_round<T>(w.w);
              if constexpr (MASK) mask(w.w, yb + t - L * R);
              q[L][C0][f].set(w.w);
            } else {
#pragma unroll
              for (int p = 0; p < NP; ++p) q[L][C0][f].w[p] = o[f][p];
            }
          }
        }
      };
      level(StripTag<1>());
      if constexpr (K >= 2) level(StripTag<2>());
      if constexpr (K >= 3) level(StripTag<3>());
      if constexpr (K >= 4) level(StripTag<4>());
      if constexpr (K >= 5) level(StripTag<5>());
      if constexpr (K >= 6) level(StripTag<6>());
      if constexpr (K >= 7) level(StripTag<7>());
      if constexpr (K >= 8) level(StripTag<8>());
      if constexpr (NF == 1) dst += nx;
      else orow += nx;
      if (!USER || t + 1 < nsteps) rd = (rd + ROWB) & (RING - 1);
    };
    // The step count is rounded up to the queue's period: the rows of the
    // first 2 K R steps whose level is not complete yet, and those past y1,
    // are computed from whatever the queue holds and dropped (no stored row
    // depends on them).
#pragma unroll 1
    for (int t = 0; t < nsteps; t += NQ) {
      step(StripTag<0>(), t);
      step(StripTag<1>(), t + 1);
      step(StripTag<2>(), t + 2);
      if constexpr (NQ == 5) {
        step(StripTag<3>(), t + 3);
        step(StripTag<4>(), t + 4);
      }
    }
    cp_async_wait<0>();
  }

  // DIR: the grid may have a Dirichlet side.
  template <bool DIR>
  static __device__ __forceinline__ void run(const Op& op, const T* const* in, T* const* out,
                                             const StripGrid& g, int x0, int y0, int y1,
                                             unsigned char* ring, const Coef* rk) {
    if constexpr (!DIR) return march<false>(op, in, out, g, x0, y0, y1, ring, rk);
    const bool dx = (g.bc[1][0] == kDirichlet && x0 - G::HL * V < 0) ||
                    (g.bc[1][1] == kDirichlet && x0 + G::VALID + G::HL * V > g.nx);
    const bool dy = (g.bc[0][0] == kDirichlet && y0 - K * R < 0) ||
                    (g.bc[0][1] == kDirichlet && y1 + K * R > g.ny);
    if (dx || dy) march<true>(op, in, out, g, x0, y0, y1, ring, rk);
    else march<false>(op, in, out, g, x0, y0, y1, ring, rk);
  }
};

// The cut of one grid into units.  Inner strips are cut into nc chunks, strips
// that touch a Dirichlet x side into nce >= nc shorter ones (their masks cost
// about half as much again per row, and with all units resident at once the
// slowest sets the time); the first chunk of a grid whose low y side is Dirichlet
// is shortened the same way (top).  Units of edge strips come first.
struct StripCut {
  int strips;      // all strips
  int el, er;      // 1: the first / last strip is cut into nce chunks
  int nc, nce;
  int hc, hce;     // rows per chunk of inner / edge strips
  int top;         // rows taken off the first chunk (Dirichlet low y side)
};

__host__ __device__ inline int strip_units(const StripCut& c) {
  const int ne = c.el + c.er;
  return ne * c.nce + (c.strips - ne) * c.nc;
}
// Unit u: its strip and rows.
__host__ __device__ inline void strip_unit(const StripCut& c, int ny, int u, int* s, int* y0, int* y1) {
  const int ne = c.el + c.er;
  int h = c.hc, i;
  if (u < ne * c.nce) {
    i = u / ne;
    const int e = u - i * ne;
    *s = c.el && e == 0 ? 0 : c.strips - 1;
    h = c.hce;
  } else {
    u -= ne * c.nce;
    const int ni = c.strips - ne;
    i = u / ni;
    *s = c.el + u - i * ni;
  }
  const int a = i * h - c.top, b = a + h;
  *y0 = a < 0 ? 0 : a;
  *y1 = b < ny ? b : ny;
}

template <class Op, class T> struct StripParams {
  Op op;
  Coef rk[4];  // Runge-Kutta: a, b of stage 2, then of stage 3
  const T* in[kMaxFields];
  T* out[kMaxFields];
  StripGrid g;
  StripCut cut;
  int units;
};

namespace {

// NWB warps per block, one unit each; neighbouring units cover neighbouring
// strips of the same rows.
template <class Op, class T, int K, int STG, int D, int NWB, int MINB, bool VEC, int PM, bool DIR>
__global__ void __launch_bounds__(32 * NWB, MINB)
    strip2d_kernel(const __grid_constant__ StripParams<Op, T> p) {
  using S = Strip<Op, T, K, STG, D, VEC, PM>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x / 32;
  const int u = blockIdx.x * NWB + warp;
  if (u >= p.units) return;
  int s, y0, y1;
  strip_unit(p.cut, p.g.ny, u, &s, &y0, &y1);
  if (y0 >= y1) return;
  S::template run<DIR>(p.op, p.in, p.out, p.g, s * S::G::VALID, y0, y1, smem_raw + warp * S::BYTES, p.rk);
}

}  // namespace
}  // namespace lope
