// Batched form: many independent grids of uneven sizes advanced together by
// one persistent, cooperatively launched kernel (trapezoid tiles), or one kernel
// per pass (register strips, below).
//
// The work list holds every (grid, tile) pair of the batch.  Each pass runs k
// fused sweeps on every tile (trap.cuh), then all blocks meet at a grid-wide
// barrier before the next pass reads what this one wrote — the one-GPU form
// of "all threads finish the loop body, then the halo transfer synchronises"
// (Sec. 3.2).  The barrier wait is bounded: after kWaitLimitNs it records a
// timeout in the error flag and the kernel returns.  The barrier's GPU-scope
// acquire, passed on to the whole block by its CTA barrier, orders every read
// of the next pass (the asynchronous window copies included) after the stores
// every block made in this one.
#include <algorithm>
#include <type_traits>

#include "strip_kernels.cuh"
#include "trap.cuh"

namespace lope {

namespace {

constexpr int kBatchThreads = 256;
constexpr int kBatchWarps = 4, kBatchRing = 8;  // strips: warps per block, staged rows per warp

__device__ __forceinline__ bool grid_sync(unsigned int* bar, unsigned int target, int* err,
                                          volatile int* s_abort, unsigned long long wait_ns,
                                          bool arrive) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (arrive) atomicAdd(bar, 1u);
    const uint64_t t0 = global_ns();
    for (;;) {
      unsigned int v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (v >= target) break;
      if (global_ns() - t0 > wait_ns) {
        raise_error(err, kErrTimeout);
        *s_abort = 1;
        break;
      }
      __nanosleep(64);
    }
    __threadfence();
  }
  __syncthreads();
  return *s_abort == 0;
}

__device__ __forceinline__ int find_grid(const BatchGrid* grids, int ngrids, int item) {
  int lo = 0, hi = ngrids - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (grids[mid].first_item <= item) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Tile policies: the variable-shape trapezoid (any tile and depth), or the
// shape fixed at compile time (TrapFixed: every tap at an immediate offset).
struct TileAny {
  template <class Op, class T>
  static __device__ __forceinline__ void run(const Op& op, const T* const* src, T* const* dst,
                                             const TrapGrid& g, int x0, int y0, int tx, int ty,
                                             int kp, C_t<T>* smem) {
    trap_tile<Op, T>(op, src, dst, g, x0, y0, tx, ty, kp, smem);
  }
};
template <int TX, int TY, int K>
struct TileFixed {
  template <class Op, class T>
  static __device__ __forceinline__ void run(const Op& op, const T* const* src, T* const* dst,
                                             const TrapGrid& g, int x0, int y0, int, int, int kp,
                                             C_t<T>* smem) {
    TrapFixed<Op, T, TX, TY, K>::tile(op, src, dst, g, x0, y0, kp, smem);
  }
};

template <class Op, class T, class Tile>
__global__ void __launch_bounds__(kBatchThreads) batch_kernel(Op op, BatchPlanDev p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ volatile int s_abort;
  if (threadIdx.x == 0) s_abort = 0;
  __syncthreads();
  const int64_t passes = (p.nsteps + p.ksteps - 1) / p.ksteps;
  for (int64_t pass = 0; pass < passes; ++pass) {
    const int64_t rem = p.nsteps - pass * p.ksteps;
    const int kp = int(rem < p.ksteps ? rem : p.ksteps);
    const bool to_out = ((passes - 1 - pass) & 1) == 0;
    for (int item = blockIdx.x; item < p.nitems; item += gridDim.x) {
      const int gi = find_grid(p.grids, p.ngrids, item);
      const BatchGrid& bg = p.grids[gi];
      // pass 0 reads in; pass q > 0 reads what pass q-1 wrote
      const T* src = pass == 0 ? static_cast<const T*>(bg.in)
                               : static_cast<const T*>(to_out ? bg.work : bg.out);
      T* dst = static_cast<T*>(to_out ? bg.out : bg.work);
      const int t = item - bg.first_item;
      const int x0 = (t % bg.tiles_x) * p.tile_x, y0 = (t / bg.tiles_x) * p.tile_y;
      TrapGrid tg;
      tg.nx = bg.nx;
      tg.ny = bg.ny;
      for (int a = 0; a < 2; ++a)
        for (int sd = 0; sd < 2; ++sd) {
          tg.bc[a][sd] = bg.bc[a][sd];
          tg.bval[a][sd] = bg.bval[a][sd];
        }
      const T* srcs[1] = {src};
      T* dsts[1] = {dst};
      Tile::template run<Op, T>(op, srcs, dsts, tg, x0, y0, p.tile_x, p.tile_y, kp,
                                reinterpret_cast<C_t<T>*>(smem_raw));
    }
    const bool arrive = !(pass == 0 && int(blockIdx.x) == p.skip_block);
    if (pass + 1 < passes &&
        !grid_sync(p.barrier, unsigned(pass + 1) * gridDim.x, p.err, &s_abort, p.wait_ns, arrive))
      return;
  }
}

// ------------------------------------------------------------------ strips
// FP32 star functions: the register strips (strip_device.cuh) over every grid
// of the batch.  A pass advances every grid by the same depth K (the plan's
// depth, then 4, 2 and 1 for what is left of the sweep count) and is one launch
// with one unit (a strip's chunk of rows of one grid) per warp; the block
// scheduler balances uneven grids.  Rows of any pitch (aligned grids stage
// whole vectors).  A persistent kernel whose warps claimed units from a counter
// kept about 45 registers of its loop alive across the march and spilled it
// (512 grids of sides 64..2048, jacobi5 x20, 5.9e8 points: 9.5 ms, with all
// depths in one kernel 11.6 ms; this form 5.09 ms, the two-sweep shared-memory
// tiles it replaced 12.5 ms).  One kernel holds the marches of aligned and of other
// rows, masked and plain, and at depth 8 still spills some (jacobi5 a 104-byte frame,
// 40 without masks).  A batch with Dirichlet sides mixes masked and
// plain units on an SM: at radius 1 all of them then run on packed pairs, whose
// code is smaller (5.60 ms on scalars, 5.40 with pairs in the masked units only);
// at radius 2 only the masked ones (256 odd grids x16 at depth 4: 3.93 ms, 4.05 on
// scalars, 4.27 all packed).  A batch without Dirichlet sides runs a kernel
// without masks, on scalars.  Bound by instruction issue: 16 grids of 4096^2
// run 3.6e12 updates/s at depth 8; odd widths (element copies and stores)
// and Dirichlet sides (masks) cost a quarter to a third.

// The grid of unit `item`: first[i] is the first unit of grid i (ascending).
// All lanes probe 32 positions of the list at once.
__device__ __forceinline__ int find_grid_warp(const int* first, int n, int item) {
  const int lane = threadIdx.x & 31;
  int lo = 0, len = n;
  while (len > 1) {
    const int step = (len + 31) / 32, i = lane * step;
    const unsigned le = __ballot_sync(0xffffffffu, i < len && first[lo + (i < len ? i : 0)] <= item);
    const int j = (__popc(le) - 1) * step;
    lo += j;
    len = min(step, len - j);
  }
  return lo;
}

// One pass of depth K over the batch; pass 0 reads in, pass q > 0 what pass q-1
// wrote.
template <class Op, int K, bool DIR>
__global__ void __launch_bounds__(32 * kBatchWarps, 4)
    batch_strip_kernel(const __grid_constant__ Op op, const __grid_constant__ BatchPlanDev p,
                       int64_t pass) {
  using G = StripGeom<float, Op::R, K>;
  constexpr int D = strip_depth_index(K);
  constexpr int PM = !DIR ? 0 : Op::R == 1 ? 2 : 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x / 32;
  const int u = blockIdx.x * kBatchWarps + warp;
  if (u >= p.units[D]) return;
  unsigned char* ring = smem_raw + warp * (kBatchRing * G::ROWB);
  const int* first = p.first + size_t(D) * (p.ngrids + 1);
  const int gi = find_grid_warp(first, p.ngrids, u);
  const BatchGrid& b = p.grids[gi];
  const bool to_out = ((p.passes - 1 - pass) & 1) == 0;
  const float* in[1] = {static_cast<const float*>(pass == 0 ? b.in : to_out ? b.work : b.out)};
  float* out[1] = {static_cast<float*>(to_out ? b.out : b.work)};
  StripGrid g;
  g.nx = b.nx;
  g.ny = b.ny;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int sd = 0; sd < 2; ++sd) {
      g.bc[a][sd] = b.bc[a][sd];
      g.bval[a][sd] = b.bval[a][sd];
    }
  const int strips = (g.nx + G::VALID - 1) / G::VALID;
  const int t = u - first[gi], c = t / strips, s = t - c * strips;
  const int y0 = c * p.chunk[D], y1 = min(g.ny, y0 + p.chunk[D]);
  if (g.nx % kStripV == 0)
    Strip<Op, float, K, 1, kBatchRing, true, PM>::template run<DIR>(op, in, out, g, s * G::VALID, y0, y1, ring, nullptr);
  else
    Strip<Op, float, K, 1, kBatchRing, false, PM>::template run<DIR>(op, in, out, g, s * G::VALID, y0, y1, ring, nullptr);
}

// Copy the plan's descriptors from page-locked host memory into the workspace
// and zero its counters.  A kernel, not copy and memset nodes: those belong to
// the allocation that held the workspace when the graph was made, and a replay
// after the caller freed and allocated it again at the same address is invalid.
__global__ void batch_upload_kernel(const uint4* src, uint4* dst, int64_t n16, uint4* counters) {
  const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i < 16) counters[i] = make_uint4(0, 0, 0, 0);
  if (i < n16) dst[i] = src[i];
}

template <class Op, class T, class Tile> struct BatchRunner {
  static cudaError_t prepare(size_t smem) {
    return cudaFuncSetAttribute(&batch_kernel<Op, T, Tile>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(smem));
  }
  static int max_blocks(size_t smem) {
    if (prepare(smem) != cudaSuccess) return 0;
    int occ = 0, dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, &batch_kernel<Op, T, Tile>, kBatchThreads,
                                                      smem) != cudaSuccess)
      return 0;
    return occ * sms;
  }
  static cudaError_t launch(const Op& op, const BatchPlanDev& p, int blocks, size_t smem,
                            cudaStream_t st) {
    cudaError_t e = prepare(smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kBatchThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, &batch_kernel<Op, T, Tile>, op, p);
    count_launches(1);
    return e;
  }
};

template <class T, class F> auto with_op(const StencilDesc& s, F&& f) {
  if (s.kind == kJacobi5) return f(OpJacobi5{s.prm[0]});
  OpStarLinear<2, 1> op;
  for (int ax = 0; ax < 3; ++ax)
    for (int d = 0; d < 3; ++d) op.w[ax][d] = s.star_w[ax][d];
  return f(op);
}

// Run F with the tile policy for (tile_x, tile_y, k): the fixed shapes the
// batch autotuner tries for FP32 storage, else the variable-shape tile.
template <class T, class F>
auto with_tile(int tx, int ty, int k, F&& f) {
  if constexpr (std::is_same<T, float>::value) {
#define LOPE_FIXED(X, Y, KK) \
    if (tx == X && ty == Y && k == KK) return f(TileFixed<X, Y, KK>());
    LOPE_FIXED(128, 32, 4) LOPE_FIXED(128, 32, 2) LOPE_FIXED(64, 32, 4) LOPE_FIXED(64, 32, 2)
    LOPE_FIXED(128, 16, 4) LOPE_FIXED(128, 16, 2) LOPE_FIXED(64, 16, 4) LOPE_FIXED(64, 16, 2)
#undef LOPE_FIXED
  }
  return f(TileAny());
}

template <class Op, int K>
cudaError_t launch_strip_pass(const Op& op, const BatchPlanDev& p, int64_t pass, cudaStream_t st) {
  constexpr size_t SMEM = size_t(kBatchWarps) * kBatchRing * StripGeom<float, Op::R, K>::ROWB;
  const int blocks = (p.units[strip_depth_index(K)] + kBatchWarps - 1) / kBatchWarps;
  if (p.dirichlet) batch_strip_kernel<Op, K, true><<<blocks, 32 * kBatchWarps, SMEM, st>>>(op, p, pass);
  else batch_strip_kernel<Op, K, false><<<blocks, 32 * kBatchWarps, SMEM, st>>>(op, p, pass);
  count_launches(1);
  return cudaGetLastError();
}

template <class Op>
cudaError_t launch_strips(const Op& op, const BatchPlanDev& p, cudaStream_t st) {
  int64_t pass = 0;
  for (int64_t left = p.nsteps; left > 0; ++pass) {
    const int k = strip_next_depth(p.ksteps, left);
    cudaError_t e = cudaErrorNotSupported;
    if constexpr (strip_kmax(1, Op::R, true) >= 8) {
      if (k == 8) e = launch_strip_pass<Op, 8>(op, p, pass, st);
    }
    if (k == 4) e = launch_strip_pass<Op, 4>(op, p, pass, st);
    if (k == 2) e = launch_strip_pass<Op, 2>(op, p, pass, st);
    if (k == 1) e = launch_strip_pass<Op, 1>(op, p, pass, st);
    if (e != cudaSuccess) return e;
    left -= k;
  }
  return cudaSuccess;
}

// Local functions of the batched strips: the 5-point Jacobi, the 9-point
// radius-2 star, and linear star tables of radius 1 or 2.
template <class F> cudaError_t with_strip_op(const StencilDesc& s, F&& f) {
  if (s.kind == kJacobi5) return f(OpJacobi5{s.prm[0]});
  if (s.kind == kStar9r2) return f(OpStar9r2{s.prm[0]});
  if (s.kind == kLinear && s.star && s.ndim == 2 && s.radius == 1) {
    OpStarLinear<2, 1> op;
    for (int ax = 0; ax < 3; ++ax) for (int d = 0; d < 3; ++d) op.w[ax][d] = s.star_w[ax][d];
    return f(op);
  }
  if (s.kind == kLinear && s.star && s.ndim == 2 && s.radius == 2) {
    OpStarLinear<2, 2> op;
    for (int ax = 0; ax < 3; ++ax) for (int d = 0; d < 5; ++d) op.w[ax][d] = s.star_w[ax][d];
    return f(op);
  }
  return cudaErrorNotSupported;
}

template <class T>
cudaError_t launch_t(const BatchPlanDev& p, const StencilDesc& s, int blocks, cudaStream_t st) {
  const size_t smem = trap_smem_bytes(sizeof(T) == 8 ? kF64 : kF32, 1, p.tile_x, p.tile_y,
                                      s.radius * p.ksteps);
  return with_op<T>(s, [&](auto op) {
    return with_tile<T>(p.tile_x, p.tile_y, p.ksteps, [&](auto tile) {
      return BatchRunner<decltype(op), T, decltype(tile)>::launch(op, p, blocks, smem, st);
    });
  });
}

template <class T> int max_blocks_t(const StencilDesc& s, int tx, int ty, int k) {
  const size_t smem = trap_smem_bytes(sizeof(T) == 8 ? kF64 : kF32, 1, tx, ty, s.radius * k);
  return with_op<T>(s, [&](auto op) {
    return with_tile<T>(tx, ty, k, [&](auto tile) {
      return BatchRunner<decltype(op), T, decltype(tile)>::max_blocks(smem);
    });
  });
}

}  // namespace

// Columns a strip of depth k advances (the cut of the batch's grids).
int batch_strip_valid(int radius, int k) {
  const int hl = (k * radius + kStripV - 1) / kStripV;
  return (32 - 2 * hl) * kStripV;
}

cudaError_t launch_batch(const BatchPlanDev& p, const StencilDesc& s, int dtype, int blocks,
                         const void* pinned, size_t bytes, cudaStream_t st) {
  {
    const int64_t n16 = int64_t((bytes + 15) / 16);
    batch_upload_kernel<<<int((std::max<int64_t>(n16, 16) + 255) / 256), 256, 0, st>>>(
        static_cast<const uint4*>(pinned), reinterpret_cast<uint4*>(const_cast<BatchGrid*>(p.grids)), n16,
        reinterpret_cast<uint4*>(p.barrier));
    count_launches(1);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (p.mode == 1) {
    if (dtype != kF32) return cudaErrorNotSupported;
    return with_strip_op(s, [&](auto op) {
      return launch_strips(op, p, st);
    });
  }
  if (!(s.kind == kJacobi5 || (s.kind == kLinear && s.star && s.ndim == 2 && s.radius == 1)))
    return cudaErrorNotSupported;
  switch (dtype) {
    case kF32: return launch_t<float>(p, s, blocks, st);
    case kF64: return launch_t<double>(p, s, blocks, st);
    case kBF16: return launch_t<__nv_bfloat16>(p, s, blocks, st);
    default: return cudaErrorNotSupported;
  }
}

int batch_max_blocks(const StencilDesc& s, int dtype, int tile_x, int tile_y, int ksteps,
                     int mode) {
  if (mode == 1) {
    if (dtype != kF32 || (ksteps != strip_kmax(1, s.radius, true) && ksteps != 4 && ksteps != 2 && ksteps != 1))
      return 0;
    // resident blocks (the units are cut for them; nothing waits on another)
    const cudaError_t e = with_strip_op(s, [](auto) { return cudaSuccess; });
    return e == cudaSuccess ? 4 * device_sms() : 0;
  }
  if (!(s.kind == kJacobi5 || (s.kind == kLinear && s.star && s.ndim == 2 && s.radius == 1)))
    return 0;
  switch (dtype) {
    case kF32: return max_blocks_t<float>(s, tile_x, tile_y, ksteps);
    case kF64: return max_blocks_t<double>(s, tile_x, tile_y, ksteps);
    case kBF16: return max_blocks_t<__nv_bfloat16>(s, tile_x, tile_y, ksteps);
    default: return 0;
  }
}

}  // namespace lope
