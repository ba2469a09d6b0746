"""Several devices of one process, without a GPU.

A kernel that needs more than 48 KB of shared memory is opted in per device.
The library's own object files are linked with a stand-in for the CUDA runtime
that has two devices, keeps the opt-ins of each, and refuses a launch whose
kernel lacks one on the current device, as the runtime does.
"""
import os
import subprocess

import pytest

HARNESS = r"""
#include <map>
#include <cstdio>
#include <cstring>
#include "lope_internal.h"
#include <cuda.h>

static int g_dev = 0, g_launches = 0, g_refused = 0;
static std::map<std::pair<int, const void*>, size_t> g_opt;
static dim3 g_grid, g_block; static size_t g_smem; static cudaStream_t g_stream;

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) { g_opt[{g_dev, f}] = size_t(v); return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetLastError() { return g_refused ? cudaErrorInvalidValue : cudaSuccess; }
static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                       const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q) {
  *p = reinterpret_cast<void*>(&encode); *q = cudaDriverEntryPointSuccess; return cudaSuccess;
}
// what the compiler's launch stubs call
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, cudaStream_t st) { g_grid = g; g_block = b; g_smem = s; g_stream = st; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = g_grid; *b = g_block; *s = g_smem; *static_cast<cudaStream_t*>(st) = g_stream; return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f)); return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t) {
  ++g_launches;
  auto it = g_opt.find({g_dev, reinterpret_cast<const void*>(k)});
  if (smem > 48 * 1024 && (it == g_opt.end() || it->second < smem)) { ++g_refused; return cudaErrorInvalidValue; }
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
}

namespace lope {
void count_launches(int64_t) {}
bool has_external(const Geom&) { return false; }
cudaError_t jit_launch(const StepArgs&, int) { return cudaErrorNotSupported; }
bool jit_tma_ok(const JitProgram*) { return false; }
cudaError_t launch_strip_swe(const StepArgs& a);
}

using namespace lope;
static StepArgs args(int ndim, int64_t nz, int64_t ny, int64_t nx, int kind, int nf, int stages, int k) {
  StepArgs a;
  std::memset(&a, 0, sizeof(a));
  a.g.ndim = a.s.ndim = ndim;
  a.g.n[0] = nz; a.g.n[1] = ny; a.g.n[2] = nx;
  a.g.dtype = kF32; a.g.nf = nf;
  a.s.kind = kind; a.s.radius = 1; a.s.stages = stages; a.s.star = kind != kSweFlux;
  for (int f = 0; f < nf; ++f) { a.in[f] = reinterpret_cast<void*>(0x10000); a.out[f] = reinterpret_cast<void*>(0x20000); }
  a.ksteps = k;
  return a;
}
int main() {
  int bad = 0;
  for (g_dev = 0; g_dev < 2; ++g_dev) {
    bad += launch_brick(args(3, 64, 256, 256, kDiff7, 1, 1, 4)) != cudaSuccess;
    bad += launch_strip_swe(args(2, 1, 512, 512, kSwe, 3, 3, 1)) != cudaSuccess;
    bad += launch_tma(args(3, 64, 256, 256, kDiff7, 1, 1, 1), nullptr) != cudaSuccess;
    bad += launch_tma(args(2, 1, 512, 512, kSwe, 3, 1, 1), nullptr) != cudaSuccess;
  }
  std::printf("launches %d refused %d failed %d\n", g_launches, g_refused, bad);
  return bad;
}
"""


def test_kernels_are_opted_in_on_every_device(lope, tmp_path):
    from paper_1502_03504_gb300 import build as B

    objs = []
    for name in ("k_brick", "k_strip_swe", "k_tma"):
        obj = os.path.join(B.BUILD, name + ".o")
        if not os.path.exists(obj):
            pytest.skip("the library was built without its object files")
        objs.append(obj)
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    inc = os.path.join(os.path.dirname(os.path.dirname(B.nvcc())), "include")
    cmd = ["g++", "-std=c++17", "-O1", "-I", B.CSRC, "-I", B.INCLUDE, "-I", inc, str(src), *objs, "-o", str(exe),
           "-lpthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and "launches 8 refused 0 failed 0" in r.stdout, r.stdout + r.stderr
