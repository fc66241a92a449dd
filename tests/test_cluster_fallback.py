"""Launches in clusters on a device that cannot hold them (a partition with few SMs together): the
selection and the Gram fall back to forms that it holds.  The launchers' own text is compiled for the
host against a fake runtime whose largest cluster the test sets."""
import ctypes
import os
import subprocess

import pytest

from paper_2605_31105_gb300 import build as build_mod
from tests.host_block import _slice

HARNESS = r"""
#include <cuda_runtime_api.h>
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <utility>
#define __host__
#define __device__
static int largest, launched, cluster_used, grid_used, kernel_used;
static int cluster_of(const cudaLaunchConfig_t* c) {
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return c->attrs[i].val.clusterDim.x;
  return 1;
}
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
template <class... P>
cudaError_t cudaFuncSetAttribute(void (*)(P...), cudaFuncAttribute, int) { return cudaSuccess; }
template <class... P>
cudaError_t cudaOccupancyMaxActiveClusters(int* n, void (*)(P...), const cudaLaunchConfig_t* c) {
  *n = cluster_of(c) <= largest ? 1 : 0;
  return cudaSuccess;
}
template <class... P, class... A>
cudaError_t cudaLaunchKernelEx(const cudaLaunchConfig_t* c, void (*k)(P...), A&&...);
namespace grkv {
struct WsLayout { size_t pooled; };
static void count_launches(int) {}
struct Shape { int U, P, pool_k; bool chained; };
%(launch)s
%(sizes)s
template <int kPer, int kCs> void k_select_reg(const float*, Shape, int32_t*) {}
void k_select(const float*, Shape, float*, int32_t*) {}
%(select)s
constexpr int kTile = 128, kClusterSms = 128, kThreadsG = 640, kSmemBytes = 230000;
struct CUtensorMap {};
struct MArgs { int U, nrb, B, ranks; };
static int ranks_used;
void k_merge_gram(const CUtensorMap, MArgs) {}
%(gram)s
}
using namespace grkv;
static void note(const MArgs& a) { ranks_used = a.ranks; }
template <class T> static void note(const T&) {}
template <class... P, class... A>
cudaError_t cudaLaunchKernelEx(const cudaLaunchConfig_t* c, void (*k)(P...), A&&... args) {
  cluster_used = cluster_of(c);
  if (cluster_used > largest) return cudaErrorInvalidClusterSize;
  ++launched;
  grid_used = c->gridDim.x;
  kernel_used = (const void*)k == (const void*)k_select;
  (note(args), ...);
  return cudaSuccess;
}
// cluster size, grid and (selection) 1 for the kernel over the pooled copy; the launch's error
extern "C" int select_launch(int U, int P, int pool, int limit, int* out) {
  largest = limit;
  launched = 0;
  Shape s{U, P, pool, false};
  const int rc = launch_select_pooled(s, nullptr, nullptr, nullptr, 0);
  out[0] = cluster_used, out[1] = grid_used, out[2] = kernel_used, out[3] = launched;
  return rc;
}
extern "C" int gram_launch(int U, int nrb, int B, int limit, int* out) {
  largest = limit;
  launched = 0;
  const int rc = launch_gram(CUtensorMap{}, MArgs{U, nrb, B, 0}, 0);
  out[0] = cluster_used, out[1] = grid_used, out[2] = ranks_used, out[3] = launched;
  return rc;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    def text(name):
        with open(os.path.join(build_mod.CSRC, name)) as f:
            return f.read()

    tmp = str(tmp_path_factory.mktemp("cluster"))
    common, sel, mrg = (text(f) for f in ("grkv_internal.cuh", "grkv_select.cu", "grkv_merge_tc.cu"))
    code = HARNESS % {
        "launch": _slice(common, "// chained: the work before this launch",
                         "// Byte offsets of the workspace"),
        "sizes": _slice(sel, "constexpr int kThr = 1024", "__device__ __forceinline__ uint32_t peer_addr"),
        "select": _slice(sel, "template <int kPer, int kCs>\ncudaError_t launch_reg",
                         "cudaError_t launch_select(const Shape").replace("}  // namespace\n", ""),
        "gram": _slice(mrg, "cudaError_t launch_gram(", "size_t merge_tc_ws_bytes(const Shape& s) {"),
    }
    src, so = os.path.join(tmp, "launch.cpp"), os.path.join(tmp, "launch.so")
    with open(src, "w") as f:
        f.write(code)
    cuda = os.path.dirname(os.path.dirname(build_mod.nvcc()))
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-w", "-I",
                    os.path.join(cuda, "include"), "-o", so, src], check=True)
    return ctypes.CDLL(so)


def _run(fn, *args):
    out = (ctypes.c_int * 4)()
    assert fn(*args, out) == 0, "the launch failed"
    assert out[3] == 1
    return tuple(out)[:3]


@pytest.mark.parametrize("P", [32769, 65536, 131072, 262144])
def test_selection(lib, P):
    assert _run(lib.select_launch, 5, P, 7, 8) == (8, 40, 0)
    for limit in (1, 2, 4):
        assert _run(lib.select_launch, 5, P, 7, limit) == (1, 5, 1)
    assert _run(lib.select_launch, 5, 32768, 7, 1) == (1, 5, 0)   # one CTA: no cluster


def test_gram(lib):
    for limit, ranks in ((8, 8), (4, 4), (2, 2), (1, 1)):
        assert _run(lib.gram_launch, 2, 1, 4096, limit) == (ranks, 2 * ranks, ranks)
    assert _run(lib.gram_launch, 33, 1, 520, 8) == (2, 66, 2)   # 66 of 128 SMs, 132 with four ranks
    assert _run(lib.gram_launch, 2, 2, 300, 8) == (2, 8, 2)     # three tiles
