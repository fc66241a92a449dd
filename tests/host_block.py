"""Runs blocks of the fp32 solve's kernels (grkv_simt_merge.cu) on the host.

The kernels' own text is compiled as C++ with every thread a fiber that runs until its
next block barrier.  Barriers are the only points where threads change over, so the order in
which the fibers run between two barriers is the test's choice: code that leaves two threads'
accesses to a word unordered gives other results in another order.  A barrier that some
threads wait at and others have left the kernel before is reported.
"""
import ctypes
import os
import re
import subprocess

import numpy as np

from paper_2605_31105_gb300 import build as build_mod

SRC = os.path.join(build_mod.CSRC, "grkv_simt_merge.cu")

HARNESS = r"""
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <ucontext.h>
#include <vector>
#define __device__
#define __global__
#define __forceinline__ inline
#define __restrict__
#define __shared__
#define __align__(n) __attribute__((aligned(n)))
#define __launch_bounds__(...)
using std::isfinite;
struct uint3_ { unsigned x; };
static uint3_ threadIdx, blockIdx;
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
static void chain_wait() {}

struct Fiber { ucontext_t ctx; std::vector<char> stack; bool done; int pred; };
static std::vector<Fiber> fibers;
static ucontext_t scheduler;
static int current, or_result;
static void (*body)();
static int __syncthreads_or(int p) {
  fibers[current].pred = p;
  swapcontext(&fibers[current].ctx, &scheduler);
  return or_result;
}
static void __syncthreads() { __syncthreads_or(0); }
static void entry() {
  body();
  fibers[current].done = true;
  swapcontext(&fibers[current].ctx, &scheduler);
}
// 0, or -1: a barrier that not all threads reached.  before(i) runs ahead of the i-th turn.
static int run_block(int threads, unsigned block, bool descending, void (*kernel)(),
                     void (*before)(int)) {
  body = kernel;
  blockIdx.x = block;
  fibers.assign(threads, Fiber());
  for (auto& f : fibers) {
    f.stack.resize(1 << 16);
    getcontext(&f.ctx);
    f.ctx.uc_stack.ss_sp = f.stack.data();
    f.ctx.uc_stack.ss_size = f.stack.size();
    f.ctx.uc_link = nullptr;
    makecontext(&f.ctx, entry, 0);
  }
  for (int turn = 0;;) {
    int done = 0;
    for (int i = 0; i < threads; ++i) {
      current = descending ? threads - 1 - i : i;
      threadIdx.x = current;
      fibers[current].pred = 0;
      if (before) before(turn++);
      swapcontext(&scheduler, &fibers[current].ctx);
      done += fibers[current].done;
    }
    if (done == threads) return 0;
    if (done) return -1;
    or_result = 0;
    for (auto& f : fibers) or_result |= f.pred;
  }
}

constexpr int kD = 128;
struct Shape { int m; };
struct SArgs { Shape s; int* state; };
alignas(16) float sm[1 << 16];
"""

ENTRY = r"""
static SArgs g_args;
static Df *g_gram, *g_rz;
extern "C" int run_chol(int m, int descending, double* gram, int* state) {
  std::vector<Df> n((size_t)m * m);
  for (size_t i = 0; i < n.size(); ++i) n[i] = {(float)gram[i], (float)(gram[i] - (float)gram[i])};
  g_args = {{m}, state};
  g_gram = n.data();
  const int rc = run_block(kChT, 0, descending, [] { k_simt_chol(g_args, g_gram); }, nullptr);
  for (size_t i = 0; i < n.size(); ++i) gram[i] = (double)n[i].hi + n[i].lo;
  return rc;
}
// Every block of one unit; turn `flip` of the first block finds the unit given to fp64 by another.
static int g_flip;
extern "C" int run_subst(int m, int descending, const double* factor, double* rz, int* state,
                         int flip) {
  std::vector<Df> n((size_t)m * m), r((size_t)m * kD);
  for (size_t i = 0; i < n.size(); ++i) n[i] = {(float)factor[i], (float)(factor[i] - (float)factor[i])};
  for (size_t i = 0; i < r.size(); ++i) r[i] = {(float)rz[i], (float)(rz[i] - (float)rz[i])};
  g_args = {{m}, state};
  g_gram = n.data();
  g_rz = r.data();
  g_flip = flip;
  int rc = 0;
  for (int b = 0; b < kD / 8; ++b)
    rc |= run_block(256, b, descending, [] { k_simt_subst(g_args, g_gram, g_rz); },
                    b == 0 && flip >= 0 ? [](int turn) { if (turn == g_flip) *g_args.state = kNeeds64; }
                                        : (void (*)(int))nullptr);
  for (size_t i = 0; i < r.size(); ++i) rz[i] = (double)r[i].hi + r[i].lo;
  return rc;
}
"""


def _slice(text, first, last):
    a, z = text.find(first), text.find(last)
    assert 0 <= a < z, f"the source no longer holds {first!r} before {last!r}"
    return text[a:z]


def load(tmp):
    """The compiled harness, built in the directory `tmp`."""
    with open(SRC) as f:
        text = f.read()
    code = (HARNESS + _slice(text, "struct alignas(8) Df {", "// Accumulator policies")
            + _slice(text, "// State of a unit's solve", "struct SArgs {")
            + _slice(text, "constexpr int kChT", "// Units left to fp64") + ENTRY)
    code = re.sub(r"#pragma unroll.*", "", code)
    src, lib = os.path.join(tmp, "block.cpp"), os.path.join(tmp, "block.so")
    with open(src, "w") as f:
        f.write(code)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", "-w",
                    "-o", lib, src], check=True)
    return ctypes.CDLL(lib)


def chol(lib, n, descending):
    """The factor that k_simt_chol leaves of the m x m matrix n, and the unit's state."""
    a, state = np.array(n, dtype=np.float64, order="C"), ctypes.c_int(0)
    rc = lib.run_chol(len(a), int(descending), a.ctypes.data_as(ctypes.c_void_p),
                      ctypes.byref(state))
    assert rc == 0, "threads of the block leave while others wait at a barrier"
    return a, state.value


def subst(lib, factor, r, descending, flip=-1):
    """Z of the residuals r [m][128] given k_simt_chol's factor, and the unit's state.  flip: the
    turn (a thread's run up to its next barrier) before which another block gives the unit to fp64."""
    f = np.array(factor, dtype=np.float64, order="C")
    z, state = np.array(r, dtype=np.float64, order="C"), ctypes.c_int(0)
    rc = lib.run_subst(len(f), int(descending), f.ctypes.data_as(ctypes.c_void_p),
                       z.ctypes.data_as(ctypes.c_void_p), ctypes.byref(state), flip)
    assert rc == 0, "threads of the block leave while others wait at a barrier"
    return z, state.value
