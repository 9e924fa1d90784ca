"""The block sums of the Wilson kernels (hp_reduce.cuh), compiled for the host and run thread by thread.

A CUDA block promises no order between its warps except at barriers.  The harness runs every warp as far as it can get before
it looks at the next one, in a given order: with the last warps first, a warp that does not wait has stored its
sums of the next call before warp 0 has read those of this one.  Sums of small integers, so every order gives the
same bits.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1302_4018_gb300", "csrc")

HARNESS = r"""
#include <ucontext.h>
#include <cstdio>
#include <cstdlib>
#include <vector>
#define __device__
#define __forceinline__ inline
#define __shared__ static
struct Dim { int x, y, z; };
static Dim threadIdx, blockIdx;
constexpr int NT = 128;
struct Fiber { ucontext_t c; std::vector<char> stack; int block_bars = 0, warp_bars = 0; bool done = false; };
static Fiber fib[NT];
static ucontext_t sched;
static int self;
static double lane_value[NT];
static void yield() { const int me = self; swapcontext(&fib[me].c, &sched); self = me; threadIdx.x = me; }
static void wait(int Fiber::*count, int first, int n) {
  const int mine = ++(fib[self].*count);
  for (;;) {
    bool all = true;
    for (int i = first; i < first + n; ++i) all = all && (fib[i].done || fib[i].*count >= mine);
    if (all) return;
    yield();
  }
}
static void __syncthreads() { wait(&Fiber::block_bars, 0, NT); }
template <typename T> static T __shfl_down_sync(unsigned, T v, int o) {
  const int w = self & ~31, lane = self & 31;
  lane_value[self] = (double)v;
  wait(&Fiber::warp_bars, w, 32);
  const T r = (T)lane_value[lane + o < 32 ? self + o : self];
  wait(&Fiber::warp_bars, w, 32);
  return r;
}
#include "hp_reduce.cuh"
constexpr int CALLS = 5, NQ = 3;
static double part[CALLS][NQ];
template <typename R> static void block() {   // a masked kernel: one call per slot
  for (int k = 0; k < CALLS; ++k) {
    R v[NQ];
    for (int q = 0; q < NQ; ++q) v[q] = (R)((self + 1) * (k + 1) + q);
    reduce_partials<R, NQ, NT>(v, part[k], 1);
  }
  fib[self].done = true;
  for (;;) yield();
}
template <typename R> static int run(const int (&order)[4]) {
  for (int i = 0; i < NT; ++i) {
    fib[i].stack.resize(65536);
    fib[i].block_bars = fib[i].warp_bars = 0;
    fib[i].done = false;
    getcontext(&fib[i].c);
    fib[i].c.uc_stack.ss_sp = fib[i].stack.data();
    fib[i].c.uc_stack.ss_size = fib[i].stack.size();
    makecontext(&fib[i].c, (void (*)())block<R>, 0);
  }
  for (int left = NT; left;) {
    for (int w : order)
      for (int pass = 0; pass < 64; ++pass)   // more than a call's warp-level steps: as far as the warp gets
        for (int i = 32 * w; i < 32 * w + 32; ++i)
          if (!fib[i].done) { self = threadIdx.x = i; swapcontext(&sched, &fib[i].c); }
    left = 0;
    for (int i = 0; i < NT; ++i) left += !fib[i].done;
  }
  int bad = 0;
  for (int k = 0; k < CALLS; ++k)
    for (int q = 0; q < NQ; ++q) bad += part[k][q] != (double)(k + 1) * NT * (NT + 1) / 2 + (double)q * NT;
  return bad;
}
int main() {
  const int orders[3][4] = {{0, 1, 2, 3}, {3, 2, 1, 0}, {2, 0, 3, 1}};
  int bad = 0;
  for (auto& o : orders) bad += run<float>(o) + run<double>(o);
  std::printf("%d wrong sums\n", bad);
  return bad != 0;
}
"""


def test_block_sums_once_per_slot_in_any_order_of_warps(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "block.cpp", tmp_path / "block"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
