"""The grid barrier's verdict is one per block: its code on host threads, with
an error flag that another block sets while the block leaves the barrier."""
from __future__ import annotations

import pytest

from tests import cpp_extract

_PROGRAM = """
#include <atomic>
#include <barrier>
#include <chrono>
#include <cstdio>
#include <thread>
#define __device__
#define __forceinline__ inline
struct Dim { unsigned x; };
static thread_local Dim threadIdx;
static Dim gridDim{2};
static int err = 0, late = 0;
static std::atomic<bool> first_left{false};
static std::barrier<> bar_(2);
static std::atomic<int> any{0};
static thread_local int calls = 0;
static void leave() {   // the second barrier of the call: thread 1 is slow to go on
  if (++calls == 2 && threadIdx.x == 1 && late) {
    while (!first_left) std::this_thread::yield();
    *(volatile int *)&err = 1;   // another block's wait runs out now
  }
}
static void __syncthreads() { bar_.arrive_and_wait(); leave(); }
static int __syncthreads_or(int v) {
  if (v) any = 1;
  bar_.arrive_and_wait();
  leave();
  return any;
}
static void __threadfence() {}
static void __nanosleep(unsigned) { std::this_thread::yield(); }
static unsigned atomicAdd(unsigned *p, unsigned v) { unsigned o = *p; *p += v; return o; }
template <typename T> static T atomicExch(T *p, T v) { T o = *p; *p = v; return o; }
static unsigned long long gtime() {
  return (unsigned long long)std::chrono::steady_clock::now().time_since_epoch().count();
}
%s
int main() {
  unsigned bar[2] = {%d, 0};   // 1: every other block has arrived; 0: the wait runs out
  late = %d;
  err = %d;
  bool ok[2];
  std::thread t[2];
  for (unsigned i = 0; i < 2; ++i)
    t[i] = std::thread([&, i] {
      threadIdx.x = i;
      ok[i] = grid_barrier(bar, &err, 1000);
      if (i == 0) first_left = true;
    });
  for (auto &x : t) x.join();
  std::printf("%%d%%d %%d", ok[0], ok[1], err);
}
"""


@pytest.mark.parametrize("arrived,late,err,want", [
    (1, 0, 0, "11 0"),   # released
    (1, 1, 0, "11 1"),   # released; the flag is set between the threads' returns
    (0, 0, 0, "00 1"),   # the wait runs out
    (1, 0, 1, "00 1"),   # the flag was set before
])
def test_verdict_is_uniform(tmp_path, arrived, late, err, want):
    body = cpp_extract.function("qisg_internal.cuh", "__device__ __forceinline__ bool grid_barrier(")
    assert cpp_extract.run(tmp_path, _PROGRAM % (body, arrived, late, err)) == want
