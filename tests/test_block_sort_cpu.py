"""The block-wide sort of block_sort.cuh, run on host threads.

Each CUDA thread is a host thread; __syncthreads and the warp shuffle are
barriers, and one warp at a time is held back after every block barrier, so
that an exchange that is not ordered by a barrier goes wrong every time.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_07265_gb300", "csrc")

HOST = r"""
#include <algorithm>
#include <barrier>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <memory>
#include <random>
#include <thread>
#include <vector>

#define __device__
#define __forceinline__ inline

struct Dim { int x; };
thread_local Dim threadIdx;
thread_local int n_sync;
int slow_warp, skip_sync;   // the block barrier of this number is left out (-1: none)
std::unique_ptr<std::barrier<>> block;
std::vector<std::unique_ptr<std::barrier<>>> warps;
std::vector<unsigned long long> lanes;

void __syncthreads() {
  if (n_sync++ == skip_sync) return;
  block->arrive_and_wait();
  if (threadIdx.x / 32 == slow_warp) std::this_thread::sleep_for(std::chrono::milliseconds(4));
}

unsigned long long __shfl_xor_sync(unsigned, unsigned long long v, int j) {
  auto &b = *warps[threadIdx.x / 32];
  lanes[threadIdx.x] = v;
  b.arrive_and_wait();
  const unsigned long long o = lanes[threadIdx.x ^ j];
  b.arrive_and_wait();
  return o;
}

#include "block_sort.cuh"

int main(int argc, char **argv) {
  const int n = std::atoi(argv[1]), threads = std::atoi(argv[2]);
  const bool leave_out = std::atoi(argv[3]) != 0;
  int live = 32;               // the threads that the sort covers
  while (live < n) live *= 2;
  int bad = 0, syncs = 0;
  for (slow_warp = 0; slow_warp < threads / 32; ++slow_warp) {
    // The barrier before the sorted values are stored is the last but one.
    skip_sync = leave_out ? std::atoi(argv[3]) - 2 : -1;
    std::mt19937_64 rng(n);
    std::vector<unsigned long long> in(threads), out(threads), left(threads), buf(threads);
    for (int i = 0; i < threads; ++i) in[i] = i < n ? rng() | 1 : 0;
    block = std::make_unique<std::barrier<>>(threads);
    warps.clear();
    for (int w = 0; w < threads / 32; ++w) warps.push_back(std::make_unique<std::barrier<>>(32));
    lanes.assign(threads, 0);
    std::vector<std::thread> pool;
    for (int t = 0; t < threads; ++t)
      pool.emplace_back([&, t] {
        threadIdx.x = t;
        n_sync = 0;
        out[t] = xs::block_sort_desc(in[t], n, buf.data());
        left[t] = buf[t ^ 1];
        if (t == 0) syncs = n_sync;
      });
    for (auto &t : pool) t.join();
    std::sort(in.begin(), in.begin() + live, std::greater<>());
    for (int i = 0; i < live; ++i) bad += out[i] != in[i] || left[i] != in[i ^ 1];
  }
  std::printf("%d barriers, %d wrong\n", syncs, bad);
  return bad != 0;
}
"""


@pytest.fixture(scope="module")
def sort(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("block_sort")
    (d / "sort.cpp").write_text(HOST)
    exe = d / "sort"
    subprocess.run(["g++", "-O1", "-std=c++20", "-pthread", "-I" + CSRC, str(d / "sort.cpp"), "-o", str(exe)],
                   check=True)

    def run(n, threads, barriers=0):
        return subprocess.run([str(exe), str(n), str(threads), str(barriers)], capture_output=True, text=True,
                              timeout=120)
    return run


@pytest.mark.parametrize("n,threads", [(1, 64), (32, 64), (33, 64), (64, 64), (65, 128), (100, 128), (128, 256)])
def test_sorted_whatever_warp_is_late(sort, n, threads):
    r = sort(n, threads)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("n", [64, 128])
def test_a_missing_barrier_before_the_store_is_found(sort, n):
    barriers = int(sort(n, n).stdout.split()[0])
    r = sort(n, n, barriers)   # the last but one of them left out
    assert r.returncode == 1 and ", 0 wrong" not in r.stdout
