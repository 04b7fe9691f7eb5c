"""The cache of device buffers (csrc/bufcache.cu) over fakes of the five runtime calls it makes: past
its limit it gives back the buffers released longest ago, it hands out the latest of a size, and no
thread waits in it while another frees (cudaFree waits for the device)."""
import os
import shutil
import subprocess

import pytest

from paper_2407_16144_gb300 import _build

pytestmark = pytest.mark.skipif(shutil.which("g++") is None or
                                (shutil.which("nvcc") is None and
                                 not os.path.exists("/usr/local/cuda/bin/nvcc")),
                                reason="no compiler or CUDA headers")

PROGRAM = r"""
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <thread>
#include <vector>
#include "bufcache.h"

static std::mutex mu;
static std::condition_variable cv;
static std::vector<long> freed;                   // in the order of the calls
static long next_ptr = 1;
static bool hold = false, in_free = false, let_go = false, timed_out = false;
static int mallocs = 0, fail_mallocs = 0;

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t) {
  std::lock_guard<std::mutex> lk(mu);
  ++mallocs;
  if (fail_mallocs > 0) { --fail_mallocs; return cudaErrorMemoryAllocation; }
  *p = (void *)(next_ptr++ << 8);
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  std::unique_lock<std::mutex> lk(mu);
  freed.push_back((long)p >> 8);
  in_free = true;
  cv.notify_all();
  if (hold && !cv.wait_for(lk, std::chrono::seconds(5), [] { return let_go; })) timed_out = true;
  return cudaSuccess;
}
}

#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); std::exit(1); } } while (0)
constexpr size_t GiB = size_t(1) << 30;
static void *get(size_t bytes) {
  void *p = nullptr;
  CHECK(rh::buf_alloc(&p, bytes) == cudaSuccess);
  return p;
}

static void order() {
  void *a[6];
  const size_t sizes[6] = {GiB, GiB, GiB / 2, GiB, GiB / 2, GiB};
  for (int i = 0; i < 6; ++i) a[i] = get(sizes[i]);            // buffers 1 to 6
  for (int i = 0; i < 5; ++i) rh::buf_release(a[i]);           // 4 GiB: full
  CHECK(freed.empty());
  rh::buf_release(a[5]);                                       // one has to go: the first
  CHECK(freed == std::vector<long>({1}));
  CHECK(get(GiB) == a[5] && get(GiB) == a[3] && get(GiB) == a[1]);   // the latest of its size
  void *n = get(GiB);
  CHECK(mallocs == 7);
  CHECK(get(GiB / 2) == a[4]);
  rh::buf_release(a[4]);
  rh::buf_release(n);                                          // 2 GiB cached: 3, 5, n
  void *big = get(3 * GiB);
  rh::buf_release(big);                                        // evicts 3 and 5, in that order
  CHECK(freed == std::vector<long>({1, 3, 5}));
  void *huge = get(5 * GiB);
  rh::buf_release(huge);                                       // over the limit by itself
  CHECK(freed.back() == ((long)huge >> 8));
  fail_mallocs = 1;                                            // out of memory: cache dropped
  CHECK(get(7) != nullptr);
  CHECK(freed.size() == 6);
  CHECK(rh::buf_drop_cache() == 0);
  for (void *p : {a[5], a[3], a[1]}) rh::buf_release(p);
  CHECK(rh::buf_drop_cache() == 3 * GiB && rh::buf_drop_cache() == 0);
}

// Another thread allocates and releases while a full cache's eviction (or a drop) is in cudaFree.
static void no_waiting(bool drop) {
  void *small = get(100), *small2 = get(100);
  std::vector<void *> a;
  for (int i = 0; i < 5; ++i) a.push_back(get(GiB - 1024));
  rh::buf_release(small);
  for (int i = 0; i < 4; ++i) rh::buf_release(a[i]);
  CHECK(get(100) == small);
  hold = true;
  std::thread t([&] { if (drop) rh::buf_drop_cache(); else rh::buf_release(a[4]); });
  {
    std::unique_lock<std::mutex> lk(mu);
    CHECK(cv.wait_for(lk, std::chrono::seconds(5), [] { return in_free; }));
  }
  rh::buf_release(small2);
  CHECK(get(100) == small2);
  {
    std::lock_guard<std::mutex> lk(mu);
    let_go = true;
  }
  cv.notify_all();
  t.join();
  CHECK(!timed_out);
}

int main(int, char **argv) {
  if (!std::strcmp(argv[1], "order")) order();
  else no_waiting(!std::strcmp(argv[1], "drop"));
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("bufcache")
    src, exe = d / "main.cpp", d / "main"
    src.write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", cuda, "-I", _build.CSRC, "-x", "c++",
                    str(src), os.path.join(_build.CSRC, "bufcache.cu"), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("what", ["order", "evict", "drop"])
def test_buffer_cache(program, what):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
