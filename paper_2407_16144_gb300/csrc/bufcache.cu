// The cache of device buffers (see bufcache.h).  Host code only.
#include "bufcache.h"

#include <algorithm>
#include <cstdint>
#include <map>
#include <mutex>
#include <unordered_map>
#include <utility>
#include <vector>

namespace rh {

namespace {
// Cached buffers are keyed by (device, size): a buffer is only ever reused on the device it was
// allocated on.  Buffers from a caller's allocator carry it (hook.free set) and are never cached.
struct BufInfo {
  int dev;
  size_t bytes;
  DevAllocator hook;
};
using Key = std::pair<int, size_t>;          // device, size
struct Cached {
  void *p;
  unsigned long long release;                // the release that brought it
};
using Freed = std::vector<std::pair<int, void *>>;   // buffers to free: device, pointer

thread_local const DevAllocator *tl_alloc = nullptr;   // set by AllocScope
std::mutex g_mu;
std::unordered_map<void *, BufInfo> g_info;            // every buffer from buf_alloc
std::map<Key, std::vector<Cached>> g_free;             // the cache, each size oldest first
std::map<unsigned long long, Key> g_by_release;        // the same buffers, oldest first
size_t g_free_bytes = 0;
unsigned long long g_releases = 0;

// Takes the cached buffers that were released longest ago out of the cache until `bytes` more fit;
// the caller holds g_mu, and frees them once it has given it up: cudaFree waits for the device, and
// every other thread's create and free would wait with it.  (Refusing the newcomer instead made every
// call that followed a larger handle allocate and free its scratch again: a KKT evaluation of a
// 30M-entry LP 640 us instead of 464.)
void unlink_oldest(size_t bytes, Freed *out) {
  while (!g_by_release.empty() && g_free_bytes + bytes > kBufferCacheBytes) {
    const Key key = g_by_release.begin()->second;
    auto it = g_free.find(key);
    void *p = it->second.front().p;          // its size's oldest is the oldest of all
    it->second.erase(it->second.begin());
    if (it->second.empty()) g_free.erase(it);
    g_by_release.erase(g_by_release.begin());
    g_free_bytes -= key.second;
    g_info.erase(p);
    out->push_back({key.first, p});
  }
}

// Frees buffers on their own devices; the caller does not hold g_mu.
void free_all(const Freed &bufs) {
  if (bufs.empty()) return;
  int cur = -1;
  cudaGetDevice(&cur);
  for (const auto &b : bufs) {
    cudaSetDevice(b.first);
    cudaFree(b.second);
  }
  if (cur >= 0) cudaSetDevice(cur);
}
}  // namespace

AllocScope::AllocScope(const DevAllocator &a) : prev_(tl_alloc), mine_(a) {
  tl_alloc = (mine_.alloc && mine_.free) ? &mine_ : nullptr;
}
AllocScope::~AllocScope() { tl_alloc = prev_; }

cudaError_t buf_alloc(void **p, size_t bytes) {
  bytes = std::max<size_t>(bytes, 1);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (tl_alloc) {
    // 256-byte alignment covers every vector load of the kernels
    void *q = tl_alloc->alloc(bytes, tl_alloc->stream, tl_alloc->ctx);
    if (!q) return cudaErrorMemoryAllocation;
    if (reinterpret_cast<uintptr_t>(q) % 256 != 0) {
      tl_alloc->free(q, tl_alloc->stream, tl_alloc->ctx);
      return cudaErrorInvalidValue;
    }
    *p = q;
    std::lock_guard<std::mutex> lk(g_mu);
    g_info[q] = BufInfo{dev, bytes, *tl_alloc};
    return cudaSuccess;
  }
  {
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_free.find({dev, bytes});
    if (it != g_free.end()) {
      *p = it->second.back().p;
      g_by_release.erase(it->second.back().release);
      it->second.pop_back();
      if (it->second.empty()) g_free.erase(it);
      g_free_bytes -= bytes;
      return cudaSuccess;
    }
  }
  e = cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    buf_drop_cache();
    e = cudaMalloc(p, bytes);
  }
  if (e == cudaSuccess) {
    std::lock_guard<std::mutex> lk(g_mu);
    g_info[*p] = BufInfo{dev, bytes, DevAllocator()};
  }
  return e;
}

void buf_release(void *p) {
  if (!p) return;
  Freed old;
  {
    std::unique_lock<std::mutex> lk(g_mu);
    auto it = g_info.find(p);
    if (it != g_info.end()) {
      const BufInfo bi = it->second;
      if (bi.hook.free) {
        g_info.erase(it);
        lk.unlock();
        bi.hook.free(p, bi.hook.stream, bi.hook.ctx);
        return;
      }
      if (bi.bytes <= kBufferCacheBytes) {
        unlink_oldest(bi.bytes, &old);
        g_free[{bi.dev, bi.bytes}].push_back({p, g_releases});
        g_by_release[g_releases++] = {bi.dev, bi.bytes};
        g_free_bytes += bi.bytes;
        lk.unlock();
        free_all(old);
        return;
      }
      g_info.erase(it);
    }
  }
  cudaFree(p);
}

size_t buf_drop_cache() {
  Freed all;
  size_t freed = 0;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    freed = g_free_bytes;
    for (auto &kv : g_free)
      for (const Cached &b : kv.second) {
        g_info.erase(b.p);
        all.push_back({kv.first.first, b.p});
      }
    g_free.clear();
    g_by_release.clear();
    g_free_bytes = 0;
  }
  free_all(all);
  return freed;
}

}  // namespace rh
