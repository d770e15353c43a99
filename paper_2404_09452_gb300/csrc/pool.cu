// Per-device cache of released device blocks.  A request takes the smallest cached
// block that holds it and is at most an eighth larger (molecules of one size
// differ by a few per cent in what screening keeps, so a new one finds the blocks
// of the last one).  The cache holds at most DFJK_CACHE_BYTES (environment, default
// 96 GiB) per device: beyond that the blocks released longest ago are freed, so
// that the blocks in use from call to call stay.  (Freeing the block being
// released instead made every later call allocate anew once the cache was full of
// other molecules' blocks: 0.5 to 7 ms a call in cudaMalloc and cudaFree.)  An
// allocation that fails first empties the cache and retries.
#include <cstdlib>
#include <map>
#include <mutex>
#include <string>
#include <unordered_map>

#include "common.cuh"
#include "pool.cuh"

namespace dfjk {

namespace {
struct DevCache {
  struct Block {
    void *p;
    uint64_t when;  // order of release
  };
  std::multimap<size_t, Block> blocks;                                     // by size
  std::map<uint64_t, std::multimap<size_t, Block>::iterator> by_time;      // oldest first
  std::unordered_map<void *, size_t> size_of;                              // every block handed out or cached
  size_t bytes = 0;
  size_t used = 0, peak = 0;  // bytes handed out, and the most since dfjk_debug_pool_peak
  uint64_t clock = 0;

  std::multimap<size_t, Block>::iterator take(std::multimap<size_t, Block>::iterator it) {
    by_time.erase(it->second.when);
    bytes -= it->first;
    return blocks.erase(it);
  }
  void hand_out(size_t b) {
    used += b;
    peak = peak > used ? peak : used;
  }
  void drop_oldest() {
    auto it = by_time.begin()->second;
    void *p = it->second.p;
    take(it);
    size_of.erase(p);
    cudaFree(p);
  }
};
std::mutex g_mu;
std::map<int, DevCache> g_cache;

size_t cache_limit() {
  static size_t lim = [] {
    const char *s = std::getenv("DFJK_CACHE_BYTES");
    return s ? (size_t)std::strtoull(s, nullptr, 10) : ((size_t)96 << 30);
  }();
  return lim;
}

int current_device() {
  int d = 0;
  DFJK_CUDA_CHECK(cudaGetDevice(&d));
  return d;
}

void trim_locked(DevCache &c) {
  while (!c.blocks.empty()) c.drop_oldest();
}
}  // namespace

void *pool_alloc(size_t bytes) {
  if (bytes == 0) return nullptr;
  const int dev = current_device();
  {
    std::lock_guard<std::mutex> lk(g_mu);
    DevCache &c = g_cache[dev];
    auto it = c.blocks.lower_bound(bytes);
    if (it != c.blocks.end() && it->first <= bytes + bytes / 8) {
      void *p = it->second.p;
      c.hand_out(it->first);
      c.take(it);
      return p;
    }
  }
  void *p = nullptr;
  cudaError_t e = cudaMalloc(&p, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    {
      std::lock_guard<std::mutex> lk(g_mu);
      trim_locked(g_cache[dev]);
    }
    e = cudaMalloc(&p, bytes);
    if (e != cudaSuccess) {
      cudaGetLastError();
      throw Error{DFJK_ERR_OOM, "cudaMalloc of " + std::to_string(bytes) + " bytes failed"};
    }
  }
  std::lock_guard<std::mutex> lk(g_mu);
  g_cache[dev].size_of[p] = bytes;
  g_cache[dev].hand_out(bytes);
  return p;
}

void pool_free(void *p, size_t) {
  if (!p) return;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaFree(p);
    return;
  }
  std::lock_guard<std::mutex> lk(g_mu);
  DevCache &c = g_cache[dev];
  const auto known = c.size_of.find(p);
  if (known != c.size_of.end()) c.used -= known->second;
  if (known == c.size_of.end() || known->second > cache_limit()) {
    if (known != c.size_of.end()) c.size_of.erase(known);
    cudaFree(p);
    return;
  }
  const size_t bytes = known->second;
  while (c.bytes + bytes > cache_limit()) c.drop_oldest();
  const auto it = c.blocks.emplace(bytes, DevCache::Block{p, c.clock});
  c.by_time.emplace(c.clock++, it);
  c.bytes += bytes;
}

void pool_trim() {
  const int dev = current_device();
  std::lock_guard<std::mutex> lk(g_mu);
  trim_locked(g_cache[dev]);
}

size_t pool_cached_bytes() {
  const int dev = current_device();
  std::lock_guard<std::mutex> lk(g_mu);
  return g_cache[dev].bytes;
}

}  // namespace dfjk

// For tests: the most bytes handed out at a time on this device since the last call.
extern "C" size_t dfjk_debug_pool_peak(void) {
  try {
    const int dev = dfjk::current_device();
    std::lock_guard<std::mutex> lk(dfjk::g_mu);
    dfjk::DevCache &c = dfjk::g_cache[dev];
    const size_t peak = c.peak;
    c.peak = c.used;
    return peak;
  } catch (const dfjk::Error &) {
    return 0;
  }
}

extern "C" int dfjk_trim_cache(void) {
  try {
    dfjk::pool_trim();
    return DFJK_OK;
  } catch (const dfjk::Error &e) {
    dfjk::set_error(e.msg);
    return e.code;
  }
}
