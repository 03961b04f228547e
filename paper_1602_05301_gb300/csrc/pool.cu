// Device memory of the library's buffers (DevBuf). A plan owns about 150 buffers,
// and cudaMalloc / cudaFree cost up to 100 us each (cudaFree also waits for the
// device), which was a fifth of the time of building and dropping a plan (8192
// nodes: 14.2 -> 11.2 ms). Blocks given back are therefore kept for later buffers of
// the same size class:
//  * at most kPoolBytes are kept per device; what exceeds that, and everything
//    when an allocation fails, goes back to the driver (an allocation that fails
//    is tried again without the rounding to its class);
//  * a block is kept only after a device synchronisation on its device, as
//    cudaFree has it, so that it may serve any stream and thread at once
//    (DeviceQuiet makes one synchronisation serve many blocks);
//  * all under one mutex.
#include <map>
#include <mutex>
#include <unordered_map>
#include <vector>

#include "qbx_internal.h"

namespace {

constexpr size_t kPoolBytes = 256u << 20;

struct Pool {
  struct Block {
    size_t size;
    int dev;
  };
  std::mutex mu;
  std::unordered_map<void*, Block> live;
  std::map<std::pair<int, size_t>, std::vector<void*>> kept;
  std::map<int, size_t> kept_bytes;
};
// never destroyed: the driver may be gone when static destructors run
Pool& pool() {
  static Pool* p = new Pool();
  return *p;
}
thread_local int t_quiet = 0;

size_t multiple(size_t n, size_t step) { return (n + step - 1) / step * step; }
// Size classes: multiples of 512 bytes to 4 KB, four steps per power of two to 2 MB,
// then multiples of 2 MB, which cudaMalloc hands out anyway: a plan's large buffers
// take no more memory than without the pool.
constexpr size_t kGranule = 2u << 20;
size_t size_class(size_t n) {
  if (n <= 4096) return multiple(n, 512);
  if (n > kGranule) return multiple(n, kGranule);
  size_t step = 1024;
  while (step * 8 < n) step *= 2;
  return multiple(n, step);
}

void drop_kept(Pool& P, int dev) {
  for (auto& e : P.kept)
    if (e.first.first == dev) {
      for (void* p : e.second) cudaFree(p);
      e.second.clear();
    }
  P.kept_bytes[dev] = 0;
}

}  // namespace

cudaError_t dev_alloc(void** out, size_t bytes) {
  *out = nullptr;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  size_t n = size_class(bytes);
  Pool& P = pool();
  std::lock_guard<std::mutex> lock(P.mu);
  auto it = P.kept.find({dev, n});
  if (it != P.kept.end() && !it->second.empty()) {
    *out = it->second.back();
    it->second.pop_back();
    P.kept_bytes[dev] -= n;
  } else {
    e = cudaMalloc(out, n);
    if (e == cudaErrorMemoryAllocation && P.kept_bytes[dev] > 0) {
      cudaGetLastError();
      drop_kept(P, dev);
      e = cudaMalloc(out, n);
    }
    if (e == cudaErrorMemoryAllocation) {  // what the buffer needs may still be there
      cudaGetLastError();
      n = multiple(bytes, 512);
      e = cudaMalloc(out, n);
    }
    if (e != cudaSuccess) {
      *out = nullptr;
      return e;
    }
  }
  P.live[*out] = {n, dev};
  return cudaSuccess;
}

void dev_free(void* p) {
  if (!p) return;
  Pool& P = pool();
  Pool::Block b;
  {
    std::lock_guard<std::mutex> lock(P.mu);
    auto it = P.live.find(p);
    if (it == P.live.end()) return;
    b = it->second;
    P.live.erase(it);
  }
  int dev = 0;
  cudaGetDevice(&dev);
  if (t_quiet == 0 || dev != b.dev) {
    if (dev != b.dev) cudaSetDevice(b.dev);
    const cudaError_t e = cudaDeviceSynchronize();
    if (dev != b.dev) cudaSetDevice(dev);
    if (e != cudaSuccess) {  // a broken context: nothing to keep
      cudaFree(p);
      return;
    }
  }
  std::lock_guard<std::mutex> lock(P.mu);
  if (P.kept_bytes[b.dev] + b.size > kPoolBytes || b.size != size_class(b.size)) {
    cudaFree(p);
    return;
  }
  P.kept[{b.dev, b.size}].push_back(p);
  P.kept_bytes[b.dev] += b.size;
}

// (where it cannot synchronise, each block tries for itself)
DeviceQuiet::DeviceQuiet() : quiet(t_quiet > 0 || cudaDeviceSynchronize() == cudaSuccess) {
  if (quiet) ++t_quiet;
}
DeviceQuiet::~DeviceQuiet() {
  if (quiet) --t_quiet;
}
