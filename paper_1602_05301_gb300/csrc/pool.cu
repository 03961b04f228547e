// Device memory of the library's buffers (DevBuf). A plan owns about 150 buffers,
// and cudaMalloc / cudaFree cost up to 100 us each (cudaFree also waits for the
// device), which was a fifth of the time of building and dropping a plan (8192
// nodes: 14.2 -> 11.2 ms). Blocks given back are therefore kept for later buffers of
// the same size class:
//  * at most kPoolBytes are kept per device; the oldest blocks beyond that, and all
//    when an allocation fails, go back to the driver (an allocation that fails is
//    tried again without the rounding to its class);
//  * qbx_release_memory gives all of them back;
//  * a block is kept only after a device synchronisation on its device, as
//    cudaFree has it, so that it may serve any stream and thread at once
//    (DeviceQuiet makes one synchronisation serve many blocks);
//  * all under one mutex.
#include <deque>
#include <map>
#include <mutex>
#include <shared_mutex>
#include <unordered_map>

#include "qbx_internal.h"

namespace {

constexpr size_t kPoolBytes = 256u << 20;

struct Pool {
  struct Block {
    size_t size;
    int dev;
  };
  std::mutex mu;
  struct Kept {
    void* p;
    unsigned long long age;  // smaller: kept for longer
  };
  std::unordered_map<void*, Block> live;
  // per device: the blocks kept by size, oldest first, and their sizes by age
  struct Device {
    std::map<size_t, std::deque<Kept>> of_size;
    std::map<unsigned long long, size_t> by_age;
    size_t bytes = 0;
  };
  std::map<int, Device> devs;
  unsigned long long clock = 0;
};
// never destroyed: the driver may be gone when static destructors run
Pool& pool() {
  static Pool* p = new Pool();
  return *p;
}
thread_local int t_quiet = 0;
std::shared_mutex g_capture;  // held alone by a capture, shared by synchronisations
thread_local bool t_capturing = false;

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

// Gives the oldest kept blocks of D back to the driver until at most `most` bytes stay.
void trim(Pool::Device& D, size_t most) {
  while (D.bytes > most) {
    const auto oldest = D.by_age.begin();
    auto it = D.of_size.find(oldest->second);
    cudaFree(it->second.front().p);
    D.bytes -= it->first;
    it->second.pop_front();
    if (it->second.empty()) D.of_size.erase(it);
    D.by_age.erase(oldest);
  }
}

}  // namespace

cudaError_t dev_sync() {
  if (t_capturing) return cudaErrorStreamCaptureUnsupported;
  std::shared_lock<std::shared_mutex> lock(g_capture);
  return cudaDeviceSynchronize();
}
CaptureScope::CaptureScope() {
  g_capture.lock();
  t_capturing = true;
}
CaptureScope::~CaptureScope() {
  t_capturing = false;
  g_capture.unlock();
}

cudaError_t dev_alloc(void** out, size_t bytes) {
  *out = nullptr;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  size_t n = size_class(bytes);
  Pool& P = pool();
  std::lock_guard<std::mutex> lock(P.mu);
  Pool::Device& D = P.devs[dev];
  auto it = D.of_size.find(n);
  if (it != D.of_size.end()) {
    *out = it->second.back().p;
    D.by_age.erase(it->second.back().age);
    it->second.pop_back();
    if (it->second.empty()) D.of_size.erase(it);
    D.bytes -= n;
  } else {
    e = cudaMalloc(out, n);
    if (e == cudaErrorMemoryAllocation && D.bytes > 0) {
      cudaGetLastError();
      trim(D, 0);
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
    const cudaError_t e = dev_sync();
    if (dev != b.dev) cudaSetDevice(dev);
    if (e != cudaSuccess) {  // a broken context or this thread's capture: not kept
      cudaFree(p);
      return;
    }
  }
  std::lock_guard<std::mutex> lock(P.mu);
  if (b.size > kPoolBytes || b.size != size_class(b.size)) {
    cudaFree(p);
    return;
  }
  Pool::Device& D = P.devs[b.dev];
  trim(D, kPoolBytes - b.size);
  D.of_size[b.size].push_back({p, P.clock});
  D.by_age[P.clock++] = b.size;
  D.bytes += b.size;
}

// (where it cannot synchronise, each block tries for itself)
DeviceQuiet::DeviceQuiet() : quiet(t_quiet > 0 || dev_sync() == cudaSuccess) {
  if (quiet) ++t_quiet;
}
DeviceQuiet::~DeviceQuiet() {
  if (quiet) --t_quiet;
}

extern "C" int64_t qbx_release_memory(void) {
  Pool& P = pool();
  std::lock_guard<std::mutex> lock(P.mu);
  size_t n = 0;
  for (auto& d : P.devs) {
    n += d.second.bytes;
    trim(d.second, 0);
  }
  return (int64_t)n;
}
