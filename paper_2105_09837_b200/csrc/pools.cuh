// Device memory, streams and events that outlive a context.
//
// A context takes a few large blocks of device memory, a stream per lane and some events.  Asking the driver for them and
// giving them back cost more than the set-up itself (10 layers of 500 on 20 000 nodes: 8 of 16 ms of pdadmm_init and 8 of
// 8 ms of pdadmm_destroy; more after large frees, when the driver clears pages first), and programs make contexts one
// after another: the greedy schedule grows one into the next, a sweep over settings rebuilds the same problem.  So what
// destroy returns is kept for the next context of the process, within bounds:
//   - device memory: at most 1/16 of the device, the oldest block goes first, and nothing while less than half of the
//     device is free (somebody else may need it; asked at most twice a second: the question goes to the driver's resource
//     manager, 0.1 ms, and 5 ms and more while other processes of the machine keep it busy); all of it goes back to the
//     driver when an allocation of this library
//     fails, and in pdadmm_release_cached_memory();
//   - at most 64 streams and 256 events of each kind per device.
// Everything is returned only after the context's device work has finished.  One lock per device; any thread.
#pragma once

#include <cuda_runtime.h>

#include <chrono>
#include <mutex>
#include <new>
#include <vector>

#include "common.cuh"

namespace pd {

struct DeviceBlock { void *p; size_t bytes; };

class DevicePool {
  static constexpr size_t MAX_STREAMS = 64, MAX_EVENTS = 256;
 public:
  DevicePool() {                           // giving a stream or an event back never allocates
    streams_.reserve(MAX_STREAMS);
    events_[0].reserve(MAX_EVENTS);
    events_[1].reserve(MAX_EVENTS);
  }
  // A block of at least `bytes` bytes, at most a quarter more; contents are undefined.  The device must be current.
  cudaError_t take(size_t bytes, DeviceBlock *out) {
    {
      std::lock_guard<std::mutex> g(m_);
      size_t best = free_.size();
      for (size_t i = 0; i < free_.size(); ++i)
        if (free_[i].bytes >= bytes && free_[i].bytes <= bytes + bytes / 4 && (best == free_.size() || free_[i].bytes < free_[best].bytes)) best = i;
      if (best != free_.size()) {
        *out = free_[best];
        free_.erase(free_.begin() + (long)best);
        held_ -= out->bytes;
        return cudaSuccess;
      }
    }
    void *p = nullptr;
    cudaError_t e = cudaMalloc(&p, bytes);
    if (e == cudaErrorMemoryAllocation) {
      cudaGetLastError();
      trim();
      e = cudaMalloc(&p, bytes);
    }
    if (e != cudaSuccess) { cudaGetLastError(); return e; }
    *out = DeviceBlock{p, bytes};
    return cudaSuccess;
  }
  // No device work may use the blocks any more.
  void give(const std::vector<DeviceBlock> &blocks) {
    if (blocks.empty()) return;
    ask();
    std::vector<DeviceBlock> out;
    try {
      std::lock_guard<std::mutex> g(m_);
      free_.reserve(free_.size() + blocks.size());
      out.reserve(free_.size() + blocks.size());
      const bool keep = roomy_;
      const size_t total = total_;
      for (const DeviceBlock &b : blocks) {
        if (!keep || b.bytes > total / 16) { out.push_back(b); continue; }
        free_.push_back(b);
        held_ += b.bytes;
      }
      while (!free_.empty() && (!keep || held_ > total / 16)) {
        out.push_back(free_.front());
        held_ -= free_.front().bytes;
        free_.erase(free_.begin());
      }
    } catch (const std::bad_alloc &) {       // no room to remember them
      for (const DeviceBlock &b : blocks) cudaFree(b.p);
      return;
    }
    for (const DeviceBlock &b : out) cudaFree(b.p);
  }
  void trim() {
    std::vector<DeviceBlock> out;
    {
      std::lock_guard<std::mutex> g(m_);
      out.swap(free_);
      held_ = 0;
    }
    for (const DeviceBlock &b : out) cudaFree(b.p);
  }
  cudaError_t take_stream(cudaStream_t *s) {
    {
      std::lock_guard<std::mutex> g(m_);
      if (!streams_.empty()) { *s = streams_.back(); streams_.pop_back(); return cudaSuccess; }
    }
    return cudaStreamCreateWithFlags(s, cudaStreamNonBlocking);
  }
  void give_stream(cudaStream_t s) {
    if (s == nullptr) return;
    {
      std::lock_guard<std::mutex> g(m_);
      if (streams_.size() < MAX_STREAMS) { streams_.push_back(s); return; }
    }
    cudaStreamDestroy(s);
  }
  cudaError_t take_event(bool timing, cudaEvent_t *ev) {
    {
      std::lock_guard<std::mutex> g(m_);
      auto &v = events_[timing];
      if (!v.empty()) { *ev = v.back(); v.pop_back(); return cudaSuccess; }
    }
    return cudaEventCreateWithFlags(ev, timing ? cudaEventDefault : cudaEventDisableTiming);
  }
  void give_event(bool timing, cudaEvent_t ev) {
    if (ev == nullptr) return;
    {
      std::lock_guard<std::mutex> g(m_);
      if (events_[timing].size() < MAX_EVENTS) { events_[timing].push_back(ev); return; }
    }
    cudaEventDestroy(ev);
  }

 private:
  // Whether half of the device is free, asked without the lock: the answer can take milliseconds, and other threads come here
  // for memory meanwhile.  They go by the answer before (nothing is kept before the first).
  void ask() {
    {
      std::lock_guard<std::mutex> g(m_);
      const auto now = std::chrono::steady_clock::now();
      if (asked_ != std::chrono::steady_clock::time_point{} && now - asked_ <= std::chrono::milliseconds(500)) return;
      asked_ = now;
    }
    size_t free_bytes = 0, total = 0;
    const bool roomy = cudaMemGetInfo(&free_bytes, &total) == cudaSuccess && free_bytes >= total / 2;
    std::lock_guard<std::mutex> g(m_);
    roomy_ = roomy;
    total_ = total;
  }
  std::mutex m_;
  std::vector<DeviceBlock> free_;          // oldest first
  size_t held_ = 0, total_ = 0;
  bool roomy_ = false;
  std::chrono::steady_clock::time_point asked_{};
  std::vector<cudaStream_t> streams_;
  std::vector<cudaEvent_t> events_[2];
};

constexpr int MAX_DEVICES = 64;
// Never destroyed: at process exit the driver may be gone before static destructors run.
inline DevicePool &device_pool(int device) {
  static DevicePool *pools = new DevicePool[MAX_DEVICES];
  return pools[device >= 0 && device < MAX_DEVICES ? device : 0];
}

}  // namespace pd
