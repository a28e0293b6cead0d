// Copies between the caller's host arrays and the library's padded device matrices.
//
// The caller's arrays are dense and usually pageable, the device matrices have padded rows.  A pageable 2-D copy left to
// the driver moves one row at a time through the driver's own staging (measured: 20 000 rows of 40 bytes 2.9 ms, 14 MB
// of weights 2.1 ms).  Here the rows go through page-locked staging blocks in dense pieces: on the way out a kernel packs a
// piece straight into the block over PCIe, on the way in the copy engine (or, for short rows, a kernel) spreads it over the padded rows; large copies
// are split among a few host threads, because one thread's memcpy (10 GB/s into fresh pages) is what bounds them.
// Page-locked caller arrays skip the staging.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <exception>
#include <thread>
#include <vector>

#include "common.cuh"
#include "pools.cuh"

namespace pd {

// ---- page-locked blocks ------------------------------------------------------------------------------------------
// Page-locking costs about half a millisecond per call, so blocks are kept for the next context or copy: at most
// PINNED_KEEP of each size (4 MB and 1 MB in all), any thread, any device (portable allocations).  A block is in
// the list only while nothing on a device uses it.
constexpr size_t STAGE_BYTES = size_t(512) << 10;      // one piece of a copy in flight
constexpr size_t CTX_PINNED_BYTES = size_t(64) << 10;  // the read-back words of one context
constexpr size_t PINNED_KEEP = 8, CTX_PINNED_KEEP = 16;
class PinnedPool {
 public:
  PinnedPool(size_t bytes, size_t keep) : bytes_(bytes), keep_(keep) { free_.reserve(keep); }     // (give never allocates)
  void *take() {
    {
      std::lock_guard<std::mutex> g(m_);
      if (!free_.empty()) { void *p = free_.back(); free_.pop_back(); return p; }
    }
    void *p = nullptr;
    if (cudaHostAlloc(&p, bytes_, cudaHostAllocPortable) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return p;
  }
  void give(void *p) {
    if (!p) return;
    {
      std::lock_guard<std::mutex> g(m_);
      if (free_.size() < keep_) { free_.push_back(p); return; }
    }
    cudaFreeHost(p);
  }
  void trim() {
    for (;;) {
      void *p = nullptr;
      {
        std::lock_guard<std::mutex> g(m_);
        if (free_.empty()) return;
        p = free_.back();
        free_.pop_back();
      }
      cudaFreeHost(p);
    }
  }
 private:
  const size_t bytes_, keep_;
  std::mutex m_;
  std::vector<void *> free_;
};
// never destroyed: at process exit the driver may be gone before static destructors run
inline PinnedPool &stage_pool() { static PinnedPool &p = *new PinnedPool(STAGE_BYTES, PINNED_KEEP); return p; }
inline PinnedPool &ctx_pinned_pool() { static PinnedPool &p = *new PinnedPool(CTX_PINNED_BYTES, CTX_PINNED_KEEP); return p; }

// Memory that the driver copies by itself: page-locked or managed, or device memory, which the host must not touch.
inline bool is_direct(const void *p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) { cudaGetLastError(); return false; }
  return a.type != cudaMemoryTypeUnregistered;
}

// rows of `width` words at a pitch of `pitch` words -> dense; T = uint4 where both allow it, so that a warp writes whole
// 512-byte runs over PCIe
template <class T>
__global__ void __launch_bounds__(256)
pack_rows_kernel(const T *__restrict__ src, size_t pitch, uint32_t width, uint32_t n, T *__restrict__ dst) {
  for (uint32_t i = blockIdx.x * 256u + threadIdx.x; i < n; i += gridDim.x * 256u) {
    const uint32_t row = i / width;
    dst[i] = src[(size_t)row * pitch + (i - row * width)];
  }
}
// The other way.  The copy engine does wide rows as fast as the link (2 KB rows 30 GB/s) and short ones slowly (400-byte
// rows 6 GB/s), so those are read over PCIe by a kernel.
constexpr size_t UNPACK_BELOW = 2048;
template <class T>
__global__ void __launch_bounds__(256)
unpack_rows_kernel(const T *__restrict__ src, size_t pitch, uint32_t width, uint32_t n, T *__restrict__ dst) {
  for (uint32_t i = blockIdx.x * 256u + threadIdx.x; i < n; i += gridDim.x * 256u) {
    const uint32_t row = i / width;
    dst[(size_t)row * pitch + (i - row * width)] = src[i];
  }
}
inline cudaError_t launch_pack(cudaStream_t st, const void *src, size_t pitch_bytes, size_t width_bytes, size_t rows, void *dst) {
  const bool wide = pitch_bytes % 16 == 0 && width_bytes % 16 == 0 && (uintptr_t)src % 16 == 0 && (uintptr_t)dst % 16 == 0;
  const uint32_t n = (uint32_t)(rows * width_bytes / (wide ? 16 : 4));
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 256), 148));
  if (wide) pack_rows_kernel<uint4><<<grid, 256, 0, st>>>((const uint4 *)src, pitch_bytes / 16, (uint32_t)(width_bytes / 16), n, (uint4 *)dst);
  else pack_rows_kernel<uint32_t><<<grid, 256, 0, st>>>((const uint32_t *)src, pitch_bytes / 4, (uint32_t)(width_bytes / 4), n, (uint32_t *)dst);
  return cudaGetLastError();           // (kept per host thread: nobody else could ask for it later)
}

inline cudaError_t queue_unpack(cudaStream_t st, const void *src, void *dst, size_t pitch, size_t width, size_t rows) {
  if (width >= UNPACK_BELOW || width % 4 || pitch % 4)
    return cudaMemcpy2DAsync(dst, pitch, src, width, width, rows, cudaMemcpyHostToDevice, st);
  const bool wide = pitch % 16 == 0 && width % 16 == 0 && (uintptr_t)src % 16 == 0 && (uintptr_t)dst % 16 == 0;
  const uint32_t n = (uint32_t)(rows * width / (wide ? 16 : 4));
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 256), 296));
  if (wide) unpack_rows_kernel<uint4><<<grid, 256, 0, st>>>((const uint4 *)src, pitch / 16, (uint32_t)(width / 16), n, (uint4 *)dst);
  else unpack_rows_kernel<uint32_t><<<grid, 256, 0, st>>>((const uint32_t *)src, pitch / 4, (uint32_t)(width / 4), n, (uint32_t *)dst);
  return cudaGetLastError();
}

// One direction of a copy, pieces piece0, piece0 + step, ... of `piece_rows` rows each.  Two staging blocks alternate, so
// that the host copies one while the device works on the other.
struct RowCopy {
  char *host; char *dev;
  size_t pitch, width, rows, piece_rows;
  bool out;                      // device -> host
  cudaStream_t st;
};
inline cudaError_t copy_pieces(const RowCopy &k, size_t piece0, size_t step, char *const (&stage)[2], const cudaEvent_t (&ev)[2]) {
  const size_t n_pieces = (size_t)ceil_div((int64_t)k.rows, (int64_t)k.piece_rows);
  auto rows_of = [&](size_t p) { return std::min(k.piece_rows, k.rows - p * k.piece_rows); };
  auto host_of = [&](size_t p) { return k.host + p * k.piece_rows * k.width; };
  auto dev_of = [&](size_t p) { return k.dev + p * k.piece_rows * k.pitch; };
  cudaError_t e = cudaSuccess;
  auto land = [&](size_t p, int b) {
    if ((e = cudaEventSynchronize(ev[b])) == cudaSuccess) memcpy(host_of(p), stage[b], rows_of(p) * k.width);
  };
  int b = 0;
  size_t before = SIZE_MAX;
  bool used[2] = {false, false};
  for (size_t p = piece0; p < n_pieces && e == cudaSuccess; p += step, b ^= 1) {
    const size_t r = rows_of(p);
    if (k.out) {
      if (k.width % 4 == 0 && k.pitch % 4 == 0) e = launch_pack(k.st, dev_of(p), k.pitch, k.width, r, stage[b]);
      else e = cudaMemcpy2DAsync(stage[b], k.width, dev_of(p), k.pitch, k.width, r, cudaMemcpyDeviceToHost, k.st);
      if (e == cudaSuccess) e = cudaEventRecord(ev[b], k.st);
      if (e == cudaSuccess && before != SIZE_MAX) land(before, b ^ 1);
      before = p;
    } else {
      if (used[b]) e = cudaEventSynchronize(ev[b]);
      if (e != cudaSuccess) break;
      memcpy(stage[b], host_of(p), r * k.width);
      e = queue_unpack(k.st, stage[b], dev_of(p), k.pitch, k.width, r);
      if (e == cudaSuccess) e = cudaEventRecord(ev[b], k.st);
      used[b] = true;
    }
  }
  if (k.out) {
    if (e == cudaSuccess && before != SIZE_MAX) land(before, b ^ 1);
  }
  // the blocks go back to the pool: nothing may still be using them
  for (int i = 0; i < 2; ++i)
    if (k.out || used[i]) { const cudaError_t f = cudaEventSynchronize(ev[i]); if (e == cudaSuccess) e = f; }
  return e;
}

// Copies `rows` rows of `width` bytes between a dense host array and device rows `pitch` bytes apart, ordered after the
// work on `st`; returns when the host array has been read or written.
// Host threads: one up to 2 MB, then one per 2 MB up to four (c5's 16 MB weight matrices: one thread 1.9 ms, four 0.7).
inline int copy_rows(int device, cudaStream_t st, void *host, void *dev, size_t pitch, size_t width, size_t rows, bool out) {
  if (rows == 0 || width == 0) return PDADMM_OK;
  if ((rows == 1 || pitch == width) && width != 4096 && rows * width > STAGE_BYTES) {      // contiguous: cut anywhere
    const size_t total = rows * width, unit = 4096, whole = total / unit;
    PD_TRY(copy_rows(device, st, host, dev, unit, unit, whole, out));
    return copy_rows(device, st, (char *)host + whole * unit, (char *)dev + whole * unit, unit, total % unit, 1, out);
  }
  if (width > STAGE_BYTES || is_direct(host)) {
    if (out) PD_CUDA(cudaMemcpy2DAsync(host, width, dev, pitch, width, rows, cudaMemcpyDefault, st));
    else PD_CUDA(cudaMemcpy2DAsync(dev, pitch, host, width, width, rows, cudaMemcpyDefault, st));
    PD_CUDA(cudaStreamSynchronize(st));
    return PDADMM_OK;
  }
  if (rows * width <= STAGE_BYTES) {             // one piece: the stream itself is what to wait for
    char *stage = (char *)stage_pool().take();
    if (stage == nullptr) return fail(PDADMM_ENOMEM, "page-locked host memory is exhausted");
    cudaError_t e = cudaSuccess;
    if (!out) {
      memcpy(stage, host, rows * width);
      e = queue_unpack(st, stage, dev, pitch, width, rows);
    } else if (width % 4 == 0 && pitch % 4 == 0) {
      e = launch_pack(st, dev, pitch, width, rows, stage);
    } else {
      e = cudaMemcpy2DAsync(stage, width, dev, pitch, width, rows, cudaMemcpyDeviceToHost, st);
    }
    const cudaError_t w = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = w;
    if (out && e == cudaSuccess) memcpy(host, stage, rows * width);
    stage_pool().give(stage);
    PD_CUDA(e);
    return PDADMM_OK;
  }
  RowCopy k{(char *)host, (char *)dev, pitch, width, rows, std::max<size_t>(1, STAGE_BYTES / width), out, st};
  const size_t n_pieces = (size_t)ceil_div((int64_t)rows, (int64_t)k.piece_rows);
  const int T = (int)std::max<size_t>(1, std::min<size_t>(std::min<size_t>(4, n_pieces), rows * width / (size_t(2) << 20)));
  struct Worker { char *stage[2] = {nullptr, nullptr}; cudaEvent_t ev[2] = {nullptr, nullptr}; cudaError_t e = cudaSuccess; };
  Worker ws[4];
  DevicePool &events = device_pool(device);        // (made before anything is taken: the first call allocates)
  cudaError_t err = cudaSuccess;
  const int n_stage = n_pieces > (size_t)T ? 2 : 1;
  for (int t = 0; t < T; ++t)
    for (int i = 0; i < 2 && err == cudaSuccess; ++i) {
      Worker &w = ws[t];
      w.stage[i] = i < n_stage ? (char *)stage_pool().take() : w.stage[0];
      if (w.stage[i] == nullptr) err = cudaErrorMemoryAllocation;
      else err = events.take_event(false, &w.ev[i]);
    }
  if (err == cudaSuccess) {
    auto body = [&](int t) {
      cudaSetDevice(device);
      ws[t].e = copy_pieces(k, (size_t)t, (size_t)T, ws[t].stage, ws[t].ev);
    };
    std::thread threads[4];
    int started = 1;
    try {
      for (; started < T; ++started) threads[started] = std::thread(body, started);
    } catch (const std::exception &) {        // no thread, or no memory for one, to be had: this one does their pieces
    }
    body(0);
    for (int t = started; t < T; ++t) body(t);
    for (int t = 1; t < started; ++t) threads[t].join();
    for (int t = 0; t < T; ++t) if (err == cudaSuccess) err = ws[t].e;
  }
  for (int t = 0; t < T; ++t)
    for (int i = 0; i < 2; ++i) {
      events.give_event(false, ws[t].ev[i]);
      if (i < n_stage) stage_pool().give(ws[t].stage[i]);
    }
  PD_CUDA(err);
  PD_CUDA(cudaGetLastError());
  return PDADMM_OK;
}

}  // namespace pd
