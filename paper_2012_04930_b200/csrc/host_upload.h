// Uploads of pageable host memory.  The driver copies pageable memory through one staging buffer with one thread
// (10.5 GB/s; 3.7 GB/s row by row); here four host threads copy through pinned buffers of their own, two each, and the
// copies run on a stream beside the caller's (40 GB/s of the 53 that pinned memory reaches; 2 threads: 20, 8: 42).
// The 8 MB of pinned memory live as long as the object.  Getting them is what an upload starts with: cudaHostAlloc pins 2 048
// small pages one by one, 3.7 to 8 ms here; four huge pages registered with the driver take 1.0 to 1.4 ms with their first touch.
#pragma once
#include <cuda_runtime.h>
#include <sys/mman.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <cstring>
#include <exception>
#include <thread>
#include <vector>

namespace gcnsa {

class HostUpload {
 public:
  static constexpr size_t kWorthwhile = 64u << 20;
  explicit HostUpload(int device) : device_(device) {}
  ~HostUpload() {
    join();
    if (stream_) {
      cudaStreamSynchronize(stream_);
      cudaStreamDestroy(stream_);
    }
    if (event_) cudaEventDestroy(event_);
    unpin();
  }
  HostUpload(const HostUpload&) = delete;
  HostUpload& operator=(const HostUpload&) = delete;

  // whether src is ordinary (neither pinned nor managed) memory
  static bool pageable(const void* src) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, src) != cudaSuccess) {
      cudaGetLastError();
      return true;
    }
    return a.type == cudaMemoryTypeUnregistered;
  }
  // false: no pinned memory or no stream to be had; the caller copies plainly
  bool open() {
    if (event_) return true;
    if (!pin() || cudaStreamCreateWithFlags(&stream_, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&event_, cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    return true;
  }
  // `rows` rows of row_bytes, src_pitch bytes apart, become dense at dst
  void add(void* dst, const void* src, size_t rows, size_t row_bytes, size_t src_pitch) {
    if (rows == 0 || row_bytes == 0) return;
    uint8_t* d = (uint8_t*)dst;
    const uint8_t* s = (const uint8_t*)src;
    if (src_pitch == row_bytes) {
      row_bytes *= rows;
      rows = 1;
    }
    const size_t per = std::max<size_t>(1, kChunk / row_bytes);
    for (size_t r = 0; r < rows; r += per) {
      const size_t n = std::min(per, rows - r);
      if (row_bytes <= kChunk) {
        chunks_.push_back({d + r * row_bytes, s + r * src_pitch, n, row_bytes, src_pitch});
      } else {  // one long row
        for (size_t b = 0; b < row_bytes; b += kChunk)
          chunks_.push_back({d + r * row_bytes + b, s + r * src_pitch + b, 1, std::min(kChunk, row_bytes - b), 0});
      }
    }
  }
  // the threads copy what was added, after the work that is on `after` now
  cudaError_t start(cudaStream_t after) {
    cudaError_t e = cudaEventRecord(event_, after);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(stream_, event_, 0);
    if (e != cudaSuccess) return e;
    next_ = 0;
    error_ = (int)cudaSuccess;
    for (int t = 0; t < kThreads; ++t) {
      try {
        threads_.emplace_back([this, t] { work(t); });
      } catch (const std::exception&) {  // no thread, or no memory for one
        break;
      }
    }
    if (threads_.empty()) work(0);
    return cudaSuccess;
  }
  // `then` waits for the copies; the host arrays are no longer read when this returns
  cudaError_t finish(cudaStream_t then) {
    join();
    chunks_.clear();
    cudaError_t e = (cudaError_t)error_.load();
    if (e == cudaSuccess) e = cudaEventRecord(event_, stream_);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(then, event_, 0);
    return e;
  }

 private:
  static constexpr int kThreads = 4;
  static constexpr size_t kChunk = 1u << 20, kPinned = 2 * kThreads * kChunk, kHuge = 2u << 20;
  struct Chunk {
    uint8_t* dst;
    const uint8_t* src;
    size_t rows, row_bytes, src_pitch;
  };
  // huge pages where the system has them to give; ordinary ones otherwise
  bool pin() {
    if (pinned_) return true;
    map_ = mmap(nullptr, kPinned + kHuge, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    if (map_ == MAP_FAILED) {
      map_ = nullptr;
      return false;
    }
    uint8_t* at = (uint8_t*)(((uintptr_t)map_ + kHuge - 1) / kHuge * kHuge);
    madvise(at, kPinned, MADV_HUGEPAGE);
    if (cudaHostRegister(at, kPinned, cudaHostRegisterDefault) != cudaSuccess) {
      unpin();
      return false;
    }
    pinned_ = at;
    return true;
  }
  void unpin() {
    if (pinned_) cudaHostUnregister(pinned_);
    if (map_) munmap(map_, kPinned + kHuge);
    pinned_ = nullptr;
    map_ = nullptr;
  }
  void join() {
    for (std::thread& t : threads_) t.join();
    threads_.clear();
  }
  void work(int id) {
    cudaError_t e = cudaSetDevice(device_);
    cudaEvent_t done[2] = {nullptr, nullptr};
    bool used[2] = {false, false};
    for (int b = 0; b < 2 && e == cudaSuccess; ++b) e = cudaEventCreateWithFlags(&done[b], cudaEventDisableTiming);
    for (int b = 0; e == cudaSuccess; b ^= 1) {
      const size_t i = next_.fetch_add(1);
      if (i >= chunks_.size()) break;
      const Chunk& c = chunks_[i];
      uint8_t* buf = pinned_ + (size_t)(2 * id + b) * kChunk;
      if (used[b]) e = cudaEventSynchronize(done[b]);
      if (e != cudaSuccess) break;
      if (c.rows == 1) std::memcpy(buf, c.src, c.row_bytes);
      else
        for (size_t r = 0; r < c.rows; ++r) std::memcpy(buf + r * c.row_bytes, c.src + r * c.src_pitch, c.row_bytes);
      e = cudaMemcpyAsync(c.dst, buf, c.rows * c.row_bytes, cudaMemcpyHostToDevice, stream_);
      if (e == cudaSuccess) e = cudaEventRecord(done[b], stream_);
      used[b] = true;
    }
    for (int b = 0; b < 2; ++b) {
      if (used[b]) {
        const cudaError_t w = cudaEventSynchronize(done[b]);
        if (e == cudaSuccess) e = w;
      }
      if (done[b]) cudaEventDestroy(done[b]);
    }
    if (e != cudaSuccess) error_ = (int)e;
  }

  int device_;
  void* map_ = nullptr;  // pinned_ lies in it, on a boundary of huge pages
  uint8_t* pinned_ = nullptr;
  cudaStream_t stream_ = nullptr;
  cudaEvent_t event_ = nullptr;
  std::vector<Chunk> chunks_;
  std::vector<std::thread> threads_;
  std::atomic<size_t> next_{0};
  std::atomic<int> error_{0};
};

}  // namespace gcnsa
