// Large transfers between pageable host memory and the device, and other host work on whole M x M
// matrices, shared out over a few threads.
#pragma once
#include <algorithm>
#include <atomic>
#include <cstddef>
#include <cstring>
#include <functional>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

namespace netmax {

// body(begin, end) on slices of [0, n), on up to 16 threads once n reaches min_parallel.
inline void parallel_rows(int64_t n, int64_t min_parallel, const std::function<void(int64_t, int64_t)>& body) {
  const unsigned hw = std::thread::hardware_concurrency();
  const int threads = (n >= min_parallel && hw > 1) ? (int)std::min<unsigned>(hw, 16) : 1;
  if (threads <= 1) {
    body(0, n);
    return;
  }
  std::vector<std::thread> pool;
  const int64_t per = (n + threads - 1) / threads;
  for (int t = 1; t < threads; ++t) {
    const int64_t a = std::min<int64_t>(n, t * per), b = std::min<int64_t>(n, a + per);
    if (a < b) pool.emplace_back(body, a, b);
  }
  body(0, std::min<int64_t>(n, per));
  for (auto& th : pool) th.join();
}

// memcpy; from 8 MB on by several threads (one core neither reaches the memory's bandwidth nor keeps up
// with the page faults of a destination that is touched for the first time).
inline void parallel_copy(void* dst, const void* src, size_t bytes) {
  const int64_t block = (int64_t)1 << 20, blocks = (int64_t)((bytes + block - 1) / block);
  parallel_rows(blocks, 8, [&](int64_t a, int64_t b) {
    const size_t from = (size_t)(a * block), to = std::min(bytes, (size_t)(b * block));
    if (from < to) std::memcpy((char*)dst + from, (const char*)src + from, to - from);
  });
}

// Copies of pageable memory by kLanes threads, each with two page-locked chunks of its own: the driver's
// own staging runs on one core (134 MB: about 13 ms each way; 5 ms with four).  For one device and one caller at a time.
class BulkCopier {
 public:
  ~BulkCopier() {
    for (auto& s : streams_)
      if (s) cudaStreamDestroy(s);
    if (stage_) cudaFreeHost(stage_);
    cudaGetLastError();
  }
  // Copies after everything enqueued on `stream`; has finished when it returns.
  cudaError_t to_device(void* dst, const void* src, size_t bytes, int device, cudaStream_t stream) {
    return run((char*)dst, (const char*)src, bytes, device, stream, true);
  }
  cudaError_t to_host(void* dst, const void* src, size_t bytes, int device, cudaStream_t stream) {
    return run((char*)dst, (const char*)src, bytes, device, stream, false);
  }

 private:
  static constexpr int kLanes = 4;
  static constexpr size_t kChunk = (size_t)1 << 20;
  unsigned char* stage_ = nullptr;
  cudaStream_t streams_[kLanes] = {};

  cudaError_t run(char* dst, const char* src, size_t bytes, int device, cudaStream_t stream, bool up) {
    cudaError_t e;
    if (!stage_) {
      void* p = nullptr;
      if ((e = cudaHostAlloc(&p, 2 * kLanes * kChunk, cudaHostAllocPortable)) != cudaSuccess) return e;
      stage_ = (unsigned char*)p;
    }
    for (auto& s : streams_)
      if (!s && (e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(stream)) != cudaSuccess) return e;  // the other streams start behind it
    const int64_t chunks = (int64_t)((bytes + kChunk - 1) / kChunk);
    std::atomic<int64_t> next{0};
    cudaError_t failed[kLanes];
    auto lane = [&](int l) {
      cudaError_t r = cudaSetDevice(device);
      cudaEvent_t done[2] = {nullptr, nullptr};
      for (auto& ev : done)
        if (r == cudaSuccess) r = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
      int64_t held[2] = {-1, -1};  // down: the chunk whose copy into half h is in flight
      auto drain = [&](int h) {
        if (held[h] < 0) return;
        if (r == cudaSuccess) r = cudaEventSynchronize(done[h]);
        if (!up && r == cudaSuccess) {
          const size_t at = (size_t)held[h] * kChunk, n = std::min(kChunk, bytes - at);
          std::memcpy(dst + at, stage_ + (size_t)(2 * l + h) * kChunk, n);
        }
        held[h] = -1;
      };
      for (int h = 0; r == cudaSuccess; h ^= 1) {
        const int64_t c = next.fetch_add(1);
        if (c >= chunks) break;
        drain(h);
        if (r != cudaSuccess) break;
        const size_t at = (size_t)c * kChunk, n = std::min(kChunk, bytes - at);
        unsigned char* buf = stage_ + (size_t)(2 * l + h) * kChunk;
        if (up) std::memcpy(buf, src + at, n);
        r = cudaMemcpyAsync(up ? (void*)(dst + at) : (void*)buf, up ? (const void*)buf : (const void*)(src + at), n,
                            up ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost, streams_[l]);
        if (r == cudaSuccess) r = cudaEventRecord(done[h], streams_[l]);
        held[h] = c;
      }
      drain(0);
      drain(1);
      if (streams_[l]) {
        const cudaError_t s = cudaStreamSynchronize(streams_[l]);
        if (r == cudaSuccess) r = s;
      }
      for (auto& ev : done)
        if (ev) cudaEventDestroy(ev);
      failed[l] = r;
    };
    std::thread pool[kLanes];
    for (int l = 1; l < kLanes; ++l) pool[l] = std::thread(lane, l);
    lane(0);
    for (int l = 1; l < kLanes; ++l) pool[l].join();
    for (cudaError_t r : failed)
      if (r != cudaSuccess) return r;
    return cudaSuccess;
  }
};

// Copiers shared by all contexts: locking their pages takes milliseconds, more than most transfers, so idle ones are
// kept for the next transfer, at most two of them.
class BulkPool {
 public:
  cudaError_t to_device(void* dst, const void* src, size_t bytes, int device, cudaStream_t stream) {
    return with(device, [&](BulkCopier& c) { return c.to_device(dst, src, bytes, device, stream); });
  }
  cudaError_t to_host(void* dst, const void* src, size_t bytes, int device, cudaStream_t stream) {
    return with(device, [&](BulkCopier& c) { return c.to_host(dst, src, bytes, device, stream); });
  }
  static BulkPool& get() {
    static BulkPool* pool = new BulkPool();  // never destroyed: contexts may outlive static destructors
    return *pool;
  }

 private:
  struct Idle {
    int device;
    std::unique_ptr<BulkCopier> copier;
  };
  std::mutex mu_;
  std::vector<Idle> idle_;

  template <typename F>
  cudaError_t with(int device, F body) {
    std::unique_ptr<BulkCopier> c;
    {
      std::lock_guard<std::mutex> lock(mu_);
      for (size_t k = 0; k < idle_.size(); ++k)
        if (idle_[k].device == device) {
          c = std::move(idle_[k].copier);
          idle_.erase(idle_.begin() + (long)k);
          break;
        }
    }
    if (!c) c.reset(new BulkCopier());
    const cudaError_t e = body(*c);
    if (e == cudaSuccess) {
      std::lock_guard<std::mutex> lock(mu_);
      if (idle_.size() < 2) idle_.push_back(Idle{device, std::move(c)});
    }
    return e;
  }
};

}  // namespace netmax
