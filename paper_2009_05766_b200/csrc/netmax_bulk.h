// Large transfers between pageable host memory and the device, and other host work on whole M x M
// matrices, shared out over a few threads.
#pragma once
#include <algorithm>
#include <atomic>
#include <cstddef>
#include <cstdint>
#include <cstring>
#include <exception>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

namespace netmax {

// Number of the current device's CUDA context, another one after every cudaDeviceReset (0: not known).  Whatever outlives
// a simulator -- page-locked blocks, copiers, kernel attributes that have been set -- belongs to the context it was made
// in and is forgotten when that is gone.
inline uint64_t context_number() {
  using Query = int (*)(void*, unsigned long long*);  // cuCtxGetId
  static const Query query = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult status;
    if (cudaGetDriverEntryPoint("cuCtxGetId", &f, cudaEnableDefault, &status) != cudaSuccess) cudaGetLastError();
    return (Query)f;
  }();
  unsigned long long id = 0;
  if (!query || query(nullptr, &id) != 0) return 0;
  return id;
}

// body(t) for t = 0 ... n - 1 at the same time, body(0) on the calling thread; n at most kMaxThreads.  Where the system has
// no thread to give, the calling one does that part as well; what a part throws is thrown here, after all have ended.
constexpr int kMaxThreads = 16;
template <typename Body>
void on_threads(int n, const Body& body) {
  std::thread pool[kMaxThreads];
  std::exception_ptr thrown[kMaxThreads];
  auto part = [&](int t) noexcept {
    try {
      body(t);
    } catch (...) {
      thrown[t] = std::current_exception();
    }
  };
  for (int t = 1; t < n; ++t) {
    try {
      pool[t] = std::thread([&part, t] { part(t); });
    } catch (...) {
      part(t);
    }
  }
  part(0);
  for (int t = 1; t < n; ++t)
    if (pool[t].joinable()) pool[t].join();
  for (int t = 0; t < n; ++t)
    if (thrown[t]) std::rethrow_exception(thrown[t]);
}

// body(begin, end) on slices of [0, n), on up to 16 threads once n reaches min_parallel.
template <typename Body>
void parallel_rows(int64_t n, int64_t min_parallel, const Body& body) {
  const unsigned hw = n >= min_parallel ? std::thread::hardware_concurrency() : 1;
  const int threads = (int)std::min<unsigned>(hw, kMaxThreads);
  if (threads <= 1) {
    body(0, n);
    return;
  }
  const int64_t per = (n + threads - 1) / threads;
  on_threads((int)((n + per - 1) / per), [&](int t) { body(t * per, std::min<int64_t>(n, (t + 1) * per)); });
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
  // Its memory and streams went with their context.
  void forget() {
    stage_ = nullptr;
    for (auto& s : streams_) s = nullptr;
  }
  // Copies after everything enqueued on `stream`; has finished when it returns.
  cudaError_t to_device(void* dst, const void* src, size_t bytes, int device, cudaStream_t stream) {
    return run((char*)dst, (const char*)src, bytes, device, stream, true);
  }
  cudaError_t to_host(void* dst, const void* src, size_t bytes, int device, cudaStream_t stream) {
    return run((char*)dst, (const char*)src, bytes, device, stream, false);
  }

 private:
  static constexpr int kLanes = 4;  // (a lane that gets no thread of its own finds its work done by the others)
  static constexpr size_t kChunk = (size_t)1 << 20;
  unsigned char* stage_ = nullptr;
  cudaStream_t streams_[kLanes] = {};

  bool prepare() {
    void* p = nullptr;
    if (!stage_ && cudaHostAlloc(&p, 2 * kLanes * kChunk, cudaHostAllocPortable) != cudaSuccess) return false;
    if (!stage_) stage_ = (unsigned char*)p;
    for (auto& s : streams_)
      if (!s && cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) return false;
    return true;
  }

  cudaError_t run(char* dst, const char* src, size_t bytes, int device, cudaStream_t stream, bool up) {
    cudaError_t e;
    if (!prepare()) {  // no memory to be locked: one plain copy
      cudaGetLastError();
      if ((e = cudaMemcpyAsync(dst, src, bytes, up ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost, stream)) != cudaSuccess) return e;
      return cudaStreamSynchronize(stream);
    }
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
    on_threads(kLanes, lane);
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
    uint64_t context;
    std::unique_ptr<BulkCopier> copier;
  };
  std::mutex mu_;
  std::vector<Idle> idle_;
  BulkPool() { idle_.reserve(2); }  // (giving a copier back allocates nothing)

  template <typename F>
  cudaError_t with(int device, F body) {
    std::unique_ptr<BulkCopier> c;
    const uint64_t context = context_number();
    {
      std::lock_guard<std::mutex> lock(mu_);
      for (size_t k = idle_.size(); k-- > 0;) {
        if (idle_[k].device != device) continue;
        if (idle_[k].context == context) {
          if (c) continue;
          c = std::move(idle_[k].copier);
        } else {
          idle_[k].copier->forget();
        }
        idle_.erase(idle_.begin() + (long)k);
      }
    }
    if (!c) c.reset(new BulkCopier());
    const cudaError_t e = body(*c);
    if (e == cudaSuccess) {
      std::lock_guard<std::mutex> lock(mu_);
      if (idle_.size() < 2) idle_.push_back(Idle{device, context, std::move(c)});
    }
    return e;
  }
};

}  // namespace netmax
