// Internal glue between the C-ABI translation units.
#pragma once
#include <cstdint>
#include <exception>
#include <new>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "netmax_bulk.h"

namespace netmax {
template <typename Fail>
int caught(const Fail& fail, int code, const char* what) noexcept {
  try {
    return fail(code, what);
  } catch (...) {
    return code;  // (no memory for the message either)
  }
}
// Ends the function-try-block of a C entry, none of which throws.  fail(code, message) records the message.
#define NM_CATCH(fail)                                                                                          \
  catch (const std::bad_alloc&) { return netmax::caught(fail, NETMAX_OOM, "host allocation failed"); }          \
  catch (const std::exception& e) { return netmax::caught(fail, NETMAX_OOM, e.what()); }

// Records the message netmax_last_error(NULL) returns on the calling thread.
void set_global_error(const std::string& msg);
// Largest eigenvalue of a symmetric tridiagonal matrix (diagonal alpha, off-diagonal beta), and an
// eigenvector of it.
double tridiagonal_top_eigenvalue(const std::vector<double>& alpha, const std::vector<double>& beta);
void tridiagonal_top_vector(const std::vector<double>& alpha, const std::vector<double>& beta, double lambda, std::vector<double>& z);

// Device memory for work on whole M x M matrices: one allocation that is carved up.  A cudaMalloc or cudaFree costs between
// half a millisecond and twenty (19 of them were a third of a policy change of 4,096 workers).  A simulator keeps the block of
// a change of links for the next one, up to kKept bytes (with one allocation per change 600 workers took 4.7 ms
// instead of 4.1, 4,096 workers 34 instead of 31); whatever else it borrows is given back when the call ends.  For one caller at a time.
class DeviceArena {
 public:
  static constexpr size_t kKept = (size_t)512 << 20;
  DeviceArena() = default;
  DeviceArena(const DeviceArena&) = delete;
  DeviceArena& operator=(const DeviceArena&) = delete;
  ~DeviceArena() { release(); }
  // Starts over with room for `bytes`; whoever used the block before has finished (its stream has been waited for).
  bool begin(size_t bytes) {
    const uint64_t context = context_number();
    if (base_ && context != context_) base_ = nullptr;  // (it went with its context)
    used_ = 0;
    if (base_ && bytes <= size_) return true;
    release();
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    base_ = (unsigned char*)p;
    size_ = bytes;
    context_ = context;
    cudaGetDevice(&device_);
    return true;
  }
  static size_t room(size_t bytes) { return (bytes + 255) & ~(size_t)255; }
  template <typename T>
  T* take(size_t count) {
    T* at = (T*)(base_ + used_);
    used_ += room(count * sizeof(T));
    return at;
  }
  void end() {
    if (size_ > kKept) release();
  }
  void release() {
    if (base_) {
      int now = -1;
      cudaGetDevice(&now);
      if (now != device_) cudaSetDevice(device_);
      if (context_number() == context_) cudaFree(base_);
      if (now >= 0 && now != device_) cudaSetDevice(now);
      cudaGetLastError();
    }
    base_ = nullptr;
    size_ = 0;
  }

 private:
  unsigned char* base_ = nullptr;
  size_t size_ = 0, used_ = 0;
  uint64_t context_ = 0;
  int device_ = 0;
};
struct ArenaUse {  // of one call
  DeviceArena& arena;
  explicit ArenaUse(DeviceArena& a) : arena(a) {}
  ~ArenaUse() { arena.end(); }
};

// A whole policy change on the current device: link speeds (host) -> link graph and iteration times ->
// Algorithm 3.  The matrices stay on the device; *d_P is P there, in `arena`.
int policy_from_links_device(int32_t M, int64_t d, const double* speed, double lr, int32_t K, int32_t R, double rho_upper,
                             int device, cudaStream_t stream, DeviceArena& arena, double** d_P, uint8_t** d_adj,
                             double* rho);
// netmax_policy_generate_device with the caller's arena, on the current device.
int policy_generate_device(int32_t M, const double* t, const uint8_t* adj, double lr, int32_t K, int32_t R, double rho_upper,
                           cudaStream_t stream, DeviceArena& arena, double* prob_out, double* rho_out, double* info_out);

// The sampler's tables from P on the device: 32-bit cumulative thresholds, last positive entry and pull
// weight of every row, bit for bit what the host builds (the prefix sums run left to right).  d_adj: the
// link graph (symmetric).  alpha_rho: fp32 alpha times rho; pull_weight > 0: the same weight on every link.
cudaError_t build_tables_device(int32_t M, const double* d_P, const uint8_t* d_adj, double alpha_rho, double pull_weight,
                                uint32_t* thr, int32_t* last_nz, float* w, cudaStream_t stream);
}  // namespace netmax
