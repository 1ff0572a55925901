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

// Device memory of one call.
class DeviceBuffers {
 public:
  ~DeviceBuffers() {
    for (void* p : ptrs_) cudaFree(p);
  }
  template <typename T>
  bool get(T** out, size_t count) {
    void* p = nullptr;
    if (cudaMalloc(&p, count * sizeof(T)) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    ptrs_.push_back(p);
    *out = (T*)p;
    return true;
  }

 private:
  std::vector<void*> ptrs_;
};

// A whole policy change on the current device: link speeds (host) -> link graph and iteration times ->
// Algorithm 3.  The matrices stay on the device; *d_P is P there, owned by `buf`.
int policy_from_links_device(int32_t M, int64_t d, const double* speed, double lr, int32_t K, int32_t R, double rho_upper,
                             int device, cudaStream_t stream, DeviceBuffers& buf, double** d_P, uint8_t** d_adj,
                             double* rho);

// The sampler's tables from P on the device: 32-bit cumulative thresholds, last positive entry and pull
// weight of every row, bit for bit what the host builds (the prefix sums run left to right).  d_adj: the
// link graph (symmetric).  alpha_rho: fp32 alpha times rho; pull_weight > 0: the same weight on every link.
cudaError_t build_tables_device(int32_t M, const double* d_P, const uint8_t* d_adj, double alpha_rho, double pull_weight,
                                uint32_t* thr, int32_t* last_nz, float* w, cudaStream_t stream);
}  // namespace netmax
