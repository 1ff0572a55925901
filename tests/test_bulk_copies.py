"""Large host transfers (netmax_bulk.h) against a CUDA runtime of a few lines on the host: whole and ragged sizes, both
directions, and a runtime that locks no memory or creates no stream (the copies are then made all the same), and a device reset in between."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_05766_b200", "csrc")

RUNTIME = r"""
// as much of the CUDA runtime's interface as netmax_bulk.h uses; copies are made at once
#pragma once
#include <atomic>
#include <cstdlib>
#include <cstring>
typedef int cudaError_t;
constexpr int cudaSuccess = 0, cudaErrorMemoryAllocation = 2;
typedef int* cudaStream_t;
typedef int* cudaEvent_t;
enum cudaMemcpyKind { cudaMemcpyHostToDevice = 1, cudaMemcpyDeviceToHost = 2 };
constexpr unsigned cudaHostAllocPortable = 1, cudaStreamNonBlocking = 1, cudaEventDisableTiming = 2;
inline std::atomic<int> locked_left{0}, streams_left{0}, locked{0}, streams{0}, copies{0};
inline cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  if (locked_left-- <= 0) return cudaErrorMemoryAllocation;
  ++locked;
  *p = std::malloc(n);
  return cudaSuccess;
}
inline cudaError_t cudaFreeHost(void* p) { --locked; std::free(p); return cudaSuccess; }
inline cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  if (streams_left-- <= 0) return cudaErrorMemoryAllocation;
  ++streams;
  *s = new int(0);
  return cudaSuccess;
}
inline cudaError_t cudaStreamDestroy(cudaStream_t s) { --streams; delete s; return cudaSuccess; }
inline cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
inline cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = new int(0); return cudaSuccess; }
inline cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
inline cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
inline cudaError_t cudaEventDestroy(cudaEvent_t e) { delete e; return cudaSuccess; }
inline cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { ++copies; std::memcpy(d, s, n); return cudaSuccess; }
typedef int cudaDriverEntryPointQueryResult;
constexpr int cudaEnableDefault = 0;
inline unsigned long long context = 1;
inline int context_id(void*, unsigned long long* id) { *id = context; return 0; }
inline cudaError_t cudaGetDriverEntryPoint(const char*, void** f, int, int*) { *f = (void*)context_id; return cudaSuccess; }
inline cudaError_t cudaSetDevice(int) { return cudaSuccess; }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
"""

PROGRAM = r"""
#include <cstdio>
#include "netmax_bulk.h"
using namespace netmax;

int main() {
  for (int locks : {0, 100})
    for (int some_streams : {0, 2, 100}) {
      BulkPool& pool = BulkPool::get();
      for (size_t bytes : {size_t(1), size_t(1000), (size_t(1) << 20) - 1, (size_t(5) << 20) + 17, size_t(23) << 20}) {
        locked_left = locks;
        streams_left = some_streams;
        std::vector<unsigned char> src(bytes), up(bytes, 0), down(bytes, 0);
        for (size_t k = 0; k < bytes; ++k) src[k] = (unsigned char)(k * 2654435761u >> 13);
        if (pool.to_device(up.data(), src.data(), bytes, 0, nullptr) != cudaSuccess) return std::printf("up: %zu\n", bytes), 1;
        if (pool.to_host(down.data(), up.data(), bytes, 0, nullptr) != cudaSuccess) return std::printf("down: %zu\n", bytes), 1;
        if (up != src || down != src) return std::printf("copy: %zu\n", bytes), 1;
      }
    }
  // a device reset takes the locked memory and the streams with it: what is kept from before is not touched again
  locked_left = streams_left = 1000;
  std::vector<unsigned char> src(1 << 20, 7), up(1 << 20);
  const int held = locked, open = streams;
  if (held < 1) return std::printf("nothing was kept\n"), 1;
  context = 2;
  for (int k = 0; k < 3; ++k)
    if (BulkPool::get().to_device(up.data(), src.data(), up.size(), 0, nullptr) != cudaSuccess || up != src) return std::printf("after a reset\n"), 1;
  if (locked != held + 1 || streams != open + 4) return std::printf("%d blocks, %d streams\n", (int)locked, (int)streams), 1;
  std::printf("fine\n");
  return 0;
}
"""


def test_copies_are_made_with_and_without_locked_memory(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    src, exe = tmp_path / "copies.cpp", tmp_path / "copies"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", str(tmp_path), "-I", CSRC, str(src), "-o", str(exe)], check=True)
    done = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert done.returncode == 0 and done.stdout.strip() == "fine", done.stdout
