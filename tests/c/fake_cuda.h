// fake_cuda.h -- the CUDA runtime calls that csrc/api.cu makes, on host memory,
// for tests of the planner and the C ABI's host code without a GPU.
//
// A copy or fill that CUDA may finish after the call has returned is kept
// pending and done when something waits for it: cudaMemcpy from pageable host
// memory to the device (documented to return once the bytes are staged) and
// cudaMemset (asynchronous to the host) run on the legacy stream, which a
// non-blocking stream is not ordered after.  Device memory starts as 0xCD.
#pragma once

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <utility>
#include <vector>

#include <cuda_runtime.h>

namespace fake {
inline int sm_count = 152;
inline std::vector<std::pair<cudaStream_t, std::function<void()>>> pending;  // (the stream, what it still does), in order

inline cudaStream_t norm(cudaStream_t s) { return s == cudaStreamLegacy ? nullptr : s; }
inline void later(cudaStream_t s, std::function<void()> work) { pending.emplace_back(norm(s), std::move(work)); }
inline void finish(cudaStream_t s) {
  std::vector<std::pair<cudaStream_t, std::function<void()>>> rest;
  for (auto& w : pending) {
    if (w.first == norm(s)) w.second();
    else rest.push_back(w);
  }
  pending.swap(rest);
}
inline void finish_all() {
  for (auto& w : pending) w.second();
  pending.clear();
}
}  // namespace fake

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = fake::sm_count; return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = std::malloc(n);
  if (*p == nullptr) return cudaErrorMemoryAllocation;
  std::memset(*p, 0xCD, n);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) { fake::finish_all(); std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind kind) {
  fake::finish(nullptr);
  if (kind != cudaMemcpyHostToDevice) {
    std::memcpy(d, s, n);
    return cudaSuccess;
  }
  const uint8_t* b = static_cast<const uint8_t*>(s);
  fake::later(nullptr, [d, staged = std::vector<uint8_t>(b, b + n)] { std::memcpy(d, staged.data(), staged.size()); });
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
  fake::later(st, [=] { std::memcpy(d, s, n); });
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { fake::later(nullptr, [=] { std::memset(d, v, n); }); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
  fake::later(st, [=] { std::memset(d, v, n); });
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { fake::finish(s); return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { fake::finish_all(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = reinterpret_cast<cudaEvent_t>(1); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
}

#include "kernels.h"

// The kernels' launchers: nothing runs.
namespace frk {
cudaError_t configure_sweep_fp() { return cudaSuccess; }
cudaError_t configure_sweep_pack() { return cudaSuccess; }
cudaError_t configure_sweep_unpack() { return cudaSuccess; }
cudaError_t configure_sweep_unpack_fp() { return cudaSuccess; }
cudaError_t launch_sweep_fp(const SweepParams&, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_sweep_pack(const SweepParams&, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_sweep_unpack(const SweepParams&, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_sweep_unpack_fp(const SweepParams&, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_list_pack(const ListParams&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_list_unpack(const ListParams&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_list_unpack_fp(const ListParams&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_finalize(int, const FinalizeParams&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_compact_flags(const uint8_t*, uint64_t, uint32_t*, uint64_t, uint64_t*, uint32_t*, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_diff(const FpEntry*, const FpEntry*, uint64_t, uint32_t*, uint64_t, uint64_t*, cudaStream_t) {
  return cudaSuccess;
}
}  // namespace frk
