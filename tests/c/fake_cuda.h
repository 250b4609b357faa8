// The part of the CUDA runtime that the library calls, on the host: memory is
// the host's, kernels are not run but listed by name, and a call can be made to
// fail. Linked in place of the runtime, it lets a CPU program drive the
// library's host code through paths a healthy GPU does not take.
#pragma once

#include <cuda_runtime_api.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>
#include <vector>

struct Launch {
  std::string kernel;
  std::vector<unsigned char> arg;  // the first parameter, if its size was asked for
};
inline std::vector<Launch> g_launches;
inline std::map<std::string, size_t> g_keep;      // kernel name -> bytes of its first parameter to keep
inline std::map<std::string, int> g_fail_at;      // call -> which of its next calls runs out of memory (1: the next)
inline std::map<std::string, int> g_calls;
inline bool g_capturing = false;
inline std::vector<size_t> g_allocs;              // sizes, in order
inline std::map<const void*, std::string> g_names;

inline cudaError_t fake_call(const char* name) {
  g_calls[name]++;
  auto f = g_fail_at.find(name);
  if (f != g_fail_at.end() && f->second > 0 && --f->second == 0) return cudaErrorMemoryAllocation;
  return cudaSuccess;
}

inline cudaError_t fake_launch(const void* fn, void** args) {
  const cudaError_t e = fake_call("launch");
  if (e != cudaSuccess) return e;
  Launch l{g_names[fn], {}};
  for (const auto& k : g_keep)
    if (l.kernel.find(k.first) != std::string::npos) {
      const unsigned char* a = static_cast<const unsigned char*>(args[0]);
      l.arg.assign(a, a + k.second);
    }
  g_launches.push_back(l);
  return cudaSuccess;
}

inline int launches_of(const char* kernel) {
  int n = 0;
  for (const auto& l : g_launches) n += l.kernel.find(kernel) != std::string::npos;
  return n;
}

extern "C" {
struct FakeConfig {
  dim3 g, b;
  size_t smem;
  cudaStream_t st;
};
static FakeConfig g_config;

void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* st) {
  g_config = FakeConfig{g, b, smem, st};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
  *g = g_config.g;
  *b = g_config.b;
  *smem = g_config.smem;
  *static_cast<cudaStream_t*>(st) = g_config.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t) const_cast<void*>(f);
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t) {
  return fake_launch(k, args);
}
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void** args, size_t, cudaStream_t) { return fake_launch(f, args); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* f, void** args) { return fake_launch(f, args); }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = (cudaEvent_t)malloc(1);
  return fake_call("cudaEventCreate");
}
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  free(e);
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) {
  const cudaError_t e = fake_call("cudaMallocAsync");
  if (e != cudaSuccess) return e;
  g_allocs.push_back(n);
  *p = aligned_alloc(256, (n + 255) / 256 * 256);
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  const cudaError_t e = fake_call("cudaMemcpyAsync");
  if (e == cudaSuccess) memcpy(d, s, n);
  return e;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  alignas(256) static unsigned char scratch[1 << 20];
  *p = scratch;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)1;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamGetDevice(cudaStream_t, int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
  *c = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
}
