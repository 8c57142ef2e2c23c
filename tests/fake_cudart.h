// A CUDA runtime of two devices that runs nothing: it records each kernel's shared-memory limit per device
// and counts launches.  Linked with the library's object files (fake_util.py) to test their host code.
#pragma once
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <utility>

#include "common.cuh"

namespace {
thread_local int t_dev = 0;
std::mutex g_m;
std::map<std::pair<int, const void*>, int> g_limit;   // (device, kernel) -> dynamic shared memory allowed
int g_bad = 0, g_seen = 0, g_large = 0;
constexpr int kSms[2] = {152, 40};

cudaError_t launch(const void* k, size_t smem) {
  std::lock_guard<std::mutex> l(g_m);
  ++g_seen;
  if (smem > 48 * 1024) {
    ++g_large;
    const auto it = g_limit.find({t_dev, k});
    if (it == g_limit.end() || (size_t)it->second < smem) ++g_bad;
  }
  return cudaSuccess;
}
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = t_dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int d) {
  *v = a == cudaDevAttrMultiProcessorCount ? kSms[d] : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
  std::lock_guard<std::mutex> l(g_m);
  g_limit[{t_dev, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { return launch(f, c->dynamicSmemBytes); }
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void**, size_t smem, cudaStream_t) {
  return launch(f, smem);
}
static thread_local size_t t_smem;
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t smem, cudaStream_t) { t_smem = smem; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t* smem, void*) { *smem = t_smem; return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t) {
  return launch((const void*)k, smem);
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyToSymbol(const void*, const void*, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}

static bool check(const char* what, bool ok) {
  std::printf("%s %s\n", ok ? "ok" : "FAIL", what);
  return ok;
}
