// Host code of the operator files against a fake CUDA runtime with two devices (compiled and run by
// test_per_device.py): what a launch needs on a device must have been set on that device.
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <thread>
#include <utility>
#include <vector>

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

using namespace chebmg;

static const char* check(const char* what, bool ok) {
  std::printf("%s %s\n", ok ? "ok" : "FAIL", what);
  return ok ? nullptr : what;
}

template <typename T>
static void operators(int64_t E, const Lattice& lat) {
  for (int Q : {3, 5, 6, 7, 9, 10})
    for (const Lattice* l : {&lat, static_cast<const Lattice*>(nullptr)})
      sem_axl<T>(Q, E, nullptr, l, static_cast<const T*>(nullptr), nullptr, nullptr, nullptr);
  for (int v : {1, 2, 4, 12, 14, 21, 22, 31, 32, 101, 102, 104, 112, 114, 121, 122, 131, 132})
    if (sem_ax8_variant_fits<T>(v)) sem_ax8<T>(E, nullptr, lat, static_cast<const T*>(nullptr), nullptr, nullptr, nullptr, v, nullptr);
  for (int v : {1, 2, 4, 11, 12, 21, 22, 101, 102, 104, 111, 112, 121, 122})
    if (sem_ax8_batched_fits<T>(2000 + v))
      sem_ax8_batched<T>(E, nullptr, lat, static_cast<const T*>(nullptr), nullptr, nullptr, nullptr, 2000 + v, 4, 512, nullptr);
}

static void all() {
  Lattice lat{};
  lat.nex = lat.ney = lat.nez = 16;
  for (int64_t E : {(int64_t)30, (int64_t)4096}) {
    operators<float>(E, lat);
    operators<double>(E, lat);
  }
  for (int v : {1, 2, 4, 101, 102, 104})
    sem_ax8_x2(4096, nullptr, lat, nullptr, nullptr, nullptr, nullptr, v, nullptr);
}

int main() {
  bool bad = false;
  // one device after the other, in one process
  for (int d : {0, 1}) {
    t_dev = d;
    const int before = g_bad, large = g_large;
    all();
    char msg[64];
    std::snprintf(msg, sizeof msg, "shared-memory limits on device %d", d);
    bad |= check(msg, g_bad == before && g_large > large) != nullptr;
  }
  // sizes that follow the device's SM count
  for (int d : {0, 1, 0}) {
    t_dev = d;
    int grid = 0, rows = 0;
    coarse_pcg_shape(30000, 1, &grid, &rows);
    char msg[64];
    std::snprintf(msg, sizeof msg, "rows per coarse block on device %d: %d", d, rows);
    bad |= check(msg, rows == (d == 0 ? 256 : 1024)) != nullptr;
    std::snprintf(msg, sizeof msg, "FP64 order-5 kernel of 300 elements on device %d", d);
    bad |= check(msg, sem_axl_chosen<double>(6, 300) == (d == 1)) != nullptr;
    std::snprintf(msg, sizeof msg, "lattice coarse blocks of 256 rows on device %d", d);
    bad |= check(msg, coarse_lat_fits(30000, 31, 256) == (d == 0)) != nullptr;
  }
  // both at once: several threads start together on fresh limits of both devices
  {
    std::vector<std::thread> th;
    const int before = g_bad;
    for (int q = 0; q < 8; ++q)
      th.emplace_back([q] {
        t_dev = q & 1;
        all();
      });
    for (auto& t : th) t.join();
    bad |= check("eight threads on two devices", g_bad == before) != nullptr;
  }
  std::printf("launches %d, with large blocks %d\n", g_seen, g_large);
  return bad ? 1 : 0;
}
