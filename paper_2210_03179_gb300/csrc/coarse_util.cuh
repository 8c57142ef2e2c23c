// Helpers shared by the persistent coarse CG kernels (kernels.cu, coarse_lat.cu): the clock of their
// bounded waits and the tagged-word exchange.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace chebmg {
namespace {

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
constexpr uint64_t kWaitNs = 1000000000ull;   // every wait gives up after about a second

// ---- tagged-word exchange ----
__device__ __forceinline__ void st_tagged(unsigned long long* p, unsigned long long w) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ void st_tagged2(unsigned long long* p, unsigned long long w0, unsigned long long w1) {
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(w0), "l"(w1) : "memory");
}
__device__ __forceinline__ unsigned long long ld_tagged(const unsigned long long* p) {
  unsigned long long w;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ void ld_tagged2(const unsigned long long* p, unsigned long long& w0,
                                           unsigned long long& w1) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(w0), "=l"(w1) : "l"(p) : "memory");
}
// One exchanged value: FP32 in one tagged word, FP64 as two (high and low halves, loaded
// and stored together; each half carries the tag, so a torn pair is never accepted).
template <typename V>
struct Tagged;
template <>
struct Tagged<float> {
  struct W {
    unsigned long long w;
  };
  static __device__ __forceinline__ unsigned long long* buf(const CoarseCG& a, unsigned gx) {
    return a.exf[gx & 1u];
  }
  static __device__ __forceinline__ void store(unsigned long long* b, int64_t g, unsigned tag, float v) {
    st_tagged(b + g, ((unsigned long long)tag << 32) | __float_as_uint(v));
  }
  static __device__ __forceinline__ W load(const unsigned long long* b, int64_t g) { return {ld_tagged(b + g)}; }
  static __device__ __forceinline__ bool ready(const W& w, unsigned tag) { return (unsigned)(w.w >> 32) == tag; }
  static __device__ __forceinline__ float value(const W& w) { return __uint_as_float((unsigned)w.w); }
  static __device__ __forceinline__ float coef(const CoarseCG& a, int64_t i) { return __ldg(&a.valf[i]); }
};
template <>
struct Tagged<double> {
  struct W {
    unsigned long long hi, lo;
  };
  static __device__ __forceinline__ unsigned long long* buf(const CoarseCG& a, unsigned gx) {
    return a.exd[gx & 1u];
  }
  static __device__ __forceinline__ void store(unsigned long long* b, int64_t g, unsigned tag, double v) {
    const unsigned long long t = (unsigned long long)tag << 32;
    st_tagged2(b + 2 * g, t | (unsigned)__double2hiint(v), t | (unsigned)__double2loint(v));
  }
  static __device__ __forceinline__ W load(const unsigned long long* b, int64_t g) {
    W w;
    ld_tagged2(b + 2 * g, w.hi, w.lo);
    return w;
  }
  static __device__ __forceinline__ bool ready(const W& w, unsigned tag) {
    return (unsigned)(w.hi >> 32) == tag && (unsigned)(w.lo >> 32) == tag;
  }
  static __device__ __forceinline__ double value(const W& w) {
    return __hiloint2double((int)(unsigned)w.hi, (int)(unsigned)w.lo);
  }
  static __device__ __forceinline__ double coef(const CoarseCG& a, int64_t i) { return __ldg(&a.val[i]); }
};

}  // namespace
}  // namespace chebmg
