// Helpers shared by the coarse CG kernels (kernels.cu, coarse_lat.cu, batched.cu): the clock of their
// bounded waits, the tagged-word exchange and block sums.
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

__device__ __forceinline__ double warp_total(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Block sums of three values, in every thread, fixed order; one warp adds through shared memory (few
// FP64 instructions).  buf: 3 blockDim.x values.  buf and res alternate between calls, so no
// barrier is needed before the writes.
__device__ __forceinline__ void block_sum3(double* buf, double* res, double& a, double& b, double& c) {
  const int T = blockDim.x;
  buf[threadIdx.x] = a;
  buf[T + threadIdx.x] = b;
  buf[2 * T + threadIdx.x] = c;
  __syncthreads();
  if (threadIdx.x < 32) {
    double t0 = 0.0, t1 = 0.0, t2 = 0.0;
    for (int q = threadIdx.x; q < T; q += 32) {
      t0 += buf[q];
      t1 += buf[T + q];
      t2 += buf[2 * T + q];
    }
    t0 = warp_total(t0);
    t1 = warp_total(t1);
    t2 = warp_total(t2);
    if (threadIdx.x == 0) {
      res[0] = t0;
      res[1] = t1;
      res[2] = t2;
    }
  }
  __syncthreads();
  a = res[0];
  b = res[1];
  c = res[2];
}

}  // namespace
}  // namespace chebmg
