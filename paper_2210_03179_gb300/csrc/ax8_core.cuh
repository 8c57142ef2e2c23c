// Building blocks of the order-7 element operator (N = 7, 8 GLL points per direction), shared
// by the operator kernels (sem_ax8.cu) and the fused smoother (sem_smooth8.cu): the shared-memory
// layout of one element, the even-odd line derivative and 8-point row loads / stores.
//
// Even-odd factorisation: the GLL derivative matrix is centro-antisymmetric,
// D[7-i][7-l] = -D[i][l], so (D u)[i] = E_i.(u_l + u_{7-l}) + O_i.(u_l - u_{7-l}) and
// (D u)[7-i] = O_i.(...) - E_i.(...) with 4 x 4 blocks E and O.  Each translation unit that
// includes this header has its own copy of the constant blocks and uploads them itself.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace chebmg {
namespace {

// even-odd blocks: [0] E of D, [1] O of D, [2] E of D^T, [3] O of D^T, each [i][l], i,l < 4
__constant__ float c_eo_f[4][4][4];
__device__ double g_eo_d[64];

template <typename T, int EB_ = 2>
struct Ax8 {
  static constexpr int EB = EB_;                       // elements per block
  static constexpr int R = 12;    // padded row stride (16-B aligned rows)
  static constexpr int P = 100;   // padded plane stride (see line_of)
  static constexpr int STAGE = 8 * P;
  static constexpr int GELEM = 6 * 512;
  static size_t smem_bytes() { return sizeof(T) * (size_t)EB * (GELEM + 3 * STAGE); }
};

// The line coefficients as a kernel uses them: FP32 constant-bank operands; FP64 in shared memory
// (an FP64 FMA issues faster with register operands than with constant ones, see Fp64Unit), rows
// loaded 16 bytes at a time where they are used.  Every thread of the block (64 at least) calls the
// constructor, which only fetches, and then stage(); a block barrier separates stage() from the first
// line8.  A kernel that gathers first stages after it, so that the fetch is in flight with the gather:
// on 8 to 64 elements a product took 0.1 to 1.0 us less (order-4 smoother from an iterate on 64
// elements, best variant 68.3 -> 67.3 us, one element per block with bulk copies 72.6 -> 68.9), on 32^3
// nothing changed.
template <typename T>
struct Coef8;
template <>
struct Coef8<float> : Arith<float> {
  static constexpr int SHARED = 1;
  __device__ __forceinline__ Coef8() {}
  __device__ __forceinline__ void stage(float*) {}
  template <int W>
  __device__ __forceinline__ void row(int i, float (&v)[4]) const {
#pragma unroll
    for (int l = 0; l < 4; ++l) v[l] = c_eo_f[W][i][l];
  }
};
template <>
struct Coef8<double> : Arith<double> {
  static constexpr int SHARED = 64;
  const double* t;
  double mine;
  __device__ __forceinline__ Coef8() : t(nullptr), mine(threadIdx.x < 64 ? __ldg(&g_eo_d[threadIdx.x]) : 0.0) {}
  __device__ __forceinline__ void stage(double* sh) {
    t = sh;
    if (threadIdx.x < 64) sh[threadIdx.x] = mine;
  }
  template <int W>
  __device__ __forceinline__ void row(int i, double (&v)[4]) const {
    const double2* p = reinterpret_cast<const double2*>(t + W * 16 + i * 4);
    const double2 a = p[0], b = p[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
  }
};

// o = D u (W = 0) or o = D^T u (W = 1) along one line of 8 points.
template <typename T, int W>
__device__ __forceinline__ void line8(const Coef8<T>& c, const T (&u)[8], T (&o)[8]) {
  T ue[4], uo[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    ue[l] = c.add(u[l], u[7 - l]);
    uo[l] = c.sub(u[l], u[7 - l]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    T e[4], d[4];
    c.template row<2 * W>(i, e);
    c.template row<2 * W + 1>(i, d);
    T se = c.mul(e[0], ue[0]);
#pragma unroll
    for (int l = 1; l < 4; ++l) se = fma(e[l], ue[l], se);
    if constexpr (sizeof(T) == 8) {
      // FP64 (bound by its FP64 issue rate): the odd chain continues from se, giving
      // o[i] = se + so directly, and o[7-i] = so - se = o[i] - 2 se in one more FMA
      // (9 operations per output pair instead of 10)
      T s = se;
#pragma unroll
      for (int l = 0; l < 4; ++l) s = fma(d[l], uo[l], s);
      o[i] = s;
      o[7 - i] = fma(c.k.m2, se, s);
    } else {
      T so = d[0] * uo[0];
#pragma unroll
      for (int l = 1; l < 4; ++l) so = fma(d[l], uo[l], so);
      o[i] = se + so;
      o[7 - i] = so - se;
    }
  }
}

// The three weighted derivatives at a point: (G row) . (ur, us, ut).
template <typename T>
__device__ __forceinline__ T dot3(const Coef8<T>& c, T g0, T a0, T g1, T a1, T g2, T a2) {
  return fma(g2, a2, fma(g1, a1, c.mul(g0, a0)));
}

__device__ __forceinline__ void ld_row(const float* p, float (&v)[8]) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void st_row(float* p, const float (&v)[8]) {
  reinterpret_cast<float4*>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
  reinterpret_cast<float4*>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void ld_row(const double* p, double (&v)[8]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const double2 a = reinterpret_cast<const double2*>(p)[q];
    v[2 * q] = a.x;
    v[2 * q + 1] = a.y;
  }
}
__device__ __forceinline__ void st_row(double* p, const double (&v)[8]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) reinterpret_cast<double2*>(p)[q] = make_double2(v[2 * q], v[2 * q + 1]);
}


}  // namespace
}  // namespace chebmg
