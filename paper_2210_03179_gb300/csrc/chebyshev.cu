// Chebyshev recurrences (Algorithms 1 and 2) and the vector updates of the smoother: the
// elementwise pass that follows each operator application.  Every kernel also takes a batch
// of right-hand sides (vector q at q * ld; per-node data such as S shared).
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace chebmg {

namespace {

inline unsigned grid_for(int64_t n, int bs) {
  int64_t g = (n + bs - 1) / bs;
  if (g > 4096 * 152) g = 4096 * 152;
  if (g < 1) g = 1;
  return (unsigned)g;
}

}  // namespace

// ===========================================================================
// Chebyshev recurrences and vector updates
// ===========================================================================
// Vector type of 16 bytes for T (float4 / double2) and its lane count.
template <typename T>
struct V16;
template <>
struct V16<float> {
  using type = float4;
  static constexpr int L = 4;
};
template <>
struct V16<double> {
  using type = double2;
  static constexpr int L = 2;
};

// The adjoint's forward recurrence (SEM) and the context-free FD smoother: separate product vector y.
// 4th-kind init: x = 0, r = b (x_is_zero) or r = b - y, y = 0; then d = c0 S r.  VEC: 16-byte accesses
// over the aligned body, scalar tail.
template <typename T, bool VEC>
__global__ void k_cheb4_init(int64_t n, const T* __restrict__ b, T* __restrict__ x, T* __restrict__ r,
                             T* __restrict__ d, T* __restrict__ y, const T* __restrict__ invD, T c0,
                             int x_is_zero, int64_t ld) {
  pdl_wait();
  { const int64_t off_ = (int64_t)blockIdx.y * ld; b += off_; x += off_; r += off_; d += off_; y += off_; }
  using VT = typename V16<T>::type;
  constexpr int L = V16<T>::L;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t nv = VEC ? n / L : 0;
  for (int64_t q = tid; q < nv; q += stride) {
    const VT bv = reinterpret_cast<const VT*>(b)[q], sv = reinterpret_cast<const VT*>(invD)[q];
    const T* bs = reinterpret_cast<const T*>(&bv);
    const T* ss = reinterpret_cast<const T*>(&sv);
    VT rv, dv;
    T* rs = reinterpret_cast<T*>(&rv);
    T* ds = reinterpret_cast<T*>(&dv);
    if (x_is_zero) {
#pragma unroll
      for (int l = 0; l < L; ++l) rs[l] = bs[l];
      reinterpret_cast<VT*>(x)[q] = VT{};
    } else {
      const VT yv = reinterpret_cast<const VT*>(y)[q];
      const T* ys = reinterpret_cast<const T*>(&yv);
#pragma unroll
      for (int l = 0; l < L; ++l) rs[l] = bs[l] - ys[l];
      reinterpret_cast<VT*>(y)[q] = VT{};
    }
#pragma unroll
    for (int l = 0; l < L; ++l) ds[l] = c0 * ss[l] * rs[l];
    reinterpret_cast<VT*>(r)[q] = rv;
    reinterpret_cast<VT*>(d)[q] = dv;
  }
  for (int64_t g = nv * L + tid; g < n; g += stride) {
    T rv;
    if (x_is_zero) {
      rv = b[g];
      x[g] = T(0);
    } else {
      rv = b[g] - y[g];
      y[g] = T(0);
    }
    r[g] = rv;
    d[g] = c0 * invD[g] * rv;
  }
}


template <typename T>
__device__ __forceinline__ void cheb4_one(T& x, T& r, T& d, T& y, T s, T beta, T c1, T c2) {
  const T dv = d;
  const T rv = r - y;
  x += beta * dv;
  r = rv;
  d = c1 * dv + c2 * s * rv;
  y = T(0);
}

// 16-byte global accesses with an L2 eviction hint.  The update streams x, r and S (evict
// first) and keeps d and y in L2 (evict last): the next operator application gathers d and
// accumulates into y, so they should still be there when it runs.
__device__ __forceinline__ uint64_t l2_policy_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t l2_policy_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
template <typename VT>
__device__ __forceinline__ VT ld16(const VT* p, uint64_t pol) {
  uint4 v;
  asm volatile("ld.global.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p), "l"(pol));
  return *reinterpret_cast<VT*>(&v);
}
template <typename VT>
__device__ __forceinline__ void st16(VT* p, const VT& val, uint64_t pol) {
  const uint4 v = *reinterpret_cast<const uint4*>(&val);
  asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z),
               "r"(v.w), "l"(pol)
               : "memory");
}

// x += beta d; r -= y; d = c1 d + c2 S r; y = 0.
template <typename T, bool VEC>
__global__ void k_cheb4_step(int64_t n, T* __restrict__ x, T* __restrict__ r, T* __restrict__ d,
                             T* __restrict__ y, const T* __restrict__ invD, T beta, T c1, T c2, int64_t ld) {
  // Everything read here is the operator kernel's output or older: wait for that kernel before
  // the first load.  (Triggering the next kernel early as well, griddepcontrol.launch_dependents,
  // was measured slower: its waiting blocks cost this grid's last wave more than they saved.)
  pdl_wait();
  { const int64_t off_ = (int64_t)blockIdx.y * ld; x += off_; r += off_; d += off_; y += off_; }
  using VT = typename V16<T>::type;
  constexpr int L = V16<T>::L;
  const int64_t nv = VEC ? n / L : 0;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const uint64_t first = l2_policy_first(), last = l2_policy_last();
  for (int64_t q = tid; q < nv; q += stride) {
    VT xv = ld16(reinterpret_cast<VT*>(x) + q, first), rv = ld16(reinterpret_cast<VT*>(r) + q, first);
    VT dv = ld16(reinterpret_cast<VT*>(d) + q, last), yv = ld16(reinterpret_cast<VT*>(y) + q, last);
    const VT sv = ld16(reinterpret_cast<const VT*>(invD) + q, first);
    T* xs = reinterpret_cast<T*>(&xv);
    T* rs = reinterpret_cast<T*>(&rv);
    T* ds = reinterpret_cast<T*>(&dv);
    T* ys = reinterpret_cast<T*>(&yv);
    const T* ss = reinterpret_cast<const T*>(&sv);
#pragma unroll
    for (int l = 0; l < L; ++l) cheb4_one<T>(xs[l], rs[l], ds[l], ys[l], ss[l], beta, c1, c2);
    st16(reinterpret_cast<VT*>(x) + q, xv, first);
    st16(reinterpret_cast<VT*>(r) + q, rv, first);
    st16(reinterpret_cast<VT*>(d) + q, dv, last);
    st16(reinterpret_cast<VT*>(y) + q, yv, last);
  }
  for (int64_t g = nv * L + tid; g < n; g += stride)
    cheb4_one<T>(x[g], r[g], d[g], y[g], invD[g], beta, c1, c2);
}

// ---- SEM smoothing: the operator subtracts A d from r in place ----
// Bytes bound these kernels.  Against the form with a product vector y (y zeroed, accumulated,
// read back and zeroed again, r rewritten) a step moves 4 n-vectors instead of 8 beside the x
// update, and x is touched every other step only: a step has both d_{i-1} and d_i at hand.
// Measured on 32^3 elements of order 7, order 6 from a zero guess, FP32: 748.7 -> 614.7 us; a whole
// mixed solve of that size 33.19 -> 31.60 ms; 64 right-hand sides on 8^3 elements 28.73 -> 27.43 ms.

// Zero guess: r = b (rin = b), d = c0 S b; or (from_r) from the residual r: d = c0 S r.  order1:
// x = w d (x += w d from a residual) instead of storing d.  b_next leaves r = b_next for the
// restriction residual.  rin and x may be one buffer (a caller's b and x), rin and r as well.
template <typename T, bool VEC>
__global__ void k_smooth_begin(int64_t n, const T* rin, T* x, T* r, T* __restrict__ d,
                               const T* __restrict__ invD, T c0, T w, int from_r, int order1, const T* b_next, int64_t ld) {
  pdl_wait();
  { const int64_t off_ = (int64_t)blockIdx.y * ld; rin += off_; x += off_; r += off_; d += off_; if (b_next) b_next += off_; }
  using VT = typename V16<T>::type;
  constexpr int L = V16<T>::L;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t nv = VEC ? n / L : 0;
  const uint64_t last = l2_policy_last();
  for (int64_t q = tid; q < nv; q += stride) {
    VT rv = reinterpret_cast<const VT*>(rin)[q], dv, xv = {};
    const VT sv = reinterpret_cast<const VT*>(invD)[q];
    if (order1 && from_r) xv = reinterpret_cast<const VT*>(x)[q];
    if (b_next && from_r) {
      const VT bv = reinterpret_cast<const VT*>(b_next)[q];
      st16(reinterpret_cast<VT*>(r) + q, bv, last);
    } else if (!from_r && (b_next || !order1)) {
      st16(reinterpret_cast<VT*>(r) + q, rv, last);
    }
    T* rs = reinterpret_cast<T*>(&rv);
    T* ds = reinterpret_cast<T*>(&dv);
    T* xs = reinterpret_cast<T*>(&xv);
    const T* ss = reinterpret_cast<const T*>(&sv);
#pragma unroll
    for (int l = 0; l < L; ++l) {
      ds[l] = c0 * ss[l] * rs[l];
      xs[l] = from_r ? xs[l] + w * ds[l] : w * ds[l];
    }
    if (order1) reinterpret_cast<VT*>(x)[q] = xv;
    else st16(reinterpret_cast<VT*>(d) + q, dv, last);
  }
  for (int64_t g = nv * L + tid; g < n; g += stride) {
    const T rv = rin[g], dv = c0 * invD[g] * rv;
    if (b_next && from_r) r[g] = b_next[g];
    else if (!from_r && (b_next || !order1)) r[g] = rv;
    if (!order1) d[g] = dv;
    else x[g] = from_r ? x[g] + w * dv : w * dv;
  }
}

// One recurrence step: d' = c1 d + c2 S r, then (XM) x += or = w0 d + w1 d'.  LAST: d' is not
// stored (nothing reads it).
template <typename T, bool VEC, int XM, bool LAST>
__global__ void k_smooth_step(int64_t n, T* __restrict__ x, T* __restrict__ r, T* __restrict__ d,
                              const T* __restrict__ invD, T c1, T c2, T w0, T w1, const T* __restrict__ b_next,
                              int64_t ld) {
  // Triggering the next kernel early (griddepcontrol.launch_dependents) was measured slower: its
  // waiting blocks cost this grid's last wave more than they saved.
  pdl_wait();
  { const int64_t off_ = (int64_t)blockIdx.y * ld; x += off_; r += off_; d += off_; if (b_next) b_next += off_; }
  using VT = typename V16<T>::type;
  constexpr int L = V16<T>::L;
  const int64_t nv = VEC ? n / L : 0;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const uint64_t first = l2_policy_first(), last = l2_policy_last();
  auto one = [&](T& xg, T& dg, T rg, T sg) {
    const T dn = c1 * dg + c2 * sg * rg;
    if (XM == SX_ADD) xg = (xg + w0 * dg) + w1 * dn;
    if (XM == SX_SET) xg = w0 * dg + w1 * dn;
    dg = dn;
  };
  for (int64_t q = tid; q < nv; q += stride) {
    VT xv = {}, rv = ld16(reinterpret_cast<const VT*>(r) + q, last);
    VT dv = ld16(reinterpret_cast<const VT*>(d) + q, last);
    if (XM == SX_ADD) xv = ld16(reinterpret_cast<const VT*>(x) + q, first);
    const VT sv = ld16(reinterpret_cast<const VT*>(invD) + q, first);
    VT bv = {};
    if (LAST && b_next) bv = ld16(reinterpret_cast<const VT*>(b_next) + q, first);
    T* xs = reinterpret_cast<T*>(&xv);
    T* ds = reinterpret_cast<T*>(&dv);
    const T* rs = reinterpret_cast<const T*>(&rv);
    const T* ss = reinterpret_cast<const T*>(&sv);
#pragma unroll
    for (int l = 0; l < L; ++l) one(xs[l], ds[l], rs[l], ss[l]);
    if (XM != SX_NONE) st16(reinterpret_cast<VT*>(x) + q, xv, LAST ? last : first);
    if (!LAST) st16(reinterpret_cast<VT*>(d) + q, dv, last);
    if (LAST && b_next) st16(reinterpret_cast<VT*>(r) + q, bv, last);
  }
  for (int64_t g = nv * L + tid; g < n; g += stride) {
    T xg = XM == SX_ADD ? x[g] : T(0), dg = d[g];
    one(xg, dg, r[g], invD[g]);
    if (XM != SX_NONE) x[g] = xg;
    if (!LAST) d[g] = dg;
    if (LAST && b_next) r[g] = b_next[g];
  }
}

template <typename T>
__global__ void k_cheb1_init(int64_t n, const T* __restrict__ b, T* __restrict__ x, T* __restrict__ r,
                             T* __restrict__ d, T* __restrict__ y, const T* __restrict__ invD,
                             T inv_theta, int x_is_zero, int64_t ld) {
  pdl_wait();
  { const int64_t off_ = (int64_t)blockIdx.y * ld; b += off_; x += off_; r += off_; d += off_; y += off_; }
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < n; g += (int64_t)gridDim.x * blockDim.x) {
    T rv;
    if (x_is_zero) {
      rv = invD[g] * b[g];
      x[g] = T(0);
    } else {
      rv = invD[g] * (b[g] - y[g]);
      y[g] = T(0);
    }
    r[g] = rv;
    d[g] = rv * inv_theta;
  }
}

template <typename T>
__global__ void k_cheb1_step(int64_t n, T* __restrict__ x, T* __restrict__ r, T* __restrict__ d,
                             T* __restrict__ y, const T* __restrict__ invD, T c1, T c2, int64_t ld) {
  pdl_wait();
  { const int64_t off_ = (int64_t)blockIdx.y * ld; x += off_; r += off_; d += off_; y += off_; }
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < n; g += (int64_t)gridDim.x * blockDim.x) {
    const T dv = d[g];
    const T rv = r[g] - invD[g] * y[g];
    x[g] += dv;
    r[g] = rv;
    d[g] = c1 * dv + c2 * rv;
    y[g] = T(0);
  }
}

template <typename T>
__global__ void k_axpy(int64_t n, T a, const T* __restrict__ d, T* __restrict__ x, int64_t ld) {
  pdl_wait();
  { const int64_t off_ = (int64_t)blockIdx.y * ld; d += off_; x += off_; }
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < n; g += (int64_t)gridDim.x * blockDim.x)
    x[g] += a * d[g];
}

template <typename Tin, typename Tout>
__global__ void k_cast(int64_t n, const Tin* __restrict__ in, Tout* __restrict__ out, int64_t ldi, int64_t ldo) {
  pdl_wait();
  in += (int64_t)blockIdx.y * ldi;
  out += (int64_t)blockIdx.y * ldo;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < n; g += (int64_t)gridDim.x * blockDim.x)
    out[g] = convert_to<Tout>(in[g]);
}

__global__ void k_masked_copy(int64_t n, const double* __restrict__ in, const double* __restrict__ invD,
                              double* __restrict__ out, int64_t ldi, int64_t ldo) {
  pdl_wait();
  in += (int64_t)blockIdx.y * ldi;
  out += (int64_t)blockIdx.y * ldo;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < n; g += (int64_t)gridDim.x * blockDim.x)
    out[g] = invD[g] != 0.0 ? in[g] : 0.0;
}

constexpr int kVecThreads = 256;

template <typename T>
void cheb4_init(int64_t n, const T* b, T* x, T* r, T* d, T* y, const T* invD, double c0, int x_is_zero,
                cudaStream_t s, int nb, int64_t ld) {
  if (!ld) ld = n;
  const uintptr_t align = (uintptr_t)b | (uintptr_t)x | (uintptr_t)r | (uintptr_t)d | (uintptr_t)y | (uintptr_t)invD;
  if (align % 16 == 0 && (nb == 1 || (ld * sizeof(T)) % 16 == 0))
    launch_dep(k_cheb4_init<T, true>, dim3(grid_for(n / V16<T>::L + 1, kVecThreads), nb), dim3(kVecThreads), 0, s,
               n, b, x, r, d, y, invD, (T)c0, x_is_zero, ld);
  else
    launch_dep(k_cheb4_init<T, false>, dim3(grid_for(n, kVecThreads), nb), dim3(kVecThreads), 0, s, n, b, x, r, d,
               y, invD, (T)c0, x_is_zero, ld);
}
template <typename T>
void cheb4_step(int64_t n, T* x, T* r, T* d, T* y, const T* invD, double beta, double c1, double c2,
                cudaStream_t s, int nb, int64_t ld) {
  if (!ld) ld = n;
  const uintptr_t align = (uintptr_t)x | (uintptr_t)r | (uintptr_t)d | (uintptr_t)y | (uintptr_t)invD;
  if (align % 16 == 0 && (nb == 1 || (ld * sizeof(T)) % 16 == 0))
    launch_dep(k_cheb4_step<T, true>, dim3(grid_for(n / V16<T>::L + 1, kVecThreads), nb), dim3(kVecThreads), 0, s, n,
               x, r, d, y, invD, (T)beta, (T)c1, (T)c2, ld);
  else
    launch_dep(k_cheb4_step<T, false>, dim3(grid_for(n, kVecThreads), nb), dim3(kVecThreads), 0, s, n, x, r, d, y,
               invD, (T)beta, (T)c1, (T)c2, ld);
}
// Whether every pointer and the batch stride allow 16-byte accesses.
template <typename T, typename... P>
static bool vec_ok(int nb, int64_t ld, const P*... p) {
  return (((uintptr_t)p | ...) % 16) == 0 && (nb == 1 || (ld * sizeof(T)) % 16 == 0);
}
template <typename T>
static void launch_begin(int64_t n, const T* rin, T* x, T* r, T* d, const T* invD, double c0, double w, int from_r,
                         int order1, const T* b_next, cudaStream_t s, int nb, int64_t ld) {
  if (!ld) ld = n;
  if (vec_ok<T>(nb, ld, rin, x, r, d, invD, b_next))
    launch_dep(k_smooth_begin<T, true>, dim3(grid_for(n / V16<T>::L + 1, kVecThreads), nb), dim3(kVecThreads), 0, s,
               n, rin, x, r, d, invD, (T)c0, (T)w, from_r, order1, b_next, ld);
  else
    launch_dep(k_smooth_begin<T, false>, dim3(grid_for(n, kVecThreads), nb), dim3(kVecThreads), 0, s, n, rin, x, r,
               d, invD, (T)c0, (T)w, from_r, order1, b_next, ld);
}
template <typename T>
void smooth_begin(int64_t n, const T* b, T* x, T* r, T* d, const T* invD, double c0, bool order1, double w,
                  const T* b_next, cudaStream_t s, int nb, int64_t ld) {
  launch_begin<T>(n, b, x, r, d, invD, c0, w, 0, order1 ? 1 : 0, b_next, s, nb, ld);
}
template <typename T>
void smooth_begin_r(int64_t n, T* x, T* r, T* d, const T* invD, double c0, bool order1, double w, const T* b_next,
                    cudaStream_t s, int nb, int64_t ld) {
  launch_begin<T>(n, r, x, r, d, invD, c0, w, 1, order1 ? 1 : 0, b_next, s, nb, ld);
}
template <typename T, int XM, bool LAST>
static void launch_smooth_step(int64_t n, T* x, T* r, T* d, const T* invD, double c1, double c2, double w0, double w1,
                               const T* b_next, cudaStream_t s, int nb, int64_t ld) {
  if (!ld) ld = n;
  if (vec_ok<T>(nb, ld, x, r, d, invD, b_next))
    launch_dep(k_smooth_step<T, true, XM, LAST>, dim3(grid_for(n / V16<T>::L + 1, kVecThreads), nb),
               dim3(kVecThreads), 0, s, n, x, r, d, invD, (T)c1, (T)c2, (T)w0, (T)w1, b_next, ld);
  else
    launch_dep(k_smooth_step<T, false, XM, LAST>, dim3(grid_for(n, kVecThreads), nb), dim3(kVecThreads), 0, s, n, x,
               r, d, invD, (T)c1, (T)c2, (T)w0, (T)w1, b_next, ld);
}
template <typename T>
void smooth_step(int64_t n, T* x, T* r, T* d, const T* invD, double c1, double c2, int xmode, double w0, double w1,
                 bool last, const T* b_next, cudaStream_t s, int nb, int64_t ld) {
  if (xmode == SX_NONE) launch_smooth_step<T, SX_NONE, false>(n, x, r, d, invD, c1, c2, w0, w1, nullptr, s, nb, ld);
  else if (xmode == SX_ADD && last)
    launch_smooth_step<T, SX_ADD, true>(n, x, r, d, invD, c1, c2, w0, w1, b_next, s, nb, ld);
  else if (xmode == SX_ADD)
    launch_smooth_step<T, SX_ADD, false>(n, x, r, d, invD, c1, c2, w0, w1, nullptr, s, nb, ld);
  else if (last) launch_smooth_step<T, SX_SET, true>(n, x, r, d, invD, c1, c2, w0, w1, b_next, s, nb, ld);
  else launch_smooth_step<T, SX_SET, false>(n, x, r, d, invD, c1, c2, w0, w1, nullptr, s, nb, ld);
}
template <typename T>
void cheb1_init(int64_t n, const T* b, T* x, T* r, T* d, T* y, const T* invD, double inv_theta,
                int x_is_zero, cudaStream_t s, int nb, int64_t ld) {
  launch_dep(k_cheb1_init<T>, dim3(grid_for(n, kVecThreads), nb), dim3(kVecThreads), 0, s, n, b, x, r, d, y, invD,
             (T)inv_theta, x_is_zero, ld ? ld : n);
}
template <typename T>
void cheb1_step(int64_t n, T* x, T* r, T* d, T* y, const T* invD, double c1, double c2, cudaStream_t s, int nb,
                int64_t ld) {
  launch_dep(k_cheb1_step<T>, dim3(grid_for(n, kVecThreads), nb), dim3(kVecThreads), 0, s, n, x, r, d, y, invD,
             (T)c1, (T)c2, ld ? ld : n);
}
template <typename T>
void axpy(int64_t n, double a, const T* d, T* x, cudaStream_t s, int nb, int64_t ld) {
  launch_dep(k_axpy<T>, dim3(grid_for(n, kVecThreads), nb), dim3(kVecThreads), 0, s, n, (T)a, d, x, ld ? ld : n);
}
template <typename Tin, typename Tout>
void cast(int64_t n, const Tin* in, Tout* out, cudaStream_t s, int nb, int64_t ldi, int64_t ldo) {
  launch_dep(k_cast<Tin, Tout>, dim3(grid_for(n, kVecThreads), nb), dim3(kVecThreads), 0, s, n, in, out,
             ldi ? ldi : n, ldo ? ldo : n);
}
void masked_copy(int64_t n, const double* in, const double* invD, double* out, cudaStream_t s, int nb, int64_t ldi,
                 int64_t ldo) {
  launch_dep(k_masked_copy, dim3(grid_for(n, kVecThreads), nb), dim3(kVecThreads), 0, s, n, in, invD, out,
             ldi ? ldi : n, ldo ? ldo : n);
}


#define CHEBMG_CHEB_INST(T)                                                                                 \
  template void smooth_begin<T>(int64_t, const T*, T*, T*, T*, const T*, double, bool, double, const T*,    \
                                cudaStream_t, int, int64_t);                                            \
  template void smooth_begin_r<T>(int64_t, T*, T*, T*, const T*, double, bool, double, const T*, cudaStream_t, \
                                  int, int64_t);                                                        \
  template void smooth_step<T>(int64_t, T*, T*, T*, const T*, double, double, int, double, double, bool,      \
                               const T*, cudaStream_t, int, int64_t);                                   \
  template void axpy<T>(int64_t, double, const T*, T*, cudaStream_t, int, int64_t);

CHEBMG_CHEB_INST(float)
CHEBMG_CHEB_INST(double)
template void cheb4_init<double>(int64_t, const double*, double*, double*, double*, double*, const double*, double, int,
                                 cudaStream_t, int, int64_t);
template void cheb4_step<double>(int64_t, double*, double*, double*, double*, const double*, double, double, double,
                                 cudaStream_t, int, int64_t);
template void cheb1_init<double>(int64_t, const double*, double*, double*, double*, double*, const double*, double, int,
                                 cudaStream_t, int, int64_t);
template void cheb1_step<double>(int64_t, double*, double*, double*, double*, const double*, double, double,
                                 cudaStream_t, int, int64_t);
template void cast<double, float>(int64_t, const double*, float*, cudaStream_t, int, int64_t, int64_t);
template void cast<float, double>(int64_t, const float*, double*, cudaStream_t, int, int64_t, int64_t);
template void cast<double, double>(int64_t, const double*, double*, cudaStream_t, int, int64_t, int64_t);
template void cast<float, float>(int64_t, const float*, float*, cudaStream_t, int, int64_t, int64_t);

}  // namespace chebmg
