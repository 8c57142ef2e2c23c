// Finite-difference kernels (Sec. 3): a constant 3x3 stencil per level (five points on the finest
// grid, Galerkin nine-point below), its transfers, and the steps of Algorithms 1 and 2 with the
// stencil inside.
//
// Grids up to a few hundred points a side stay in L2, so launches and the FP64 pipe bound these
// kernels.  A Chebyshev step is one kernel: the stencil of d, the residual update, the recurrence
// (d out of place, since neighbours read it) and the x update; S = diag(A)^{-1} is one number, so
// it is folded into the coefficients.  From a zero guess the first step works on b directly
// (d_0 = c0 S b is never stored), and the restriction residual is formed in shared memory by the
// restriction itself.  Stencil coefficients are moved into registers (in_register): an FP64 FMA
// with a constant operand issues slower, and a five-point stencil skips its zero corners.
// Separate operator and update kernels -> these: order-4 smoothing of 511 x 511 from a nonzero guess
// 46.2 -> 30.8 us (of which about 15 us FP64 issue), a symmetric order-2 cycle on 63 x 63
// 96.6 -> 32.1 us (27 -> 7 launches, the dense coarse product 45.9 us -> a few, small blocks).
#include <cuda_runtime.h>

#include "common.cuh"

namespace chebmg {

namespace {

constexpr int kBX = 32, kBY = 8;   // threads of a block over the grid (kBY: at most)

// A kernel parameter as a register operand the compiler cannot fold back.  Call it with whole warps.
__device__ __forceinline__ double in_register(double v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ float in_register(float v) { return v; }

// Which of the nine entries a stencil uses: all, or centre and edges.
template <bool NINE>
__device__ __forceinline__ constexpr bool used(int q) {
  return NINE || q == 4 || (q & 1);
}
template <typename T, bool NINE>
__device__ __forceinline__ void load_stencil(const Stencil9<T>& p, T (&c)[9]) {
#pragma unroll
  for (int q = 0; q < 9; ++q) c[q] = used<NINE>(q) ? in_register(p.c[q]) : T(0);
}

// sum_q c[q] u(neighbour q) at (i, j), zero outside the grid; uc = u(i, j).  The terms cancel, so
// the caller adds its residual to the finished sum rather than starting the chain with it (which
// saves one operation and was measured four times less exact).
template <typename T, bool NINE>
__device__ __forceinline__ T stencil_sum(const Arith<T>& ar, const T* u, int mx, int my, int i, int j,
                                         const T (&c)[9], T& uc) {
  const T* p = u + (int64_t)j * mx + i;
  T v[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    if (!used<NINE>(q)) continue;
    const int a = q / 3 - 1, b = q % 3 - 1;
    const bool in = (a == 0 || (a < 0 ? j > 0 : j + 1 < my)) && (b == 0 || (b < 0 ? i > 0 : i + 1 < mx));
    v[q] = in ? p[a * mx + b] : T(0);
  }
  T acc = ar.mul(c[NINE ? 0 : 1], v[NINE ? 0 : 1]);
#pragma unroll
  for (int q = NINE ? 1 : 2; q < 9; ++q)
    if (used<NINE>(q)) acc = fma(c[q], v[q], acc);
  uc = v[4];
  return acc;
}

struct Pt {
  int i, j;
  bool in;
  int64_t g;
};
__device__ __forceinline__ Pt point(int mx, int my) {
  Pt p;
  p.i = blockIdx.x * kBX + threadIdx.x;
  p.j = blockIdx.y * blockDim.y + threadIdx.y;
  p.in = p.i < mx && p.j < my;
  p.g = (int64_t)p.j * mx + p.i;
  return p;
}

// y = A u
template <typename T, bool NINE>
__global__ void __launch_bounds__(kBX * kBY)
k_fd_apply(int mx, int my, Stencil9<T> st, const T* __restrict__ u, T* __restrict__ y, int64_t ld) {
  T c[9];
  const Arith<T> ar;
  load_stencil<T, NINE>(st, c);
  pdl_wait();
  const Pt p = point(mx, my);
  if (!p.in) return;
  const int64_t o = (int64_t)blockIdx.z * ld;   // right-hand side of a batch
  T uc;
  y[o + p.g] = stencil_sum<T, NINE>(ar, u + o, mx, my, p.i, p.j, c, uc);
}

// First step from a zero guess: with d_0 = c0 b (c0 includes S), r = b - A d_0 (st = -c0 A),
// d = c1 d_0 + c2 r, x = w0 d_0 + w1 d (unless x is null).  last: r and d are not stored.
template <typename T, bool NINE>
__global__ void __launch_bounds__(kBX * kBY)
k_fd_first(int mx, int my, Stencil9<T> st, const T* __restrict__ b, T* __restrict__ x, T* __restrict__ r,
           T* __restrict__ d, T c0, T c1, T c2, T w0, T w1, int last, int64_t ld) {
  T c[9];
  const Arith<T> ar;
  load_stencil<T, NINE>(st, c);
  pdl_wait();
  const Pt p = point(mx, my);
  if (!p.in) return;
  const int64_t o = (int64_t)blockIdx.z * ld;
  const T b0 = b[o + p.g];
  T uc;
  const T rv = ar.add(stencil_sum<T, NINE>(ar, b + o, mx, my, p.i, p.j, c, uc), b0);
  const T d0 = c0 * b0, dn = c1 * d0 + c2 * rv;
  if (x) x[o + p.g] = w0 * d0 + w1 * dn;
  if (last) return;
  r[o + p.g] = rv;
  d[o + p.g] = dn;
}

// One step: r -= A d (st = -A), d' = c1 d + c2 r (c2 includes S), then x = or += w0 d + w1 d'.
// last: r and d' are not stored.  rin is r, or the residual to start from (r_out = rin - A d).
template <typename T, bool NINE>
__global__ void __launch_bounds__(kBX * kBY)
k_fd_step(int mx, int my, Stencil9<T> st, const T* __restrict__ d, T* __restrict__ dn, const T* rin, T* r, T* x, T c1,
          T c2, int xmode, T w0, T w1, int last, int64_t ld) {
  T c[9];
  const Arith<T> ar;
  load_stencil<T, NINE>(st, c);
  pdl_wait();
  const Pt p = point(mx, my);
  if (!p.in) return;
  const int64_t o = (int64_t)blockIdx.z * ld + p.g;
  const T r0 = rin[o], x0 = xmode == SX_ADD ? x[o] : T(0);
  T dc;
  const T rv = ar.add(stencil_sum<T, NINE>(ar, d + (int64_t)blockIdx.z * ld, mx, my, p.i, p.j, c, dc), r0);
  const T v = c1 * dc + c2 * rv;
  if (xmode != SX_NONE) x[o] = (x0 + w0 * dc) + w1 * v;
  if (last) return;
  r[o] = rv;
  dn[o] = v;
}

// r = b - A x (st = -A), and d = c0 r where d is given (c0 includes S).
template <typename T, bool NINE>
__global__ void __launch_bounds__(kBX * kBY)
k_fd_resid(int mx, int my, Stencil9<T> st, const T* __restrict__ b, const T* __restrict__ x, T* __restrict__ r,
           T* __restrict__ d, T c0, int64_t ld) {
  T c[9];
  const Arith<T> ar;
  load_stencil<T, NINE>(st, c);
  pdl_wait();
  const Pt p = point(mx, my);
  if (!p.in) return;
  const int64_t o = (int64_t)blockIdx.z * ld;
  T xc;
  const T b0 = b[o + p.g];
  const T rv = ar.add(stencil_sum<T, NINE>(ar, x + o, mx, my, p.i, p.j, c, xc), b0);
  r[o + p.g] = rv;
  if (d) d[o + p.g] = c0 * rv;
}

// rc = P^T (b - A x) for coarsening by two (st = -A): a block forms the residual of the fine points
// under its tile of coarse points in shared memory (one row and column shared with the next tile).
// TY coarse rows per block: 8, or 2 where 8 leave SMs idle (a block's points are FP64 work in series).
constexpr int kTX = 16, kRestrictThreads = 256;
template <typename T, bool NINE, int TY>
__global__ void __launch_bounds__(kRestrictThreads)
k_fd_resid_restrict(int mx, int my, int mcx, int mcy, Stencil9<T> st, const T* __restrict__ b,
                    const T* __restrict__ x, T* __restrict__ rc, int64_t ldf, int64_t ldc) {
  constexpr int FX = 2 * kTX + 1, FY = 2 * TY + 1;
  __shared__ T sr[FY][FX + 1];
  T c[9];
  const Arith<T> ar;
  load_stencil<T, NINE>(st, c);
  pdl_wait();
  b += (int64_t)blockIdx.z * ldf;
  x += (int64_t)blockIdx.z * ldf;
  rc += (int64_t)blockIdx.z * ldc;
  const int I0 = blockIdx.x * kTX, J0 = blockIdx.y * TY;
  for (int q = threadIdx.x; q < FX * FY; q += kRestrictThreads) {
    const int fi = q % FX, fj = q / FX, i = 2 * I0 + fi, j = 2 * J0 + fj;
    T v = T(0), xc;
    if (i < mx && j < my) v = ar.add(stencil_sum<T, NINE>(ar, x, mx, my, i, j, c, xc), b[(int64_t)j * mx + i]);
    sr[fj][fi] = v;
  }
  __syncthreads();
  const int tx = threadIdx.x % kTX, ty = threadIdx.x / kTX, I = I0 + tx, J = J0 + ty;
  if (ty >= TY || I >= mcx || J >= mcy) return;
  T acc = T(0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const T* row = sr[2 * ty + a] + 2 * tx;
    const T v = T(0.5) * (row[0] + row[2]) + row[1];
    acc += (a == 1 ? T(1) : T(0.5)) * v;
  }
  rc[(int64_t)J * mcx + I] = acc;
}

// Orders 1 and 2 from a zero guess with the restriction of their residual: x depends on b alone, so a
// block forms x on the fine points under its coarse tile and a rim of one, the residual there, and
// restricts it; it writes the x it owns.  One launch instead of two, x not read back.
template <typename T, bool NINE, int TY>
__global__ void __launch_bounds__(kRestrictThreads)
k_fd_smooth_restrict(int mx, int my, int mcx, int mcy, Stencil9<T> st, const T* __restrict__ b, T* __restrict__ x,
                     T* __restrict__ rc, int order, T c0, T c1, T c2, T w0, T w1, int64_t ldf, int64_t ldc) {
  constexpr int FX = 2 * kTX + 1, FY = 2 * TY + 1;
  __shared__ T sx[FY + 2][FX + 2];
  __shared__ T sr[FY][FX + 1];
  T c[9];
  const Arith<T> ar;
  load_stencil<T, NINE>(st, c);    // -A
  pdl_wait();
  b += (int64_t)blockIdx.z * ldf;
  x += (int64_t)blockIdx.z * ldf;
  rc += (int64_t)blockIdx.z * ldc;
  const int I0 = blockIdx.x * kTX, J0 = blockIdx.y * TY;
  const bool lastx = blockIdx.x + 1 == gridDim.x, lasty = blockIdx.y + 1 == gridDim.y;
  for (int q = threadIdx.x; q < (FX + 2) * (FY + 2); q += kRestrictThreads) {
    const int sj = q / (FX + 2), si = q - sj * (FX + 2), i = 2 * I0 + si - 1, j = 2 * J0 + sj - 1;
    T v = T(0);
    if (i >= 0 && i < mx && j >= 0 && j < my) {
      const int64_t g = (int64_t)j * mx + i;
      if (order == 1) {
        v = w0 * (c0 * b[g]);
      } else {
        T b0;
        const T s = stencil_sum<T, NINE>(ar, b, mx, my, i, j, c, b0);
        const T rv = fma(c0, s, b0), d0 = c0 * b0, dn = c1 * d0 + c2 * rv;
        v = w0 * d0 + w1 * dn;
      }
      if (si >= 1 && sj >= 1 && (si <= 2 * kTX || lastx) && (sj <= 2 * TY || lasty)) x[g] = v;
    }
    sx[sj][si] = v;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < FX * FY; q += kRestrictThreads) {
    const int fj = q / FX, fi = q - fj * FX, i = 2 * I0 + fi, j = 2 * J0 + fj;
    T v = T(0);
    if (i < mx && j < my) {
      T acc = ar.mul(c[4], sx[fj + 1][fi + 1]);
#pragma unroll
      for (int k = 0; k < 9; ++k)
        if (k != 4 && used<NINE>(k)) acc = fma(c[k], sx[fj + k / 3][fi + k % 3], acc);
      v = ar.add(acc, b[(int64_t)j * mx + i]);
    }
    sr[fj][fi] = v;
  }
  __syncthreads();
  const int tx = threadIdx.x % kTX, ty = threadIdx.x / kTX, I = I0 + tx, J = J0 + ty;
  if (ty >= TY || I >= mcx || J >= mcy) return;
  T acc = T(0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const T* row = sr[2 * ty + a] + 2 * tx;
    const T v = T(0.5) * (row[0] + row[2]) + row[1];
    acc += (a == 1 ? T(1) : T(0.5)) * v;
  }
  rc[(int64_t)J * mcx + I] = acc;
}

// (P xc)(i, j), coarsening by two: even points lie between two coarse ones.
template <typename T>
__device__ __forceinline__ T interpolate2(const T* __restrict__ xc, int mcx, int mcy, int i, int j) {
  const int I = ((i + 1) >> 1) - 1, J = ((j + 1) >> 1) - 1;
  const bool di = !(i & 1), dj = !(j & 1);
  const bool i0 = I >= 0, i1 = di && I + 1 < mcx, j0 = J >= 0, j1 = dj && J + 1 < mcy;
  const T* r0 = xc + (int64_t)J * mcx + I;
  const T a = (i0 && j0 ? r0[0] : T(0)), b = (i1 && j0 ? r0[1] : T(0));
  const T e = (i0 && j1 ? r0[mcx] : T(0)), f = (i1 && j1 ? r0[mcx + 1] : T(0));
  T s = dj ? (a + e) : a;
  if (di) s += dj ? (b + f) : b;
  return s * ((di ? T(0.5) : T(1)) * (dj ? T(0.5) : T(1)));
}

// x = xp + P xc (xm = x if given); with r: r = b - A x (st = -A), d = c0 r.  Out of place, so that a
// block can form x on its tile and a rim of one and take the residual at once.
template <typename T, bool NINE, int BY>
__global__ void __launch_bounds__(kBX * BY)
k_fd_prolong_resid(int mx, int my, int mcx, int mcy, Stencil9<T> st, const T* __restrict__ xp,
                   const T* __restrict__ xc, const T* __restrict__ b, T* __restrict__ x, T* __restrict__ xm,
                   T* __restrict__ r, T* __restrict__ d, T c0, int64_t ldf, int64_t ldc) {
  __shared__ T s[BY + 2][kBX + 2];
  T c[9];
  const Arith<T> ar;
  load_stencil<T, NINE>(st, c);
  pdl_wait();
  const int64_t o = (int64_t)blockIdx.z * ldf;
  xc += (int64_t)blockIdx.z * ldc;
  const Pt p = point(mx, my);
  if (!r) {
    if (p.in) x[o + p.g] = xp[o + p.g] + interpolate2(xc, mcx, mcy, p.i, p.j);
    return;
  }
  const int i0 = blockIdx.x * kBX - 1, j0 = blockIdx.y * BY - 1;
  const int tid = threadIdx.y * kBX + threadIdx.x;
  for (int q = tid; q < (kBX + 2) * (BY + 2); q += kBX * BY) {
    const int sj = q / (kBX + 2), si = q - sj * (kBX + 2), i = i0 + si, j = j0 + sj;
    T v = T(0);
    if (i >= 0 && i < mx && j >= 0 && j < my)
      v = xp[o + (int64_t)j * mx + i] + interpolate2(xc, mcx, mcy, i, j);
    s[sj][si] = v;
  }
  const T b0 = p.in ? b[o + p.g] : T(0);
  __syncthreads();
  if (!p.in) return;
  const int si = threadIdx.x + 1, sj = threadIdx.y + 1;
  T acc = ar.mul(c[4], s[sj][si]);
#pragma unroll
  for (int k = 0; k < 9; ++k)
    if (k != 4 && used<NINE>(k)) acc = fma(c[k], s[sj + k / 3 - 1][si + k % 3 - 1], acc);
  const T rv = ar.add(acc, b0);
  x[o + p.g] = s[sj][si];
  if (xm) xm[o + p.g] = s[sj][si];
  r[o + p.g] = rv;
  d[o + p.g] = c0 * rv;
}

// rc(I,J) = sum_{|a|,|b| < c} w_a w_b rf(c(I+1)-1+b, c(J+1)-1+a), w_d = (c - |d|)/c.  C: the factor
// when known at compile time (2), else 0.
template <typename T, int C>
__global__ void __launch_bounds__(256)
k_fd_restrict(int mfx, int mfy, int mcx, int mcy, int cr, const T* __restrict__ rf, T* __restrict__ rc, int64_t ldf,
              int64_t ldc) {
  pdl_wait();
  rf += (int64_t)blockIdx.z * ldf;
  rc += (int64_t)blockIdx.z * ldc;
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int Jc = blockIdx.y * blockDim.y + threadIdx.y;
  if (I >= mcx || Jc >= mcy) return;
  const int c = C ? C : cr;
  const int fi = c * (I + 1) - 1, fj = c * (Jc + 1) - 1;
  const T inv_c = C == 2 ? T(0.5) : T(1) / T(c);
  T acc = 0;
#pragma unroll
  for (int a = -(c - 1); a <= c - 1; ++a) {
    const int jj = fj + a;
    if (jj < 0 || jj >= mfy) continue;
    const T wa = T(c - (a < 0 ? -a : a)) * inv_c;
    T row = 0;
#pragma unroll
    for (int b = -(c - 1); b <= c - 1; ++b) {
      const int ii = fi + b;
      if (ii < 0 || ii >= mfx) continue;
      row += T(c - (b < 0 ? -b : b)) * inv_c * rf[(size_t)jj * mfx + ii];
    }
    acc += wa * row;
  }
  rc[(size_t)Jc * mcx + I] = acc;
}

// zf (+)= P zc, bilinear.
template <typename T, int C>
__global__ void __launch_bounds__(256)
k_fd_prolong(int mfx, int mfy, int mcx, int mcy, int cr, const T* __restrict__ zc, T* __restrict__ zf, int accumulate,
             int64_t ldf, int64_t ldc) {
  pdl_wait();
  zf += (int64_t)blockIdx.z * ldf;
  zc += (int64_t)blockIdx.z * ldc;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= mfx || j >= mfy) return;
  const int c = C ? C : cr;
  const T inv_c = C == 2 ? T(0.5) : T(1) / T(c);
  const int I0 = (i + 1) / c - 1, J0 = (j + 1) / c - 1;
  const int di = i - (c * (I0 + 1) - 1), dj = j - (c * (J0 + 1) - 1);
  const T wi[2] = {T(c - di) * inv_c, T(di) * inv_c};
  const T wj[2] = {T(c - dj) * inv_c, T(dj) * inv_c};
  T acc = 0;
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int Jc = J0 + a;
    if (Jc < 0 || Jc >= mcy || (a == 1 && dj == 0)) continue;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int I = I0 + b;
      if (I < 0 || I >= mcx || (b == 1 && di == 0)) continue;
      acc += wj[a] * wi[b] * zc[(size_t)Jc * mcx + I];
    }
  }
  T* dst = &zf[(size_t)j * mfx + i];
  *dst = accumulate ? *dst + acc : acc;
}

// y = M x for a dense row-major n x n matrix, a warp per row (coalesced reads, one shuffle sum); a
// block's rows are read once for every right-hand side it covers.  (A thread per row read the matrix
// uncoalesced and summed n products in one chain: 45.9 us at n = 225.)
constexpr int kDenseWarps = 4;
__global__ void __launch_bounds__(32 * kDenseWarps)
k_dense_matvec(int n, const double* __restrict__ M, const double* __restrict__ x, double* __restrict__ y, int nb,
               int64_t ld) {
  pdl_wait();
  const int lane = threadIdx.x & 31, i = blockIdx.x * kDenseWarps + (threadIdx.x >> 5);
  if (i >= n) return;
  const double* row = M + (size_t)i * n;
  for (int q = blockIdx.y; q < nb; q += gridDim.y) {
    const double* xq = x + (int64_t)q * ld;
    double a0 = 0.0, a1 = 0.0;
    int j = lane;
    for (; j + 32 < n; j += 64) {
      a0 = fma(row[j], xq[j], a0);
      a1 = fma(row[j + 32], xq[j + 32], a1);
    }
    if (j < n) a0 = fma(row[j], xq[j], a0);
    a0 += a1;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) a0 += __shfl_down_sync(0xffffffffu, a0, s);
    if (lane == 0) y[(int64_t)q * ld + i] = a0;
  }
}

// ---- adjoint of a smoother application (recurrences at the top of adjoint.cu) ----
__device__ __forceinline__ double block_dot(double v) {   // sum over the block, result in thread (0, 0)
  __shared__ double sh[kBY];
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) v += __shfl_down_sync(0xffffffffu, v, s);
  if (threadIdx.x == 0) sh[threadIdx.y] = v;
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    v = 0.0;
#pragma unroll
    for (int q = 0; q < kBY; ++q) v += sh[q];
  }
  return v;
}
__device__ __forceinline__ int64_t part_index(int dot) {   // partials of one dot: [right-hand side][block]
  const int64_t nblk = (int64_t)gridDim.x * gridDim.y;
  return ((int64_t)dot * gridDim.z + blockIdx.z) * nblk + (int64_t)blockIdx.y * gridDim.x + blockIdx.x;
}

// One step: rho' = rho + k delta (with FIRST: rho = 0 and delta = bk xbar), the partial <delta, r>, then
//   a middle step: delta' = beta xbar + c1 delta - A rho';
//   the last (LAST): bbar = or += rho', and x0bar = xbar - A rho' where x0bar is given.
// st = -A.  rho' of the tile and its rim is formed in shared memory, so A needs no pass of its own.
template <bool NINE, bool FIRST, bool LAST>
__global__ void __launch_bounds__(kBX * kBY)
k_fd_adj_step(int mx, int my, Stencil9<double> st, const double* __restrict__ rho, const double* __restrict__ del,
              const double* __restrict__ xbar, const double* __restrict__ r, double k, double bk, double beta,
              double c1, double* __restrict__ rho_out, double* __restrict__ del_out, double* bbar, int set_bbar,
              double* __restrict__ x0bar, double* __restrict__ part, int dot, int64_t ld) {
  __shared__ double s[kBY + 2][kBX + 2];
  double c[9];
  const Arith<double> ar;
  load_stencil<double, NINE>(st, c);
  k = in_register(k);
  pdl_wait();
  const int64_t o = (int64_t)blockIdx.z * ld;
  const int i0 = blockIdx.x * kBX - 1, j0 = blockIdx.y * kBY - 1;
  const int tid = threadIdx.y * kBX + threadIdx.x;
  for (int q = tid; q < (kBX + 2) * (kBY + 2); q += kBX * kBY) {
    const int sj = q / (kBX + 2), si = q - sj * (kBX + 2), i = i0 + si, j = j0 + sj;
    double v = 0.0;
    if (i >= 0 && i < mx && j >= 0 && j < my) {
      const int64_t g = o + (int64_t)j * mx + i;
      v = FIRST ? ar.mul(k, bk * xbar[g]) : fma(k, del[g], rho[g]);
    }
    s[sj][si] = v;
  }
  const Pt p = point(mx, my);
  double xb = 0.0, dv = 0.0, rv = 0.0;
  if (p.in) {
    xb = xbar[o + p.g];
    dv = FIRST ? bk * xb : del[o + p.g];
    rv = r[o + p.g];
  }
  __syncthreads();
  if (p.in) {
    const int si = threadIdx.x + 1, sj = threadIdx.y + 1;
    double acc = 0.0;
    if (!LAST || x0bar) {
#pragma unroll
      for (int q = 0; q < 9; ++q)
        if (used<NINE>(q)) acc = fma(c[q], s[sj + q / 3 - 1][si + q % 3 - 1], acc);
    }
    const double rn = s[sj][si];
    if constexpr (LAST) {
      bbar[o + p.g] = set_bbar ? rn : bbar[o + p.g] + rn;
      if (x0bar) x0bar[o + p.g] = xb + acc;
    } else {
      rho_out[o + p.g] = rn;
      del_out[o + p.g] = fma(beta, xb, fma(c1, dv, acc));
    }
  }
  const double t = block_dot(dv * rv);
  if (tid == 0) part[part_index(dot)] = t;
}

// Partial <xbar, d_i> for up to kAdjDots vectors.
constexpr int kAdjDots = 8;
struct AdjVecs {
  const double* p[kAdjDots];
};
__global__ void __launch_bounds__(kBX * kBY)
k_fd_adj_dots(int mx, int my, int nv, AdjVecs d, const double* __restrict__ xbar, double* __restrict__ part, int dot0,
              int64_t ld) {
  pdl_wait();
  const Pt p = point(mx, my);
  const int64_t o = (int64_t)blockIdx.z * ld + p.g;
  const double xb = p.in ? xbar[o] : 0.0;
#pragma unroll
  for (int v = 0; v < kAdjDots; ++v) {
    if (v >= nv) break;
    const double t = block_dot(p.in ? xb * d.p[v][o] : 0.0);
    if (threadIdx.x == 0 && threadIdx.y == 0) part[part_index(dot0 + v)] = t;
    __syncthreads();
  }
}

// acc[i] += coef[i] * dot i for i < K (block i), acc[lslot] += sum_i coef[K + i] * dot (K + i) (block
// K); a dot is the sum of its `count` partials, in fixed order.
constexpr int kAdjMaxOrder = 64;
struct AdjCoef {
  double c[2 * kAdjMaxOrder];
};
__global__ void __launch_bounds__(256)
k_fd_adj_finish(int K, int64_t count, const double* __restrict__ part, const __grid_constant__ AdjCoef coef,
                double* __restrict__ acc, int lslot) {
  pdl_wait();
  __shared__ double sh[8];
  const bool lam = (int)blockIdx.x == K;
  const int d0 = blockIdx.x, nd = lam ? K : 1;
  double s = 0.0;
  for (int d = 0; d < nd; ++d) {
    double t0 = 0.0, t1 = 0.0;
    const double* p = part + (int64_t)(d0 + d) * count;
    int64_t q = threadIdx.x;
    for (; q + 256 < count; q += 512) {
      t0 += p[q];
      t1 += p[q + 256];
    }
    if (q < count) t0 += p[q];
    s += coef.c[d0 + d] * (t0 + t1);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < 8; ++q) s += sh[q];
    acc[lam ? lslot : d0] += s;
  }
}

// bbar = or += rb, x0bar -= A rb (st = -A)
template <bool NINE>
__global__ void __launch_bounds__(kBX * kBY)
k_fd_adj_mid(int mx, int my, Stencil9<double> st, const double* __restrict__ rb, double* __restrict__ bbar,
             int set_bbar, double* __restrict__ x0bar, int64_t ld) {
  double c[9];
  const Arith<double> ar;
  load_stencil<double, NINE>(st, c);
  pdl_wait();
  const Pt p = point(mx, my);
  if (!p.in) return;
  const int64_t o = (int64_t)blockIdx.z * ld;
  double uc;
  const double acc = stencil_sum<double, NINE>(ar, rb + o, mx, my, p.i, p.j, c, uc);
  x0bar[o + p.g] += acc;
  bbar[o + p.g] = set_bbar ? uc : bbar[o + p.g] + uc;
}

template <typename T>
bool nine(const Stencil9<T>& st) {
  return st.c[0] != T(0) || st.c[2] != T(0) || st.c[6] != T(0) || st.c[8] != T(0);
}
template <typename T>
Stencil9<T> scaled(const Stencil9<double>& st, double f) {
  Stencil9<T> o;
  for (int q = 0; q < 9; ++q) o.c[q] = (T)(f * st.c[q]);
  return o;
}
dim3 grid_of(int mx, int my, int nb, int by = kBY) { return dim3((mx + kBX - 1) / kBX, (my + by - 1) / by, nb); }
// Rows per block: `many`, or `few` where that leaves SMs without a block -- small grids are bound by the
// FP64 work that the busiest SM does in series.  A symmetric order-2 cycle, tall blocks alone -> this:
// 63 x 63 40.7 -> 32.1 us, 127 x 127 54.5 -> 42.8, 511 x 511 (its coarse levels) 103.0 -> 90.5.
int rows_for(int mx, int my, int nb, int bx, int many, int few) {
  return (int64_t)((mx + bx - 1) / bx) * ((my + many - 1) / many) * nb < sm_count() ? few : many;
}

}  // namespace

// Launches K<T, true> or K<T, false> by the stencil's corners, a thread per point.
#define FD_LAUNCH(K, st, ...)                                                      \
  do {                                                                             \
    const int by_ = rows_for(mx, my, nb, kBX, kBY, 2);                              \
    const dim3 grid_ = grid_of(mx, my, nb, by_), block_(kBX, by_);                   \
    if (nine(st)) launch_dep(K<T, true>, grid_, block_, 0, s, __VA_ARGS__);          \
    else launch_dep(K<T, false>, grid_, block_, 0, s, __VA_ARGS__);                  \
  } while (0)
// The same for the tiled kernels, with ROWS (of `few` or `many`) rows per block.
#define FD_LAUNCH_TILED(K, st, rows, few, many, grid, block, ...)                       \
  do {                                                                                  \
    if (nine(st)) {                                                                     \
      if (rows == few) launch_dep(K<T, true, few>, grid, block, 0, s, __VA_ARGS__);       \
      else launch_dep(K<T, true, many>, grid, block, 0, s, __VA_ARGS__);                  \
    } else {                                                                            \
      if (rows == few) launch_dep(K<T, false, few>, grid, block, 0, s, __VA_ARGS__);      \
      else launch_dep(K<T, false, many>, grid, block, 0, s, __VA_ARGS__);                 \
    }                                                                                   \
  } while (0)

template <typename T>
void fd_apply(int mx, int my, const Stencil9<double>& st, const T* u, T* y, cudaStream_t s, int nb, int64_t ld) {
  const Stencil9<T> a = scaled<T>(st, 1.0);
  FD_LAUNCH(k_fd_apply, a, mx, my, a, u, y, ld);
}

template <typename T>
void fd_first(int mx, int my, const Stencil9<double>& st, const T* b, T* x, T* r, T* d, double c0, double c1, double c2,
              double w0, double w1, bool last, cudaStream_t s, int nb, int64_t ld) {
  const double S = 1.0 / st.c[4];
  const Stencil9<T> a = scaled<T>(st, -c0 * S);
  FD_LAUNCH(k_fd_first, a, mx, my, a, b, x, r, d, (T)(c0 * S), (T)c1, (T)(c2 * S),
            (T)w0, (T)w1, last ? 1 : 0, ld);
}

template <typename T>
void fd_step(int mx, int my, const Stencil9<double>& st, const T* d, T* dn, const T* rin, T* r, T* x, double c1,
             double c2, int xmode, double w0, double w1, bool last, cudaStream_t s, int nb, int64_t ld) {
  const Stencil9<T> a = scaled<T>(st, -1.0);
  FD_LAUNCH(k_fd_step, a, mx, my, a, d, dn, rin, r, x, (T)c1,
            (T)(c2 / st.c[4]), xmode, (T)w0, (T)w1, last ? 1 : 0, ld);
}

template <typename T>
void fd_resid(int mx, int my, const Stencil9<double>& st, const T* b, const T* x, T* r, T* d, double c0, cudaStream_t s,
              int nb, int64_t ld) {
  const Stencil9<T> a = scaled<T>(st, -1.0);
  FD_LAUNCH(k_fd_resid, a, mx, my, a, b, x, r, d, (T)(c0 / st.c[4]), ld);
}

template <typename T>
void fd_resid_restrict(int mx, int my, int mcx, int mcy, const Stencil9<double>& st, const T* b, const T* x, T* rc,
                       cudaStream_t s, int nb, int64_t ldf, int64_t ldc) {
  const Stencil9<T> a = scaled<T>(st, -1.0);
  const int ty = rows_for(mcx, mcy, nb, kTX, 8, 2);
  const dim3 grid((mcx + kTX - 1) / kTX, (mcy + ty - 1) / ty, nb);
  FD_LAUNCH_TILED(k_fd_resid_restrict, a, ty, 2, 8, grid, dim3(kRestrictThreads), mx, my, mcx, mcy, a, b, x, rc, ldf, ldc);
}

template <typename T>
void fd_smooth_restrict(int mx, int my, int mcx, int mcy, const Stencil9<double>& st, const T* b, T* x, T* rc, int order,
                        double c0, double c1, double c2, double w0, double w1, cudaStream_t s, int nb, int64_t ldf,
                        int64_t ldc) {
  const double S = 1.0 / st.c[4];
  const Stencil9<T> a = scaled<T>(st, -1.0);
  const int ty = rows_for(mcx, mcy, nb, kTX, 8, 2);
  const dim3 grid((mcx + kTX - 1) / kTX, (mcy + ty - 1) / ty, nb);
  FD_LAUNCH_TILED(k_fd_smooth_restrict, a, ty, 2, 8, grid, dim3(kRestrictThreads), mx, my, mcx, mcy, a, b, x, rc, order, (T)(c0 * S), (T)c1,
            (T)(c2 * S), (T)w0, (T)w1, ldf, ldc);
}

template <typename T>
void fd_prolong_resid(int mx, int my, int mcx, int mcy, const Stencil9<double>& st, const T* xp, const T* xc, const T* b,
                      T* x, T* xm, T* r, T* d, double c0, cudaStream_t s, int nb, int64_t ldf, int64_t ldc) {
  const Stencil9<T> a = scaled<T>(st, -1.0);
  const int by = rows_for(mx, my, nb, kBX, 8, 4);
  FD_LAUNCH_TILED(k_fd_prolong_resid, a, by, 4, 8, grid_of(mx, my, nb, by), dim3(kBX, by), mx, my, mcx, mcy, a, xp, xc, b, x, xm, r, d,
            (T)(c0 / st.c[4]), ldf, ldc);
}

template <typename T>
void fd_restrict(int mfx, int mfy, int mcx, int mcy, int c, const T* rf, T* rc, cudaStream_t s, int nb,
                 int64_t ldf, int64_t ldc) {
  const dim3 bs(16, 16), gs((mcx + 15) / 16, (mcy + 15) / 16, nb);
  if (c == 2) launch_dep(k_fd_restrict<T, 2>, gs, bs, 0, s, mfx, mfy, mcx, mcy, c, rf, rc, ldf, ldc);
  else launch_dep(k_fd_restrict<T, 0>, gs, bs, 0, s, mfx, mfy, mcx, mcy, c, rf, rc, ldf, ldc);
}

template <typename T>
void fd_prolong(int mfx, int mfy, int mcx, int mcy, int c, const T* zc, T* zf, int accumulate,
                cudaStream_t s, int nb, int64_t ldf, int64_t ldc) {
  const dim3 bs(32, 8), gs((mfx + 31) / 32, (mfy + 7) / 8, nb);
  if (c == 2) launch_dep(k_fd_prolong<T, 2>, gs, bs, 0, s, mfx, mfy, mcx, mcy, c, zc, zf, accumulate, ldf, ldc);
  else launch_dep(k_fd_prolong<T, 0>, gs, bs, 0, s, mfx, mfy, mcx, mcy, c, zc, zf, accumulate, ldf, ldc);
}

void dense_matvec(int n, const double* M, const double* x, double* y, cudaStream_t s, int nb, int64_t ld) {
  // rows of a few right-hand sides per block: enough blocks to fill the GPU for small n
  const unsigned by = (unsigned)(nb < 16 ? nb : 16);
  launch_dep(k_dense_matvec, dim3((n + kDenseWarps - 1) / kDenseWarps, by), dim3(32 * kDenseWarps), 0, s, n, M, x, y,
             nb, ld);
}

int64_t fd_adj_partials(int mx, int my, int nb, int order) {
  const dim3 g = grid_of(mx, my, nb);
  return 2 * (int64_t)order * g.x * g.y * g.z;
}

void fd_adj_step(int mx, int my, const Stencil9<double>& st, const FdAdjStep& a, cudaStream_t s, int nb, int64_t ld) {
  const Stencil9<double> m = scaled<double>(st, -1.0);
  const dim3 grid = grid_of(mx, my, nb), block(kBX, kBY);
  const double k = a.k / st.c[4];   // S folded in
  auto go = [&](auto kernel) {
    launch_dep(kernel, grid, block, 0, s, mx, my, m, a.rho, a.del, a.xbar, a.r, k, a.bk, a.beta, a.c1, a.rho_out,
               a.del_out, a.bbar, a.set_bbar ? 1 : 0, a.x0bar, a.part, a.dot, ld);
  };
  const bool first = a.rho == nullptr;
  if (nine(m)) {
    if (first && a.last) go(k_fd_adj_step<true, true, true>);
    else if (first) go(k_fd_adj_step<true, true, false>);
    else if (a.last) go(k_fd_adj_step<true, false, true>);
    else go(k_fd_adj_step<true, false, false>);
  } else {
    if (first && a.last) go(k_fd_adj_step<false, true, true>);
    else if (first) go(k_fd_adj_step<false, true, false>);
    else if (a.last) go(k_fd_adj_step<false, false, true>);
    else go(k_fd_adj_step<false, false, false>);
  }
}

void fd_adj_dots(int mx, int my, int nv, const double* const* d, const double* xbar, double* part, cudaStream_t s,
                 int nb, int64_t ld) {
  for (int v0 = 0; v0 < nv; v0 += kAdjDots) {
    AdjVecs a{};
    const int n = nv - v0 < kAdjDots ? nv - v0 : kAdjDots;
    for (int v = 0; v < n; ++v) a.p[v] = d[v0 + v];
    launch_dep(k_fd_adj_dots, grid_of(mx, my, nb), dim3(kBX, kBY), 0, s, mx, my, n, a, xbar, part, v0, ld);
  }
}

void fd_adj_finish(int mx, int my, int nb, int order, const double* coef, const double* part, double* acc, int lslot,
                   cudaStream_t s) {
  AdjCoef c{};
  for (int q = 0; q < 2 * order; ++q) c.c[q] = coef[q];
  const dim3 g = grid_of(mx, my, nb);
  launch_dep(k_fd_adj_finish, dim3(order + 1), dim3(256), 0, s, order, (int64_t)g.x * g.y * g.z, part, c, acc, lslot);
}

void fd_adj_mid(int mx, int my, const Stencil9<double>& st, const double* rb, double* bbar, bool set_bbar,
                double* x0bar, cudaStream_t s, int nb, int64_t ld) {
  const Stencil9<double> m = scaled<double>(st, -1.0);
  const dim3 grid = grid_of(mx, my, nb), block(kBX, kBY);
  if (nine(m)) launch_dep(k_fd_adj_mid<true>, grid, block, 0, s, mx, my, m, rb, bbar, set_bbar ? 1 : 0, x0bar, ld);
  else launch_dep(k_fd_adj_mid<false>, grid, block, 0, s, mx, my, m, rb, bbar, set_bbar ? 1 : 0, x0bar, ld);
}

#define FD_INST(T)                                                                                               \
  template void fd_apply<T>(int, int, const Stencil9<double>&, const T*, T*, cudaStream_t, int, int64_t);        \
  template void fd_first<T>(int, int, const Stencil9<double>&, const T*, T*, T*, T*, double, double, double,     \
                            double, double, bool, cudaStream_t, int, int64_t);                                   \
  template void fd_step<T>(int, int, const Stencil9<double>&, const T*, T*, const T*, T*, T*, double, double,    \
                           int, double, double, bool, cudaStream_t, int, int64_t);                               \
  template void fd_resid<T>(int, int, const Stencil9<double>&, const T*, const T*, T*, T*, double, cudaStream_t, \
                            int, int64_t);                                                                       \
  template void fd_resid_restrict<T>(int, int, int, int, const Stencil9<double>&, const T*, const T*, T*,        \
                                     cudaStream_t, int, int64_t, int64_t);                                       \
  template void fd_smooth_restrict<T>(int, int, int, int, const Stencil9<double>&, const T*, T*, T*, int,        \
                                      double, double, double, double, double, cudaStream_t, int, int64_t,        \
                                      int64_t);                                                                  \
  template void fd_prolong_resid<T>(int, int, int, int, const Stencil9<double>&, const T*, const T*, const T*,   \
                                    T*, T*, T*, T*, double, cudaStream_t, int, int64_t, int64_t);                \
  template void fd_restrict<T>(int, int, int, int, int, const T*, T*, cudaStream_t, int, int64_t, int64_t);      \
  template void fd_prolong<T>(int, int, int, int, int, const T*, T*, int, cudaStream_t, int, int64_t, int64_t);

FD_INST(float)
FD_INST(double)

}  // namespace chebmg
