// Element operator for the polynomial orders other than 1, 3 and 7 (Sec. 1, Eq. 1.3; orders 3 and 7
// have kernels of their own, order 1 is the assembled coarse level), by line passes.
//
// Q = N + 1 points per direction, Q^2 threads per element: in each of the six 1-D contractions a
// thread owns one whole grid line, reads its Q values once and produces Q outputs, so a value read
// from shared memory feeds about Q/2 FMAs (the one-thread-per-point form reads two shared values
// for every FMA and is bound by them).  The derivative matrix is centro-antisymmetric,
// D[Q-1-i][Q-1-l] = -D[i][l]: sums and differences of mirrored points halve the multiplications
// (h = Q / 2 of each; odd Q has a middle point that joins the even half and a middle row of
// differences alone).
// Strides R (rows) and P (planes) are those with the fewest bank conflicts over the passes.
//
// Measured, one thread per point -> line passes, with the zeroing of the output (6 to 12 us):
// FP32 order 9 on 23^3 elements 215.5 -> 116.9 us and on 13^3 44.9 -> 24.6, order 8 on 25^3
// 242.5 -> 92.3, order 5 on 38^3 164.8 -> 91.3, order 2 on 42^3 26.7 -> 22.5; FP64 order 9 on 23^3
// 1555 -> 1334, order 5 on 38^3 932 -> 874, order 2 on 42^3 109.7 -> 102.4.  Then, with the FP64
// coefficients in shared memory: order 9 1334 -> 1216 us, order 5 874 -> 833; and with the FP32 factors
// read where they are used instead of held in registers (twice the elements in flight per SM): order
// 9 116.9 -> 87.2 us on 23^3 and 18.9 -> 13.4 on 12^3, order 8 90.3 -> 75.2, order 5 87.5 -> 83.1.
#include <cuda_runtime.h>

#include "common.cuh"

namespace chebmg {

namespace {

constexpr int kMaxH = 5, kRow = 6;   // Q <= 10; rows padded to 16-byte multiples
// [0] of D, [1] of D^T: even blocks e[i][l] (column h: the middle point), odd blocks o[i][l],
// middle row m[l]
template <typename T>
struct LineTab {
  T e[2][kMaxH][kRow], o[2][kMaxH][kRow], m[2][kRow];
};
__constant__ LineTab<float> c_tab_f[11];
__device__ LineTab<double> g_tab_d[11];

// The line coefficients as a kernel uses them: FP32 constant-bank operands; FP64 staged in shared
// memory (register operands issue faster, see Fp64Unit), rows loaded where they are used.  Every
// thread of the block calls the constructor; a block barrier separates it from the first line.
template <typename T, int Q>
struct Coef;
template <int Q>
struct Coef<float, Q> : Arith<float> {
  using Shared = float;
  __device__ __forceinline__ explicit Coef(float*) {}
  template <int W, int K>   // K: 0 even, 1 odd, 2 middle
  __device__ __forceinline__ void row(int i, float (&v)[kRow]) const {
    const LineTab<float>& t = c_tab_f[Q];
#pragma unroll
    for (int l = 0; l < Q / 2 + (K == 0 ? Q % 2 : 0); ++l) v[l] = K == 0 ? t.e[W][i][l] : K == 1 ? t.o[W][i][l] : t.m[W][l];
  }
};
template <int Q>
struct Coef<double, Q> : Arith<double> {
  using Shared = LineTab<double>;
  const Shared* t;
  __device__ __forceinline__ explicit Coef(Shared* sh) : t(sh) {
    const double* src = reinterpret_cast<const double*>(&g_tab_d[Q]);
    for (int q = threadIdx.x; q < (int)(sizeof(Shared) / sizeof(double)); q += blockDim.x)
      reinterpret_cast<double*>(sh)[q] = __ldg(src + q);
  }
  template <int W, int K>
  __device__ __forceinline__ void row(int i, double (&v)[kRow]) const {
    const double2* p = reinterpret_cast<const double2*>(K == 0 ? t->e[W][i] : K == 1 ? t->o[W][i] : t->m[W]);
#pragma unroll
    for (int l = 0; l < (Q / 2 + (K == 0 ? Q % 2 : 0) + 1) / 2; ++l) {
      const double2 x = p[l];
      v[2 * l] = x.x;
      v[2 * l + 1] = x.y;
    }
  }
};

// EB elements per block.
template <typename T, int Q, int EB_>
struct AxL {
  static constexpr bool F = sizeof(T) == 4;
  static constexpr int QQ = Q * Q, NP = Q * Q * Q, EB = EB_;
  // FP32 reads the factors where they are used, with small blocks and many of them per SM; at order 6
  // holding them in registers was faster (87.2 against 91.3 us on 33^3 elements)
  static constexpr bool GREG = F && (Q == 7 || Q == 3);
  static constexpr int THREADS = (EB * QQ + 31) / 32 * 32;
  // blocks per SM to fit registers for
  static constexpr int MINB = EB == 1 && !(F && Q >= 9) ? 1
                              : F ? (Q == 10 ? 9 : Q == 9 ? 10 : Q == 6 ? 4 : Q == 5 ? 8 : 1) : (Q == 9 ? 2 : 1);
  static constexpr int R = F ? (Q == 3 ? 4 : Q == 5 ? 6 : Q == 6 ? 9 : Q == 7 ? 8 : Q) : (Q == 6 ? 9 : Q);
  static constexpr int P = F ? (Q == 3 ? 35 : Q == 5 ? 37 : Q == 6 ? 70 : Q == 7 ? 71 : Q == 9 ? 81 : 101)
                             : (Q == 3 ? 19 : Q == 5 ? 25 : Q == 6 ? 54 : Q == 7 ? 55 : Q == 9 ? 89 : 106);
  static constexpr int STAGE = Q * P;
  static constexpr size_t SMEM = sizeof(T) * (size_t)EB * 3 * STAGE;
};

// o = D u (W = 0) or D^T u (W = 1) along a line of Q points.
template <typename T, int Q, int W>
__device__ __forceinline__ void line(const Coef<T, Q>& c, const T (&u)[Q], T (&o)[Q]) {
  constexpr int H = Q / 2;
  T ue[H], uo[H];
#pragma unroll
  for (int l = 0; l < H; ++l) {
    ue[l] = c.add(u[l], u[Q - 1 - l]);
    uo[l] = c.sub(u[l], u[Q - 1 - l]);
  }
#pragma unroll
  for (int i = 0; i < H; ++i) {
    T e[kRow], d[kRow];
    c.template row<W, 0>(i, e);
    c.template row<W, 1>(i, d);
    T se = c.mul(e[0], ue[0]);
#pragma unroll
    for (int l = 1; l < H; ++l) se = fma(e[l], ue[l], se);
    if (Q % 2) se = fma(e[H], u[H], se);
    if constexpr (sizeof(T) == 8) {   // the odd chain continues the even one: one FMA gives the mirror
      T s = se;
#pragma unroll
      for (int l = 0; l < H; ++l) s = fma(d[l], uo[l], s);
      o[i] = s;
      o[Q - 1 - i] = fma(c.k.m2, se, s);
    } else {
      T so = d[0] * uo[0];
#pragma unroll
      for (int l = 1; l < H; ++l) so = fma(d[l], uo[l], so);
      o[i] = se + so;
      o[Q - 1 - i] = so - se;
    }
  }
  if constexpr (Q % 2) {
    T d[kRow];
    c.template row<W, 2>(0, d);
    T s = c.mul(d[0], uo[0]);
#pragma unroll
    for (int l = 1; l < H; ++l) s = fma(d[l], uo[l], s);
    o[H] = s;
  }
}

template <typename T, int Q, int EB, bool IMPLICIT>
__global__ void __launch_bounds__(AxL<T, Q, EB>::THREADS, AxL<T, Q, EB>::MINB)
k_sem_axl(int64_t E, const uint32_t* __restrict__ gid, Lattice lat, const T* __restrict__ G,
          const T* __restrict__ u, T* __restrict__ y, int64_t ld, uint32_t neg) {
  using C = AxL<T, Q, EB>;
  constexpr int R = C::R, P = C::P, QQ = C::QQ, NP = C::NP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) typename Coef<T, Q>::Shared sCoef;
  const Coef<T, Q> cf(&sCoef);
  T* sm = reinterpret_cast<T*>(smem_raw);
  const int tid = threadIdx.x;
  const bool in = tid < C::EB * QQ;           // the last warp may have spare threads
  const int le = in ? tid / QQ : 0, t = in ? tid - le * QQ : 0, a = t % Q, b = t / Q;
  const int64_t e = (int64_t)blockIdx.x * C::EB + le;
  const bool valid = in && e < E;
  T* su = sm + (size_t)le * 3 * C::STAGE;
  T* sr = su + C::STAGE;
  T* ss = sr + C::STAGE;
  const T* Ge = G + (valid ? e : 0) * (6 * NP) + t;
  constexpr bool GREG = C::GREG;
  T gr[GREG ? 6 : 1][GREG ? Q : 1];
  if constexpr (GREG) {
#pragma unroll
    for (int c = 0; c < 6; ++c)
#pragma unroll
      for (int k = 0; k < Q; ++k) gr[c][k] = __ldg(Ge + c * NP + k * QQ);
  }
  uint32_t g[Q];
  if (!valid) {
#pragma unroll
    for (int k = 0; k < Q; ++k) g[k] = kGidDirichlet;
  } else if constexpr (IMPLICIT) {
    const uint32_t ee = (uint32_t)e, exy = (uint32_t)lat.nex * (uint32_t)lat.ney;
    const uint32_t ez = ee / exy, rem = ee - ez * exy, ey = rem / (uint32_t)lat.nex, ex = rem - ey * (uint32_t)lat.nex;
    const uint32_t gx = ex * (Q - 1) + a, gy = ey * (Q - 1) + b;
    const bool side = gx == 0 || gx == (uint32_t)lat.NX - 1 || gy == 0 || gy == (uint32_t)lat.NY - 1;
    const uint32_t plane = (uint32_t)lat.NX * (uint32_t)lat.NY;
    const uint32_t g0 = (ez * (Q - 1) * (uint32_t)lat.NY + gy) * (uint32_t)lat.NX + gx;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const uint32_t gz = ez * (Q - 1) + k;
      g[k] = (g0 + k * plane) | ((side || gz == 0 || gz == (uint32_t)lat.NZ - 1) ? kGidDirichlet : 0u);
    }
  } else {
#pragma unroll
    for (int k = 0; k < Q; ++k) g[k] = __ldg(gid + e * NP + k * QQ + t);
  }
  u += (int64_t)blockIdx.y * ld;   // right-hand side of a batch
  y += (int64_t)blockIdx.y * ld;
  pdl_wait();   // u and y may come from the kernel before (programmatic dependent launch)
  T col[Q], ut[Q];
#pragma unroll
  for (int k = 0; k < Q; ++k) col[k] = (g[k] & kGidDirichlet) ? T(0) : u[g[k] & kGidMask];
  if (in) {
#pragma unroll
    for (int k = 0; k < Q; ++k) su[k * P + b * R + a] = col[k];
  }
  __syncthreads();
  line<T, Q, 0>(cf, col, ut);                    // t: thread (i = a, j = b)
  T v[Q], o[Q];
  if (in) {
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = su[b * P + a * R + i];   // r: thread (j = a, k = b)
    line<T, Q, 0>(cf, v, o);
#pragma unroll
    for (int i = 0; i < Q; ++i) sr[b * P + a * R + i] = o[i];
#pragma unroll
    for (int j = 0; j < Q; ++j) v[j] = su[b * P + j * R + a];   // s: thread (i = a, k = b)
    line<T, Q, 0>(cf, v, o);
#pragma unroll
    for (int j = 0; j < Q; ++j) ss[b * P + j * R + a] = o[j];
  }
  __syncthreads();
  if (in) {
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const int q = k * P + b * R + a;
      T g00, g01, g02, g11, g12, g22;
      if constexpr (GREG) {
        g00 = gr[0][k]; g01 = gr[1][k]; g02 = gr[2][k]; g11 = gr[3][k]; g12 = gr[4][k]; g22 = gr[5][k];
      } else {
        const T* p = Ge + k * QQ;
        g00 = __ldg(p); g01 = __ldg(p + NP); g02 = __ldg(p + 2 * NP);
        g11 = __ldg(p + 3 * NP); g12 = __ldg(p + 4 * NP); g22 = __ldg(p + 5 * NP);
      }
      const T ur = sr[q], us = ss[q], utk = ut[k];
      sr[q] = fma(g02, utk, fma(g01, us, cf.mul(g00, ur)));
      ss[q] = fma(g12, utk, fma(g11, us, cf.mul(g01, ur)));
      v[k] = fma(g22, utk, fma(g12, us, cf.mul(g02, ur)));
    }
    line<T, Q, 1>(cf, v, ut);                    // ut now holds the t contribution
  }
  __syncthreads();
  if (in) {
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = sr[b * P + a * R + i];
    line<T, Q, 1>(cf, v, o);
#pragma unroll
    for (int i = 0; i < Q; ++i) su[b * P + a * R + i] = o[i];
  }
  __syncthreads();
  if (in) {
#pragma unroll
    for (int j = 0; j < Q; ++j) v[j] = ss[b * P + j * R + a];
    line<T, Q, 1>(cf, v, o);
#pragma unroll
    for (int j = 0; j < Q; ++j) su[b * P + j * R + a] = cf.add(su[b * P + j * R + a], o[j]);
  }
  __syncthreads();
  if (valid) {
#pragma unroll
    for (int k = 0; k < Q; ++k)
      if (!(g[k] & kGidDirichlet)) atomicAdd(&y[g[k] & kGidMask], flip_sign(cf.add(su[k * P + b * R + a], ut[k]), neg));
  }
}

template <typename T, int Q, int EB>
void launch_eb(int64_t E, const uint32_t* gid, const Lattice* lat, const T* G, const T* u, T* y, cudaStream_t s,
               int nb, int64_t ld, uint32_t neg) {
  using C = AxL<T, Q, EB>;
  static PerDevice smem_lat, smem_map;
  const dim3 blocks((unsigned)((E + EB - 1) / EB), nb);
  if (lat) {
    allow_smem(smem_lat, (const void*)k_sem_axl<T, Q, EB, true>, C::SMEM);
    launch_dep(k_sem_axl<T, Q, EB, true>, blocks, dim3(C::THREADS), C::SMEM, s, E, gid, *lat, G, u, y, ld, neg);
  } else {
    allow_smem(smem_map, (const void*)k_sem_axl<T, Q, EB, false>, C::SMEM);
    launch_dep(k_sem_axl<T, Q, EB, false>, blocks, dim3(C::THREADS), C::SMEM, s, E, gid, Lattice{}, G, u, y, ld, neg);
  }
}

// Elements per block: the number that fills whole warps best (FP64 issue is paid for every lane of a
// warp), or fewer where the busiest SM then has fewer warps to issue for: one where that leaves SMs idle
// (36 elements of order 9 in FP64: 72.1 us in blocks of five, 21.6 in blocks of one), and at order 5 in FP64,
// whose blocks of seven are the largest, five or four where that makes a smaller last wave (order-4
// smoothing of 1,100 elements 135 -> 94.6 us, of 2,200 199 -> 157).
template <typename T, int Q>
void launch(int64_t E, const uint32_t* gid, const Lattice* lat, const T* G, const T* u, T* y, cudaStream_t s, int nb,
            int64_t ld, uint32_t neg) {
  constexpr int EB = Q == 3 ? 14 : Q == 5 ? 5 : Q == 6 ? 7 : Q == 7 ? 5 : sizeof(T) == 4 ? 1 : Q == 9 ? 3 : 5;
  constexpr int SMALL = Q == 3 ? 3 : 1;
  if constexpr (EB > SMALL) {
    const int sms = sm_count();
    auto warps = [&](int eb, int threads) {   // of the busiest SM
      const int64_t blocks = (E + eb - 1) / eb * nb;
      return (blocks + sms - 1) / sms * (threads / 32);
    };
    int64_t least = warps(EB, AxL<T, Q, EB>::THREADS);
    int eb = EB;
    auto consider = [&](int e, int threads) {
      const int64_t w = warps(e, threads);
      if (w < least) least = w, eb = e;
    };
    if constexpr (sizeof(T) == 8 && Q == 6) {
      consider(5, AxL<T, Q, 5>::THREADS);
      consider(4, AxL<T, Q, 4>::THREADS);
    }
    consider(SMALL, AxL<T, Q, SMALL>::THREADS);
    if (eb == SMALL) return launch_eb<T, Q, SMALL>(E, gid, lat, G, u, y, s, nb, ld, neg);
    if constexpr (sizeof(T) == 8 && Q == 6) {
      if (eb == 5) return launch_eb<T, Q, 5>(E, gid, lat, G, u, y, s, nb, ld, neg);
      if (eb == 4) return launch_eb<T, Q, 4>(E, gid, lat, G, u, y, s, nb, ld, neg);
    }
  }
  launch_eb<T, Q, EB>(E, gid, lat, G, u, y, s, nb, ld, neg);
}

template <typename T>
void fill(const double* S, int Q, LineTab<T>& t) {   // S: symmetrised D, [Q][Q]
  const int H = Q / 2;
  for (int w = 0; w < 2; ++w) {
    auto at = [&](int i, int l) { return w == 0 ? S[i * Q + l] : S[l * Q + i]; };
    for (int i = 0; i < H; ++i) {
      for (int l = 0; l < H; ++l) {
        t.e[w][i][l] = (T)(0.5 * (at(i, l) + at(i, Q - 1 - l)));
        t.o[w][i][l] = (T)(0.5 * (at(i, l) - at(i, Q - 1 - l)));
      }
      if (Q % 2) t.e[w][i][H] = (T)at(i, H);
    }
    if (Q % 2)
      for (int l = 0; l < H; ++l) t.m[w][l] = (T)at(H, l);
  }
}

}  // namespace

// On few elements a thread per point has the shorter serial chains, and the line passes' fewer
// operations count only once every SM has warps enough to keep FP64 issue busy.  Four products of a
// smoother, thread per point against line passes: order 4 on 512 elements 41.5 / 47.3 us, on 640 61.2 /
// 47.3; order 5 on 294 39.4 / 57.4, on 512 60.0 / 80.0, on 640 82.7 / 82.5; order 6 on 294 55.8 / 65.6, on
// 448 76.3 / 79.5, on 640 114.8 / 98.2; order 8 on 150 68.2 / 85.6, on 180 114.2 / 105.0; order 9 on 150
// 91.7 / 97.9, on 180 170.0 / 155.9.  Order 2: even at every size.
// FP32, the same: order 4 on 64 elements 15.8 / 16.7 us, on 512 16.6 / 18.1, on 729 19.1 / 18.1; order 5 on 64
// 16.0 / 17.8, on 343 18.2 / 18.2, on 512 19.7 / 20.6, on 729 21.4 / 20.1; order 6 on 64 16.0 / 18.1, on 125
// 16.3 / 18.2, on 216 18.6 / 18.6, on 343 21.4 / 18.8.  Orders 2, 8 and 9 are even on the fewest (order 9 on
// 64 elements 22.7 / 23.4) and line passes soon the faster.
template <typename T>
bool sem_axl_chosen(int Q, int64_t elements) {
  const int64_t few = sizeof(T) == 4 ? (Q == 5 || Q == 6 ? 4 : Q == 7 ? 1 : 0)   // elements per SM
                                     : Q == 3 ? 0 : Q >= 9 ? 1 : 4;
  return sem_axl_supported(Q) && (few == 0 || elements > few * sm_count());
}
template bool sem_axl_chosen<float>(int, int64_t);
template bool sem_axl_chosen<double>(int, int64_t);

bool sem_axl_supported(int Q) { return Q == 3 || (Q >= 5 && Q <= 10 && Q != 8); }

cudaError_t sem_axl_set_D(int Q, const double* D) {
  if (!sem_axl_supported(Q)) return cudaErrorInvalidValue;
  double S[100];
  for (int i = 0; i < Q; ++i)
    for (int l = 0; l < Q; ++l) S[i * Q + l] = 0.5 * (D[i * Q + l] - D[(Q - 1 - i) * Q + (Q - 1 - l)]);
  LineTab<float> f{};
  LineTab<double> d{};
  fill(S, Q, f);
  fill(S, Q, d);
  const cudaError_t e = cudaMemcpyToSymbol(c_tab_f, &f, sizeof(f), (size_t)Q * sizeof(f));
  return e != cudaSuccess ? e : cudaMemcpyToSymbol(g_tab_d, &d, sizeof(d), (size_t)Q * sizeof(d));
}

template <typename T>
bool sem_axl(int Q, int64_t E, const uint32_t* gid, const Lattice* lat, const T* G, const T* u, T* y, cudaStream_t s,
             int nb, int64_t ld, bool subtract) {
  const uint32_t neg = subtract ? kSignBit : 0u;
  switch (Q) {
    case 3: launch<T, 3>(E, gid, lat, G, u, y, s, nb, ld, neg); return true;
    case 5: launch<T, 5>(E, gid, lat, G, u, y, s, nb, ld, neg); return true;
    case 6: launch<T, 6>(E, gid, lat, G, u, y, s, nb, ld, neg); return true;
    case 7: launch<T, 7>(E, gid, lat, G, u, y, s, nb, ld, neg); return true;
    case 9: launch<T, 9>(E, gid, lat, G, u, y, s, nb, ld, neg); return true;
    case 10: launch<T, 10>(E, gid, lat, G, u, y, s, nb, ld, neg); return true;
    default: return false;
  }
}
template bool sem_axl<float>(int, int64_t, const uint32_t*, const Lattice*, const float*, const float*, float*,
                             cudaStream_t, int, int64_t, bool);
template bool sem_axl<double>(int, int64_t, const uint32_t*, const Lattice*, const double*, const double*, double*,
                              cudaStream_t, int, int64_t, bool);

}  // namespace chebmg
