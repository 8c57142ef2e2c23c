// The persistent coarse CG (N = 1, FP64, polynomial preconditioner) on a box lattice: the method, the
// status words and the tagged-word exchange of k_coarse_pcg (kernels.cu), with each product reading
// its vector from shared memory.
//
// The solve is a chain of about 200 products, each an exchange between blocks through the L2, so
// what a product does beside that round trip is what there is to save.  A block owns a contiguous
// range of rows, one per thread.  The 27 neighbours of its rows lie in three bands of the lattice
// (the range itself and the ranges one plane below and above, each widened by a row and a point),
// so it loads each word of the bands once -- three or four per thread instead of 27 -- takes its own
// rows from registers, and computes from shared memory, with the row's 27 coefficients in registers.
// Two shared buffers alternate, so one barrier per product is enough.  Every row in the bands is
// read, boundary (Dirichlet) rows too, which are published as zeros: then two blocks that read
// each other's rows always do so both ways, which the exchange's double buffering needs.
// Sums over the grid travel as tagged words as well: every block posts three values and reads all
// blocks' values itself, one round trip, no counter.
// The block size (64 .. 1024 rows) is timed at setup: small blocks spread the FP64 products over
// more SMs.
//
// Measured, a coarse solve with the products reading the L2 (or the cluster kernel where that was
// faster) -> this, FP32 / FP64 preconditioner: 32^3 elements 594 -> 430 / 967 -> 826 us (141 blocks of
// 256; FP64 there is half FP64 issue), 24^3 473 -> 328 / 768 -> 532, 16^3 311 -> 250 / 550 -> 377 (39 blocks
// of 128 instead of 20 of 256), 8^3 207 -> 167 / 361 -> 218, 45^3 2857 -> 1328 / 5676 -> 3329.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "coarse_util.cuh"
#include "common.cuh"

namespace chebmg {

namespace {

struct Band {
  int bw, pad;    // words per band; own rows start at bw + pad
};
__host__ __device__ constexpr Band band_of(int block, int nx) { return {block + 2 * (nx + 1), nx + 1}; }

// Shared memory: FP64 and FP32 bands, two buffers each, and two buffers for the block sums.
size_t lat_smem(int block, int nx) {
  const size_t w = 3 * (size_t)band_of(block, nx).bw;
  return 2 * w * (sizeof(double) + sizeof(float)) + 2 * 3 * sizeof(double) * (size_t)block;
}

// M: band words a thread loads per product (at most); MAXT: threads per block (at most).  Up to 256
// threads the coefficients stay in registers.
template <bool PF32, int M, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_coarse_lat(CoarseCG a) {
  constexpr bool REG = MAXT <= 256;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ CoarseCoef coef;
  __shared__ double s_res[2][3];
  __shared__ double s_div[2];
  const int T = blockDim.x, tid = threadIdx.x, nx = a.lat_nx, nxy = a.lat_nxy;
  const Band bd = band_of(T, nx);
  const int W = 3 * bd.bw;
  double* sd = reinterpret_cast<double*>(smem_raw);           // [2][W]
  double* sum = sd + 2 * W;                                   // [2][3 T]
  float* sf = reinterpret_cast<float*>(sum + 2 * 3 * T);      // [2][W]
  const int n = (int)a.n, base = blockIdx.x * T, g = base + tid;
  const bool live = g < n;
  const bool lead = blockIdx.x == 0 && tid == 0;
  const int nblk = (int)gridDim.x + (int)a.phantom_blocks;
  for (int q = tid; q < 2 * W; q += T) {                      // words outside the lattice stay zero
    sd[q] = 0.0;
    sf[q] = 0.f;
  }
  // band words this thread loads: position tid + m T, the row there, -1 if none (own or outside)
  // (bands of the block's real rows: the last block's spare threads would make it read blocks that
  // do not read it)
  const int own = min(T, n - base);
  int row[M];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int q = tid + m * T, k = q / bd.bw, o = q - k * bd.bw, r = base + (k - 1) * nxy - bd.pad + o;
    const bool in = q < W && o < own + 2 * bd.pad && r >= 0 && r < n;
    row[m] = in && !(k == 1 && r >= base && r < base + own) ? r : -1;
  }
  const double S = live ? __ldg(&a.invD[g]) : 0.0;
  double r = (live && S != 0.0) ? a.b[g] : 0.0;
  double x = 0.0, p = 0.0, z = 0.0, y = 0.0, ro = 0.0;
  const double c0 = 4.0 / (3.0 * a.lmax);
  coarse_coef_fill(coef, a.degree, a.lmax);
  float cf[REG && PF32 ? 27 : 1];
  double cd[REG && !PF32 ? 27 : 1];
  if constexpr (REG) {
#pragma unroll
    for (int k = 0; k < 27; ++k) {
      if constexpr (PF32) cf[k] = live ? __ldg(&a.valf[(int64_t)k * n + g]) : 0.f;
      else cd[k] = live ? __ldg(&a.val[(int64_t)k * n + g]) : 0.0;
    }
  }
  unsigned gb = 0, gx = 0;   // generations: grid sums, exchanges
  __syncthreads();

  // y = A v on this thread's row: publish v, collect the bands (bounded waits), multiply.  False in
  // every thread if a wait ran out.
  auto product = [&](auto v, auto& out) -> bool {
    using V = decltype(v);
    using TW = typename Tagged<V>::W;
    ++gx;
    const unsigned tag = a.gen0 + gx;
    unsigned long long* buf = Tagged<V>::buf(a, gx);
    V* s = (sizeof(V) == 8 ? reinterpret_cast<V*>(sd) : reinterpret_cast<V*>(sf)) + (gx & 1u) * W;
    if (live) Tagged<V>::store(buf, g, tag, v);
    s[bd.bw + bd.pad + tid] = v;
    V cc[REG && PF32 && sizeof(V) == 8 ? 27 : 1];
    if constexpr (REG && PF32 && sizeof(V) == 8) {   // once per iteration: fetched behind the exchange
#pragma unroll
      for (int k = 0; k < 27; ++k) cc[k] = live ? (V)__ldg(&a.val[(int64_t)k * n + g]) : V(0);
    }
    TW w[M];
    unsigned miss = 0;
    bool ok = true;
#pragma unroll
    for (int m = 0; m < M; ++m)
      if (row[m] >= 0) w[m] = Tagged<V>::load(buf, row[m]);
#pragma unroll
    for (int m = 0; m < M; ++m)
      if (row[m] >= 0 && !Tagged<V>::ready(w[m], tag)) miss |= 1u << m;
    if (miss) {
      const uint64_t t0 = global_ns();
      for (unsigned it = 1; miss; ++it) {
        if (it > 64) __nanosleep(32);
#pragma unroll
        for (int m = 0; m < M; ++m)
          if (miss >> m & 1u) w[m] = Tagged<V>::load(buf, row[m]);
#pragma unroll
        for (int m = 0; m < M; ++m)
          if ((miss >> m & 1u) && Tagged<V>::ready(w[m], tag)) miss &= ~(1u << m);
        if (miss && (it & 63u) == 0 && global_ns() - t0 > kWaitNs) {
          atomicMax((int*)&a.ctl[4], (int)CS_TIMEOUT);
          ok = false;
          break;
        }
      }
    }
#pragma unroll
    for (int m = 0; m < M; ++m)
      if (row[m] >= 0) s[tid + m * T] = Tagged<V>::value(w[m]);
    // the barrier also ends every read of the other shared buffer and of this exchange's words
    if (!__syncthreads_and(ok)) return false;
    V acc = V(0);
    const V* s0 = s + bd.pad + tid;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      const V* q = s0 + (j / 3) * bd.bw + (j % 3 - 1) * nx;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const int k = 3 * j + i;
        V ck;
        if constexpr (!REG) ck = live ? Tagged<V>::coef(a, (int64_t)k * n + g) : V(0);
        else if constexpr (sizeof(V) == 4) ck = cf[PF32 ? k : 0];
        else if constexpr (PF32) ck = cc[k];
        else ck = cd[k];
        acc = fma(ck, q[i - 1], acc);
      }
    }
    out = acc;
    return true;
  };
  // grid sums of three values (see block_sum3): posted and collected as tagged words
  auto grid_sum3 = [&](double& u, double& v, double& w) -> bool {
    block_sum3(sum + (gb & 1u) * 3 * T, s_res[0], u, v, w);
    ++gb;
    const unsigned tag = a.gen0 + gb;
    unsigned long long* buf = a.red + (size_t)(gb & 1u) * kCoarseRedWords * nblk;
    const unsigned long long th = (unsigned long long)tag << 32;
    if (tid < 3) {
      const double val = tid == 0 ? u : tid == 1 ? v : w;
      st_tagged2(buf + (size_t)kCoarseRedWords * blockIdx.x + 2 * tid, th | (unsigned)__double2hiint(val),
                 th | (unsigned)__double2loint(val));
    }
    double s[3] = {0.0, 0.0, 0.0};
    bool ok = true;
    for (int q = tid; q < nblk && ok; q += T) {
      const unsigned long long* src = buf + (size_t)kCoarseRedWords * q;
      Tagged<double>::W t[3];
      const uint64_t t0 = global_ns();
      for (unsigned it = 1;; ++it) {
#pragma unroll
        for (int k = 0; k < 3; ++k) ld_tagged2(src + 2 * k, t[k].hi, t[k].lo);
        if (Tagged<double>::ready(t[0], tag) && Tagged<double>::ready(t[1], tag) && Tagged<double>::ready(t[2], tag))
          break;
        if (it > 64) __nanosleep(32);
        if ((it & 63u) == 0 && global_ns() - t0 > kWaitNs) {
          atomicMax((int*)&a.ctl[4], (int)CS_TIMEOUT);
          ok = false;
          break;
        }
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) s[k] += Tagged<double>::value(t[k]);
    }
    if (!__syncthreads_and(ok)) return false;
    // the same alternating buffer serves again: the barrier above ended its reads
    block_sum3(sum + ((gb + 1) & 1u) * 3 * T, s_res[1], s[0], s[1], s[2]);
    u = s[0];
    v = s[1];
    w = s[2];
    return true;
  };
  // z = M r: Algorithm 2 (beta = 1) from a zero guess
  auto precond = [&]() -> bool {
    using V = std::conditional_t<PF32, float, double>;
    const V sv = PF32 ? (V)(live ? __ldg(&a.invDf[g]) : 0.f) : (V)S;
    V rv = (V)r, d = (V)c0 * sv * rv, zv = V(0), yv = V(0);
    for (int i = 1; i < a.degree; ++i) {
      zv += d;
      if (!product(d, yv)) return false;
      const V c1 = PF32 ? (V)coef.c1f[i] : (V)coef.c1[i], c2 = PF32 ? (V)coef.c2f[i] : (V)coef.c2[i];
      rv -= yv;
      d = c1 * d + c2 * sv * rv;
    }
    z = (double)(zv + d);
    return true;
  };
  auto finish = [&](int status, int it) {
    if (live) a.x[g] = x;
    if (lead) {
      a.ctl[2] = (unsigned)status;
      a.ctl[3] = (unsigned)it;
      if (status == CS_BREAKDOWN) atomicMax((int*)&a.ctl[4], (int)CS_BREAKDOWN);
    }
  };
  if (!precond()) return;
  p = z;
  double rz = r * z, rr = r * r, spare = 0.0;
  if (!grid_sum3(rz, rr, spare)) return;
  double gam = rz;
  if (!(rr > 0.0) || !(gam >= 0.0)) {
    finish(rr == 0.0 ? CS_OK : CS_BREAKDOWN, 0);
    return;
  }
  const double tol2 = a.rtol * a.rtol * rr;
  for (int it = 1; it <= a.maxit; ++it) {
    if (!product(p, y)) return;
    double pq = p * y, z1 = 0.0, z2 = 0.0;
    if (!grid_sum3(pq, z1, z2)) return;
    if (!(pq > 0.0)) {
      finish(CS_BREAKDOWN, it);
      return;
    }
    const double alpha = block_div(&s_div[0], gam, pq);
    ro = r;
    x = fma(alpha, p, x);
    r = fma(-alpha, y, r);
    if (!precond()) return;
    double rz2 = r * z, rr2 = r * r;
    z1 = PF32 ? ro * z : 0.0;
    if (!grid_sum3(rz2, rr2, z1)) return;
    if (!(rr2 == rr2)) {
      finish(CS_BREAKDOWN, it);
      return;
    }
    if (rr2 <= tol2) {
      finish(CS_OK, it);
      return;
    }
    // Fletcher-Reeves for the exact (symmetric) FP64 preconditioner; Polak-Ribiere
    // (z_new, r_new - r_old) / (z_old, r_old) for the FP32 one
    const double beta = block_div(&s_div[1], PF32 ? rz2 - z1 : rz2, gam);
    gam = rz2;
    p = fma(beta, p, z);
  }
  finish(CS_NOTCONV, a.maxit);
}

template <bool PF32>
const void* lat_kernel(int block, int loads) {
  if (block <= 256) return loads <= 4 ? (const void*)k_coarse_lat<PF32, 4, 256> : (const void*)k_coarse_lat<PF32, 8, 256>;
  return loads <= 4 ? (const void*)k_coarse_lat<PF32, 4, 1024> : (const void*)k_coarse_lat<PF32, 8, 1024>;
}
int loads_of(int block, int nx) { return (3 * band_of(block, nx).bw + block - 1) / block; }

}  // namespace

bool coarse_lat_fits(int64_t n, int nx, int block) {
  static PerDevice smem_max;
  const int optin = smem_max([] { return device_attribute(cudaDevAttrMaxSharedMemoryPerBlockOptin); });
  return n < (int64_t)1 << 30 && (n + block - 1) / block <= sm_count() && loads_of(block, nx) <= 8 &&
         lat_smem(block, nx) + 4096 <= (size_t)optin;
}

bool coarse_lat_launch(const CoarseCG& a, cudaStream_t s, cudaError_t* err) {
  CoarseCG arg = a;
  void* params[] = {&arg};
  const size_t smem = lat_smem(a.lat_block, a.lat_nx);
  const int loads = loads_of(a.lat_block, a.lat_nx);
  const void* fn = a.pf32 ? lat_kernel<true>(a.lat_block, loads) : lat_kernel<false>(a.lat_block, loads);
  cudaError_t e = cudaSuccess;
  if (smem > 40 * 1024) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)
    e = cudaLaunchCooperativeKernel(fn, dim3((unsigned)((a.n + a.lat_block - 1) / a.lat_block)), dim3(a.lat_block),
                                    params, smem, s);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  if (err) *err = e;
  return e == cudaSuccess;
}

}  // namespace chebmg
