// p-multigrid interpolation and restriction (Sec. 4.1) for fixed order pairs (7->3, 3->1 and
// the 7->5->3 steps of the 7-5-3-1 schedule), on the box lattice of the library's meshes.
//
// P z_c = W Q_f^T (J x J x J) Q_c z_c and P^T r_f = Q_c^T (J^T x J^T x J^T) O^T r_f, where
// O^T keeps each fine node only in its owner element (equal to Q_f W on the continuous range
// of J3 Q_c).  QF^2 threads per element, a thread per fine column: its global ids step by one
// lattice plane, so a column costs one set of coordinates instead of one per point, its loads are
// in flight together, and the contraction along it needs no shared memory; the two others go
// through shared memory with every thread busy (lines split over threads where there are more
// threads than lines).  Element ends are points of both orders, so the first and last row of J are
// unit rows and only the interior ones are multiplied.
// FP64 loads J's distinct entries (J[QF-1-f][QC-1-c] = J[f][c]) instead of taking them as constant
// operands, with which an FMA issues slower (see Fp64Unit).
//
// An id and ownership test per point, divisions per thread and passes with idle threads -> this
// (restriction / interpolation / accumulating, us): FP32 7 <-> 3 on 32^3 elements
// 33.0 / 26.6 / 30.7 -> 23.1 / 22.4 / 24.2, 3 <-> 1 18.6 / 14.4 / 14.7 -> 7.6 / 5.8 / 5.7;
// FP64 7 <-> 3 250 / 235 / 271 -> 157 / 188 / 188, 3 <-> 1 57 / 48 / 55 -> 15 / 14 / 17.  FP32 is bound by
// instruction issue, FP64 by its pipe.
#include <cuda_runtime.h>

#include "common.cuh"

namespace chebmg {

namespace {

// J[fine point][coarse point] per supported pair: FP32 constant, FP64 in global memory.
__constant__ float c_J84_f[8 * 4];
__constant__ float c_J42_f[4 * 2];
__constant__ float c_J86_f[8 * 6];
__constant__ float c_J64_f[6 * 4];
__device__ double g_J84_d[8 * 4];
__device__ double g_J42_d[4 * 2];
__device__ double g_J86_d[8 * 6];
__device__ double g_J64_d[6 * 4];

template <int QF, int QC>
__device__ __forceinline__ const float* table_f() {
  return QF == 4 ? c_J42_f : QF == 6 ? c_J64_f : QC == 4 ? c_J84_f : c_J86_f;
}
template <int QF, int QC>
__device__ __forceinline__ const double* table_d() {
  return QF == 4 ? g_J42_d : QF == 6 ? g_J64_d : QC == 4 ? g_J84_d : g_J86_d;
}

// J(f, c) for interior rows 1 <= f <= QF - 2.
template <typename T, int QF, int QC>
struct Interp;
template <int QF, int QC>
struct Interp<float, QF, QC> : Arith<float> {
  __device__ __forceinline__ float at(int f, int c) const { return table_f<QF, QC>()[f * QC + c]; }
};
template <int QF, int QC>
struct Interp<double, QF, QC> : Arith<double> {
  double v[QF / 2][QC];   // rows 1 .. QF/2 - 1 used
  __device__ __forceinline__ Interp() {
#pragma unroll
    for (int f = 1; f < QF / 2; ++f)
#pragma unroll
      for (int c = 0; c < QC; ++c) v[f][c] = __ldg(table_d<QF, QC>() + f * QC + c);
  }
  __device__ __forceinline__ double at(int f, int c) const { return f < QF / 2 ? v[f][c] : v[QF - 1 - f][QC - 1 - c]; }
};

// (J^T v)[c] with v[QF - 1] = 0
template <typename T, int QF, int QC>
__device__ __forceinline__ T down(const Interp<T, QF, QC>& J, const T (&v)[QF], int c) {
  T acc = J.mul(J.at(1, c), v[1]);
#pragma unroll
  for (int f = 2; f < QF - 1; ++f) acc = fma(J.at(f, c), v[f], acc);
  if (c == 0) acc = J.add(acc, v[0]);
  return acc;
}
// (J v)[f]
template <typename T, int QF, int QC>
__device__ __forceinline__ T up(const Interp<T, QF, QC>& J, const T (&v)[QC], int f) {
  if (f == 0) return v[0];
  if (f == QF - 1) return v[QC - 1];
  T acc = J.mul(J.at(f, 0), v[0]);
#pragma unroll
  for (int c = 1; c < QC; ++c) acc = fma(J.at(f, c), v[c], acc);
  return acc;
}

// J into shared memory for the passes whose output index differs between lanes.
template <typename T, int QF, int QC>
__device__ __forceinline__ void stage_J(T* sJ) {
  for (int q = threadIdx.x; q < QF * QC; q += blockDim.x) {
    if constexpr (sizeof(T) == 8) sJ[q] = __ldg(table_d<QF, QC>() + q);
    else sJ[q] = table_f<QF, QC>()[q];
  }
}

template <int QF>
constexpr int kElements = QF == 8 ? 2 : QF == 6 ? 7 : 16;        // elements per block: whole warps, nearly
template <int QF, int EB_>
struct Shape {
  static constexpr int T = QF * QF;                              // threads per element
  static constexpr int EB = EB_;
  static constexpr int THREADS = (EB * T + 31) / 32 * 32;
};

// Element coordinates without a division: e / d = high half of e * (floor(2^64 / d) + 1), exact for
// e d < 2^64.
struct BoxDiv {
  uint64_t m_xy, m_x;
};
BoxDiv box_div(const Lattice& L) {
  const uint64_t xy = (uint64_t)L.nex * (uint64_t)L.ney, x = (uint64_t)L.nex;
  return {xy > 1 ? ~0ull / xy + 1 : 0, x > 1 ? ~0ull / x + 1 : 0};   // 0: divisor 1
}
struct ElemCoord {
  int ex, ey, ez;
};
__device__ __forceinline__ ElemCoord elem_coord(int64_t e, const Lattice& L, const BoxDiv& d) {
  const uint32_t ee = (uint32_t)e, exy = (uint32_t)L.nex * (uint32_t)L.ney;
  const uint32_t ez = d.m_xy ? (uint32_t)__umul64hi(ee, d.m_xy) : ee;
  const uint32_t rem = ee - ez * exy;
  const uint32_t ey = d.m_x ? (uint32_t)__umul64hi(rem, d.m_x) : rem;
  return {(int)(rem - ey * (uint32_t)L.nex), (int)ey, (int)ez};
}

// Point i of Q along one direction of element ex of nex: on the box's boundary (Dirichlet)?
template <int Q>
__device__ __forceinline__ bool edge(int i, int ex, int nex) {
  return (i == 0 && ex == 0) || (i == Q - 1 && ex == nex - 1);
}
// Id of point (i, j, 0) of element c at Q points per direction, and the step to the next k.
template <int Q>
__device__ __forceinline__ uint32_t column_id(const Lattice& L, ElemCoord c, int i, int j, uint32_t& plane) {
  constexpr int N = Q - 1;
  plane = (uint32_t)L.NX * (uint32_t)L.NY;
  return (uint32_t)(c.ez * N) * plane + (uint32_t)(c.ey * N + j) * (uint32_t)L.NX + (uint32_t)(c.ex * N + i);
}

// rc += P^T rf (rc zeroed by the caller; coarse contributions summed by atomics).  An element owns
// its points below N in every direction, and a last element its end points too, which are
// boundary points: the free fine values of an element are those with i, j, k < N, so the last
// value of every line is zero.
template <typename T, int QF, int QC, int EB>
__global__ void __launch_bounds__(Shape<QF, EB>::THREADS)
k_restrict_box(int64_t E, Lattice Lf, Lattice Lc, BoxDiv bd, const T* __restrict__ rf, T* __restrict__ rc,
               int64_t ldf, int64_t ldc) {
  using S = Shape<QF, EB>;
  constexpr int NF = QF - 1;
  constexpr int NT = S::T, PB = QF * QF + 8, PC = QC * QF + 4;      // padded planes
  constexpr int L1 = QF * QC, S1 = NT / L1 < 1 ? 1 : (NT / L1 > QC ? QC : NT / L1), O1 = QC / S1;
  constexpr int L2 = QC * QC, S2 = NT / L2 < 1 ? 1 : (NT / L2 > QC ? QC : NT / L2), O2 = QC / S2;
  static_assert(O1 * S1 == QC && O2 * S2 == QC, "outputs split evenly");
  __shared__ T sB[S::EB][QC * PB];
  __shared__ T sC[S::EB][QC * PC];
  __shared__ T sJ[QF * QC];
  const Interp<T, QF, QC> J;
  stage_J<T, QF, QC>(sJ);
  const int le = threadIdx.x / NT, t = threadIdx.x - le * NT, a = t % QF, b = t / QF;
  const int64_t e = (int64_t)blockIdx.x * S::EB + le;
  const bool in = le < S::EB, valid = in && e < E;
  const ElemCoord c = valid ? elem_coord(e, Lf, bd) : ElemCoord{0, 0, 0};
  T* B = sB[in ? le : 0];
  T* C = sC[in ? le : 0];
  uint32_t plane;
  const uint32_t g0 = column_id<QF>(Lf, c, a, b, plane);
  const bool use = valid && a < NF && b < NF && !(a == 0 && c.ex == 0) && !(b == 0 && c.ey == 0);
  pdl_wait();   // rf (and the zeroed rc) may come from the kernel before
  rf += (int64_t)blockIdx.y * ldf;   // right-hand side of a batch
  rc += (int64_t)blockIdx.y * ldc;
  T v[QF];
#pragma unroll
  for (int k = 0; k < NF; ++k) v[k] = use && (k > 0 || c.ez > 0) ? rf[g0 + k * plane] : T(0);
  if (in && b < NF) {
#pragma unroll
    for (int kc = 0; kc < QC; ++kc) B[kc * PB + b * QF + a] = down<T, QF, QC>(J, v, kc);
  }
  __syncthreads();
  if (in && t < L1 * S1 && t % QF < NF) {   // along j: line (i, kc), O1 of its outputs
    const int i = t % QF, kc = (t / QF) % QC, part = t / L1;
#pragma unroll
    for (int l = 0; l < NF; ++l) v[l] = B[kc * PB + l * QF + i];
#pragma unroll
    for (int jc = 0; jc < QC; ++jc)
      if (jc / O1 == part) C[kc * PC + jc * QF + i] = down<T, QF, QC>(J, v, jc);
  }
  __syncthreads();
  if (valid && t < L2 * S2) {      // along i: line (jc, kc), O2 of its outputs
    const int part = t % S2, jc = (t / S2) % QC, kc = t / (S2 * QC);
#pragma unroll
    for (int l = 0; l < NF; ++l) v[l] = C[kc * PC + jc * QF + l];
    uint32_t cplane;
    const uint32_t cg = column_id<QC>(Lc, c, 0, jc, cplane) + kc * cplane;
    const bool out = edge<QC>(jc, c.ey, Lc.ney) || edge<QC>(kc, c.ez, Lc.nez);
#pragma unroll
    for (int o = 0; o < O2; ++o) {
      const int ic = part * O2 + o;
      T acc;
      if constexpr (S2 == 1) {
        acc = down<T, QF, QC>(J, v, o);
      } else {                     // the output differs between the lanes of a warp: J from shared memory
        acc = J.mul(sJ[ic], v[0]);
#pragma unroll
        for (int l = 1; l < NF; ++l) acc = fma(sJ[l * QC + ic], v[l], acc);
      }
      if (!out && !edge<QC>(ic, c.ex, Lc.nex)) atomicAdd(&rc[cg + ic], acc);
    }
  }
}

// zf (+)= P zc at the owned fine copies (boundary nodes: zero when not accumulating)
template <typename T, int QF, int QC, int EB>
__global__ void __launch_bounds__(Shape<QF, EB>::THREADS)
k_prolong_box(int64_t E, Lattice Lf, Lattice Lc, BoxDiv bd, const T* __restrict__ zc, T* __restrict__ zf,
              int accumulate, int64_t ldf, int64_t ldc) {
  using S = Shape<QF, EB>;
  constexpr int NF = QF - 1;
  constexpr int NT = S::T, PB = QC * QF + 4, PC = QF * QF + 8;
  constexpr int L1 = QC * QC, S1 = NT / L1 < 1 ? 1 : (NT / L1 > QF / 2 ? QF / 2 : NT / L1), O1 = (QF + S1 - 1) / S1;
  constexpr int L2 = QF * QC, S2 = NT / L2 < 1 ? 1 : NT / L2, O2 = (QF + S2 - 1) / S2;
  static_assert(O1 * S1 == QF && O2 * S2 == QF, "outputs split evenly");
  __shared__ T sA[S::EB][QC * QC * QC];
  __shared__ T sB[S::EB][QC * PB];
  __shared__ T sC[S::EB][QC * PC];
  __shared__ T sJ[QF * QC];
  const Interp<T, QF, QC> J;
  stage_J<T, QF, QC>(sJ);
  const int le = threadIdx.x / NT, t = threadIdx.x - le * NT, a = t % QF, b = t / QF;
  const int64_t e = (int64_t)blockIdx.x * S::EB + le;
  const bool in = le < S::EB, valid = in && e < E;
  const ElemCoord c = valid ? elem_coord(e, Lf, bd) : ElemCoord{0, 0, 0};
  T* A = sA[in ? le : 0];
  T* B = sB[in ? le : 0];
  T* C = sC[in ? le : 0];
  uint32_t plane;
  const uint32_t g0 = column_id<QF>(Lf, c, a, b, plane);
  // owned column, free of the side faces; its bottom point is free unless ez = 0, its top one
  // (owned by a last element alone) never
  const bool own = valid && (a < NF || c.ex == Lf.nex - 1) && (b < NF || c.ey == Lf.ney - 1);
  const bool inner = own && !edge<QF>(a, c.ex, Lf.nex) && !edge<QF>(b, c.ey, Lf.ney);
  pdl_wait();   // zc and zf may come from the kernels before
  zf += (int64_t)blockIdx.y * ldf;
  zc += (int64_t)blockIdx.y * ldc;
  T* col = zf + g0;
  // the fine column's old values first: in flight during the whole interpolation
  T old[NF];
#pragma unroll
  for (int k = 0; k < NF; ++k) old[k] = accumulate && inner && (k > 0 || c.ez > 0) ? col[(size_t)k * plane] : T(0);
  if (in)
    for (int p = t; p < QC * QC * QC; p += NT) {
      const int i = p % QC, j = (p / QC) % QC, k = p / (QC * QC);
      uint32_t cplane;
      const uint32_t cg = column_id<QC>(Lc, c, i, j, cplane) + k * cplane;
      const bool out = edge<QC>(i, c.ex, Lc.nex) || edge<QC>(j, c.ey, Lc.ney) || edge<QC>(k, c.ez, Lc.nez);
      A[p] = (valid && !out) ? zc[cg] : T(0);
    }
  __syncthreads();
  T v[QC];
  if (in && t < L1 * S1) {         // along i: line (jc, kc), O1 of its outputs
    const int part = t % S1, line = t / S1, jc = line % QC, kc = line / QC;
#pragma unroll
    for (int l = 0; l < QC; ++l) v[l] = A[line * QC + l];
#pragma unroll
    for (int o = 0; o < O1; ++o) {
      const int f = part * O1 + o;
      T acc;
      if constexpr (S1 == 1) {
        acc = up<T, QF, QC>(J, v, o);
      } else {                     // the output differs between the lanes of a warp: J from shared memory
        acc = J.mul(sJ[f * QC], v[0]);
#pragma unroll
        for (int l = 1; l < QC; ++l) acc = fma(sJ[f * QC + l], v[l], acc);
      }
      B[kc * PB + jc * QF + f] = acc;
    }
  }
  __syncthreads();
  if (in && t < L2 * S2) {         // along j: line (i, kc), O2 of its outputs
    const int i = t % QF, kc = (t / QF) % QC, part = t / L2;
#pragma unroll
    for (int l = 0; l < QC; ++l) v[l] = B[kc * PB + l * QF + i];
#pragma unroll
    for (int f = 0; f < QF; ++f)
      if (f / O2 == part) C[kc * PC + f * QF + i] = up<T, QF, QC>(J, v, f);
  }
  __syncthreads();
  if (inner) {                     // along k: fine column (a, b)
#pragma unroll
    for (int l = 0; l < QC; ++l) v[l] = C[l * PC + b * QF + a];
#pragma unroll
    for (int k = 0; k < NF; ++k) {
      const T acc = up<T, QF, QC>(J, v, k);
      if (k > 0 || c.ez > 0) col[(size_t)k * plane] = accumulate ? J.add(acc, old[k]) : acc;
    }
  }
  if (!accumulate && own) {        // boundary points
    const bool top = c.ez == Lf.nez - 1;
#pragma unroll
    for (int k = 0; k < QF; ++k)
      if (k == NF ? top : !inner || (k == 0 && c.ez == 0)) col[(size_t)k * plane] = T(0);
  }
}

}  // namespace

template <int QF, int QC>
static cudaError_t set_J(const double* J, const void* sym_d, const void* sym_f) {
  // the kernels use unit end rows and the mirror symmetry of the interior ones (to rounding)
  for (int c = 0; c < QC; ++c)
    if (J[c] != (c == 0 ? 1.0 : 0.0) || J[(QF - 1) * QC + c] != (c == QC - 1 ? 1.0 : 0.0)) return cudaErrorInvalidValue;
  float f[QF * QC];
  for (int q = 0; q < QF * QC; ++q) f[q] = (float)J[q];
  cudaError_t e = cudaMemcpyToSymbol(sym_d, J, sizeof(double) * QF * QC);
  return e != cudaSuccess ? e : cudaMemcpyToSymbol(sym_f, f, sizeof(f));
}

cudaError_t transfer_box_set_J(int Qf, int Qc, const double* J) {
  if (Qf == 8 && Qc == 4) return set_J<8, 4>(J, g_J84_d, c_J84_f);
  if (Qf == 4 && Qc == 2) return set_J<4, 2>(J, g_J42_d, c_J42_f);
  if (Qf == 8 && Qc == 6) return set_J<8, 6>(J, g_J86_d, c_J86_f);
  if (Qf == 6 && Qc == 4) return set_J<6, 4>(J, g_J64_d, c_J64_f);
  return cudaErrorInvalidValue;
}

bool transfer_box_supported(int Qf, int Qc) {
  return (Qf == 8 && Qc == 4) || (Qf == 4 && Qc == 2) || (Qf == 8 && Qc == 6) || (Qf == 6 && Qc == 4);
}

// Elements per block at order 5 in FP64: seven, or fewer where the busiest SM then has fewer warps to issue
// for -- a full block's seven elements are FP64 work in series on one SM.  One element on up to 456
// elements (a single 5 -> 3 interpolation, with its synchronisation, on 64 to 392 elements 20.4 -> 18.2 us,
// a restriction 20.8 -> 18.4), five where seven make a nearly empty last wave (1,100 elements 22.3 -> 21.0).
// Order 7 has two elements in a block, order 3 little work in each, and FP32 is not bound by its issue on
// so few.
template <int QF>
int elements_per_block(int64_t E, int nb) {
  const int sms = sm_count();
  int eb = 0;
  int64_t least = 0;
  auto consider = [&](int e, int threads) {
    const int64_t w = ((E + e - 1) / e * nb + sms - 1) / sms * (threads / 32);
    if (eb == 0 || w < least) least = w, eb = e;
  };
  consider(kElements<QF>, Shape<QF, kElements<QF>>::THREADS);
  consider(1, Shape<QF, 1>::THREADS);
  consider(5, Shape<QF, 5>::THREADS);
  return eb;
}

template <typename T, int QF, int QC, int EB>
static void launch_restrict_eb(int64_t E, const Lattice& Lf, const Lattice& Lc, const T* rf, T* rc, cudaStream_t s,
                               int nb, int64_t ldf, int64_t ldc) {
  launch_dep(k_restrict_box<T, QF, QC, EB>, dim3((unsigned)((E + EB - 1) / EB), nb), dim3(Shape<QF, EB>::THREADS), 0,
             s, E, Lf, Lc, box_div(Lf), rf, rc, ldf, ldc);
}
template <typename T, int QF, int QC, int EB>
static void launch_prolong_eb(int64_t E, const Lattice& Lf, const Lattice& Lc, const T* zc, T* zf, int accumulate,
                              cudaStream_t s, int nb, int64_t ldf, int64_t ldc) {
  launch_dep(k_prolong_box<T, QF, QC, EB>, dim3((unsigned)((E + EB - 1) / EB), nb), dim3(Shape<QF, EB>::THREADS), 0,
             s, E, Lf, Lc, box_div(Lf), zc, zf, accumulate, ldf, ldc);
}
template <typename T, int QF, int QC>
static void launch_restrict(int64_t E, const Lattice& Lf, const Lattice& Lc, const T* rf, T* rc, cudaStream_t s, int nb,
                            int64_t ldf, int64_t ldc) {
  if constexpr (sizeof(T) == 8 && QF == 6) {
    const int eb = elements_per_block<QF>(E, nb);
    if (eb == 1) return launch_restrict_eb<T, QF, QC, 1>(E, Lf, Lc, rf, rc, s, nb, ldf, ldc);
    if (eb == 5) return launch_restrict_eb<T, QF, QC, 5>(E, Lf, Lc, rf, rc, s, nb, ldf, ldc);
  }
  launch_restrict_eb<T, QF, QC, kElements<QF>>(E, Lf, Lc, rf, rc, s, nb, ldf, ldc);
}
template <typename T, int QF, int QC>
static void launch_prolong(int64_t E, const Lattice& Lf, const Lattice& Lc, const T* zc, T* zf, int accumulate,
                           cudaStream_t s, int nb, int64_t ldf, int64_t ldc) {
  if constexpr (sizeof(T) == 8 && QF == 6) {
    const int eb = elements_per_block<QF>(E, nb);
    if (eb == 1) return launch_prolong_eb<T, QF, QC, 1>(E, Lf, Lc, zc, zf, accumulate, s, nb, ldf, ldc);
    if (eb == 5) return launch_prolong_eb<T, QF, QC, 5>(E, Lf, Lc, zc, zf, accumulate, s, nb, ldf, ldc);
  }
  launch_prolong_eb<T, QF, QC, kElements<QF>>(E, Lf, Lc, zc, zf, accumulate, s, nb, ldf, ldc);
}

template <typename T>
void restrict_box(int Qf, int Qc, int64_t E, const Lattice& Lf, const Lattice& Lc, const T* rf, T* rc,
                  cudaStream_t s, int nb, int64_t ldf, int64_t ldc) {
  if (Qf == 8 && Qc == 4) launch_restrict<T, 8, 4>(E, Lf, Lc, rf, rc, s, nb, ldf, ldc);
  else if (Qf == 8 && Qc == 6) launch_restrict<T, 8, 6>(E, Lf, Lc, rf, rc, s, nb, ldf, ldc);
  else if (Qf == 6 && Qc == 4) launch_restrict<T, 6, 4>(E, Lf, Lc, rf, rc, s, nb, ldf, ldc);
  else launch_restrict<T, 4, 2>(E, Lf, Lc, rf, rc, s, nb, ldf, ldc);
}

template <typename T>
void prolong_box(int Qf, int Qc, int64_t E, const Lattice& Lf, const Lattice& Lc, const T* zc, T* zf,
                 int accumulate, cudaStream_t s, int nb, int64_t ldf, int64_t ldc) {
  if (Qf == 8 && Qc == 4) launch_prolong<T, 8, 4>(E, Lf, Lc, zc, zf, accumulate, s, nb, ldf, ldc);
  else if (Qf == 8 && Qc == 6) launch_prolong<T, 8, 6>(E, Lf, Lc, zc, zf, accumulate, s, nb, ldf, ldc);
  else if (Qf == 6 && Qc == 4) launch_prolong<T, 6, 4>(E, Lf, Lc, zc, zf, accumulate, s, nb, ldf, ldc);
  else launch_prolong<T, 4, 2>(E, Lf, Lc, zc, zf, accumulate, s, nb, ldf, ldc);
}

template void restrict_box<float>(int, int, int64_t, const Lattice&, const Lattice&, const float*, float*,
                                  cudaStream_t, int, int64_t, int64_t);
template void restrict_box<double>(int, int, int64_t, const Lattice&, const Lattice&, const double*, double*,
                                   cudaStream_t, int, int64_t, int64_t);
template void prolong_box<float>(int, int, int64_t, const Lattice&, const Lattice&, const float*, float*, int,
                                 cudaStream_t, int, int64_t, int64_t);
template void prolong_box<double>(int, int, int64_t, const Lattice&, const Lattice&, const double*, double*, int,
                                  cudaStream_t, int, int64_t, int64_t);

}  // namespace chebmg
