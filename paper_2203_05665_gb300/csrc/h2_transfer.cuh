// Transfer steps of the H^2 product (Algorithms 1 and 2) with the factored
// transfer matrices E = Ex (x) Ey (x) Ez of tensor Chebyshev interpolation
// (Eq. (9)): three m x m mode products per child instead of one k x k
// product.  Shared by the single-matrix and the batched products.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "h2_dd.cuh"
#include "h2_launch.cuh"

namespace h2 {
namespace {

constexpr int kMaxM = 5;

// storage -> compute conversion of a transfer factor
template <class TC, class TS>
__device__ __forceinline__ TC to_compute(TS v) {
  return convert<TC, TS>(v);
}
template <>
__device__ __forceinline__ float to_compute<float, __nv_bfloat16>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}
template <>
__device__ __forceinline__ float to_compute<float, __half>(__half v) {
  return __half2float(v);
}

// ---------------------------------------------------------------------------
// Register transfer kernels for m = 3 and m = 4 (k = m^3): 64 threads per
// parent and 16 columns (grid.y runs over groups of 16 columns), thread
// (j, jz) = (column, z index; jz < m, the fourth lane of a column idles for
// m = 3) holds the m x m slab nu = jx + m jy + m^2 jz of one column in
// registers.  The x and y mode products run in registers, the z mode product
// takes the slab entries of the threads of the column (adjacent lanes) by
// warp shuffles, so no barrier separates the three mode products.  Every output
// is formed by m multiply-adds and one renormalisation, axes x, y, z in turn.
// Used for the wide upward levels in FP32 (launch_up_m).
constexpr int kRegParents = 4;   // parents per 256-thread CTA

__device__ __forceinline__ float shfl_t(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// out[a] = sum_b F[a][b] in[b] (plain, E) or sum_b F[b][a] in[b] (trans, E^T)
template <class T, bool TRANS, int M>
__device__ __forceinline__ T modem_out(const T *F, const T (&in)[M], int a) {
  T acc;
  acc_mul(acc, F[TRANS ? a : a * M], in[0]);
#pragma unroll
  for (int b = 1; b < M; ++b) acc_fma(acc, TRANS ? F[b * M + a] : F[a * M + b], in[b]);
  acc_norm(acc);
  return acc;
}

// the transfer factors of the children of this CTA's parents: F[q][ch][axis][M x M]
template <class TS, class T, int M, int P = kRegParents>
__device__ __forceinline__ void load_factors(const TS *__restrict__ Ef, int64_t par0, int64_t npar,
                                             T (*F)[2][3][M * M]) {
  constexpr int kPer = 6 * M * M, kChild = 3 * M * M;
  for (int i = threadIdx.x; i < P * kPer; i += blockDim.x) {
    const int q = i / kPer, o = i % kPer;
    const int64_t pi = (int64_t)blockIdx.x * P + q;
    const int64_t pp = par0 + pi;
    F[q][o / kChild][(o % kChild) / (M * M)][o % (M * M)] =
        pi < npar ? to_compute<T>(Ef[(2 * pp + 1) * kChild + o]) : zero_of<T>();
  }
  __syncthreads();
}

// Upward (Algorithm 1): x^_parent = sum over both children of E_c^T x^_c.
// With xmax, also the largest |x^_parent| (|hi| for double-float) of every
// column over the launch, as float bits (atomicMax; infinities and NaN are above all
// others).
__device__ __forceinline__ float mag_of(float v) { return fabsf(v); }
__device__ __forceinline__ float mag_of(double v) { return (float)fabs(v); }
__device__ __forceinline__ float mag_of(dd v) { return fabsf(v.hi); }

template <class TS, class T, int M>
__global__ void __launch_bounds__(256, 2) k_up_reg(const TS *__restrict__ Ef, int rp, int64_t par0, int64_t npar,
                                                   T *__restrict__ xhat, unsigned *__restrict__ xmax) {
  pdl_wait();
  pdl_go();
  constexpr int K = M * M * M;
  __shared__ T F[kRegParents][2][3][M * M];
  __shared__ unsigned loc[16];
  if (threadIdx.x < 16) loc[threadIdx.x] = 0u;
  load_factors<TS, T, M>(Ef, par0, npar, F);
  const int pl = threadIdx.x >> 6, t = threadIdx.x & 63, j = (t >> 2) + 16 * blockIdx.y, jz = t & 3;
  const int64_t pi = (int64_t)blockIdx.x * kRegParents + pl, par = par0 + pi;
  const bool act = pi < npar && j < rp && jz < M;
  const int base = (threadIdx.x & 31) & ~3;
  const int zq = jz < M ? jz : 0;
  T out[M][M];
#pragma unroll 1
  for (int ch = 0; ch < 2; ++ch) {
    const int64_t c = 2 * par + 1 + ch;
    const T *Fx = F[pl][ch][0], *Fy = F[pl][ch][1], *Fz = F[pl][ch][2];
    T v[M][M], a[M][M], b[M][M];
#pragma unroll
    for (int jy = 0; jy < M; ++jy)
#pragma unroll
      for (int jx = 0; jx < M; ++jx)
        v[jy][jx] = act ? xhat[(c * K + jx + M * jy + M * M * jz) * rp + j] : zero_of<T>();
#pragma unroll
    for (int jy = 0; jy < M; ++jy)
#pragma unroll
      for (int jx = 0; jx < M; ++jx) a[jy][jx] = modem_out<T, true, M>(Fx, v[jy], jx);
#pragma unroll
    for (int jx = 0; jx < M; ++jx) {
      T col[M];
#pragma unroll
      for (int jy = 0; jy < M; ++jy) col[jy] = a[jy][jx];
#pragma unroll
      for (int jy = 0; jy < M; ++jy) b[jy][jx] = modem_out<T, true, M>(Fy, col, jy);
    }
#pragma unroll
    for (int jy = 0; jy < M; ++jy)
#pragma unroll
      for (int jx = 0; jx < M; ++jx) {
        T in[M];
#pragma unroll
        for (int q = 0; q < M; ++q) in[q] = shfl_t(b[jy][jx], base + q);
        const T r = modem_out<T, true, M>(Fz, in, zq);
        out[jy][jx] = ch == 0 ? zero_of<T>() + r : out[jy][jx] + r;
      }
  }
  unsigned mx = 0u;
#pragma unroll
  for (int jy = 0; jy < M; ++jy)
#pragma unroll
    for (int jx = 0; jx < M; ++jx) {
      if (act) xhat[(par * K + jx + M * jy + M * M * jz) * rp + j] = out[jy][jx];
      if (act) mx = max(mx, __float_as_uint(mag_of(out[jy][jx])));
    }
  if (xmax) {
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    if (act && jz == 0 && mx) atomicMax(&loc[j & 15], mx);
    __syncthreads();
    if (threadIdx.x < 16 && loc[threadIdx.x]) atomicMax(&xmax[16 * blockIdx.y + threadIdx.x], loc[threadIdx.x]);
  }
}

// Child-split variants: 128 threads per parent, the two 64-thread halves
// taking one child each (two parents per 256-thread CTA), so every thread
// forms half the mode products.  On levels with few parents a CTA's time is
// the latency of one thread's chain of operations, which this
// halves.  The second child's part is added to the first through shared memory
// in the order of k_up_reg (same bits).
constexpr int kSplitParents = 2;   // parents per 256-thread CTA
// upward levels of at most this many parents take the split kernel (measured
// at 327,680 triangles, 16 right-hand sides)
constexpr int64_t kUpSplitMax = 4096;

template <class TS, class T, int M>
__global__ void __launch_bounds__(256, 2) k_up_split(const TS *__restrict__ Ef, int rp, int64_t par0, int64_t npar,
                                                     T *__restrict__ xhat, unsigned *__restrict__ xmax) {
  pdl_wait();
  pdl_go();
  constexpr int K = M * M * M;
  __shared__ T F[kSplitParents][2][3][M * M];
  __shared__ T R[kSplitParents][M * M][64];   // the second child's part
  __shared__ unsigned loc[16];
  if (threadIdx.x < 16) loc[threadIdx.x] = 0u;
  load_factors<TS, T, M, kSplitParents>(Ef, par0, npar, F);
  const int pl = threadIdx.x >> 7, ch = (threadIdx.x >> 6) & 1, t = threadIdx.x & 63;
  const int j = (t >> 2) + 16 * blockIdx.y, jz = t & 3;
  const int64_t pi = (int64_t)blockIdx.x * kSplitParents + pl, par = par0 + pi;
  const bool act = pi < npar && j < rp && jz < M;
  const int base = (threadIdx.x & 31) & ~3;
  const int zq = jz < M ? jz : 0;
  const int64_t c = 2 * par + 1 + ch;
  const T *Fx = F[pl][ch][0], *Fy = F[pl][ch][1], *Fz = F[pl][ch][2];
  T v[M][M], a[M][M], b[M][M];
#pragma unroll
  for (int jy = 0; jy < M; ++jy)
#pragma unroll
    for (int jx = 0; jx < M; ++jx)
      v[jy][jx] = act ? xhat[(c * K + jx + M * jy + M * M * jz) * rp + j] : zero_of<T>();
#pragma unroll
  for (int jy = 0; jy < M; ++jy)
#pragma unroll
    for (int jx = 0; jx < M; ++jx) a[jy][jx] = modem_out<T, true, M>(Fx, v[jy], jx);
#pragma unroll
  for (int jx = 0; jx < M; ++jx) {
    T col[M];
#pragma unroll
    for (int jy = 0; jy < M; ++jy) col[jy] = a[jy][jx];
#pragma unroll
    for (int jy = 0; jy < M; ++jy) b[jy][jx] = modem_out<T, true, M>(Fy, col, jy);
  }
  // the z mode product into a (the slab is free again)
#pragma unroll
  for (int jy = 0; jy < M; ++jy)
#pragma unroll
    for (int jx = 0; jx < M; ++jx) {
      T in[M];
#pragma unroll
      for (int q = 0; q < M; ++q) in[q] = shfl_t(b[jy][jx], base + q);
      a[jy][jx] = modem_out<T, true, M>(Fz, in, zq);
    }
  if (ch == 1)
#pragma unroll
    for (int jy = 0; jy < M; ++jy)
#pragma unroll
      for (int jx = 0; jx < M; ++jx) R[pl][jx + M * jy][t] = a[jy][jx];
  __syncthreads();
  unsigned mx = 0u;
  if (ch == 0)
#pragma unroll
    for (int jy = 0; jy < M; ++jy)
#pragma unroll
      for (int jx = 0; jx < M; ++jx) {
        const T o = (zero_of<T>() + a[jy][jx]) + R[pl][jx + M * jy][t];
        if (act) xhat[(par * K + jx + M * jy + M * M * jz) * rp + j] = o;
        if (act) mx = max(mx, __float_as_uint(mag_of(o)));
      }
  if (xmax) {
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    if (ch == 0 && act && jz == 0 && mx) atomicMax(&loc[j & 15], mx);
    __syncthreads();
    if (threadIdx.x < 16 && loc[threadIdx.x]) atomicMax(&xmax[16 * blockIdx.y + threadIdx.x], loc[threadIdx.x]);
  }
}

// ---------------------------------------------------------------------------
// Transfer kernels with one output pair per thread: a parent has M^3 x NP
// threads, thread (nu, p) forms the coefficient nu of two neighbouring columns
// (one 16-byte value pair for double-float) in each of the three mode products,
// which exchange their tensors through shared memory.  The children of a
// parent are taken in turn.  Threads exist for the columns there are, PP
// parents share a CTA, and a thread's chain is twelve multiply-adds per child
// instead of the register kernels' hundreds (whose unrolled code also misses
// the instruction cache on narrow levels).  Every output is formed by the same
// operations in the same order as there, so the bits are the same.  Narrow
// levels: 8 - 9 us per level with the register kernels (order 4, double-float),
// 4 - 5 us here; 81,920 triangles, order 4, one column, all upward levels 122
// -> 64 us (51 us with the shorter sums of mode_pair).
template <class T>
struct alignas(2 * sizeof(T)) Pair {
  T a, b;
};

// columns of a CTA in pairs (grid.y runs over groups of this many)
template <int M>
__host__ __device__ constexpr int pair_max() { return M == 5 ? 4 : 8; }

// sum_b F[b][j] (up) or F[j][b] (down) in[base + b stride], both columns.  The
// first term is a plain product: added to zero like the others it cost 8 of 54
// FP32 instructions per double-float sum (327,680 triangles, order 4, 16 columns:
// upward 409 -> 386 us with the digit cut, downward 291 -> 271 us).
template <class T, bool TRANS, int M>
__device__ __forceinline__ Pair<T> mode_pair(const T *F, int j, const Pair<T> *in, int stride) {
  Pair<T> o;
#pragma unroll
  for (int b = 0; b < M; ++b) {
    const T f = TRANS ? F[b * M + j] : F[j * M + b];
    const Pair<T> v = in[b * stride];
    if (b == 0) {
      acc_mul(o.a, f, v.a);
      acc_mul(o.b, f, v.b);
    } else {
      acc_fma(o.a, f, v.a);
      acc_fma(o.b, f, v.b);
    }
  }
  acc_norm(o.a);
  acc_norm(o.b);
  return o;
}

template <class TS, class T, int M>
__device__ __forceinline__ void pair_factors(const TS *__restrict__ Ef, int64_t par, int64_t npar_left, int pp, T *F) {
  constexpr int kPer = 6 * M * M;
  const int n = npar_left < pp ? (int)npar_left : pp;
  for (int i = threadIdx.x; i < n * kPer; i += blockDim.x)
    F[i] = to_compute<T>(Ef[(2 * par + 1) * (3 * M * M) + i]);   // the children of consecutive parents are consecutive
}

// The bodies: CTA bx of the launch (or of its part of a batched launch), column
// group by; psm: shared memory of pair_smem bytes, loc: 16 shared words.
template <class TS, class T, int M>
__device__ __forceinline__ void up_pair(const TS *__restrict__ Ef, int rp, int np, int pp, int64_t par0, int64_t npar,
                                        T *__restrict__ xhat, unsigned *__restrict__ xmax, int bx, int by,
                                        unsigned char *psm, unsigned *loc) {
  constexpr int K = M * M * M;
  const int tpp = K * np, pl = (int)threadIdx.x / tpp, rem = (int)threadIdx.x - pl * tpp;
  Pair<T> *buf = reinterpret_cast<Pair<T> *>(psm);          // [2][pp][K][np]
  T *F = reinterpret_cast<T *>(buf + 2 * pp * tpp);         // [pp][2][3][M x M]
  if (threadIdx.x < 16) loc[threadIdx.x] = 0u;
  const int64_t p0 = (int64_t)bx * pp, par = par0 + p0 + pl;
  const int nu = rem / np, p = rem - nu * np, col = 2 * (pair_max<M>() * by + p);
  const int jx = nu % M, jy = (nu / M) % M, jz = nu / (M * M);
  const bool act = pl < pp && p0 + pl < npar && col < rp;
  pair_factors<TS, T, M>(Ef, par0 + p0, npar - p0, pp, F);
  pdl_wait();
  pdl_go();
  Pair<T> v[2];
#pragma unroll
  for (int ch = 0; ch < 2; ++ch)
    v[ch] = act ? *reinterpret_cast<const Pair<T> *>(xhat + ((2 * par + 1 + ch) * K + nu) * rp + col)
                : Pair<T>{zero_of<T>(), zero_of<T>()};
  const int slot = pl < pp ? (int)threadIdx.x : 0, at = pl < pp ? pl * tpp + p : 0;
  const T *Fp = F + (pl < pp ? pl : 0) * 6 * M * M;
  Pair<T> acc;
#pragma unroll
  for (int ch = 0; ch < 2; ++ch) {
    Pair<T> *A = buf + (ch ? pp * tpp : 0), *Bf = buf + (ch ? 0 : pp * tpp);
    const T *Fc = Fp + ch * 3 * M * M;
    if (pl < pp) A[slot] = v[ch];
    __syncthreads();
    Pair<T> o = mode_pair<T, true, M>(Fc, jx, A + at + (nu - jx) * np, np);
    if (pl < pp) Bf[slot] = o;
    __syncthreads();
    o = mode_pair<T, true, M>(Fc + M * M, jy, Bf + at + (nu - M * jy) * np, M * np);
    if (pl < pp) A[slot] = o;
    __syncthreads();
    o = mode_pair<T, true, M>(Fc + 2 * M * M, jz, A + at + (nu - M * M * jz) * np, M * M * np);
    acc = ch == 0 ? o : Pair<T>{acc.a + o.a, acc.b + o.b};
  }
  if (act) *reinterpret_cast<Pair<T> *>(xhat + (par * K + nu) * rp + col) = acc;
  if (xmax) {
    if (act) {
      atomicMax(&loc[2 * p], __float_as_uint(mag_of(acc.a)));
      atomicMax(&loc[2 * p + 1], __float_as_uint(mag_of(acc.b)));
    }
    __syncthreads();
    unsigned *dst = xmax + 2 * pair_max<M>() * by + threadIdx.x;
    if (threadIdx.x < 16 && loc[threadIdx.x] && loc[threadIdx.x] > __ldcg(dst)) atomicMax(dst, loc[threadIdx.x]);
  }
}

template <class TS, class T, int M>
__global__ void __launch_bounds__(512, 3) k_up_pair(const TS *__restrict__ Ef, int rp, int np, int pp, int64_t par0,
                                                    int64_t npar, T *__restrict__ xhat, unsigned *__restrict__ xmax) {
  extern __shared__ __align__(16) unsigned char psm[];
  __shared__ unsigned loc[16];
  up_pair<TS, T, M>(Ef, rp, np, pp, par0, npar, xhat, xmax, (int)blockIdx.x, (int)blockIdx.y, psm, loc);
}

template <class TS, class T, int M>
__device__ __forceinline__ void down_pair(const TS *__restrict__ Ef, int rp, int np, int pp, int64_t par0,
                                          int64_t npar, T *__restrict__ yhat, int bx, int by, unsigned char *psm) {
  constexpr int K = M * M * M;
  const int tpp = K * np, pl = (int)threadIdx.x / tpp, rem = (int)threadIdx.x - pl * tpp;
  Pair<T> *P = reinterpret_cast<Pair<T> *>(psm), *A = P + pp * tpp, *Bf = A + pp * tpp;   // [pp][K][np] each
  T *F = reinterpret_cast<T *>(Bf + pp * tpp);
  const int64_t p0 = (int64_t)bx * pp, par = par0 + p0 + pl;
  const int nu = rem / np, p = rem - nu * np, col = 2 * (pair_max<M>() * by + p);
  const int jx = nu % M, jy = (nu / M) % M, jz = nu / (M * M);
  const bool act = pl < pp && p0 + pl < npar && col < rp;
  const Pair<T> zero{zero_of<T>(), zero_of<T>()};
  pair_factors<TS, T, M>(Ef, par0 + p0, npar - p0, pp, F);
  pdl_wait();
  pdl_go();
  const Pair<T> v = act ? *reinterpret_cast<const Pair<T> *>(yhat + (par * K + nu) * rp + col) : zero;
  Pair<T> yc[2];
#pragma unroll
  for (int ch = 0; ch < 2; ++ch)
    yc[ch] = act ? *reinterpret_cast<const Pair<T> *>(yhat + ((2 * par + 1 + ch) * K + nu) * rp + col) : zero;
  const int slot = pl < pp ? (int)threadIdx.x : 0, at = pl < pp ? pl * tpp + p : 0;
  const T *Fp = F + (pl < pp ? pl : 0) * 6 * M * M;
  if (pl < pp) P[slot] = v;
  __syncthreads();
#pragma unroll
  for (int ch = 0; ch < 2; ++ch) {
    const T *Fc = Fp + ch * 3 * M * M;
    Pair<T> o = mode_pair<T, false, M>(Fc, jx, P + at + (nu - jx) * np, np);
    if (pl < pp) A[slot] = o;
    __syncthreads();
    o = mode_pair<T, false, M>(Fc + M * M, jy, A + at + (nu - M * jy) * np, M * np);
    if (pl < pp) Bf[slot] = o;
    __syncthreads();
    o = mode_pair<T, false, M>(Fc + 2 * M * M, jz, Bf + at + (nu - M * M * jz) * np, M * M * np);
    if (act)
      *reinterpret_cast<Pair<T> *>(yhat + ((2 * par + 1 + ch) * K + nu) * rp + col) =
          Pair<T>{yc[ch].a + o.a, yc[ch].b + o.b};
  }
}

template <class TS, class T, int M>
__global__ void __launch_bounds__(512, 3) k_down_pair(const TS *__restrict__ Ef, int rp, int np, int pp, int64_t par0,
                                                      int64_t npar, T *__restrict__ yhat) {
  extern __shared__ __align__(16) unsigned char psm[];
  down_pair<TS, T, M>(Ef, rp, np, pp, par0, npar, yhat, (int)blockIdx.x, (int)blockIdx.y, psm);
}

// shared memory of a CTA: two (up) or three (down) tensors per parent and the factors
template <class T>
inline size_t pair_smem(int m, int np, int pp, bool down) {
  return (size_t)pp * ((down ? 3 : 2) * m * m * m * np * sizeof(Pair<T>) + 6 * m * m * sizeof(T));
}

// parents of a CTA of the pair kernels: 512 threads on wide levels, fewer where
// that leaves SMs without a CTA
inline int pair_parents(int m, int64_t npar, int np) {
  const int most = std::max(1, 512 / (m * m * m * np));
  return (int)std::max<int64_t>(1, std::min<int64_t>(most, npar / (2 * 152)));
}

// Upward levels that take the pair kernel: every level in double-float (and
// double) arithmetic, orders other than 3 and 4, and in FP32 up to 8 columns
// and narrow levels.  Wide FP32 levels of more columns are bound by the pair
// kernel's shared-memory reads (eight per four multiply-adds): 327,680
// triangles, order 4, 16 columns 210 us with the register kernels, 238 us
// without; 1.3 M triangles, order 3, 4 columns 150 us with them, 95 us without.
// Downward the pair kernel was never slower (1.3 M, 4 columns 193 -> 93 us;
// 327,680, 16 columns FP32 146 -> 133 us, double-float 343 -> 306 us; 81,920,
// one column, double-float order 4 121 -> 64 us; now 113, 271 and 33 us).
template <class T>
inline bool pair_up(int m, int64_t npar, int rp) {
  return sizeof(T) == 8 || (m != 3 && m != 4) || rp <= 8 || npar * rp <= 4096;
}

template <class TS, class T, int M>
void launch_up_m(const TS *Ef, int rp, int64_t par0, int64_t npar, T *xhat, unsigned *xmax, cudaStream_t st) {
  if (pair_up<T>(M, npar, rp)) {
    const int np = std::min(pair_max<M>(), rp / 2), pp = pair_parents(M, npar, np), thr = (pp * M * M * M * np + 31) / 32 * 32;
    const dim3 grid((unsigned)((npar + pp - 1) / pp), (rp / 2 + np - 1) / np);
    pdl(k_up_pair<TS, T, M>, grid, thr, pair_smem<T>(M, np, pp, false), st, 
        Ef, rp, np, pp, par0, npar, xhat, xmax);
    return;
  }
  if constexpr (sizeof(T) == 4 && (M == 3 || M == 4)) {   // the only ones pair_up leaves
    const int gy = (rp + 15) / 16;
    if (npar <= kUpSplitMax)
      pdl(k_up_split<TS, T, M>, dim3((unsigned)((npar + kSplitParents - 1) / kSplitParents), gy), 256, 0, st, 
          Ef, rp, par0, npar, xhat, xmax);
    else
      pdl(k_up_reg<TS, T, M>, dim3((unsigned)((npar + kRegParents - 1) / kRegParents), gy), 256, 0, st, 
          Ef, rp, par0, npar, xhat, xmax);
  }
}

template <class TS, class T, int M>
void launch_down_m(const TS *Ef, int rp, int64_t par0, int64_t npar, T *yhat, cudaStream_t st) {
  const int np = std::min(pair_max<M>(), rp / 2), pp = pair_parents(M, npar, np), thr = (pp * M * M * M * np + 31) / 32 * 32;
  const dim3 grid((unsigned)((npar + pp - 1) / pp), (rp / 2 + np - 1) / np);
  pdl(k_down_pair<TS, T, M>, grid, thr, pair_smem<T>(M, np, pp, true), st, 
      Ef, rp, np, pp, par0, npar, yhat);
}

// the upward step for parents par0 .. par0 + npar - 1, and the downward step below them
template <class TS, class T>
void launch_up(const TS *Ef, int m, int rp, int64_t par0, int64_t npar, T *xhat, unsigned *xmax, cudaStream_t st) {
  switch (m) {
    case 1: return launch_up_m<TS, T, 1>(Ef, rp, par0, npar, xhat, xmax, st);
    case 2: return launch_up_m<TS, T, 2>(Ef, rp, par0, npar, xhat, xmax, st);
    case 3: return launch_up_m<TS, T, 3>(Ef, rp, par0, npar, xhat, xmax, st);
    case 4: return launch_up_m<TS, T, 4>(Ef, rp, par0, npar, xhat, xmax, st);
    default: return launch_up_m<TS, T, 5>(Ef, rp, par0, npar, xhat, xmax, st);
  }
}
template <class TS, class T>
void launch_down(const TS *Ef, int m, int rp, int64_t par0, int64_t npar, T *yhat, cudaStream_t st) {
  switch (m) {
    case 1: return launch_down_m<TS, T, 1>(Ef, rp, par0, npar, yhat, st);
    case 2: return launch_down_m<TS, T, 2>(Ef, rp, par0, npar, yhat, st);
    case 3: return launch_down_m<TS, T, 3>(Ef, rp, par0, npar, yhat, st);
    case 4: return launch_down_m<TS, T, 4>(Ef, rp, par0, npar, yhat, st);
    default: return launch_down_m<TS, T, 5>(Ef, rp, par0, npar, yhat, st);
  }
}

}  // namespace
}  // namespace h2
