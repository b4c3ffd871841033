// Device helpers of the tensor-core phases (h2_tc.cu, h2_tile.cu): tcgen05
// issue and tensor-memory reads, operand layouts, and the digit cut of
// double-float and FP32 values.
#pragma once

#include <cuda_fp8.h>

#include "h2_dd.cuh"
#include "h2_internal.hpp"
#include "h2_digits.hpp"
#include "h2_ptx.cuh"

namespace h2 {
namespace {

constexpr int kTcN = 16;                 // columns of one tensor-core pass (right-hand sides, padded)
constexpr int kTcSlices = 10;            // 5-bit digits of an FP64-accurate value
constexpr int kTcFixBits = 49;           // |X| <= 2^49
constexpr int kTileDigits = 11;          // digits of the input values of the small tiles (h2_tile.cu)
constexpr int kTileFixBits = 54;         // |X| <= 2^54: the first ten digits are those of the rounding to 49 bits
constexpr uint32_t kTmemCols = 512;      // tensor memory of one SM
constexpr int kXmaxCols = kLevelCols;

// instruction descriptor of tcgen05.mma kind::f8f6f4: D FP32 (bits 4-5 =
// 1), A and B E4M3 (bits 7-9 = 0, bits 10-12 = 0), both K-major (bits 15, 16
// = 0), N / 8 at bits 17-22, M / 16 at bits 24-28
__host__ __device__ constexpr uint32_t tc_idesc(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}


// Issue by one elected lane of a converged warp (every lane calls it): the
// operands stay warp-uniform, which a branch on the lane number hides from the
// compiler (FP32 coupling at 327,680 triangles, 16 right-hand sides: 1,515 ->
// 1,460 us).
__device__ __forceinline__ void tc_mma(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

// arrive on bar once every MMA issued so far by this warp's elected lane has completed
__device__ __forceinline__ void tc_commit(uint64_t *bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 consecutive 32-bit columns of this warp's 32 tensor-memory lanes; the
// registers are valid after tmem_wait()
__device__ __forceinline__ void tmem_ld16_nw(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Column indices of the blocks a producer thread streams, eight at a time and
// eight ahead, so that no bulk copy waits on a global load.  Without a column
// array (col = NULL) block e lies in column e.
struct ColAhead {
  const int32_t *col;
  int64_t end;
  int32_t nxt[8];
  __device__ __forceinline__ void load(int64_t e) {
#pragma unroll
    for (int u = 0; u < 8; ++u) nxt[u] = col && e + u < end ? col[e + u] : (int32_t)(e + u);
  }
  __device__ __forceinline__ ColAhead(const int32_t *cl, int64_t e0, int64_t e1) : col(cl), end(e1) { load(e0); }
  // the columns of blocks e .. e + 7; afterwards those of e + 8 .. are in flight
  __device__ __forceinline__ void take(int64_t e, int32_t (&c)[8]) {
#pragma unroll
    for (int u = 0; u < 8; ++u) c[u] = nxt[u];
    load(e + 8);
  }
};

__device__ __forceinline__ void named_sync_id(uint32_t id, uint32_t nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// 2^e as a float for -126 <= e <= 127 (exact; used for power-of-two scaling)
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }


// a digit (|s| <= 16, an integer) as its exact FP8 E4M3 byte
__device__ __forceinline__ unsigned char e4m3(int s) {
  return (unsigned char)__nv_cvt_float_to_fp8((float)s, __NV_SATFINITE, __NV_E4M3);
}

__device__ __forceinline__ int tc_level(int64_t c) { return 63 - __clzll(c + 1); }

// F = 2 + floor(log2 max): |hi + lo| < 2^(F-1)
__device__ __forceinline__ int tc_colexp(unsigned bits) {
  return bits ? (int)((bits >> 23) & 0xFF) - 127 + 2 : 0;
}

// v 2^sc for the coefficient scalings (|v 2^sc| <= 2^49, |sc| < 252): two
// power-of-two factors that are normal floats, so the product is exact
// unless it is far below 1/2, where it rounds to the integer 0 anyway
__device__ __forceinline__ float scale2(float v, int sc) {
  const int h = sc >> 1;
  return v * pow2f(h) * pow2f(sc - h);
}

// the ND digits (exact floats) of round(v 2^sc) for a double-float or FP32 value
template <int ND>
__device__ __forceinline__ void digits_of(dd v, int sc, float (&f)[ND]) {
  split_digits_f<ND>(scale2(v.hi, sc), scale2(v.lo, sc), f);
}
template <int ND>
__device__ __forceinline__ void digits_of(float v, int sc, float (&f)[ND]) {
  split_digits_f<ND>(scale2(v, sc), 0.0f, f);
}

// two digits as their E4M3 bytes, the first in the low byte
__device__ __forceinline__ uint32_t e4m3x2(float a, float b) {
  return (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(a, b), __NV_SATFINITE, __NV_E4M3);
}

// The digit planes of NV (8 or 16) consecutive values of one column, each scaled by
// 2^sc: plane i as NV / 4 words (the bytes in value order), a row, or half a row, of
// one core matrix of the MMA layout.
template <int ND, int NV, class T>
__device__ __forceinline__ void cut_row(const T (&v)[NV], int sc, uint32_t (&u)[ND][NV / 4]) {
#pragma unroll
  for (int q = 0; q < NV / 2; ++q) {
    float f0[ND], f1[ND];
    digits_of<ND>(v[2 * q], sc, f0);
    digits_of<ND>(v[2 * q + 1], sc, f1);
#pragma unroll
    for (int i = 0; i < ND; ++i) {
      const uint32_t h = e4m3x2(f0[i], f1[i]);
      u[i][q >> 1] = (q & 1) ? (u[i][q >> 1] | (h << 16)) : h;
    }
  }
}

__device__ __forceinline__ dd dd_scale(dd v, int e) {
  if (e >= -126 && e <= 127) {
    const float w = pow2f(e);
    return dd{v.hi * w, v.lo * w};
  }
  return dd{ldexpf(v.hi, e), ldexpf(v.lo, e)};
}

// byte offset of (row r, contraction index c) in a K-major one-byte operand
// of 32 contraction values per row: two core matrices along K (128 bytes
// apart), then the next 8 rows (256 bytes on)
__host__ __device__ __forceinline__ int core_off32(int r, int c) {
  return ((r >> 3) * 2 + (c >> 4)) * 128 + (r & 7) * 16 + (c & 15);
}
__device__ __forceinline__ uint64_t sdesc32(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(256u >> 4) << 32) |
         (1ull << 46);
}

}  // namespace
}  // namespace h2
