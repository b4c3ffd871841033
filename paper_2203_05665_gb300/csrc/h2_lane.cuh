// One output row of the FP32 block rows (h2_lane.cu, h2_batch.cu); the design is
// described in h2_lane.cu.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstdint>
#include <type_traits>

#include "h2_internal.hpp"
#include "h2_ptx.cuh"

namespace h2 {
namespace {

constexpr int kLaneWarps = 4;
constexpr int kPiece = 32;            // contraction values of a piece

__device__ __forceinline__ uint64_t dup2(float a) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ void fma2(uint64_t &d, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

__device__ __forceinline__ void add2(uint64_t &d, uint64_t a) {
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(d) : "l"(a));
}

// four neighbouring stored values (aligned to the four)
__device__ __forceinline__ float4 val4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 val4(const __nv_bfloat16 *p) {
  const uint2 v = *reinterpret_cast<const uint2 *>(p);
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xffff0000u));
}
__device__ __forceinline__ float4 val4(const __half *p) {
  const uint2 v = *reinterpret_cast<const uint2 *>(p);
  const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&v.x));
  const float2 b = __half22float2(*reinterpret_cast<const __half2 *>(&v.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
// only half storage is scaled (powers of two)
__device__ __forceinline__ float4 scaled(const __half *, float4 v, float s) {
  return make_float4(v.x * s, v.y * s, v.z * s, v.w * s);
}
__device__ __forceinline__ float4 scaled(const float *, float4 v, float) { return v; }
__device__ __forceinline__ float4 scaled(const __nv_bfloat16 *, float4 v, float) { return v; }

// how the rows of one launch (or of one part of a batched launch) are worked on
struct LaneShape {
  int vpieces, gpieces, ppb; // pieces of the V tile, of the self tile, of a block
  uint32_t xoff, stage;      // X region of a stage, stage bytes
  int c0, ncol, xp;          // columns of the pass, their pitch in shared memory
};

// Output row `row` of g by one warp (wpr = 1) or, as warp w, by four (wpr = 4,
// all warps of the CTA; red: shared memory for their sums).  ring: the warp's NST
// stages.  BPP: whole blocks of a piece (more than one only for K <= kPiece, ppb = 1).
template <class TS, class TV, int TC, int TPL, int NST, int BPP = 1>
__device__ __forceinline__ void lane_row(const LaneRows &g, const LaneShape &a, int wpr, int64_t row, int w,
                                         unsigned char *ring, unsigned char *red_smem) {
  const int lane = threadIdx.x & 31;
  const int64_t e0 = g.ptr ? g.ptr[row] : row;
  const int64_t e1 = min(g.ptr ? (g.pend ? g.pend[row] : g.ptr[row + 1]) : row + 1, e0 + g.cap);
  const int nb = (int)(e1 - e0), lead = a.vpieces + a.gpieces;
  const int np = lead + (BPP == 1 ? nb * a.ppb : (nb + BPP - 1) / BPP);
  const int first = wpr == 1 ? 0 : w, n = (np - first + wpr - 1) / wpr;
  const int M = g.M, Mp = g.Mp, K = g.K, rp = g.rp, xp = a.xp;

  // column, stored block and scale of blocks e0 + base + lane
  int base = 0;
  int32_t bc = 0, bb = 0;
  float bs = 1.0f;
  auto batch = [&](int b) {
    base = b;
    const int64_t e = e0 + b + lane;
    if (e < e1) {
      bc = g.col ? g.col[e] : (int32_t)e;
      bb = g.blk ? g.blk[e] : (int32_t)e;
      bs = g.scale ? g.scale[bb] : 1.0f;
    }
  };
  batch(0);

  // copies of kc rows of A (ab bytes) and of X as block u of stage st
  auto copy = [&](unsigned char *st, int u, const unsigned char *src, uint32_t ab, const float *x, int kc) {
    unsigned char *sa = st + u * ab;
    for (uint32_t o = 16u * lane; o < ab; o += 512u) cp_async16(sa + o, src + o);
    float *sx = reinterpret_cast<float *>(st + a.xoff) + u * kc * xp;
    if (rp == xp) {
      for (int o = 4 * lane; o < kc * xp; o += 128) cp_async16(sx + o, x + o);
    } else {
      const int c4 = a.ncol / 4;
      for (int o = lane; o < kc * c4; o += 32) {
        const int mu = o / c4, q = o - mu * c4;
        cp_async16(sx + mu * xp + 4 * q, x + (int64_t)mu * rp + a.c0 + 4 * q);
      }
    }
  };
  // copies of the warp's i-th piece
  auto issue = [&](int i) {
    if (i < n) {
      const int p = first + i * wpr;
      unsigned char *st = ring + ((uint32_t)i % NST) * (size_t)a.stage;
      const unsigned char *src;
      const float *x;
      int kc, b = nb;   // b: the piece's first block
      uint32_t ab;
      float sc = 1.0f;
      if (p < a.vpieces) {
        kc = min(kPiece, g.kv - kPiece * p);
        src = reinterpret_cast<const unsigned char *>(static_cast<const TV *>(g.V) +
                                                      (row * g.kv + kPiece * p) * (int64_t)Mp);
        ab = (uint32_t)(sizeof(TV) * kc * Mp);
        x = g.Y + (row * g.kv + kPiece * p) * (int64_t)rp;
        if (g.vscale) sc = g.vscale[row];
      } else if (p < lead) {
        const int k0 = kPiece * (p - a.vpieces);
        kc = min(kPiece, K - k0);
        src = reinterpret_cast<const unsigned char *>(g.G + (row * K + k0) * (int64_t)Mp);
        ab = (uint32_t)(sizeof(float) * kc * Mp);
        x = g.X + (row * K + k0) * (int64_t)rp;
      } else {
        const int t = p - lead;
        b = BPP > 1 ? BPP * t : a.ppb == 1 ? t : t / a.ppb;
        const int k0 = BPP > 1 ? 0 : kPiece * (t - b * a.ppb);
        if (b - base >= 32) batch(b & ~31);
        const int32_t c = __shfl_sync(0xffffffffu, bc, b - base), k = __shfl_sync(0xffffffffu, bb, b - base);
        sc = __shfl_sync(0xffffffffu, bs, b - base);
        kc = min(kPiece, K - k0);
        src = reinterpret_cast<const unsigned char *>(static_cast<const TS *>(g.A) + ((int64_t)k * K + k0) * Mp);
        ab = (uint32_t)(sizeof(TS) * kc * Mp);
        x = g.X + ((int64_t)c * K + k0) * rp;
      }
      copy(st, 0, src, ab, x, kc);
      if (lane == 0) *reinterpret_cast<float *>(st + a.stage - 16) = sc;
#pragma unroll
      for (int u = 1; u < BPP; ++u) {   // BPP divides 32: the blocks share a batch of columns
        if (b + u >= nb) break;
        const int32_t c = __shfl_sync(0xffffffffu, bc, b + u - base), k = __shfl_sync(0xffffffffu, bb, b + u - base);
        sc = __shfl_sync(0xffffffffu, bs, b + u - base);
        copy(st, u, reinterpret_cast<const unsigned char *>(static_cast<const TS *>(g.A) + (int64_t)k * K * Mp), ab,
             g.X + (int64_t)c * K * rp, kc);
        if (lane == 0) *reinterpret_cast<float *>(st + a.stage - 16 + 4 * u) = sc;
      }
    }
    cp_async_commit();
  };

  // register tiles: tile q = rows 4 (q mod rg) .., columns TC (q div rg) ..; spare lanes
  // take further slices of the contraction
  const int rg = (M + 3) / 4, tiles = rg * (xp / TC), slices = TPL == 1 ? 32 / tiles : 1;
  const int ks = TPL == 1 ? lane / tiles : 0, q0 = TPL == 1 ? lane - ks * tiles : lane;
  int row4[TPL], colt[TPL];
  uint64_t acc[TPL][4][TC / 2];
#pragma unroll
  for (int t = 0; t < TPL; ++t) {
    const int q = min(q0 + 32 * t, tiles - 1);
    row4[t] = 4 * (q % rg);
    colt[t] = TC * (q / rg);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < TC / 2; ++c) acc[t][r][c] = 0ull;
  }

  auto multiply = [&](const auto *sA, const float *sX, int kc, float sc) {
    if (ks >= slices) return;
    uint64_t part[TPL][4][TC / 2];
#pragma unroll
    for (int t = 0; t < TPL; ++t)
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < TC / 2; ++c) part[t][r][c] = 0ull;
    // longer code misses the instruction cache around the short 4-column steps
#pragma unroll(TC == 8 ? 4 : 1)
    for (int mu = ks; mu < kc; mu += slices)
#pragma unroll
      for (int t = 0; t < TPL; ++t) {
        const float4 v = scaled(sA, val4(sA + mu * Mp + row4[t]), sc);
        const uint64_t av[4] = {dup2(v.x), dup2(v.y), dup2(v.z), dup2(v.w)};
        const ulonglong2 *xr = reinterpret_cast<const ulonglong2 *>(sX + mu * xp + colt[t]);
#pragma unroll
        for (int c = 0; c < TC / 4; ++c) {
          const ulonglong2 xv = xr[c];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            fma2(part[t][r][2 * c], av[r], xv.x);
            fma2(part[t][r][2 * c + 1], av[r], xv.y);
          }
        }
      }
#pragma unroll
    for (int t = 0; t < TPL; ++t)
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < TC / 2; ++c) add2(acc[t][r][c], part[t][r][c]);
  };

#pragma unroll
  for (int i = 0; i < NST - 1; ++i) issue(i);
  for (int i = 0; i < n; ++i) {
    cp_async_wait<NST - 2>();
    __syncwarp();
    issue(i + NST - 1);   // into the stage of piece i - 1
    const unsigned char *st = ring + ((uint32_t)i % NST) * (size_t)a.stage;
    const float *sX = reinterpret_cast<const float *>(st + a.xoff);
    const float sc = *reinterpret_cast<const float *>(st + a.stage - 16);
    const int p = first + i * wpr;
    if (p < a.vpieces) {
      multiply(reinterpret_cast<const TV *>(st), sX, min(kPiece, g.kv - kPiece * p), sc);
    } else if (p < lead) {
      multiply(reinterpret_cast<const float *>(st), sX, min(kPiece, K - kPiece * (p - a.vpieces)), 1.0f);
    } else {
      const int t = p - lead, k0 = a.ppb == 1 ? 0 : kPiece * (t % a.ppb);
      const TS *sA = reinterpret_cast<const TS *>(st);
      if (BPP == 1) {
        multiply(sA, sX, min(kPiece, K - k0), sc);
      } else {
        const int m = min(BPP, nb - BPP * t);
        if (std::is_same<TS, __half>::value)   // a scale per block
          for (int u = 0; u < m; ++u)
            multiply(sA + u * K * Mp, sX + u * K * xp, K, *reinterpret_cast<const float *>(st + a.stage - 16 + 4 * u));
        else
          multiply(sA, sX, m * K, sc);
      }
    }
  }
  cp_async_wait<0>();

  float out[TPL][4][TC];
#pragma unroll
  for (int t = 0; t < TPL; ++t)
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < TC / 2; ++c) {
        const float2 v = unpack2(acc[t][r][c]);
        out[t][r][2 * c] = v.x;
        out[t][r][2 * c + 1] = v.y;
      }
  if (TPL == 1)
    for (int z = 1; z < slices; ++z) {
      const int from = min(31, q0 + z * tiles);
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < TC; ++c) {
          // the first slice's lanes read the others' sums, which nobody changes
          const float v = __shfl_sync(0xffffffffu, out[0][r][c], from);
          if (ks == 0) out[0][r][c] += v;
        }
    }
  if (wpr > 1) {
    // the warps' sums, added in order
    __syncthreads();
    float *red = reinterpret_cast<float *>(red_smem);   // [warp][value][lane]
#pragma unroll
    for (int t = 0; t < TPL; ++t)
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < TC; ++c) red[(((w * TPL + t) * 4 + r) * TC + c) * 32 + lane] = out[t][r][c];
    __syncthreads();
    if (w > 0) return;
    for (int v = 1; v < kLaneWarps; ++v)
#pragma unroll
      for (int t = 0; t < TPL; ++t)
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < TC; ++c) out[t][r][c] += red[(((v * TPL + t) * 4 + r) * TC + c) * 32 + lane];
  }
  if (ks > 0) return;
#pragma unroll
  for (int t = 0; t < TPL; ++t) {
    if (q0 + 32 * t >= tiles) continue;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (row4[t] + r >= M) continue;
      float *o = g.out + (row * M + row4[t] + r) * (int64_t)rp + a.c0 + colt[t];
#pragma unroll
      for (int c = 0; c < TC; c += 4)
        if (colt[t] + c < a.ncol) {
          float4 v = make_float4(out[t][r][c], out[t][r][c + 1], out[t][r][c + 2], out[t][r][c + 3]);
          if (g.accumulate) {
            const float4 u = *reinterpret_cast<const float4 *>(o + c);
            v = make_float4(u.x + v.x, u.y + v.y, u.z + v.z, u.w + v.w);
          }
          *reinterpret_cast<float4 *>(o + c) = v;
        }
    }
  }
}

// bytes of a stage (and the offset of its X region): the largest piece of A, V or G, the rows of X
// beside it, and the scales
inline uint32_t lane_stage(const LaneRows &g, size_t sa, size_t sv, int xp, int bpp, uint32_t *xoff) {
  const int k1 = g.K < kPiece ? g.K : kPiece, kb = bpp * k1, kvb = g.V ? (g.kv < kPiece ? g.kv : kPiece) : 0;
  size_t ab = sa * kb * g.Mp;
  if (sv * kvb * g.Mp > ab) ab = sv * kvb * g.Mp;
  if (g.G && sizeof(float) * k1 * g.Mp > ab) ab = sizeof(float) * k1 * g.Mp;
  *xoff = (uint32_t)((ab + 15) / 16 * 16);
  return *xoff + (uint32_t)((kb > kvb ? kb : kvb) * xp * sizeof(float)) + 16;
}

inline void lane_pieces(const LaneRows &g, LaneShape &t) {
  t.vpieces = g.V ? (g.kv + kPiece - 1) / kPiece : 0;
  t.gpieces = g.G ? (g.K + kPiece - 1) / kPiece : 0;
  t.ppb = (g.K + kPiece - 1) / kPiece;
}

// columns of a pass; returns the columns of a register tile
inline int lane_columns(int ncol, LaneShape &t) {
  const int tc = ncol <= 4 ? 4 : 8;
  t.ncol = ncol;
  t.xp = (ncol + tc - 1) / tc * tc;
  return tc;
}

}  // namespace
}  // namespace h2
