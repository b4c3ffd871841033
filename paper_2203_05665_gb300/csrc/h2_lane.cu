// Block rows in FP32 arithmetic, one warp (or four) per output row: the leaf
// forward step, the stored FP32 coupling of orders up to 3 (and of order 4
// beyond 16 right-hand sides), and the nearfield together with the leaf
// backward step, of FP32, bfloat16 and half handles with tiles of at most 64
// rows.
//
// A row is a sequence of pieces of at most 32 contraction values.  The warp
// copies the next piece (a tile A, stored [contraction][row], and the rows of X
// it meets) into the other of its two shared-memory stages (cp.async) while it
// multiplies the current one (deeper rings cost more in resident warps than
// they hide: four stages 217 us, three 164, two 162 for the coupling below).  A lane owns a register tile of 4 output rows by
// TC = 8 (4 for up to 4 columns) columns, two of them for large tiles; lanes
// that are left take further slices of the contraction.  The tile shape is set
// by the shared-memory return bandwidth (128 bytes per cycle and SM, also for
// broadcasts): 12 words feed 32 multiply-adds (packed pairs, fma.rn.f32x2, each
// half rounded like fmaf); a lane per output row with 32 columns would read 33
// words for them and measured 2.5 times slower.  A piece is summed from zero and
// then added to the row, so that a row of hundreds of terms keeps the rounding
// error of short sums.  Column indices (and the scales and stored blocks that go
// with them) are loaded 32 at a time and handed out by shuffles.  Contraction
// slices, and with four warps per row (matrices that hold rows far longer than
// the average, where one warp would finish last alone; warp w takes every fourth
// piece) the warps' sums, are added in a fixed order.
//
// The pipelined block-row kernel of h2_matvec.cu, which ran these steps before,
// synchronises a whole CTA per row and holds a barrier pair per block; blocks of
// 20 to 32 rows leave it bound by latency (16 to 25 % of the issue slots).
// Before -> now: FP32, 81,920 triangles, order 3, 32 columns: coupling 308 ->
// 149 us, leaf backward + nearfield 124 -> 85 us; FP32, 327,680, order 4, 16
// columns: leaf forward 88 -> 44 us, leaf backward + nearfield 356 -> 174 us;
// bfloat16, 1.3 M, order 3, 4 columns: leaf forward 158 -> 66 us, leaf backward +
// nearfield 896 -> 371 us (bound by the instructions around the 20 x 20 pieces:
// half of the issue slots at 24 warps per SM).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstdint>

#include "h2_internal.hpp"
#include "h2_ptx.cuh"

namespace h2 {
namespace {

constexpr int kLaneWarps = 4;
constexpr int kPiece = 32;            // contraction values of a piece
constexpr size_t kLaneSmemMax = 227 * 1024;

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

struct LaneArgs {
  LaneRows r;
  int wpr;                   // warps per row
  int vpieces, gpieces, ppb; // pieces of the V tile, of the self tile, of a block
  uint32_t xoff, stage;      // X region of a stage, stage bytes
  int c0, ncol, xp;          // columns of the pass, their pitch in shared memory
};

template <class TS, class TV, int TC, int TPL>
__global__ void __launch_bounds__(32 * kLaneWarps) k_lane_rows(const __grid_constant__ LaneArgs a) {
  extern __shared__ __align__(16) unsigned char lsm[];
  const LaneRows &g = a.r;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t row = a.wpr == 1 ? (int64_t)blockIdx.x * kLaneWarps + w : (int64_t)blockIdx.x;
  if (row >= g.nrows) return;   // whole warps; with four warps per row every row exists
  unsigned char *ring = lsm + (size_t)w * 2 * a.stage;
  const int64_t e0 = g.ptr ? g.ptr[row] : row, e1 = g.ptr ? g.ptr[row + 1] : row + 1;
  const int lead = a.vpieces + a.gpieces, np = lead + (int)(e1 - e0) * a.ppb;
  const int first = a.wpr == 1 ? 0 : w, n = (np - first + a.wpr - 1) / a.wpr;
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

  // copies of the warp's i-th piece
  auto issue = [&](int i) {
    if (i < n) {
      const int p = first + i * a.wpr;
      unsigned char *st = ring + (size_t)(i & 1) * a.stage;
      const unsigned char *src;
      const float *x;
      int kc;
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
        const int t = p - lead, b = a.ppb == 1 ? t : t / a.ppb, k0 = kPiece * (t - b * a.ppb);
        if (b - base >= 32) batch(b & ~31);
        const int32_t c = __shfl_sync(0xffffffffu, bc, b - base), k = __shfl_sync(0xffffffffu, bb, b - base);
        sc = __shfl_sync(0xffffffffu, bs, b - base);
        kc = min(kPiece, K - k0);
        src = reinterpret_cast<const unsigned char *>(static_cast<const TS *>(g.A) + ((int64_t)k * K + k0) * Mp);
        ab = (uint32_t)(sizeof(TS) * kc * Mp);
        x = g.X + ((int64_t)c * K + k0) * rp;
      }
      for (uint32_t o = 16u * lane; o < ab; o += 512u) cp_async16(st + o, src + o);
      float *sx = reinterpret_cast<float *>(st + a.xoff);
      if (rp == xp) {
        for (int o = 4 * lane; o < kc * xp; o += 128) cp_async16(sx + o, x + o);
      } else {
        const int c4 = a.ncol / 4;
        for (int o = lane; o < kc * c4; o += 32) {
          const int mu = o / c4, q = o - mu * c4;
          cp_async16(sx + mu * xp + 4 * q, x + (int64_t)mu * rp + a.c0 + 4 * q);
        }
      }
      if (lane == 0) *reinterpret_cast<float *>(st + a.stage - 16) = sc;
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
#pragma unroll(TC == 8 ? 4 : 2)
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

  issue(0);
  for (int i = 0; i < n; ++i) {
    cp_async_wait<0>();
    __syncwarp();
    issue(i + 1);   // into the stage of piece i - 1
    const unsigned char *st = ring + (size_t)(i & 1) * a.stage;
    const float *sX = reinterpret_cast<const float *>(st + a.xoff);
    const float sc = *reinterpret_cast<const float *>(st + a.stage - 16);
    const int p = first + i * a.wpr;
    if (p < a.vpieces) {
      multiply(reinterpret_cast<const TV *>(st), sX, min(kPiece, g.kv - kPiece * p), sc);
    } else if (p < lead) {
      multiply(reinterpret_cast<const float *>(st), sX, min(kPiece, K - kPiece * (p - a.vpieces)), 1.0f);
    } else {
      const int t = p - lead, k0 = a.ppb == 1 ? 0 : kPiece * (t % a.ppb);
      multiply(reinterpret_cast<const TS *>(st), sX, min(kPiece, K - k0), sc);
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
  if (a.wpr > 1) {
    // the warps' sums, added in order
    __syncthreads();
    float *red = reinterpret_cast<float *>(lsm);   // [warp][value][lane]
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
        if (colt[t] + c < a.ncol)
          *reinterpret_cast<float4 *>(o + c) =
              make_float4(out[t][r][c], out[t][r][c + 1], out[t][r][c + 2], out[t][r][c + 3]);
    }
  }
}

template <class TS, class TV, int TC, int TPL>
int lane_launch(LaneArgs a, cudaStream_t st) {
  const LaneRows &g = a.r;
  const int kb = std::min(g.K, kPiece), kvb = std::min(g.kv, kPiece);
  size_t ab = sizeof(TS) * kb * g.Mp;
  if (g.V) ab = std::max(ab, sizeof(TV) * kvb * g.Mp);
  if (g.G) ab = std::max(ab, sizeof(float) * kb * g.Mp);
  a.xoff = (uint32_t)((ab + 15) / 16 * 16);
  a.stage = a.xoff + (uint32_t)(std::max(kb, kvb) * a.xp * sizeof(float)) + 16;
  const size_t sm = std::max<size_t>((size_t)kLaneWarps * 2 * a.stage,
                                     a.wpr > 1 ? (size_t)kLaneWarps * TPL * 4 * TC * 32 * sizeof(float) : 0);
  if (sm > kLaneSmemMax) return fail(H2_EINVAL, "block-row tile does not fit in shared memory");
  if (sm > 48 * 1024)
    H2_CUDA_TRY(cudaFuncSetAttribute((const void *)k_lane_rows<TS, TV, TC, TPL>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLaneSmemMax));
  const int64_t grid = a.wpr == 1 ? (g.nrows + kLaneWarps - 1) / kLaneWarps : g.nrows;
  k_lane_rows<TS, TV, TC, TPL><<<(unsigned)grid, 32 * kLaneWarps, sm, st>>>(a);
  H2_CUDA_TRY(cudaGetLastError());
  return H2_OK;
}

template <class TS, class TV>
int lane_run(const LaneRows &g, int64_t *launches, cudaStream_t st) {
  LaneArgs a{};
  a.r = g;
  a.vpieces = g.V ? (g.kv + kPiece - 1) / kPiece : 0;
  a.gpieces = g.G ? (g.K + kPiece - 1) / kPiece : 0;
  a.ppb = (g.K + kPiece - 1) / kPiece;
  // four warps per row where one row is far longer than the rows a warp gets through meanwhile
  a.wpr = g.longest > 64 ? kLaneWarps : 1;
  for (a.c0 = 0; a.c0 < g.rp; a.c0 += 32) {
    a.ncol = std::min(32, g.rp - a.c0);
    const int tc = a.ncol <= 4 ? 4 : 8;
    a.xp = (a.ncol + tc - 1) / tc * tc;
    const int tiles = (g.M + 3) / 4 * (a.xp / tc);
    const int rc = tc == 4 ? lane_launch<TS, TV, 4, 1>(a, st)
                   : tiles <= 32 ? lane_launch<TS, TV, 8, 1>(a, st) : lane_launch<TS, TV, 8, 2>(a, st);
    if (rc) return rc;
    if (launches) ++*launches;
  }
  return H2_OK;
}

}  // namespace

int lane_rows(const LaneRows &g, int prec, bool v32, int64_t *launches, cudaStream_t st) {
  if (g.nrows <= 0) return H2_OK;
  using bf = __nv_bfloat16;
  switch (prec) {
    case H2_F32: return lane_run<float, float>(g, launches, st);
    case H2_BF16: return v32 ? lane_run<bf, float>(g, launches, st) : lane_run<bf, bf>(g, launches, st);
    case H2_F16: return v32 ? lane_run<__half, float>(g, launches, st) : lane_run<__half, __half>(g, launches, st);
    default: return fail(H2_EINVAL, "the FP32 block rows run in FP32 arithmetic only");
  }
}

}  // namespace h2
