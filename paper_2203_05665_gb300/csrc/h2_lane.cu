// Block rows in FP32 arithmetic, one warp (or four) per output row: the leaf
// forward step, the stored FP32 coupling of orders up to 3 (and of order 4
// beyond 16 right-hand sides), and the nearfield together with the leaf
// backward step, of FP32, bfloat16 and half handles with tiles of at most 64
// rows.
//
// A row is a sequence of pieces of at most 32 contraction values (or of two
// whole blocks).  The warp copies the next piece (a tile A, stored
// [contraction][row], and the rows of X it meets) into the other of its two
// shared-memory stages (cp.async) while it multiplies the current one (deeper
// rings cost more in resident warps than they hide: four stages 217 us, three
// 164, two 162 for the coupling below).  A lane owns a register tile of 4 output
// rows by TC = 8 (4 for up to 4 columns) columns, two of them for large tiles; lanes
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
// columns: leaf forward 88 -> 43 us, leaf backward + nearfield 356 -> 156 us;
// bfloat16, 1.3 M, order 3, 4 columns: leaf forward 158 -> 62 us, leaf backward +
// nearfield 896 -> 305 us (bound by the instructions around the 20 x 20 pieces:
// half of the issue slots at 24 warps per SM).  The last two take two blocks per
// piece, which spares half of the waits, copies' set-up and additions of pieces
// (one block per piece: 178 and 347 us).
#include <algorithm>

#include "h2_internal.hpp"
#include "h2_lane.cuh"
#include "h2_launch.cuh"

namespace h2 {
namespace {

constexpr size_t kLaneSmemMax = 227 * 1024;
constexpr size_t kLaneSmemAll = 220 * 1024;   // shared memory of an SM's CTAs (each takes 1 KB more)

struct LaneArgs {
  LaneRows r;
  LaneShape t;
  int wpr;                   // warps per row
};

// CTAs an SM holds
constexpr int lane_ctas(int tc, int tpl) { return tc == 4 ? 6 : tpl == 1 ? 4 : 2; }

template <class TS, class TV, int TC, int TPL, int BPP>
__global__ void __launch_bounds__(32 * kLaneWarps, lane_ctas(TC, TPL)) k_lane_rows(const __grid_constant__ LaneArgs a) {
  pdl_wait();
  pdl_go();
  extern __shared__ __align__(16) unsigned char lsm[];
  const int w = threadIdx.x >> 5;
  const int64_t row = a.wpr == 1 ? (int64_t)blockIdx.x * kLaneWarps + w : (int64_t)blockIdx.x;
  if (row >= a.r.nrows) return;   // whole warps; with four warps per row every row exists
  lane_row<TS, TV, TC, TPL, 2, BPP>(a.r, a.t, a.wpr, row, w, lsm + (size_t)w * 2 * a.t.stage, lsm);
}

template <class TS, class TV, int TC, int TPL, int BPP>
int lane_start(LaneArgs a, cudaStream_t st) {
  const LaneRows &g = a.r;
  a.t.stage = lane_stage(g, sizeof(TS), sizeof(TV), a.t.xp, BPP, &a.t.xoff);
  const size_t sm = std::max<size_t>((size_t)kLaneWarps * 2 * a.t.stage,
                                     a.wpr > 1 ? (size_t)kLaneWarps * TPL * 4 * TC * 32 * sizeof(float) : 0);
  if (sm > kLaneSmemMax) return fail(H2_EINVAL, "block-row tile does not fit in shared memory");
  if (sm > 48 * 1024)
    H2_CUDA_TRY(cudaFuncSetAttribute((const void *)k_lane_rows<TS, TV, TC, TPL, BPP>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLaneSmemMax));
  const int64_t grid = a.wpr == 1 ? (g.nrows + kLaneWarps - 1) / kLaneWarps : g.nrows;
  pdl(k_lane_rows<TS, TV, TC, TPL, BPP>, (unsigned)grid, 32 * kLaneWarps, sm, st, a);
  H2_CUDA_TRY(cudaGetLastError());
  return H2_OK;
}

template <class TS, class TV, int TC, int TPL>
int lane_launch(const LaneArgs &a, cudaStream_t st) {
  // two blocks per piece where the rows have blocks (ptr) of at most kPiece contraction
  // values and the larger stages leave the SM its CTAs (measured above; with 32 columns
  // they would not, and one block per piece measured the same, 87 us)
  uint32_t xoff;
  const LaneRows &g = a.r;
  const size_t stage2 = lane_stage(g, sizeof(TS), sizeof(TV), a.t.xp, 2, &xoff);
  const bool two = g.ptr && a.t.ppb == 1 && lane_ctas(TC, TPL) * kLaneWarps * 2 * stage2 <= kLaneSmemAll;
  return two ? lane_start<TS, TV, TC, TPL, 2>(a, st) : lane_start<TS, TV, TC, TPL, 1>(a, st);
}

template <class TS, class TV>
int lane_run(const LaneRows &g, int64_t *launches, cudaStream_t st) {
  LaneArgs a{};
  a.r = g;
  lane_pieces(g, a.t);
  // Four warps per row where one row is far longer than the rows a warp gets through
  // meanwhile.  FP32 coupling, order 3, 8 columns, one and four warps: longest row of 120
  // blocks (cube, 30,000 triangles) 138 and 56 us, 115 (ellipsoid, 81,920) 182 and 125 us;
  // of 16 (cube, 120,000) 75 and 97 us, 20 (sphere, 81,920) 82 and 100 us.  The line lies
  // between; meshes that do not fill the GPU with one warp per row (4,800 triangles: 24
  // and 14 us) are not told apart.
  a.wpr = g.longest > 64 ? kLaneWarps : 1;
  for (a.t.c0 = 0; a.t.c0 < g.rp; a.t.c0 += 32) {
    const int tc = lane_columns(std::min(32, g.rp - a.t.c0), a.t);
    const int tiles = (g.M + 3) / 4 * (a.t.xp / tc);
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
