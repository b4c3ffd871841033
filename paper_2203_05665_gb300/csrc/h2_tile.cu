// Block rows with small tiles on the tensor cores (tcgen05, FP8 E4M3
// operands, FP32 accumulation in tensor memory), FP64 accuracy: output rows
// of R <= 32 values whose blocks contract over at most 32 values.  The
// nearfield of H2_F64 handles (R = L triangles per leaf, y|t += sum G_ts x|s,
// Algorithm 3 over the inadmissible leaf pairs) and the coupling of order-3
// handles (R = 27, y^_t += sum S_ts x^_s) run on it for any number of
// right-hand sides, 16 columns per launch.
//
// The arithmetic is the exact digit splitting of h2_tc.cu: every row nu of
// the blocks of one block row gets a power of two 2^E, every column j of the
// input (of each tree level, for the coupling) a power of two 2^F.  A block's value
// becomes X = round(v 2^(49-E)), |X| <= 2^49, cut into ten signed 5-bit digits i =
// 0 .. 9 of weight 2^(-4 - 5 i), an input value X = round(v 2^(54-F)) and eleven
// digits.  All digit pairs of levels i + k <= 10 are summed (and some above): the
// pairs left out stay below 2^-53 of the scales' product, the rounding of a block's
// value below 2^-50 of its row's scale, that of an input value below 2^-55 of its
// column's scale (at most four times the largest value).
//
// Range.  Double-float arithmetic, which this replaces, rounds every input value to
// 2^-48 of itself, the digits to 2^-53 of the column's largest.  A column takes the
// digits if at least half of its non-zero entries reach 2^-5 of the largest
// (k_permute_in counts): those keep their 48 bits, and in the 2-norm the rounding
// is at most 2^-53 2^5 sqrt(2) = 2^-47.5 of the column.  Evenly distributed columns do by a wide margin (uniform 97 %, normal
// 87 % at 10^6 entries), and so do unit vectors; a column that does not (a few
// entries far above the rest, values over many orders of magnitude) is summed in
// double-float by the same CTAs over the same rows (rows_dd), after the digits of
// the pass's other columns (its own are cut as zeros), so that no column's result
// depends on another's values.
// Errors in the 2-norm, 5,120 triangles graded 55 : 1 in size, order 3, 20
// columns of entries in [-1, 1] and one of 1e8: 1.0e-10 without that rule, 1.3e-14
// now, 1.7e-14 in double-float block rows.  The rule and the eleventh digit cost even
// columns about 1 % (81,920 triangles, 32 columns).
//
// Layout.  The digit planes of a block are stacked four to a 128-row MMA
// operand: digit i (from 0) of row nu lies in group i / 4, row (i mod 4) R +
// nu (three groups; K = 32 bytes, zero padded, K-major core matrices).  The
// input digits of a column tile are the N side: digit k (from 0), column j in
// row W k + j, W = 4, 8 or 16 columns per digit as the right-hand sides ask,
// (the rows up to a multiple of 16 are zero).  Group g multiplies the planes k =
// 0 .. 10 - 4 g into accumulator columns W (4 g + k) + j: the planes of a
// group differ in i by their lane quarter only, so column block c = 4 g + k
// holds, in lanes R q + nu, the sum of every pair of level i + k = c + q
// (from 0), and the tensor cores add the pairs of a level themselves.  One
// accumulator set is 11 W columns (176, 88 or 44) instead of one per group,
// and the epilogue reads 11 column blocks instead of 14.  The last group holds
// two digits; its other two plane rows are zeros that stay in shared memory.
//
// Exactness: a set sums at most three groups of nb blocks of products of
// magnitude <= 2^8 over R values: 3 x 2^8 x nb R <= 2^18.9 for nb R <= 661, so
// that two neighbouring column blocks combine exactly in FP32 (32 D_c +
// D_(c+1) < 2^24) before they enter the double-float sum.  Longer rows are cut
// into segments of that length.
//
// Roles (one CTA per SM, ten warps): warp 0 streams the blocks through a
// shared-memory ring (bulk copies completing on mbarriers), warp 1 issues the
// MMAs, warps 2-5 and 6-9 are two epilogue groups that take the rows in turn,
// each with its own accumulator set and exchange area.
//
// What bounds it: the copy stream and the MMA warp's issue.  Nearfield of
// 327,680 triangles (leaves of 20, 179,008 blocks of 6.4 KB and as many input
// tiles of 5.6 KB), 16 columns: 480 us before (one epilogue group, separate
// accumulator columns per plane group, single-stage commits), 298 us now, 7.2
// TB/s into shared memory.  Leaves of 30 (cube, 30,000 triangles, 5 columns):
// 161 us in double-float block rows, 44 us now; 32 right-hand sides, 81,920
// triangles: 414 us in double-float, 184 us now (two passes, with the digit cuts).  Order-3
// coupling, double-float block rows before: 81,920 triangles, 32 right-hand
// sides (75,224 blocks of 9.0 KB, two passes) 1,070 us, now 339 us with the
// digit cuts; cube of 30,000 triangles, 5 columns 195 us, now 54 us; 5,120
// triangles, one column 35 us, now 17 us.
#include <algorithm>
#include <functional>
#include <queue>
#include <utility>
#include <vector>

#include "h2_internal.hpp"
#include "h2_kernel.cuh"
#include "h2_launch.cuh"
#include "h2_tc.cuh"

namespace h2 {
namespace {

constexpr int kTileMax = 32;              // rows of a tile, contraction length
constexpr int kTileThreads = 64 + 256;    // producer, MMA, two epilogue groups
constexpr uint32_t kTilePad = 4096;       // an MMA reads 128 rows from a group's start: past the last stage at most this far
constexpr int kTileMaxStages = 24;
// stages released by one commit: a tcgen05.commit costs its thread about as
// much as the three MMAs of a block (327,680 triangles, leaves of 20, 16
// columns: 424 us with one per block, 342 us with one per four)
constexpr int kTileGroup = 4;
constexpr int64_t kSchedChunk = 12;       // blocks and rows of a scheduling chunk (see row_schedule)
constexpr uint32_t kTileSmemMax = 227 * 1024;

// N rows (bytes / 32) of an input digit tile, columns of an accumulator set
template <int W>
__host__ __device__ constexpr int tile_n() { return (kTileDigits * W + 15) / 16 * 16; }

// bytes of a four-plane group, of the stored last (two-plane) group and of a stored block
__host__ __device__ inline uint32_t tile_group(int R) { return (uint32_t)((4 * R + 7) / 8 * 8) * 32u; }
__host__ __device__ inline uint32_t tile_last(int R) { return (uint32_t)((2 * R + 7) / 8 * 8) * 32u; }
__host__ __device__ inline uint32_t tile_bytes(int R) { return 2 * tile_group(R) + tile_last(R); }
// blocks per exact segment
__host__ __device__ inline int tile_seg(int R) { return 661 / R; }

// byte offset of digit i (from 0), row nu, contraction index c of a block
__device__ __forceinline__ uint32_t tile_off(int R, int i, int nu, int c) {
  return (uint32_t)(i >> 2) * tile_group(R) + (uint32_t)core_off32((i & 3) * R + nu, c);
}

struct TileArgs {
  const unsigned char *A;     // stored blocks, abytes each
  const unsigned char *X;     // input digit tiles, 32 tile_n<W>() bytes each
  const int64_t *ptr;         // CSR over the scheduled rows (row_schedule)
  const int32_t *col;
  const int32_t *row;         // output row of every scheduled row
  const int32_t *E;           // [output row][R] powers of two
  const unsigned *xmax;       // column maxima (bits of a float)
  const int32_t *split;       // [gridDim.x + 1]: rows of every CTA
  dd *out;                    // [row][R][rp], at the first column of the pass
  // the same rows in double-float (rows_dd), for the columns that need it; spread NULL: none
  const int *spread;          // per column: negative where too few entries come near the largest
  const unsigned long long *colmax;   // per column: 0 where the input vanishes
  const dd *B, *Xd;           // blocks [K = R][Bp] (contraction index major), inputs [item][R][rp]
  const int64_t *bptr;        // CSR over the output rows (from row0 on)
  const int32_t *bcol;
  int Bp;
  int R, ncol, rp, nst, accumulate;
  int64_t row0;               // output row of scheduled row value 0 (E, out, xmax are indexed from it)
  int by_level;               // xmax holds kXmaxCols maxima per tree level, output rows are clusters
  uint32_t stage, xch;        // bytes of a stage, of one exchange area
};

// The CTA's rows of the columns in mask in double-float: two blocks and their inputs at a time, staged three
// deep (cp.async); one of 256 threads sums four output rows of two columns, spare ones
// take further slices of the contraction, added in order.  Every four blocks are summed
// from zero and then added to the row, so that long rows keep the rounding error of
// short sums.  Threads and slices are those of all columns of the pass, whichever are
// in mask.  Bound by the FP32 pipe (two warps per scheduler; the other two warps only
// copy).  Whole products of wide columns, 81,920 triangles, order 3, 1 / 5 / 16 / 32
// columns: 573 / 714 / 1,185 / 2,310 us, one among even ones 572 / 882 / 1,359 / 2,677 us; pipelined block rows on the same sums 531 / 637 / 1,053 / 1,871 us
// (every product, before the digits).
constexpr int kDdStages = 3, kDdThreads = 256;
__host__ __device__ inline uint32_t rows_dd_stage(int R, int Bp, int ncol) {
  return (uint32_t)(2 * R * (Bp + ncol) * (int)sizeof(dd));
}
__device__ __noinline__ void rows_dd(const TileArgs &a, int64_t r_begin, int64_t r_end, unsigned char *smem,
                                     uint32_t mask) {
  const int R = a.R, Bp = a.Bp, nc = a.ncol, tid = threadIdx.x;
  const uint32_t stage = rows_dd_stage(R, Bp, nc);
  dd *red = reinterpret_cast<dd *>(smem + kDdStages * stage);   // [slice][tile][8], at most 8 values per thread
  const int rg = (R + 3) / 4, tiles = rg * (nc / 2), slices = max(1, min(kDdThreads / tiles, R));
  const int ks = tid / tiles, q = tid - ks * tiles, nu = 4 * (q % rg), c = 2 * (q / rg);
  const bool on = ks < slices && (mask >> c & 3u);
  const int xo = 2 * tid / nc * a.rp + 2 * tid % nc;   // this thread's two values of an input
  // The copies run ahead of the sums across rows: block pb (of blocks to pe - 1 of scheduled
  // row pr) comes next; the bounds of the row after and the row after that are on their way.
  int64_t pr = r_begin - 1, pb = 0, pe = 0, nb0 = 0, nb1 = 0;
  int32_t t1 = r_begin < r_end ? a.row[r_begin] : 0, t2 = r_begin + 1 < r_end ? a.row[r_begin + 1] : 0, col[2];
  if (r_begin < r_end) {
    nb0 = a.bptr[t1];
    nb1 = a.bptr[t1 + 1];
  }
  auto next_row = [&] {
    pb = nb0;
    pe = nb1;
    if (++pr + 1 < r_end) {
      nb0 = a.bptr[t2];
      nb1 = a.bptr[t2 + 1];
      if (pr + 2 < r_end) t2 = a.row[pr + 2];
    }
  };
  auto seek = [&] {   // the next block's row and the columns of the next copy
    while (pb >= pe && pr < r_end) next_row();
#pragma unroll
    for (int u = 0; u < 2; ++u) col[u] = pb + u < pe ? a.bcol[pb + u] : -1;
  };
  auto copy = [&](uint32_t i) {
    if (pr < r_end) {
      dd *sB = reinterpret_cast<dd *>(smem + (i % kDdStages) * stage), *sX = sB + 2 * R * Bp;
      const dd *B = a.B + pb * R * Bp;
      const int vals = (pb + 1 < pe ? 2 : 1) * R * Bp;
      for (int o = 2 * tid; o < vals; o += 2 * kTileThreads) cp_async16(sB + o, B + o);
      if (2 * tid < R * nc)
#pragma unroll
        for (int u = 0; u < 2; ++u)
          if (col[u] >= 0) cp_async16(sX + u * R * nc + 2 * tid, a.Xd + (int64_t)col[u] * R * a.rp + xo);
      pb = min(pb + 2, pe);
    }
    cp_async_commit();
    seek();
  };
  seek();
  for (int i = 0; i < kDdStages - 1; ++i) copy(i);
  uint32_t step = 0;
  for (int64_t r = r_begin; r < r_end; ++r) {
    const int32_t t = t1;
    const int nb = (int)(a.bptr[t + 1] - a.bptr[t]);
    if (r + 1 < r_end) t1 = a.row[r + 1];
    dd s[4][2] = {}, p[4][2] = {};
    for (int i = 0; i < nb; i += 2, ++step) {
      cp_async_wait<kDdStages - 2>();
      __syncthreads();
      copy(step + kDdStages - 1);   // into the stage before this one
      if (on) {
        const dd *sB = reinterpret_cast<const dd *>(smem + (step % kDdStages) * stage), *sX = sB + 2 * R * Bp;
        const int K = (i + 1 < nb ? 2 : 1) * R;
#pragma unroll 2
        for (int mu = ks; mu < K; mu += slices) {
          const float4 v0 = *reinterpret_cast<const float4 *>(sB + mu * Bp + nu);
          const float4 v1 = *reinterpret_cast<const float4 *>(sB + mu * Bp + nu + 2);
          const float4 x = *reinterpret_cast<const float4 *>(sX + mu * nc + c);
          const dd v[4] = {{v0.x, v0.y}, {v0.z, v0.w}, {v1.x, v1.y}, {v1.z, v1.w}};
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            acc_fma(p[u][0], v[u], dd{x.x, x.y});
            acc_fma(p[u][1], v[u], dd{x.z, x.w});
          }
        }
        if ((i & 2) || i + 2 >= nb)
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int w = 0; w < 2; ++w) {
              acc_norm(p[u][w]);
              s[u][w] = s[u][w] + p[u][w];
              p[u][w] = dd{0.0f, 0.0f};
            }
      }
    }
    // the slices' sums, added in order by a thread per output
    if (on)
#pragma unroll
      for (int u = 0; u < 8; ++u) red[(ks * tiles + q) * 8 + u] = s[u >> 1][u & 1];
    __syncthreads();
    for (int o = tid; o < R * nc; o += kTileThreads) {
      const int ro = o / nc, co = o - ro * nc;
      if (!(mask >> co & 1u)) continue;
      const dd *v = red + ((co >> 1) * rg + (ro >> 2)) * 8 + (ro & 3) * 2 + (co & 1);
      dd sum = v[0];
      for (int z = 1; z < slices; ++z) sum = sum + v[z * tiles * 8];
      dd *y = a.out + ((a.row0 + t) * R + ro) * a.rp + co;
      *y = a.accumulate ? *y + sum : sum;
    }
    __syncthreads();   // red is free again
  }
  cp_async_wait<0>();
}

template <int W>
__global__ void __launch_bounds__(kTileThreads, 1) k_tile_tc(const __grid_constant__ TileArgs a) {
  constexpr int N0 = tile_n<W>(), SET = W == 16 ? 256 : 128;
  constexpr uint32_t kX = (uint32_t)N0 * 32u;
  extern __shared__ __align__(1024) unsigned char smem[];
  const int R = a.R, nst = a.nst;
  const uint32_t ga = tile_group(R), ab = tile_bytes(R);
  dd *xch = reinterpret_cast<dd *>(smem + (size_t)nst * a.stage + kTilePad);
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + (size_t)nst * a.stage + kTilePad + 2 * a.xch);
  uint64_t *empty = full + kTileMaxStages;
  uint64_t *accf = empty + kTileMaxStages;   // [2]: the MMAs of a segment have completed
  uint64_t *acce = accf + 2;                 // [2]: the epilogue has read the set
  uint64_t *done = acce + 2;
  uint32_t *tslot = reinterpret_cast<uint32_t *>(done + 1);
  volatile int *abort = reinterpret_cast<volatile int *>(tslot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t r_begin = a.split[blockIdx.x], r_all = a.split[blockIdx.x + 1], e_begin = a.ptr[r_begin];
  int64_t r_end = r_all, e_end = a.ptr[r_all];   // the rows multiplied as digits

  if (tid == 0) {
    for (int s = 0; s < nst; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int u = 0; u < 2; ++u) {
      mbar_init(&accf[u], 1);
      mbar_init(&acce[u], 4);
    }
    mbar_init(done, 1);
    *abort = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(2 * SET)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // the zero plane rows of the last group, in every stage (the copies never touch them)
  {
    const int words = (int)(3 * ga - ab) / 16;
    for (int i = tid; i < words * nst; i += kTileThreads)
      *reinterpret_cast<uint4 *>(smem + (size_t)(i / words) * a.stage + ab + 16 * (i % words)) = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = *tslot;
  const int64_t seg = tile_seg(R);
  pdl_wait();   // everything above is set-up data and this CTA's own
  // narrow tiles: CTAs of the next kernel beside a long tail cost more than their early start
  // gives.  Products of 5 columns with and without: 5,120 triangles 66 and 60 us, 20,480 124
  // and 119, 81,920 337 and 334, cubes of 4,800 64 and 60, 30,000 155 and 150, 129,792 343
  // and 340; one column the same either way
  if (W == 16) pdl_go();
  // columns in double-float (the same in every warp); without any other that does not
  // vanish no row is multiplied as digits
  uint32_t wide = 0u;
  if (a.spread) {
    const bool in = lane < a.ncol, w = in && a.spread[min(lane, a.ncol - 1)] < 0;
    const bool zero = a.colmax[min(lane, a.ncol - 1)] == 0ull;
    wide = __ballot_sync(0xffffffffu, w);
    if (wide && !__any_sync(0xffffffffu, in && !w && !zero)) {
      wide = 0xffffffffu;
      r_end = r_begin;
      e_end = e_begin;
    }
  }

  if (warp == 0) {
    // ---------------- producer: the digits of every block of the range and of its column tile
    if (lane == 0) {
      int64_t e = e_begin;
      ColAhead ca(a.col, e, e_end);
      const uint64_t pol_stream = l2_evict_first(), pol_keep = l2_evict_last();
      int s = 0;
      uint32_t ph = 1;   // parity of the stage's previous release
      bool ok = true;
      while (e < e_end && ok) {
        int32_t cb[8];
        ca.take(e, cb);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (e >= e_end || !ok) break;
          if (s % kTileGroup == 0 && e - e_begin >= nst && !mbar_wait_or_abort(&empty[s / kTileGroup], ph, abort)) {
            ok = false;
            break;
          }
          unsigned char *st = smem + (size_t)s * a.stage;
          mbar_expect_tx(&full[s], ab + kX);
          bulk_g2s_hint(st + 3 * ga, a.X + (int64_t)cb[u] * kX, kX, &full[s], pol_keep);
          bulk_g2s_hint(st, a.A + e * (int64_t)ab, ab, &full[s], pol_stream);
          ++e;
          if (++s == nst) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (*abort) {
        // let the copies in flight land before the CTA leaves (bounded)
        const int64_t j0 = e - nst > e_begin ? e - nst : e_begin;
        for (int64_t j = j0; j < e; ++j) {
          const int64_t ij = j - e_begin;
          mbar_wait_bounded(&full[ij % nst], (uint32_t)((ij / nst) & 1));
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (the whole warp waits, an elected lane issues)
    {
      int s = 0;
      uint32_t ph = 0, use[2] = {0, 0}, set = 1;
      bool ok = true;
      int64_t pnext = a.ptr[r_begin];   // row pointers loaded one row ahead
      for (int64_t r = r_begin; r < r_end && ok; ++r) {
        const int64_t b0 = pnext;
        pnext = a.ptr[r + 1];
        const int64_t nb = pnext - b0;
        if (nb > 0) set ^= 1;   // the rows that have blocks alternate between the two groups
        for (int64_t s0 = 0; s0 < nb && ok; s0 += seg) {
          const uint32_t u = set ? use[1]++ : use[0]++;
          if (u > 0 && !mbar_wait_or_abort(&acce[set], (u - 1) & 1, abort)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d0 = tbase + set * SET;
          const int64_t sn = nb - s0 < seg ? nb - s0 : seg;
          for (int64_t t = 0; t < sn; ++t) {
            if (!mbar_wait_or_abort(&full[s], ph, abort)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t A0 = smem_u32(smem + (size_t)s * a.stage);
            const uint64_t dA = sdesc32(A0), dB = sdesc32(A0 + 3 * ga);
            // group 0 covers every column of the set, so its MMA of the first block overwrites it
#pragma unroll
            for (int g = 0; g < 3; ++g)
              tc_mma(d0 + 4 * g * W, dA + (uint64_t)((g * ga) >> 4), dB, tc_idesc(((11 - 4 * g) * W + 15) / 16 * 16),
                     (t > 0 || g > 0) ? 1u : 0u);
            // the stages of a group are free once these MMAs have read them
            if (s % kTileGroup == kTileGroup - 1) tc_commit(&empty[s / kTileGroup]);
            if (++s == nst) {
              s = 0;
              ph ^= 1;
            }
          }
          if (ok) tc_commit(&accf[set]);
        }
      }
      // every MMA issued has completed before the tensor memory is released
      tc_commit(done);
      mbar_wait_bounded(done, 0);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue group grp: warps read tensor-memory lanes 32 (warp % 4) ..
    const uint32_t grp = (uint32_t)(warp - 2) >> 2;
    const int quad = warp & 3, tl = quad * 32 + lane;
    const int pitch = 4 * R + 1, nout = R * a.ncol;
    dd *xg = xch + (size_t)grp * (a.xch / sizeof(dd));
    const uint32_t bar_or = 1 + 2 * grp, bar_x = 2 + 2 * grp;
    const uint32_t tset = tbase + ((uint32_t)(quad * 32) << 16) + grp * SET;
    const bool plane = tl < 4 * R;
    const float wq = pow2f(-5 * (plane ? tl / R : 0));
    // this thread's outputs o = tl + 128 u: row o / ncol, column o % ncol
    constexpr int UO = W / 4;
    int orow[UO], ocol[UO], fexp[UO];
#pragma unroll
    for (int u = 0; u < UO; ++u) {
      const int o = tl + 128 * u;
      orow[u] = o < nout ? o / a.ncol : 0;
      ocol[u] = o < nout ? o % a.ncol : 0;
      fexp[u] = tc_colexp(a.xmax[ocol[u]]);
    }
    uint32_t use = 0, set = 1;
    int64_t pnext = a.ptr[r_begin];
    int32_t rnext = r_begin < r_end ? a.row[r_begin] : 0;
    for (int64_t r = r_begin; r < r_end; ++r) {
      const int64_t b0 = pnext, orow_id = a.row0 + rnext;
      pnext = a.ptr[r + 1];
      if (r + 1 < r_end) rnext = a.row[r + 1];
      const int64_t nb = pnext - b0;
      dd *yrow = a.out + orow_id * R * a.rp;
      if (nb == 0) {
        if (!a.accumulate && grp == 0)
#pragma unroll
          for (int u = 0; u < UO; ++u)
            if (tl + 128 * u < nout) yrow[orow[u] * a.rp + ocol[u]] = dd{0.0f, 0.0f};
        continue;
      }
      set ^= 1;
      if (set != grp) continue;
      bool stop = false;
      for (int64_t s0 = 0; s0 < nb; s0 += seg, ++use) {
        // row powers and previous values are loaded before the wait
        int eo[UO];
        dd yold[UO];
#pragma unroll
        for (int u = 0; u < UO; ++u) {
          eo[u] = 0;
          yold[u] = dd{0.0f, 0.0f};
          if (tl + 128 * u < nout) {
            if (a.by_level) fexp[u] = tc_colexp(a.xmax[tc_level(orow_id) * kXmaxCols + ocol[u]]);
            eo[u] = a.E[orow_id * R + orow[u]] + fexp[u];
            if (s0 > 0 || a.accumulate) yold[u] = yrow[orow[u] * a.rp + ocol[u]];
          }
        }
        const bool ready = !*abort && mbar_wait_or_abort(&accf[grp], use & 1, abort);
        if (named_sync_or_id(bar_or, 128, ready ? 0 : 1)) {
          stop = true;
          break;
        }
        tc_fence_after();
        // column blocks c, c + 1 combine exactly; weight 2^(-8 - 5 (c + 1)), times 2^(-5 q) at the
        // end.  Rolled for 16 columns: unrolled, the three roles' code missed the instruction
        // cache, the first of the stalls, and the kernel's time moved by 4 % with the code
        // around it (81,920 triangles, order 3, 32 columns: product 873 us unrolled, 795 rolled;
        // 327,680, order 4, 16 columns: nearfield and leaf backward 581 and 514 us; 8 columns
        // or fewer 143 us unrolled, 145 rolled)
        dd acc[W];
#pragma unroll
        for (int j = 0; j < W; ++j) acc[j] = dd{0.0f, 0.0f};
#pragma unroll(W == 16 ? 1 : 4)
        for (int base = 0; base < N0; base += 64) {
          uint32_t raw[4][16];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (base + 16 * u < N0) tmem_ld16_nw(tset + (uint32_t)(base + 16 * u), raw[u]);
          tmem_wait();
#pragma unroll
          for (int cb = 0; cb < 64 / W; cb += 2) {
            const int c = base / W + cb;
            if (c < 11) {
              const float w = pow2f(-8 - 5 * (c + 1));
#pragma unroll
              for (int j = 0; j < W; ++j) {
                const int p = cb * W + j, p1 = p + W;
                float v = 32.0f * __uint_as_float(raw[p >> 4][p & 15]);
                if (c + 1 < 11) v += __uint_as_float(raw[(p1 >> 4) & 3][p1 & 15]);
                float s, e;
                two_sum(acc[j].hi, v * w, s, e);
                acc[j].hi = s;
                acc[j].lo += e;
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce[grp]);
        if (plane)
#pragma unroll
          for (int j = 0; j < W; ++j) {
            acc_norm(acc[j]);
            xg[j * pitch + tl] = dd{acc[j].hi * wq, acc[j].lo * wq};
          }
        named_sync_id(bar_x, 128);
#pragma unroll
        for (int u = 0; u < UO; ++u) {
          if (tl + 128 * u >= nout) continue;
          const dd *xc = xg + ocol[u] * pitch + orow[u];
          dd v = xc[0];
#pragma unroll
          for (int q = 1; q < 4; ++q) v = v + xc[q * R];
          v = dd_scale(v, eo[u]);
          if (s0 > 0 || a.accumulate) v = v + yold[u];
          yrow[orow[u] * a.rp + ocol[u]] = v;
        }
        named_sync_id(bar_x, 128);
      }
      if (stop) break;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(2 * SET) : "memory");
  if (wide) rows_dd(a, r_begin, r_all, smem, wide);   // every copy and MMA of the digits is complete
}

// The input digit tiles of items first .. first + count - 1 (R rows of rp
// values each, columns 0 .. ncol - 1 of x): 4 W threads per item, thread (j, g)
// cuts rows 8 g .. 8 g + 7 of column j in registers (zero beyond R and ncol) and
// writes half a 16-byte row of a core matrix per plane, and of the zero rows behind the
// eleven planes.  Columns of wide range (spread, NULL: none) are cut as zeros.  (Sixteen values per thread took 168 registers.)
template <int W>
__global__ void __launch_bounds__(128) k_tile_cut(const dd *__restrict__ x, int64_t first, int64_t count, int R,
                                                  int rp, int ncol, const unsigned *__restrict__ xmax, int by_level,
                                                  const int *__restrict__ spread, unsigned char *__restrict__ X) {
  pdl_wait();
  pdl_go();
  constexpr int N0 = tile_n<W>();
  const int64_t i = (int64_t)blockIdx.x * (32 / W) + threadIdx.x / (4 * W);
  if (i >= count) return;
  const int64_t t = first + i;
  // the halves of a core-matrix row are neighbouring lanes, then the columns
  const int h = threadIdx.x & 1, j = (threadIdx.x >> 1) % W, c = (threadIdx.x / (2 * W)) & 1, g = 2 * c + h;
  const int sc = kTileFixBits - tc_colexp(j < ncol ? xmax[(by_level ? tc_level(t) * kXmaxCols : 0) + j] : 0u);
  const bool cut = j < ncol && !(spread && spread[j] < 0);
  dd v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int mu = 8 * g + q;
    v[q] = mu < R && cut ? x[(t * R + mu) * rp + j] : dd{0.0f, 0.0f};
  }
  uint32_t w[kTileDigits][2];
  cut_row<kTileDigits, 8>(v, sc, w);
  unsigned char *dst = X + t * (int64_t)(32 * N0) + c * 128 + h * 8;
#pragma unroll
  for (int k = 0; k < kTileDigits; ++k) {
    const int n = W * k + j;
    *reinterpret_cast<uint2 *>(dst + (n >> 3) * 256 + (n & 7) * 16) = make_uint2(w[k][0], w[k][1]);
  }
  for (int n = W * kTileDigits + j; n < N0; n += W)
    *reinterpret_cast<uint2 *>(dst + (n >> 3) * 256 + (n & 7) * 16) = make_uint2(0, 0);
}

// E[t][nu] = 1 + floor(log2 max |G_b[nu][mu]|) over the near blocks b of leaf row t (0 if none)
__global__ void k_near_rowexp(const dd *__restrict__ near, const int64_t *__restrict__ ptr, int64_t nleaf, int L,
                              int Lp, int32_t *__restrict__ E) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= nleaf * L) return;
  const int64_t t = e / L;
  const int nu = (int)(e % L);
  float mx = 0.0f;
  for (int64_t b = ptr[t]; b < ptr[t + 1]; ++b)
    for (int mu = 0; mu < L; ++mu) mx = fmaxf(mx, fabsf(near[(b * L + mu) * Lp + nu].hi));
  E[e] = mx > 0.0f ? ilogbf(mx) + 1 : 0;
}

// the ten digit planes of scheduled block d (near block src[d], row leaf brow[d]), row nu,
// contraction indices 16 cg .. 16 cg + 15
__global__ void k_near_slice(const dd *__restrict__ near, const int32_t *__restrict__ src,
                             const int32_t *__restrict__ brow, const int32_t *__restrict__ E, int64_t nnear, int L,
                             int Lp, unsigned char *__restrict__ A) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= nnear * L * 2) return;
  const int64_t d = e / (2 * L), b = src[d];
  const int nu = (int)((e / 2) % L), cg = (int)(e % 2);
  const int sc = kTcFixBits - E[(int64_t)brow[d] * L + nu];
  __align__(16) unsigned char out[kTcSlices][16];
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int mu = 16 * cg + q;
    long long X = 0;
    if (mu < L) {
      const dd v = near[(b * L + mu) * Lp + nu];
      X = llrint(ldexp((double)v.hi + (double)v.lo, sc));
    }
    int sl[kTcSlices];
    split_digits(X, sl);
#pragma unroll
    for (int i = 0; i < kTcSlices; ++i) out[i][q] = e4m3(sl[i]);
  }
  unsigned char *base = A + d * (int64_t)tile_bytes(L);
#pragma unroll
  for (int i = 0; i < kTcSlices; ++i)
    *reinterpret_cast<uint4 *>(base + tile_off(L, i, nu, 16 * cg)) = *reinterpret_cast<const uint4 *>(out[i]);
}

// ---------------------------------------------------------------- order-3 coupling
// interpolation point nu of cluster c (tensor Chebyshev points, Eq. (6c))
__device__ __forceinline__ void cheb_point(const double *cheb, int m, int64_t c, int nu, double *x) {
  x[0] = cheb[(3 * c + 0) * m + nu % m];
  x[1] = cheb[(3 * c + 1) * m + (nu / m) % m];
  x[2] = cheb[(3 * c + 2) * m + nu / (m * m)];
}

// E[t][nu] = 1 + floor(log2 max |S_ts[nu][mu]|) over the blocks of row t (0 if none)
__global__ void k_cpl_rowexp(const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                             const double *__restrict__ cheb, int m, int64_t row0, int64_t nclu, KernelFn kf,
                             int32_t *__restrict__ E) {
  const int k = m * m * m;
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (nclu - row0) * k) return;
  const int64_t t = row0 + e / k;
  const int nu = (int)(e % k);
  double x[3], y[3], mx = 0.0;
  cheb_point(cheb, m, t, nu, x);
  for (int64_t b = ptr[t]; b < ptr[t + 1]; ++b)
    for (int mu = 0; mu < k; ++mu) {
      cheb_point(cheb, m, col[b], mu, y);
      mx = fmax(mx, fabs(kernel_value(kf, x, y)));
    }
  E[t * k + nu] = mx > 0.0 ? ilogb(mx) + 1 : 0;
}

// the ten digit planes of scheduled block b (row cluster row0 + brow[b], column cluster col[b]), row
// nu, contraction indices 16 cg .. 16 cg + 15
__global__ void k_cpl_slice(const int32_t *__restrict__ brow, const int32_t *__restrict__ col, int64_t row0,
                            const double *__restrict__ cheb, int m, const int32_t *__restrict__ E, int64_t nblk,
                            KernelFn kf, unsigned char *__restrict__ A) {
  const int k = m * m * m;
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= nblk * k * 2) return;
  const int64_t b = e / (2 * k), t = row0 + brow[b];
  const int nu = (int)((e / 2) % k), cg = (int)(e % 2);
  const int sc = kTcFixBits - E[t * k + nu];
  double x[3], y[3];
  cheb_point(cheb, m, t, nu, x);
  __align__(16) unsigned char out[kTcSlices][16];
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int mu = 16 * cg + q;
    long long X = 0;
    if (mu < k) {
      cheb_point(cheb, m, col[b], mu, y);
      X = llrint(ldexp(kernel_value(kf, x, y), sc));
    }
    int sl[kTcSlices];
    split_digits(X, sl);
#pragma unroll
    for (int i = 0; i < kTcSlices; ++i) out[i][q] = e4m3(sl[i]);
  }
  unsigned char *base = A + b * (int64_t)tile_bytes(k);
#pragma unroll
  for (int i = 0; i < kTcSlices; ++i)
    *reinterpret_cast<uint4 *>(base + tile_off(k, i, nu, 16 * cg)) = *reinterpret_cast<const uint4 *>(out[i]);
}

// xmax[c] = largest |hi| of column c of x ([rows][rp], rp <= 64), as float
// bits: every thread keeps one column
__global__ void __launch_bounds__(256) k_row_max(const dd *__restrict__ x, int64_t rows, int rp,
                                                 unsigned *__restrict__ xmax) {
  pdl_wait();
  pdl_go();
  __shared__ unsigned loc[kXmaxCols];
  if (threadIdx.x < kXmaxCols) loc[threadIdx.x] = 0u;
  __syncthreads();
  const int per = (int)blockDim.x / rp, c = (int)threadIdx.x % rp, q = (int)threadIdx.x / rp;
  float mx = 0.0f;
  if (q < per)
    for (int64_t r = blockIdx.x * (int64_t)per + q; r < rows; r += (int64_t)gridDim.x * per)
      mx = fmaxf(mx, fabsf(x[r * rp + c].hi));
  if (mx > 0.0f) atomicMax(&loc[c], __float_as_uint(mx));
  __syncthreads();
  if ((int)threadIdx.x < rp && loc[threadIdx.x]) atomicMax(&xmax[threadIdx.x], loc[threadIdx.x]);
}

// W of a pass over ncol columns
int tile_width(int ncol) { return ncol <= 4 ? 4 : ncol <= 8 ? 8 : 16; }

template <int W>
int tile_launch(TileArgs a, int grid, cudaStream_t st) {
  a.xch = (uint32_t)((W * (4 * a.R + 1) * (int)sizeof(dd) + 127) / 128 * 128);
  a.stage = 3 * tile_group(a.R) + 32 * tile_n<W>();
  const uint32_t fixed = kTilePad + 2 * a.xch + 8 * (2 * kTileMaxStages + 5) + 16;
  a.nst = (int)std::min<uint32_t>(kTileMaxStages, (kTileSmemMax - fixed) / a.stage) / kTileGroup * kTileGroup;
  // rows_dd's stages and sums take less than the ring's stages
  if (a.spread && kDdStages * rows_dd_stage(a.R, a.Bp, a.ncol) + 8 * kDdThreads * sizeof(dd) > a.nst * a.stage + fixed)
    return fail(H2_EINVAL, "double-float rows do not fit in shared memory");
  H2_CUDA_TRY(cudaFuncSetAttribute((const void *)k_tile_tc<W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kTileSmemMax));
  pdl(k_tile_tc<W>, grid, kTileThreads, a.nst * a.stage + fixed, st, a);
  H2_CUDA_TRY(cudaGetLastError());
  return H2_OK;
}

int tile_run(const TileArgs &a, int width, int grid, cudaStream_t st) {
  switch (width) {
    case 4: return tile_launch<4>(a, grid, st);
    case 8: return tile_launch<8>(a, grid, st);
    default: return tile_launch<16>(a, grid, st);
  }
}

template <int W>
void cut_launch(const dd *x, int64_t first, int64_t count, int R, int rp, int ncol, const unsigned *xmax, int by_level,
                const int *spread, unsigned char *X, cudaStream_t st) {
  constexpr int per = 32 / W;
  pdl(k_tile_cut<W>, (unsigned)((count + per - 1) / per), 128, 0, st, x, first, count, R, rp, ncol, xmax, by_level, spread,
      X);
}

void tile_cut(const dd *x, int64_t first, int64_t count, int R, int rp, int ncol, const unsigned *xmax, int by_level,
              const int *spread, unsigned char *X, int width, cudaStream_t st) {
  switch (width) {
    case 4: return cut_launch<4>(x, first, count, R, rp, ncol, xmax, by_level, spread, X, st);
    case 8: return cut_launch<8>(x, first, count, R, rp, ncol, xmax, by_level, spread, X, st);
    default: return cut_launch<16>(x, first, count, R, rp, ncol, xmax, by_level, spread, X, st);
  }
}

}  // namespace

// The order in which the CTAs of a block-row kernel take their rows, laid out
// at set-up.  Rows are cut into chunks of neighbouring rows (a few dozen
// blocks) and every chunk, in row order, goes to the CTA that has the least to
// do so far: the CTAs work through the rows side by side, so that they read
// the input tiles of one neighbourhood of the tree at a time (all of them
// together exceed L2), and their shares differ by less than a chunk.  A row
// counts its blocks and one more for its epilogue.  The stored blocks follow
// this order, so that a CTA's blocks are one contiguous stream, and its row
// range is two loads instead of two binary searches of the row pointers
// (chains of some 15 dependent loads each).  Chunks of 12 / 32 / 128 / 512
// blocks and rows at 327,680 triangles, 16 right-hand sides: F64 coupling
// 1,905 / 1,911 / 1,925 / 2,004 us, nearfield 354 / 361 / 373 / 383 us.
int row_schedule(Dev &d, const int64_t *ptr, const int32_t *col, int64_t nrows, RowSched &s, SchedTmp &tmp,
                 cudaStream_t st) {
  int dev = 0, sms = 0;
  H2_CUDA_TRY(cudaGetDevice(&dev));
  H2_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int g = (int)std::max<int64_t>(1, std::min<int64_t>(sms, nrows));
  const int64_t nblk = ptr[nrows] - ptr[0];
  const int64_t chunk = std::min<int64_t>(kSchedChunk, (nblk + nrows) / (8 * g));
  std::vector<std::vector<int32_t>> mine(g);
  // (load, CTA), least load first, ties to the lower CTA
  std::priority_queue<std::pair<int64_t, int>, std::vector<std::pair<int64_t, int>>, std::greater<>> next;
  for (int w = 0; w < g; ++w) next.push({0, w});
  for (int64_t r = 0; r < nrows;) {
    auto [load, w] = next.top();
    next.pop();
    int64_t c = 0;
    do {
      mine[w].push_back((int32_t)r);
      c += ptr[r + 1] - ptr[r] + 1;
      ++r;
    } while (r < nrows && c + (ptr[r + 1] - ptr[r]) + 1 <= chunk);
    next.push({load + c, w});
  }
  std::vector<int32_t> row, split(g + 1), cols, src, brow;
  std::vector<int64_t> p2;
  row.reserve(nrows);
  p2.reserve(nrows + 1);
  cols.reserve(nblk);
  src.reserve(nblk);
  brow.reserve(nblk);
  for (int w = 0; w < g; ++w) {
    split[w] = (int32_t)row.size();
    for (int32_t r : mine[w]) {
      row.push_back(r);
      p2.push_back((int64_t)cols.size());
      for (int64_t e = ptr[r]; e < ptr[r + 1]; ++e) {
        cols.push_back(col[e]);
        src.push_back((int32_t)e);
        brow.push_back(r);
      }
    }
  }
  split[g] = (int32_t)row.size();
  p2.push_back((int64_t)cols.size());
  int rc;
  auto up = [&](void **dst, const void *from, size_t bytes) -> int {
    int r = dev_alloc(d, dst, bytes);
    if (r) return r;
    if (bytes) H2_CUDA_TRY(cudaMemcpyAsync(*dst, from, bytes, cudaMemcpyHostToDevice, st));
    return H2_OK;
  };
  if ((rc = up((void **)&s.row, row.data(), row.size() * 4)) || (rc = up((void **)&s.ptr, p2.data(), p2.size() * 8)) ||
      (rc = up((void **)&s.col, cols.data(), cols.size() * 4)) ||
      (rc = up((void **)&s.split, split.data(), split.size() * 4)))
    return rc;
  for (auto [dst, from] : {std::pair<int32_t **, std::vector<int32_t> *>{&tmp.src, &src}, {&tmp.brow, &brow}}) {
    if (dmalloc(dst, std::max<size_t>(from->size() * 4, 16)) != cudaSuccess) {
      cudaGetLastError();
      return fail(H2_ENOMEM, "device set-up buffer");
    }
    H2_CUDA_TRY(cudaMemcpyAsync(*dst, from->data(), from->size() * 4, cudaMemcpyHostToDevice, st));
  }
  H2_CUDA_TRY(cudaStreamSynchronize(st));
  s.grid = g;
  return H2_OK;
}

SchedTmp::~SchedTmp() {
  if (src) cudaFree(src);
  if (brow) cudaFree(brow);
}

// FP64-accurate handles with leaves of at most 32 triangles, unless the
// digits would take more than half of the free device memory
bool ntc_eligible(const Dev &d) {
  if (!(d.prec == H2_F64 && d.tensor == 0 && d.lmax <= kTileMax && d.nnear > 0)) return false;
  size_t fr = 0, tot = 0;
  if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) return false;
  return (double)d.nnear * tile_bytes((int)d.lmax) + (double)d.nleaf * 32 * tile_n<kTcN>() <= 0.5 * (double)fr;
}

int ntc_build(Ctx &c) {
  Dev &d = c.d;
  cudaStream_t st = c.stream;
  const int L = (int)d.lmax, Lp = (int)d.lp;
  const uint32_t ab = tile_bytes(L);
  int rc;
  if ((rc = dev_alloc(d, (void **)&d.ntc_E, sizeof(int32_t) * (size_t)d.nleaf * L))) return rc;
  if ((rc = dev_alloc(d, &d.Ntc, (size_t)d.nnear * ab))) return rc;
  if ((rc = dev_alloc(d, &d.xnt, (size_t)d.nleaf * 32 * tile_n<kTcN>()))) return rc;
  SchedTmp tmp;
  if ((rc = row_schedule(d, c.plan.near_ptr.data(), c.plan.near_col.data(), d.nleaf, d.ntc_s, tmp, st))) return rc;
  H2_CUDA_TRY(cudaMemsetAsync(d.Ntc, 0, (size_t)d.nnear * ab, st));
  const int64_t nr = d.nleaf * L;
  k_near_rowexp<<<(unsigned)((nr + 127) / 128), 128, 0, st>>>((const dd *)d.near, d.near_ptr, d.nleaf, L, Lp,
                                                              d.ntc_E);
  const int64_t ns = d.nnear * L * 2;
  k_near_slice<<<(unsigned)((ns + 255) / 256), 256, 0, st>>>((const dd *)d.near, tmp.src, tmp.brow, d.ntc_E, d.nnear, L,
                                                             Lp, (unsigned char *)d.Ntc);
  H2_CUDA_TRY(cudaGetLastError());
  if ((rc = tc_leaf_build(c))) return rc;
  H2_CUDA_TRY(cudaStreamSynchronize(st));
  d.ntc = true;
  return H2_OK;
}

// the digit tiles of columns c0 .. c0 + ncol - 1 of the permuted input
void ntc_input(Ctx &c, const void *xpad, int rp, int c0, int ncol, bool wide, bool ranged) {
  Dev &d = c.d;
  tile_cut(static_cast<const dd *>(xpad) + c0, 0, d.nleaf, (int)d.lmax, rp, ncol, d.ntc_xmax + c0, 0,
           ranged ? d.spread + c0 : nullptr, (unsigned char *)d.xnt, wide ? kTcN : tile_width(ncol), c.stream);
}

// The nearfield phase (y_pad += or = the near sums), 16 columns per pass.
// The input's column maxima are in place (k_permute_in); have_input: so are
// the wide digit tiles of the one pass of at most 16 columns.  ranged: columns of
// wide range in double-float (their counts are in place too).
int ntc_near(Ctx &c, const void *xpad, void *ypad, int rp, int accumulate, int64_t *launches, bool ranged,
             bool have_input) {
  Dev &d = c.d;
  int64_t nl = 0;
  for (int c0 = 0; c0 < rp; c0 += kTcN) {
    const int ncol = std::min(kTcN, rp - c0);
    if (!have_input) {
      ntc_input(c, xpad, rp, c0, ncol, false, ranged);
      ++nl;
    }
    TileArgs a{};
    a.A = (const unsigned char *)d.Ntc;
    a.X = (const unsigned char *)d.xnt;
    a.ptr = d.ntc_s.ptr;
    a.col = d.ntc_s.col;
    a.row = d.ntc_s.row;
    a.split = d.ntc_s.split;
    a.E = d.ntc_E;
    a.xmax = d.ntc_xmax + c0;
    a.spread = ranged ? d.spread + c0 : nullptr;
    a.colmax = d.colmax + c0;
    a.B = static_cast<const dd *>(d.near);
    a.Bp = (int)d.lp;
    a.bptr = d.near_ptr;
    a.bcol = d.near_col;
    a.Xd = static_cast<const dd *>(xpad) + c0;
    a.out = static_cast<dd *>(ypad) + c0;
    a.R = (int)d.lmax;
    a.ncol = ncol;
    a.rp = rp;
    a.accumulate = accumulate;
    const int rc = tile_run(a, have_input ? kTcN : tile_width(ncol), d.ntc_s.grid, c.stream);
    if (rc) return rc;
    ++nl;
  }
  H2_CUDA_TRY(cudaGetLastError());
  if (launches) *launches = nl;
  return H2_OK;
}

// Coupling of FP64-accurate order-3 handles with stored coupling (k = 27),
// unless the digits would take more than half of the free device memory or
// the handle's products are single launches
bool tct_eligible(const Dev &d) {
  if (!(d.prec == H2_F64 && d.tensor == 0 && !d.gca && d.coupling == 0 && d.m == 3 && d.nadm > 0)) return false;
  if (d.fused && d.n <= kFusedMaxN) return false;
  size_t fr = 0, tot = 0;
  if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) return false;
  return (double)d.nadm * tile_bytes(d.k) + (double)d.nclu * 32 * tile_n<kTcN>() <= 0.5 * (double)fr;
}

int tct_build(Ctx &c) {
  Dev &d = c.d;
  cudaStream_t st = c.stream;
  const int64_t row0 = ((int64_t)1 << d.first_adm_level) - 1;
  const uint32_t ab = tile_bytes(d.k);
  int rc;
  SchedTmp tmp;
  if ((rc = row_schedule(d, c.plan.adm_ptr.data() + row0, c.plan.adm_col.data(), d.nclu - row0, d.tc_s, tmp, st)))
    return rc;
  if ((rc = dev_alloc(d, (void **)&d.tc_E, sizeof(int32_t) * (size_t)d.nclu * d.k))) return rc;
  if ((rc = dev_alloc(d, &d.Stc, (size_t)d.nadm * ab))) return rc;
  if ((rc = dev_alloc(d, &d.xtc, (size_t)d.nclu * 32 * tile_n<kTcN>()))) return rc;
  H2_CUDA_TRY(cudaMemsetAsync(d.tc_E, 0, sizeof(int32_t) * (size_t)d.nclu * d.k, st));
  H2_CUDA_TRY(cudaMemsetAsync(d.Stc, 0, (size_t)d.nadm * ab, st));
  const int64_t nr = (d.nclu - row0) * d.k, ns = d.nadm * d.k * 2;
  k_cpl_rowexp<<<(unsigned)((nr + 127) / 128), 128, 0, st>>>(d.adm_ptr, d.adm_col, d.cheb, d.m, row0, d.nclu,
                                                             d.kernel, d.tc_E);
  k_cpl_slice<<<(unsigned)((ns + 255) / 256), 256, 0, st>>>(tmp.brow, d.tc_s.col, row0, d.cheb, d.m, d.tc_E, d.nadm,
                                                            d.kernel, (unsigned char *)d.Stc);
  H2_CUDA_TRY(cudaGetLastError());
  H2_CUDA_TRY(cudaStreamSynchronize(st));
  d.tct = true;
  return H2_OK;
}

// column maxima of the leaf coefficients (where the leaf step does not take them)
void tct_leaf_max(Ctx &c, const void *xhat, int rp) {
  const Dev &d = c.d;
  const int64_t rows = d.nleaf * d.k, per = 256 / rp;
  const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((rows + 8 * per - 1) / (8 * per), 152 * 8));
  pdl(k_row_max, grid, 256, 0, c.stream, static_cast<const dd *>(xhat) + (d.nleaf - 1) * d.k * (int64_t)rp, rows, rp,
                                        d.tc_xmax + d.depth * kXmaxCols);
}

// the coupling phase, 16 columns per pass; the column maxima of every level and the input's
// counts are in place
int tct_coupling(Ctx &c, const void *xhat, void *yhat, int rp, int64_t *launches) {
  Dev &d = c.d;
  const int64_t row0 = ((int64_t)1 << d.first_adm_level) - 1;
  int64_t nl = 0;
  for (int c0 = 0; c0 < rp; c0 += kTcN) {
    const int ncol = std::min(kTcN, rp - c0);
    tile_cut(static_cast<const dd *>(xhat) + c0, row0, d.nclu - row0, d.k, rp, ncol, d.tc_xmax + c0, 1,
             d.spread + c0, (unsigned char *)d.xtc, tile_width(ncol), c.stream);
    TileArgs a{};
    a.A = (const unsigned char *)d.Stc;
    a.X = (const unsigned char *)d.xtc;
    a.ptr = d.tc_s.ptr;
    a.col = d.tc_s.col;
    a.row = d.tc_s.row;
    a.split = d.tc_s.split;
    a.E = d.tc_E;
    a.xmax = d.tc_xmax + c0;
    a.spread = d.spread + c0;
    a.colmax = d.colmax + c0;
    a.B = static_cast<const dd *>(d.S);
    a.Bp = d.kp;
    a.bptr = d.adm_ptr + row0;
    a.bcol = d.adm_col;
    a.Xd = static_cast<const dd *>(xhat) + c0;
    a.out = static_cast<dd *>(yhat) + c0;
    a.R = d.k;
    a.ncol = ncol;
    a.rp = rp;
    a.row0 = row0;
    a.by_level = 1;
    const int rc = tile_run(a, tile_width(ncol), d.tc_s.grid, c.stream);
    if (rc) return rc;
    nl += 2;
  }
  H2_CUDA_TRY(cudaGetLastError());
  if (launches) *launches = nl;
  return H2_OK;
}

// this file's device error word (its bounded waits)
int tile_take_error(cudaStream_t st) {
  int v = 0, zero = 0;
  H2_CUDA_TRY(cudaMemcpyFromSymbolAsync(&v, g_h2_device_error, sizeof(int), 0, cudaMemcpyDeviceToHost, st));
  H2_CUDA_TRY(cudaStreamSynchronize(st));
  if (v) {
    H2_CUDA_TRY(cudaMemcpyToSymbolAsync(g_h2_device_error, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, st));
    H2_CUDA_TRY(cudaStreamSynchronize(st));
    return fail(H2_ETIMEOUT, "a bounded device wait of the tensor-core block rows ran out");
  }
  return H2_OK;
}

}  // namespace h2
