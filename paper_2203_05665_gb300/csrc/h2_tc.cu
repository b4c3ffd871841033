// Coupling phase of order-4 handles (k = 64) on the tensor cores (tcgen05, FP8
// E4M3 operands, FP32 accumulation in tensor memory), up to 16 right-hand sides,
// in FP64 accuracy (ten digits per value) or FP32 accuracy (six digits), and the
// FP64-accurate leaf forward step of leaves of at most 21 triangles.  Block rows
// with smaller tiles (nearfield, order-3 coupling) are in h2_tile.cu.
//
// GB300 runs FP64 at 1/58 of its FP32 rate, and double-float arithmetic on
// the FP32 pipe leaves the coupling (Algorithm 3, y^_t = sum S_ts x^_s)
// bound by instruction issue far below the memory roofline.  This path
// computes the same sums exactly enough for FP64 parity with integer digits
// on the tensor cores (the splitting scheme of Ozaki et al.):
//
//  * every row nu of the coupling matrices of row cluster t gets a power of
//    two 2^E (E[t][nu], common to all blocks of the row, |S| < 2^E), every
//    column j of the coefficients of tree level l a power of two 2^F;
//  * a value v becomes the integer X = round(v 2^(49-E)), |X| <= 2^49,
//    split into ten signed 5-bit digits, X = sum_i s_i 2^(50-5i),
//    |s_i| <= 16: every digit is exact in FP8 E4M3 (one byte);
//  * D_ik = sum_blocks sum_mu s_i[nu][mu] t_k[mu][j] is a sum of at most
//    64 x 64 products of magnitude <= 2^8, an integer of at most 2^20: the
//    tensor cores accumulate it exactly in FP32, and the at most five D_ik
//    of one level i + k add exactly in FP32 too;
//  * y^_t[nu][j] = 2^(E + F) sum_{i + k <= 11} 2^(2-5(i+k)) D_ik, the ten
//    levels summed in double-float; the dropped pairs and the rounding of X
//    stay below 2^-46 of the row's scale.  With six digits (FP32 handles):
//    |X| <= 2^29, pairs i + k <= 7, below 2^-27.
//
// The digits of S are cut once at set-up, straight into the layout the
// tensor cores read from shared memory (K-major, 8 x 16-byte core matrices,
// no swizzle), 10 bytes per entry, so bulk copies (TMA engine) move a block
// as it is stored; the coefficients are cut once per product.  One MMA
// instruction (kind::f8f6f4, K = 32) multiplies two stacked digit planes of
// S (M = 128 rows: digits i and i+1) by the digit planes of x^ it pairs with
// (N = 16 columns per plane, 160 down to 32): five such groups, two K steps
// each, 10 instructions per block.  The groups write their pairs so that the
// pairs of one level i + k land in the same accumulator columns (the tensor
// cores add them, exactly), so a segment's results take 160 columns and
// there are three accumulator sets, one per epilogue group: the MMAs of one row
// overlap the epilogues of the two before it.
//
// Kernel roles (one CTA per SM, 14 warps): warp 0 streams the digits of each
// block through a shared-memory ring (bulk copies completing on mbarriers;
// the digit stream evict-first in L2, the coefficient tiles evict-last),
// warp 1 allocates tensor memory and issues the MMAs of a row segment (at
// most 64 blocks) into the row's accumulator set, three groups of four warps take
// the rows in turn, each with its own set: they read it back (tcgen05.ld), add
// the levels in double-float, and write y^_t.  The rows follow row_schedule
// (h2_tile.cu), so that the CTAs read the coefficient tiles of one
// neighbourhood at a time and L2 holds them.  327,680 triangles, 16 right-hand
// sides: FP64-accurate 2,197 -> 1,905 us (6.6 TB/s of stored digits, 0.97 of the
// copy bandwidth), FP32 1,515 -> 1,173 us (6.4 TB/s).  Every wait is bounded; on a timeout the
// device error word is raised, every role stops, copies and MMAs in flight
// are waited for and the tensor memory is released before the CTA exits.
#include <cuda_fp8.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "h2_dd.cuh"
#include "h2_digits.hpp"
#include "h2_internal.hpp"
#include "h2_kernel.cuh"
#include "h2_launch.cuh"
#include "h2_ptx.cuh"
#include "h2_tc.cuh"
#include "h2_transfer.cuh"

namespace h2 {
namespace {

constexpr int kTcK = 64;                 // rank k = m^3, m = 4
constexpr int kLeafTcMax = 21;           // largest leaf of the tensor-core leaf forward step
constexpr int kTcSegBlocks = 64;         // blocks accumulated in one exact segment (sums <= 2^20)
constexpr uint32_t kSliceA = kTcK * kTcK;              // 4096 bytes: one digit plane of S_b (64 x 64 E4M3)

// The coupling's digit layout for ND digits per value: ND = 10 for FP64
// accuracy (|X| <= 2^49, pairs i + k <= 11), ND = 6 for FP32 accuracy (|X| <=
// 2^29, pairs i + k <= 7: the dropped pairs stay below 2^-27 of the row's
// scale).  Group g pairs S digits 2g+1 (accumulator lanes 0-63) and 2g+2
// (lanes 64-127) with x^ digits k = 1 .. ND - 2g (N = 16 (ND - 2g)) and
// writes them from accumulator column 2 W g on: x^ digit k of group g lands in
// column block 2g + k - 1, so column block c holds, in lanes 0-63, the sum of
// every pair of level i + k = c + 2 and, in lanes 64-127, of level c + 3.  The
// tensor cores thus add the pairs of one level themselves (exactly: at most
// five sums of at most 2^20 each), an accumulator set is W ND columns wide
// (160 or 96 for W = 16), and each epilogue group has a set of its own, so that the
// MMAs of the next rows run while it reads its row.
//
// KB is the contraction length of one block in bytes: 64 for the coupling
// matrices (two MMA K steps), 32 for the leaf bases V_t^T of the leaf forward
// step (the L <= 32 triangles of a leaf, zero padded; one K step).
//
// W is the columns of a product the tiles are laid out for: 16, or 8 for up to
// 8 right-hand sides of the coupling (half the coefficient digits, accumulator
// columns and epilogue arithmetic).  FP64-accurate, 81,920 triangles, with the leaf
// forward step in double-float and narrow nearfield tiles at these widths: one
// column 705 -> 648 us, Helmholtz with 8 real columns 1,651 -> 1,559 us.
template <int ND, int KB = kTcK, int W = kTcN>
struct Dig {
  static constexpr int kFix = 5 * ND - 1;
  static constexpr int kTop = ND + 1;
  static constexpr int kGroups = ND / 2;
  static constexpr int kKSteps = KB / 32;
  static constexpr uint32_t kPlaneA = kTcK * KB;   // one digit plane of a block: 64 rows x KB
  static constexpr uint32_t kPlaneB = W * KB;      // one digit plane of the coefficients: W rows x KB
  static constexpr uint32_t kTileA = ND * kPlaneA;
  static constexpr uint32_t kTileB = ND * kPlaneB;
  static constexpr uint32_t kStage = kTileA + kTileB;
  static constexpr int kStages = (ND == 10 ? 4 : 6) * (kTcK / KB);
  // stages released by one commit (with one commit per block the MMA warp bounded the
  // coupling: FP32, 327,680 triangles, 16 right-hand sides 1,457 us, per two 1,415 us;
  // one-block rows wait for every block's results anyway)
  static constexpr int kRel = KB == kTcK ? 2 : 1;
  static constexpr uint32_t kW = W * ND;         // columns of an accumulator set
  static constexpr int kSets = 3;   // one per epilogue group
  __host__ __device__ static constexpr int nx(int g) { return ND - 2 * g; }
  __host__ __device__ static constexpr uint32_t col(int g) { return (uint32_t)(2 * W * g); }
};
static_assert(Dig<10>::kSets * Dig<10>::kW <= 512 && Dig<6>::kSets * Dig<6>::kW <= 512, "accumulator sets");
// epilogue warp groups, one per accumulator set (one group for all three sets held up
// the rows: with its arithmetic left out the F64 coupling at 327,680 triangles and 16
// right-hand sides took 2,018 instead of 2,118 us)
constexpr int kRowGroups = 3;
constexpr int kTcThreads = 64 + kRowGroups * 128;   // producer, MMA, epilogue warps
// each epilogue group has an exchange area of 64 rows x W double-float values
template <int ND, int KB = kTcK, int W = kTcN>
__host__ __device__ constexpr uint32_t tc_bar_off() {
  return Dig<ND, KB, W>::kStages * Dig<ND, KB, W>::kStage + kRowGroups * (64 * W * 8);
}
template <int ND, int KB = kTcK, int W = kTcN>
__host__ __device__ constexpr uint32_t tc_smem() { return tc_bar_off<ND, KB, W>() + 40 * 8 + 16; }

// byte offset of (row r, contraction index c) in a K-major one-byte operand
// of 64 contraction values per row: core matrices of 8 rows x 16 bytes, four
// along K (128 bytes apart), then the next 8 rows (512 bytes on)
__host__ __device__ __forceinline__ int core_off(int r, int c) {
  return ((r >> 3) * 4 + (c >> 4)) * 128 + (r & 7) * 16 + (c & 15);
}

// shared-memory matrix descriptor (no swizzle) of rows of KB contraction
// bytes: start address, leading byte offset 128 (next core matrix along K),
// stride byte offset 8 KB (next 8 rows), descriptor version 1
template <int KB>
__device__ __forceinline__ uint64_t sdesc_kb(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16) |
         ((uint64_t)((8u * KB) >> 4) << 32) | (1ull << 46);
}

// interpolation point nu of cluster c (tensor Chebyshev points, Eq. (6c))
__device__ __forceinline__ void tc_point(const double *cheb, int64_t c, int nu, double *x) {
  x[0] = cheb[(3 * c + 0) * 4 + (nu & 3)];
  x[1] = cheb[(3 * c + 1) * 4 + ((nu >> 2) & 3)];
  x[2] = cheb[(3 * c + 2) * 4 + (nu >> 4)];
}

// ---------------------------------------------------------------- set-up
// E[t][nu]: 1 + floor(log2 max |S_ts[nu][mu]|) over the blocks of row t (0 if none)
__global__ void k_tc_rowexp(const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                            const double *__restrict__ cheb, int64_t row0, int64_t nclu, KernelFn kf,
                            int32_t *__restrict__ E) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (nclu - row0) * kTcK) return;
  const int64_t t = row0 + e / kTcK;
  const int nu = (int)(e % kTcK);
  double x[3], y[3], mx = 0.0;
  tc_point(cheb, t, nu, x);
  for (int64_t b = ptr[t]; b < ptr[t + 1]; ++b)
    for (int mu = 0; mu < kTcK; ++mu) {
      tc_point(cheb, col[b], mu, y);
      mx = fmax(mx, fabs(kernel_value(kf, x, y)));
    }
  E[t * kTcK + nu] = mx > 0.0 ? ilogb(mx) + 1 : 0;
}

// the ND E4M3 digit planes of scheduled block b (row cluster row0 + brow[b]), row nu, contraction
// indices 16 cg .. 16 cg + 15
template <int ND>
__global__ void k_tc_slice_s(const int32_t *__restrict__ brow, const int32_t *__restrict__ col, int64_t row0,
                             const double *__restrict__ cheb, const int32_t *__restrict__ E, int64_t nblk,
                             KernelFn kf, unsigned char *__restrict__ Stc) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= nblk * kTcK * 4) return;
  const int64_t b = e / (kTcK * 4);
  const int nu = (int)((e / 4) % kTcK), cg = (int)(e % 4);
  const int64_t t = row0 + brow[b], s = col[b];
  double x[3], y[3];
  tc_point(cheb, t, nu, x);
  const int sc = Dig<ND>::kFix - E[t * kTcK + nu];
  __align__(16) unsigned char out[ND][16];
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    tc_point(cheb, s, 16 * cg + q, y);
    const long long X = llrint(ldexp(kernel_value(kf, x, y), sc));
    int sl[ND];
    split_digits<ND>(X, sl);
#pragma unroll
    for (int i = 0; i < ND; ++i) out[i][q] = e4m3(sl[i]);
  }
  unsigned char *base = Stc + b * (int64_t)Dig<ND>::kTileA + core_off(nu, 16 * cg);
#pragma unroll
  for (int i = 0; i < ND; ++i)
    *reinterpret_cast<uint4 *>(base + i * kSliceA) = *reinterpret_cast<const uint4 *>(out[i]);
}

// ---------------------------------------------------------------- per product
// xmax[j] = largest |x| (double-float: |hi|) of column j over rows [0, rows) of x
// ([rows][rp], as float bits, infinities and NaN above all others).  A warp reads 32 / LPR rows at a time with 16-byte
// loads (LPR lanes per row of 16 columns, lane l: row l / LPR, its EPV columns
// from EPV (l % LPR)), so the reads are contiguous and every lane keeps fixed
// columns; rp is a multiple of EPV (rows are padded to 16 bytes).
template <class T>
__global__ void k_tc_levmax(const T *__restrict__ x, int64_t rows, int rp, unsigned *__restrict__ xmax) {
  pdl_wait();
  pdl_go();
  constexpr int EPV = 16 / (int)sizeof(T), LPR = kTcN / EPV, RPW = 32 / LPR;
  __shared__ unsigned loc[kTcN];
  if (threadIdx.x < kTcN) loc[threadIdx.x] = 0u;
  __syncthreads();
  const int lane = threadIdx.x & 31, sub = lane % LPR, nv = rp / EPV;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const int64_t w = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
  unsigned m[EPV];
#pragma unroll
  for (int e = 0; e < EPV; ++e) m[e] = 0u;
  if (sub < nv)
    for (int64_t r = RPW * w + lane / LPR; r < rows; r += RPW * warps) {
      const T *p = x + r * rp + EPV * sub;
#pragma unroll
      for (int e = 0; e < EPV; ++e) m[e] = max(m[e], __float_as_uint(mag_of(p[e])));
    }
#pragma unroll
  for (int e = 0; e < EPV; ++e)
    for (int o = LPR; o < 32; o <<= 1) m[e] = max(m[e], __shfl_xor_sync(0xffffffffu, m[e], o));
  if (lane < nv)
#pragma unroll
    for (int e = 0; e < EPV; ++e)
      if (m[e]) atomicMax(&loc[EPV * lane + e], m[e]);
  __syncthreads();
  if (threadIdx.x < kTcN && loc[threadIdx.x]) atomicMax(&xmax[threadIdx.x], loc[threadIdx.x]);
}

// The ND E4M3 digit planes of the coefficients x^_c ([64][rp]) of clusters
// c0 .. c0 + ncl - 1, each with the column maxima of its own tree level:
// 4 W threads per cluster (64 / W per CTA), thread (g, j) cuts the values
// mu = 16 g .. 16 g + 15 of column j in registers and writes one 16-byte row
// of a core matrix per plane (zero digits for the columns j >= rp).
template <class T, int ND, int W>
__global__ void __launch_bounds__(256) k_tc_slice_x(const T *__restrict__ xhat, int64_t c0, int64_t ncl, int rp,
                                                    const unsigned *__restrict__ xmax, unsigned char *__restrict__ xtc) {
  pdl_wait();
  pdl_go();
  const int64_t ci = (int64_t)blockIdx.x * (64 / W) + threadIdx.x / (4 * W);
  if (ci >= ncl) return;
  const int64_t c = c0 + ci;
  const int g = (threadIdx.x / W) & 3, j = threadIdx.x % W;
  const T *xc = xhat + c * kTcK * rp;
  const int sc = Dig<ND>::kFix - tc_colexp(xmax[tc_level(c) * kXmaxCols + j]);
  T v[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) v[q] = j < rp ? xc[(16 * g + q) * rp + j] : T{};
  uint32_t w[ND][4];
  cut_row<ND, 16>(v, sc, w);
  unsigned char *dst = xtc + c * (int64_t)Dig<ND, kTcK, W>::kTileB + core_off(j, 16 * g);
#pragma unroll
  for (int i = 0; i < ND; ++i)
    *reinterpret_cast<uint4 *>(dst + i * Dig<ND, kTcK, W>::kPlaneB) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
}

// The coupling kernel (see the top of the file).  Rows t = row0 + r for r
// in [0, nrows); each CTA takes a contiguous range of rows holding about
// 1/gridDim of the blocks.
// T: the coefficient type (dd with ND = 10, float with ND = 6).
// DIAG: row r holds the single block r in column r (ptr = col = NULL), its
// row powers of two are E[r][nu] and the column powers xmax[j] (one level):
// the leaf forward step x^_t = V_t^T x|t with KB = 32, the V_t^T digit
// planes as the blocks and the input digit planes of leaf t as the
// coefficients (with ymax, the largest |hi| of every column of the results
// is taken too, as float bits).  Three epilogue warp groups then take every
// third row, and two
// neighbouring digit levels are combined exactly in FP32 before entering
// double-float: a level sum of one block is at most 5 x 32 x 16^2 < 2^15.4,
// so 32 D_L + D_(L+1) < 2^21.
__device__ __forceinline__ dd to_dd(dd v) { return v; }
__device__ __forceinline__ dd to_dd(float v) { return dd{v, 0.0f}; }
__device__ __forceinline__ void store_as(dd v, dd *p) { *p = v; }
__device__ __forceinline__ void store_as(dd v, float *p) { *p = v.hi + v.lo; }

template <int ND, class T, int KB = kTcK, bool DIAG = false, int W = kTcN>
__global__ void __launch_bounds__(kTcThreads, 1)
    k_coupling_tc(const unsigned char *__restrict__ Stc, const unsigned char *__restrict__ xtc,
                  const int64_t *__restrict__ ptr, const int32_t *__restrict__ col, const int32_t *__restrict__ row,
                  const int32_t *__restrict__ split, const int32_t *__restrict__ E, const unsigned *__restrict__ xmax,
                  int64_t row0, int64_t nrows, int rp, T *__restrict__ yhat, unsigned *__restrict__ ymax, uint32_t xstride) {
  using D = Dig<ND, KB, W>;
  static_assert(!DIAG || W == kTcN, "one-block rows read tiles of 16 columns");
  // first block of scheduled row r; one block per row without ptr
  auto pt = [&](int64_t r) -> int64_t { return DIAG ? r : ptr[r]; };
  constexpr int kTcStages = D::kStages, kTcGroups = D::kGroups;
  constexpr uint32_t kStage = D::kStage, kTileA = D::kTileA, kTileB = D::kTileB;
  extern __shared__ __align__(1024) unsigned char smem[];
  dd *xch = reinterpret_cast<dd *>(smem + kTcStages * kStage);
  constexpr int kSets = D::kSets;
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + tc_bar_off<ND, KB, W>());
  uint64_t *empty = full + kTcStages;
  uint64_t *accf = empty + kTcStages;   // [kSets]: the MMAs of a segment have completed
  uint64_t *acce = accf + kSets;        // [kSets]: the epilogue has read the set
  uint64_t *done = acce + kSets;
  uint32_t *tslot = reinterpret_cast<uint32_t *>(done + 1);
  volatile int *abort = reinterpret_cast<volatile int *>(tslot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // rows of this CTA: laid out at set-up, or an equal share of one-block rows
  const int64_t r_begin = DIAG ? nrows * blockIdx.x / gridDim.x : split[blockIdx.x];
  const int64_t r_end = DIAG ? nrows * (blockIdx.x + 1) / gridDim.x : split[blockIdx.x + 1];
  const int64_t e_begin = pt(r_begin), e_end = pt(r_end);

  if (tid == 0) {
    for (int s = 0; s < kTcStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int u = 0; u < kSets; ++u) {
      mbar_init(&accf[u], 1);
      mbar_init(&acce[u], 4);
    }
    mbar_init(done, 1);
    *abort = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = *tslot;
  pdl_wait();   // everything above is set-up data and this CTA's own
  pdl_go();

  if (warp == 0) {
    // ---------------- producer: the slices of every block of the range
    if (lane == 0) {
      int64_t e = e_begin;
      ColAhead ca(col, e, e_end);
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
          if (s % D::kRel == 0 && e - e_begin >= kTcStages && !mbar_wait_or_abort(&empty[s / D::kRel], ph, abort)) {
            ok = false;
            break;
          }
          unsigned char *st = smem + (size_t)s * kStage;
          mbar_expect_tx(&full[s], kStage);
          // the coefficient digits (read by every block of their column: kept in L2) and
          // S (read once: evicted first)
          bulk_g2s_hint(st + kTileA, xtc + (int64_t)cb[u] * xstride, kTileB, &full[s], pol_keep);
          bulk_g2s_hint(st, Stc + e * (int64_t)kTileA, kTileA, &full[s], pol_stream);
          ++e;
          if (++s == kTcStages) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (*abort) {
        // let the copies in flight land before the CTA leaves (bounded)
        const int64_t j0 = e - kTcStages > e_begin ? e - kTcStages : e_begin;
        for (int64_t j = j0; j < e; ++j) {
          const int64_t ij = j - e_begin;
          mbar_wait_bounded(&full[ij % kTcStages], (uint32_t)((ij / kTcStages) & 1));
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (the whole warp waits, an elected lane issues)
    {
      int s = 0, set = kSets - 1;
      uint32_t ph = 0, use[kSets] = {};
      bool ok = true;
      int64_t pnext = pt(r_begin);   // row pointers loaded one row ahead
      for (int64_t r = r_begin; r < r_end && ok; ++r) {
        const int64_t b0 = pnext;
        pnext = pt(r + 1);
        const int64_t nb = pnext - b0;
        if (nb > 0) set = set == kSets - 1 ? 0 : set + 1;   // the rows that have blocks take the sets in turn
        for (int64_t s0 = 0; s0 < nb && ok; s0 += kTcSegBlocks) {
          // the set is free once its epilogue group has read its previous use
          uint32_t u = 0;
#pragma unroll
          for (int v = 0; v < kSets; ++v)
            if (set == v) u = use[v]++;
          if (u > 0 && !mbar_wait_or_abort(&acce[set], (u - 1) & 1, abort)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t dset = tbase + (uint32_t)set * D::kW;
          const int64_t sn = nb - s0 < kTcSegBlocks ? nb - s0 : kTcSegBlocks;
          for (int64_t t = 0; t < sn; ++t) {
            if (!mbar_wait_or_abort(&full[s], ph, abort)) {
              ok = false;
              break;
            }
            tc_fence_after();
            // descriptors of the stage; offsets below 256 KB add to the 14-bit address field.
            // Group g: S digits 2g+1, 2g+2 (M = 128 rows) times x^ digits 1 .. ND - 2g into
            // column blocks 2g .. ND - 1 of the set.  Group 0 covers every column, so its
            // first MMA of a segment overwrites the set and all later ones accumulate.
            // K steps (32 bytes, two core matrices) outermost.
            const uint32_t A0 = smem_u32(smem + (size_t)s * kStage), B0 = A0 + kTileA;
            const uint64_t dA = sdesc_kb<KB>(A0), dB = sdesc_kb<KB>(B0);
#pragma unroll
            for (int kk = 0; kk < D::kKSteps; ++kk)
#pragma unroll
              for (int g = 0; g < kTcGroups; ++g)
                tc_mma(dset + D::col(g), dA + (uint64_t)((2 * g * D::kPlaneA + kk * 256) >> 4),
                       dB + (uint64_t)(kk * 16), tc_idesc(W * D::nx(g)), (t > 0 || kk > 0 || g > 0) ? 1u : 0u);
            // the stages of a release group are free once these MMAs have read them
            if (s % D::kRel == D::kRel - 1) tc_commit(&empty[s / D::kRel]);
            if (++s == kTcStages) {
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
  } else if (DIAG) {
    // ---------------- one-block rows: warps 2-5 (group 0), 6-9 (group 1) and
    // 10-13 (group 2) take every third row; each reads tensor-memory lanes
    // 32 (warp % 4) ..
    const int grp = (warp - 2) >> 2;
    const int quad = warp & 3, tl = quad * 32 + lane, half = tl >> 6, nu = tl & 63;
    dd *xg = xch + grp * (64 * kTcN);
    const uint32_t bar_or = 1 + 2 * grp, bar_x = 2 + 2 * grp;
    int cx[kTcN];
    float cm[kTcN];   // column maxima of the rows this thread writes
#pragma unroll
    for (int j = 0; j < kTcN; ++j) {
      cx[j] = tc_colexp(xmax[j]);
      cm[j] = 0.0f;
    }
    int64_t r = r_begin + grp;
    int Enext = r < r_end ? E[r * kTcK + nu] : 0;   // the row's powers, loaded a row ahead
    for (; r < r_end; r += kRowGroups) {
      const int64_t q = r - r_begin, t = row0 + r;
      const int Er = Enext;
      if (r + kRowGroups < r_end) Enext = E[(r + kRowGroups) * kTcK + nu];
      T *yrow = yhat + (t * kTcK + nu) * rp;
      const int set = (int)(q % kSets);
      const bool ready = !*abort && mbar_wait_or_abort(&accf[set], (uint32_t)((q / kSets) & 1), abort);
      if (named_sync_or_id(bar_or, 128, ready ? 0 : 1)) break;
      tc_fence_after();
      dd acc[kTcN];
#pragma unroll
      for (int j = 0; j < kTcN; ++j) acc[j] = dd{0.0f, 0.0f};
      // column block c holds level L = c + 2 + half; blocks c, c + 1 combine as
      // (32 D_L + D_(L+1)) 2^(2 - 5 (L + 1)), in increasing L
      const uint32_t tset = tbase + ((uint32_t)(quad * 32) << 16) + (uint32_t)set * D::kW;
#pragma unroll
      for (int c0 = 0; c0 < ND; c0 += 4) {
        uint32_t raw[4][16];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (c0 + u < ND) tmem_ld16_nw(tset + (uint32_t)((c0 + u) * kTcN), raw[u]);
        tmem_wait();
#pragma unroll
        for (int u = 0; u < 4; u += 2) {
          const int L = c0 + u + 2 + half;
          if (c0 + u < ND && L <= D::kTop) {
            const float w = pow2f(2 - 5 * (L + 1));
            const float c1 = L + 1 <= D::kTop ? 1.0f : 0.0f;
#pragma unroll
            for (int j = 0; j < kTcN; ++j) {
              const float v = 32.0f * __uint_as_float(raw[u][j]) + c1 * __uint_as_float(raw[u + 1][j]);
              acc[j] = acc[j] + dd{v * w, 0.0f};
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acce[set]);
      if (half == 1)
#pragma unroll
        for (int j = 0; j < kTcN; ++j) xg[j * 64 + nu] = acc[j];
      named_sync_id(bar_x, 128);
      if (half == 0) {
#pragma unroll
        for (int j = 0; j < kTcN; ++j) {
          if (j >= rp) break;
          const dd v = dd_scale(acc[j] + xg[j * 64 + nu], Er + cx[j]);
          store_as(v, yrow + j);
          cm[j] = fmaxf(cm[j], fabsf(v.hi));
        }
      }
      named_sync_id(bar_x, 128);
    }
    if (ymax && half == 0) {
#pragma unroll
      for (int j = 0; j < kTcN; ++j) {
        float m = cm[j];
#pragma unroll
        for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0 && j < rp && m > 0.0f) atomicMax(&ymax[j], __float_as_uint(m));
      }
    }
  } else {
    // ---------------- epilogue groups (warps 2-5, 6-9, 10-13; each warp reads
    // tensor-memory lanes 32 (warp % 4) ..): they take the rows that have blocks in
    // turn, each with its own accumulator set
    const int grp = (warp - 2) >> 2;
    const int quad = warp & 3, tl = quad * 32 + lane, half = tl >> 6, nu = tl & 63;
    dd *xg = xch + grp * (64 * W);
    const uint32_t bar_or = 1 + 2 * grp, bar_x = 2 + 2 * grp;
    uint32_t use = 0;
    int turn = kSets - 1;
    int64_t pnext = pt(r_begin);
    int32_t rnext = r_begin < r_end ? row[r_begin] : 0;
    for (int64_t r = r_begin; r < r_end; ++r) {
      const int64_t t = row0 + rnext, b0 = pnext;
      pnext = pt(r + 1);
      if (r + 1 < r_end) rnext = row[r + 1];
      const int64_t nb = pnext - b0;
      T *yrow = yhat + (t * kTcK + nu) * rp;
      if (nb == 0) {
        if (half == 0 && grp == 0)
          for (int j = 0; j < rp; ++j) store_as(dd{0.0f, 0.0f}, yrow + j);
        continue;
      }
      turn = turn == kSets - 1 ? 0 : turn + 1;
      if (turn != grp) continue;
      const int Er = E[t * kTcK + nu];
      const int lvl = tc_level(t);
      int Fc[W];
#pragma unroll
      for (int j = 0; j < W; ++j) Fc[j] = Er + tc_colexp(xmax[lvl * kXmaxCols + j]);
      bool stop = false;
      for (int64_t s0 = 0; s0 < nb; s0 += kTcSegBlocks, ++use) {
        const int set = grp;
        const bool ready = !*abort && mbar_wait_or_abort(&accf[set], use & 1, abort);
        if (named_sync_or_id(bar_or, 128, ready ? 0 : 1)) {   // the group's warps agree to stop
          stop = true;
          break;
        }
        tc_fence_after();
        dd acc[W];
#pragma unroll
        for (int j = 0; j < W; ++j) acc[j] = dd{0.0f, 0.0f};
        // column block c of lane nu (+ 64) holds the sum of every digit pair of level
        // L = c + 2 (+ 1) (integers, exact in FP32); the levels share the weight
        // 2^(2-5L) and enter the double-float result once each, in increasing order
        // (L <= ND + 1: lanes 64-127 skip their last block)
        const uint32_t tset = tbase + ((uint32_t)(quad * 32) << 16) + (uint32_t)set * D::kW;
#pragma unroll
        for (int c0 = 0; c0 < ND; c0 += 4) {
          uint32_t raw[4 * W / 16][16];   // four column blocks
#pragma unroll
          for (int u = 0; u < 4 * W / 16; ++u)
            if (c0 * W + 16 * u < ND * W) tmem_ld16_nw(tset + (uint32_t)(c0 * W + 16 * u), raw[u]);
          tmem_wait();
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int L = c0 + u + 2 + half;
            if (c0 + u < ND && L <= D::kTop) {
              const float w = pow2f(2 - 5 * L);
#pragma unroll
              for (int j = 0; j < W; ++j)
                acc[j] = acc[j] + dd{__uint_as_float(raw[(u * W + j) >> 4][(u * W + j) & 15]) * w, 0.0f};
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce[set]);
        if (half == 1)
#pragma unroll
          for (int j = 0; j < W; ++j) xg[j * 64 + nu] = acc[j];   // consecutive lanes, consecutive words
        named_sync_id(bar_x, 128);
        if (half == 0) {
#pragma unroll
          for (int j = 0; j < W; ++j) {
            if (j >= rp) break;
            dd v = dd_scale(acc[j] + xg[j * 64 + nu], Fc[j]);
            if (s0 > 0) v = v + to_dd(yrow[j]);
            store_as(v, yrow + j);
          }
        }
        named_sync_id(bar_x, 128);
      }
      if (stop) break;
    }
  }
  // tensor memory is released once every role is done
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(kTmemCols) : "memory");
}


// Leaf forward step on the tensor cores (Algorithm 1 at the leaves,
// x^_t = V_t^T x|t, FP64-accurate handles of order 4 with leaves of at most
// 21 triangles and 9 to 16 columns): the blocks are V_t^T (64 rows nu, the leaf's triangles r as
// the contraction index, zero padded to 32 bytes), cut once into the ten
// digit planes of the coupling with a power of two per row,
// Ev[t][nu] = 1 + floor(log2 max_r |V_t[r][nu]|); the coefficients are the
// wide input digit tiles of leaf t that the nearfield reads too (ntc_input).
__global__ void k_tcv_rowexp(const dd *__restrict__ V, int64_t nleaf, int L, int kp, int32_t *__restrict__ Ev) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= nleaf * kTcK) return;
  const int64_t t = e / kTcK;
  const int nu = (int)(e % kTcK);
  float mx = 0.0f;
  for (int r = 0; r < L; ++r) mx = fmaxf(mx, fabsf(V[(t * L + r) * kp + nu].hi));
  Ev[e] = mx > 0.0f ? ilogbf(mx) + 1 : 0;
}

// the ten digit planes of V_t^T, row nu, contraction indices 16 cg .. 16 cg + 15
__global__ void k_tcv_slice(const dd *__restrict__ V, const int32_t *__restrict__ Ev, int64_t nleaf, int L, int kp,
                            unsigned char *__restrict__ Vtc) {
  using D = Dig<kTcSlices, 32>;
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= nleaf * kTcK * 2) return;
  const int64_t t = e / (kTcK * 2);
  const int nu = (int)((e / 2) % kTcK), cg = (int)(e % 2);
  const int sc = kTcFixBits - Ev[t * kTcK + nu];
  __align__(16) unsigned char out[kTcSlices][16];
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int r = 16 * cg + q;
    long long X = 0;
    if (r < L) {
      const dd v = V[(t * L + r) * kp + nu];
      X = llrint(ldexp((double)v.hi + (double)v.lo, sc));
    }
    int sl[kTcSlices];
    split_digits(X, sl);
#pragma unroll
    for (int i = 0; i < kTcSlices; ++i) out[i][q] = e4m3(sl[i]);
  }
  unsigned char *base = Vtc + t * (int64_t)D::kTileA + core_off32(nu, 16 * cg);
#pragma unroll
  for (int i = 0; i < kTcSlices; ++i)
    *reinterpret_cast<uint4 *>(base + i * D::kPlaneA) = *reinterpret_cast<const uint4 *>(out[i]);
}

}  // namespace

// ---------------------------------------------------------------- host side
// CTAs of k_tc_levmax: 8 warps of 4 rows each per pass, at most 8 CTAs per SM
static unsigned levmax_grid(int64_t rows) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((rows + 31) / 32, 152 * 8));
}

// FP64-accurate (ten digits) or FP32-accurate (six digits) coupling of an
// order-4 handle with stored coupling matrices
bool tc_eligible(const Dev &d) {
  return (d.prec == H2_F64 || d.prec == H2_F32) && d.coupling == 0 && d.m == 4 && d.kp == kTcK;
}

namespace {

template <int ND>
int tc_build_nd(Ctx &c) {
  Dev &d = c.d;
  cudaStream_t st = c.stream;
  const int64_t row0 = ((int64_t)1 << d.first_adm_level) - 1;
  int rc;
  SchedTmp tmp;
  if ((rc = row_schedule(d, c.plan.adm_ptr.data() + row0, c.plan.adm_col.data(), d.nclu - row0, d.tc_s, tmp, st)))
    return rc;
  if ((rc = dev_alloc(d, (void **)&d.tc_E, sizeof(int32_t) * (size_t)d.nclu * kTcK))) return rc;
  if ((rc = dev_alloc(d, &d.Stc, (size_t)d.nadm * Dig<ND>::kTileA))) return rc;
  if ((rc = dev_alloc(d, &d.xtc, (size_t)d.nclu * Dig<ND>::kTileB))) return rc;
  if (!d.tc_xmax && (rc = dev_alloc(d, (void **)&d.tc_xmax, sizeof(unsigned) * 32 * kXmaxCols))) return rc;
  H2_CUDA_TRY(cudaMemsetAsync(d.tc_E, 0, sizeof(int32_t) * (size_t)d.nclu * kTcK, st));
  H2_CUDA_TRY(cudaMemsetAsync(d.xtc, 0, (size_t)d.nclu * Dig<ND>::kTileB, st));
  const int64_t nr = (d.nclu - row0) * kTcK;
  k_tc_rowexp<<<(unsigned)((nr + 127) / 128), 128, 0, st>>>(d.adm_ptr, d.adm_col, d.cheb, row0, d.nclu, d.kernel,
                                                             d.tc_E);
  const int64_t ns = d.nadm * kTcK * 4;
  k_tc_slice_s<ND><<<(unsigned)((ns + 255) / 256), 256, 0, st>>>(tmp.brow, d.tc_s.col, row0, d.cheb, d.tc_E, d.nadm,
                                                                 d.kernel, (unsigned char *)d.Stc);
  H2_CUDA_TRY(cudaGetLastError());
  H2_CUDA_TRY(cudaStreamSynchronize(st));
  d.tc_nd = ND;
  d.tc = true;
  return H2_OK;
}

// Upward pass of a product on the tensor-core path: the transfers of
// Algorithm 1, each level's column maxima taken on the way (launch_up; the leaves' by the
// leaf step or k_tc_levmax), then the coefficient digits of
// every far-field level in one launch (k_tc_slice_x, each cluster with its
// level's maxima).  Cutting a level's digits inside the next level's
// transfer launch was slower: the transfer threads are latency bound.
// Returns the launches made.
template <class T, int ND>
int tc_upward_t(Ctx &c, T *xhat, int rp, int64_t *launches, bool leaf_max) {
  Dev &d = c.d;
  cudaStream_t st = c.stream;
  const int D = d.depth, lmin = d.first_adm_level;
  if (lmin > D) return H2_OK;
  const int64_t leaf0 = d.nleaf - 1;
  int64_t nl = 0;
  if (!leaf_max) {
    // FP64-accurate products clear all their maxima at the start
    if (d.prec != H2_F64) H2_CUDA_TRY(cudaMemsetAsync(d.tc_xmax, 0, sizeof(unsigned) * 32 * kXmaxCols, st));
    const int64_t lrows = d.nleaf * kTcK;
    pdl(k_tc_levmax<T>, levmax_grid(lrows), 256, 0, st, xhat + leaf0 * kTcK * rp, lrows, rp, d.tc_xmax + D * kXmaxCols);
    ++nl;
  }
  for (int l = D - 1; l >= lmin; --l) {
    // level l from level l + 1, with the column maxima of level l
    const int64_t np = (int64_t)1 << l;
    launch_up<T, T>((const T *)d.Ef, 4, rp, np - 1, np, xhat, d.tc_xmax + l * kXmaxCols, st);
    ++nl;
  }
  // the digits of every level at once (all maxima are complete)
  const int64_t c0 = ((int64_t)1 << lmin) - 1, ncl = d.nclu - c0;
  if (rp <= 8)
    pdl(k_tc_slice_x<T, ND, 8>, (unsigned)((ncl + 7) / 8), 256, 0, st, xhat, c0, ncl, rp, d.tc_xmax,
        (unsigned char *)d.xtc);
  else
    pdl(k_tc_slice_x<T, ND, kTcN>, (unsigned)((ncl + 3) / 4), 256, 0, st, xhat, c0, ncl, rp, d.tc_xmax,
        (unsigned char *)d.xtc);
  ++nl;
  H2_CUDA_TRY(cudaGetLastError());
  if (launches) *launches = nl;
  return H2_OK;
}

template <class T, int ND, int W>
int tc_coupling_w(Ctx &c, T *yhat, int rp) {
  Dev &d = c.d;
  const int64_t row0 = ((int64_t)1 << d.first_adm_level) - 1, nrows = d.nclu - row0;
  if (nrows <= 0) return H2_OK;
  static_assert(tc_smem<ND, kTcK, W>() <= 227 * 1024, "tensor-core coupling does not fit in shared memory");
  H2_CUDA_TRY(cudaFuncSetAttribute((const void *)k_coupling_tc<ND, T, kTcK, false, W>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(227 * 1024)));
  pdl(k_coupling_tc<ND, T, kTcK, false, W>, d.tc_s.grid, kTcThreads, tc_smem<ND, kTcK, W>(), c.stream,
      (const unsigned char *)d.Stc, (const unsigned char *)d.xtc, d.tc_s.ptr, d.tc_s.col, d.tc_s.row, d.tc_s.split,
      d.tc_E, d.tc_xmax, row0, nrows, rp, yhat, nullptr, Dig<ND, kTcK, W>::kTileB);
  H2_CUDA_TRY(cudaGetLastError());
  return H2_OK;
}

template <class T, int ND>
int tc_coupling_t(Ctx &c, T *yhat, int rp) {
  return rp <= 8 ? tc_coupling_w<T, ND, 8>(c, yhat, rp) : tc_coupling_w<T, ND, kTcN>(c, yhat, rp);
}

}  // namespace

int tc_build(Ctx &c) {
  Dev &d = c.d;
  if (d.first_adm_level > d.depth || d.nadm == 0) return H2_OK;
  return d.prec == H2_F64 ? tc_build_nd<10>(c) : tc_build_nd<6>(c);
}

int tc_upward(Ctx &c, void *xhat, int rp, int64_t *launches, bool leaf_max) {
  if (rp > kTcN) return fail(H2_EINVAL, "the tensor-core coupling takes at most 16 right-hand sides");
  if (c.d.tc_nd == 10) return tc_upward_t<dd, 10>(c, static_cast<dd *>(xhat), rp, launches, leaf_max);
  return tc_upward_t<float, 6>(c, static_cast<float *>(xhat), rp, launches, leaf_max);
}

// the coupling phase: the coefficient digits exist (tc_upward)
int tc_coupling(Ctx &c, const void *xhat, void *yhat, int rp) {
  (void)xhat;
  if (rp > kTcN) return fail(H2_EINVAL, "the tensor-core coupling takes at most 16 right-hand sides");
  if (c.d.tc_nd == 10) return tc_coupling_t<dd, 10>(c, static_cast<dd *>(yhat), rp);
  return tc_coupling_t<float, 6>(c, static_cast<float *>(yhat), rp);
}

// the V_t^T digit planes of the tensor-core leaf forward step, for FP64-accurate
// handles with tensor-core coupling and nearfield and leaves of at most 21 triangles
int tc_leaf_build(Ctx &c) {
  Dev &d = c.d;
  const int L = (int)d.lmax;
  if (!(d.tc && d.tc_nd == kTcSlices && d.k == kTcK && d.kp == kTcK && L <= kLeafTcMax)) return H2_OK;
  using DV = Dig<kTcSlices, 32>;
  int rc;
  if ((rc = dev_alloc(d, (void **)&d.tcv_E, sizeof(int32_t) * (size_t)d.nleaf * kTcK))) return rc;
  if ((rc = dev_alloc(d, &d.Vtc, (size_t)d.nleaf * DV::kTileA))) return rc;
  const int64_t nv = d.nleaf * kTcK;
  k_tcv_rowexp<<<(unsigned)((nv + 127) / 128), 128, 0, c.stream>>>((const dd *)d.V, d.nleaf, L, (int)d.kp, d.tcv_E);
  k_tcv_slice<<<(unsigned)((2 * nv + 255) / 256), 256, 0, c.stream>>>((const dd *)d.V, d.tcv_E, d.nleaf, L,
                                                                      (int)d.kp, (unsigned char *)d.Vtc);
  H2_CUDA_TRY(cudaGetLastError());
  return H2_OK;
}

// the leaf forward step on the tensor cores: x^ of the leaf clusters from the
// input digits (ntc_input) and the stored V_t^T digits, with their column
// maxima for the upward pass
int tc_leaf_forward(Ctx &c, void *xhat_v, int rp) {
  Dev &d = c.d;
  cudaStream_t st = c.stream;
  if (rp > kTcN || !d.Vtc) return fail(H2_EINVAL, "no tensor-core leaf forward step for this handle");
  constexpr int KB = 32;
  constexpr uint32_t sm = tc_smem<kTcSlices, KB>();
  static_assert(sm <= 227 * 1024, "tensor-core leaf step does not fit in shared memory");
  H2_CUDA_TRY(cudaFuncSetAttribute((const void *)k_coupling_tc<kTcSlices, dd, KB, true>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(227 * 1024)));
  int sms = 0, dev = 0;
  H2_CUDA_TRY(cudaGetDevice(&dev));
  H2_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int grid = (int)std::min<int64_t>(sms, d.nleaf);
  // the leaf level's column maxima of the upward pass are taken here (tc_upward with leaf_max)
  pdl(k_coupling_tc<kTcSlices, dd, KB, true>, grid, kTcThreads, sm, st, 
      (const unsigned char *)d.Vtc, (const unsigned char *)d.xnt, nullptr, nullptr, nullptr, nullptr, d.tcv_E, d.ntc_xmax,
      d.nleaf - 1, d.nleaf, rp, static_cast<dd *>(xhat_v), d.tc_xmax + d.depth * kXmaxCols, 32 * 11 * kTcN);
  H2_CUDA_TRY(cudaGetLastError());
  return H2_OK;
}

// the tensor-core path's own device error word (bounded waits of this file)
int tc_take_error(cudaStream_t st) {
  int v = 0, zero = 0;
  H2_CUDA_TRY(cudaMemcpyFromSymbolAsync(&v, g_h2_device_error, sizeof(int), 0, cudaMemcpyDeviceToHost, st));
  H2_CUDA_TRY(cudaStreamSynchronize(st));
  if (v) {
    H2_CUDA_TRY(cudaMemcpyToSymbolAsync(g_h2_device_error, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, st));
    H2_CUDA_TRY(cudaStreamSynchronize(st));
    return fail(H2_ETIMEOUT, "a bounded device wait of the tensor-core coupling ran out");
  }
  return H2_OK;
}

}  // namespace h2
