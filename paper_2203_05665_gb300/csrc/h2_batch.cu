// Batched H^2 products over independent matrices of uneven sizes (FP32
// storage and arithmetic, stored coupling).
//
// Every block-row phase of the product (leaf forward, coupling, leaf backward,
// nearfield: Algorithms 1-3) runs as ONE launch over the rows of all problems.  Rows differ in shape from problem to problem (rank k =
// m^3 for m = 3 or 4, leaf sizes up to 64, 1 to 16 right-hand sides); a warp
// looks up its row's problem and takes the row as the single-matrix kernel does
// (lane_row, h2_lane.cu): double-buffered pieces in its own shared-memory
// stages, 4 x 8 (4 x 4) register tiles.  Rows of many terms are cut in chunk
// rows whose partial sums are added in order, so that no warp finishes long
// after the others; results are bit-reproducible.
//
// The transfer passes run level-synchronously across problems (up_pair and
// down_pair, h2_transfer.cuh): step s of the upward pass treats level D_p - 1 - s
// of every problem p, step s of the downward pass level lmin_p + s.  The
// permutations in and out are one launch each over the packed vectors of all
// problems.  The whole sequence is captured once in a CUDA graph and replayed.
//
// The warps per CTA and stages per warp of every block-row phase are chosen by
// measurement (h2_batch_tune).
//
// Six problems (20,480 to 130,000 triangles, order 3 and 4, leaves of 64, 1 to 8
// right-hand sides), default launch shapes: 1,124 us per product with a
// persistent kernel of four warps per SM and one output row per lane (coupling
// 416, leaf backward + nearfield 442, transfers 210), 415 us now (136, 183, 68);
// bound by the instructions around pieces of 27 to 64 rows and 4 columns.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "h2_internal.hpp"
#include "h2_lane.cuh"
#include "h2_launch.cuh"
#include "h2_transfer.cuh"

namespace h2 {
namespace {

// One problem's rows in one block-row phase; first: its first row among the phase's
struct BRows {
  LaneRows g;
  LaneShape t;
  int64_t first;
  int tc;                // columns of a register tile
};

// One problem's parents in one transfer step.
struct BTr {
  const float *Ef;
  float *hat;
  int64_t par0, npar;
  int cta0, m, rp, np, pp;   // first CTA of the entry, order, columns, column pairs, parents per CTA
};

// One problem's part of the packed input / output vectors.
struct BPerm {
  const int32_t *pad_src;
  float *pad;
  int64_t n, npad, xoff, e0;
  int nrhs, rp;
};

constexpr int kBatchMaxRows = 64;   // output rows of a tile (k or the leaf size)
constexpr int kBatchMaxRp = 16;     // padded right-hand sides

// The batched block-row kernel (see the top of the file): warp per row, the
// rows of the phase's problems one after the other.
template <int NST>
__global__ void __launch_bounds__(256) k_batch_rows(const BRows *__restrict__ pr, int np, int64_t total,
                                                    uint32_t stage) {
  pdl_wait();
  pdl_go();
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + w;
  if (row >= total) return;
  // the row's problem: the last one that starts at or before it
  int p = -1;
  for (int b = 0; b < np; b += 32)
    p += __popc(__ballot_sync(0xffffffffu, b + lane < np && pr[min(b + lane, np - 1)].first <= row));
  const LaneRows g = pr[p].g;
  const LaneShape t = pr[p].t;
  unsigned char *ring = smem + (size_t)w * NST * stage;
  if (pr[p].tc == 4) lane_row<float, float, 4, 1, NST>(g, t, 1, row - pr[p].first, w, ring, nullptr);
  else lane_row<float, float, 8, 1, NST>(g, t, 1, row - pr[p].first, w, ring, nullptr);
}

// ---------------------------------------------------------------------------
// transfers: CTA per group of parents; CTA b belongs to the last entry that
// starts at or before it
__device__ __forceinline__ int find_entry(const BTr *__restrict__ te, int ne, int b) {
  int lo = 0, hi = ne - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (te[mid].cta0 <= b) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

template <bool UP>
__global__ void __launch_bounds__(512, 3) k_batch_transfer(const BTr *__restrict__ te, int ne) {
  extern __shared__ __align__(16) unsigned char psm[];
  __shared__ unsigned loc[16];
  const BTr t = te[find_entry(te, ne, (int)blockIdx.x)];
  const int bx = (int)blockIdx.x - t.cta0;
  auto go = [&](auto order) {
    constexpr int M = decltype(order)::value;
    if (UP) up_pair<float, float, M>(t.Ef, t.rp, t.np, t.pp, t.par0, t.npar, t.hat, nullptr, bx, 0, psm, loc);
    else down_pair<float, float, M>(t.Ef, t.rp, t.np, t.pp, t.par0, t.npar, t.hat, bx, 0, psm);
  };
  switch (t.m) {
    case 1: return go(std::integral_constant<int, 1>{});
    case 2: return go(std::integral_constant<int, 2>{});
    case 3: return go(std::integral_constant<int, 3>{});
    default: return go(std::integral_constant<int, 4>{});
  }
}

// rows cut in chunks: out (+)= the partial sums of the chunk rows, in chunk order
struct BRed {
  float *out;            // the output row (already holding the first chunk's sum)
  const float *part;     // nch partial rows of len values each
  int nch, len;
};

__global__ void k_batch_reduce(const BRed *__restrict__ rd) {
  pdl_wait();
  pdl_go();
  const BRed &q = rd[blockIdx.x];
  for (int i = threadIdx.x; i < q.len; i += blockDim.x) {
    float v = q.out[i];
    for (int j = 0; j < q.nch; ++j) v += q.part[(int64_t)j * q.len + i];
    q.out[i] = v;
  }
}

// ---------------------------------------------------------------------------
// permutations over the packed vectors: element e of the padded space of all
// problems; each thread walks increasing e, so its problem index only grows
__device__ __forceinline__ int perm_problem(const BPerm *__restrict__ pp, int np, int64_t e) {
  int lo = 0, hi = np - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (pp[mid].e0 <= e) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__global__ void k_batch_permute_in(const BPerm *__restrict__ pp, int np, int64_t total, const float *__restrict__ x) {
  pdl_wait();
  pdl_go();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  int p = perm_problem(pp, np, e);
  for (; e < total; e += stride) {
    while (p + 1 < np && pp[p + 1].e0 <= e) ++p;
    const BPerm &q = pp[p];
    const int64_t l = e - q.e0, i = l / q.rp;
    const int c = (int)(l - i * q.rp);
    const int32_t src = q.pad_src[i];
    q.pad[l] = (src >= 0 && c < q.nrhs) ? x[q.xoff + src + (int64_t)c * q.n] : 0.0f;
  }
}

__global__ void k_batch_permute_out(const BPerm *__restrict__ pp, int np, int64_t total, float *__restrict__ y) {
  pdl_wait();
  pdl_go();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  int p = perm_problem(pp, np, e);
  for (; e < total; e += stride) {
    while (p + 1 < np && pp[p + 1].e0 <= e) ++p;
    const BPerm &q = pp[p];
    const int64_t l = e - q.e0, i = l / q.rp;
    const int c = (int)(l - i * q.rp);
    const int32_t src = q.pad_src[i];
    if (src >= 0 && c < q.nrhs) y[q.xoff + src + (int64_t)c * q.n] = q.pad[l];
  }
}

constexpr int kRowPhases = 4;   // leaf forward, coupling, leaf backward, nearfield
constexpr int64_t kChunkTerms = 24;   // rows with more terms are cut in chunks of this many terms
constexpr int kPermThreads = 256;
constexpr size_t kBatchSmemMax = 227 * 1024;

// launch shapes of the block-row kernel the tuner chooses from
struct Shape {
  int wpb, nst;   // warps per CTA, stages per warp
};
constexpr Shape kShapes[] = {{4, 2}, {8, 2}, {2, 2}, {1, 2}, {4, 3}, {2, 3}, {6, 2}, {6, 3}};
constexpr int kNumShapes = sizeof(kShapes) / sizeof(kShapes[0]);
// the largest stage (a piece of 32 x 64 entries, 16 columns) fits every shape
static_assert(6 * 3 * (32 * 64 * 4 + 32 * 16 * 4 + 16) <= 227 * 1024, "batched block-row stages");

}  // namespace
}  // namespace h2

using namespace h2;

struct h2_batch_s {
  struct Prob {
    h2_ctx *h = nullptr;
    int nrhs = 0, rp = 0;
    int64_t xoff = 0;
    float *xpad = nullptr, *ypad = nullptr, *xhat = nullptr, *yhat = nullptr;
  };
  int device = 0;
  cudaStream_t stream = nullptr;       // launches (NULL: the legacy default stream)
  cudaStream_t cap = nullptr;          // capture stream
  std::vector<Prob> probs;
  int64_t packed = 0;                  // elements of the packed x and y
  int64_t dofs = 0;                    // sum of n nrhs
  void *work = nullptr;                // all work vectors
  int64_t work_bytes = 0;
  // block-row phases
  std::vector<BRows> rows[kRowPhases];
  BRows *d_rows[kRowPhases] = {};
  int64_t total[kRowPhases] = {};      // rows
  uint32_t stage[kRowPhases] = {};     // bytes of the largest stage
  int shape[kRowPhases] = {0, 0, 0, 0};
  // rows cut in chunks (coupling and nearfield): chunk bounds, partial sums, reductions
  int64_t *d_chunks[kRowPhases] = {};
  float *scratch[kRowPhases] = {};
  BRed *d_red[kRowPhases] = {};
  int nred[kRowPhases] = {};
  // transfers: per step, entries (device arrays) and parents
  std::vector<BTr *> d_up, d_down;
  struct Step {
    int entries, ctas, threads;
    size_t smem;
  };
  std::vector<Step> s_up, s_down;
  // permutations
  BPerm *d_perm_in = nullptr, *d_perm_out = nullptr;
  int64_t perm_total = 0;
  // graph
  cudaGraphExec_t exec = nullptr;
  const float *gx = nullptr;
  float *gy = nullptr;
  bool gprof = false;
  // profiling
  bool prof = false;
  cudaEvent_t ev[H2_NPHASE + 1] = {};
  double ms[H2_NPHASE] = {0};
  int64_t launches[H2_NPHASE] = {0};
  int64_t products = 0;
  int64_t graph_launches = 0;          // kernel launches per product
};

namespace h2 {
namespace {

// shapes, row offsets and device copies of a phase's rows
int upload_rows(h2_batch_s &b, int ph) {
  b.total[ph] = 0;
  b.stage[ph] = 0;
  for (BRows &q : b.rows[ph]) {
    q.first = b.total[ph];
    b.total[ph] += q.g.nrows;
    q.t = LaneShape{};
    lane_pieces(q.g, q.t);
    q.tc = lane_columns(q.g.rp, q.t);
    q.t.stage = lane_stage(q.g, sizeof(float), sizeof(float), q.t.xp, 1, &q.t.xoff);
    if (q.g.nrows > 0) b.stage[ph] = std::max(b.stage[ph], q.t.stage);
  }
  if (b.rows[ph].empty()) return H2_OK;
  H2_CUDA_TRY(cudaMemcpy(b.d_rows[ph], b.rows[ph].data(), sizeof(BRows) * b.rows[ph].size(), cudaMemcpyHostToDevice));
  H2_CUDA_TRY(cudaFuncSetAttribute((const void *)k_batch_rows<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kBatchSmemMax));
  H2_CUDA_TRY(cudaFuncSetAttribute((const void *)k_batch_rows<3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kBatchSmemMax));
  return H2_OK;
}

void launch_rows_phase(h2_batch_s &b, int ph, cudaStream_t st) {
  if (b.total[ph] == 0) return;
  const Shape &s = kShapes[b.shape[ph]];
  const unsigned grid = (unsigned)((b.total[ph] + s.wpb - 1) / s.wpb);
  const size_t sm = (size_t)s.wpb * s.nst * b.stage[ph];
  if (s.nst == 2)
    pdl(k_batch_rows<2>, grid, 32 * s.wpb, sm, st, b.d_rows[ph], (int)b.rows[ph].size(), b.total[ph], b.stage[ph]);
  else
    pdl(k_batch_rows<3>, grid, 32 * s.wpb, sm, st, b.d_rows[ph], (int)b.rows[ph].size(), b.total[ph], b.stage[ph]);
}

// enqueue one product on st; returns the number of kernel launches
int64_t enqueue(h2_batch_s &b, const float *x, float *y, cudaStream_t st, bool events) {
  int64_t nl = 0;
  const int np = (int)b.probs.size();
  // inside a capture, external event nodes stay visible to the host (timing)
  auto mark = [&](int ph) {
    if (events) cudaEventRecordWithFlags(b.ev[ph], st, cudaEventRecordExternal);
  };
  const int pgrid = (int)std::max<int64_t>(1, std::min<int64_t>((b.perm_total + kPermThreads - 1) / kPermThreads, 152 * 16));
  mark(H2_PH_PERMUTE_IN);
  pdl(k_batch_permute_in, pgrid, kPermThreads, 0, st, b.d_perm_in, np, b.perm_total, x);
  ++nl;
  mark(H2_PH_LEAF_FORWARD);
  if (b.total[0]) launch_rows_phase(b, 0, st), ++nl;
  mark(H2_PH_UPWARD);
  for (size_t i = 0; i < b.d_up.size(); ++i) {
    pdl(k_batch_transfer<true>, b.s_up[i].ctas, b.s_up[i].threads, b.s_up[i].smem, st, b.d_up[i], b.s_up[i].entries);
    ++nl;
  }
  mark(H2_PH_COUPLING);
  if (b.total[1]) launch_rows_phase(b, 1, st), ++nl;
  if (b.nred[1]) pdl(k_batch_reduce, b.nred[1], 128, 0, st, b.d_red[1]), ++nl;
  mark(H2_PH_DOWNWARD);
  for (size_t i = 0; i < b.d_down.size(); ++i) {
    pdl(k_batch_transfer<false>, b.s_down[i].ctas, b.s_down[i].threads, b.s_down[i].smem, st, b.d_down[i],
                                                                                            b.s_down[i].entries);
    ++nl;
  }
  mark(H2_PH_LEAF_NEAR);
  if (b.total[2]) launch_rows_phase(b, 2, st), ++nl;
  if (b.total[3]) launch_rows_phase(b, 3, st), ++nl;
  if (b.nred[3]) pdl(k_batch_reduce, b.nred[3], 128, 0, st, b.d_red[3]), ++nl;
  mark(H2_PH_PERMUTE_OUT);
  pdl(k_batch_permute_out, pgrid, kPermThreads, 0, st, b.d_perm_out, np, b.perm_total, y);
  ++nl;
  mark(H2_NPHASE);
  return nl;
}

void drop_graph(h2_batch_s &b) {
  if (b.exec) cudaGraphExecDestroy(b.exec);
  b.exec = nullptr;
  b.gx = nullptr;
  b.gy = nullptr;
}

int capture(h2_batch_s &b, const float *x, float *y) {
  drop_graph(b);
  cudaGraph_t g = nullptr;
  H2_CUDA_TRY(cudaStreamBeginCapture(b.cap, cudaStreamCaptureModeThreadLocal));
  b.graph_launches = enqueue(b, x, y, b.cap, b.prof);
  cudaError_t e = cudaStreamEndCapture(b.cap, &g);
  if (e != cudaSuccess) {
    if (g) cudaGraphDestroy(g);
    return cuda_fail(e, "capture of the batched product");
  }
  e = cudaGraphInstantiate(&b.exec, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) {
    b.exec = nullptr;
    return cuda_fail(e, "instantiation of the batched product graph");
  }
  b.gx = x;
  b.gy = y;
  b.gprof = b.prof;
  return H2_OK;
}

void free_batch(h2_batch_s *b) {
  if (!b) return;
  cudaSetDevice(b->device);
  if (b->stream) cudaStreamSynchronize(b->stream);
  else cudaDeviceSynchronize();
  drop_graph(*b);
  for (auto &d : b->d_rows)
    if (d) cudaFree(d);
  for (int ph = 0; ph < kRowPhases; ++ph) {
    if (b->d_chunks[ph]) cudaFree(b->d_chunks[ph]);
    if (b->scratch[ph]) cudaFree(b->scratch[ph]);
    if (b->d_red[ph]) cudaFree(b->d_red[ph]);
  }
  for (auto p : b->d_up) cudaFree(p);
  for (auto p : b->d_down) cudaFree(p);
  if (b->d_perm_in) cudaFree(b->d_perm_in);
  if (b->d_perm_out) cudaFree(b->d_perm_out);
  if (b->work) cudaFree(b->work);
  for (auto e : b->ev)
    if (e) cudaEventDestroy(e);
  if (b->cap) cudaStreamDestroy(b->cap);
  delete b;
}

}  // namespace
}  // namespace h2

extern "C" {

int h2_batch_create(const h2_handle *hs, int nprob, const int *nrhs, void *stream, h2_batch *out) {
  if (!out) return fail(H2_EINVAL, "out is NULL");
  *out = nullptr;
  if (!hs || !nrhs || nprob < 1) return fail(H2_EINVAL, "a batch needs at least one handle and its nrhs");
  for (int p = 0; p < nprob; ++p) {
    const h2_ctx *h = hs[p];
    if (!h) return fail(H2_EINVAL, "NULL handle in the batch");
    if (h->d.prec != H2_F32) return fail(H2_EINVAL, "batched products need H2_F32 handles");
    if (h->d.gca) return fail(H2_EINVAL, "batched products need interpolation handles (not GCA-H^2)");
    if (h->d.coupling != 0) return fail(H2_EINVAL, "batched products need stored coupling matrices");
    if (h->d.k > kBatchMaxRows || h->d.lmax > kBatchMaxRows)
      return fail(H2_EINVAL, "batched products need rank k <= 64 (order <= 4) and leaves of at most 64 triangles");
    if (nrhs[p] < 1 || padded_rhs(nrhs[p], 4) > kBatchMaxRp) return fail(H2_EINVAL, "batched nrhs must be in [1, 16]");
    if (h->device != hs[0]->device) return fail(H2_EINVAL, "all handles of a batch must live on one device");
  }
  h2_batch_s *b = new (std::nothrow) h2_batch_s();
  if (!b) return fail(H2_ENOMEM, "batch");
  b->device = hs[0]->device;
  b->stream = (cudaStream_t)stream;
  auto bail = [&](int rc) {
    free_batch(b);
    return rc;
  };
  cudaError_t ce = cudaSetDevice(b->device);
  if (ce != cudaSuccess) return bail(cuda_fail(ce, "cudaSetDevice"));
  if ((ce = cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking)) != cudaSuccess)
    return bail(cuda_fail(ce, "capture stream"));
  for (auto &e : b->ev)
    if ((ce = cudaEventCreate(&e)) != cudaSuccess) return bail(cuda_fail(ce, "events"));

  // work vectors of every problem in one allocation (256-byte aligned parts)
  b->probs.resize(nprob);
  auto r256 = [](int64_t v) { return (v + 63) / 64 * 64; };   // floats
  int64_t off = 0, xoff = 0;
  std::vector<int64_t> offs(4 * (size_t)nprob);
  for (int p = 0; p < nprob; ++p) {
    auto &P = b->probs[p];
    P.h = hs[p];
    P.nrhs = nrhs[p];
    P.rp = padded_rhs(nrhs[p], 4);
    P.xoff = xoff;
    const Dev &d = P.h->d;
    xoff += d.n * P.nrhs;
    b->dofs += d.n * P.nrhs;
    const int64_t vec = r256(d.npad * P.rp), coef = r256(d.nclu * (int64_t)d.k * P.rp);
    offs[4 * p] = off;
    offs[4 * p + 1] = off + vec;
    offs[4 * p + 2] = off + 2 * vec;
    offs[4 * p + 3] = off + 2 * vec + coef;
    off += 2 * vec + 2 * coef;
  }
  b->packed = xoff;
  b->work_bytes = off * 4;
  if ((ce = dmalloc(&b->work, (size_t)b->work_bytes)) != cudaSuccess)
    return bail(cuda_fail(ce, "batched work vectors"));
  if ((ce = cudaMemset(b->work, 0, (size_t)b->work_bytes)) != cudaSuccess) return bail(cuda_fail(ce, "memset"));
  float *wf = static_cast<float *>(b->work);
  for (int p = 0; p < nprob; ++p) {
    auto &P = b->probs[p];
    P.xpad = wf + offs[4 * p];
    P.ypad = wf + offs[4 * p + 1];
    P.xhat = wf + offs[4 * p + 2];
    P.yhat = wf + offs[4 * p + 3];
  }

  // block-row phases
  for (int ph = 0; ph < kRowPhases; ++ph) b->rows[ph].resize(nprob);
  int max_steps = 0;
  for (int p = 0; p < nprob; ++p) {
    const auto &P = b->probs[p];
    const Dev &d = P.h->d;
    const int k = d.k, kp = d.kp, L = (int)d.lmax, Lp = (int)d.lp, rp = P.rp;
    const bool far = d.first_adm_level <= d.depth;
    const int64_t leaf0 = d.nleaf - 1, row0 = ((int64_t)1 << d.first_adm_level) - 1;
    LaneRows &fw = b->rows[0][p].g;
    fw.A = d.V;
    fw.X = P.xpad;
    fw.out = P.xhat + leaf0 * k * rp;
    fw.nrows = far ? d.nleaf : 0;
    fw.M = k, fw.Mp = kp, fw.K = L, fw.rp = rp;
    LaneRows &cp = b->rows[1][p].g;
    cp.A = d.S;
    cp.X = P.xhat;
    cp.ptr = d.adm_ptr + row0;
    cp.col = d.adm_col;
    cp.out = P.yhat + row0 * k * rp;
    cp.nrows = far ? d.nclu - row0 : 0;
    cp.M = k, cp.Mp = kp, cp.K = k, cp.rp = rp;
    LaneRows &bw = b->rows[2][p].g;
    bw.A = d.Vt;
    bw.X = P.yhat + leaf0 * k * rp;
    bw.out = P.ypad;
    bw.nrows = far ? d.nleaf : 0;
    bw.M = L, bw.Mp = Lp, bw.K = k, bw.rp = rp;
    LaneRows &nr = b->rows[3][p].g;
    nr.A = d.near;
    nr.X = P.xpad;
    nr.ptr = d.near_ptr;
    nr.col = d.near_col;
    nr.accumulate = far ? 1 : 0;
    nr.out = P.ypad;
    nr.nrows = d.nleaf;
    nr.M = L, nr.Mp = Lp, nr.K = L, nr.rp = rp;
    if (far) max_steps = std::max(max_steps, d.depth - d.first_adm_level);
  }

  // rows of the coupling and the nearfield with more than kChunkTerms terms
  // (cube surfaces produce clusters with hundreds of blocks): the row keeps
  // its first kChunkTerms terms, the rest become chunk rows of their own that
  // write partial sums, added to the row afterwards in chunk order
  for (int ph : {1, 3}) {
    std::vector<int64_t> cb, ce_;
    std::vector<BRed> red;
    std::vector<LaneRows> extra;
    for (int p = 0; p < nprob; ++p) {
      LaneRows &q = b->rows[ph][p].g;
      if (q.nrows == 0) continue;
      const Plan &pl = b->probs[p].h->plan;
      const int64_t *hp = ph == 1 ? pl.adm_ptr.data() + (((int64_t)1 << pl.first_adm_level) - 1) : pl.near_ptr.data();
      LaneRows x = q;
      x.nrows = 0;
      const int64_t first_chunk = (int64_t)cb.size();
      for (int64_t r = 0; r < q.nrows; ++r) {
        const int64_t nt = hp[r + 1] - hp[r];
        if (nt <= kChunkTerms) continue;
        const int64_t nch = (nt - 1) / kChunkTerms;   // chunks beyond the first
        BRed rd{};
        rd.out = q.out + r * q.M * q.rp;
        rd.part = nullptr;   // set once the partial rows are allocated
        rd.nch = (int)nch;
        rd.len = q.M * q.rp;
        red.push_back(rd);
        for (int64_t j = 1; j <= nch; ++j) {
          cb.push_back(hp[r] + j * kChunkTerms);
          ce_.push_back(std::min(hp[r + 1], hp[r] + (j + 1) * kChunkTerms));
        }
        x.nrows += nch;
      }
      if (x.nrows == 0) continue;
      q.cap = kChunkTerms;
      x.ptr = reinterpret_cast<const int64_t *>(first_chunk);   // rebased below
      x.accumulate = 0;
      x.cap = kChunkTerms;
      extra.push_back(x);
    }
    if (extra.empty()) continue;
    // partial rows: float offsets of every extra entry (rows of M rp values)
    int64_t floats = 0;
    std::vector<int64_t> fl_off(extra.size());
    for (size_t i = 0; i < extra.size(); ++i) {
      fl_off[i] = floats;
      floats += extra[i].nrows * extra[i].M * extra[i].rp;
    }
    const size_t nc = cb.size();
    if ((ce = dmalloc((void **)&b->d_chunks[ph], 2 * nc * sizeof(int64_t))) != cudaSuccess ||
        (ce = dmalloc((void **)&b->scratch[ph], (size_t)floats * sizeof(float))) != cudaSuccess ||
        (ce = dmalloc((void **)&b->d_red[ph], red.size() * sizeof(BRed))) != cudaSuccess)
      return bail(cuda_fail(ce, "chunk rows"));
    std::vector<int64_t> both(cb);
    both.insert(both.end(), ce_.begin(), ce_.end());
    if ((ce = cudaMemcpy(b->d_chunks[ph], both.data(), both.size() * sizeof(int64_t), cudaMemcpyHostToDevice)) !=
        cudaSuccess)
      return bail(cuda_fail(ce, "chunk rows"));
    // rebase: chunk bounds and partial rows of each extra entry
    size_t ri = 0;
    for (size_t i = 0; i < extra.size(); ++i) {
      LaneRows &x = extra[i];
      const int64_t c0 = reinterpret_cast<int64_t>(x.ptr);
      x.ptr = b->d_chunks[ph] + c0;
      x.pend = b->d_chunks[ph] + nc + c0;
      x.out = b->scratch[ph] + fl_off[i];
      // the reductions of this entry's rows, in row order
      int64_t row_in_entry = 0;
      while (ri < red.size() && row_in_entry < x.nrows) {
        red[ri].part = x.out + row_in_entry * x.M * x.rp;
        row_in_entry += red[ri].nch;
        ++ri;
      }
      BRows br{};
      br.g = x;
      b->rows[ph].push_back(br);
    }
    if ((ce = cudaMemcpy(b->d_red[ph], red.data(), red.size() * sizeof(BRed), cudaMemcpyHostToDevice)) != cudaSuccess)
      return bail(cuda_fail(ce, "chunk reductions"));
    b->nred[ph] = (int)red.size();
  }
  for (int ph = 0; ph < kRowPhases; ++ph) {
    if ((ce = dmalloc((void **)&b->d_rows[ph], sizeof(BRows) * b->rows[ph].size())) != cudaSuccess)
      return bail(cuda_fail(ce, "batch descriptors"));
    int rc = upload_rows(*b, ph);
    if (rc) return bail(rc);
  }

  // transfer steps
  for (int up = 0; up < 2; ++up) {
    for (int s = 0; s < max_steps; ++s) {
      std::vector<BTr> ent;
      h2_batch_s::Step step{0, 0, 32, 0};
      for (int p = 0; p < nprob; ++p) {
        const auto &P = b->probs[p];
        const Dev &d = P.h->d;
        if (d.first_adm_level > d.depth || s >= d.depth - d.first_adm_level) continue;
        const int l = up ? d.depth - 1 - s : d.first_adm_level + s;   // parent level
        BTr t{};
        t.Ef = (const float *)d.Ef;
        t.hat = up ? P.xhat : P.yhat;
        t.npar = (int64_t)1 << l;
        t.par0 = t.npar - 1;
        t.cta0 = step.ctas;
        t.m = d.m;
        t.rp = P.rp;
        t.np = P.rp / 2;
        t.pp = pair_parents(d.m, t.npar, t.np);
        ent.push_back(t);
        step.ctas += (int)((t.npar + t.pp - 1) / t.pp);
        step.threads = std::max(step.threads, (t.pp * d.k * t.np + 31) / 32 * 32);
        step.smem = std::max(step.smem, pair_smem<float>(d.m, t.np, t.pp, !up));
      }
      step.entries = (int)ent.size();
      BTr *dp = nullptr;
      if ((ce = dmalloc((void **)&dp, sizeof(BTr) * ent.size())) != cudaSuccess)
        return bail(cuda_fail(ce, "transfer descriptors"));
      (up ? b->d_up : b->d_down).push_back(dp);
      if ((ce = cudaMemcpy(dp, ent.data(), sizeof(BTr) * ent.size(), cudaMemcpyHostToDevice)) != cudaSuccess)
        return bail(cuda_fail(ce, "transfer descriptors"));
      (up ? b->s_up : b->s_down).push_back(step);
    }
  }
  // permutations
  std::vector<BPerm> pin(nprob), pout(nprob);
  int64_t e0 = 0;
  for (int p = 0; p < nprob; ++p) {
    const auto &P = b->probs[p];
    const Dev &d = P.h->d;
    BPerm q{d.pad_src, P.xpad, d.n, d.npad, P.xoff, e0, P.nrhs, P.rp};
    pin[p] = q;
    q.pad = P.ypad;
    pout[p] = q;
    e0 += d.npad * P.rp;
  }
  b->perm_total = e0;
  if ((ce = dmalloc((void **)&b->d_perm_in, sizeof(BPerm) * nprob)) != cudaSuccess ||
      (ce = dmalloc((void **)&b->d_perm_out, sizeof(BPerm) * nprob)) != cudaSuccess)
    return bail(cuda_fail(ce, "permutation descriptors"));
  if ((ce = cudaMemcpy(b->d_perm_in, pin.data(), sizeof(BPerm) * nprob, cudaMemcpyHostToDevice)) != cudaSuccess ||
      (ce = cudaMemcpy(b->d_perm_out, pout.data(), sizeof(BPerm) * nprob, cudaMemcpyHostToDevice)) != cudaSuccess)
    return bail(cuda_fail(ce, "permutation descriptors"));
  *out = b;
  return H2_OK;
}

int h2_batch_offsets(h2_batch b, int64_t *offsets) {
  if (!b || !offsets) return fail(H2_EINVAL, "NULL argument");
  for (size_t p = 0; p < b->probs.size(); ++p) offsets[p] = b->probs[p].xoff;
  offsets[b->probs.size()] = b->packed;
  return H2_OK;
}

int h2_batch_matvec(h2_batch b, const float *x, float *y) {
  if (!b || !x || !y) return fail(H2_EINVAL, "NULL argument");
  H2_CUDA_TRY(cudaSetDevice(b->device));
  if (!b->exec || b->gx != x || b->gy != y || b->gprof != b->prof) {
    int rc = capture(*b, x, y);
    if (rc) return rc;
  }
  H2_CUDA_TRY(cudaGraphLaunch(b->exec, b->stream));
  if (b->prof) {
    H2_CUDA_TRY(cudaEventSynchronize(b->ev[H2_NPHASE]));
    for (int i = 0; i < H2_NPHASE; ++i) {
      float t = 0;
      H2_CUDA_TRY(cudaEventElapsedTime(&t, b->ev[i], b->ev[i + 1]));
      b->ms[i] += t;
    }
    b->products++;
  }
  return H2_OK;
}

int h2_batch_tune(h2_batch b, int reps, int *choice) {
  if (!b) return fail(H2_EINVAL, "NULL batch");
  if (reps < 1) reps = 3;
  H2_CUDA_TRY(cudaSetDevice(b->device));
  H2_CUDA_TRY(cudaStreamSynchronize(b->stream));
  drop_graph(*b);
  // the kernels of one phase only read their inputs and (over)write their
  // outputs, so a phase can be launched on its own repeatedly; the work
  // vectors hold whatever the last product left
  cudaEvent_t t0, t1;
  H2_CUDA_TRY(cudaEventCreate(&t0));
  H2_CUDA_TRY(cudaEventCreate(&t1));
  int rc = H2_OK;
  for (int ph = 0; ph < kRowPhases && !rc; ++ph) {
    if (b->total[ph] == 0) continue;
    int best = b->shape[ph];
    float best_ms = 1e30f;
    for (int s = 0; s < kNumShapes && !rc; ++s) {
      b->shape[ph] = s;
      launch_rows_phase(*b, ph, b->cap);   // warm-up
      cudaEventRecord(t0, b->cap);
      for (int i = 0; i < reps; ++i) launch_rows_phase(*b, ph, b->cap);
      cudaEventRecord(t1, b->cap);
      cudaError_t e = cudaEventSynchronize(t1);
      if (e != cudaSuccess) {
        rc = cuda_fail(e, "tuning run");
        break;
      }
      float ms = 0;
      cudaEventElapsedTime(&ms, t0, t1);
      if (ms < best_ms) {
        best_ms = ms;
        best = s;
      }
    }
    b->shape[ph] = best;
    // a phase that accumulates was run repeatedly: the next product rewrites it
  }
  cudaEventDestroy(t0);
  cudaEventDestroy(t1);
  if (rc) return rc;
  if (choice)
    for (int ph = 0; ph < kRowPhases; ++ph) choice[ph] = b->shape[ph];
  return H2_OK;
}

int h2_batch_set_shapes(h2_batch b, const int *choice) {
  if (!b || !choice) return fail(H2_EINVAL, "NULL argument");
  for (int ph = 0; ph < kRowPhases; ++ph)
    if (choice[ph] < 0 || choice[ph] >= kNumShapes)
      return fail(H2_EINVAL, "unknown launch shape");
  H2_CUDA_TRY(cudaSetDevice(b->device));
  H2_CUDA_TRY(cudaStreamSynchronize(b->stream));
  drop_graph(*b);
  for (int ph = 0; ph < kRowPhases; ++ph) {
    b->shape[ph] = choice[ph];
  }
  return H2_OK;
}

int h2_batch_profile(h2_batch b, int enable) {
  if (!b) return fail(H2_EINVAL, "NULL batch");
  b->prof = enable != 0;
  for (double &v : b->ms) v = 0.0;
  b->products = 0;
  return H2_OK;
}

int h2_batch_phase_times(h2_batch b, double *ms, int64_t *launches, int64_t *products) {
  if (!b) return fail(H2_EINVAL, "NULL batch");
  H2_CUDA_TRY(cudaSetDevice(b->device));
  H2_CUDA_TRY(cudaStreamSynchronize(b->stream));
  if (ms)
    for (int i = 0; i < H2_NPHASE; ++i) ms[i] = b->ms[i];
  if (launches) {
    launches[H2_PH_PERMUTE_IN] = 1;
    launches[H2_PH_LEAF_FORWARD] = b->total[0] ? 1 : 0;
    launches[H2_PH_UPWARD] = (int64_t)b->d_up.size();
    launches[H2_PH_COUPLING] = (b->total[1] ? 1 : 0) + (b->nred[1] ? 1 : 0);
    launches[H2_PH_DOWNWARD] = (int64_t)b->d_down.size();
    launches[H2_PH_LEAF_NEAR] = (b->total[2] ? 1 : 0) + (b->total[3] ? 1 : 0) + (b->nred[3] ? 1 : 0);
    launches[H2_PH_PERMUTE_OUT] = 1;
  }
  if (products) *products = b->products;
  return H2_OK;
}

int h2_batch_info(h2_batch b, int64_t *info) {
  if (!b || !info) return fail(H2_EINVAL, "NULL argument");
  info[0] = (int64_t)b->probs.size();
  info[1] = b->packed;
  info[2] = b->dofs;
  info[3] = b->work_bytes;
  int64_t nl = 2 + (int64_t)b->d_up.size() + (int64_t)b->d_down.size();
  for (int ph = 0; ph < kRowPhases; ++ph) nl += (b->total[ph] ? 1 : 0) + (b->nred[ph] ? 1 : 0);
  info[4] = nl;
  for (int ph = 0; ph < kRowPhases; ++ph) info[5 + ph] = b->shape[ph];
  return H2_OK;
}

int h2_batch_sync(h2_batch b) {
  if (!b) return fail(H2_EINVAL, "NULL batch");
  H2_CUDA_TRY(cudaSetDevice(b->device));
  H2_CUDA_TRY(cudaStreamSynchronize(b->stream));
  return H2_OK;
}

int h2_batch_destroy(h2_batch b) {
  free_batch(b);
  return H2_OK;
}

}  // extern "C"
