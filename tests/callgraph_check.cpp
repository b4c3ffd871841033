// Host check of the call graphs' bookkeeping (paper_2203_05665_gb300/csrc/h2_callgraph.hpp)
// with failing driver calls.  Exit status 0 on success.
#include <cstdio>
#include <map>
#include <new>

#include "h2_callgraph.hpp"

using h2::CallGraph;

static int bad = 0;
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); ++bad; } } while (0)

// nodes 1 and 2 read x, node 3 writes y; a call whose n-th exchange fails leaves some of
// them on the old vectors
static void aim_after_failure(int failing) {
  CallGraph g;
  std::map<cudaGraphNode_t, const void *> at;
  double v[4];
  const void *x0 = &v[0], *x1 = &v[1];
  void *y0 = &v[2], *y1 = &v[3];
  for (uintptr_t i = 1; i <= 3; ++i) {
    const cudaGraphNode_t n = reinterpret_cast<cudaGraphNode_t>(i);
    g.nodes.push_back({n, 0, 1, i == 3});
    at[n] = i == 3 ? y0 : x0;
  }
  g.x = x0;
  g.y = y0;
  int count = 0;
  const void *x = nullptr;
  void *y = nullptr;
  auto set = [&](const CallGraph::Node &nd) {
    if (++count == failing) return cudaErrorInvalidValue;
    at[nd.node] = nd.out ? y : x;
    return cudaSuccess;
  };
  auto aim = [&](const void *nx, void *ny) {
    x = nx;
    y = ny;
    return h2::aim_nodes(g, nx, ny, set);
  };
  auto aimed = [&] {
    bool ok = true;
    for (const CallGraph::Node &nd : g.nodes) ok = ok && at[nd.node] == (nd.out ? y : x);
    return ok;
  };
  CHECK(aim(x0, y0) == cudaSuccess && count == 0 && aimed());   // nothing to exchange
  CHECK(aim(x1, y1) == cudaErrorInvalidValue);
  CHECK(aim(x0, y0) == cudaSuccess && aimed());                 // the vectors of before
  CHECK(aim(x0, y1) == cudaSuccess && aimed());
  const int before = count;
  CHECK(aim(x0, y1) == cudaSuccess && count == before);
}

// a product that throws while its stream is replaced
static void stream_after_throw() {
  cudaStream_t own = reinterpret_cast<cudaStream_t>(uintptr_t(8)), cap = reinterpret_cast<cudaStream_t>(uintptr_t(16));
  cudaStream_t stream = own;
  CHECK(!h2::run_on(stream, cap, [&]() -> bool { throw std::bad_alloc(); }) && stream == own);
  CHECK(!h2::run_on(stream, cap, [&] { return stream != cap; }) && stream == own);
  CHECK(h2::run_on(stream, cap, [&] { return stream == cap; }) && stream == own);
}

static void first(const float *, int, double *) {}
static void last(const float *, int, int, double *) {}

int main() {
  const h2::VectorKernel in = h2::reads_x(first), out = h2::writes_y(last);
  CHECK(!in.out && in.arg == 0 && in.count == 3 && in.kernel == reinterpret_cast<const void *>(first));
  CHECK(out.out && out.arg == 3 && out.count == 4 && out.kernel == reinterpret_cast<const void *>(last));
  stream_after_throw();
  for (int failing = 1; failing <= 3; ++failing) aim_after_failure(failing);
  return bad != 0;
}
