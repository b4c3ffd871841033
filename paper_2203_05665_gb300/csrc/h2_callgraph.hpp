// Products captured as CUDA graphs for repeated calls (run_matvec, h2_matvec.cu):
// what is kept and how a kept graph is pointed at a call's vectors.  The driver calls
// come in as functions, so that their failures can be played on the host.
#pragma once

#include <cuda_runtime_api.h>

#include <cstdint>
#include <tuple>
#include <type_traits>
#include <vector>

namespace h2 {

// A product with a given number of right-hand sides: only the nodes that read x or
// write y change from call to call
struct CallGraph {
  struct Node {
    cudaGraphNode_t node;
    int arg, count;               // index of the x or y parameter, number of parameters
    bool out;
  };
  int nrhs = 0;
  bool io64 = false, acc = false;
  int64_t work_gen = -1;          // work buffers the capture refers to
  uint64_t used = 0;              // call count of the last use
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr; // NULL until the second call
  const void *x = nullptr;        // the vectors that every node points at; NULL: not all the same
  void *y = nullptr;
  std::vector<Node> nodes;
};
constexpr int kMaxCallGraphs = 4;

// How a kernel's node is pointed at a vector, from the kernel's own signature: x is the
// first parameter of those that read it, y the last of those that write it.
struct VectorKernel {
  const void *kernel;
  int arg, count;
  bool out;
};
constexpr int kMaxParams = 16;
template <class T, class... P>
VectorKernel reads_x(void (*kernel)(const T *, P...)) {
  static_assert(sizeof...(P) < kMaxParams, "parameters");
  return {reinterpret_cast<const void *>(kernel), 0, 1 + (int)sizeof...(P), false};
}
template <class... P>
VectorKernel writes_y(void (*kernel)(P...)) {
  using Last = std::tuple_element_t<sizeof...(P) - 1, std::tuple<P...>>;
  static_assert(sizeof...(P) <= kMaxParams, "parameters");
  static_assert(std::is_pointer<Last>::value && !std::is_const<std::remove_pointer_t<Last>>::value, "y comes last");
  return {reinterpret_cast<const void *>(kernel), (int)sizeof...(P) - 1, (int)sizeof...(P), true};
}

// Point the graph's nodes at this call's x and y: set(node) exchanges a node's
// parameter.  After a failure some nodes point at the new vectors and some at the
// old: neither is recorded, so that the next call sets every node.
template <class Set>
cudaError_t aim_nodes(CallGraph &g, const void *x, void *y, Set set) {
  const void *ox = g.x;
  void *oy = g.y;
  g.x = nullptr;
  g.y = nullptr;
  for (const CallGraph::Node &nd : g.nodes) {
    if (nd.out ? y == oy : x == ox) continue;
    const cudaError_t e = set(nd);
    if (e != cudaSuccess) return e;
  }
  g.x = x;
  g.y = y;
  return cudaSuccess;
}

// Run body with the handle's stream replaced by cap and put it back however body ends;
// false where it failed or threw (an error message that could not be allocated), so that
// the caller ends the capture on cap in any case.
template <class Body>
bool run_on(cudaStream_t &stream, cudaStream_t cap, Body body) {
  const cudaStream_t own = stream;
  stream = cap;
  bool ok = false;
  try {
    ok = body();
  } catch (...) {
  }
  stream = own;
  return ok;
}

}  // namespace h2
