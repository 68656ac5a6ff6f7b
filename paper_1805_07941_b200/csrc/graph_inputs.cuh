// The kernels of a captured CUDA graph that read the network's float input, so that a replay can read another
// buffer of the same shape in place: the graph's node is given the new pointer instead of the input being copied
// to a fixed address first (that copy reads and writes the whole float batch: 51 us of a 961 us MobileNet step at
// batch 256, 28 us of 497 us on the inception blocks).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <memory>
#include <tuple>
#include <utility>
#include <vector>

namespace qc {

// One kernel node whose first argument points into the input.
struct GraphInputNode {
  cudaGraphNode_t node = nullptr;
  size_t offset = 0;                       // bytes from the start of the input
  virtual ~GraphInputNode() = default;
  virtual cudaError_t set(cudaGraphExec_t exec, const void* input) = 0;
};

template <typename First, typename... Rest>
struct GraphInputNodeOf final : GraphInputNode {
  void (*kernel)(First, Rest...);
  dim3 grid, block;
  size_t smem;
  std::tuple<First, Rest...> args;
  GraphInputNodeOf(void (*k)(First, Rest...), dim3 g, dim3 b, size_t s, First first, Rest... rest)
      : kernel(k), grid(g), block(b), smem(s), args(first, rest...) {}
  cudaError_t set(cudaGraphExec_t exec, const void* input) override {
    std::get<0>(args) = reinterpret_cast<First>(static_cast<const char*>(input) + offset);
    return apply(exec, std::index_sequence_for<First, Rest...>{});
  }

 private:
  template <size_t... I>
  cudaError_t apply(cudaGraphExec_t exec, std::index_sequence<I...>) {
    void* ptrs[] = {static_cast<void*>(&std::get<I>(args))...};
    cudaKernelNodeParams p = {};
    p.func = reinterpret_cast<void*>(kernel);
    p.gridDim = grid;
    p.blockDim = block;
    p.sharedMemBytes = static_cast<unsigned int>(smem);
    p.kernelParams = ptrs;
    return cudaGraphExecKernelNodeSetParams(exec, node, &p);
  }
};

// What the calling thread is recording (between qgraph_record_begin and qgraph_record_end).
struct GraphInputRecord {
  const char* base = nullptr;
  size_t bytes = 0;
  bool complete = true;                    // false: a reader of the input could not be noted
  std::vector<std::unique_ptr<GraphInputNode>> nodes;
};

// Notes the kernel that the calling thread has just launched on `st` if that stream is being captured and the
// kernel's input lies in the recorded range.
template <typename First, typename... Rest>
void note_graph_input(GraphInputRecord* rec, cudaStream_t st, void (*kernel)(First, Rest...), dim3 grid, dim3 block,
                      size_t smem, First first, Rest... rest) {
  if (!rec) return;
  const char* p = reinterpret_cast<const char*>(first);
  if (p < rec->base || p >= rec->base + rec->bytes) return;
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  const cudaGraphNode_t* deps = nullptr;
  const cudaGraphEdgeData* edges = nullptr;
  size_t n = 0;
  if (cudaStreamGetCaptureInfo_v3(st, &status, nullptr, nullptr, &deps, &edges, &n) != cudaSuccess) {
    cudaGetLastError();
    rec->complete = false;
    return;
  }
  if (status != cudaStreamCaptureStatusActive) return;
  if (n != 1) {                            // right after a launch the stream depends on that launch alone
    rec->complete = false;
    return;
  }
  auto node = std::make_unique<GraphInputNodeOf<First, Rest...>>(kernel, grid, block, smem, first, rest...);
  node->node = deps[0];
  node->offset = static_cast<size_t>(p - rec->base);
  rec->nodes.push_back(std::move(node));
}

}  // namespace qc
