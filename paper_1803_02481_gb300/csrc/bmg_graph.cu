// The nodes of a recorded graph (GraphRecorder in bmg_internal.h).
#include "bmg_internal.h"

#include <cstring>

namespace bmg {

namespace {
thread_local GraphRecorder* g_recorder = nullptr;
}  // namespace

GraphRecorder* recorder() { return g_recorder; }

GraphRecorder::GraphRecorder(cudaGraph_t graph) : graph_(graph), outer_(g_recorder) { g_recorder = this; }
GraphRecorder::~GraphRecorder() { g_recorder = outer_; }

cudaError_t GraphRecorder::added(cudaGraphNode_t node, cudaError_t e, bool kernel) {
  if (e != cudaSuccess) {
    if (status_ == cudaSuccess) status_ = e;
    return e;
  }
  last_ = node;
  last_kernel_ = kernel;
  return e;
}

cudaError_t GraphRecorder::kernel(const void* func, dim3 grid, dim3 block, size_t smem, void** params,
                                  bool programmatic, unsigned cluster) {
  // zeroed storage: the struct's unions have no default constructor
  alignas(cudaGraphNodeParams) unsigned char raw[sizeof(cudaGraphNodeParams)];
  std::memset(raw, 0, sizeof(raw));
  cudaGraphNodeParams& p = *reinterpret_cast<cudaGraphNodeParams*>(raw);
  p.type = cudaGraphNodeTypeKernel;
  p.kernel.func = const_cast<void*>(func);
  p.kernel.gridDim = grid;
  p.kernel.blockDim = block;
  p.kernel.sharedMemBytes = unsigned(smem);
  p.kernel.kernelParams = params;
  cudaGraphEdgeData edge;
  std::memset(&edge, 0, sizeof(edge));
  if (programmatic && last_kernel_) {
    edge.from_port = cudaGraphKernelNodePortProgrammatic;
    edge.type = cudaGraphDependencyTypeProgrammatic;
  }
  cudaGraphNode_t node = nullptr;
  cudaError_t e = cudaGraphAddNode(&node, graph_, last_ ? &last_ : nullptr, last_ ? &edge : nullptr, last_ ? 1 : 0, &p);
  if (e == cudaSuccess && cluster > 1) {
    cudaLaunchAttributeValue v;
    std::memset(&v, 0, sizeof(v));
    v.clusterDim.x = cluster;
    v.clusterDim.y = v.clusterDim.z = 1;
    e = cudaGraphKernelNodeSetAttribute(node, cudaLaunchAttributeClusterDimension, &v);
  }
  return added(node, e, true);
}

cudaError_t GraphRecorder::copy_to_host(void* dst, const void* src, size_t bytes) {
  cudaGraphNode_t node = nullptr;
  const cudaError_t e = cudaGraphAddMemcpyNode1D(&node, graph_, last_ ? &last_ : nullptr, last_ ? 1 : 0, dst, src,
                                                 bytes, cudaMemcpyDeviceToHost);
  return added(node, e, false);
}

cudaGraph_t GraphRecorder::loop(cudaGraphConditionalHandle handle) {
  alignas(cudaGraphNodeParams) unsigned char raw[sizeof(cudaGraphNodeParams)];
  std::memset(raw, 0, sizeof(raw));
  cudaGraphNodeParams& p = *reinterpret_cast<cudaGraphNodeParams*>(raw);
  p.type = cudaGraphNodeTypeConditional;
  p.conditional.handle = handle;
  p.conditional.type = cudaGraphCondTypeWhile;
  p.conditional.size = 1;
  cudaGraphNode_t node = nullptr;
  const cudaError_t e = cudaGraphAddNode(&node, graph_, last_ ? &last_ : nullptr, nullptr, last_ ? 1 : 0, &p);
  if (added(node, e, false) != cudaSuccess) return nullptr;
  return p.conditional.phGraph_out[0];
}

}  // namespace bmg
