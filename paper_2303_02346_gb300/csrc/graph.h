// Capture of a handle's work into an executable CUDA graph.
#pragma once

#include <cuda_runtime.h>

namespace mpm {

// Captures the work that fn enqueues on `stream` (a capture stream, with nothing
// else on it) and instantiates it into *exec; nullptr on any error, which is
// returned. A launch that is refused need not end the capture: its graph then only
// lacks that kernel, and would replay without it and without an error. So launch
// errors are read before the graph is kept. An error that was pending at entry is
// returned without running fn, and stays pending.
template <class Fn>
cudaError_t capture_graph(cudaStream_t stream, unsigned long long flags, Fn fn, cudaGraphExec_t* exec) {
  *exec = nullptr;
  cudaError_t e = cudaPeekAtLastError();
  if (e != cudaSuccess) return e;
  e = cudaStreamBeginCapture(stream, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e;
  }
  fn(stream);
  const cudaError_t launch = cudaGetLastError();
  cudaGraph_t graph = nullptr;
  e = cudaStreamEndCapture(stream, &graph);
  if (launch != cudaSuccess) e = launch;
  if (e == cudaSuccess && !graph) e = cudaErrorUnknown;
  if (e == cudaSuccess) e = cudaGraphInstantiate(exec, graph, flags);
  if (graph) cudaGraphDestroy(graph);
  if (e != cudaSuccess) {
    *exec = nullptr;
    cudaGetLastError();
  }
  return e;
}

}  // namespace mpm
