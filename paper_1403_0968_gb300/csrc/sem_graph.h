// Blocks of solver iterations as CUDA graphs (host code).
#pragma once

#include <cuda_runtime.h>

#include <string>

#include "sem_internal.h"

// The graph of a block of iterations, captured at its first use and kept for the rest of the solve.
struct StepGraph {
  cudaGraphExec_t e = nullptr;
  bool refused = false;  // the capture was refused: launch one by one
  StepGraph() = default;
  StepGraph(const StepGraph &) = delete;
  StepGraph &operator=(const StepGraph &) = delete;
  ~StepGraph() {
    if (e) cudaGraphExecDestroy(e);
  }
};

// Captures what `body` launches and makes it an executable graph.  The legacy default stream cannot be
// captured: its work is captured on a stream of its own and replayed on the default one.
template <typename F>
sem_status capture_graph(cudaStream_t st, cudaGraphExec_t *exec, F body) {
  cudaStream_t cap = st;
  cudaGraph_t g = nullptr;
  sem_status s = SEM_OK;
  cudaError_t ce = st ? cudaSuccess : cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
  if (ce == cudaSuccess) ce = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
  if (ce == cudaSuccess) {
    s = body(cap);
    ce = cudaStreamEndCapture(cap, &g);
  }
  if (!st && cap) cudaStreamDestroy(cap);
  if (s == SEM_OK && ce != cudaSuccess)
    s = sem_fail(SEM_ERR_CUDA, std::string("graph capture: ") + cudaGetErrorString(ce));
  if (s == SEM_OK) {
    ce = cudaGraphInstantiate(exec, g, 0);
    if (ce != cudaSuccess) {
      *exec = nullptr;
      s = sem_fail(SEM_ERR_CUDA, std::string("graph instantiate: ") + cudaGetErrorString(ce));
    }
  }
  if (g) cudaGraphDestroy(g);
  return s;
}

// Launches a block of iterations as one graph.  A refused capture ends a solve on the caller's own stream;
// on the default stream, whose caller never asked for another one, the block is launched one by one instead.
template <typename F>
sem_status replay(cudaStream_t st, StepGraph *g, F body) {
  if (!g->e && !g->refused) {
    const sem_status s = capture_graph(st, &g->e, body);
    if (s != SEM_OK && st) return s;
    if (s != SEM_OK) {
      g->refused = true;
      cudaGetLastError();
    }
  }
  if (g->refused) return body(st);
  const cudaError_t ce = cudaGraphLaunch(g->e, st);
  return ce == cudaSuccess ? SEM_OK : sem_fail(SEM_ERR_CUDA, std::string("graph launch: ") + cudaGetErrorString(ce));
}
