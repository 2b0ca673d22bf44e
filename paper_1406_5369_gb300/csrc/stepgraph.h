// CUDA graphs of a solve step (one V-cycle and its residual norm) for the
// contexts that solve on a stream of their own: the cell-centred and the
// complex-diffusion ones. A step is some 100 short launches; replaying them
// as one graph takes about 1.3 us each, launching them 2.5 us.
//
// A graph holds the context's buffers, which live as long as the context, and
// is keyed by the live-buffer state it was captured in. The first two steps of
// a context's first solve run without one: short solves never pay for capture.
#pragma once

#include <cuda_runtime.h>

namespace mg {

struct StepGraphs {
  struct Slot {
    bool valid;
    unsigned key, post;
    cudaGraphExec_t exec;
  } slot[4];  // two live-buffer states, each with and without polished sweeps
  int next;
  cudaStream_t cap;  // private capture stream, created on first use
};

inline void drop(StepGraphs &g) {
  for (auto &s : g.slot) {
    if (s.valid) cudaGraphExecDestroy(s.exec);
    s.valid = false;
  }
  if (g.cap) cudaStreamDestroy(g.cap);
  g.cap = nullptr;
}

// Step `k` of a solve on `stream`, a reference to the stream that record()
// launches on. key() reads and set_key() sets the live-buffer state; record()
// returns 0 or the caller's status.
template <typename Key, typename SetKey, typename Record>
cudaError_t step(StepGraphs &g, int k, cudaStream_t &stream, Key key, SetKey set_key, Record record, int *status) {
  *status = 0;
  const unsigned now = key();
  for (auto &s : g.slot)
    if (s.valid && s.key == now) {
      const cudaError_t e = cudaGraphLaunch(s.exec, stream);
      if (e == cudaSuccess) set_key(s.post);
      return e;
    }
  if (k < 2) {
    *status = record();
    return cudaSuccess;
  }
  cudaError_t e = cudaSuccess;
  if (!g.cap && (e = cudaStreamCreateWithFlags(&g.cap, cudaStreamNonBlocking)) != cudaSuccess) return e;
  StepGraphs::Slot &s = g.slot[g.next];
  g.next = (g.next + 1) & 3;
  if (s.valid) cudaGraphExecDestroy(s.exec);
  s.valid = false;
  if ((e = cudaStreamBeginCapture(g.cap, cudaStreamCaptureModeThreadLocal)) != cudaSuccess) return e;
  const cudaStream_t user = stream;
  stream = g.cap;
  *status = record();
  stream = user;
  s.post = key();
  set_key(now);
  cudaGraph_t graph = nullptr;
  e = cudaStreamEndCapture(g.cap, &graph);
  if (*status == 0 && e == cudaSuccess && (e = cudaGraphInstantiate(&s.exec, graph, 0)) == cudaSuccess) {
    s.valid = true;
    s.key = now;
  }
  if (graph) cudaGraphDestroy(graph);
  if (!s.valid) return e;
  e = cudaGraphLaunch(s.exec, stream);
  if (e == cudaSuccess) set_key(s.post);
  return e;
}

}  // namespace mg
