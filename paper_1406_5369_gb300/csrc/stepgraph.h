// CUDA graphs of a solve step (one V-cycle and its residual norm) for the
// contexts that solve on a stream of their own: the cell-centred and the
// complex-diffusion ones. A step is some 100 short launches; replaying them
// as one graph takes about 1.3 us each, launching them 2.5 us.
//
// A graph holds the context's buffers, which live as long as the context, and
// is keyed by the live-buffer state it was captured in. The first two steps of
// a context's first solve run without one: short solves never pay for capture. So
// does every step for which none can be made.
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
  // Another thread's capture in the global mode forbids the calls below in threads
  // of that mode, and would be spoilt by them: not so in the thread-local mode.
  struct Mode {
    cudaStreamCaptureMode m = cudaStreamCaptureModeThreadLocal;
    Mode() { cudaThreadExchangeStreamCaptureMode(&m); }
    ~Mode() { cudaThreadExchangeStreamCaptureMode(&m); }
  } mode;
  StepGraphs::Slot &s = g.slot[g.next];
  if ((g.cap || cudaStreamCreateWithFlags(&g.cap, cudaStreamNonBlocking) == cudaSuccess) &&
      cudaStreamBeginCapture(g.cap, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
    g.next = (g.next + 1) & 3;
    if (s.valid) cudaGraphExecDestroy(s.exec);
    s.valid = false;
    const cudaStream_t user = stream;
    stream = g.cap;
    *status = record();
    stream = user;
    s.post = key();
    set_key(now);
    cudaGraph_t graph = nullptr;
    const cudaError_t e = cudaStreamEndCapture(g.cap, &graph);
    s.valid = *status == 0 && e == cudaSuccess && cudaGraphInstantiate(&s.exec, graph, 0) == cudaSuccess;
    s.key = now;
    if (graph) cudaGraphDestroy(graph);
    if (s.valid) {
      const cudaError_t launched = cudaGraphLaunch(s.exec, stream);
      if (launched == cudaSuccess) set_key(s.post);
      return launched;
    }
  }
  // no graph (no memory for one, say): the step's launches themselves
  cudaGetLastError();
  *status = record();
  return cudaSuccess;
}

}  // namespace mg
