// A call of the C ABI as one graph launch (host code; the CUDA runtime calls are the only dependency, so that the paths taken
// when one of them fails are tested with fakes, without a GPU).
#pragma once
#include <cuda_runtime_api.h>

#include "../../include/lp.h"

namespace lp {

// Executable graph of one entry point of a handle.
struct CallGraph {
  cudaGraphExec_t exec = nullptr;
  int direct_calls = 0;            // of the first kDirectCalls
  int rebuilt = 0, kept = 0;       // executable graphs given up; launches since the last one
  bool off = false;
};
// The first calls of a kind are launched directly: a program that makes one or two does not pay for a graph.
constexpr int kDirectCalls = 2;
// A caller that changes the launches of a call (multipliers given or not, another loss) pays for a new executable graph:
// once in a while it is worth it, at every other call it is not.  After kMaxRebuilt of them without kForgiveAfter launches
// of one graph in a row the calls are launched directly.
constexpr int kMaxRebuilt = 4, kForgiveAfter = 16;

// What a handle's calls are recorded with, and how they were made.  A kernel of a graph runs at the priority of the stream it was recorded on, so
// it has the priority of the caller's stream (of the first one that a call is recorded for; calls on streams of another
// priority are launched directly).
struct CallRecorder {
  cudaStream_t stream = nullptr;
  int priority = 0;
  bool failed = false;
  long long launched = 0, built = 0, direct = 0;   // graph launches; executable graphs; calls launched directly
};
inline cudaStream_t capture_stream_for(CallRecorder& c, cudaStream_t st) {
  int priority = 0;
  if (c.failed || cudaStreamGetPriority(st, &priority) != cudaSuccess) { cudaGetLastError(); return nullptr; }
  if (!c.stream) {
    if (cudaStreamCreateWithPriority(&c.stream, cudaStreamNonBlocking, priority) != cudaSuccess) {
      cudaGetLastError();
      c.stream = nullptr;
      c.failed = true;
      return nullptr;
    }
    c.priority = priority;
  }
  return c.priority == priority ? c.stream : nullptr;
}

// Runs `enqueue(stream)` as ONE graph launch on `st`.  A call is some hundred launches of a few microseconds each; made one
// by one, each costs the host 3 to 5 us, so that small networks wait for the host (ResNet-56 on 20 images in three calls:
// 915 us, 362 as graph launches) and large ones lose the overlap of launches across streams.  The call is recorded anew every
// time, with this call's pointers and arguments, on a stream of the handle's own (recording a launch costs a fraction of
// making it), the executable graph of the previous call is updated to the recording, and launched; only its topology and
// memory are kept.  The first two calls of a kind, calls inside a caller's capture, and profiled calls launch
// directly.  `enqueue` changes host state (which gradients are fresh, launch counts) as if its work had been launched:
// `restore` puts that back wherever a recording does not become a launch.
template <typename Enqueue, typename Restore>
int run_as_graph(CallGraph& g, CallRecorder& rec, cudaStream_t st, bool profiled, Enqueue enqueue, Restore restore) {
  const auto direct = [&]() -> int { ++rec.direct; return enqueue(st); };
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) { cudaGetLastError(); return direct(); }
  if (cs != cudaStreamCaptureStatusNone || profiled || g.off) return direct();
  if (g.direct_calls < kDirectCalls) { ++g.direct_calls; return direct(); }
  const cudaStream_t capture = capture_stream_for(rec, st);
  if (!capture) return direct();
  // (relaxed, as lp_graph_begin: a kernel that is launched for the first time may be loaded then)
  if (cudaStreamBeginCapture(capture, cudaStreamCaptureModeRelaxed) != cudaSuccess) {
    cudaGetLastError();
    g.off = true;
    return direct();
  }
  const int rc = enqueue(capture);
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamEndCapture(capture, &graph);
  if (rc != LP_OK && rc != LP_ERR_CUDA) {   // refused (nothing has run): a direct call would be too
    if (graph) cudaGraphDestroy(graph);
    cudaGetLastError();
    restore();
    return rc;
  }
  if (rc == LP_ERR_CUDA) e = cudaErrorUnknown;   // something that a recording does not take, or a real error: direct, below
  if (e == cudaSuccess && g.exec) {
    cudaGraphExecUpdateResultInfo info;
    if (cudaGraphExecUpdate(g.exec, graph, &info) != cudaSuccess) {   // other options than last time: other nodes
      cudaGetLastError();
      cudaGraphExecDestroy(g.exec);
      g.exec = nullptr;
      g.kept = 0;
      g.off = ++g.rebuilt >= kMaxRebuilt;
    } else if (++g.kept >= kForgiveAfter) {
      g.rebuilt = g.kept = 0;
    }
  }
  if (e == cudaSuccess && !g.exec) {
    e = cudaGraphInstantiate(&g.exec, graph, 0);
    if (e == cudaSuccess) ++rec.built;
  }
  if (e == cudaSuccess) e = cudaGraphLaunch(g.exec, st);
  if (graph) cudaGraphDestroy(graph);
  if (e != cudaSuccess) {          // recording does not work here: launch directly from now on
    cudaGetLastError();
    g.off = true;
    restore();
    return direct();
  }
  ++rec.launched;
  return LP_OK;
}

}  // namespace lp
