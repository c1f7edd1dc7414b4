"""Calls of the C ABI as graph launches (csrc/call_graph.h) against a fake CUDA runtime: what happens where a step of the
recording fails.  Compiled with g++; needs no GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2112_05387_b200", "csrc")

FAKE_RUNTIME = """
#pragma once
typedef int cudaError_t;
enum { cudaSuccess = 0, cudaErrorFake = 1, cudaErrorUnknown = 999 };
typedef struct FakeStream* cudaStream_t;
typedef struct FakeGraph* cudaGraph_t;
typedef struct FakeExec* cudaGraphExec_t;
enum cudaStreamCaptureStatus { cudaStreamCaptureStatusNone = 0, cudaStreamCaptureStatusActive = 1 };
enum cudaStreamCaptureMode { cudaStreamCaptureModeGlobal, cudaStreamCaptureModeThreadLocal, cudaStreamCaptureModeRelaxed };
struct cudaGraphExecUpdateResultInfo { int result; };
struct FakeStream { bool capturing = false, invalid = false; int recorded = 0, topology = 0, priority = 0; };
struct FakeGraph { int nodes, topology; };
struct FakeExec { int nodes, topology; };
// how often each call has been made, and which of them fail from now on
struct Fake { int begin, end, update, instantiate, launch, live_graphs, live_execs, live_streams, launched_nodes; bool fail_begin, fail_end, fail_instantiate, fail_launch, fail_stream; cudaStreamCaptureMode mode; };
extern Fake fake;

inline cudaError_t cudaGetLastError() { return cudaSuccess; }
inline cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* c) {
  *c = s->capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
enum { cudaStreamNonBlocking = 1 };
inline cudaError_t cudaStreamGetPriority(cudaStream_t s, int* p) { *p = s->priority; return cudaSuccess; }
inline cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int p) {
  if (fake.fail_stream) return cudaErrorFake;
  *s = new FakeStream; (*s)->priority = p;
  ++fake.live_streams;
  return cudaSuccess;
}
inline cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode m) {
  ++fake.begin; fake.mode = m;
  if (fake.fail_begin) return cudaErrorFake;
  s->capturing = true; s->invalid = false; s->recorded = 0;
  return cudaSuccess;
}
inline cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
  ++fake.end;
  s->capturing = false;
  *g = nullptr;
  if (fake.fail_end || s->invalid) return cudaErrorFake;
  *g = new FakeGraph{s->recorded, s->topology};
  ++fake.live_graphs;
  return cudaSuccess;
}
inline cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete g; --fake.live_graphs; return cudaSuccess; }
inline cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { delete e; --fake.live_execs; return cudaSuccess; }
inline cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
  ++fake.instantiate;
  if (fake.fail_instantiate) return cudaErrorFake;
  *e = new FakeExec{g->nodes, g->topology};
  ++fake.live_execs;
  return cudaSuccess;
}
inline cudaError_t cudaGraphExecUpdate(cudaGraphExec_t e, cudaGraph_t g, cudaGraphExecUpdateResultInfo*) {
  ++fake.update;
  if (e->topology != g->topology) return cudaErrorFake;
  e->nodes = g->nodes;
  return cudaSuccess;
}
inline cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
  ++fake.launch;
  if (fake.fail_launch) return cudaErrorFake;
  fake.launched_nodes += e->nodes;
  return cudaSuccess;
}
"""

PRELUDE = """
#include <cstdio>
#include <cstdlib>
#include "call_graph.h"
Fake fake = {};
using namespace lp;
// A handle's host state and a call that changes it: five launches and a flag.
struct Handle {
  CallGraph g;
  CallRecorder capture;
  FakeStream user;
  bool fresh = false;
  int launches = 0, done = 0;      // launches counted; launched directly
  int topology = 0, rc = LP_OK, rc_recording = LP_OK;
  bool profiled = false;
  int recorded_priority = 99;
  int call() {
    const bool f = fresh; const int l = launches;
    return run_as_graph(g, capture, &user, profiled, [&](cudaStream_t s) -> int {
      fresh = true;
      launches += 5;
      if (s->capturing) { s->recorded = 5; recorded_priority = s->priority; s->topology = topology; if (rc_recording != LP_OK) return rc_recording; }
      else done += 5;
      return rc;
    }, [&] { fresh = f; launches = l; });
  }
  int ran() const { return done + fake.launched_nodes; }
};
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\\n", __LINE__, #x); std::exit(1); } } while (0)
"""

SCENARIOS = {
    "first two calls direct, then one graph launch each": """
      for (int i = 1; i <= 10; ++i) { CHECK(h.call() == LP_OK); CHECK(h.ran() == 5 * i && h.launches == 5 * i); }
      CHECK(h.done == 10 && fake.launch == 8 && fake.instantiate == 1 && fake.update == 7);
      CHECK(fake.live_graphs == 0 && fake.live_execs == 1);
      CHECK(h.capture.launched == 8 && h.capture.built == 1 && h.capture.direct == 2);
    """,
    "an argument error while recording leaves the state of before": """
      h.call(); h.call(); h.call();
      h.fresh = false; h.rc = LP_ERR_UNSUPPORTED;
      const int ran = h.ran(), launches = h.launches;
      CHECK(h.call() == LP_ERR_UNSUPPORTED);
      CHECK(h.ran() == ran && h.launches == launches && !h.fresh);     // nothing has run, nothing is fresh
      h.rc = LP_OK;
      CHECK(h.call() == LP_OK && h.ran() == ran + 5 && h.fresh);
      CHECK(fake.live_graphs == 0);
    """,
    "a launch that fails is made directly, once": """
      h.call(); h.call();
      fake.fail_launch = true;
      CHECK(h.call() == LP_OK && h.done == 15 && h.launches == 15 && h.fresh);
      CHECK(h.call() == LP_OK && h.done == 20 && fake.begin == 1);
    """,
    "an instantiation that fails is made directly": """
      h.call(); h.call();
      fake.fail_instantiate = true;
      CHECK(h.call() == LP_OK && h.done == 15 && h.launches == 15);
      CHECK(fake.live_graphs == 0 && fake.live_execs == 0);
    """,
    "a recording that cannot begin is made directly": """
      h.call(); h.call();
      fake.fail_begin = true;
      CHECK(h.call() == LP_OK && h.done == 15 && h.launches == 15);
    """,
    "what only a recording refuses is made directly, now and from then on": """
      h.call(); h.call(); h.call();
      h.rc_recording = LP_ERR_CUDA;
      CHECK(h.call() == LP_OK && h.done == 15 && h.launches == 20 && h.fresh);
      CHECK(h.call() == LP_OK && h.done == 20 && fake.begin == 2);
      CHECK(fake.live_graphs == 0);
    """,
    "an error of the direct call too is returned": """
      h.call(); h.call();
      h.rc = LP_ERR_CUDA;
      CHECK(h.call() == LP_ERR_CUDA && fake.launch == 0);
    """,
    "a recording that cannot be ended is made directly": """
      h.call(); h.call();
      fake.fail_end = true;
      CHECK(h.call() == LP_OK && h.done == 15 && h.launches == 15);
    """,
    "the mode of lp_graph_begin": """
      h.call(); h.call(); h.call();
      CHECK(fake.mode == cudaStreamCaptureModeRelaxed);
    """,
    "launches that change now and then stay graph launches": """
      h.call(); h.call();
      for (int epoch = 0; epoch < 12; ++epoch) {
        h.topology = epoch & 1;
        for (int i = 0; i < 20; ++i) h.call();
      }
      CHECK(fake.instantiate == 12 && h.done == 10 && fake.launch == 240 && fake.live_execs == 1);
    """,
    "launches that change all the time are made directly": """
      h.call(); h.call();
      for (int i = 0; i < 40; ++i) { h.topology = i & 1; CHECK(h.call() == LP_OK); }
      CHECK(fake.instantiate == 5 && h.ran() == 5 * 42 && h.done == 5 * (2 + 35));
    """,
    "no count runs over": """
      for (int i = 0; i < 100; ++i) h.call();
      CHECK(h.g.direct_calls == 2 && h.g.rebuilt == 0 && h.g.kept < kForgiveAfter);   // the only counts that a call keeps
    """,
    "recorded at the priority of the caller's stream": """
      h.user.priority = -5;
      for (int i = 0; i < 4; ++i) h.call();
      CHECK(h.recorded_priority == -5 && fake.launch == 2 && fake.live_streams == 1);
      h.user.priority = 0;                       // another stream: neither recorded at -5 nor a graph of its own
      CHECK(h.call() == LP_OK && h.done == 15 && fake.launch == 2 && fake.live_streams == 1);
      h.user.priority = -5;
      CHECK(h.call() == LP_OK && fake.launch == 3);
    """,
    "no stream to record on": """
      fake.fail_stream = true;
      for (int i = 1; i <= 5; ++i) CHECK(h.call() == LP_OK && h.done == 5 * i);
      CHECK(fake.begin == 0);
    """,
    "profiled calls and calls inside a caller's capture are enqueued as they are": """
      h.call(); h.call();
      h.profiled = true;
      CHECK(h.call() == LP_OK && h.done == 15 && fake.begin == 0);
      h.profiled = false; h.user.capturing = true;
      CHECK(h.call() == LP_OK && h.user.recorded == 5 && fake.begin == 0);
    """,
    "another topology is another executable graph": """
      for (int i = 0; i < 4; ++i) h.call();
      h.topology = 1;
      CHECK(h.call() == LP_OK && fake.instantiate == 2 && fake.live_execs == 1 && h.ran() == 25);
    """,
}


def run_scenario(tmp_path, body):
    inc = tmp_path / "inc"
    inc.mkdir()
    (inc / "cuda_runtime_api.h").write_text(FAKE_RUNTIME)
    src = tmp_path / "t.cpp"
    src.write_text(PRELUDE + "int main() { static Handle h; {" + body + "} return 0; }\n")
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover", "-Wall", "-Werror", "-I", str(inc),
                    "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("name", list(SCENARIOS))
def test_calls_as_graph_launches(tmp_path, name):
    run_scenario(tmp_path, SCENARIOS[name])
