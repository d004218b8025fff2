"""Graph capture (csrc/graph.h) against a fake CUDA runtime: a launch that is
refused inside a capture must not leave a graph behind that replays without it."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUNTIME = r"""
#pragma once
#include <cstdio>
typedef int cudaError_t;
typedef struct St* cudaStream_t;
typedef struct Gr { int n; }* cudaGraph_t;
typedef struct Ex { int n; }* cudaGraphExec_t;
enum { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorMemoryAllocation = 2, cudaErrorStreamCaptureInvalidated = 901,
       cudaErrorUnknown = 999 };
enum { cudaStreamCaptureModeThreadLocal = 1 };
// what the next calls return, and what is left behind
static int last, begin_ret, end_ret, inst_ret, begun, graphs_alive, execs;
static Gr the_graph;
static Ex the_exec;
inline cudaError_t cudaPeekAtLastError() { return last; }
inline cudaError_t cudaGetLastError() { int e = last; last = 0; return e; }
inline cudaError_t note(int e) { if (e) last = e; return e; }
inline cudaError_t cudaStreamBeginCapture(cudaStream_t, int) { if (!begin_ret) ++begun; return note(begin_ret); }
inline cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  --begun;
  *g = nullptr;
  if (!end_ret) { *g = &the_graph; ++graphs_alive; }
  return note(end_ret);
}
inline cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
  if (!inst_ret) { *x = &the_exec; ++execs; }
  return note(inst_ret);
}
inline cudaError_t cudaGraphDestroy(cudaGraph_t) { --graphs_alive; return 0; }
"""

MAIN = r"""
#include <cstdlib>
#include "graph.h"
int main(int argc, char** argv) {
  last = atoi(argv[1]); begin_ret = atoi(argv[2]); const int launch = atoi(argv[3]);
  end_ret = atoi(argv[4]); inst_ret = atoi(argv[5]);
  int ran = 0;
  cudaGraphExec_t x = &the_exec;
  const int e = mpm::capture_graph(nullptr, 0, [&](cudaStream_t) { ++ran; if (launch) last = launch; }, &x);
  printf("%d %d %d %d %d %d %d\n", e, ran, x != nullptr, execs, begun, graphs_alive, last);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("graph")
    (d / "cuda_runtime.h").write_text(RUNTIME)
    (d / "main.cpp").write_text(MAIN)
    exe = d / "main"
    csrc = os.path.join(ROOT, "paper_2303_02346_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", f"-I{d}", f"-I{csrc}", str(d / "main.cpp"), "-o", str(exe)], check=True)
    return str(exe)


# pending error, BeginCapture, launch, EndCapture, Instantiate ->
# returned error, runs of fn, exec given, execs made, captures open, graphs not destroyed, error left pending
@pytest.mark.parametrize("given,want", [
    ((0, 0, 0, 0, 0), (0, 1, 1, 1, 0, 0, 0)),
    ((0, 0, 1, 0, 0), (1, 1, 0, 0, 0, 0, 0)),      # a refused launch that the capture survives
    ((0, 0, 1, 901, 0), (1, 1, 0, 0, 0, 0, 0)),    # one that ends the capture: the launch's own error is told
    ((0, 0, 0, 901, 0), (901, 1, 0, 0, 0, 0, 0)),
    ((0, 0, 0, 0, 2), (2, 1, 0, 0, 0, 0, 0)),
    ((0, 2, 0, 0, 0), (2, 0, 0, 0, 0, 0, 0)),
    ((2, 0, 0, 0, 0), (2, 0, 0, 0, 0, 0, 2)),      # another's error: not run, left pending
])
def test_capture(program, given, want):
    out = subprocess.run([program, *map(str, given)], capture_output=True, text=True, check=True).stdout
    assert tuple(map(int, out.split())) == want
