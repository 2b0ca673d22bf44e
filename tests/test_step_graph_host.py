"""A solve step whose CUDA graph cannot be made (csrc/stepgraph.h) runs its launches
themselves, and capture leaves another thread's alone. Compiled on the host against
a stand-in for the CUDA calls it makes, each failing in turn."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1406_5369_gb300", "csrc")

CUDA = """#pragma once
typedef int cudaError_t;
typedef int *cudaStream_t, *cudaGraph_t, *cudaGraphExec_t;
enum { cudaSuccess = 0, cudaStreamNonBlocking = 1 };
enum cudaStreamCaptureMode { cudaStreamCaptureModeGlobal = 0, cudaStreamCaptureModeThreadLocal = 1 };
extern int fail, mode, outside, launched, made;  // the call that fails; calls made outside the thread-local mode
extern int object;
inline cudaError_t call(int which) { if (mode != cudaStreamCaptureModeThreadLocal) outside++; return which == fail; }
inline cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, int) { if (call(1)) return 1; *s = &object; return 0; }
inline cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return call(2); }
inline cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = nullptr; if (call(3)) return 1; *g = &object; return 0; }
inline cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, int) { if (call(4)) return 1; *x = &object; made++; return 0; }
inline cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { launched++; return 0; }
inline cudaError_t cudaGraphDestroy(cudaGraph_t) { return 0; }
inline cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return 0; }
inline cudaError_t cudaStreamDestroy(cudaStream_t) { return 0; }
inline cudaError_t cudaGetLastError() { return 0; }
inline cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *m) { int t = mode; mode = *m; *m = (cudaStreamCaptureMode)t; return 0; }
"""

MAIN = """#include "stepgraph.h"
#include <stdio.h>
int fail = 0, mode = 0, outside = 0, launched = 0, made = 0, object = 0;
int main() {
  for (fail = 0; fail <= 4; fail++) {
    mg::StepGraphs g = {};
    int user_object = 0, direct = 0, captured = 0;
    cudaStream_t user = &user_object;
    unsigned key = 0;
    outside = launched = made = 0;
    bool ok = true;
    for (int k = 0; k < 6; k++) {
      int status = -1;
      const unsigned before = key;
      const int e = mg::step(g, k, user, [&] { return key; }, [&](unsigned v) { key = v; },
                             [&] { (user == &user_object ? direct : captured)++; key ^= 1; return 0; }, &status);
      ok = ok && e == 0 && status == 0 && key == (before ^ 1) && user == &user_object;
    }
    printf("%d:%d direct %d made %d launched %d outside %d mode %d\\n", fail, ok, direct, made, launched, outside, mode);
  }
}
"""

WANT = """0:1 direct 2 made 2 launched 4 outside 0 mode 0
1:1 direct 6 made 0 launched 0 outside 0 mode 0
2:1 direct 6 made 0 launched 0 outside 0 mode 0
3:1 direct 6 made 0 launched 0 outside 0 mode 0
4:1 direct 6 made 0 launched 0 outside 0 mode 0
"""


def test_steps_without_a_graph(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no C++ compiler")
    (tmp_path / "cuda_runtime.h").write_text(CUDA)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run([gxx, "-std=c++17", "-I", str(tmp_path), "-I", CSRC, str(tmp_path / "main.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout == WANT
