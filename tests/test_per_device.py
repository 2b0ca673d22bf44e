"""Kernel attributes are per device: what csrc/perdevice.h keeps is found once for
each device, and again after a failure. Compiled on the host against a stand-in
for the one CUDA call it makes."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1406_5369_gb300", "csrc")

CUDA = """#pragma once
typedef int cudaError_t;
enum { cudaSuccess = 0 };
extern int g_dev, g_err;
inline cudaError_t cudaGetDevice(int *d) { *d = g_dev; return g_err; }
"""

MAIN = """#include "perdevice.h"
#include <stdio.h>
int g_dev = 0, g_err = 0, asked = 0;
static mg::PerDevice p;
static long long get(long long v) { return mg::per_device(p, [&] { asked++; return v; }); }
int main() {
  printf("%lld ", get(16)); printf("%lld ", get(1)); printf("%d ", asked);   // 16 16 1
  g_dev = 1;
  printf("%lld ", get(-7)); printf("%lld ", get(8)); printf("%lld ", get(1)); printf("%d ", asked);  // -7 8 8 3
  g_dev = 0;
  printf("%lld %d ", get(1), asked);                                         // 16 3
  g_dev = 64;
  printf("%lld ", get(5)); printf("%lld ", get(6));                          // 5 6: not kept
  g_dev = 2; g_err = 1;
  printf("%lld ", get(9)); g_err = 0; printf("%lld", get(4));                // 9 4
}
"""


def test_found_once_per_device(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no C++ compiler")
    (tmp_path / "cuda_runtime.h").write_text(CUDA)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run([gxx, "-std=c++17", "-I", str(tmp_path), "-I", CSRC, str(tmp_path / "main.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout == "16 16 1 -7 8 8 3 16 3 5 6 9 4"


@pytest.mark.parametrize("name", ["fx2d.cuh", "fx3d.cuh", "small2d.cu"])
def test_attributes_are_set_where_the_value_is_per_device(name):
    """No process-wide flag says that a kernel's attributes are set."""
    with open(os.path.join(CSRC, name)) as fh:
        src = fh.read()
    assert "cudaFuncSetAttribute" in src and "PerDevice" in src
    assert not re.search(r"static (?!PerDevice)(int|long long|bool) \w+ = ", src)
    assert not re.search(r"^int g_\w+ = ", src, re.M)
