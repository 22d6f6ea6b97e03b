"""Kernel set-up that is done once on every device, not once in a process."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_09422_gb300", "csrc")
CUDA = "/usr/local/cuda/include"

PROGRAM = r"""
#include "per_device.hpp"
#include <cstdio>
static int device = 0, calls = 0;
static cudaError_t result = cudaSuccess;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
static PerDevice ready;
static int go(int d) { device = d; return (int)ready.once([] { calls++; return result; }); }
int main()
{
    const int devs[] = {0, 0, 3, 0, 3, 63, 63, 64, 64};
    for (int d : devs) { go(d); printf("%d ", calls); }
    result = cudaErrorInvalidValue;  // a set-up that failed is tried again
    printf("%d ", go(5) == cudaErrorInvalidValue);
    result = cudaSuccess;
    go(5); printf("%d ", calls);
    go(5); printf("%d\n", calls);
}
"""


@pytest.mark.skipif(not os.path.exists(os.path.join(CUDA, "cuda_runtime_api.h")), reason="no CUDA headers")
def test_set_up_once_on_every_device(tmp_path):
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", CUDA, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert out == "1 1 2 2 2 3 3 4 5 1 7 7".split()


@pytest.mark.parametrize("name", ["cno_api.cu", "lb_api.cu"])
def test_no_launcher_keeps_a_process_wide_flag(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    assert not re.search(r"^\s+static bool \w+ = false", text, re.M)
    assert len(re.findall(r"static PerDevice \w+;", text)) >= 2
