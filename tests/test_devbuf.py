"""The owning device buffer (devbuf.h) after an allocation that failed: empty.
Callers compare its size with what they need before they use it, so a buffer
that kept the size without the memory would hand out a null pointer on the
next call.  cudaMalloc is replaced at compile time by one that fails."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_17917_gb300", "csrc")
MAIN = r"""
#include <cstddef>
#include <cstdio>
#include <cstdlib>
enum cudaError_t { cudaSuccess = 0, cudaErrorMemoryAllocation = 2 };
static bool full = false;
static cudaError_t cudaMalloc(void **p, size_t n)
{
    if (full) return cudaErrorMemoryAllocation;
    *p = malloc(n);
    return cudaSuccess;
}
static void cudaFree(void *p) { free(p); }
#include "devbuf_host.h"
int main()
{
    dg::DevBuf<double> b;
    if (b.alloc(4) != cudaSuccess || b.n != 4 || !b.ptr) return 1;
    full = true;
    if (b.alloc(8) != cudaErrorMemoryAllocation) return 2;
    if (b.n != 0 || b.ptr) return 3;
    full = false;
    if (b.alloc(8) != cudaSuccess || b.n != 8 || !b.ptr) return 4;
    return b.alloc(0) == cudaSuccess && b.n == 0 && !b.ptr ? 0 : 5;
}
"""


def test_a_failed_allocation_leaves_it_empty(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    text = open(os.path.join(CSRC, "devbuf.h")).read().replace("#include <cuda_runtime.h>\n", "")
    (tmp_path / "devbuf_host.h").write_text(text)
    (tmp_path / "main.cpp").write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-o", str(tmp_path / "t"), str(tmp_path / "main.cpp")], check=True)
    assert subprocess.run([str(tmp_path / "t")]).returncode == 0
