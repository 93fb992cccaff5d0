"""The buffers of one call (csrc/ns_workspace.h) against a CUDA runtime that
counts: whichever allocation fails, and at a return from the middle of a call,
every buffer is freed once, after the stream has been waited for; and the
gradient's workspace is made of nothing else.  No GPU needed."""
from __future__ import annotations

import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1705_06149_gb300", "csrc")

RUNTIME = """#pragma once
#include <cstddef>
#include <cstdlib>
#include <set>
typedef void* cudaStream_t;
typedef int cudaError_t;
enum { cudaSuccess = 0, cudaErrorMemoryAllocation = 2 };
inline std::set<void*> live;
inline int waits = 0, calls = 0, fail_at = -1;
inline cudaError_t cudaMalloc(void** p, size_t n) {
    if (calls++ == fail_at) return cudaErrorMemoryAllocation;
    live.insert(*p = std::malloc(n));
    return cudaSuccess;
}
inline cudaError_t cudaFree(void* p) {
    if (waits == 0 || live.erase(p) != 1) std::abort();
    std::free(p);
    return cudaSuccess;
}
inline cudaError_t cudaStreamSynchronize(cudaStream_t) { ++waits; return cudaSuccess; }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
"""

MAIN = """#include "ns_workspace.h"
static int body(bool leave) {
    Workspace ws(nullptr);
    double* a = ws.get<double>(100);
    float* b = ws.get<float>(0);
    if (leave) return 1;
    char* c = ws.get<char>(7);
    if (!ws.ok()) return 2;
    a[99] = 1.0;
    c[6] = 2;
    b[3] = 3.0f;
    return 0;
}
int main(int, char** argv) {
    fail_at = std::atoi(argv[1]);
    const int want = fail_at < 0 ? 0 : 2;
    if (body(false) != want || !live.empty()) return 1;
    calls = 0;
    if (body(true) != 1 || !live.empty()) return 2;
    return 0;
}
"""


@pytest.mark.parametrize("fail_at", [-1, 0, 1, 2])
def test_every_buffer_is_freed_however_the_call_ends(tmp_path, fail_at):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = tmp_path / "main"
    r = subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-Werror",
                        "-fsanitize=address,undefined", "-I", str(tmp_path), "-I", CSRC,
                        str(tmp_path / "main.cpp"), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe), str(fail_at)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])


def test_the_gradient_allocates_from_its_workspace_alone():
    src = open(os.path.join(CSRC, "ns_api.cu")).read()
    a = src.index("ns_status adjoint_impl(")
    body = src[a:src.index("\n}\n", a)]
    assert "cudaMalloc" not in body and "Workspace ws(" in body
    # the gather's buffer and kernels belong to FP64 grids
    assert re.search(r"acc = tiled \? nullptr", body)
    assert body.index("if constexpr (sizeof(T) == 8)") < body.index("k_adj_rhs<T>")
