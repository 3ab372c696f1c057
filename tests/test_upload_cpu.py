"""Uploads from host arrays that live only as long as the call.

The CUDA runtime may copy from pageable memory after cudaMemcpyAsync has returned (it does
not stage where the device reads host pages itself).  A small program with a runtime of its
own, which makes every asynchronous copy at the next synchronisation of its stream, uploads
an array, overwrites it and looks at what arrived.  No GPU is involved.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <vector>
#include "internal.cuh"

static std::vector<std::function<void()>> pending;
static cudaError_t flush() {
    for (auto& f : pending) f();
    pending.clear();
    return cudaSuccess;
}
extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::malloc(n); return cudaSuccess; }
cudaError_t cudaFree(void* p) { flush(); std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    pending.push_back([=] { std::memcpy(d, s, n); });
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return flush(); }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return ""; }
const char* cudaGetErrorName(cudaError_t) { return ""; }
}

int main() {
    oasis::DBuf<int32_t> b;
    std::vector<int32_t> v(1000);
    for (int k = 0; k < 1000; ++k) v[k] = 3 * k + 1;
    b.upload(v.data(), v.size(), nullptr);
    for (auto& x : v) x = -1;
    cudaStreamSynchronize(nullptr);
    for (int k = 0; k < 1000; ++k)
        if (b.p[k] != 3 * k + 1) {
            std::printf("entry %d is %d\n", k, b.p[k]);
            return 1;
        }
    return 0;
}
"""


def test_upload_is_done_with_the_host_array(tmp_path):
    cc = shutil.which("g++")
    from paper_1602_03643_gb300 import build
    try:
        cuda = os.path.dirname(os.path.dirname(build.nvcc()))
    except RuntimeError:
        cuda = None
    if not cc or not cuda:
        pytest.skip("no C++ compiler or CUDA headers")
    src, exe = tmp_path / "upload.cpp", tmp_path / "upload"
    src.write_text(PROGRAM)
    subprocess.run([cc, "-std=c++17", "-I", os.path.join(ROOT, "paper_1602_03643_gb300", "csrc"), "-I",
                    os.path.join(ROOT, "include"), "-I", os.path.join(cuda, "include"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
