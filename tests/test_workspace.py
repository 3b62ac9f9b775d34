"""The context workspace against a fake of the CUDA allocator (host code only): an
optional workspace that did not fit is had once the memory is free again, is not tried
while it is not, and costs the present workspace nothing during a capture."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#pragma once
#include <cstddef>
#include <cstdlib>
#include <map>
typedef int cudaError_t;
typedef void *cudaStream_t;
enum { cudaSuccess = 0, cudaErrorMemoryAllocation = 2 };
enum cudaStreamCaptureStatus { cudaStreamCaptureStatusNone = 0, cudaStreamCaptureStatusActive = 1 };
static size_t device_free = 1000000;
static int frees = 0, mallocs = 0, captured = 0;
static std::map<void *, size_t> held;
static cudaError_t cudaMalloc(void **p, size_t n) {
    ++mallocs;
    if (n > device_free) return cudaErrorMemoryAllocation;
    *p = malloc(1);
    held[*p] = n;
    device_free -= n;
    return cudaSuccess;
}
static cudaError_t cudaFree(void *p) {
    ++frees;
    device_free += held[p];
    held.erase(p);
    free(p);
    return cudaSuccess;
}
static cudaError_t cudaGetLastError() { return cudaSuccess; }
static cudaError_t cudaMemGetInfo(size_t *f, size_t *t) {
    *f = device_free;
    *t = 1000000;
    return cudaSuccess;
}
static cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
    *s = captured ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
"""

MAIN = r"""
#include <cstdio>
#include "workspace.h"
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
    using namespace pcl;
    pcl_ctx c;
    CHECK(ensure_ws(&c, 10000) == PCL_OK && c.ws_bytes == ws_request(10000));
    device_free -= 900000;  // another allocator
    CHECK(!ensure_ws_optional(&c, 500000, nullptr) && c.err.empty());
    CHECK(ensure_ws(&c, 10000) == PCL_OK);
    const int m = mallocs, f = frees;
    for (int k = 0; k < 5; ++k) CHECK(!ensure_ws_optional(&c, 500000, nullptr));
    CHECK(mallocs == m && frees == f && c.ws);
    device_free += 900000;
    captured = 1;
    CHECK(!ensure_ws_optional(&c, 500000, nullptr) && mallocs == m && frees == f);
    captured = 0;
    CHECK(ensure_ws_optional(&c, 500000, nullptr) && c.ws_bytes == ws_request(500000));
    CHECK(ensure_ws_optional(&c, 400000, nullptr) && mallocs == m + 1);
    CHECK(ensure_ws(&c, 900000) == PCL_ERR_OOM && !c.err.empty() && !c.ws && c.ws_bytes == 0);
    return 0;
}
"""


def test_refused_workspace_is_had_again(tmp_path):
    (tmp_path / "cuda_runtime_api.h").write_text(FAKE)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = tmp_path / "main"
    subprocess.check_call(["g++", "-std=c++17", "-I", str(tmp_path), "-I", os.path.join(ROOT, "include"), "-I",
                           os.path.join(ROOT, "paper_2512_13133_gb300", "csrc"), str(tmp_path / "main.cpp"), "-o",
                           str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
