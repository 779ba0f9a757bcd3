"""A refused allocation leaves no CUDA error behind (csrc/alloc.h): a launch
helper that ends with cudaGetLastError() would take it for its own launch's.
The helpers against a fake CUDA runtime whose allocations fail, on the CPU, and
no allocation of the library past them."""
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_07152_gb300", "csrc")

FAKE = r"""
#pragma once
#include <cstddef>
#include <cstdlib>
typedef int cudaError_t;
typedef void* cudaMemPool_t;
typedef void* cudaStream_t;
enum { cudaSuccess = 0, cudaErrorMemoryAllocation = 2 };
inline int g_last = 0, g_calls = 0;
inline bool g_refuse = false;
inline cudaError_t fake(void** p, size_t n) {
    ++g_calls;
    if (g_refuse) return g_last = cudaErrorMemoryAllocation;
    *p = std::malloc(n);
    return cudaSuccess;
}
inline cudaError_t cudaMalloc(void** p, size_t n) { return fake(p, n); }
inline cudaError_t cudaMallocHost(void** p, size_t n) { return fake(p, n); }
inline cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) {
    return fake(p, n);
}
inline cudaError_t cudaGetLastError() { const int e = g_last; g_last = 0; return e; }
"""

MAIN = r"""
#include "alloc.h"
#include <cstdio>
int main() {
    int bad = 0;
    for (int k = 0; k < 2; ++k) {
        const bool refuse = k == 1;
        g_refuse = refuse;
        float* a = reinterpret_cast<float*>(8);
        long* b = reinterpret_cast<long*>(8);
        char* c = reinterpret_cast<char*>(8);
        const int want = refuse ? cudaErrorMemoryAllocation : cudaSuccess;
        bad += pvs::device_alloc(&a, 10) != want || (a == nullptr) != refuse || g_last != 0;
        bad += pvs::pinned_alloc(&b, 0) != want || (b == nullptr) != refuse || g_last != 0;
        bad += pvs::pool_alloc(&c, 10, nullptr, nullptr) != want || (c == nullptr) != refuse ||
               g_last != 0;
    }
    g_last = cudaErrorMemoryAllocation;
    bad += pvs::taken(cudaErrorMemoryAllocation) != cudaErrorMemoryAllocation || g_last != 0;
    printf("%d %d\n", bad, g_calls);
    return 0;
}
"""


def test_a_refusal_is_returned_and_not_left_behind(tmp_path):
    (tmp_path / "cuda_runtime_api.h").write_text(FAKE)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = tmp_path / "main"
    subprocess.run(["g++", "-std=c++17", "-I", str(tmp_path), "-I", CSRC,
                    str(tmp_path / "main.cpp"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert out.split() == ["0", "6"]


def test_every_allocation_goes_through_the_helpers():
    for path in glob.glob(os.path.join(CSRC, "*")):
        if os.path.basename(path) == "alloc.h":
            continue
        text = re.sub(r"//.*", "", open(path).read())
        found = re.findall(r"\bcuda(?:Malloc\w*|HostAlloc|MemAllocPool\w*)\s*\(", text)
        assert not found, (path, found)
