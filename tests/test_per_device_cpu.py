"""Host state of a kernel per device (csrc/per_device.h) against a stand-in for the runtime's calls:
every device gets its own shared-memory limit and its own count of resident blocks, once, whatever
thread comes first; a failed call is not kept."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROGRAM = r"""
#include <cassert>
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"

static thread_local int g_dev = 0;
static std::atomic<int> g_limit[100], g_calls{0};
static cudaError_t g_fail = cudaSuccess;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int bytes) {
    if (g_fail != cudaSuccess) return g_fail;
    ++g_calls;
    g_limit[g_dev] = bytes;
    return cudaSuccess;
}
extern "C" cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
    *n = g_dev;  // none on device 0
    return cudaSuccess;
}
static void kernel(int, float) {}

int main() {
    lat::PerDevice limit;
    g_fail = cudaErrorInvalidValue;
    assert(lat::raise_smem(limit, kernel, 1000) == cudaErrorInvalidValue);
    g_fail = cudaSuccess;
    for (int rep = 0; rep < 2; ++rep)
        for (g_dev = 0; g_dev < 3; ++g_dev) {
            assert(lat::raise_smem(limit, kernel, 1000 + g_dev) == cudaSuccess);
            assert(g_limit[g_dev] == 1000 + g_dev);
        }
    assert(g_calls == 3);
    lat::PerDevice res;
    int n = 0;
    for (int d : {0, 3, 5, 3, 80, 80}) {  // 80: beyond what is kept
        g_dev = d;
        assert(lat::resident_blocks(res, kernel, 128, 2000, &n) == cudaSuccess);
        assert(n == (d ? d : 1) && g_limit[d] == 2000);
    }
    assert(g_calls == 3 + 5);
    lat::PerDevice shared;
    std::vector<std::thread> t;
    for (int i = 0; i < 8; ++i)
        t.emplace_back([&, i] {
            g_dev = i % 4;
            for (int r = 0; r < 1000; ++r) {
                int v = 0;
                assert(lat::resident_blocks(shared, kernel, 128, 3000 + i % 4, &v) == cudaSuccess);
                assert(v == std::max(1, i % 4) && g_limit[i % 4] == 3000 + i % 4);
            }
        });
    for (auto& q : t) q.join();
    std::puts("ok");
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no C++ compiler")
def test_kernel_state_is_kept_per_device(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I" + os.path.join(CUDA, "include"),
                    "-I" + os.path.join(ROOT, "paper_1508_02899_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == "ok\n"


def test_no_kernel_keeps_its_state_for_the_process():
    csrc = os.path.join(ROOT, "paper_1508_02899_gb300", "csrc")
    for name in os.listdir(csrc):
        with open(os.path.join(csrc, name)) as fh:
            text = fh.read()
        for word in ("static bool ", "static int "):
            assert not any(line.strip().startswith(word) and line.rstrip().endswith(";")
                           and "(" not in line for line in text.splitlines()), name
