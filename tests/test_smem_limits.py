"""The record of what a kernel's shared-memory limit has been raised to, driven by threads at their first calls (host code, no GPU)."""
import os
import subprocess

import pytest

from paper_2609_19104_b200 import build

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "rm_common.cuh"
int rm_last_cuda_error = 0;
int main() {
    int wrong = 0, calls = 0;
    for (int round = 0; round < 20; ++round) {
        rm_smem_configured configured = {};
        std::atomic<int> limit{0}, set_calls{0}, go{0}, bad{0};         // `limit` stands for the kernel's attribute
        std::vector<std::thread> threads;
        for (int i = 0; i < 8; ++i)
            threads.emplace_back([&, i] {
                const int need = 60000 + 4000 * ((i * 5 + round) % 8);
                while (!go) std::this_thread::yield();
                const int rc = configured.raise(0, need, [&] {
                    std::this_thread::sleep_for(std::chrono::microseconds(200 * (8 - i)));
                    limit = need;
                    ++set_calls;
                    return (int)RM_OK;
                });
                if (rc != RM_OK) ++bad;
                for (int k = 0; k < 20; ++k) {                           // launches of this size
                    if (limit < need) ++bad;
                    std::this_thread::sleep_for(std::chrono::microseconds(100));
                }
            });
        go = 1;
        for (auto& t : threads) t.join();
        wrong += bad;
        calls += set_calls;
        if (configured.raise(0, 1000, [] { return (int)RM_ERR_CUDA; }) != RM_OK) ++wrong;                    // (covered)
        if (configured.raise(0, 1 << 20, [] { return (int)RM_ERR_CUDA; }) != RM_ERR_CUDA) ++wrong;
        if (configured.covers(0, 1 << 20) || configured.covers(1, 1000)) ++wrong;
    }
    std::printf("%d %d\n", wrong, calls);
    return wrong != 0;
}
"""


def test_threads_raise_a_kernels_limit_and_never_lower_it(tmp_path):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "limits.cu", tmp_path / "limits"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                    "-o", str(exe), str(src)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
