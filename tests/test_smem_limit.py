"""The helper that raises a kernel's shared-memory limit, called by two threads with different sizes for one kernel.

Compiled for the CPU against a stand-in for the CUDA runtime whose attribute call of the smaller size waits (at most
half a second) until the larger one has been set, which is the order in which an unsynchronised check-then-set lowers the
limit again.  Whatever the order, the limit that ends up in force has to cover both sizes and what the helper remembers.
"""
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent

HARNESS = r"""
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include "common.cuh"

using namespace conv2d_b200;

static const size_t kSmall = 57744, kLarge = 68208;
static std::atomic<size_t> limit{0};
static std::atomic<bool> small_arrived{false};

extern "C" cudaError_t CUDARTAPI cudaGetDevice(int* dev) { *dev = DEVICE; return cudaSuccess; }
extern "C" cudaError_t CUDARTAPI cudaFuncGetAttributes(cudaFuncAttributes* a, const void*)
{
    a->maxDynamicSharedSizeBytes = (int)limit.load();
    return cudaSuccess;
}
extern "C" cudaError_t CUDARTAPI cudaFuncSetAttribute(const void*, cudaFuncAttribute, int bytes)
{
    const auto until = std::chrono::steady_clock::now() + std::chrono::milliseconds(500);
    if ((size_t)bytes == kSmall) {
        small_arrived = true;
        while (limit < kLarge && std::chrono::steady_clock::now() < until) std::this_thread::yield();
    }
    limit = (size_t)bytes;
    return cudaSuccess;
}

int main()
{
    static SmemLimit done;
    int dummy = 0;
    std::thread small([&] { raise_smem_limit(&dummy, kSmall, done); });
    while (!small_arrived) std::this_thread::yield();
    std::thread large([&] { raise_smem_limit(&dummy, kLarge, done); });
    small.join();
    large.join();
    if (limit < kLarge) { std::printf("limit lowered to %zu\n", limit.load()); return 1; }
    raise_smem_limit(&dummy, 60768, done);            // between the two: nothing to raise, nothing to lower
    if (limit < kLarge) { std::printf("limit lowered to %zu by a later call\n", limit.load()); return 1; }
    return 0;
}
"""


@pytest.mark.parametrize("device", [0, 70])          # a device that the helper keeps a record of, and one beyond its table
def test_two_threads_never_lower_the_limit(tmp_path, device):
    src = tmp_path / "smem_limit.cpp"
    src.write_text(HARNESS.replace("DEVICE", str(device)))
    exe = tmp_path / "smem_limit"
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-x", "c++", "-I", str(ROOT / "include"),
                    "-I", str(ROOT / "paper_1705_10591_b200" / "csrc"), "-I", "/usr/local/cuda/include", str(src), "-o", str(exe)],
                   check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert run.returncode == 0, run.stdout
