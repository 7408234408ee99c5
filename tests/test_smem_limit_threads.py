"""The record of raised shared memory limits on the CPU: the library's own
function, compiled against stand-ins for the two CUDA calls that it makes."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STANDINS = r"""
#include <atomic>
#include <chrono>
#include <map>
#include <mutex>
#include <thread>

std::atomic<int> slow{0}, begun{0}, calls{0};
static std::mutex mu;
static std::map<const void*, int> limits;
int limit_of(const void* f) { return limits.count(f) ? limits[f] : 0; }

extern "C" int cudaGetDevice(int* d) { *d = 0; return 0; }
extern "C" int cudaFuncSetAttribute(const void* f, int, int bytes) {
    ++calls;
    if (bytes == slow) {  // a thread that is held up between its look and its call
        begun = 1;
        std::this_thread::sleep_for(std::chrono::milliseconds(300));
    }
    std::lock_guard<std::mutex> lock(mu);
    limits[f] = bytes;
    return 0;
}
"""

HARNESS = r"""
#include <atomic>
#include <cstdio>
#include <thread>

#include "dgs_internal.cuh"

extern std::atomic<int> slow, begun, calls;
int limit_of(const void* f);
void kernel_a(int) {}
void kernel_b(int) {}

#define EXPECT(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

int main() {
    const void* a = reinterpret_cast<const void*>(&kernel_a);
    const void* b = reinterpret_cast<const void*>(&kernel_b);
    slow = 50000;
    std::thread small([] { dgs::ensure_smem_limit<kernel_a>(50000); });
    while (!begun) std::this_thread::yield();
    dgs::ensure_smem_limit<kernel_a>(200000);
    small.join();
    EXPECT(limit_of(a) == 200000);
    const int n = calls;
    EXPECT(dgs::ensure_smem_limit<kernel_a>(60000) == cudaSuccess && calls == n && limit_of(a) == 200000);
    EXPECT(limit_of(b) == 0);
    EXPECT(dgs::ensure_smem_limit<kernel_b>(60000) == cudaSuccess && limit_of(b) == 60000);
    return 0;
}
"""


def test_the_limit_only_grows_and_belongs_to_its_kernel(tmp_path):
    from paper_1106_5694_gb300 import build_ext

    nvcc = build_ext._nvcc()
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc")
    src, standins, exe = tmp_path / "limits.cu", tmp_path / "standins.cpp", tmp_path / "limits"
    src.write_text(HARNESS)
    standins.write_text(STANDINS)
    subprocess.check_call([nvcc, *build_ext.ARCH, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-cudart", "shared",
                           "-I", build_ext.CSRC, "-o", str(exe), str(src), str(standins), "-lpthread"])
    libs = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "lib64")
    env = {**os.environ, "LD_LIBRARY_PATH": libs + ":" + os.environ.get("LD_LIBRARY_PATH", "")}
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60, env=env)
    assert r.returncode == 0, r.stdout + r.stderr
