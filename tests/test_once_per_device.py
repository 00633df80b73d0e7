"""A kernel's attributes are set before anyone launches it, also where two threads meet on its first use and where setting
them failed at first: the header's helper, compiled on the host against a stand-in for the device query."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include "tb_internal.h"
static thread_local int device = 3;
extern "C" cudaError_t cudaGetDevice(int* dev) { *dev = device; return device < 0 ? cudaErrorInitializationError : cudaSuccess; }
static tb::DeviceFlags late, failing, outside;
int main() {
    // one thread is still setting the attributes when another arrives: that one does not go on without them
    std::atomic<int> inside{0}, set{0};
    std::thread first([&] {
        tb::once_per_device(late, [&] {
            inside = 1;
            std::this_thread::sleep_for(std::chrono::milliseconds(300));
            return ++set, cudaSuccess;
        });
    });
    while (!inside) std::this_thread::yield();
    int calls = 0;
    if (tb::once_per_device(late, [&] { return ++set, ++calls, cudaSuccess; }) != cudaSuccess || set < 1) return 1;
    first.join();
    if (tb::once_per_device(late, [&] { return ++calls, cudaSuccess; }) != cudaSuccess || calls != 1) return 2;
    device = 4;                                        // another device has its own
    if (tb::once_per_device(late, [&] { return ++calls, cudaSuccess; }) != cudaSuccess || calls != 2) return 3;
    // a failure is told, and not remembered as done
    if (tb::once_per_device(failing, [&] { return cudaErrorInvalidValue; }) != cudaErrorInvalidValue) return 4;
    calls = 0;
    if (tb::once_per_device(failing, [&] { return ++calls, cudaSuccess; }) != cudaSuccess || calls != 1) return 5;
    // devices that are not kept account of, or not known: every time
    for (int d : {64, -1}) {
        device = d, calls = 0;
        for (int i = 0; i < 2; ++i) tb::once_per_device(outside, [&] { return ++calls, cudaSuccess; });
        if (calls != 2) return 6;
    }
    return 0;
}
"""


def test_nobody_launches_a_kernel_before_its_attributes_are_set(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-pthread", "-I" + os.path.join(ROOT, "paper_2503_07518_b200", "csrc"),
                           "-I/usr/local/cuda/include", str(src), "-o", str(exe)])
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
