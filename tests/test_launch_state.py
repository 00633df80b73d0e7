"""What the launchers keep per device or context, compiled on the host against stand-ins for the queries.

A kernel's attributes are set before anyone launches it, also where two threads meet on its first use and where setting
them failed at first.  How many clusters fit is asked again after a failure, and in another context."""
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
static unsigned long long context = 1;
static CUresult context_id(CUcontext, unsigned long long* id) { *id = context; return context ? CUDA_SUCCESS : CUDA_ERROR_INVALID_CONTEXT; }
extern "C" cudaError_t cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* found) {
    *fn = (void*)&context_id, *found = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
static tb::DeviceFlags late, failing, outside;
static int asked;
static int fit(int blocks, int answer) { return tb::clusters_that_fit(blocks, [&] { return ++asked, answer; }); }
static int clusters() {
    device = 0;
    if (fit(8, -1) != -1 || fit(8, 16) != 16 || asked != 2) return 11;             // a failure is not an answer to keep
    if (fit(8, 5) != 16 || asked != 2) return 12;
    if (fit(16, 0) != 0 || fit(16, 9) != 0 || asked != 3) return 13;               // none is
    context = 2;
    if (fit(8, 3) != 3 || fit(8, 5) != 3 || fit(16, 1) != 1 || asked != 5) return 14;
    device = 1;
    if (fit(8, 7) != 7 || asked != 6) return 15;
    device = 0;
    if (fit(8, 5) != 3 || asked != 6) return 16;
    for (int d : {64, -1}) {
        device = d;
        if (fit(8, 4) != 4 || fit(8, 6) != 6) return 17;
    }
    device = 0, context = 0;                           // no current context, or a driver that does not number them
    return fit(8, 4) != 4 || fit(8, 6) != 6 ? 18 : 0;
}
int main() {
    if (const int r = clusters()) return r;
    device = 3;
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


def test_what_is_kept_per_device_and_context(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-pthread", "-I" + os.path.join(ROOT, "paper_2503_07518_b200", "csrc"),
                           "-I/usr/local/cuda/include", str(src), "-o", str(exe)])
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
