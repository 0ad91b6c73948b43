"""Host code that several threads may enter at once, against a stand-in for the runtime that holds the calls where they would
meet.  Plain C++, compiled here with g++; no GPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2602_04163_b200", "csrc")

ENCODER = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include <cuda_runtime_api.h>
#include "bpdq_tma.cuh"
using namespace std::chrono_literals;
static int entry;                                     // stands for the driver's function
extern "C" cudaError_t cudaGetDriverEntryPoint(const char*, void** f, unsigned long long, cudaDriverEntryPointQueryResult* q) {
    std::this_thread::sleep_for(300ms);               // the second thread asks meanwhile
    *f = &entry;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
int main() {
    bool a = false, b = false;
    std::thread first([&] { a = bpdq::encode_tiled_fn() != nullptr; });
    std::this_thread::sleep_for(100ms);
    std::thread second([&] { b = bpdq::encode_tiled_fn() != nullptr; });
    first.join();
    second.join();
    printf("%d %d\n", a, b);
}
"""

SMEM = r"""
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include "bpdq_internal.h"
using namespace std::chrono_literals;
static std::atomic<int> inside{0};
static std::atomic<int> attribute{0};
static std::atomic<bool> large_set{false}, small_done{false};
static void until(std::atomic<bool>& flag) { for (int k = 0; k < 30 && !flag; ++k) std::this_thread::sleep_for(10ms); }
// both threads inside (if the code lets them): the large size is set, then the small one, and the small request returns first
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int bytes) {
    ++inside;
    for (int k = 0; k < 30 && inside < 2; ++k) std::this_thread::sleep_for(10ms);
    if (bytes > 100000) {
        attribute = bytes;
        large_set = true;
        until(small_done);
    } else {
        until(large_set);
        attribute = bytes;
    }
    return cudaSuccess;
}
extern "C" const char* cudaGetErrorString(cudaError_t) { return ""; }
namespace bpdq { int set_error(int code, const char*, ...) { return code; } }
int main() {
    static bpdq::SmemOptin record;
    const void* kernel = &record;
    int a = -1, b = -1;
    std::thread large([&] { a = bpdq::ensure_smem_optin(kernel, record, 0, 200 * 1024, "large"); });
    std::thread small([&] { b = bpdq::ensure_smem_optin(kernel, record, 0, 60 * 1024, "small"); small_done = true; });
    large.join();
    small.join();
    printf("%d %d %d %d\n", a, b, (int)attribute, record.bytes[0]);
}
"""


def run(tmp_path, driver, *sources):
    src, exe = tmp_path / "driver.cpp", tmp_path / "driver"
    src.write_text(driver)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include",
                    str(src), *(os.path.join(CSRC, s) for s in sources), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout.split()


def test_the_tensor_map_encoder_is_there_for_every_thread(tmp_path):
    """Two threads create their first handles: a thread that asked while the other was still looking got none, its handle had no
    tensor maps, and a later launch with 3 to 128 tokens handed the copies an address next to zero."""
    assert run(tmp_path, ENCODER, "bpdq_driver.cpp") == ["1", "1"]


def test_a_smaller_request_does_not_take_back_a_larger_opt_in(tmp_path):
    """Two threads opt in to different sizes of one kernel's shared memory (the gather of two handles with other row lengths): the
    attribute has to end at the larger one, as the record says, or later launches of that size fail for the rest of the process."""
    assert run(tmp_path, SMEM) == ["0", "0", str(200 * 1024), str(200 * 1024)]
