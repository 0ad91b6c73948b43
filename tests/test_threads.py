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
