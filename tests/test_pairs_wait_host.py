"""The pinned word and event that `rasterize` reads a pair count with, on a
runtime that only counts (no GPU): a thread that alternates between devices
makes one of each per device, another thread its own, and a thread's end gives
all of its own back."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_08551_gb300", "csrc")

RUNTIME = """
#pragma once
#include <cstdlib>
typedef int cudaError_t;
typedef void* cudaEvent_t;
enum { cudaSuccess = 0, cudaHostAllocDefault = 0, cudaEventDisableTiming = 2 };
extern thread_local int device;
extern int made, freed, fail;
inline cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
inline cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { if (fail) return 2; ++made; *p = std::malloc(n); return 0; }
inline cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { ++made; *e = std::malloc(1); return 0; }
inline cudaError_t cudaEventDestroy(cudaEvent_t e) { ++freed; std::free(e); return 0; }
inline cudaError_t cudaFreeHost(void* p) { ++freed; std::free(p); return 0; }
"""

MAIN = """
#include <cstdio>
#include <thread>
#include "pairs_wait.cuh"
thread_local int device = 0;
int made = 0, freed = 0, fail = 0;
int main() {
    std::thread([] {
        fail = 1;
        if (gi::pairs_wait()) std::puts("a word without memory");
        fail = 0;
        gi::PairsWait* first[2] = {nullptr, nullptr};
        for (int i = 0; i < 100; ++i) {
            device = i % 2;
            gi::PairsWait* w = gi::pairs_wait();
            if (!w || !w->k || !w->ev) std::puts("no word");
            if (i < 2) first[device] = w;
            if (w != first[device] || first[0] == first[1]) std::puts("not the device's own");
        }
        std::thread([] { gi::pairs_wait(); }).join();
    }).join();
    std::printf("%d %d", made, freed);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no g++")
def test_one_word_and_event_per_thread_and_device(tmp_path):
    (tmp_path / "cuda_runtime_api.h").write_text(RUNTIME)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = tmp_path / "main"
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", str(tmp_path), "-x", "c++", "-I", CSRC,
                    str(tmp_path / "main.cpp"), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == "6 6"
