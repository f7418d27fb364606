"""Which array arguments kernels read where they are, against a runtime whose
answers the test makes up (no GPU: a second device's memory among them)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "pointers.h"
#include <cstdio>
static cudaMemoryType type;
static int where, current;
static cudaError_t answer;
extern "C" cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) {
    a->type = type;
    a->device = where;
    return answer;
}
extern "C" cudaError_t cudaGetDevice(int *d) { *d = current; return cudaSuccess; }
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
static int ask(cudaMemoryType t, int w, int c, cudaError_t e = cudaSuccess) {
    type = t; where = w; current = c; answer = e;
    return dtws::readable_in_place(nullptr);
}
int main() {
    printf("%d%d%d%d%d%d%d\n", ask(cudaMemoryTypeDevice, 0, 0), ask(cudaMemoryTypeDevice, 1, 0),
           ask(cudaMemoryTypeDevice, 0, 1), ask(cudaMemoryTypeManaged, 1, 0), ask(cudaMemoryTypeHost, 0, 0),
           ask(cudaMemoryTypeUnregistered, -2, 0), ask(cudaMemoryTypeDevice, 0, 0, cudaErrorInvalidValue));
}
"""


def test_memory_of_another_device_is_not_read_in_place(tmp_path):
    include = "/usr/local/cuda/include"
    if not shutil.which("g++") or not os.path.exists(os.path.join(include, "cuda_runtime_api.h")):
        pytest.skip("no host compiler or CUDA headers")
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I" + include, "-I" + os.path.join(ROOT, "paper_1812_10302_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    got = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip()
    # this device, another one's (both ways), managed, pinned host, pageable host, no answer
    assert got == "1001000"
