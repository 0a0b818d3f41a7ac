"""Which vectors the preconditioner's kernels take where they are: this device's memory on a double's boundary. Another
GPU's memory, managed memory and odd addresses, which a copy takes, go through one; host memory is no device memory.
The host code is compiled against a runtime with made-up allocations."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1708_06065_gb300", "csrc")

PROGRAM = r"""
#include "pointers.h"

struct Range { uintptr_t at; cudaMemoryType type; int device; };
static const Range ranges[] = {{0x10000, cudaMemoryTypeDevice, 1}, {0x20000, cudaMemoryTypeDevice, 0},
                               {0x30000, cudaMemoryTypeManaged, 1}, {0x40000, cudaMemoryTypeHost, 1},
                               {0x50000, cudaMemoryTypeUnregistered, -2}};
static int errors;

extern "C" cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    for (const Range &r : ranges)
        if (reinterpret_cast<uintptr_t>(p) >> 16 == r.at >> 16) {
            *a = cudaPointerAttributes();
            a->type = r.type;
            a->device = r.device;
            return cudaSuccess;
        }
    return cudaErrorInvalidValue;
}
extern "C" cudaError_t cudaGetDevice(int *dev) { *dev = 1; return cudaSuccess; }
extern "C" cudaError_t cudaGetLastError() { ++errors; return cudaSuccess; }

int main() {
    struct { uintptr_t p; bool device, kernels; } want[] = {
        {0x10000, true, true}, {0x10008, true, true}, {0x10004, true, false}, {0x10001, true, false},
        {0x20000, true, false},                                                   // another GPU's
        {0x30000, true, false}, {0x40000, false, false}, {0x50000, false, false}, // managed, pinned, pageable
        {0x60000, false, false}};                                                 // unknown to the runtime
    for (auto &w : want) {
        const double *p = reinterpret_cast<const double *>(w.p);
        if (lair::is_device_ptr(p) != w.device || lair::kernels_take(p) != w.kernels) return 1 + (int)(w.p >> 16);
    }
    return errors == 2 ? 0 : 100;   // the error of an unknown pointer does not stay behind
}
"""


def test_which_vectors_kernels_take(tmp_path):
    nvcc = shutil.which("nvcc")
    if shutil.which("g++") is None or nvcc is None:
        pytest.skip("no host compiler or CUDA headers")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    src, exe = tmp_path / "pointers.cpp", tmp_path / "pointers"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", include, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], timeout=20).returncode == 0
