"""Copies from pageable host arrays: the source lives until the stream has been synchronised. The host code is compiled
against a runtime that reads the sources of all copies only at the synchronisation."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1708_06065_gb300", "csrc")

PROGRAM = r"""
#include "host_copies.h"
#include <cstring>

struct Copy { void *dst; const void *src; size_t bytes; };
static std::vector<Copy> pending;
static int gone;

extern "C" cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t bytes, cudaMemcpyKind, cudaStream_t) {
    pending.push_back(Copy{dst, src, bytes});
    return cudaSuccess;
}
static void synchronize() {
    for (auto &c : pending) memcpy(c.dst, c.src, c.bytes);
    pending.clear();
}

struct Item {   // counts how many have been given back
    int v;
    explicit Item(int x) : v(x) {}
    Item(const Item &) = default;
    ~Item() { ++gone; }
};

int main() {
    lair::HostSources sources;
    std::vector<int> dst(6, 0);
    {
        for (int k = 0; k < 2; ++k) {   // two sources on the way at once
            auto v = std::make_shared<std::vector<Item>>();
            v->reserve(3);
            for (int i = 0; i < 3; ++i) v->emplace_back(10 * k + i);
            gone = 0;
            if (sources.upload(reinterpret_cast<Item *>(dst.data() + 3 * k), v, nullptr) != cudaSuccess) return 1;
        }
        auto none = std::make_shared<std::vector<Item>>();
        if (sources.upload(static_cast<Item *>(nullptr), none, nullptr) != cudaSuccess || pending.size() != 2) return 2;
    }
    if (gone != 0) return 3;   // freed with its copy in flight
    synchronize();
    for (int i = 0; i < 6; ++i)
        if (dst[i] != 10 * (i / 3) + i % 3) return 4;
    sources.release();
    return gone == 6 ? 0 : 5;
}
"""


def test_sources_outlive_their_copies(tmp_path):
    nvcc = shutil.which("nvcc")
    if shutil.which("g++") is None or nvcc is None:
        pytest.skip("no host compiler or CUDA headers")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    src, exe = tmp_path / "copies.cpp", tmp_path / "copies"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", include, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], timeout=20).returncode == 0
