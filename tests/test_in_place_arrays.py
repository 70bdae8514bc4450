"""Which arrays a training step reads where they lie (mlp_internal.h): only
those in the memory of the problem's own device, on a 16-byte boundary.  The
rule is host code over pointer attributes, compiled here with the system's
C++ compiler -- no GPU needed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "mlp_internal.h"
#include <cstdio>
int main() {
    const cudaMemoryType types[] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice,
                                    cudaMemoryTypeManaged};
    for (cudaMemoryType t : types)
        for (int owner = 0; owner < 3; ++owner)
            for (int device = 0; device < 3; ++device)
                for (int off = 0; off < 32; off += 2) {
                    cudaPointerAttributes at = {};
                    at.type = t;
                    at.device = owner;
                    const void* v = reinterpret_cast<const void*>(static_cast<uintptr_t>(0x7f0000000000ull + off));
                    const bool want = t == cudaMemoryTypeDevice && owner == device && off % 16 == 0;
                    if (comet::mlp::usable_in_place(at, device, v) != want) {
                        std::printf("type %d owner %d device %d offset %d\n", (int)t, owner, device, off);
                        return 1;
                    }
                }
    return 0;
}
"""


def test_only_own_aligned_device_memory_is_read_in_place(tmp_path):
    cxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if cxx is None or not os.path.exists(nvcc):
        pytest.skip("no C++ compiler or CUDA headers")
    src, exe = tmp_path / "in_place.cpp", tmp_path / "in_place"
    src.write_text(SRC)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    inc = [os.path.join(ROOT, "include"), os.path.join(ROOT, "paper_2609_21803_gb300", "csrc"), cuda]
    subprocess.run([cxx, "-std=c++17"] + [a for i in inc for a in ("-I", i)] + [str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
