"""The table of resident CTAs is kept per kernel: two kernels of one signature, as the plain sweep's two forms
are, keep their own counts whichever is asked for first. Compiled for the host with stand-ins for the
CUDA calls."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "occupancy.h"
static void sweep(int, float*) {}
static void prefetched(int, float*) { static volatile int other; other = 1; }
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int threads, size_t smem) {
    *n = f == reinterpret_cast<const void*>(&sweep) ? 2048 / threads : (int)((224 << 10) / smem);
    return cudaSuccess;
}
int slots(int form, int threads) {
    return form == 0 ? stg::resident_ctas<sweep>(threads) : stg::resident_ctas<prefetched>(threads, (size_t)threads * 560);
}
}
"""


@pytest.mark.parametrize("first", [0, 1])
def test_resident_ctas_do_not_depend_on_the_order_of_calls(tmp_path, first):
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    (tmp_path / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I",
                    os.path.join(ROOT, "paper_1410_5561_gb300", "csrc"),
                    "-I", cuda, str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t.so")], check=True)
    lib = ctypes.CDLL(str(tmp_path / "t.so"))
    want = {(0, 256): 152 * 8, (1, 256): 152 * 1, (0, 160): 152 * 12, (1, 160): 152 * 2}
    for threads in (256, 160):
        for form in (first, 1 - first, first):
            assert lib.slots(form, threads) == want[form, threads], (form, threads)
