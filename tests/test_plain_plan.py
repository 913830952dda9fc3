"""Launch plans of the plain sweep, compiled for the host from the header that the launches use."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "plain_plan.h"
extern "C" long prefetch(int nx, int V, int rows, long bytes, int alone, int* threads, long* smem) {
    const stg::PrefetchShape p = stg::prefetch_shape(nx, V, rows, (size_t)bytes, alone != 0);
    *threads = p.threads;
    *smem = (long)p.smem;
    return p.width;
}
"""
SM_SHARED, CTA_SHARED, CTA_MOST = 228 << 10, 1 << 10, 227 << 10


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1410_5561_gb300", "csrc"), str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    L = ctypes.CDLL(str(d / "t.so"))
    L.prefetch.restype = ctypes.c_long
    return L


@pytest.mark.parametrize("V,bytes_", [(4, 560), (4, 832), (2, 832)])  # 25 points: BF16, FP32, FP64
def test_prefetched_25_point_rows_of_several_ctas_run_one_an_sm(lib, V, bytes_):
    for nx in range(1, 1400):
        t, m = ctypes.c_int(), ctypes.c_long()
        w = lib.prefetch(nx, V, 8, ctypes.c_long(bytes_), 1, ctypes.byref(t), ctypes.byref(m))
        ctas = -(-nx // (32 * V))
        assert 1 <= w <= 32 and w * V * ctas >= nx and w * 8 <= t.value <= 256 and t.value % 32 == 0
        assert t.value * bytes_ <= m.value <= max(256 * bytes_, SM_SHARED // 2) <= CTA_MOST
        if ctas > 1:
            assert 2 * (m.value + CTA_SHARED) > SM_SHARED, nx
