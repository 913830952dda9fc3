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
extern "C" int split(int ny, long rows, long units, long* xblocks, long* seg) {
    const stg::CopySplit c = stg::copy_split(ny, rows, units);
    *xblocks = c.xblocks;
    *seg = (long)c.seg;
    return c.lg;
}
extern "C" int early(long ctas, int slots, int planes) { return stg::early_fp64(ctas, slots, planes) ? 1 : 0; }
extern "C" long want() { return (long)stg::COPY_WANT; }
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


@pytest.mark.parametrize("ny", [1, 2, 3, 4, 7, 8, 9, 33, 4000])
@pytest.mark.parametrize("nz", [1, 2, 5, 3000])
def test_copies_cover_every_row_once_with_warps_for_the_gpu(lib, ny, nz):
    """Segments of a row follow one another and end with it, rows of a CTA likewise; few rows give as
    many warps as the GPU wants, or as there are passes of a warp; many rows are not cut."""
    lib.want.restype = ctypes.c_long
    for units in (1, 2, 31, 127, 128, 129, 1000, 4097, 20000, 250000, 1 << 21):
        xb, seg = ctypes.c_long(), ctypes.c_long()
        lg = lib.split(ny, ctypes.c_long(ny * nz), ctypes.c_long(units), ctypes.byref(xb), ctypes.byref(seg))
        per, seg, xb = 8 >> lg, seg.value, xb.value
        assert 1 << lg <= max(ny, 1) and (1 << lg) * per == 8
        segs = -(-units // seg)
        assert (xb - 1) * per < segs <= xb * per and -(-ny // (1 << lg)) * xb < 2 ** 31
        passes = -(-units // 128)
        assert seg % 128 == 0
        assert 2 * ny * nz * segs >= min(lib.want(), ny * nz * passes)
        if ny * nz >= lib.want():
            assert segs == 1


@pytest.mark.parametrize("ctas,slots,planes,want", [
    (232, 456, 29, 0), (375, 608, 30, 0), (432, 608, 16, 0), (483, 608, 14, 0),  # measured 0.76 to 0.98 when early
    (608, 608, 23, 1), (505, 608, 21, 1), (570, 760, 2, 1), (513, 608, 1, 1), (41, 608, 1, 1),
    (609, 608, 1, 0), (1200, 608, 30, 0),  # several waves
])
def test_fp64_steps_set_up_early(lib, ctas, slots, planes, want):
    assert lib.early(ctypes.c_long(ctas), slots, planes) == want
