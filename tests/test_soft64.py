"""FP64 add and multiplication by integer operations against the hardware's, bit for bit, wherever the
integer form takes the operands: compiled for the host from the header that the kernels use."""
import ctypes
import subprocess
import os

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "soft64.cuh"
extern "C" void run(const double* a, const double* b, long n, double* add, double* mul, unsigned* bad) {
    for (long i = 0; i < n; ++i) {
        uint32_t p = 0, q = 0;
        add[i] = stg::soft_add(a[i], b[i], p);
        mul[i] = stg::soft_mul(stg::SoftFactor(a[i]), b[i], q);
        bad[i] = p | q << 1;
    }
}
"""
SPECIAL = [0.0, 5e-324, 2.2250738585072014e-308, 2.0 ** -960, 2.0 ** -959, 2.0 ** -53, 1.5 * 2.0 ** -53, 2.0 ** -54,
           1.0 - 2.0 ** -53, 1.0, 1.0 + 2.0 ** -52, 1.5, 2.0 ** 52, 2.0 ** 53, 2.0 ** 54, 2.0 ** 1022, 2.0 ** 1023,
           1.7976931348623157e308, np.inf, np.nan]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("soft64")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-x", "c++", "-I",
                    os.path.join(ROOT, "paper_1410_5561_gb300", "csrc"), str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


def _operands(name, rng, n=200000):
    if name == "special":
        v = np.array(SPECIAL + [-x for x in SPECIAL])
        return [x.ravel() for x in np.meshgrid(v, v)]
    if name == "field":  # what a sweep adds
        return [rng.uniform(-1, 1, n) for _ in range(2)]
    if name == "bits":
        return [rng.integers(0, 2 ** 64, n, dtype=np.uint64).view(np.float64) for _ in range(2)]
    if name == "ties":  # few significant bits, exponents up to 60 apart
        return [np.ldexp(rng.integers(-64, 64, n).astype(float), rng.integers(-30, 30, n)) for _ in range(2)]
    a = rng.uniform(-1, 1, n)  # cancellation down to a few units in the last place
    return [a, ((-a).view(np.int64) + rng.integers(-3, 4, n)).view(np.float64)]


@pytest.mark.parametrize("name", ["special", "field", "bits", "ties", "cancel"])
def test_soft_operations_give_the_hardware_bits(lib, name):
    a, b = (np.ascontiguousarray(x) for x in _operands(name, np.random.default_rng(7)))
    n = a.size
    add, mul, bad = np.empty(n), np.empty(n), np.empty(n, np.uint32)
    p = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    lib.run(p(a), p(b), ctypes.c_long(n), p(add), p(mul), p(bad))
    with np.errstate(all="ignore"):
        for got, ref, bit in ((add, a + b, 1), (mul, a * b, 2)):
            ok = (bad & bit) == 0
            assert np.array_equal(got[ok].view(np.int64), ref[ok].view(np.int64))
            if name == "field":
                assert ok.all()
