"""The two forms of the word conversions (csrc/od_arith.cuh), with branches for
passes over a field and by selection for redone cells, on the host: the same
words and values for every kind of double."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_12734_gb300", "csrc")

SOURCE = """
#include "od_arith.cuh"
extern "C" int64_t differ(const double *x, int64_t n, uint32_t e0) {
    int64_t bad = 0;
    for (int64_t i = 0; i < n; ++i) {
        const uint64_t w = od::fx_encode(x[i], e0);
        bad += w != od::fx_encode_any(x[i], e0);
        bad += od::f64_bits(od::fx_decode(w, e0)) != od::f64_bits(od::fx_decode_any(w, e0));
        bad += od::f64_bits(od::fx_decode_any(w, e0)) != od::f64_bits(x[i]);
    }
    return bad;
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("forms")
    (d / "f.cpp").write_text(SOURCE)
    so = str(d / "f.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(d / "f.cpp"), "-o",
                    so], check=True)
    lib = ctypes.CDLL(so)
    lib.differ.restype = ctypes.c_int64
    return lib


@pytest.mark.parametrize("e0", [0, 1, 2, 248, 255, 256, 1015, 1016, 1700, 1772])
def test_both_forms_agree(fx, e0):
    rng = np.random.default_rng(e0)
    n = 400000
    # every exponent of both signs but the positive ones that a field of words does not hold
    top = 1790 if e0 else 2048
    e = rng.integers(0, top, n).astype(np.uint64)
    neg = rng.random(n) < 0.3
    e[neg] = rng.integers(0, 2048, int(neg.sum())).astype(np.uint64)
    m = rng.integers(0, 1 << 52, n).astype(np.uint64)
    m[::7] = 0
    m[1::7] = (1 << 52) - 1
    b = (neg.astype(np.uint64) << np.uint64(63)) | (e << np.uint64(52)) | m
    b[:4] = [0, 1 << 63, 0x7FF0000000000000, 0x7FF8000000000000]  # zeros, infinity, NaN
    assert fx.differ(b.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(n), ctypes.c_uint32(e0)) == 0
