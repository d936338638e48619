"""The arithmetic of fixed-point field words (csrc/od_arith.cuh) on the host:
the words of a double and back, and every update that stays in the window
against the IEEE operations, bit for bit.  The routines are the same source
that the kernels compile."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_12734_gb300", "csrc")

SOURCE = """
#include "od_arith.cuh"
extern "C" {
void words(const double *x, int64_t n, uint32_t e0, uint64_t *w, double *back) {
    for (int64_t i = 0; i < n; ++i) { w[i] = od::fx_encode(x[i], e0); back[i] = od::fx_decode(w[i], e0); }
}
// dims 3: six operands an element, 2: four; ok[i] = 1 where the update stays in the window
void update(int dims, const double *x, int64_t n, uint32_t e0, double *out, uint8_t *ok) {
    const int k = dims == 3 ? 6 : 4;
    for (int64_t i = 0; i < n; ++i) {
        uint64_t w[6];
        for (int j = 0; j < k; ++j) w[j] = od::fx_encode(x[k * i + j], e0);
        bool good;
        const uint64_t q = dims == 3 ? od::fx_update3(w[0], w[1], w[2], w[3], w[4], w[5], good)
                                     : od::fx_update2(w[0], w[1], w[2], w[3], good);
        out[i] = od::fx_decode(q, e0);
        ok[i] = good;
    }
}
uint32_t anchor(uint64_t vmax) { return od::fx_anchor(vmax); }
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("words")
    src, so = str(d / "words.cpp"), str(d / "words.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, src, "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def bits(x):
    return np.ascontiguousarray(x).view(np.uint64)


def words(fx, x, e0):
    w, back = np.empty(x.size, np.uint64), np.empty(x.size)
    fx.words(x.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(x.size), ctypes.c_uint32(e0),
             w.ctypes.data_as(ctypes.c_void_p), back.ctypes.data_as(ctypes.c_void_p))
    return w, back


def update(fx, dims, x, e0):
    n = x.size // (6 if dims == 3 else 4)
    out, ok = np.empty(n), np.empty(n, np.uint8)
    fx.update(ctypes.c_int(dims), x.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(n), ctypes.c_uint32(e0),
              out.ctypes.data_as(ctypes.c_void_p), ok.ctypes.data_as(ctypes.c_void_p))
    return out, ok.astype(bool)


def significands(rng, n):
    """53-bit significands: random, few bits set, runs of ones, the ends."""
    m = rng.integers(0, 2 ** 52, n, dtype=np.uint64)
    kind = rng.integers(0, 5, n)
    sh = rng.integers(0, 52, n, dtype=np.uint64)
    ones = np.uint64(2 ** 52 - 1)
    m = np.where(kind == 1, (m >> sh) << sh, m)
    m = np.where(kind == 2, m | (ones >> sh), m)
    m = np.where(kind == 3, m & np.uint64(3), m)
    return np.where(kind == 4, ones - (m & np.uint64(3)), m)


@pytest.mark.parametrize("e0", [1, 4, 250, 256, 1015, 1772])
def test_words_round_trip(fx, e0):
    rng = np.random.default_rng(e0)
    n = 200000
    # every exponent but the positive ones that stand for the tiny values
    e = rng.integers(0, 1790, n, dtype=np.uint64)
    neg = rng.integers(0, 2, n, dtype=np.uint64)
    e = np.where(neg == 1, rng.integers(0, 2048, n, dtype=np.uint64), e)
    x = ((neg << np.uint64(63)) | (e << np.uint64(52)) | significands(rng, n)).view(np.float64)
    special = np.array([0.0, -0.0, 5e-324, -5e-324, 2.2250738585072014e-308, np.inf, -np.inf,
                        2.0 ** (e0 - 1023), np.nextafter(2.0 ** (e0 + 8 - 1023), 0.0)])
    x = np.concatenate([x, special])
    w, back = words(fx, x, e0)
    assert np.array_equal(bits(back), bits(x))
    ex = bits(x) >> np.uint64(52)
    inside = (ex >= e0) & (ex <= e0 + 7)
    small = (w >> np.uint64(60)) == 0
    assert np.array_equal(small, inside | (bits(x) == 0))  # only window words and zero have no top bits


@pytest.mark.parametrize("dims", [2, 3])
@pytest.mark.parametrize("spread", [1, 2, 5, 8])
def test_updates_in_the_window(fx, dims, spread):
    rng = np.random.default_rng(100 * dims + spread)
    k, n, e0 = (6, 400000, 1015) if dims == 3 else (4, 400000, 1015)
    e = np.uint64(e0) + rng.integers(0, spread, n * k, dtype=np.uint64)
    x = ((e << np.uint64(52)) | significands(rng, n * k)).view(np.float64)
    x[rng.integers(0, 20, n * k) == 0] = 0.0
    x[: 6 * k] = 0.0  # whole cells of zeros
    out, ok = update(fx, dims, x, e0)
    v = x.reshape(n, k)
    s = v[:, 0] + v[:, 1]
    for j in range(2, k):
        s = s + v[:, j]
    want = s / float(k)
    exp = bits(want) >> np.uint64(52)
    # the fast form applies exactly when the quotient lies in the window or is zero
    assert np.array_equal(ok, (exp >= e0) | (want == 0.0))
    assert np.array_equal(bits(out[ok]), bits(want[ok]))


def test_updates_leave_the_window_flagged(fx):
    # one operand outside: negative, infinite, NaN, too large, too small, subnormal
    e0 = 1015
    for bad in (-0.5, np.inf, np.nan, 1.0, 2.0 ** -9, 5e-324, -0.0, 1e300):
        for pos in range(6):
            x = np.full(6, 0.5)
            x[pos] = bad
            assert not update(fx, 3, x, e0)[1][0], (bad, pos)
        for pos in range(4):
            x = np.full(4, 0.5)
            x[pos] = bad
            assert not update(fx, 2, x, e0)[1][0], (bad, pos)


def test_anchor(fx):
    def anchor(x):
        return fx.anchor(ctypes.c_uint64(int(bits(np.array([x]))[0])))
    fx.anchor.restype = ctypes.c_uint32
    assert anchor(np.nextafter(1.0, 0.0)) == 1015 and anchor(1.0) == 1016  # the window's top binade holds the maximum
    assert anchor(0.0) == 1 and anchor(5e-324) == 1 and anchor(2.0 ** -1015) == 1
    assert anchor(2.0 ** 756) == 1772 and anchor(2.0 ** 757) == 0 and anchor(1e308) == 0
