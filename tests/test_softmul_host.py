"""The integer products of the particle gather (softmul.cuh, compiled here with the host compiler)
against the processor's FP64 operations, bit for bit: weights f, 1 - f and their products, and a
weight times any double that the function takes."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = """
#include "softmul.cuh"
using namespace saamg;
// bits of the weight w(f0) w(f1) w(f2), each f or 1 - f by the bits of `side`
static Unpacked weight(const uint64_t* f, int side) {
  Unpacked u[3];
  for (int k = 0; k < 3; ++k)
    u[k] = (side >> k) & 1 ? unpack_fraction(f[k]) : unpack_complement(f[k]);
  return mul_unpacked(mul_unpacked(u[0], u[1]), u[2]);
}
extern "C" void weights(int n, const uint64_t* f, int side, uint64_t* out) {
  for (int i = 0; i < n; ++i) out[i] = pack_bits(weight(f + 3 * i, side));
}
extern "C" void products(int n, const uint64_t* f, int side, const uint64_t* v, uint64_t* out,
                         uint8_t* ok) {
  for (int i = 0; i < n; ++i) {
    bool o = false;
    out[i] = mul_bits(weight(f + 3 * i, side), v[i], o);
    ok[i] = o;
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("softmul")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_0907_4863_gb300", "csrc"), str(d / "shim.cpp"), "-o",
                    str(d / "shim.so")], check=True)
    return C.CDLL(str(d / "shim.so"))


def fractions(rng, n):
    """Fractions in units of 2^-64 with at most 53 significant bits, as the gather forms them from
    coordinates that are 0 or at least 2^-11: random ones, 0, the least, neighbours of 1/2 and 1,
    few and many bits."""
    k = rng.integers(0, 12, n).astype(np.uint64)
    f = (rng.integers(1 << 52, 1 << 53, n, dtype=np.uint64) << np.uint64(11)) >> k
    f &= ~np.uint64(0) << (np.uint64(11) - np.minimum(k, np.uint64(11)))
    for share, values in ((40, [0, 1 << 63, 1 << 11, 3 << 11, (1 << 64) - (1 << 11), 1 << 53,
                                (1 << 63) - (1 << 11), (1 << 63) + (1 << 11), 1 << 62, 3 << 62]),):
        pick = rng.integers(0, share, n)
        for q, v in enumerate(values):
            f[pick == q] = np.uint64(v)
    short = rng.integers(0, 8, n) == 0
    f[short] &= ~np.uint64(0) << np.uint64(50)
    return f


def as_double(f):
    return np.ldexp(f.astype(np.float64), -64)


def native_weight(f, side):
    with np.errstate(all="ignore"):
        w = [as_double(f[:, k]) if (side >> k) & 1 else 1.0 - as_double(f[:, k]) for k in range(3)]
        return (w[0] * w[1]) * w[2]


def ptr(a):
    return a.ctypes.data_as(C.c_void_p)


@pytest.mark.parametrize("side", range(8))
def test_weights(lib, side):
    rng = np.random.default_rng(side)
    n = 200_000
    f = np.ascontiguousarray(fractions(rng, 3 * n).reshape(n, 3))
    assert np.array_equal(as_double(f).astype(np.longdouble) * 2.0 ** 64, f.astype(np.longdouble))
    out = np.empty(n, np.uint64)
    lib.weights(n, ptr(f), side, ptr(out))
    assert np.array_equal(out, native_weight(f, side).view(np.uint64))


@pytest.mark.parametrize("side", range(8))
def test_products(lib, side):
    rng = np.random.default_rng(100 + side)
    n = 200_000
    f = np.ascontiguousarray(fractions(rng, 3 * n).reshape(n, 3))
    v = rng.standard_normal(n)
    anybits = rng.integers(0, 3, n) == 0
    v[anybits] = rng.integers(0, 1 << 64, n, dtype=np.uint64).view(np.float64)[anybits]
    pick = rng.integers(0, 40, n)
    tiny = np.finfo(np.float64).tiny
    for q, x in enumerate([0.0, -0.0, 5e-324, -1e-310, tiny, -tiny, 2.0 * tiny, 1e-300,
                           np.finfo(np.float64).max, -1.7e308, np.inf, -np.inf, np.nan, 1.0, -2.0]):
        v[pick == q] = x
    out, ok = np.empty(n, np.uint64), np.empty(n, np.uint8)
    lib.products(n, ptr(f), side, ptr(v.view(np.uint64)), ptr(out), ptr(ok))
    w = native_weight(f, side)
    with np.errstate(all="ignore"):
        ref = w * v
    ok = ok != 0
    # a product by a zero v is +0 here, of either sign in FP64
    assert np.all(out[ok & (v == 0.0)] == 0) and np.all(ok[v == 0.0])
    same = ok & (v != 0.0)
    assert np.array_equal(out[same], ref.view(np.uint64)[same])
    # what it must not take: operands and products that are not normal numbers
    assert not np.any(ok & ~np.isfinite(v)) and not np.any(ok & (v != 0.0) & (np.abs(v) < tiny))
    assert not np.any(ok & (v != 0.0) & ((w == 0.0) | (np.abs(ref) < tiny)))
    # and what it has to: normal numbers with a product away from the ends of the range
    plain = (w != 0.0) & (np.abs(v) > 1e-200) & (np.abs(v) < 1e300)
    assert np.all(ok[plain])
