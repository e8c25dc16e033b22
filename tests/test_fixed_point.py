"""The fixed-point arithmetic of the double sampler (csrc/fixed_point.cuh, host
and device code) compiled for the host: its Box-Muller pairs against the
oracle's libm Box-Muller on the same Philox words, and its products and
conversions against Python's integers."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from oracle import mc

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1105_0542_gb300", "csrc")
SRC = r"""
#include "fixed_point.cuh"
using namespace su;
static const fx::Tables T = fx::make_tables();
extern "C" void normals(const uint32_t *w, long n, double *z) {
    for (long i = 0; i < n; ++i, w += 4) {
        int64_t a, b;
        fx::normals(((uint64_t)w[0] << 21) | (w[1] >> 11), ((uint64_t)w[2] << 21) | (w[3] >> 11), &T, a, b);
        z[2 * i] = fx::to_double(a, -fx::kZScale);
        z[2 * i + 1] = fx::to_double(b, -fx::kZScale);
    }
}
static const fx::TanhTable H = fx::make_tanh_table();
extern "C" int64_t tanh2(int64_t w) { return fx::tanh2(w, H.n); }
extern "C" int64_t mul(int64_t x, int64_t f) { return fx::mul(x, fx::limbs(f)); }
extern "C" int64_t square(int64_t x) { return fx::square(fx::limbs(x)); }
extern "C" double to_double(int64_t x, int s) { return fx::to_double(x, s); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cpp").write_text(SRC)
    so = str(d / "fx.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(d / "fx.cpp"), "-o", so],
                   check=True)
    L = ctypes.CDLL(so)
    i64 = ctypes.c_int64
    L.mul.argtypes, L.mul.restype = [i64, i64], i64
    L.square.argtypes, L.square.restype = [i64], i64
    L.tanh2.argtypes, L.tanh2.restype = [i64], i64
    L.to_double.argtypes, L.to_double.restype = [i64, ctypes.c_int], ctypes.c_double
    return L


def test_normals(lib):
    n = 4000
    w = np.array([mc.philox_words(77, 3, 1000 + i, 0) for i in range(n)], dtype=np.uint32)
    # u1 at and next to 0 and 1, u2 next to the octants' edges
    edge = [(0, 0), (0, 0x800), (0xFFFFFFFF, 0xFFFFFFFF), (0xFFFFFFFF, 0xFFFFF000), (0xBFFFFFFF, 0xFFFFFFFF), (0xC0000000, 0)]
    turn = [(0, 0), (0xFFFFFFFF, 0xFFFFFFFF)] + [(k << 29, 0) for k in range(8)] + [((k << 29) - 1, 0xFFFFFFFF) for k in range(1, 8)]
    w = np.concatenate([w, np.array([e + t for e in edge for t in turn], dtype=np.uint32)])
    z = np.empty(2 * len(w))
    lib.normals(w.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(len(w)), z.ctypes.data_as(ctypes.c_void_p))
    a = (w[:, 0].astype(np.uint64) << np.uint64(21)) | (w[:, 1].astype(np.uint64) >> np.uint64(11))
    b = (w[:, 2].astype(np.uint64) << np.uint64(21)) | (w[:, 3].astype(np.uint64) >> np.uint64(11))
    u1, u2 = (a.astype(np.float64) + 0.5) * 2.0 ** -53, (b.astype(np.float64) + 0.5) * 2.0 ** -53
    r = np.sqrt(-2 * np.log(u1))
    ref = np.stack([r * np.cos(2 * np.pi * u2), r * np.sin(2 * np.pi * u2)], axis=1).reshape(-1)
    # the reference's own rounding of 2 pi u2 (up to 2^-51) and of the logarithm, per unit of the radius
    assert np.max(np.abs(z - ref) / (1 + np.repeat(r, 2))) <= 1e-15


def test_products_and_conversions(lib):
    rng = np.random.default_rng(5)
    xs = [int(v) for v in rng.integers(-2 ** 63 + 1, 2 ** 63 - 1, 300)] + [0, 1, -1, 2 ** 63 - 1, -2 ** 63 + 1, 2 ** 32, -2 ** 32]
    fs = [int(v) for v in rng.integers(0, 2 ** 63 - 2 ** 32, 300)] + [0, 1, 2 ** 31, 2 ** 62, 2 ** 63 - 2 ** 32]
    for x in xs:
        for f in fs[::17] + fs[-5:]:
            assert -2 <= lib.mul(x, f) - x * f / 2 ** 64 <= 2 or abs(lib.mul(x, f) - (x * f >> 64)) <= 2
        if abs(x) < 2 ** 63 - 2 ** 32:
            assert 0 <= (x * x >> 64) - lib.square(x) <= 2
        assert lib.to_double(x, -57) == pytest.approx(x * 2.0 ** -57, rel=2.0 ** -53)


def test_tanh2(lib):
    """z = tanh^2(w 2^-59) in units of 2^-62 against the same in double: the
    argument's rounding to a double and tanh's own are below 4 2^-53 z."""
    rng = np.random.default_rng(6)
    ws = [int(v) for v in rng.integers(0, 384 * 2 ** 53, 2000)] + [(i << 53) + e for i in (0, 1, 63, 383) for e in (0, 1, 2 ** 53 - 1)]
    for w in ws:
        z = np.tanh(w * 2.0 ** -59) ** 2
        assert abs(lib.tanh2(w) * 2.0 ** -62 - z) <= 2.0 ** -57 + 2.0 ** -51 * z
