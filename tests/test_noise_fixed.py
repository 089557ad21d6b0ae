"""The FP64 mode's Box-Muller in 64-bit fixed point (csrc/smerf_fixed.cuh), compiled for the host,
against 160-bit arithmetic at the words' extremes (u0 next to 0 and 1 and to every power of two,
every octant's edges of u1) and at random words: correctly scaled, within 0.52 units in the last
place (0.5 of rounding, 2^-59 of the fixed-point steps)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1709_10314_gb300", "csrc")
SOURCE = """
#include "smerf_fixed.cuh"
extern "C" void products(const int64_t* a, const uint64_t* turns, int64_t* out, int n)
{
    for (int i = 0; i < n; ++i) {
        int64_t c, s;
        int32_t axh, axl, ayh, ayl, ch, cl, sh, sl;
        smerf::fx_cis62(turns[i], c, s);
        smerf::fx_split(a[2 * i], axh, axl), smerf::fx_split(a[2 * i + 1], ayh, ayl);
        smerf::fx_split(c, ch, cl), smerf::fx_split(s, sh, sl);
        out[4 * i] = smerf::fx_dot<true>(axh, axl, ch, cl, ayh, ayl, sh, sl);
        out[4 * i + 1] = smerf::fx_dot<false>(axh, axl, sh, sl, ayh, ayl, ch, cl);
        out[4 * i + 2] = c, out[4 * i + 3] = s;
    }
}
extern "C" void round_trip(const uint64_t* d, const int* S, int64_t* fixed, uint64_t* back, int n)
{
    for (int i = 0; i < n; ++i) fixed[i] = smerf::fx_from_double(d[i], S[i]), back[i] = smerf::fx_to_double(fixed[i], S[i]);
}
extern "C" void pairs(const uint32_t* a, const uint32_t* b, double* out, int n)
{
    for (int i = 0; i < n; ++i)
        smerf::fx_box_muller(a[i], b[i], smerf::kFxLog[smerf::fx_log_index(a[i])], out[2 * i], out[2 * i + 1]);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    src, lib = str(d / "pairs.cpp"), str(d / "pairs.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, src, "-o", lib], check=True)
    return ctypes.CDLL(lib)


def _p(v):
    return v.ctypes.data_as(ctypes.c_void_p)


@pytest.fixture(scope="module")
def pairs(lib):
    def call(a, b):
        out = np.zeros((len(a), 2))
        lib.pairs(_p(a), _p(b), _p(out), len(a))
        return out
    return call


def _worst_ulp(pairs, a, b):
    with mp.workprec(160):
        out, worst = pairs(a, b), 0.0
        for i in range(len(a)):
            r = mp.sqrt(-2 * mp.log((2 * mp.mpf(int(a[i])) + 1) / mp.mpf(2) ** 33))
            t = mp.pi * (2 * mp.mpf(int(b[i])) + 1) / mp.mpf(2) ** 32
            for got, want in zip(out[i], (r * mp.cos(t), r * mp.sin(t))):
                ulp = mp.mpf(2) ** (mp.floor(mp.log(abs(want), 2)) - 52)
                worst = max(worst, float(abs(mp.mpf(float(got)) - want) / ulp))
    return worst


def test_words_extremes(pairs):
    ends = {0, 1, 2 ** 32 - 1} | {2 ** k + d for k in range(32) for d in (-1, 0, 1)} | {2 ** 32 - 2 ** k for k in range(32)}
    a = sorted(v for v in ends if 0 <= v < 2 ** 32)
    b = sorted({o * 2 ** 29 + d for o in range(8) for d in (0, 1, 2 ** 28 - 1, 2 ** 28, 2 ** 29 - 1)})
    pick = [(x, b[(7 * i + j) % len(b)]) for i, x in enumerate(a) for j in range(6)] + [(x, y) for y in b for x in (0, 77, 2 ** 32 - 1)]
    A, B = (np.array(v, dtype=np.uint32) for v in zip(*pick))
    assert _worst_ulp(pairs, A, B) < 0.52


def test_log_table_edges(pairs):
    # the 64 intervals of the logarithm's table: both ends of each, at u0 near 1/2 .. 1 and lower
    a = [v for i in range(65) for s in (0, 5) for v in ((2 ** 31 + i * 2 ** 25 - 1) >> s, (2 ** 31 + i * 2 ** 25) >> s) if v < 2 ** 32]
    A = np.array(a, dtype=np.uint32)
    B = (np.arange(len(a), dtype=np.uint64) * 2654435761 % 2 ** 32).astype(np.uint32)
    assert _worst_ulp(pairs, A, B) < 0.52


def test_random_words(pairs):
    w = np.random.default_rng(3).integers(0, 2 ** 32, (2, 1500), dtype=np.uint64).astype(np.uint32)
    assert _worst_ulp(pairs, np.ascontiguousarray(w[0]), np.ascontiguousarray(w[1])) < 0.52


def test_fixed_point_complex_products(lib):
    """The FP64 FFT's products a e^{2 pi i p} in 64-bit fixed point, |a| < 2^62: factors to one unit of
    2^-62, products to three (half a unit of rounding, the dropped low words' products of up to half a
    unit each, the factor's own error), at random values, at the words' sign edges and on the axes."""
    rng = np.random.default_rng(8)
    r, t = 2.0 ** rng.uniform(0, 61.99, 4000), rng.uniform(0, 2 * np.pi, 4000)
    a = np.stack([r * np.cos(t), r * np.sin(t)], 1).astype(np.int64)
    a[:1000] = (a[:1000] & ~np.int64(0xFFFFFFFF)) | rng.choice([0, 1, 0x7FFFFFFF, 0x80000000, 0xFFFFFFFF], (1000, 2))
    a[:8] = [(2 ** 62 - 1, 0), (0, 1 - 2 ** 62), (-2 ** 31, 2 ** 31), (2 ** 61, -2 ** 61), (0, 0), (-1, 1), (1, 0), (0, -1)]
    turns = rng.integers(0, 2 ** 64, 4000, dtype=np.uint64)
    turns[::5] = (np.arange(800, dtype=np.uint64) * np.uint64(2 ** 55)) << np.uint64(1)
    out = np.zeros((4000, 4), dtype=np.int64)
    lib.products(_p(a), _p(turns), _p(out), 4000)
    with mp.workprec(200):
        for i in range(4000):
            w = mp.expjpi(2 * mp.mpf(int(turns[i])) / mp.mpf(2) ** 64)
            assert abs(int(out[i, 2]) - w.real * 2 ** 62) <= 1 and abs(int(out[i, 3]) - w.imag * 2 ** 62) <= 1
            z = mp.mpc(int(a[i, 0]), int(a[i, 1])) * w
            assert abs(int(out[i, 0]) - z.real) <= 3 and abs(int(out[i, 1]) - z.imag) <= 3


def test_fixed_point_round_trip(lib):
    """Doubles to fixed point and back at every scale the FFT takes (|v| 2^S < 2^60): within half a
    unit, exact when the unit reaches the last bit, zeros and tiny values to zero."""
    rng = np.random.default_rng(9)
    S = rng.integers(-400, 900, 3000).astype(np.int32)
    v = rng.uniform(1, 2, 3000) * 2.0 ** (59 - S - rng.integers(0, 70, 3000)) * rng.choice([-1.0, 1.0], 3000)
    v[:4] = [0.0, -0.0, 5e-324, 2.0 ** -1022]
    S[:4] = 60
    fixed, back = np.zeros(3000, np.int64), np.zeros(3000, np.float64)
    lib.round_trip(_p(v), _p(S), _p(fixed), _p(back), 3000)
    for i in range(3000):
        exact = mp.mpf(float(v[i])) * mp.mpf(2) ** int(S[i])
        assert abs(int(fixed[i]) - exact) <= mp.mpf(1) / 2
        assert back[i] == float(mp.mpf(int(fixed[i])) / mp.mpf(2) ** int(S[i]))
