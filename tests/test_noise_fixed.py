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
extern "C" void pairs(const uint32_t* a, const uint32_t* b, double* out, int n)
{
    for (int i = 0; i < n; ++i)
        smerf::fx_box_muller(a[i], b[i], smerf::kFxLog[smerf::fx_log_index(a[i])], out[2 * i], out[2 * i + 1]);
}
"""


@pytest.fixture(scope="module")
def pairs(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    src, lib = str(d / "pairs.cpp"), str(d / "pairs.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, src, "-o", lib], check=True)
    L = ctypes.CDLL(lib)

    def call(a, b):
        out = np.zeros((len(a), 2))
        p = [v.ctypes.data_as(ctypes.c_void_p) for v in (a, b, out)]
        L.pairs(p[0], p[1], p[2], len(a))
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
