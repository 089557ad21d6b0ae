"""The FP64 mode's ring FFT in 64-bit fixed point (csrc/smerf_fixed.cuh), compiled for the host: whole
transforms by the passes of grp_fx_c2r, against long double sums, beside the same passes in FP64 with
correctly rounded factors."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1709_10314_gb300", "csrc")
SOURCE = r"""
#include <complex>
#include <cstring>
#include <vector>
#include "smerf_fixed.cuh"
using namespace smerf;
typedef long double ld;
struct fxc { int64_t x, y; };
static uint64_t bits(double v) { uint64_t b; memcpy(&b, &v, 8); return b; }
static double back(uint64_t b) { double v; memcpy(&v, &b, 8); return v; }
static fxc add(fxc a, fxc b) { return {a.x + b.x, a.y + b.y}; }
static fxc sub(fxc a, fxc b) { return {a.x - b.x, a.y - b.y}; }
static fxc conj(fxc a) { return {a.x, -a.y}; }
static fxc muli(fxc a) { return {-a.y, a.x}; }
static fxc mul(fxc a, int64_t k, int lgn, int d)  // by e^{2 pi i k / 2^lgn}
{
    int64_t c, s;
    int32_t ch, cl, sh, sl;
    fx_cis62((uint64_t)k << (64 - lgn), c, s);
    fx_split(c, ch, cl), fx_split(s, sh, sl);
    return fx_cmul(a, ch, cl, sh, sl, d);
}
typedef std::complex<double> cd;
static cd root(int64_t k, int lgn) { ld t = 2 * 3.14159265358979323846264338327950288L * k / ((ld)(1ll << lgn)); return cd((double)cosl(t), (double)sinl(t)); }

extern "C" double to_double(int64_t x, int S) { return back(fx_to_double(x, S)); }
// g: 2^lg coefficients (slot 0 = g_0, Re g_M); fx, fp: the ring's 2^(lg + 1) values; returns the largest
// |component| of any intermediate value over 2^62
extern "C" double transform(const double* g, int lg, double* fx, double* fp)
{
    const int N = 1 << lg;
    int top = 0;
    unsigned sum = 0;
    for (int i = 0; i < 2 * N; ++i) { int e = (int)((bits(g[i]) >> 52) & 0x7ff); if (e > top) top = e; }
    for (int i = 0; i < 2 * N; ++i) sum += fx_share((uint32_t)(bits(g[i]) >> 32) & 0x7fffffffu, top) + 1u;
    const bool flat = lg <= 7;  // one unit for the whole transform (kFxFlat)
    const int spread = fx_spread(sum), S = fx_unit(top, spread, flat ? lg : 2);
    std::vector<fxc> X(N), Y(N);
    std::vector<cd> A(N), B(N);
    double worst = 0;
    auto see = [&](fxc v) { worst = fmax(worst, fmax(fabs((double)v.x), fabs((double)v.y)) * 0x1p-62); };
    auto get = [&](int i) { return fxc{fx_from_double(bits(g[2 * i]), S), fx_from_double(bits(g[2 * i + 1]), S)}; };
    for (int s = 0; s <= N / 2; ++s) {
        const fxc a = get(s);
        const cd u(g[2 * s], g[2 * s + 1]);
        if (s == 0) { X[0] = {a.x + a.y, a.x - a.y}; A[0] = cd(u.real() + u.imag(), u.real() - u.imag()); continue; }
        const fxc b = conj(get(N - s));
        const fxc e = add(a, b), o = muli(mul(sub(a, b), s, lg + 1, 0));
        X[s] = add(e, o);
        if (2 * s < N) X[N - s] = conj(sub(e, o));
        const cd v = std::conj(cd(g[2 * (N - s)], g[2 * (N - s) + 1])), ee = u + v, oo = cd(0, 1) * (root(s, lg + 1) * (u - v));
        A[s] = ee + oo;
        if (2 * s < N) A[N - s] = std::conj(ee - oo);
    }
    for (int s = 0; s < N; ++s) see(X[s]);
    for (int ln = 0; ln < lg;) {
        const int LR = lg - ln >= 2 ? 2 : 1, R = 1 << LR, Ns = 1 << ln, nb = N >> LR, d = ln && !flat ? fx_shift(spread, ln, LR) : 0;
        for (int j = 0; j < nb; ++j) {
            const int kk = j & (Ns - 1), idx = ((j - kk) << LR) + kk;
            fxc v[4];
            cd w[4];
            for (int i = 0; i < R; ++i) {
                v[i] = X[j + i * nb];
                w[i] = A[j + i * nb];
                if (ln) v[i] = i ? mul(v[i], (int64_t)i * kk, ln + LR, d) : fx_cshift(v[i], d);
                if (ln && i) w[i] *= root((int64_t)i * kk, ln + LR);
            }
            if (R == 4) {
                const fxc p = add(v[0], v[2]), q = sub(v[0], v[2]), r = add(v[1], v[3]), t = muli(sub(v[1], v[3]));
                v[0] = add(p, r), v[1] = add(q, t), v[2] = sub(p, r), v[3] = sub(q, t);
                const cd P = w[0] + w[2], Q = w[0] - w[2], T = w[1] + w[3], U = w[1] - w[3], W(-U.imag(), U.real());
                w[0] = P + T, w[1] = Q + W, w[2] = P - T, w[3] = Q - W;
            } else {
                const fxc p = v[0];
                v[0] = add(p, v[1]), v[1] = sub(p, v[1]);
                const cd P = w[0];
                w[0] = P + w[1], w[1] = P - w[1];
            }
            for (int i = 0; i < R; ++i) { Y[idx + i * Ns] = v[i]; see(v[i]); B[idx + i * Ns] = w[i]; }
        }
        X.swap(Y), A.swap(B);
        ln += LR;
    }
    const int E = fx_unit(top, spread, lg);
    for (int s = 0; s < N; ++s) {
        fx[2 * s] = back(fx_to_double(X[s].x, E)), fx[2 * s + 1] = back(fx_to_double(X[s].y, E));
        fp[2 * s] = A[s].real(), fp[2 * s + 1] = A[s].imag();
    }
    return worst;
}
// squared deviations of fx and fp from the ring's exact values, and the values' own square, over every
// step-th point
extern "C" void errors(const double* g, int lg, const double* fx, const double* fp, int step, double* out)
{
    const int N = 1 << lg, n = 2 * N;
    std::vector<ld> c(n), s(n);
    for (int i = 0; i < n; ++i) { ld t = 2 * 3.14159265358979323846264338327950288L * i / n; c[i] = cosl(t), s[i] = sinl(t); }
    out[0] = out[1] = out[2] = 0;
    for (int j = 0; j < n; j += step) {
        ld v = g[0] + (j & 1 ? -(ld)g[1] : (ld)g[1]);
        for (int m = 1; m < N; ++m) {
            const int k = (int)((int64_t)m * j % n);
            v += 2 * (g[2 * m] * c[k] - g[2 * m + 1] * s[k]);
        }
        out[0] += (double)((fx[j] - v) * (fx[j] - v)), out[1] += (double)((fp[j] - v) * (fp[j] - v)), out[2] += (double)(v * v);
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed_fft")
    src, so = str(d / "fft.cpp"), str(d / "fft.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, src, "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.transform.restype = ctypes.c_double
    return L


def _p(v):
    return v.ctypes.data_as(ctypes.c_void_p)


def _transform(lib, g):
    """Squared errors of the fixed-point and the FP64 ring relative to its square, the largest value."""
    g = np.ascontiguousarray(g, dtype=np.float64).ravel()
    lg = int(np.log2(len(g) // 2))
    fx, fp, out = np.zeros(len(g)), np.zeros(len(g)), np.zeros(3)
    largest = lib.transform(_p(g), lg, _p(fx), _p(fp))
    lib.errors(_p(g), lg, _p(fx), _p(fp), 1 if lg < 9 else 2 ** (lg - 8) - 1, _p(out))
    return out[0] / out[2], out[1] / out[2], largest


@pytest.mark.parametrize("lg", range(2, 13))
@pytest.mark.parametrize("falling", [0.0, 0.5, 1.0, 2.0, 6.0])
def test_whole_transforms_err_no_more_than_fp64(lib, lg, falling):
    """Rings of 8 to 8192 points whose coefficients are flat or fall as m^-falling (a field's spectrum
    below and above kappa): the error is not above that of the same passes in FP64."""
    rng, N, fx, fp = np.random.default_rng(lg), 1 << lg, 0.0, 0.0
    for _ in range(4):
        e = _transform(lib, rng.normal(size=(N, 2)) * (1.0 + np.arange(N))[:, None] ** -falling * 2.0 ** rng.integers(-300, 300))
        fx, fp = fx + e[0], fp + e[1]
        assert e[2] < 1
    assert fx <= fp


@pytest.mark.parametrize("lg", [2, 3, 5, 6, 8, 11, 12])
def test_values_stay_below_the_bound(lib, lg):
    """Coefficients of the largest magnitude below a power of two, aligned to add up in one place or to stay
    apart, and a single one."""
    rng, N, big = np.random.default_rng(lg), 1 << lg, 2 - 2.0 ** -52
    k = np.arange(N) * (2 * np.pi * 3 / (2 * N))
    cases = [np.full((N, 2), big), np.full((N, 2), big) * [1, -1], np.stack([np.cos(k), np.sin(k)], 1)]
    cases += [big * (np.arange(N) == i)[:, None] * np.ones(2) for i in (0, 1, N // 2, N - 1)]
    cases += [rng.choice([-big, big, 0.0, 0.5], size=(N, 2)) + [[1e-9, 0]] for _ in range(20)]
    for g in cases:
        fx, fp, largest = _transform(lib, g)
        assert largest < 1 and fx < 2 * fp + 2.0 ** -106


def test_overflow_is_infinity(lib):
    """Fixed point to doubles at the top of their range: the largest finite value, then infinities."""
    lib.to_double.restype = ctypes.c_double
    one = lambda x, S: lib.to_double(ctypes.c_int64(x), S)  # noqa: E731
    assert one(2 ** 62, -961) == 2.0 ** 1023 and one(-2 ** 62, -961) == -2.0 ** 1023
    assert one(2 ** 53 - 1, -971) == np.finfo(np.float64).max
    for x, S in ((2 ** 62, -962), (2 ** 62 - 1, -962), (2 ** 62, -1500), (2 ** 61, -964)):
        assert one(x, S) == np.inf and one(-x, S) == -np.inf
