// smerf_fixed.cuh -- Box-Muller in 64-bit fixed point for the FP64 recursion mode.
//
// GB300 has 2 FP64 lanes per SM beside 128 integer lanes, so a logarithm, a square root and a
// sine / cosine in FP64 (about 70 FP64 instructions per pair of normals) kept the FP64 pipe of the
// sampling kernels 85 % busy, two thirds of it on noise.  Here the pair is formed on the integer
// lanes, exact words in, correctly scaled doubles out, with no FP64 instruction: polynomials in
// 64-bit fixed point (their high-order terms, below 2^-24 of the result, in 32 bits), a 64-entry
// table for the logarithm (Tang, "Table-driven implementation of the logarithm function in IEEE
// floating-point arithmetic", ACM TOMS 16, 1990: c ~ 1/f from the leading bits, then the
// logarithm of c f = 1 - z by its series), and Newton's iteration for the square root.  Every
// quantity keeps at least 60 significant bits (the small radius near u0 = 1 and the small sine
// included), so a normal is within 0.51 units in the last place of its exact value.
// 1024 x 2048, p = 2, 16 realisations: 6.92 -> 2.27 ms a call; 20001 realisations of 32 x 64:
// 10.9 -> 5.36 ms; 64 x 128, p = 1, Alg. 2's order: 205 -> 166 us; the error of the fields
// against 64-bit references is unchanged (8.7e-13, 3.9e-15, 3.5e-15).  With the fixed-point ring FFT
// (grp_fx_c2r) and the band kernel the same calls take 1.34 ms, 2.03 ms and 24.6 us.
// Plain integer code: it compiles for the host too, where the tests hold it against long
// arithmetic at the words' extremes.
#pragma once

#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define SMERF_HD __host__ __device__ __forceinline__
#else
#define SMERF_HD inline
#endif

namespace smerf {

SMERF_HD uint64_t fx_mulhi(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
// the same without the low words' product: 0 to 2 below the exact high word, with three of the four
// widening multiplies (32 per SM and clock) and half of the carries.  For everything whose last
// bits do not count
SMERF_HD uint64_t fx_mulh(uint64_t a, uint64_t b)
{
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    return (uint64_t)ah * bh + (uint32_t)(((uint64_t)ah * bl) >> 32) + (uint32_t)(((uint64_t)al * bh) >> 32);
}
SMERF_HD uint32_t fx_mulhi(uint32_t a, uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
SMERF_HD int fx_clz(uint64_t a)  // a != 0
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)a);
#else
    return __builtin_clzll(a);
#endif
}
SMERF_HD double fx_double(uint64_t bits)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)bits);
#else
    union { uint64_t u; double d; } v;
    v.u = bits;
    return v.d;
#endif
}

// c_i = C 2^-16, the largest such value with c_i f <= 1 on f in [1/2 + i/128, 1/2 + (i+1)/128)
// (so z = 1 - c_i f is in [0, 0.0154)), and ln c_i as a 64-bit fraction
struct alignas(16) FxLog { uint32_t c; uint64_t l; };
#ifdef __CUDACC__
__device__
#endif
static const FxLog kFxLog[64] = {
    {0x1f81f, 0xad79c0e1a9ccfbbbull}, {0x1f07c, 0xa99161343342b993ull}, {0x1e913, 0xa5b7dd7cb7fefb85ull}, {0x1e1e1, 0xa1ec8797acfe1db1ull},
    {0x1dae6, 0x9e303c61b5f5a919ull}, {0x1d41d, 0x9a81216ce9dc2dd3ull}, {0x1cd85, 0x96df70bd80681549ull}, {0x1c71c, 0x934ad0899edc926dull},
    {0x1c0e0, 0x8fc2dafe28b2c589ull}, {0x1bacf, 0x8c471e07841d3010ull}, {0x1b4e8, 0x88d7b11e3a553cd7ull}, {0x1af28, 0x857377167aa7d0c6ull},
    {0x1a98e, 0x821a71f3855556f7ull}, {0x1a41a, 0x7ecd3abde602106cull}, {0x19ec8, 0x7b89f55aa7cf84caull}, {0x19999, 0x7851c8688a9b31d3ull},
    {0x1948b, 0x7523ff1b7bb7add7ull}, {0x18f9c, 0x71ffd71d14d3248cull}, {0x18acb, 0x6ee5266df249e7f4ull}, {0x18618, 0x6bd465491b374048ull},
    {0x18181, 0x68ccba088577dfe7ull}, {0x17d05, 0x65cde90c18d2a0ccull}, {0x178a4, 0x62d85ea20897c5c4ull}, {0x1745d, 0x5febd8ef5fd46fb2ull},
    {0x1702e, 0x5d075ddb19e6c585ull}, {0x16c16, 0x5a2a98fa4d88439eull}, {0x16816, 0x57569b7d54f4baa5ull}, {0x1642c, 0x548a581cd08f5ab8ull},
    {0x16058, 0x51c62709c6906c14ull}, {0x15c98, 0x4f08e9dcbac60a55ull}, {0x158ed, 0x4c53ad874c218eacull}, {0x15555, 0x49a54844cb6e488cull},
    {0x151d0, 0x46fe058d57ae4ef7ull}, {0x14e5e, 0x445e32089f71ef78ull}, {0x14afd, 0x41c48f81283f8700ull}, {0x147ae, 0x3f3228d966e6f2f6ull},
    {0x1446f, 0x3ca5b3ffb82e1e15ull}, {0x14141, 0x3a203be4c574f5f9ull}, {0x13e22, 0x37a06a70432943aeull}, {0x13b13, 0x35274a78ed33b7aeull},
    {0x13813, 0x32b44bb9d810f836ull}, {0x13521, 0x3046d6ca697f6995ull}, {0x1323e, 0x2ddff916e70d76caull}, {0x12f68, 0x2b7e40d6a07b62a2ull},
    {0x12c9f, 0x2921e1063918af29ull}, {0x129e4, 0x26cbe9602aa02c5aull}, {0x12735, 0x247ad85493520348ull}, {0x12492, 0x222edd0447c8f667ull},
    {0x121fb, 0x1fe82739c5e35f86ull}, {0x11f70, 0x1da6e7637c46a0fbull}, {0x11cf0, 0x1b6a688d9b5b1760ull}, {0x11a7b, 0x1932d65d35297be3ull},
    {0x11811, 0x17005d0acf8ed899ull}, {0x115b1, 0x14d23d5cc8b67be7ull}, {0x1135c, 0x12a98ca42af79bc2ull}, {0x11111, 0x108588b59dba0683ull},
    {0x10ecf, 0x0e6567e6e1b762f6ull}, {0x10c97, 0x0c4a410a4f11a190ull}, {0x10a68, 0x0a33476a1671f4c1ull}, {0x10842, 0x08209ec4f3222233ull},
    {0x10624, 0x06117149d7127c61ull}, {0x10410, 0x0407d5961cd6107dull}, {0x10204, 0x0201faaeb0fbce24ull}, {0x10000, 0x0000000000000000ull},
};

// y = -ln u, u = (a + 1/2) 2^-32, as m 2^x with the top bit of m set.  lt: kFxLog's entry for the
// index fx_log_index(a).
SMERF_HD int fx_log_index(uint32_t a)
{
    const uint64_t X = 2 * (uint64_t)a + 1;  // u = X 2^-33
    return (int)((X << fx_clz(X)) >> 57) & 63;
}
SMERF_HD void fx_neg_log(uint32_t a, FxLog lt, uint64_t& m, int& x)
{
    const uint64_t X = 2 * (uint64_t)a + 1;
    const int lz = fx_clz(X);                          // 31 .. 63
    const uint64_t F = (X << lz) >> 31;                 // f = F 2^-33 in [1/2, 1), u = f 2^(31 - lz)
    const uint64_t z = ((1ull << 49) - (uint64_t)lt.c * F) << 15;  // 1 - c f as a 64-bit fraction, exact
    const uint64_t zs = z << 6;                         // 64 z < 1
    const uint32_t zt = (uint32_t)(zs >> 32);
    // -ln(1 - z) = z + z (z H), H = 1/2 + z/3 + z^2/4 + ...
    uint32_t t = 0x0000071cu + fx_mulhi(zt, 0x0000001au);
    t = 0x00020000u + fx_mulhi(zt, t);
    t = 0x00924925u + fx_mulhi(zt, t);
    t = 0x2aaaaaabu + fx_mulhi(zt, t);
    uint64_t h = 0x00000ccccccccccdull + fx_mulh(zs, (uint64_t)t << 8);
    h = 0x0004000000000000ull + fx_mulh(zs, h);
    h = 0x0155555555555555ull + fx_mulh(zs, h);
    h = 0x8000000000000000ull + fx_mulh(zs, h);
    const uint64_t zh = fx_mulhi(z, h);
    // f near 1 (c = 1) and no power of two: y = z (1 + zH) alone, from z's own leading bit on;
    // otherwise ln c + the series + k ln 2, to 2^-59 of values above 2^-7
    const int s = fx_clz(z | 1) - 1;
    const uint64_t zn = z << s;
    const int k = lz - 31;
    const bool one = lt.c == 0x10000u && k == 0;
    uint64_t y = lt.l + z + fx_mulhi(z, zh);
    int e = -64;
    if (k > 0) {
        y = (y >> 5) + (uint64_t)k * 0x058b90bfbe8e7bcdull;
        e = -59;
    }
    if (one) {
        y = zn + fx_mulh(zn, zh);
        e = -64 - s;
    }
    const int n = fx_clz(y);
    m = y << n;
    x = e - n;
}

// sqrt(2 m 2^x) (top bit of m set) as r 2^(xr - 64), r in [2^63, 2^64)
SMERF_HD void fx_sqrt2(uint64_t m, int x, uint64_t& r, int& xr)
{
    // 2 m 2^x = v 2^(2 xr), v = V 2^-64 in [1/4, 1)
    const int E = x + 65;
    const uint64_t V = m >> (E & 1);
    xr = (E + (E & 1)) >> 1;
    // q ~ 1/sqrt(v) from the 32-bit rsqrt; s0 = v q; two Newton corrections s += q (v - s^2) / 2
    // (2^-21 -> 2^-42 -> below 2^-63)
    const float vf = (float)(uint32_t)(V >> 32) * 0x1p-32f;
#ifdef __CUDA_ARCH__
    const float qf = rsqrtf(vf);
#else
    const float qf = 1.0f / sqrtf(vf);
#endif
    const uint64_t q = (uint64_t)(uint32_t)(qf * 0x1p30f) << 32;  // q 2^-62, in (1, 2]
    const uint64_t s0 = fx_mulh(V, q) << 1;                       // s 2^-63
    const int64_t d0 = (int64_t)((V >> 2) - fx_mulh(s0, s0));     // v - s0^2, 2^-62, |d0| < 2^42
    const int64_t c0 = ((d0 >> 8) * (int64_t)(q >> 34)) >> 20;      // q d0 / 2: 2^-54 2^-28 2^-1 2^20 = 2^-63
    const uint64_t s1 = s0 + (uint64_t)c0;
    // v - s1^2 to 2^-94: the exact 128-bit product's bits below 2^-62
    const uint64_t ph = fx_mulhi(s1, s1), pl = s1 * s1;
    const uint64_t dh = (V >> 2) - ph, vl = V << 62;
    const int64_t d1 = (int64_t)(((dh - (uint64_t)(vl < pl)) << 32) | ((vl - pl) >> 32));  // 2^-94
    const int64_t c1 = ((d1 >> 16) * (int64_t)(q >> 40)) >> 37;      // q d1 / 2: 2^-78 2^-22 2^-1 2^37 = 2^-64
    r = (s1 << 1) + (uint64_t)c1;
    if (!(r >> 63)) r = s1 > (3ull << 61) ? ~0ull : 1ull << 63;  // within rounding of 1 or of 1/2
}

// (r 2^(xr - 64)) (t 2^(xt - 64)) rounded to a double
SMERF_HD double fx_normal(uint64_t r, int xr, uint64_t t, int xt, bool neg)
{
    const uint64_t p = fx_mulh(r, t);
    const int n = fx_clz(p);
    const uint64_t m = ((p << n) >> 11) + (((p << n) >> 10) & 1);  // 2^52 .. 2^53
    // value = m 2^(xr + xt - n - 53); a carry to 2^53 moves the exponent by itself
    const uint64_t bits = ((uint64_t)(uint32_t)(1022 + xr + xt - n - 1) << 52) + m;
    return fx_double(bits | (neg ? 0x8000000000000000ull : 0ull));
}
// t = T 2^-64 in [0, 1): S with sin(pi/4 t) = t S 2^-64, and cos(pi/4 t) as a 64-bit fraction, to
// 2^-60
SMERF_HD void fx_octant(uint64_t T, uint64_t& sn, uint64_t& cs)
{
    const uint64_t T2 = fx_mulh(T, T);
    const uint32_t th = (uint32_t)(T2 >> 32);
    // sin(pi/4 t) = t S(t^2), cos(pi/4 t) = 1 - t^2 D(t^2): Taylor series
    uint32_t q = 0x0000b7d7u - fx_mulhi(th, 0x0000006bu);
    q = 0x00f47a1au - fx_mulhi(th, q);
    q = 0xf183a7efu - fx_mulhi(th, q);
    uint64_t S = 0x00000541e0d21fbaull - fx_mulh(T2, (uint64_t)q << 3);
    S = 0x000265a599cc57b1ull - fx_mulh(T2, S);
    S = 0x00a335e33bad570full - fx_mulh(T2, S);
    S = 0x14abbce625be52bfull - fx_mulh(T2, S);
    S = 0xc90fdaa22168c235ull - fx_mulh(T2, S);
    q = 0x00009063u - fx_mulhi(th, 0x0000004bu);
    q = 0x00db7128u - fx_mulhi(th, q);
    q = 0xfce9c51cu - fx_mulhi(th, q);
    uint64_t D = 0x00000069b47ca881ull - fx_mulh(T2, (uint64_t)(q >> 1));
    D = 0x00003c3ea0d12375ull - fx_mulh(T2, D);
    D = 0x00155d3c7e3cbffaull - fx_mulh(T2, D);
    D = 0x040f07c206d6b0edull - fx_mulh(T2, D);
    D = 0x4ef4f326f9177969ull - fx_mulh(T2, D);
    sn = S;
    cs = 0ull - (fx_mulh(T2, D) | 1);  // in [0.707, 1)
}
// The same to about a unit, for tables of factors: each coefficient normalised (c 2^(64 + shift)), so
// that a term's rounding counts by its own size, and every product rounded
SMERF_HD uint64_t fx_mulr(uint64_t a, uint64_t b) { return fx_mulhi(a, b) + ((a * b) >> 63); }
SMERF_HD uint64_t fx_horner(uint64_t T2, const uint64_t* c, const int* shift, int n)
{
    uint64_t v = c[n - 1];
    for (int k = n - 2; k >= 0; --k) {
        const int d = shift[k + 1] - shift[k];
        const uint64_t p = fx_mulr(T2, v);
        v = c[k] - (d > 0 ? (p >> d) + ((p >> (d - 1)) & 1) : p);
    }
    return v;
}
SMERF_HD void fx_octant_exact(uint64_t T, uint64_t& sn, uint64_t& cs)
{
    const uint64_t c[10] = {0xc90fdaa22168c235ull, 0xa55de7312df295f5ull, 0xa335e33bad570e92ull, 0x9969667315ec2df3ull,
                            0xa83c1a43f73c0dc8ull, 0xf183a7ef4438fb12ull, 0xf47a1a680c6b1994ull, 0xb7d6dcf8aaba1c8bull,
                            0xd5761957c99ac950ull, 0xc5202108fcaa382eull};
    const int cx[10] = {0, 3, 8, 14, 21, 29, 37, 45, 54, 63};
    const uint64_t d[10] = {0x9de9e64df22ef2d2ull, 0x81e0f840dad61d9bull, 0xaae9e3f1e5ffcfe3ull, 0xf0fa83448dd5d7a3ull,
                            0xd368f95102545d4dull, 0xfce9c51bb1e6146full, 0xdb7127a25894796eull, 0x9063161796bfa54cull,
                            0x95062c8d7c18a243ull, 0xf7b71846b68e1c74ull};
    const int dx[10] = {1, 5, 11, 18, 25, 33, 41, 49, 58, 68};
    const uint64_t T2 = fx_mulr(T, T);
    sn = fx_horner(T2, c, cx, 10);
    const uint64_t p = fx_mulr(T2, fx_horner(T2, d, dx, 10));  // 2 (1 - cos)
    cs = 0ull - (((p >> 1) + (p & 1)) | (p == 0));
}
// e^{2 pi i p}, p = ph 2^-64 turns, in units of 2^-62 (to one unit)
SMERF_HD void fx_cis62(uint64_t ph, int64_t& c, int64_t& s)
{
    const int o = (int)(ph >> 61);
    uint64_t T = ph << 3, S, cs;
    if (o & 1) T = ~T;
    fx_octant_exact(T, S, cs);
    const uint64_t sn = fx_mulr(T, S);
    const int64_t a = (int64_t)((sn >> 2) + ((sn >> 1) & 1)), b = (int64_t)((cs >> 2) + ((cs >> 1) & 1));
    const bool swap = (o + 1) & 2;
    c = ((o + 2) & 4) ? -(swap ? a : b) : (swap ? a : b);
    s = (o & 4) ? -(swap ? b : a) : (swap ? b : a);
}
// e^{2 pi i p}, p = ph 2^-64 turns, to 2^-63 (four FP64 instructions)
SMERF_HD void fx_cis(uint64_t ph, double& c, double& s)
{
    const int o = (int)(ph >> 61);
    uint64_t T = ph << 3, S, cs;
    if (o & 1) T = ~T;
    fx_octant(T, S, cs);
    const double a = (double)(int64_t)(fx_mulhi(T, S) >> 1) * 0x1p-63, b = (double)(int64_t)(cs >> 1) * 0x1p-63;
    const bool swap = (o + 1) & 2;
    c = ((o + 2) & 4) ? -(swap ? a : b) : (swap ? a : b);
    s = (o & 4) ? -(swap ? b : a) : (swap ? b : a);
}
// Box-Muller: n0 + i n1 = sqrt(-2 ln u0) e^{2 pi i u1}, u = (word + 1/2) 2^-32
SMERF_HD void fx_box_muller(uint32_t a, uint32_t b, FxLog lt, double& n0, double& n1)
{
    uint64_t m, r, S, cs;
    int x, xr;
    fx_neg_log(a, lt, m, x);
    fx_sqrt2(m, x, r, xr);
    // octant and the angle pi/4 T 2^-64 within it, reflected in the odd ones
    const int o = (int)(b >> 29);
    uint32_t w = 2 * (b & 0x1fffffffu) + 1;  // of 2^30
    if (o & 1) w = (1u << 30) - w;
    const uint64_t T = (uint64_t)w << 34;
    fx_octant(T, S, cs);
    const int lw = fx_clz(T);
    const uint64_t sn = fx_mulh(T << lw, S);  // sin 2^(64 + lw)
    const bool swap = (o + 1) & 2;
    n0 = fx_normal(r, xr, swap ? sn : cs, swap ? -lw : 0, (o + 2) & 4);
    n1 = fx_normal(r, xr, swap ? cs : sn, swap ? 0 : -lw, o & 4);
}

// ---- 64-bit fixed-point values of a ring's FFT
// v in units of 2^-S, |v| 2^S < 2^62 (round to nearest)
SMERF_HD int64_t fx_from_double(uint64_t bits, int S)
{
    const int e = (int)((bits >> 52) & 0x7ff), k = e - 1075 + S;
    const uint64_t m = (bits & 0xfffffffffffffull) | 0x10000000000000ull;
    uint64_t v = 0;
    if (e > 0 && k > -54) v = k >= 0 ? m << k : (m + (1ull << (-k - 1))) >> -k;
    return (int64_t)(bits >> 63 ? 0 - v : v);
}
// x 2^-S rounded to a double (below the normal range: 0; above: infinity; TOP = false: S >= kFxTop, from
// which on nothing lies above)
constexpr int kFxTop = -960;
template <bool TOP = true> SMERF_HD uint64_t fx_to_double(int64_t x, int S)
{
    const uint64_t sign = (uint64_t)x & 0x8000000000000000ull, a = x < 0 ? 0 - (uint64_t)x : (uint64_t)x;
    const int n = fx_clz(a | 1), e = 1022 + 63 - n - S;
    const uint64_t m = a << n, bits = ((uint64_t)(uint32_t)e << 52) + (m >> 11) + ((m >> 10) & 1);
    return a == 0 || e <= 0 ? sign : (TOP && e > 2045 ? 0x7ff0000000000000ull : bits) | sign;
}
// a factor of magnitude at most 1 in units of 2^-62 as two signed words, hi 2^32 + lo
SMERF_HD void fx_split(int64_t w, int32_t& hi, int32_t& lo)
{
    lo = (int32_t)(uint32_t)w;
    hi = (int32_t)((w - lo) >> 32);
}
// a.x w.x - a.y w.y (SUB) or a.x w.x + a.y w.y over 2^d, from the parts (w in units of 2^-62, |a| < 2^62,
// |w| <= 1 as complex numbers, so that the middle sum stays below 2^63; d = 0 .. 2): the high words'
// products to all bits, the mixed ones rounded, the low words' products (below one unit) left out
template <bool SUB>
SMERF_HD int64_t fx_dot(int32_t axh, int32_t axl, int32_t wxh, int32_t wxl, int32_t ayh, int32_t ayl, int32_t wyh, int32_t wyl, int d = 0)
{
    const int64_t h0 = (int64_t)axh * wxh, h1 = (int64_t)ayh * wyh;
    const int64_t m0 = (int64_t)axh * wxl + (int64_t)axl * wxh, m1 = (int64_t)ayh * wyl + (int64_t)ayl * wyh;
    const int64_t hh = SUB ? h0 - h1 : h0 + h1, mid = SUB ? m0 - m1 : m0 + m1;
    return (int64_t)((uint64_t)hh << (2 - d)) + ((mid + ((int64_t)1 << (29 + d))) >> (30 + d));
}
// a w / 2^d, w as fx_split's words (Re hi, lo, Im hi, lo), and a / 2^d, rounded
template <class C> SMERF_HD C fx_cmul(C a, int32_t wxh, int32_t wxl, int32_t wyh, int32_t wyl, int d)
{
    int32_t axh, axl, ayh, ayl;
    fx_split(a.x, axh, axl);
    fx_split(a.y, ayh, ayl);
    C r;
    r.x = fx_dot<true>(axh, axl, wxh, wxl, ayh, ayl, wyh, wyl, d);
    r.y = fx_dot<false>(axh, axl, wyh, wyl, ayh, ayl, wxh, wxl, d);
    return r;
}
template <class C> SMERF_HD C fx_cshift(C a, int d)
{
    const int64_t half = ((int64_t)1 << d) >> 1;
    a.x = (a.x + half) >> d;
    a.y = (a.y + half) >> d;
    return a;
}

// The unit of a ring's values.  With 2^(top - 1022) above every |Re|, |Im| of the coefficients g, a packed
// value is at most 2^(top - 1020) and one after sub-transforms of 2^lgL points 2^(lgL + top - 1020); and
// all are below 2 sqrt(2) sum |g|.  The unit 2^-S, S = fx_unit(top, spread, lgL), keeps the smaller of the
// two bounds within 2^62; the sum comes as `sum` of all fx_share values.  A pass from 2^lgNs to
// 2^(lgNs + lgR) points divides its inputs by 2^fx_shift, 0 .. lgR bits.  Against long sums a
// transform of 8 to 4096 points then errs by 0.2 to 0.9 of what the same passes in FP64 do, at
// flat and falling spectra alike (at 2048 points, of the ring's deviation: flat 6.7e-17 against 2.4e-16,
// m^-1/2 1.6e-16 against 2.2e-16, m^-2 1.2e-16 against 1.8e-16; one unit for the whole transform, that of the sum,
// rounded the early passes to 2^-49 of a flat coefficient: 1.5e-15; up to 256 points one unit is as good).
SMERF_HD unsigned fx_share(uint32_t h, int top)  // of 2^(top - 1039), rounded up but for a unit; h: high word of |v|
{
    const int s = top - (int)(h >> 20);
    return s > 20 ? 0u : ((h & 0xfffffu) | 0x100000u) >> 4 >> s;
}
SMERF_HD int fx_spread(unsigned sum)  // log2 of the bound by the sum over the bound by the maximum at one point
{
#ifdef __CUDA_ARCH__
    return 15 - __clz(sum - (sum >> 2));
#else
    return 15 - __builtin_clz(sum - (sum >> 2));
#endif
}
SMERF_HD int fx_least(int a, int b) { return a < b ? a : b; }
SMERF_HD int fx_unit(int top, int spread, int lgL) { return 61 - (top - 1021) - fx_least(lgL, spread); }
SMERF_HD int fx_shift(int spread, int lgNs, int lgR) { return fx_least(lgNs + lgR, spread) - fx_least(lgNs, spread); }

}  // namespace smerf
