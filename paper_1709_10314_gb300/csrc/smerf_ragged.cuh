// smerf_ragged.cuh -- rings of their own point count and offset (the paper's Sec. 1 remark: the method
// holds on any iso-latitude grid).  Included by smerf_sample_impl.cuh.
//
// A ring of n points from phi0: Y_q = sum over m = q (mod n) of c_m e^{i m phi0} is formed and packed
// for an n/2-point complex FFT, which runs in Stockham passes over the factors of n/2 (4, 2, then
// the odd primes), one output point per thread from r terms with the roots of unity from a table of
// the ring's own.  HEALPix's polar rings (4i points) took O(n^2) terms in the FFT warps of one CTA
// per segment before: Nside 128, 16 realisations, 4266 -> 113 us a call.
#pragma once

namespace smerf {

// e^{2 pi i p}, p = ph 2^-64 turns
template <class Real> __device__ __forceinline__ cplx<Real> cis_turns(uint64_t ph)
{
    Real sn, cs;
    if constexpr (sizeof(Real) == 4) sincospif((float)(int32_t)(ph >> 32) * 0x1p-31f, &sn, &cs);
    else fx_cis(ph, cs, sn);
    return cmk<cplx<Real>>(cs, sn);
}

// threads that share a ring of its own point count, in the band kernel: a warp for rings up
// to 512 points, the whole CTA from 4096 on
__host__ __device__ inline int band_group(int Nc) { return Nc <= 256 ? 32 : Nc >= 2048 ? 256 : Nc / 8; }

// barrier of a ring's thread group (one warp, or gs threads on named barrier bar)
__device__ __forceinline__ void ragged_sync(int gs, int bar)
{
    if (gs == 32) __syncwarp();
    else bar_sync(bar, gs);
}

// Y_q of the ring's coefficients X (slot 0 = (g_0, Re g_M), slot m = g_m, M = Nc): the real field
// T(phi) = sum_{|m| <= M} c_m e^{i m phi}, c_0 = g_0, c_{+-m} = g_m, conj g_m, c_{+-M} = Re g_M / 2, has
// Y_q = sum over m = q (mod n) of c_m e^{i m phi0} (modes above the ring's own Nyquist alias onto it).
// This is part `part` of 2^lp of it.
template <class Real>
__device__ __forceinline__ cplx<Real> ring_fold(const cplx<Real>* X, int Nc, int n, uint64_t ph, int q, int part, int lp)
{
    using C = cplx<Real>;
    C acc = cmk<C>(0, 0);
    auto term = [&](int m) {
        const C g = m == 0 ? cmk<C>(X[0].x, 0) : (m == Nc ? cmk<C>((Real)0.5 * X[0].y, 0) : X[m]);
        return ph == 0 ? g : cmul(g, cis_turns<Real>((uint64_t)m * ph));
    };
    for (int m = q + n * part; m <= Nc; m += n << lp) acc = cadd(acc, term(m));
    for (int m = (q == 0 ? n : n - q) + n * part; m <= Nc; m += n << lp) acc = cadd(acc, cconj(term(m)));  // -m < 0
    return acc;
}

// One ring of n = 2 N points from its coefficients in X (destroyed) with W as second buffer and
// RT for the N roots e^{2 pi i t / n} (roots: formed here, else there already), by the gs threads of a
// group (lane l; named barrier bar)
template <class Real>
__device__ __noinline__ void ragged_ring(cplx<Real>* X, cplx<Real>* W, cplx<Real>* RT, bool roots, int Nc, int n,
                                         uint64_t ph, cplx<Real>* gout, int l, int gs, int bar)
{
    using C = cplx<Real>;
    const int N = n / 2;
    if (roots) {
        // t / n as a 64-bit fraction: t (2^64 / n) with the division's remainder r < n < 2^14 (t r < 2^27)
        const uint64_t q = ~0ull / (unsigned)n;
        const unsigned r = (unsigned)(~0ull - q * (unsigned)n) + 1u;
        for (int t = l; t < N; t += gs) RT[t] = cis_turns<Real>((uint64_t)t * q + ((unsigned)t * r) / (unsigned)n);
    }
    ragged_sync(gs, bar);
    // fold and C2R packing (c2r_pack's Z), the pair q, N - q together.  A pair sums 4 Nc / n terms: on short
    // rings 2^lp neighbouring lanes share it, else a few threads would sum all modes one after another (lp
    // by the band kernel's groups everywhere, so that the sums are the same on either kernel)
    int lp = 0;
    while (lp < 5 && (N / 2 + 1) << (lp + 1) <= band_group(Nc)) ++lp;
    for (int q0 = 0; 2 * q0 <= N; q0 += gs >> lp) {
        const int q = q0 + (l >> lp), part = l & ((1 << lp) - 1);
        C a = cmk<C>(0, 0), b = a;
        if (2 * q <= N) {
            a = ring_fold<Real>(X, Nc, n, ph, q, part, lp);
            b = ring_fold<Real>(X, Nc, n, ph, N - q, part, lp);
        }
        for (int o = 1 << lp >> 1; o > 0; o >>= 1) {
            a = cadd(a, cmk<C>(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o)));
            b = cadd(b, cmk<C>(__shfl_xor_sync(0xffffffffu, b.x, o), __shfl_xor_sync(0xffffffffu, b.y, o)));
        }
        if (part || 2 * q > N) continue;
        b = cconj(b);
        if (q == 0) {
            W[0] = cmk<C>(a.x + b.x, a.x - b.x);
        } else {
            const C e = cadd(a, b), o = cmuli(cmul(RT[q], csub(a, b)));
            W[q] = cadd(e, o);
            if (2 * q < N) W[N - q] = cconj(csub(e, o));
        }
    }
    ragged_sync(gs, bar);
    C* src = W;
    C* dst = X;
    int Ns = 1, rem = N, p = 3;
    while (rem > 1) {
        int r;
        if ((rem & 3) == 0) r = 4;
        else if ((rem & 1) == 0) r = 2;
        else {
            while (p * p <= rem && rem % p) p += 2;
            r = rem % p ? rem : p;
        }
        rem /= r;
        const int Wn = Ns * r, m = N / r, unit = N / Wn;
        for (int e = l; e < N; e += gs) {
            const int blk = e / Wn, w = e - blk * Wn, st = w * unit;  // w = kk + a Ns
            const C* in = src + blk * Ns + w % Ns;
            C acc = in[0];
            int t = st;
            auto term = [&](int i) {
                const int u = 2 * t;  // root of order N: e^{2 pi i t / N} = e^{2 pi i u / n}, half a turn from t = N / 2 on
                const C x = in[i * m], y = u < N ? RT[u] : RT[u - N];
                const C z = cmul(x, y);
                acc = u < N ? cadd(acc, z) : csub(acc, z);
                t += st;
                if (t >= N) t -= N;
            };
            if (sizeof(Real) == 8 || r <= 256) {
                for (int i = 1; i < r; ++i) term(i);
            } else {
                // large primes in FP32 in parts of 64 terms, so that a sum rounds 64 + r / 64 times and not r times
                C sum = acc;
                for (int i = 1; i < r; i += 64) {
                    acc = cmk<C>(0, 0);
                    const int end = i + 64 < r ? i + 64 : r;
                    for (int k = i; k < end; ++k) term(k);
                    sum = cadd(sum, acc);
                }
                acc = sum;
            }
            if (rem == 1) __stcs(gout + e, acc);
            else dst[e] = acc;
        }
        Ns = Wn;
        ragged_sync(gs, bar);
        C* s = src;
        src = dst;
        dst = s;
    }
    if (N == 1 && l == 0) __stcs(gout, W[0]);
}

}  // namespace smerf
