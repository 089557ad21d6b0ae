// smerf_band.cuh -- the segment kernel for requests that leave most of the GPU idle (few
// segments, few realisations) and for plans with ring-dependent longitudes.  Included by
// smerf_sample_impl.cuh.
//
// The warp-specialised kernel walks a segment ring by ring, so a request of a few segments takes
// the latency of a whole ring (noise, step, FFT: 2 us and more) for each ring of a segment while
// most SMs idle.  Here a CTA takes one realisation's segment in chunks of rings and does each
// part of the work for the whole chunk at once, with every thread:
//   1. the noise of every (ring, unit) of the chunk, which depends on no state;
//   2. the recursion, one thread per unit, nothing but its table rows and a few multiply-adds per
//      ring (Eq. (state_space), with step_state's operations in step_state's order, so that the
//      field is the warp-specialised kernel's bit for bit);
//   3. the C2R FFTs of the chunk's rings side by side, written straight to the output.
// A segment can be split further over `splits` CTAs: each repeats parts 1 and 2 from the
// segment's start (they are cheap) and synthesises only its own share of the rings.
// Rings with their own point count: smerf_ragged.cuh, a group of threads per ring.  One FP64
// realisation of 64 x 128 in Alg. 2's order: 166 -> 24.6 us (the fixed-point FFT among them); one of
// 181 x 512, p = 2: 31 -> 20 to 24 us between runs (the anchor tiles among them).
#pragma once

namespace smerf {

constexpr int kBandThreads = 256;      // two CTAs per SM
constexpr int kBandThreadsFew = 512;   // requests of at most one CTA per SM (band_config)

// Table rows of unit u at one position, G rows of step_row(M) values, converted to Real
template <class Real, class TabT, int M>
__device__ __forceinline__ void band_rows(const TabT* tb, int u, Real (&t)[kG<M>][step_row(M)])
{
    constexpr int G = kG<M>, ROW = step_row(M);
#pragma unroll
    for (int g = 0; g < G; ++g) load_row<Real, TabT, ROW>(tb + (size_t)(G * u + g) * ROW, t[g]);
}

// One ring's step of a unit (table rows t, the Nyquist chain's row ny, normals nr, the right
// anchor's states xr), as in ws_body
template <class Real, int M>
__device__ __forceinline__ void band_step(const Real (&t)[kG<M>][step_row(M)], const Real* ny, bool first_unit,
                                          bool has_right, const Real* nr, const Real* xr, Real (&x)[unit_vals(M)])
{
    constexpr int G = kG<M>, ROW = step_row(M);
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            Real(&xs)[M] = *reinterpret_cast<Real(*)[M]>(&x[g * 2 * M + part * M]);
            const Real* xi = nr + g * 2 * M + part * M;
            const Real* xq = xr + g * 2 * M + part * M;
            if (g == 0 && part == 1 && first_unit) {
                Real tn[ROW];  // slot 0, second part: the Nyquist chain
                VecN<Real, ROW>::ld(ny, tn);
                if (has_right) step_state<Real, M, true>(tn, xs, xi, xq);
                else step_state<Real, M, false>(tn, xs, xi, nullptr);
            } else if (has_right) {
                step_state<Real, M, true>(t[g], xs, xi, xq);
            } else {
                step_state<Real, M, false>(t[g], xs, xi, nullptr);
            }
        }
}

// Reals of a unit's staged table rows: an odd number of 16-byte words, so that neighbouring units'
// vector accesses fall on different banks
template <class Real, int M>
__host__ __device__ constexpr int band_row_reals()
{
    const int v = unit_slots(M) * step_row(M), w = 16 / (int)sizeof(Real);
    return (v / w) % 2 == 0 ? v + w : v;
}

// Shared memory (cplx = 2 Real), rb realisations: X [rb][chunk][Nc] cplx; the normals [rb][chunk][units][NU]
// Real, the same memory then the FFTs' second buffer [rb][chunk][Nc] cplx; the staged rows
// [chunk][units][RV] Real; the states [rb][units][NU] Real; the Nyquist chain's rows [chunk][ROW] Real;
// the root tables [groups][Nc] cplx (ring-dependent longitudes only).  Where that does not fit (the
// longest ring-dependent plans, one ring per chunk), lean = 1: the root tables lie behind the FFTs'
// second buffer in the normals' memory (p = 2 and 3: the normals are two and three times that
// buffer; p = 3 with 4096 complex points in FP32: 229472 bytes of 262240); lean = 2, Alg. 2's order:
// the states stay in the anchors' scratch, whose start-ring entry of a chain and realisation
// belongs to this CTA alone (no other segment, no splits)
template <class Real> constexpr bool band_global_states(int M) { return M == 1 || (M == 2 && sizeof(Real) == 8); }
template <class Real, int M>
__host__ __device__ inline size_t band_noise_reals(int Nc, int chunk, int rb, int lean)
{
    const size_t nz = (size_t)Nc / unit_slots(M) * unit_vals(M), fft = (size_t)2 * Nc * (1 + kBandThreads / band_group(Nc));
    return lean ? (nz > fft ? nz : fft) : rb * chunk * nz;
}
template <class Real, int M, bool STAGE>
__host__ __device__ inline size_t band_smem(int Nc, int chunk, int rb, bool rings, int lean)
{
    const int units = Nc / unit_slots(M);
    const size_t x = (size_t)Nc * 2 * sizeof(Real), nz = (size_t)units * unit_vals(M) * sizeof(Real);
    const size_t rows = (STAGE ? (size_t)units * band_row_reals<Real, M>() : 0) * sizeof(Real) + step_row(M) * sizeof(Real);
    return chunk * (rb * x + rows) + band_noise_reals<Real, M>(Nc, chunk, rb, lean) * sizeof(Real) + (lean == 2 ? 0 : rb * nz) +
           (rings && !lean ? (kBandThreads / band_group(Nc)) * x : 0);
}

// grid (splits, realisations / rb, segments)
// STAGE: the chunk's table rows go through shared memory, loaded in part 1 beside the noise by
// every thread, so that the recursion waits for no global load
// GS: lean = 2
template <class Real, class TabT, int M, bool STAGE, int NT, bool GS>
__global__ void __launch_bounds__(NT, NT == kBandThreads ? 2 : 1) segment_band_kernel(SampleParams P, int chunk, int rb, int lean)
{
    using C = cplx<Real>;
    constexpr int G = kG<M>, ROW = step_row(M), NU = unit_vals(M), NC = unit_calls(M);
    constexpr int RV = band_row_reals<Real, M>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint4 rk[2][kKeyWords];  // rb <= 2
    __shared__ int fxred[sizeof(Real) == 8 ? 2 * kFxRings : 1];
    (void)fxred;

    const Segment sg = P.segs[blockIdx.z];
    const int r = blockIdx.y * rb, c = sg.chain, nr = min(rb, P.n_samples - r);  // realisations r .. r + nr - 1
    constexpr int nt = NT;
    const bool rings = NT == kBandThreads && P.ring_n;  // the ragged rings' groups are of kBandThreads
    const int tid = threadIdx.x;
    const int Nc = P.Nc, n_units = P.n_units;
    const size_t mp = P.n_modes_pad;
    const bool has_right = sg.right >= 0;
    // this CTA's share of the segment's rings (the start ring is written by the northern chain)
    const int first = (c == 1 && sg.p0 == 0) ? 1 : sg.p0, len = sg.p1 - first;
    const int own0 = first + (int)((long long)len * blockIdx.x / gridDim.x);
    const int own1 = first + (int)((long long)len * (blockIdx.x + 1) / gridDim.x);
    if (own0 >= own1) return;

    const int cn = chunk * n_units;  // units of a realisation's chunk
    C* X = reinterpret_cast<C*>(smem_raw);
    Real* NZ = reinterpret_cast<Real*>(X + (size_t)rb * chunk * Nc);
    C* W = reinterpret_cast<C*>(NZ);
    constexpr bool LEAN = !STAGE && NT == kBandThreads;  // builds that lean layouts run on
    Real* RW = NZ + (LEAN ? band_noise_reals<Real, M>(Nc, chunk, rb, lean) : (size_t)rb * cn * NU);
    Real* S = RW + (STAGE ? (size_t)cn * RV : 0);
    Real* NY = S + (GS ? 0 : (size_t)rb * n_units * NU);
    C* RT = LEAN && lean ? W + Nc : reinterpret_cast<C*>(NY + (size_t)chunk * ROW);
    Real* anc = (Real*)P.anc;
    const size_t anc_r = aoff<M>(P, 0, 1, 0, 0, 0);  // from one realisation's anchor states to the next's
    const Real* xrg = anc + aoff<M>(P, c, r, has_right ? sg.right : 0, 0, 0);
    Real* xlg = anc + aoff<M>(P, c, r, sg.left, 0, 0);
    const TabT* steps = (const TabT*)(c == 0 ? P.steps[0] : P.steps[1]);
    if (tid < rb * kKeyWords) rk[tid / kKeyWords][tid % kKeyWords] = round_key_word(P.seed + (uint64_t)(r + tid / kKeyWords), tid % kKeyWords);
    __syncthreads();

    for (int c0 = sg.p0; c0 < own1; c0 += chunk) {
        const int nk = min(chunk, own1 - c0);
        const int ring0 = c == 0 ? P.k0 - c0 : P.k0 + c0, dir = c == 0 ? -1 : 1;  // ring of pos c0 + k: ring0 + dir k
        for (int idx = tid; idx < nk * n_units; idx += nt) {
            const int k = idx / n_units, u = idx - k * n_units;
            if (c0 + k == sg.p0) continue;  // the segment's left end: its state is the anchor's
            const TabT* tb = steps + (size_t)(c0 + k) * mp * ROW;
            if constexpr (STAGE) {
                Real t[G][ROW];
                band_rows<Real, TabT, M>(tb, u, t);
#pragma unroll
                for (int g = 0; g < G; ++g) VecN<Real, ROW>::st(RW + (size_t)idx * RV + g * ROW, t[g]);
            }
            if (u == 0) {
                Real tn[ROW];
                load_row<Real, TabT, ROW>(tb + (size_t)Nc * ROW, tn);
                VecN<Real, ROW>::st(NY + (size_t)k * ROW, tn);
            }
#pragma unroll 1
            for (int z = 0; z < nr; ++z) {
                Real xi[NU];
                unit_normals_rk<Real, NC>(rk[z], (uint32_t)u, (uint32_t)(ring0 + dir * k), xi);
                VecN<Real, NU>::st(NZ + ((size_t)z * cn + idx) * NU, xi);
            }
        }
        if (c0 == sg.p0) {
            // the anchors' states, the first values of the launch before this one
            wait_launch();
            for (int idx = tid; idx < (GS ? 0 : nr * n_units); idx += nt) {
                const int z = idx / n_units, u = idx - z * n_units;
                Real v[NU];
                VecN<Real, NU>::ldcg(xlg + z * anc_r + (size_t)NU * u, v);
                VecN<Real, NU>::st(S + (size_t)NU * idx, v);
            }
        }
        __syncthreads();
        if constexpr (STAGE) {
            // one thread per real chain f (slot f / 2, Re or Im): a small grid has few units, and in
            // FP64 a warp's multiply-add holds the SM's two lanes for 16 cycles
            for (int zf = tid; zf < nr * 2 * Nc; zf += nt) {
                const int z = zf / (2 * Nc), f = zf - z * 2 * Nc;
                const int u = f / (2 * G), in_unit = f - u * 2 * G;
                Real x[M], xr[M];
#pragma unroll
                for (int q = 0; q < M; ++q) {
                    x[q] = S[(size_t)zf * M + q];
                    xr[q] = has_right ? __ldcg(xrg + z * anc_r + (size_t)f * M + q) : (Real)0;
                }
#pragma unroll 2
                for (int k = 0; k < nk; ++k) {
                    const int pos = c0 + k;
                    if (pos > sg.p0) {
                        const Real* w = NZ + ((size_t)z * cn + (size_t)k * n_units + u) * NU;
                        // chain 1 is the Nyquist mode's (its own table row)
                        const Real* row = f == 1 ? NY + (size_t)k * ROW : RW + ((size_t)k * n_units + u) * RV + (in_unit >> 1) * ROW;
                        Real t[ROW], xi[M];
                        VecN<Real, ROW>::ld(row, t);
#pragma unroll
                        for (int q = 0; q < M; ++q) xi[q] = w[in_unit * M + q];
                        if (has_right) step_state<Real, M, true>(t, x, xi, xr);
                        else step_state<Real, M, false>(t, x, xi, nullptr);
                    }
                    if (pos >= own0) reinterpret_cast<Real*>(X)[((size_t)z * chunk + k) * 2 * Nc + f] = x[0];
                }
#pragma unroll
                for (int q = 0; q < M; ++q) S[(size_t)zf * M + q] = x[q];
            }
        } else {
            for (int u = tid; u < n_units; u += nt) {
                Real x[NU], xr[NU];
                if constexpr (GS) VecN<Real, NU>::ldcg(xlg + (size_t)NU * u, x);
                else VecN<Real, NU>::ld(S + (size_t)NU * u, x);
                if (has_right) VecN<Real, NU>::ldcg(xrg + (size_t)NU * u, xr);
#pragma unroll 2
                for (int k = 0; k < nk; ++k) {
                    const int pos = c0 + k;
                    if (pos > sg.p0) {
                        Real xi[NU], t[G][ROW];
                        VecN<Real, NU>::ld(NZ + ((size_t)k * n_units + u) * NU, xi);
                        band_rows<Real, TabT, M>(steps + (size_t)pos * mp * ROW, u, t);
                        band_step<Real, M>(t, NY + (size_t)k * ROW, u == 0, has_right, xi, xr, x);
                    }
                    if (pos >= own0) put_unit<C, Real, M>(X + (size_t)k * Nc, u, x);
                }
                if constexpr (GS) VecN<Real, NU>::st(xlg + (size_t)NU * u, x);  // this thread's own in the next chunk
                else VecN<Real, NU>::st(S + (size_t)NU * u, x);
            }
        }
        __syncthreads();
        const int k0 = max(0, own0 - c0);
        if (k0 >= nk) continue;  // nothing of this chunk is this CTA's (NZ is rewritten: no reader is left)
        if (rings) {
            // whole rings with an offset become whole rings without one; rings of their own
            // point count are synthesised by the thread groups
            const int gs = band_group(Nc), g = tid / gs, groups = nt / gs;
            for (int k = k0; k < nk; ++k) {
                const int ring = ring0 + dir * k;
                const uint64_t ph = P.ring_ph[ring];
                if (P.ring_n[ring] != P.n_phi || ph == 0) continue;
                C* x = X + (size_t)k * Nc;
                for (int s = tid; s < Nc; s += nt) {
                    if (s == 0) x[0].y *= cis_turns<Real>((uint64_t)Nc * ph).x;
                    else x[s] = cmul(x[s], cis_turns<Real>((uint64_t)s * ph));
                }
            }
            int turn = 0;
            for (int k = k0; k < nk; ++k) {
                const int ring = ring0 + dir * k, n = P.ring_n[ring];
                if (n == P.n_phi) continue;
                if (turn++ % groups != g) continue;
                ragged_ring<Real>(X + (size_t)k * Nc, W + (size_t)k * Nc, RT + (size_t)g * Nc, true, Nc, n, P.ring_ph[ring],
                                  (C*)((Real*)P.out + (size_t)r * P.ring_total + P.ring_off[ring]), tid - g * gs, gs, 6 + g);
            }
            __syncthreads();
        }
        if constexpr (sizeof(Real) == 8) {
            if (rb > 1) {
                // every realisation's rings of this chunk together (none are ring-dependent); chunks that
                // begin before this CTA's share hold rings to skip, so each realisation's rings move up
                C* base = (C*)((Real*)P.out + ((size_t)r * P.n_theta + ring0 + dir * k0) * (size_t)P.n_phi);
                const int per = nk - k0;
                if (per < chunk) {
                    for (int z = 0; z < nr; ++z) {
                        for (int i = tid; i < per * Nc; i += nt) {
                            const C v = X[((size_t)z * chunk + k0) * Nc + i];
                            W[(size_t)z * per * Nc + i] = v;
                        }
                    }
                    __syncthreads();
                    for (int i = tid; i < nr * per * Nc; i += nt) X[i] = W[i];
                    __syncthreads();
                }
                // rb > 1 only on short rings (band_config)
                grp_fx_c2r<false, true>(X, W, nr * per, P.lgNc, (const int4*)P.twx, (const int4*)P.prex,
                                        RingOut2<C>{base, (size_t)((long long)dir * Nc), (size_t)P.n_theta * Nc, per}, fxred, tid, nt, kBarFft);
                __syncthreads();
                continue;
            }
        }
        for (int k = k0; k < nk;) {
            // a run of whole rings: their FFTs together
            int e = nk;
            const int ring = ring0 + dir * k;
            C* base = (C*)((Real*)P.out + ((size_t)r * P.n_theta + ring) * (size_t)P.n_phi);
            if (rings) {
                if (P.ring_n[ring] != P.n_phi) {
                    ++k;
                    continue;
                }
                for (e = k + 1; e < nk && P.ring_n[ring0 + dir * e] == P.n_phi;) ++e;
                base = (C*)((Real*)P.out + (size_t)r * P.ring_total + P.ring_off[ring]);
            }
            const RingOut<C> gout{base, (size_t)((long long)dir * Nc), (reinterpret_cast<uintptr_t>(base) & 15) == 0};
            C* x = X + (size_t)k * Nc;
            C* w = W + (size_t)k * Nc;
            const C* pre = (const C*)P.pre;
            if constexpr (sizeof(Real) == 4) {
                if (!P.fft_r4) hr_c2r<C, 2, 12, true>(P.lgNc, x, w, e - k, (const C*)P.tw, (const C*)P.tw2, pre, gout, tid, nt);
                else grp_c2r_rt<C>(x, w, e - k, P.lgNc, (const C*)P.tw, pre, gout, tid, nt);
            } else {
                if (P.lgNc <= kFxFlat)
                    grp_fx_c2r<false, true>(x, w, e - k, P.lgNc, (const int4*)P.twx, (const int4*)P.prex, gout, fxred, tid, nt, kBarFft);
                else
                    grp_fx_c2r<false, false>(x, w, e - k, P.lgNc, (const int4*)P.twx, (const int4*)P.prex, gout, fxred, tid, nt, kBarFft);
                __syncthreads();  // fxred serves the next run
            }
            k = e;
        }
        __syncthreads();  // X and W (the noise) are rewritten by the next chunk
    }
}

}  // namespace smerf
