// smerf_setup.cu -- FP64 set-up of the conditional-covariance tables on the GPU
// (Alg. 1 of Creasey & Lang, arXiv 1709.10314, with the efficient covariance of Sec. 3).
//
// Everything lives in the "northern frame": a chain runs from its start angle toward the
// north pole (theta decreasing).  The southern chain is the mirror image z -> -z of the
// northern problem (Sec. 4 obtains the southern rings from the mirror symmetry); its tables act
// on the mirrored state S x, S = diag((-1)^q).
//
// Notation (Sec. 3).  kappa-hat_i = kappa_i^2 = -l_i (l_i + 1).  For integer order mu,
//   P^mu_l(z)  = (Q_mu / mu!) t^mu F_mu(x),   P^mu_l(-z) = (Q_mu / mu!) t^-mu F_mu(1-x),
//   t = tan(theta/2), x = sin^2(theta/2) = (1-z)/2,
//   Q_mu = prod_{j<mu} (j(j+1) + kappa^2) = (-l)_mu (1+l)_mu,
//   F_mu(x) = 2F1(-l, l+1; 1+mu; x)          (Eq. (Legendre_hypergeometric)),
// whose series has positive terms with ratio (n(n+1) + kappa^2) x / ((n+1+mu)(n+1)).
//
// U-basis state x_q = U^q_m g_m (Eq. (Jmatrix_more_efficient)), q < p.  The solution
// matrix regular at the north pole is U(z)_{q,i} = P^{m+q}_{l_i}(z).  Gaussian
// conditioning (Eqs. (trans_matrix), (innov_matrix)) with the product form of the
// cross covariance (Eq. (Jmatrix_efficient)) gives, for a northward step z1 -> z2:
//   A = U(z2) U(z1)^{-1}                                               (transition)
//   Q = Cov(x(z2) | x(z1)) = (A_amp / 2 pi) int_{z1}^{z2} phi phi^T ds / (1 - s^2),
//       phi(s) = U(z2) U(s)^{-1} e_{p-1}.
// The second form follows from the state-space model of the process: its covariance
// operator is (2 pi D_m)^{-1} (Lemma 2.1 and the orthonormality of sqrt(2 pi) L_lm in
// dz), D_m has leading coefficient (-1)^p (1-z^2)^p, so only the last U-component is
// driven, with intensity A_amp / (2 pi (1 - s^2)).  It needs only the regular solution,
// i.e. 2F1 at x <= 1/2, and has no cancellation when z1 and z2 are close.
// The start covariance J(z0, z0) of a real spectrum comes from ratios of neighbouring orders on both sides of z0
// (start_kernel); a complex one takes Eq. (Jmatrix_efficient) with its Gamma factors (start_kernel_c).
// Both solutions are needed at |z0| ~ 0 only, where both series converge fast.
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <chrono>
#include <vector>

#include <cuda/std/complex>

#include "smerf_internal.cuh"
#include "smerf_setup.h"

using namespace smerf;

namespace {

struct Spec {
    int M;
    double k2[kMaxP];     // kappa_i^2
    double b[kMaxP];      // partial-fraction weights (Eq. (C_ell_efficient))
    double A;
    double kmax;
    int n_theta, k0, n_modes, n_modes_pad;
    const double* theta;  // device: ring colatitudes (null: equiangular, pi (k + 1/2) / n_theta)
};

// colatitude of ring k (the plan's table, or the equiangular grid)
__device__ __host__ inline double ring_colat(const double* theta, int n_theta, int k)
{
    return theta ? theta[k] : SMERF_PI * ((double)k + 0.5) / (double)n_theta;
}

// 2F1(-l, l+1; 1+mu; x) for kappa^2 = k2 (a positive series) as S * 1e250^E.  Terms are
// taken two at a time with one division: r0 = a0/d0 and r1 = a1/d1 from 1/(d0 d1).
__device__ void hyp_scaled(double k2, int mu, double x, double& S, int& E)
{
    double s = 1.0, t = 1.0;
    int e = 0;
    const double m1 = (double)mu + 1.0;
    for (int n = 0; n < 1000000; n += 2) {
        const double dn = (double)n;
        const double a0 = (dn * (dn + 1.0) + k2) * x, d0 = (dn + m1) * (dn + 1.0);
        const double a1 = ((dn + 1.0) * (dn + 2.0) + k2) * x, d1 = (dn + 1.0 + m1) * (dn + 2.0);
        const double inv = 1.0 / (d0 * d1);
        const double r0 = a0 * d1 * inv, r1 = a1 * d0 * inv;
        t *= r0;
        s += t;
        if (t < 1e-17 * s && r0 < 0.9) break;
        t *= r1;
        s += t;
        if (t < 1e-17 * s && r1 < 0.9) break;
        if (s > 1e250) { s *= 1e-250; t *= 1e-250; ++e; }
    }
    S = s;
    E = e;
}

// the series relative to a reference value sref * 1e250^eref (given as 1/sref and eref)
__device__ inline double hyp_rel(double k2, int mu, double x, double sref_inv, int eref)
{
    double s;
    int e;
    hyp_scaled(k2, mu, x, s, e);
    double v = s * sref_inv;
    for (int d = e - eref; d > 0; --d) v *= 1e250;
    for (int d = e - eref; d < 0; ++d) v *= 1e-250;
    return v;
}

// ring angle of position pos in chain c, in the northern frame
__device__ __host__ inline double chain_theta(const Spec& sp, int c, int pos)
{
    const int k = (c == 0) ? sp.k0 - pos : sp.n_theta - 1 - sp.k0 - pos;
    return ring_colat(sp.theta, sp.n_theta, k);
}

// ---------------------------------------------------------------- small matrices
template <int M> struct Mat { double a[M][M]; };

template <int M> __device__ inline Mat<M> mzero() { Mat<M> r; for (int i = 0; i < M; ++i) for (int j = 0; j < M; ++j) r.a[i][j] = 0.0; return r; }
template <int M> __device__ inline Mat<M> meye() { Mat<M> r = mzero<M>(); for (int i = 0; i < M; ++i) r.a[i][i] = 1.0; return r; }
template <int M> __device__ inline Mat<M> mmul(const Mat<M>& x, const Mat<M>& y)
{
    Mat<M> r;
    for (int i = 0; i < M; ++i)
        for (int j = 0; j < M; ++j) {
            double s = 0.0;
            for (int k = 0; k < M; ++k) s += x.a[i][k] * y.a[k][j];
            r.a[i][j] = s;
        }
    return r;
}
template <int M> __device__ inline Mat<M> mT(const Mat<M>& x) { Mat<M> r; for (int i = 0; i < M; ++i) for (int j = 0; j < M; ++j) r.a[i][j] = x.a[j][i]; return r; }
template <int M> __device__ inline Mat<M> madd(const Mat<M>& x, const Mat<M>& y) { Mat<M> r; for (int i = 0; i < M; ++i) for (int j = 0; j < M; ++j) r.a[i][j] = x.a[i][j] + y.a[i][j]; return r; }
template <int M> __device__ inline Mat<M> msym(const Mat<M>& x) { Mat<M> r; for (int i = 0; i < M; ++i) for (int j = 0; j < M; ++j) r.a[i][j] = 0.5 * (x.a[i][j] + x.a[j][i]); return r; }

// inverse of a 3 x 3 matrix by its adjugate (cofactors, the transposed minors) over the
// determinant; T is a real or complex matrix type, S its scalar
template <class T, class S> __device__ inline T inv3(const T& x)
{
    const auto& a = x.a;
    T r;
    r.a[0][0] = a[1][1] * a[2][2] - a[1][2] * a[2][1];
    r.a[0][1] = a[0][2] * a[2][1] - a[0][1] * a[2][2];
    r.a[0][2] = a[0][1] * a[1][2] - a[0][2] * a[1][1];
    r.a[1][0] = a[1][2] * a[2][0] - a[1][0] * a[2][2];
    r.a[1][1] = a[0][0] * a[2][2] - a[0][2] * a[2][0];
    r.a[1][2] = a[0][2] * a[1][0] - a[0][0] * a[1][2];
    r.a[2][0] = a[1][0] * a[2][1] - a[1][1] * a[2][0];
    r.a[2][1] = a[0][1] * a[2][0] - a[0][0] * a[2][1];
    r.a[2][2] = a[0][0] * a[1][1] - a[0][1] * a[1][0];
    const S d = a[0][0] * r.a[0][0] + a[0][1] * r.a[1][0] + a[0][2] * r.a[2][0];
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) r.a[i][j] = r.a[i][j] / d;
    return r;
}

// inverse of a general M x M matrix (M <= 3)
template <int M> __device__ inline Mat<M> minv(const Mat<M>& x);
template <> __device__ inline Mat<1> minv<1>(const Mat<1>& x) { Mat<1> r; r.a[0][0] = 1.0 / x.a[0][0]; return r; }
template <> __device__ inline Mat<2> minv<2>(const Mat<2>& x)
{
    const double d = x.a[0][0] * x.a[1][1] - x.a[0][1] * x.a[1][0];
    Mat<2> r;
    r.a[0][0] = x.a[1][1] / d; r.a[0][1] = -x.a[0][1] / d;
    r.a[1][0] = -x.a[1][0] / d; r.a[1][1] = x.a[0][0] / d;
    return r;
}
template <> __device__ inline Mat<3> minv<3>(const Mat<3>& x) { return inv3<Mat<3>, double>(x); }

// lower Cholesky factor of a symmetric positive semi-definite matrix (0 where it degenerates)
template <int M> __device__ inline Mat<M> mchol(const Mat<M>& x)
{
    Mat<M> L = mzero<M>();
    for (int j = 0; j < M; ++j) {
        double d = x.a[j][j];
        for (int k = 0; k < j; ++k) d -= L.a[j][k] * L.a[j][k];
        const double ljj = d > 0.0 ? sqrt(d) : 0.0;
        L.a[j][j] = ljj;
        for (int i = j + 1; i < M; ++i) {
            double s = x.a[i][j];
            for (int k = 0; k < j; ++k) s -= L.a[i][k] * L.a[j][k];
            L.a[i][j] = ljj > 0.0 ? s / ljj : 0.0;
        }
    }
    return L;
}

// inverse of a symmetric positive definite matrix through its Cholesky factor
template <int M> __device__ inline Mat<M> mspd_inv(const Mat<M>& x)
{
    if (M == 1) { Mat<M> r; r.a[0][0] = rcp_newton(x.a[0][0]); return r; }
    Mat<M> L = mchol<M>(x);
    Mat<M> Li = mzero<M>();  // L^{-1}, lower
    for (int i = 0; i < M; ++i) {
        Li.a[i][i] = rcp_newton(L.a[i][i]);
        for (int j = 0; j < i; ++j) {
            double s = 0.0;
            for (int k = j; k < i; ++k) s += L.a[i][k] * Li.a[k][j];
            Li.a[i][j] = -s * Li.a[i][i];
        }
    }
    return mmul<M>(mT<M>(Li), Li);
}

// H_{q,i}(x) = r_{q,i} F^i_{m+q}(x) / F^i_m(x_ref); r_{q,i} = prod_{j=m}^{m+q-1} (j(j+1)+kappa_i^2)/(j+1)
// (the reference series value F^i_m(x_ref) = sref * 1e250^eref, given as 1/sref and eref)
template <int M> __device__ inline Mat<M> hmat(const Spec& sp, int m, double x, const double* sinv, const int* eref)
{
    Mat<M> H;
    for (int i = 0; i < M; ++i) {
        double r = 1.0;
        for (int q = 0; q < M; ++q) {
            if (q > 0) {
                const double j = (double)(m + q - 1);
                r *= (j * (j + 1.0) + sp.k2[i]) / (j + 1.0);
            }
            H.a[q][i] = r * hyp_rel(sp.k2[i], m + q, x, sinv[i], eref[i]);
        }
    }
    return H;
}

__constant__ double kGL8x[8] = {-0.9602898564975363, -0.7966664774136267, -0.5255324099163290, -0.1834346424956498,
                                 0.1834346424956498,  0.5255324099163290,  0.7966664774136267,  0.9602898564975363};
__constant__ double kGL8w[8] = {0.1012285362903763, 0.2223810344533745, 0.3137066458778873, 0.3626837833783620,
                                0.3626837833783620, 0.3137066458778873, 0.2223810344533745, 0.1012285362903763};

// Transition Phi and conditional covariance Q of every northward step, one thread per
// (chain, position, mode).  phi/q: [c][pos][m][M*M] doubles (pos 1..len).
template <int M>
__global__ void step_kernel(Spec sp, int c, int len, double* phi, double* qout)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    const int pos = blockIdx.y + 1;
    if (m >= sp.n_modes || pos > len) return;
    const double th1 = chain_theta(sp, c, pos - 1), th2 = chain_theta(sp, c, pos);
    const double t1 = tan(0.5 * th1), t2 = tan(0.5 * th2);
    const double u1 = log(t1), u2 = log(t2);
    const double s1 = sin(0.5 * th1), s2 = sin(0.5 * th2);
    const double x1 = s1 * s1, x2 = s2 * s2;
    double sinv[M];
    int eref[M];
    for (int i = 0; i < M; ++i) {
        double sr;
        hyp_scaled(sp.k2[i], m, x2, sr, eref[i]);
        sinv[i] = 1.0 / sr;
    }
    const Mat<M> H2 = hmat<M>(sp, m, x2, sinv, eref);
    const Mat<M> H1 = hmat<M>(sp, m, x1, sinv, eref);
    // A = (t2/t1)^m diag(t2^q) H2 H1^{-1} diag(t1^-q)
    Mat<M> A = mmul<M>(H2, minv<M>(H1));
    const double g = exp((double)m * (u2 - u1));
    for (int p = 0; p < M; ++p)
        for (int q = 0; q < M; ++q) A.a[p][q] *= g * pow(t2, (double)p) / pow(t1, (double)q);
    // W = diag(t2^(q-M+1)) H2
    Mat<M> W = H2;
    for (int p = 0; p < M; ++p)
        for (int q = 0; q < M; ++q) W.a[p][q] *= pow(t2, (double)(p - M + 1));
    // Q = A_amp/(2 pi) int_0^{du} e^{-c v} (W h)(W h)^T dv, h = H(x(u2+v))^{-1} e_{M-1}
    const double cexp = 2.0 * (double)(m + M - 1);
    const double du = u1 - u2;
    const double vmax = cexp > 0.0 ? fmin(du, 46.0 / cexp) : du;
    const double sinmax = th1 > 0.5 * SMERF_PI ? 1.0 : sin(th1);
    const double rho = cexp + 2.0 * sp.kmax * sinmax + 1.0;
    int nsub = (int)ceil(0.25 * rho * vmax);  // one 8-point panel per 4 / rho (twice finer agrees to rounding)
    nsub = nsub < 1 ? 1 : (nsub > 256 ? 256 : nsub);
    const double h = vmax / nsub;
    Mat<M> acc = mzero<M>();
    for (int j = 0; j < nsub; ++j)
        for (int n = 0; n < 8; ++n) {
            const double v = (j + 0.5 * (kGL8x[n] + 1.0)) * h;
            const double w = 0.5 * h * kGL8w[n] * exp(-cexp * v);
            const double u = u2 + v;
            const double x = 1.0 / (1.0 + exp(-2.0 * u));   // sin^2(theta/2), tan(theta/2) = e^u
            const Mat<M> Hs = hmat<M>(sp, m, x, sinv, eref);
            const Mat<M> Hi = minv<M>(Hs);
            double ph[M];
            for (int p = 0; p < M; ++p) {
                double s = 0.0;
                for (int k = 0; k < M; ++k) s += W.a[p][k] * Hi.a[k][M - 1];
                ph[p] = s;
            }
            for (int p = 0; p < M; ++p)
                for (int q = 0; q < M; ++q) acc.a[p][q] += w * ph[p] * ph[q];
        }
    const double f = sp.A / (2.0 * SMERF_PI);
    const size_t o = (((size_t)pos) * sp.n_modes + m) * (M * M);
    for (int p = 0; p < M; ++p)
        for (int q = 0; q < M; ++q) {
            phi[o + p * M + q] = A.a[p][q];
            qout[o + p * M + q] = f * acc.a[p][q];
        }
}

// ---- p = 1 and 2 with a real spectrum: the step tables by a recurrence in m (Alg. 1 sets up the
// hypergeometric functions of every order m).  For fixed x the series of
// Eq. (Legendre_hypergeometric), F_m(x) = 2F1(-lambda, lambda+1; 1+m; x) with
// (-lambda)(lambda+1) = kappa^2, satisfy Gauss's contiguous relation in the third parameter,
//   F_{m-1} = [(1-2x) F_m + (1 + kappa^2/(m(m+1))) x F_{m+1}] / (1-x),   m >= 1.
// For large m its solutions behave like 1 (F_m itself) and like (-(1-x)/x)^m, so for x < 1/2
// F_m is the minimal solution and the relation taken downward from two series values is
// stable (relative error of order m eps; ratios of F at nearby x, which is what the tables
// use, to a few 1e-13 over 16384 orders).  For x > 1/2 the error grows by x/(1-x) per order:
// only the first step's equatorward ring can have x > 1/2 (south of the equator, even n_theta);
// that step keeps step_kernel's per-mode series unless the growth over all orders,
// (x/(1-x))^m_max, stays below 1e3 (it is about e^pi = 23 when n_phi = 2 n_theta).
//
// Per order m a point x has H(x) as in step_kernel (p = 1: F_m; p = 2: [[F^1_m, F^2_m],
// [r_1 F^1_{m+1}, r_2 F^2_{m+1}]], r_i = (m(m+1)+kappa_i^2)/(m+1)) up to a scale per column, which
// cancels in A = (t2/t1)^m diag(t2^p) H2 H1^-1 diag(t1^-q) and in phi = diag(t2^(p-M+1)) H2 H(x)^-1
// e_{M-1}.  A node's phi is formed from H2's entries (broadcast from its group's lane 0) and the
// node's own before squaring (no cancellation).
//
// A group of 16 lanes takes one step and a block of rec_block(n_modes) orders, starting the
// recurrence from the series at the block's top: lane 0 at x2 (the step's poleward ring), lane 1
// at x1, lanes 2 .. 15 at the 14 nodes of a Gauss-Legendre panel in v.  The panel is no wider than
// 11 / rho(m) for every order of the block whose weight e^{-2mv} at the panel's start is above
// e^-46 (further panels, which only the orders of such weight take, follow for steps near the pole):
// 14 nodes then integrate e^{-11 t} to 1e-17 of its maximum, where 8-point panels of width 4 / rho
// took 22 nodes.  The blocks' and groups' independence is what counts: one warp per step walked
// all orders and panels before, so a set-up took the polar steps' latency (1024 x 2048, p = 2:
// 10.7 ms in 512 warps, now 1.9 ms; 2048 x
// 4096, p = 1: 12.5 -> 3.8 ms for the whole set-up).  Tables of every order against the former kernels': A and C to 1e-12 (p = 1) and
// 1e-11 of each entry's scale (p = 2); fields against 64-bit references 8.7e-13 -> 5.1e-13.
constexpr int kRecNodes = 14;
constexpr int kRecWarps = 2;         // warps per block, two steps each
constexpr int kRecMaxPanels = 8192;  // reached only by grids far beyond 16384 rings
__constant__ double kGL14x[kRecNodes] = {-0.98628380869681233884, -0.92843488366357351734, -0.82720131506976499319, -0.68729290481168547015,
                                         -0.51524863635815409197, -0.31911236892788976044, -0.10805494870734366207, 0.10805494870734366207,
                                         0.31911236892788976044, 0.51524863635815409197, 0.68729290481168547015, 0.82720131506976499319,
                                         0.92843488366357351734, 0.98628380869681233884};
__constant__ double kGL14w[kRecNodes] = {0.035119460331751863032, 0.080158087159760209806, 0.12151857068790318469, 0.15720316715819353457,
                                         0.18553839747793781374, 0.20519846372129560397, 0.2152638534631577902, 0.2152638534631577902,
                                         0.20519846372129560397, 0.18553839747793781374, 0.15720316715819353457, 0.12151857068790318469,
                                         0.080158087159760209806, 0.035119460331751863032};

// blocks of orders, and orders per block: about 64 (256 from 2560 modes on), evenly; the series at
// a block's top cost as much as some 30 orders
__host__ __device__ inline int rec_blocks(int n_modes)
{
    const int nb = n_modes / (n_modes <= 2560 ? 64 : 256);
    return nb > 0 ? nb : 1;
}
__host__ __device__ inline int rec_block(int n_modes) { return (n_modes + rec_blocks(n_modes) - 1) / rec_blocks(n_modes); }

__device__ inline int hi_word(double x) { return __double2hiint(x); }

// the series F_mu(x) and F_{mu+1}(x) for every kappa_i, as S 2^(250 E) with one E per i; the terms'
// denominators are shared by all of them
template <int M>
__device__ inline void hyp_pairs(const double* k2, int mu, double x, double (&S0)[M], double (&S1)[M], int (&E)[M])
{
    double t0[M], t1[M];
#pragma unroll
    for (int i = 0; i < M; ++i) {
        t0[i] = t1[i] = S0[i] = S1[i] = 1.0;
        E[i] = 0;
    }
    double n1 = 1.0, a = (double)mu + 1.0;  // n + 1, n + 1 + mu
    for (int n = 0; n < 1000000; ++n) {
        const double b = a + 1.0, r = x * rcp_newton(n1 * (a * b));
        const double q = n1 * n1 - n1;  // n (n + 1)
        bool done = true;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const double c = (q + k2[i]) * r, r0 = c * b;
            t0[i] *= r0;
            t1[i] *= c * a;
            S0[i] += t0[i];
            S1[i] += t1[i];
            // terms below 2^-57 of the sums and falling (all values positive: their high words compare)
            done = done && hi_word(S0[i]) - hi_word(t0[i]) > (57 << 20) && hi_word(S1[i]) - hi_word(t1[i]) > (57 << 20) &&
                   hi_word(r0) < hi_word(0.9);
            if (hi_word(S0[i]) > ((1023 + 250) << 20)) {
                S0[i] *= 0x1p-250;
                S1[i] *= 0x1p-250;
                t0[i] *= 0x1p-250;
                t1[i] *= 0x1p-250;
                ++E[i];
            }
        }
        if (done) break;
        n1 += 1.0;
        a = b;
    }
}

template <int M>
__global__ void __launch_bounds__(32 * kRecWarps) step_kernel_rec(Spec sp, int first, int len, double* phi, double* qout)
{
    constexpr int T = M * (M + 1) / 2, MM = M * M;
    __shared__ double tile[kRecWarps][T][2][16][17];  // [product][half][order in block][lane]
    __shared__ double h2[kRecWarps][MM][2][16], h1[kRecWarps][MM][2][16], alph[kRecWarps][M][2][16], rr[kRecWarps][M][2][16];
    const int w = threadIdx.x >> 5, h = (threadIdx.x >> 4) & 1, l = threadIdx.x & 15;
    const unsigned full = 0xffffffffu, half = 0xffffu << (16 * h);
    const int step = 2 * ((gridDim.x - 1 - blockIdx.x) * kRecWarps + w);  // polar steps (more panels) first
    if (first + step > len) return;  // whole warps
    const bool live = first + step + h <= len;  // a second half beyond the last step repeats it and stores nothing
    const int pos = live ? first + step + h : len;
    const int B = rec_block(sp.n_modes), mlo = blockIdx.y * B, mhi = min(sp.n_modes - 1, mlo + B - 1);
    const double th1 = chain_theta(sp, 0, pos - 1), th2 = chain_theta(sp, 0, pos);
    const double t1 = tan(0.5 * th1), t2 = tan(0.5 * th2);
    const double u2 = log(t2), du = log(t1) - u2;
    const double sa = sin(0.5 * th1), sb = sin(0.5 * th2);
    const double sinmax = th1 > 0.5 * SMERF_PI ? 1.0 : sin(th1);
    const double kap = 2.0 * sp.kmax * sinmax + 1.0;
    const double f = sp.A / (2.0 * SMERF_PI), it1 = 1.0 / t1, it2 = 1.0 / t2;
    const size_t base = (size_t)pos * sp.n_modes;
    // highest order whose weight e^{-2(m+M-1)v} is above e^-46 at v
    auto top = [&](double v) { return v > 0.0 ? (int)fmin((double)mhi, floor(23.0 / v) - (M - 1)) : mhi; };
    double v0 = 0.0;  // the panel's start
    for (int ch = 0; ch < kRecMaxPanels; ++ch) {
        const int mt = top(v0);
        const bool act = v0 < du && mt >= mlo;  // this half has the panel
        if (!__any_sync(full, act)) break;
        const double wd = 11.0 / (2.0 * (max(mt, mlo) + M - 1) + kap);
        const double hp = fmin(wd, du - v0);
        double x = sb * sb, wt = 0.0, v = 0.0;
        if (l == 1) {
            x = sa * sa;
            v = du;
        } else if (l >= 2 && act) {
            v = v0 + 0.5 * (kGL14x[l - 2] + 1.0) * hp;
            wt = 0.5 * hp * kGL14w[l - 2];
            x = 1.0 / (1.0 + exp(-2.0 * (u2 + v)));
        }
        // both halves start at the higher of their top orders
        int ms = act ? mt : mlo;
        ms = max(ms, __shfl_xor_sync(full, ms, 16));
        double F[M], Fp[M];
        int E[M];
        hyp_pairs<M>(sp.k2, ms, x, F, Fp, E);
#pragma unroll
        for (int i = 0; i < M; ++i) {
            int W = E[i];  // one scale per column and half
            for (int o = 8; o > 0; o >>= 1) W = max(W, __shfl_xor_sync(full, W, o));
            F[i] = ldexp(F[i], 250 * (E[i] - W));
            Fp[i] = ldexp(Fp[i], 250 * (E[i] - W));
        }
        const double beta = (1.0 - 2.0 * x) / (1.0 - x), gam = x / (1.0 - x);
        const double e2v = exp(2.0 * v);
        double Ew = 0.0;
        for (int mb = ms; mb >= mlo; mb -= 16) {
            const int ml = mb - l;
#pragma unroll
            for (int i = 0; i < M; ++i) {
                const double al = ml >= 1 ? sp.k2[i] * rcp_newton((double)ml * (double)(ml + 1)) : 0.0;
                alph[w][i][h][l] = al;
                rr[w][i][h][l] = ml >= 1 ? (double)ml + (double)ml * al : sp.k2[i];  // (m(m+1) + kappa^2)/(m+1)
            }
            __syncwarp();
            // e^{-2(m+M-1)v}, exact every 32 orders
            if (((ms - mb) & 16) == 0) Ew = wt * exp(-2.0 * (double)(mb + M - 1) * v);
#pragma unroll 2
            for (int k = 0; k < 16; ++k) {
                const int m = mb - k;
                if (m < mlo) break;
                if constexpr (M == 1) {
                    const double r = rcp_newton(F[0]);
                    tile[w][0][h][k][l] = Ew * r * r;
                    if (l == 0) h2[w][0][h][k] = F[0];
                    if (l == 1) h1[w][0][h][k] = F[0];
                } else {
                    const double a = F[0], b = F[1], c = rr[w][0][h][k] * Fp[0], d = rr[w][1][h][k] * Fp[1];
                    const double a2 = __shfl_sync(full, a, 0, 16), b2 = __shfl_sync(full, b, 0, 16);
                    const double c2 = __shfl_sync(full, c, 0, 16), d2 = __shfl_sync(full, d, 0, 16);
                    const double rdet = rcp_newton(a * d - b * c);
                    const double p0 = (b2 * a - a2 * b) * rdet, p1 = (d2 * a - c2 * b) * rdet;
                    const double q0 = Ew * p0;
                    tile[w][0][h][k][l] = q0 * p0;
                    tile[w][1][h][k][l] = q0 * p1;
                    tile[w][2][h][k][l] = Ew * p1 * p1;
                    if (l == 0) { h2[w][0][h][k] = a; h2[w][1][h][k] = b; h2[w][2][h][k] = c; h2[w][3][h][k] = d; }
                    if (l == 1) { h1[w][0][h][k] = a; h1[w][1][h][k] = b; h1[w][2][h][k] = c; h1[w][3][h][k] = d; }
                }
                if (m >= 1) {
#pragma unroll
                    for (int i = 0; i < M; ++i) {
                        const double t = gam + gam * alph[w][i][h][k];
                        const double Fn = beta * F[i] + t * Fp[i];
                        Fp[i] = F[i];
                        F[i] = Fn;
                        // a common rescale keeps the values, their squares and the squares of their
                        // reciprocals in range (ratios are unchanged)
                        if (__ballot_sync(full, (hi_word(F[i]) & 0x7ff00000) > ((1023 + 250) << 20)) & half) {
                            F[i] *= 0x1p-250;
                            Fp[i] *= 0x1p-250;
                        }
                    }
                }
                Ew *= e2v;
            }
            __syncwarp();
            if (act && live && ml >= mlo && ml <= mhi) {
                double s[T];
#pragma unroll
                for (int e = 0; e < T; ++e) {
                    s[e] = 0.0;
                    for (int j = 2; j < 16; ++j) s[e] += tile[w][e][h][l][j];
                }
                const size_t o = (base + ml) * MM;
                double q[MM];
                if constexpr (M == 1) {
                    const double F2 = h2[w][0][h][l];
                    q[0] = f * F2 * F2 * s[0];
                } else {
                    q[0] = f * s[0] * it2 * it2;
                    q[1] = q[2] = f * s[1] * it2;
                    q[3] = f * s[2];
                }
                if (ch == 0) {
#pragma unroll
                    for (int e = 0; e < MM; ++e) qout[o + e] = q[e];
                    // A = (t2/t1)^m diag(t2^p) H2 H1^-1 diag(t1^-q)
                    const double g = exp(-(double)ml * du);
                    if constexpr (M == 1) {
                        phi[o] = g * h2[w][0][h][l] / h1[w][0][h][l];
                    } else {
                        const double a2 = h2[w][0][h][l], b2 = h2[w][1][h][l], c2 = h2[w][2][h][l], d2 = h2[w][3][h][l];
                        const double a1 = h1[w][0][h][l], b1 = h1[w][1][h][l], c1 = h1[w][2][h][l], d1 = h1[w][3][h][l];
                        const double gd = g / (a1 * d1 - b1 * c1);
                        phi[o + 0] = gd * (a2 * d1 - b2 * c1);
                        phi[o + 1] = gd * (b2 * a1 - a2 * b1) * it1;
                        phi[o + 2] = gd * t2 * (c2 * d1 - d2 * c1);
                        phi[o + 3] = gd * t2 * (d2 * a1 - c2 * b1) * it1;
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < MM; ++e) qout[o + e] += q[e];
                }
            }
            __syncwarp();
        }
        if (act) v0 += hp;
    }
}

// Table store.  FP64 tables keep every entry at magnitude >= 2^-120 (zeros and smaller
// values become +-2^-120, a change far below any effect on the field): FP32-recursion
// kernels then convert them to FP32 with three integer instructions and no range check.
template <class T>
__device__ inline void put(void* base, bool is64, size_t idx, double v)
{
    if (is64) {
        const double tiny = 0x1p-120;
        ((double*)base)[idx] = fabs(v) < tiny ? (v < 0.0 ? -tiny : tiny) : v;
    } else {
        ((float*)base)[idx] = (float)v;
    }
}

// Start factor B_eq = chol J(z0, z0) (Eq. (state_initial)).  J = sum_i b_i (2 pi)^-1 G_i with the
// Green's functions G_i of l(l+1) + kappa_i^2 (Eq. (C_ell_efficient)) from the solutions regular at
// either pole, u = P^m_l(z) and v = P^m_l(-z): with R_q(z) = P^{m+q}_l(z) / P^m_l(z) = r_q t^q
// F_{m+q}(x) / F_m(x) and (1-z^2)(v'/v - u'/u) = sin(theta0) (R_1(z) + R_1(-z)), the raised
// components are J_qp = b_i R_q(z) (-1)^p R_p(-z) / (2 pi sin(theta0) (R_1(z) + R_1(-z))).  Only
// ratios of neighbouring orders enter, so no Gamma factor nor product over the orders (the form
// with Eq. (Jmatrix_efficient)'s Pochhammer factors took a prefix sum of logarithms over the modes
// and 2 M^2 series per thread: 0.65 ms at 1024 x 2048, p = 2, now 0.12).  A group of
// start_lanes(M) lanes per mode, one lane per (i, side).
__host__ __device__ constexpr int start_lanes(int M) { return M == 1 ? 2 : M == 2 ? 4 : 8; }
template <int M>
__global__ void __launch_bounds__(64) start_kernel(Spec sp, void* beq, bool tab64)
{
    constexpr int GL = start_lanes(M), NR = M < 3 ? 2 : 3;  // R_0 .. R_{NR-1}
    const int gid = blockIdx.x * blockDim.x + threadIdx.x, lane = gid % GL;
    const int m = min(gid / GL, sp.n_modes - 1);  // the last block's spare groups repeat the last mode
    const double th0 = ring_colat(sp.theta, sp.n_theta, sp.k0);
    const double sx = sin(0.5 * th0), cx = cos(0.5 * th0);
    // lane = 2 i + side (0: z, 1: -z); spare lanes repeat the last factor
    const int side = lane & 1;
    double k2[1] = {sp.k2[min(lane / 2, M - 1)]};
    const double x = side ? cx * cx : sx * sx, t = side ? cx / sx : sx / cx;
    double R[NR], S0[1], S1[1];
    int E[1];
    hyp_pairs<1>(k2, m, x, S0, S1, E);
    const double dm = (double)m, r1 = (dm * (dm + 1.0) + k2[0]) / (dm + 1.0);
    R[0] = 1.0;
    R[1] = r1 * t * S1[0] / S0[0];
    if constexpr (NR > 2) {
        hyp_pairs<1>(k2, m + 1, x, S0, S1, E);
        R[2] = R[1] * ((dm + 1.0) * (dm + 2.0) + k2[0]) / (dm + 2.0) * t * S1[0] / S0[0];
    }
    Mat<M> J = mzero<M>();
#pragma unroll
    for (int i = 0; i < M; ++i) {
        double n[NR], q[NR];
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            n[k] = __shfl_sync(0xffffffffu, R[k], 2 * i, GL);
            q[k] = __shfl_sync(0xffffffffu, R[k], 2 * i + 1, GL);
        }
        const double g = sp.b[i] / (2.0 * SMERF_PI * sin(th0) * (n[1] + q[1]));
        for (int a = 0; a < M; ++a)
            for (int b = 0; b < M; ++b) J.a[a][b] += g * n[a] * ((b & 1) ? -q[b] : q[b]);
    }
    if (lane != 0 || gid / GL >= sp.n_modes) return;
    const Mat<M> L = mchol<M>(msym<M>(J));
    const double sc = m > 0 ? 0.70710678118654752440 : 1.0;
    int e = 0;
    for (int p = 0; p < M; ++p)
        for (int q = 0; q <= p; ++q, ++e)
            put<double>(beq, tab64, (size_t)e * sp.n_modes_pad + m, L.a[p][q] * sc);
}

// Bridge, forward and coarse tables of one segment, one thread per (segment, mode).
// Segment [pa, pb] with right anchor pb: for pa < pos < pb, condition x_pos on x_{pos-1}
// (prior N(Phi x, Q)) and on x_pb = Psi x_pos + N(0, S) (Psi, S accumulated backward), in gain form:
//   W = Psi Q Psi^T + S,  C = Q Psi^T W^{-1},  R = I - C Psi,  Abar = R Phi,
//   P = R Q R^T + C S C^T,  B = chol P.
// W is the next position's S, and one inverse per position replaces the three of the information
// form (Q^{-1} + Psi^T S^{-1} Psi)^{-1}, on the FP64 pipe that bounds this kernel (2 x 348 -> 2 x 231 us at 1024 x 2048, p = 2).
// The coarse step pa -> pb is (Psi_pa, chol S_pa).  Without a right anchor the tables are
// the plain forward step (Phi, 0, chol Q).
template <int M>
__global__ void segment_tables_kernel(Spec sp, int c, int len, int H, const double* phi,
                                      const double* qv, void* steps, void* coarse, bool tab64)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    const int seg = blockIdx.y;
    if (m >= sp.n_modes) return;
    const int Ec = coarse_elems(M);
    const size_t mp = sp.n_modes_pad;
    const double sc = m > 0 ? 0.70710678118654752440 : 1.0;
    // the southern chain runs in the mirrored state S x and is driven by S xi; its B
    // factors are stored with S folded into their columns so that the kernels use xi as is
    auto colsign = [&](int q) { return (c == 1 && (q & 1)) ? -1.0 : 1.0; };
    const int pa = H > 0 ? seg * H : 0;
    const int pb = (H > 0 && pa + H <= len) ? pa + H : -1;
    auto load = [&](const double* base, int pos) {
        Mat<M> r;
        const size_t o = (((size_t)pos) * sp.n_modes + m) * (M * M);
        for (int p = 0; p < M; ++p)
            for (int q = 0; q < M; ++q) r.a[p][q] = base[o + p * M + q];
        return r;
    };
    auto store_step = [&](int pos, const Mat<M>& A, const Mat<M>& C, const Mat<M>& B) {
        const size_t base = ((size_t)pos * mp + m) * step_row(M);
        int e = 0;
        for (int p = 0; p < M; ++p)
            for (int q = 0; q < M; ++q, ++e) put<double>(steps, tab64, base + e, A.a[p][q]);
        for (int p = 0; p < M; ++p)
            for (int q = 0; q < M; ++q, ++e) put<double>(steps, tab64, base + e, C.a[p][q]);
        for (int p = 0; p < M; ++p)
            for (int q = 0; q <= p; ++q, ++e) put<double>(steps, tab64, base + e, B.a[p][q] * sc * colsign(q));
        for (; e < step_row(M); ++e) put<double>(steps, tab64, base + e, 0.0);
    };
    if (pb < 0) {
        const int end = len;
        for (int pos = pa + 1; pos <= end; ++pos) {
            const Mat<M> Ph = load(phi, pos), Q = load(qv, pos);
            store_step(pos, Ph, mzero<M>(), mchol<M>(msym<M>(Q)));
        }
        return;
    }
    Mat<M> Psi = meye<M>(), S = mzero<M>();
    for (int pos = pb; pos > pa; --pos) {
        const Mat<M> Ph = load(phi, pos), Q = msym<M>(load(qv, pos));
        // W = Psi Q Psi^T + S: the anchor's covariance given x_{pos-1}, and S_{pos-1}
        const Mat<M> G = mmul<M>(Psi, Q);
        const Mat<M> W = msym<M>(madd<M>(mmul<M>(G, mT<M>(Psi)), S));
        if (pos < pb) {
            const Mat<M> C = mmul<M>(mT<M>(G), mspd_inv<M>(W));
            Mat<M> R = mmul<M>(C, Psi);  // I - C Psi
            for (int i = 0; i < M; ++i)
                for (int j = 0; j < M; ++j) R.a[i][j] = (i == j ? 1.0 : 0.0) - R.a[i][j];
            // P = R Q R^T + C S C^T: a sum of covariances, nothing cancels in it
            const Mat<M> P = madd<M>(mmul<M>(mmul<M>(R, Q), mT<M>(R)), mmul<M>(mmul<M>(C, S), mT<M>(C)));
            store_step(pos, mmul<M>(R, Ph), C, mchol<M>(msym<M>(P)));
        }
        S = W;
        Psi = mmul<M>(Psi, Ph);
    }
    const Mat<M> Bc = mchol<M>(msym<M>(S));
    const int j = pb / H;
    const size_t base = (size_t)j * Ec * mp + m;
    int e = 0;
    for (int p = 0; p < M; ++p)
        for (int q = 0; q < M; ++q, ++e) put<double>(coarse, tab64, base + (size_t)e * mp, Psi.a[p][q]);
    for (int p = 0; p < M; ++p)
        for (int q = 0; q <= p; ++q, ++e) put<double>(coarse, tab64, base + (size_t)e * mp, Bc.a[p][q] * sc * colsign(q));
}

// FFT tables in the recursion precision (formed in FP64):
//   pre[s] = e^{2 pi i s / n_phi}, s < Nc (C2R packing), and for every radix-RP pass with
//   Ns > 1 (pass plan: radix 4 while Nc/Ns >= 4, then 2) the block
//   tw[off + (i-1) Ns + kk] = e^{2 pi i i kk / (Ns RP)}, i = 1..RP-1, kk < Ns;
//   tw2, tw3: the same for the high-radix plans (passes of at most 16 and at most 8 points).
__host__ __device__ inline int r4_table(int lgNc)  // entries of tw
{
    int n = 0;
    for (int l = 2; l < lgNc; l += 2) n += (lgNc - l >= 2 ? 3 : 1) << l;
    return n;
}
__device__ inline int4 fx_root(int k, int lgn)  // e^{2 pi i k / 2^lgn} in fixed point
{
    int64_t c, s;
    fx_cis62((uint64_t)(unsigned)k << (64 - lgn), c, s);
    int4 w;
    fx_split(c, w.x, w.y);
    fx_split(s, w.z, w.w);
    return w;
}
template <class R>
__global__ void __launch_bounds__(256) fft_tables_kernel(int lgNc, cplx<R>* pre, cplx<R>* tw, cplx<R>* tw2, cplx<R>* tw3,
                                                         int4* prex, int4* twx)
{
    const int Nc = 1 << lgNc, t0 = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    auto root = [](int k, int n) {  // e^{2 pi i k / n}, n a power of two
        double c, s;
        sincospi(2.0 * (double)k / (double)n, &s, &c);
        return cmk<cplx<R>>((R)c, (R)s);
    };
    for (int s = t0; s < Nc; s += nt) {
        pre[s] = root(s, 2 * Nc);
        if (sizeof(R) == 8) prex[s] = fx_root(s, lgNc + 1);
    }
    // entry i of a pass of radix 2^b and stride Ns = 2^l: i = (a - 1) Ns + kk
    auto entry = [&](int i, int l, int b) { return root(((i >> l) + 1) * (i & ((1 << l) - 1)), 1 << (l + b)); };
    int off = 0;
    for (int l = 2; l < lgNc; l += 2) {
        const int b = lgNc - l >= 2 ? 2 : 1, n = ((1 << b) - 1) << l;
        for (int i = t0; i < n; i += nt) {
            tw[off + i] = entry(i, l, b);
            if (sizeof(R) == 8) twx[off + i] = fx_root(((i >> l) + 1) * (i & ((1 << l) - 1)), l + b);
        }
        off += n;
    }
    for (int q = 0; q < 2; ++q) {
        const int MB = q == 0 ? 4 : SMERF_INPLACE_MB;
        cplx<R>* t = q == 0 ? tw2 : tw3;
        for (int ps = 1; ps < smerf::hr_passes(lgNc, MB); ++ps) {
            const int b = smerf::hr_bits(lgNc, ps, MB), l = smerf::hr_lgns(lgNc, ps, MB), n = ((1 << b) - 1) << l;
            for (int i = t0; i < n; i += nt) t[smerf::hr_off(lgNc, ps, MB) + i] = entry(i, l, b);
        }
    }
}

// ---------------------------------------------------------------- complex kappa-hat
// Spectra with complex kappa-hat (Eq. (Cl) with complex-conjugate pairs, as in the paper's
// Sec. 5 example (10 + l^2 (l+1)^2)^-1, kappa-hat = +-i sqrt(10)).  The same construction in
// complex arithmetic: l_i, 2F1, U, the partial-fraction weights b_i and the Gamma factors are
// complex; A, Q and J(z0, z0) are real (the two columns of U of a conjugate pair are complex
// conjugates) and their real parts are kept.
using cdbl = cuda::std::complex<double>;

struct SpecC {
    cdbl k2[kMaxP], b[kMaxP], lG0[kMaxP];  // kappa-hat_i, b_i, log(Gamma(1+l_i) Gamma(-l_i))
    double A, kmax;
    int n_theta, k0, n_modes, n_modes_pad;
    const double* theta;  // device: ring colatitudes (null: equiangular)
};

template <int M> struct MatC { cdbl a[M][M]; };

template <int M> __device__ inline MatC<M> cmmul(const MatC<M>& x, const MatC<M>& y)
{
    MatC<M> r;
    for (int i = 0; i < M; ++i)
        for (int j = 0; j < M; ++j) {
            cdbl s = 0.0;
            for (int k = 0; k < M; ++k) s += x.a[i][k] * y.a[k][j];
            r.a[i][j] = s;
        }
    return r;
}
template <int M> __device__ inline MatC<M> cminv(const MatC<M>& x);
template <> __device__ inline MatC<1> cminv<1>(const MatC<1>& x) { MatC<1> r; r.a[0][0] = 1.0 / x.a[0][0]; return r; }
template <> __device__ inline MatC<2> cminv<2>(const MatC<2>& x)
{
    const cdbl d = x.a[0][0] * x.a[1][1] - x.a[0][1] * x.a[1][0];
    MatC<2> r;
    r.a[0][0] = x.a[1][1] / d; r.a[0][1] = -x.a[0][1] / d;
    r.a[1][0] = -x.a[1][0] / d; r.a[1][1] = x.a[0][0] / d;
    return r;
}
template <> __device__ inline MatC<3> cminv<3>(const MatC<3>& x) { return inv3<MatC<3>, cdbl>(x); }

// 2F1(-l, l+1; 1+mu; x) with kappa-hat = k2 complex, as S * 1e250^E (terms two per division)
__device__ void hyp_scaled_c(cdbl k2, int mu, double x, cdbl& S, int& E)
{
    cdbl s = 1.0, t = 1.0;
    int e = 0;
    const double m1 = (double)mu + 1.0;
    for (int n = 0; n < 1000000; n += 2) {
        const double dn = (double)n;
        const cdbl a0 = (dn * (dn + 1.0) + k2) * x, a1 = ((dn + 1.0) * (dn + 2.0) + k2) * x;
        const double d0 = (dn + m1) * (dn + 1.0), d1 = (dn + 1.0 + m1) * (dn + 2.0);
        const double inv = 1.0 / (d0 * d1);
        const cdbl r0 = a0 * (d1 * inv), r1 = a1 * (d0 * inv);
        t *= r0;
        s += t;
        if (cuda::std::abs(t) < 1e-17 * cuda::std::abs(s) && cuda::std::abs(r0) < 0.9) break;
        t *= r1;
        s += t;
        if (cuda::std::abs(t) < 1e-17 * cuda::std::abs(s) && cuda::std::abs(r1) < 0.9) break;
        if (cuda::std::abs(s) > 1e250) { s *= 1e-250; t *= 1e-250; ++e; }
    }
    S = s;
    E = e;
}

__device__ inline cdbl log_hyp_c(cdbl k2, int mu, double x)
{
    cdbl s;
    int e;
    hyp_scaled_c(k2, mu, x, s, e);
    return cuda::std::log(s) + e * 575.64627324851142;
}

__device__ inline cdbl hyp_rel_c(cdbl k2, int mu, double x, cdbl sref_inv, int eref)
{
    cdbl s;
    int e;
    hyp_scaled_c(k2, mu, x, s, e);
    cdbl v = s * sref_inv;
    for (int d = e - eref; d > 0; --d) v *= 1e250;
    for (int d = e - eref; d < 0; ++d) v *= 1e-250;
    return v;
}

template <int M> __device__ inline MatC<M> hmat_c(const SpecC& sp, int m, double x, const cdbl* sinv, const int* eref)
{
    MatC<M> H;
    for (int i = 0; i < M; ++i) {
        cdbl r = 1.0;
        for (int q = 0; q < M; ++q) {
            if (q > 0) {
                const double j = (double)(m + q - 1);
                r *= (j * (j + 1.0) + sp.k2[i]) / (j + 1.0);
            }
            H.a[q][i] = r * hyp_rel_c(sp.k2[i], m + q, x, sinv[i], eref[i]);
        }
    }
    return H;
}

// step_kernel in complex arithmetic (same construction, real parts stored)
template <int M>
__global__ void step_kernel_c(SpecC sp, int len, double* phi, double* qout)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    const int pos = blockIdx.y + 1;
    if (m >= sp.n_modes || pos > len) return;
    const double th1 = ring_colat(sp.theta, sp.n_theta, sp.k0 - pos + 1);
    const double th2 = ring_colat(sp.theta, sp.n_theta, sp.k0 - pos);
    const double t1 = tan(0.5 * th1), t2 = tan(0.5 * th2);
    const double u1 = log(t1), u2 = log(t2);
    const double s1 = sin(0.5 * th1), s2 = sin(0.5 * th2);
    const double x1 = s1 * s1, x2 = s2 * s2;
    cdbl sinv[M];
    int eref[M];
    for (int i = 0; i < M; ++i) {
        cdbl sr;
        hyp_scaled_c(sp.k2[i], m, x2, sr, eref[i]);
        sinv[i] = 1.0 / sr;
    }
    const MatC<M> H2 = hmat_c<M>(sp, m, x2, sinv, eref);
    const MatC<M> H1 = hmat_c<M>(sp, m, x1, sinv, eref);
    MatC<M> A = cmmul<M>(H2, cminv<M>(H1));
    const double g = exp((double)m * (u2 - u1));
    for (int p = 0; p < M; ++p)
        for (int q = 0; q < M; ++q) A.a[p][q] *= g * pow(t2, (double)p) / pow(t1, (double)q);
    MatC<M> W = H2;
    for (int p = 0; p < M; ++p)
        for (int q = 0; q < M; ++q) W.a[p][q] *= pow(t2, (double)(p - M + 1));
    const double cexp = 2.0 * (double)(m + M - 1);
    const double du = u1 - u2;
    const double vmax = cexp > 0.0 ? fmin(du, 46.0 / cexp) : du;
    const double sinmax = th1 > 0.5 * SMERF_PI ? 1.0 : sin(th1);
    const double rho = cexp + 2.0 * sp.kmax * sinmax + 1.0;
    int nsub = (int)ceil(0.25 * rho * vmax);
    nsub = nsub < 1 ? 1 : (nsub > 256 ? 256 : nsub);
    const double h = vmax / nsub;
    double acc[M][M];
    for (int p = 0; p < M; ++p)
        for (int q = 0; q < M; ++q) acc[p][q] = 0.0;
    for (int j = 0; j < nsub; ++j)
        for (int n = 0; n < 8; ++n) {
            const double v = (j + 0.5 * (kGL8x[n] + 1.0)) * h;
            const double w = 0.5 * h * kGL8w[n] * exp(-cexp * v);
            const double u = u2 + v;
            const double x = 1.0 / (1.0 + exp(-2.0 * u));
            const MatC<M> Hi = cminv<M>(hmat_c<M>(sp, m, x, sinv, eref));
            double ph[M];
            for (int p = 0; p < M; ++p) {
                cdbl s = 0.0;
                for (int k = 0; k < M; ++k) s += W.a[p][k] * Hi.a[k][M - 1];
                ph[p] = s.real();  // phi is real (conjugate columns)
            }
            for (int p = 0; p < M; ++p)
                for (int q = 0; q < M; ++q) acc[p][q] += w * ph[p] * ph[q];
        }
    const double f = sp.A / (2.0 * SMERF_PI);
    const size_t o = (((size_t)pos) * sp.n_modes + m) * (M * M);
    for (int p = 0; p < M; ++p)
        for (int q = 0; q < M; ++q) {
            phi[o + p * M + q] = A.a[p][q].real();
            qout[o + p * M + q] = f * acc[p][q];
        }
}

// start_kernel in complex arithmetic
template <int M>
__global__ void start_kernel_c(SpecC sp, void* beq, bool tab64)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= sp.n_modes) return;
    const double th0 = ring_colat(sp.theta, sp.n_theta, sp.k0);
    const double t0 = tan(0.5 * th0);
    const double sx = sin(0.5 * th0), cx = cos(0.5 * th0);
    const double x0 = sx * sx, xb0 = cx * cx;
    Mat<M> J = mzero<M>();
    for (int i = 0; i < M; ++i) {
        const cdbl k2 = sp.k2[i];
        cdbl lq = 0.0;  // log Q_m / (m!)^2
        for (int j = 0; j < m; ++j) lq += cuda::std::log((j * (j + 1.0) + k2) / ((j + 1.0) * (j + 1.0)));
        cdbl lF0[M], lF1[M], r[M];
        cdbl rr = 1.0;
        for (int q = 0; q < M; ++q) {
            if (q > 0) {
                const double j = (double)(m + q - 1);
                rr *= (j * (j + 1.0) + k2) / (j + 1.0);
            }
            r[q] = rr;
            lF0[q] = log_hyp_c(k2, m + q, x0);
            lF1[q] = log_hyp_c(k2, m + q, xb0);
        }
        const cdbl lb = cuda::std::log(sp.b[i]) + sp.lG0[i] - log(4.0 * SMERF_PI) + lq;
        for (int p = 0; p < M; ++p)
            for (int q = 0; q < M; ++q) {
                const cdbl v = cuda::std::exp(lb + lF1[p] + lF0[q]) * r[p] * r[q] * pow(t0, (double)(q - p));
                J.a[p][q] += ((p & 1) ? -v : v).real();
            }
    }
    const Mat<M> L = mchol<M>(msym<M>(J));
    const double sc = m > 0 ? 0.70710678118654752440 : 1.0;
    int e = 0;
    for (int p = 0; p < M; ++p)
        for (int q = 0; q <= p; ++q, ++e)
            put<double>(beq, tab64, (size_t)e * sp.n_modes_pad + m, L.a[p][q] * sc);
}

// host: the complex spectrum's constants
static SpecC make_spec_c(const smerf_plan* pl)
{
    SpecC sc = SpecC();  // value-initialised: every member zero
    const int M = pl->p;
    sc.A = pl->A;
    sc.kmax = 0.0;
    for (int i = 0; i < M; ++i) {
        const cdbl kh(pl->khat_re[i], pl->khat_im[i]);
        sc.k2[i] = kh;
        sc.kmax = fmax(sc.kmax, sqrt(cuda::std::abs(kh)));
        cdbl b = pl->A;
        for (int j = 0; j < M; ++j)
            if (j != i) b /= cdbl(pl->khat_re[j], pl->khat_im[j]) - kh;
        sc.b[i] = b;
        // l = -1/2 + sqrt(1/4 - kappa-hat); Gamma(1+l) Gamma(-l) = -pi / sin(pi l)
        const cdbl lam = -0.5 + cuda::std::sqrt(0.25 - kh);
        const cdbl I(0.0, 1.0), z = SMERF_PI * lam;
        const cdbl ls = z.imag() > 0.0 ? -I * z + cuda::std::log(I * 0.5) + cuda::std::log(1.0 - cuda::std::exp(2.0 * I * z))
                                       : I * z + cuda::std::log(-I * 0.5) + cuda::std::log(1.0 - cuda::std::exp(-2.0 * I * z));
        sc.lG0[i] = cuda::std::log(cdbl(-SMERF_PI, 0.0)) - ls;
    }
    sc.n_theta = pl->n_theta;
    sc.k0 = pl->k0;
    sc.n_modes = pl->n_modes;
    sc.n_modes_pad = pl->n_modes_pad;
    sc.theta = pl->theta_dev;
    return sc;
}

#define CK(x)                                                                     \
    do {                                                                          \
        cudaError_t e_ = (x);                                                     \
        if (e_ != cudaSuccess) {                                                  \
            fprintf(stderr, "smerf setup: %s at %s:%d\n", cudaGetErrorString(e_), \
                    __FILE__, __LINE__);                                          \
            rc = (e_ == cudaErrorMemoryAllocation) ? SMERF_ENOMEM : SMERF_ECUDA;  \
            goto done;                                                            \
        }                                                                         \
    } while (0)

// p = 1 FP32 step rows [position][mode][A, C, B, pad] -> [position][A, C, B][mode]
__global__ void repack_rows_kernel(const float* __restrict__ rows, float* __restrict__ packed, int mp)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    const size_t pos = blockIdx.y;
    if (m >= mp) return;
    const float4 r = reinterpret_cast<const float4*>(rows)[pos * mp + m];
    packed[(pos * 3 + 0) * mp + m] = r.x;
    packed[(pos * 3 + 1) * mp + m] = r.y;
    packed[(pos * 3 + 2) * mp + m] = r.z;
}

// A set-up's temporaries: from the library's scratch pool (which keeps its memory between calls, so
// that a program that makes plan after plan maps none), or, when large or beyond the share of the
// pool that set-ups have, from the default pool, which returns them at the set-up's end
cudaError_t setup_alloc(void** p, size_t bytes, bool pooled, int dev, cudaStream_t st)
{
    return pooled ? smerf_scratch_alloc(p, bytes, dev, st) : smerf::dev_malloc_async(p, bytes, st);
}

template <int M>
int setup_impl(smerf_plan* pl, cudaStream_t st, bool sync, size_t* held)
{
    int rc = SMERF_OK;
    Spec sp;
    memset(&sp, 0, sizeof(sp));
    sp.M = M;
    sp.A = pl->A;
    sp.kmax = 0.0;
    for (int i = 0; i < M && !pl->complex_spec; ++i) {
        const double k = pl->kappa[i];
        sp.k2[i] = k * k;
        sp.kmax = fmax(sp.kmax, k);
        double b = pl->A;
        for (int j = 0; j < M; ++j)
            if (j != i) b /= pl->kappa[j] * pl->kappa[j] - k * k;
        sp.b[i] = b;
    }
    sp.n_theta = pl->n_theta;
    sp.k0 = pl->k0;
    sp.n_modes = pl->n_modes;
    sp.n_modes_pad = pl->n_modes_pad;
    sp.theta = pl->theta_dev;

    const bool t64 = pl->tab64;
    const size_t es = t64 ? 8 : 4;
    const size_t mp = pl->n_modes_pad;
    double* phi = nullptr;
    double* qv = nullptr;
    const int threads = 128;
    const int gm = (pl->n_modes + threads - 1) / threads;
    auto t_start = std::chrono::steady_clock::now();

    pl->table_bytes = 0;
    pl->step_table_bytes = 0;
    {
        // the start factor, the coarse tables and the FFT tables share one allocation (an allocation
        // and its release cost 40 us each, as much as many a set-up's kernels)
        int lg = 0;
        while ((2 << lg) < pl->n_phi) ++lg;
        const size_t cs = 2 * (pl->recur64 ? 8 : 4);
        size_t end = 0;
        auto part = [&end](size_t bytes) { const size_t o = end; end += (bytes + 255) / 256 * 256 + 256; return o; };
        const size_t beq_b = (size_t)tri(M) * mp * es;
        size_t coarse_b[2];
        for (int c = 0; c < 2; ++c) coarse_b[c] = (size_t)(pl->chain[c].n_anchors + 1) * coarse_elems(M) * mp * es;
        const size_t o_beq = part(beq_b), o_c0 = part(coarse_b[0]), o_c1 = part(coarse_b[1]), tables_end = end;
        const size_t o_pre = part(cs << lg), o_tw = part(cs * r4_table(lg)),
                     o_tw2 = part(cs * smerf::hr_off(lg, smerf::hr_passes(lg, 4), 4)),
                     o_tw3 = part(cs * smerf::hr_off(lg, smerf::hr_passes(lg, SMERF_INPLACE_MB), SMERF_INPLACE_MB)),
                     o_prex = part(pl->recur64 ? sizeof(int4) << lg : 0), o_twx = part(pl->recur64 ? sizeof(int4) * r4_table(lg) : 0);
        CK(smerf::dev_malloc((void**)&pl->shared, end));
        CK(cudaMemsetAsync(pl->shared, 0, tables_end, st));
        unsigned char* at = (unsigned char*)pl->shared;
        pl->beq = at + o_beq;
        pl->coarse[0] = at + o_c0;
        pl->coarse[1] = at + o_c1;
        pl->pre = at + o_pre;
        pl->tw = at + o_tw;
        pl->tw2 = at + o_tw2;
        pl->tw3 = at + o_tw3;
        pl->prex = at + o_prex;
        pl->twx = at + o_twx;
        pl->table_bytes += beq_b + coarse_b[0] + coarse_b[1];
        const int blocks = ((4 << lg) + 255) / 256 < 152 ? ((4 << lg) + 255) / 256 : 152;
        if (pl->recur64) fft_tables_kernel<double><<<blocks, 256, 0, st>>>(lg, (double2*)pl->pre, (double2*)pl->tw, (double2*)pl->tw2, (double2*)pl->tw3,
                                                                           (int4*)pl->prex, (int4*)pl->twx);
        else fft_tables_kernel<float><<<blocks, 256, 0, st>>>(lg, (float2*)pl->pre, (float2*)pl->tw, (float2*)pl->tw2, (float2*)pl->tw3, nullptr, nullptr);
        CK(cudaGetLastError());
    }
    for (int c = 0; c < 2; ++c) {
        const size_t sb = (size_t)(pl->chain[c].len + 1) * step_row(M) * mp * es;
        CK(smerf::dev_malloc((void**)&pl->steps[c], sb));
        CK(cudaMemsetAsync(pl->steps[c], 0, sb, st));
        pl->table_bytes += sb;
        pl->step_table_bytes += sb;
    }
    if (pl->complex_spec) start_kernel_c<M><<<gm, threads, 0, st>>>(make_spec_c(pl), pl->beq, t64);
    else {
        start_kernel<M><<<((unsigned)pl->n_modes * start_lanes(M) + 63) / 64, 64, 0, st>>>(sp, pl->beq, t64);
    }
    CK(cudaGetLastError());
    {
        // Step transitions and covariances of the northern chain.  On a grid symmetric about the
        // equator the southern chain's steps are their mirror images (z -> -z): in the northern
        // frame its step pos is the northern step pos + shift, shift = 1 for even n_theta (start
        // ring south of the equator) and 0 for odd n_theta, so one computation serves both
        // chains.  On any other grid a second pass computes them as the northern chain of the
        // mirrored grid theta'_j = pi - theta_{n_theta-1-j} (stored after the grid's own
        // colatitudes) from its start ring n_theta - 1 - k0, whose ring k0' - pos is the southern
        // chain's ring k0 + pos.
        const int len0 = pl->chain[0].len, len1 = pl->chain[1].len;
        const bool sym = smerf_grid_symmetric(pl->theta_host, pl->n_theta);
        const int shift = (pl->n_theta % 2 == 0) ? 1 : 0;
        if (sym && len1 + shift > len0) { rc = SMERF_EUNSUPPORTED; goto done; }
        for (int pass = 0; pass < (sym ? 1 : 2); ++pass) {
            const int len = pass == 0 ? len0 : len1;
            Spec s = sp;
            SpecC sc = pl->complex_spec ? make_spec_c(pl) : SpecC();
            // colatitude of the pass's start ring in its own frame
            double th = ring_colat(pl->theta_host, pl->n_theta, pl->k0);
            if (pass == 1) {
                s.theta = sc.theta = pl->theta_dev + pl->n_theta;
                s.k0 = sc.k0 = pl->n_theta - 1 - pl->k0;
                th = SMERF_PI - th;
            }
            if (len > 0) {
                const size_t nb = (size_t)(len + 1) * pl->n_modes * M * M * sizeof(double);
                const bool pooled = nb <= ((size_t)128 << 20) && smerf_setup_reserve(2 * nb, held);
                CK(setup_alloc((void**)&phi, nb, pooled, pl->dev, st));
                CK(setup_alloc((void**)&qv, nb, pooled, pl->dev, st));
                if (len > 65535) { rc = SMERF_EUNSUPPORTED; goto done; }
                dim3 grid(gm, len);
                if (pl->complex_spec) step_kernel_c<M><<<grid, threads, 0, st>>>(sc, len, phi, qv);
                else if (M == 3) step_kernel<M><<<grid, threads, 0, st>>>(s, 0, len, phi, qv);  // per-mode series
                else {
                    // the recurrence in m, but for a first step whose equatorward ring (x > 1/2)
                    // would amplify rounding errors by more than 1e3 over the orders: that one by
                    // the per-mode series (the start ring is the ring nearest the equator, so no
                    // later step starts south of it)
                    const double x1 = sin(0.5 * th) * sin(0.5 * th);
                    const bool first_series = x1 > 0.5 && (double)(pl->n_modes - 1) * log(x1 / (1.0 - x1)) > log(1e3);
                    const int first = first_series ? 2 : 1;
                    if (first_series) step_kernel<M><<<dim3(gm, 1), threads, 0, st>>>(s, 0, 1, phi, qv);
                    if (len >= first) {
                        const int n = len - first + 1;
                        if constexpr (M < 3)
                            step_kernel_rec<M><<<dim3((n + 2 * kRecWarps - 1) / (2 * kRecWarps), rec_blocks(pl->n_modes)),
                                                 32 * kRecWarps, 0, st>>>(s, first, len, phi, qv);
                    }
                }
                CK(cudaGetLastError());
            }
            // the chains whose tables this pass's steps give: both (symmetric grid), or one
            for (int c = sym ? 0 : pass; c < (sym ? 2 : pass + 1); ++c) {
                const int lc = pl->chain[c].len;
                if (lc == 0) continue;
                const size_t off = (sym && c == 1) ? (size_t)shift * pl->n_modes * M * M : 0;
                const int H = pl->H;
                const int nseg = H > 0 ? (lc / H + 1) : 1;
                dim3 grid(gm, nseg);
                segment_tables_kernel<M><<<grid, threads, 0, st>>>(sp, c, lc, H, phi + off, qv + off, pl->steps[c],
                                                             pl->coarse[c], t64);
                CK(cudaGetLastError());
            }
            if (phi) CK(cudaFreeAsync(phi, st));
            if (qv) CK(cudaFreeAsync(qv, st));
            phi = qv = nullptr;
        }
    }
    if (M == 1 && pl->packed) {
        // the ring kernel's packed p = 1 layout: [position][A, C, B][mode]
        for (int c = 0; c < 2; ++c) {
            const int len = pl->chain[c].len;
            const size_t rb = (size_t)(len + 1) * step_row(M) * mp * es;
            const size_t pb = (size_t)(len + 1) * 3 * mp * es;
            void* packed = nullptr;
            CK(smerf::dev_malloc(&packed, pb > 0 ? pb : 16));
            repack_rows_kernel<<<dim3((unsigned)((mp + 255) / 256), (unsigned)(len + 1)), 256, 0, st>>>(
                (const float*)pl->steps[c], (float*)packed, (int)mp);
            CK(cudaGetLastError());
            CK(cudaStreamSynchronize(st));
            cudaFree(pl->steps[c]);
            pl->steps[c] = packed;
            pl->table_bytes = pl->table_bytes - rb + pb;
            pl->step_table_bytes = pl->step_table_bytes - rb + pb;
        }
    }
    if (sync) {
        CK(cudaStreamSynchronize(st));
        pl->setup_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t_start).count();
    }
done:
    if (phi || qv) {
        cudaStreamSynchronize(st);
        if (phi) cudaFree(phi);
        if (qv) cudaFree(qv);
    }
    return rc;
}

}  // namespace

bool smerf_grid_symmetric(const double* theta, int n_theta)
{
    if (!theta) return true;
    for (int k = 0; k < n_theta; ++k)
        if (fabs(theta[k] + theta[n_theta - 1 - k] - SMERF_PI) > 1e-12 * SMERF_PI) return false;
    return true;
}

int smerf_start_ring(const double* theta, int n_theta)
{
    if (smerf_grid_symmetric(theta, n_theta)) return n_theta / 2;
    int k0 = 0;
    for (int k = 1; k < n_theta; ++k)
        if (fabs(theta[k] - 0.5 * SMERF_PI) <= fabs(theta[k0] - 0.5 * SMERF_PI)) k0 = k;
    return k0;
}

int smerf_setup_tables(smerf_plan* pl, cudaStream_t st, bool sync, size_t* held)
{
    switch (pl->p) {
        case 1: return setup_impl<1>(pl, st, sync, held);
        case 2: return setup_impl<2>(pl, st, sync, held);
        case 3: return setup_impl<3>(pl, st, sync, held);
        default: return SMERF_EUNSUPPORTED;
    }
}
