// Small dense kernels of libvne: the tridiagonal eigensolve + Gauss
// quadrature (Section 4, eq. rational-krylov-approximation-quadform), the
// Lanczos matvec coefficients f(T) e1, and the Hutch++ sketch linear algebra
// (Gram matrices, block products, pivoted Cholesky-QR factor).
//
// Tridiagonal eigenproblems use the implicit symmetric QR iteration with a
// Wilkinson shift (Golub & Van Loan, Matrix Computations, Sec. 8.3), in
// FP64.  Only the first row of the eigenvector matrix is needed for the
// quadrature (the Golub-Welsch weights u_{1j}^2), so the per-column kernel
// tracks that row alone; the matvec kernel keeps the full eigenvector matrix
// in shared memory, one warp per column, lanes owning its rows.
#include <cooperative_groups.h>
#include <float.h>
#include <math.h>
#include <stdlib.h>

#include "kernels.h"

namespace vne {

__host__ __device__ __forceinline__ double f_entropy(double x) { return x > 0.0 ? -x * log(x) : 0.0; }

#ifndef __CUDA_ARCH__
static inline double rsqrt(double v) { return 1.0 / sqrt(v); }
#endif

// One implicit QR sweep framework.  d[0..n), e[0..n-1) are overwritten by the
// eigenvalues / zeros; `rot(k, c, s)` is called for every Givens rotation
// acting on columns k, k+1 of the eigenvector matrix.  Returns false if the
// iteration cap was hit.
template <typename Rot>
__host__ __device__ bool symtri_qr(double* d, double* e, int n, Rot rot) {
    const double eps = DBL_EPSILON;
    int hi = n - 1;
    int iters = 0;
    const int max_iters = 40 * n + 40;
    while (hi > 0) {
        if (fabs(e[hi - 1]) <= eps * (fabs(d[hi - 1]) + fabs(d[hi]))) {
            e[hi - 1] = 0.0;
            hi--;
            continue;
        }
        int lo = hi - 1;
        while (lo > 0 && fabs(e[lo - 1]) > eps * (fabs(d[lo - 1]) + fabs(d[lo]))) lo--;
        if (lo > 0) e[lo - 1] = 0.0;
        if (++iters > max_iters) return false;
        // Wilkinson shift: eigenvalue of the trailing 2x2 closer to d[hi]
        double delta = 0.5 * (d[hi - 1] - d[hi]);
        double b2 = e[hi - 1] * e[hi - 1];
        double den = delta + copysign(sqrt(delta * delta + b2), delta == 0.0 ? 1.0 : delta);
        double mu = d[hi] - b2 / den;
        double x = d[lo] - mu, y = e[lo];
        for (int k = lo; k < hi; k++) {
            // Givens rotation from one reciprocal square root (cheaper than
            // hypot and two divisions on an FP64-poor GPU)
            double r2 = x * x + y * y;
            double c, s, r;
            if (r2 == 0.0) {
                c = 1.0;
                s = 0.0;
                r = 0.0;
            } else {
                double inv = rsqrt(r2);
                c = x * inv;
                s = -y * inv;
                r = r2 * inv;
            }
            if (k > lo) e[k - 1] = r;
            double a = d[k], b = e[k], cc = d[k + 1];
            double cs = c * s, c2 = c * c, s2 = s * s;
            d[k] = a * c2 - 2.0 * b * cs + cc * s2;
            d[k + 1] = a * s2 + 2.0 * b * cs + cc * c2;
            e[k] = (a - cc) * cs + b * (c2 - s2);
            rot(k, c, s);
            if (k < hi - 1) {
                x = e[k];
                y = -s * e[k + 1];
                e[k + 1] = c * e[k + 1];
            }
        }
    }
    return true;
}

// Implicit QR with `nr` rows of the eigenvector matrix tracked alongside (the
// quadrature needs the first row only; f(T) e1 needs all rows, spread over
// the lanes of a warp).  The sweep's running values (d_k, e_k and each
// tracked row's entry k) are carried in registers, so the dependent chain of
// one rotation touches no memory; old values of the next position are loaded
// ahead of their use.
template <int R>
__host__ __device__ inline bool symtri_qr_rows(double* d, double* e, int n, double* const* zr, int nr) {
    const double eps = DBL_EPSILON;
    int hi = n - 1;
    int iters = 0;
    const int max_iters = 40 * n + 40;
    while (hi > 0) {
        if (fabs(e[hi - 1]) <= eps * (fabs(d[hi - 1]) + fabs(d[hi]))) {
            e[hi - 1] = 0.0;
            hi--;
            continue;
        }
        int lo = hi - 1;
        while (lo > 0 && fabs(e[lo - 1]) > eps * (fabs(d[lo - 1]) + fabs(d[lo]))) lo--;
        if (lo > 0) e[lo - 1] = 0.0;
        if (++iters > max_iters) return false;
        const double delta = 0.5 * (d[hi - 1] - d[hi]);
        const double b2 = e[hi - 1] * e[hi - 1];
        const double den = delta + copysign(sqrt(delta * delta + b2), delta == 0.0 ? 1.0 : delta);
        const double mu = d[hi] - b2 / den;
        double dk = d[lo], ek = e[lo];
        double zk[R];
#pragma unroll
        for (int q = 0; q < R; q++) zk[q] = (q < nr) ? zr[q][lo] : 0.0;
        double x = dk - mu, y = ek;
        for (int k = lo; k < hi; k++) {
            const double dk1 = d[k + 1];
            const double ek1 = (k + 1 < hi) ? e[k + 1] : 0.0;
            double zk1[R];
#pragma unroll
            for (int q = 0; q < R; q++) zk1[q] = (q < nr) ? zr[q][k + 1] : 0.0;
            const double r2 = x * x + y * y;
            double c, s, r;
            if (r2 == 0.0) {
                c = 1.0;
                s = 0.0;
                r = 0.0;
            } else {
                const double inv = rsqrt(r2);
                c = x * inv;
                s = -y * inv;
                r = r2 * inv;
            }
            if (k > lo) e[k - 1] = r;
            const double cs = c * s, c2 = c * c, s2 = s * s;
            const double a = dk, b = ek;
            d[k] = a * c2 - 2.0 * b * cs + dk1 * s2;
            const double ndk1 = a * s2 + 2.0 * b * cs + dk1 * c2;
            const double nek = (a - dk1) * cs + b * (c2 - s2);
#pragma unroll
            for (int q = 0; q < R; q++) {
                if (q < nr) zr[q][k] = c * zk[q] - s * zk1[q];
                zk[q] = s * zk[q] + c * zk1[q];
            }
            dk = ndk1;
            if (k < hi - 1) {
                x = nek;
                y = -s * ek1;
                ek = c * ek1;
            } else {
                e[k] = nek;
            }
        }
        d[hi] = dk;
#pragma unroll
        for (int q = 0; q < R; q++)
            if (q < nr) zr[q][hi] = zk[q];
    }
    return true;
}

__host__ __device__ inline bool symtri_qr_first_row(double* d, double* e, double* z, int n) {
    double* rows[1] = {z};
    return symtri_qr_rows<1>(d, e, n, rows, 1);
}

// ---------------------------------------------------------------------------
// Gauss quadrature psi = ||c||^2 sum_j u_{1j}^2 f(sigma theta_j) of the
// leading unreduced block of T (Golub & Meurant, Matrices, Moments and
// Quadrature, Ch. 6), one CTA per tridiagonal with the eigenvalues spread
// over the threads.  GB300 retires FP64 instructions slowly, so one long
// sequential QR chain per column is the slowest possible schedule; here every
// lane runs short independent chains:
//  * theta_j by bisection on the Sturm count #{theta < z} (number of k with
//    sign p_k(z) = sign p_{k-1}(z), p_k = det(z I - T_k) by the three-term
//    recurrence, rescaled by powers of two every eight steps; Wilkinson, The
//    Algebraic Eigenvalue Problem, Ch. 5): FP32 counts first narrow the
//    Gershgorin interval, FP64 counts check the bracket, a bracket that holds
//    one eigenvalue goes to Newton's iteration on p_n, others are searched on
//    with FP64 counts (four trial points per pass and eigenvalue);
//  * u_{1j}^2 from the eigenvector of the twisted factorisation
//    T - theta I = N_r Delta_r N_r^T at the twist index r of smallest
//    |gamma_r| (Parlett & Dhillon, Lin. Alg. Appl. 309, 2000): z_r = 1,
//    components above r from the top-down pivots, below r from the bottom-up
//    pivots, u_{1j}^2 = z_1^2 / ||z||^2;
//  * eigenvalues closer than kClusterGap * span to a neighbour (or closer
//    than 16 x the half-width of the group being formed) form a cluster,
//    whose individual weights are ill-conditioned; its summed weight W and
//    first and second moments come from the resolvent e1^T (z I - T)^{-1} e1
//    (continued fraction) integrated by the trapezoid rule on a circle
//    around it, and it contributes W f(tbar) + f''(tbar) W var / 2 (weighted
//    mean tbar, variance var).  A cluster closer than 16 x its half-width to
//    the previous group sends the column to the sequential implicit QR
//    (lane 0), which keeps the kernel correct for any input.
constexpr double kClusterGap = 1e-5;
constexpr int kContourPoints = 32;

// Power of two that brings |x| (the largest of the values passed) to [1, 2):
// multiplying the recurrence state by it keeps signs and ratios.
__device__ __forceinline__ double pow2_rescale(long long maxbits) {
    int se = 2046 - (int)(maxbits >> 52);
    se = se < 1 ? 1 : (se > 2046 ? 2046 : se);
    return __longlong_as_double((long long)se << 52);
}

__device__ __forceinline__ long long absbits(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffLL; }

// #{eigenvalues of the leading n x n block < z[q]} for NC points at once
// (independent recurrences, interleaved for instruction-level parallelism):
// the number of k with sign p_k = sign p_{k-1}, p_0 = 1.  b2[k] =
// beta_{k-1}^2, b2[0] = 0.  A p_k that is exactly +0 counts as positive (a
// perturbation of z by one ulp).
template <int NC>
__device__ __forceinline__ void sturm_counts(const double* a, const double* b2, int n, const double (&z)[NC],
                                             int (&cnt)[NC]) {
    double p2[NC], p1[NC];  // p_{k-2}, p_{k-1}
    int hprev[NC], changes[NC];
#pragma unroll
    for (int q = 0; q < NC; q++) {
        p2[q] = 0.0;
        p1[q] = 1.0;
        hprev[q] = 0;
        changes[q] = 0;
    }
    for (int k = 0; k < n; k++) {
        const double ak = a[k], bk = b2[k];
#pragma unroll
        for (int q = 0; q < NC; q++) {
            const double p = fma(z[q] - ak, p1[q], -(bk * p2[q]));
            const int h = __double2hiint(p);
            changes[q] += (int)((unsigned)(h ^ hprev[q]) >> 31);
            hprev[q] = h;
            p2[q] = p1[q];
            p1[q] = p;
        }
        if ((k & 7) == 7) {
#pragma unroll
            for (int q = 0; q < NC; q++) {
                const long long m1 = absbits(p1[q]), m2 = absbits(p2[q]);
                const double fsc = pow2_rescale(m1 > m2 ? m1 : m2);
                p1[q] *= fsc;
                p2[q] *= fsc;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < NC; q++) cnt[q] = n - changes[q];
}

// p_n(z) / p_n'(z) for the characteristic polynomial p_n(z) = det(z I - T)
// and the Sturm count at z, from one recurrence (p_k' = p_{k-1} +
// (z - a_k) p_{k-1}' - b2_k p_{k-2}'), for NC points.
template <int NC>
__device__ __forceinline__ void newton_counts(const double* a, const double* b2, int n, const double (&z)[NC],
                                              double (&ratio)[NC], int (&cnt)[NC]) {
    double p2[NC], p1[NC], d2[NC], d1[NC];
    int hprev[NC], changes[NC];
#pragma unroll
    for (int q = 0; q < NC; q++) {
        p2[q] = 0.0;
        p1[q] = 1.0;
        d2[q] = 0.0;
        d1[q] = 0.0;
        hprev[q] = 0;
        changes[q] = 0;
    }
    for (int k = 0; k < n; k++) {
        const double ak = a[k], bk = b2[k];
#pragma unroll
        for (int q = 0; q < NC; q++) {
            const double zk = z[q] - ak;
            const double p = fma(zk, p1[q], -(bk * p2[q]));
            const double d = fma(zk, d1[q], p1[q]) - bk * d2[q];
            const int h = __double2hiint(p);
            changes[q] += (int)((unsigned)(h ^ hprev[q]) >> 31);
            hprev[q] = h;
            p2[q] = p1[q];
            p1[q] = p;
            d2[q] = d1[q];
            d1[q] = d;
        }
        if ((k & 7) == 7) {
#pragma unroll
            for (int q = 0; q < NC; q++) {
                long long m = absbits(p1[q]);
                m = max(m, absbits(p2[q]));
                m = max(m, absbits(d1[q]));
                m = max(m, absbits(d2[q]));
                const double fsc = pow2_rescale(m);
                p1[q] *= fsc;
                p2[q] *= fsc;
                d1[q] *= fsc;
                d2[q] *= fsc;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < NC; q++) {
        ratio[q] = p1[q] / d1[q];
        cnt[q] = n - changes[q];
    }
}

// FP32 Sturm count on the FP32-rounded block (pivots d_k of T - zI,
// #{d_k < 0}), used only to narrow the FP64 search interval; the interval is
// checked with FP64 counts before it is trusted.
__device__ __forceinline__ int sturm_count_f32(const float* a, const float* b2, int n, float z, float pivmin) {
    int cnt = 0;
    float d = 1.f;
    for (int k = 0; k < n; k++) {
        d = (a[k] - z) - __fdividef(b2[k], d);
        if (fabsf(d) < pivmin) d = -pivmin;
        cnt += d < 0.f;
    }
    return cnt;
}

__device__ __forceinline__ double guard_pivot(double x, double pivmin) {
    // compared by their bits: an FP64 comparison would take a slot of the FP64 port
    return absbits(x) < absbits(pivmin) ? copysign(pivmin, x == 0.0 ? 1.0 : x) : x;
}

// Point q of the K-point trapezoid rule on the circle z = c + rho e^{i phi}:
// Re F(z) dz^p, p = 1, 2, 3, with dz = z - c and F(z) = e1^T (z I - T)^{-1} e1
// by the bottom-up continued fraction.  (1/K) times their sums over q are the
// summed weight and the first and second moments about c of the eigenvalues
// inside the circle.
__device__ void resolvent_point(const double* a, const double* b, int n, double c, double rho, int q, double& re1,
                                double& re2, double& re3) {
    double sph, cph;
    sincospi((2.0 * q + 1.0) / kContourPoints, &sph, &cph);
    const double dzr = rho * cph, dzi = rho * sph;
    const double zr = c + dzr, zi = dzi;
    double gr = zr - a[n - 1], gi = zi;
    for (int k = n - 2; k >= 0; k--) {
        // g <- (z - a_k) - b_k^2 / g
        const double t = b[k] * b[k] / (gr * gr + gi * gi);
        gr = (zr - a[k]) - t * gr;
        gi = zi + t * gi;
    }
    const double den = gr * gr + gi * gi;
    const double fr = gr / den, fi = -gi / den;                        // F = 1 / g
    const double pr = fr * dzr - fi * dzi, pim = fr * dzi + fi * dzr;  // F dz
    re1 = pr;
    const double p2r = pr * dzr - pim * dzi, p2i = pr * dzi + pim * dzr;  // F dz^2
    re2 = p2r;
    re3 = p2r * dzr - p2i * dzi;  // Re(F dz^3)
}

// Fallback: the quadrature by the sequential implicit QR of the whole
// (scaled) block, run by lane 0 of the warp.
template <int MAXM>
__device__ void quad_by_qr(const double* sa, const double* sb, int n, double sc, double norm2, int lane,
                           double* out) {
    if (lane != 0) return;
    double d[MAXM], ee[MAXM], z[MAXM];
    for (int k = 0; k < n; k++) {
        d[k] = sa[k];
        ee[k] = sb[k];
        z[k] = 0.0;
    }
    z[0] = 1.0;
    const bool ok = symtri_qr_first_row(d, ee, z, n);
    double s = 0.0;
    for (int k = 0; k < n; k++) s += z[k] * z[k] * f_entropy(sc * d[k]);
    *out = ok ? norm2 * s : nan("");
}

// Shapes of the spectral kernels.  FP64 bounds them: GB300 issues one FP64
// instruction per warp and sub-partition in 64 cycles whatever its
// independence (measured: 0.5 lane operations per cycle for one warp, 1.7 per
// SM; a division takes 9, a reciprocal 6, a logarithm 32 such slots), while
// FP32, integer and conversion instructions run at full rate.  One warp per
// tridiagonal therefore leaves three of an SM's four FP64 issue ports idle
// and pays for every lane loop in full, so a CTA of 4 MAXM threads takes one
// tridiagonal: four lanes per eigenvalue in the searches (one trial point
// each), one lane in Newton's iteration, two lanes in the twisted
// factorisation (top-down and bottom-up pivots at the same time).
// Measured (a CTA per tridiagonal against one warp): 104 quadratures of order
// 50 in 0.10 ms (0.59); 3072 of order 40 in 1.30 ms (2.38); one Krylov check
// of a server (quadrature and 512 grid points of Theorem 4.4, some hundred
// columns of order 3 to 9) in 0.071 ms (0.320 in two kernels).
template <int MAXM>
struct TqCfg {
    static constexpr int NT = 4 * MAXM;                 // threads per CTA
    static constexpr int NW = NT / 32;
    static constexpr int RB = MAXM < 64 ? MAXM : 64;    // eigenvectors per pass of the pivot scratch
    static constexpr int LD = RB + 1;                   // row stride of the scratch (conflict-free both ways)
    static constexpr int kSmem = 2 * MAXM * LD * (int)sizeof(double);
};

// Shared state of the spectral kernels for one tridiagonal (one CTA).
template <int MAXM>
struct TqShared {
    double a[MAXM], b[MAXM], b2[MAXM + 1];  // scaled block, b2[k] = beta_{k-1}^2, b2[n] = 0
    double th[MAXM], bw[MAXM];              // eigenvalues (ascending), bracket widths
    double z1[MAXM], zn[MAXM], nrm[MAXM];   // first / last entry and squared norm of the twisted eigenvectors
    double c0[MAXM], c1[MAXM];              // per-eigenvalue terms of the final sums
    double k0[MAXM / 2], k1[MAXM / 2], k2[MAXM / 2];  // per-cluster terms
    float a32[MAXM], b2_32[MAXM + 1];
    double cc[MAXM / 2], rho[MAXM / 2], half[MAXM / 2];  // clusters: centre, circle radius, half-width
    int gfirst[MAXM + 1], glast[MAXM], cl_of_group[MAXM];
    int clo[MAXM], chi[MAXM];  // Sturm counts at the ends of the brackets (searches)
    int ngroups, ncl, fallback, n, finite;
    double span, s2, pivmin, glo, ghi;
    float pivmin32;
    unsigned long long gmin, gmax;
};

// Choose the sub-interval of [lo, hi] that holds eigenvalue j from the counts
// of four ascending interior points, one per lane of the quad (all four lanes
// of the quad end with the same bracket).
__device__ __forceinline__ void quad_choose(int j, int lane, double z, int cnt, double& lo, double& hi, int& clo,
                                            int& chi) {
    const int base = lane & 28;
    const unsigned above = (__ballot_sync(0xffffffffu, cnt > j) >> base) & 15u;
    const int i = above ? __ffs(above) - 1 : 4;  // first point above eigenvalue j
    const double zu = __shfl_sync(0xffffffffu, z, base + (i < 4 ? i : 3));
    const int cu = __shfl_sync(0xffffffffu, cnt, base + (i < 4 ? i : 3));
    const double zl = __shfl_sync(0xffffffffu, z, base + (i > 0 ? i - 1 : 0));
    const int cl = __shfl_sync(0xffffffffu, cnt, base + (i > 0 ? i - 1 : 0));
    if (i < 4) hi = zu, chi = cu;
    if (i > 0) lo = zl, clo = cl;
}

// Eigenvalues and their grouping for the leading unreduced block of
// tridiagonal c (every thread of the CTA calls it).  Returns false if the
// block has a non-finite entry.
template <int MAXM>
__device__ bool tq_spectrum(const double* __restrict__ alpha, const double* __restrict__ beta, int c, int m, int ld,
                            TqShared<MAXM>& S) {
    constexpr int NT = TqCfg<MAXM>::NT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double* sa = S.a;
    double* sb = S.b;
    double* sb2 = S.b2;
    double* sth = S.th;
    double* sbw = S.bw;
    float* sa32 = S.a32;
    float* sb2_32 = S.b2_32;
    if (warp == 0) {
        // leading unreduced block: n = 1 + first j with beta_j == 0
        int n = m;
        for (int j0 = 0; j0 < m - 1; j0 += 32) {
            const int j = j0 + lane;
            const bool zero = j < m - 1 && beta[(size_t)j * ld + c] == 0.0;
            const unsigned zb = __ballot_sync(0xffffffffu, zero);
            if (zb) {
                n = j0 + __ffs(zb);
                break;
            }
        }
        bool finite = true;
        double glo = INFINITY, ghi = -INFINITY, bmax = 0.0;
        for (int j = lane; j < n; j += 32) {
            const double aj = alpha[(size_t)j * ld + c];
            const double bj = (j + 1 < n) ? beta[(size_t)j * ld + c] : 0.0;
            const double bp = (j > 0) ? beta[(size_t)(j - 1) * ld + c] : 0.0;
            sa[j] = aj;
            sb[j] = bj;
            const double bj2 = bj * bj;
            sb2[j + 1] = bj2;
            finite = finite && isfinite(aj) && isfinite(bj);
            const double r = fabs(bj) + fabs(bp);
            glo = fmin(glo, aj - r);
            ghi = fmax(ghi, aj + r);
            bmax = fmax(bmax, bj2);
        }
        if (lane == 0) {
            sb2[0] = 0.0;
            sb2_32[0] = 0.f;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, off));
            ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, off));
            bmax = fmax(bmax, __shfl_xor_sync(0xffffffffu, bmax, off));
        }
        finite = __all_sync(0xffffffffu, finite);
        __syncwarp();
        // scale the block by the power of two s2 that brings its Gershgorin
        // radius to [1, 2) (exact: eigenvalues scale by s2, weights do not), so
        // the unnormalised Sturm recurrences stay far from overflow
        const double s2 = pow2_rescale(absbits(fmax(fmax(fabs(glo), fabs(ghi)), DBL_MIN)));
        for (int j = lane; j < n; j += 32) {
            sa[j] *= s2;
            sb[j] *= s2;
            sb2[j + 1] *= s2 * s2;
            sa32[j] = (float)sa[j];
            sb2_32[j + 1] = (float)sb2[j + 1];
        }
        if (lane == 0) {
            glo *= s2;
            ghi *= s2;
            bmax *= s2 * s2;
            const double span = fmax(fmax(fabs(glo), fabs(ghi)), DBL_MIN);
            S.n = n;
            S.finite = finite;
            S.span = span;
            S.s2 = s2;
            S.glo = glo - (4.0 * DBL_EPSILON * span + DBL_MIN);
            S.ghi = ghi + (4.0 * DBL_EPSILON * span + DBL_MIN);
            S.pivmin = DBL_MIN * fmax(1.0, bmax);
            S.pivmin32 = FLT_MIN * fmaxf(1.f, (float)bmax);
        }
    }
    __syncthreads();
    if (!S.finite) return false;
    const int n = S.n;
    const double span = S.span, glo = S.glo, ghi = S.ghi;
    // 1. eigenvalues, ascending: theta_j is the j-th smallest; four lanes
    //    search for it, each with one trial point per pass.  Warps without an
    //    eigenvalue skip the arithmetic.
    const int j = tid >> 2, q = tid & 3;
    const bool busy = warp * 8 < n, live = j < n;
    double lo = glo, hi = ghi;
    int clo = 0, chi = n;
    bool widened = false;
    if (busy) {
        // (a) FP32 search (factor 5 per pass) down to ~1e-6 of the span
        const float pivmin32 = S.pivmin32;
        float l32 = (float)glo, h32 = (float)ghi;
        for (int it = 0; it < 9; it++) {
            const float w = h32 - l32;
            const float z = l32 + 0.2f * (float)(q + 1) * w;
            const bool gt = sturm_count_f32(sa32, sb2_32, n, z, pivmin32) > j;
            const unsigned above = (__ballot_sync(0xffffffffu, gt) >> (lane & 28)) & 15u;
            const int i = above ? __ffs(above) - 1 : 4;
            if (i < 4) h32 = l32 + 0.2f * (float)(i + 1) * w;
            if (i > 0) l32 = l32 + 0.2f * (float)i * w;
        }
        const double wd = 4e-6 * span + 8.0 * (double)FLT_EPSILON * fabs((double)h32);
        lo = fmax(glo, (double)l32 - wd);
        hi = fmin(ghi, (double)h32 + wd);
        // (b) FP64 counts at the ends and two interior points: the bracket is
        //     trusted only if count(lo) <= j < count(hi)
        double zc[1] = {q == 3 ? hi : fma((double)q * (1.0 / 3.0), hi - lo, lo)};
        int cn[1];
        sturm_counts<1>(sa, sb2, n, zc, cn);
        const int c_lo = __shfl_sync(0xffffffffu, cn[0], lane & 28);
        const int c_hi = __shfl_sync(0xffffffffu, cn[0], (lane & 28) + 3);
        clo = c_lo;
        chi = c_hi;
        quad_choose(j, lane, zc[0], cn[0], lo, hi, clo, chi);
        if (live && !(c_lo <= j && c_hi > j)) {
            lo = glo;
            hi = ghi;
            clo = 0;
            chi = n;
            widened = true;
        }
    }
    // (c) FP64 search (factor 5 per pass) while some bracket holds more than
    //     one eigenvalue: 4 passes from the FP32 bracket (below 1e-8 span),
    //     13 from the Gershgorin interval.  Isolated brackets go straight to
    //     Newton's iteration.
    const int any = __syncthreads_or((live && chi - clo != 1 ? 1 : 0) | (widened ? 2 : 0));
    const int wide = __syncthreads_or(widened ? 1 : 0);
    if (any && busy) {
        const int passes = wide ? 13 : 4;
        for (int it = 0; it < passes; it++) {
            double zq[1] = {fma(0.2 * (q + 1), hi - lo, lo)};
            int cq[1];
            sturm_counts<1>(sa, sb2, n, zq, cq);
            quad_choose(j, lane, zq[0], cq[0], lo, hi, clo, chi);
        }
    }
    if (live && q == 0) {
        S.c0[j] = lo;
        S.c1[j] = hi;
        S.clo[j] = clo;
        S.chi[j] = chi;
    }
    __syncthreads();
    // (d) safeguarded Newton on p_n, one lane per eigenvalue (each step also
    //     counts, so the bracket keeps shrinking): a root alone in its bracket
    //     converges quadratically and stops; roots sharing a bracket (tight
    //     clusters) halve it four times and are handled as a cluster below
    if (warp * 32 < n) {
        const int jr = min(tid, n - 1);
        double l = S.c0[jr], h = S.c1[jr];
        int cl = S.clo[jr], ch = S.chi[jr];
        double zn[1] = {0.5 * (l + h)};
        double w = 0.0;
        bool done = false;
        for (int it = 0; it < 48; it++) {
            double ratio[1];
            int cn[1];
            newton_counts<1>(sa, sb2, n, zn, ratio, cn);
            if (!done) {
                if (cn[0] > jr) {
                    h = zn[0];
                    ch = cn[0];
                } else {
                    l = zn[0];
                    cl = cn[0];
                }
                const double zt = zn[0] - ratio[0];
                const bool alone = (ch - cl) == 1, inside = zt >= l && zt <= h;
                w = h - l;
                if (alone && inside) {
                    zn[0] = zt;
                    // the step left an error of ratio^2 / gap, gap >= kClusterGap span
                    if (fabs(ratio[0]) <= 1e-11 * span) {
                        w = 8.0 * DBL_EPSILON * span;
                        done = true;
                    }
                } else {
                    zn[0] = 0.5 * (l + h);
                    if (!alone && it >= 3) done = true;
                    if (w <= 4.0 * DBL_EPSILON * span) done = true;
                }
            }
            if (__all_sync(0xffffffffu, done)) break;
        }
        if (tid < n) {
            sth[jr] = zn[0];
            sbw[jr] = w;
        }
    }
    __syncthreads();
    // 2. groups of eigenvalues: a group grows while the next gap is below
    //    kClusterGap * span or below 16 x its half-width, and absorbs the
    //    previous group while the gap to it is below 17 x its half-width;
    //    one-member groups are isolated eigenvalues, the others clusters.  A
    //    cluster closer than 16 x its half-width to a neighbouring group sends
    //    the column to the sequential QR.  When no gap is that small (the
    //    usual case, tested by all threads at once) every group has one member.
    const double tau = kClusterGap * span;
    double* s_cc = S.cc;
    double* s_rho = S.rho;
    double* s_half = S.half;
    int* s_gfirst = S.gfirst;
    int* s_glast = S.glast;
    int* s_cl_of_group = S.cl_of_group;
    bool close = false;
    if (tid + 1 < n) {
        const double gap = sth[tid + 1] - sth[tid];
        close = gap < tau || gap < 8.0 * sbw[tid];
    }
    if (!__syncthreads_or(close)) {
        for (int g = tid; g < n; g += NT) {
            s_gfirst[g] = g;
            s_glast[g] = g;
            s_cl_of_group[g] = -1;
        }
        if (tid == 0) {
            s_gfirst[n] = n;
            S.ngroups = n;
            S.ncl = 0;
            S.fallback = 0;
        }
    } else if (tid == 0) {
        auto halfw = [&](int f, int l) {
            double h = 0.5 * (sth[l] - sth[f]);
            for (int i = f; i <= l; i++) h = fmax(h, 0.5 * sbw[i]);
            return h;
        };
        int ng = 0;
        for (int i = 0; i < n;) {
            int f = i, e = i;
            for (;;) {
                while (e + 1 < n) {
                    const double gap = sth[e + 1] - sth[e];
                    if (!(gap < tau || gap < 16.0 * halfw(f, e))) break;
                    e++;
                }
                if (ng > 0 && e > f && sth[f] - sth[s_glast[ng - 1]] < 17.0 * halfw(f, e)) {
                    f = s_gfirst[--ng];  // absorb the previous group
                    continue;
                }
                break;
            }
            s_gfirst[ng] = f;
            s_glast[ng] = e;
            ng++;
            i = e + 1;
        }
        int ncl = 0, fb = 0;
        for (int g = 0; g < ng; g++) {
            const int f = s_gfirst[g], e = s_glast[g];
            s_cl_of_group[g] = -1;
            if (e == f) continue;
            const double half = fmax(halfw(f, e), 4.0 * DBL_EPSILON * span);
            const double dl = g > 0 ? sth[f] - sth[s_glast[g - 1]] : INFINITY;
            const double dr = g + 1 < ng ? sth[s_gfirst[g + 1]] - sth[e] : INFINITY;
            const double D = fmin(dl, dr) - half;
            if (!(D >= 16.0 * half)) fb = 1;
            // circle radius: D / 8 for a tight cluster, else the geometric mean
            // of half-width and distance (both error terms (half / D)^(K/2))
            s_cc[ncl] = 0.5 * (sth[f] + sth[e]);
            s_rho[ncl] = !isfinite(D) ? 0.25 * span : (D >= 64.0 * half ? D / 8.0 : sqrt(half * D));
            s_half[ncl] = half;
            s_cl_of_group[g] = ncl++;
        }
        s_gfirst[ng] = n;
        S.ngroups = ng;
        S.ncl = ncl;
        S.fallback = fb;
    }
    __syncthreads();
    return true;
}

// Twisted-factorisation eigenvectors of the eigenvalues [rb0, rb0 + nb), nb <=
// RB: squared norm, first and last component (the entry at the twist index is
// 1) to S.nrm, S.z1, S.zn.  Two lanes per eigenvalue: lane 0 of the pair runs
// the top-down pivots D_k and the components above the twist, lane 1 the
// bottom-up pivots R_k and those below; both keep reciprocals in P ([2][MAXM]
// [LD]), which the components need (one reciprocal per pivot, no division).
// With KEEP the components replace the first half of P.  Every thread of the
// CTA calls it.
template <int MAXM, bool KEEP>
__device__ void tq_vectors(TqShared<MAXM>& S, double* P, int rb0, int nb) {
    constexpr int LD = TqCfg<MAXM>::LD;
    const int tid = threadIdx.x;
    const int r = tid >> 1, side = tid & 1, n = S.n;
    if ((tid >> 5) * 16 < nb) {  // warp-uniform
        const bool live = r < nb;
        const int rr = live ? r : nb - 1;
        const double th = S.th[rb0 + rr], pivmin = S.pivmin;
        const double *sa = S.a, *sb = S.b, *sb2 = S.b2;
        double* P0 = P + rr;
        double* P1 = P + MAXM * LD + rr;
        double* mine = side ? P1 : P0;
        double inv = 0.0;
        for (int i = 0; i < n; i++) {
            const int k = side ? n - 1 - i : i;
            const double d = guard_pivot(fma(-sb2[side ? k + 1 : k], inv, sa[k] - th), pivmin);
            inv = 1.0 / d;
            if (live) mine[k * LD] = inv;
        }
        __syncwarp();
        // twist index: smallest |gamma_k| = |D_k + R_k - (a_k - theta)|
        long long best = 0x7ff0000000000000LL;
        int tw = n - 1;
        for (int k = n - 1 - side; k >= 0; k -= 2) {
            const double up = k > 0 ? P0[(k - 1) * LD] : 0.0, dn = k + 1 < n ? P1[(k + 1) * LD] : 0.0;
            const long long g = absbits(fma(-sb2[k + 1], dn, fma(-sb2[k], up, sa[k] - th)));
            if (g < best) {
                best = g;
                tw = k;
            }
        }
        const long long ob = __shfl_xor_sync(0xffffffffu, best, 1);
        const int ot = __shfl_xor_sync(0xffffffffu, tw, 1);
        if (ob < best || (ob == best && ot > tw)) tw = ot;
        __syncwarp();  // both lanes have read the reciprocals that KEEP overwrites
        // components away from the twist
        double z = 1.0, s = 0.0;
        const int steps = side ? n - 1 - tw : tw;
        for (int i = 1; i <= steps; i++) {
            const int k = side ? tw + i : tw - i;
            z = -(sb[side ? k - 1 : k] * z) * mine[k * LD];
            s = fma(z, z, s);
            if (KEEP && live) P0[k * LD] = z;
        }
        if (KEEP && live && side == 0) P0[tw * LD] = 1.0;
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        if (live) {
            if (side == 0) {
                S.nrm[rb0 + r] = 1.0 + s;
                S.z1[rb0 + r] = z;
            } else {
                S.zn[rb0 + r] = z;
            }
        }
    }
    __syncthreads();
}

// The Gauss quadrature from the spectrum and the twisted eigenvectors of all
// eigenvalues (S.nrm, S.z1): isolated eigenvalues by their weights, clusters
// by the contour, a warp per cluster and a lane per contour point.  Every
// thread of the CTA calls it; thread 0 writes *psi.
template <int MAXM>
__device__ void tq_quadrature(TqShared<MAXM>& S, double sc, double norm2, double* psi) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = S.n;
    for (int g = tid; g < S.ngroups; g += blockDim.x) {
        if (S.cl_of_group[g] >= 0) {
            S.c0[g] = S.c1[g] = 0.0;
            continue;
        }
        const int i = S.gfirst[g];
        const double w = S.z1[i] * S.z1[i] / S.nrm[i];
        S.c0[g] = w * f_entropy(sc * S.th[i]);
        S.c1[g] = w;
    }
    for (int cl = warp; cl < S.ncl; cl += TqCfg<MAXM>::NW) {
        double W, M1, M2;
        resolvent_point(S.a, S.b, n, S.cc[cl], S.rho[cl], lane, W, M1, M2);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            W += __shfl_xor_sync(0xffffffffu, W, off);
            M1 += __shfl_xor_sync(0xffffffffu, M1, off);
            M2 += __shfl_xor_sync(0xffffffffu, M2, off);
        }
        if (lane == 0) {
            W /= kContourPoints;
            M1 /= kContourPoints;
            M2 /= kContourPoints;
            // sum_j w_j f(theta_j) over the cluster ~ W f(tbar) + f''(tbar) W var / 2
            // with the weighted mean tbar and variance var; a cluster whose weight
            // is at rounding level (eigenvectors that vanish at row 1) keeps its
            // centre and no correction
            const double cc = S.cc[cl], half = S.half[cl];
            double contrib = W * f_entropy(sc * cc), errb = 0.0;
            if (W > 0.0 && fabs(M1) <= 2.0 * half * W) {
                const double mu = M1 / W, tbar = cc + mu;
                const double var = fmax(M2 / W - mu * mu, 0.0);
                contrib = W * f_entropy(sc * tbar);
                if (tbar > 0.0) contrib -= 0.5 * (sc / tbar) * W * var;  // d2/dt2 f(sc t) = -sc / t
            }
            if (half > 1e-3 * fabs(cc)) {
                // a cluster at the origin: the expansion does not hold, but its
                // members lie in [cc - half, cc + half] and f >= 0 increases from
                // 0, so the error is below W f(cc + half)
                errb = fmax(W, 0.0) * f_entropy(fmin(sc * fmax(cc + half, 0.0), 0.36787944117144233));
            }
            S.k0[cl] = contrib;
            S.k1[cl] = W;
            S.k2[cl] = errb;
        }
    }
    __syncthreads();
    if (warp == 0) {
        double acc = 0.0, wsum = 0.0, errb = 0.0;
        for (int g = lane; g < S.ngroups; g += 32) {
            acc += S.c0[g];
            wsum += S.c1[g];
        }
        for (int cl = lane; cl < S.ncl; cl += 32) {
            acc += S.k0[cl];
            wsum += S.k1[cl];
            errb += S.k2[cl];
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            acc += __shfl_xor_sync(0xffffffffu, acc, off);
            wsum += __shfl_xor_sync(0xffffffffu, wsum, off);
            if (S.ncl) errb += __shfl_xor_sync(0xffffffffu, errb, off);
        }
        if (!(errb <= 1e-10 * fabs(acc))) {
            quad_by_qr<MAXM>(S.a, S.b, n, sc, norm2, lane, psi);
        } else if (lane == 0) {
            // the weights sum to one; dividing by the computed sum removes their
            // common rounding
            *psi = norm2 * (acc / wsum);
        }
    }
}

template <int MAXM>
__global__ void __launch_bounds__(TqCfg<MAXM>::NT)
    k_tridiag_quad(const double* __restrict__ alpha, const double* __restrict__ beta,
                   const double* __restrict__ norm2, const double* __restrict__ scale, int count, int m_all, int ld,
                   double* __restrict__ psi, const int32_t* __restrict__ cols, const int32_t* __restrict__ mcol) {
    __shared__ TqShared<MAXM> S;
    extern __shared__ double piv[];  // pivot scratch of tq_vectors
    if ((int)blockIdx.x >= count) return;
    // entry blockIdx.x: column c (of the ld-strided arrays) after m steps
    const int c = cols ? cols[blockIdx.x] : (int)blockIdx.x;
    const int m = mcol ? mcol[blockIdx.x] : m_all;
    if (!tq_spectrum<MAXM>(alpha, beta, c, m, ld, S)) {
        if (threadIdx.x == 0) psi[c] = nan("");
        return;
    }
    const double sc = scale[c] / S.s2;  // f is applied to the unscaled eigenvalues
    if (S.fallback) {
        if (threadIdx.x < 32) quad_by_qr<MAXM>(S.a, S.b, S.n, sc, norm2[c], threadIdx.x, psi + c);
        return;
    }
    for (int rb = 0; rb < S.n; rb += TqCfg<MAXM>::RB)
        tq_vectors<MAXM, false>(S, piv, rb, min(TqCfg<MAXM>::RB, S.n - rb));
    tq_quadrature<MAXM>(S, sc, norm2[c], psi + c);
}

// f(T) e1 by the sequential implicit QR with the full eigenvector matrix Z
// (n x n, row-major, in shared memory): every lane runs the scalar
// recurrence on its own copies (uniform control flow) and rotates the rows of
// Z it owns (rows lane, lane + 32, ...).  Fallback of k_tridiag_fvec.
template <int MAXM>
__device__ void fvec_by_qr(const double* sa, const double* sb, int n, int m, double sc, int lane, double* Z,
                           double* __restrict__ zvec, int ld, int c) {
    constexpr int R = MAXM / 32;
    for (int idx = lane; idx < n * n; idx += 32) Z[idx] = ((idx / n) == (idx % n)) ? 1.0 : 0.0;
    double dl[MAXM], el[MAXM];
    for (int j = 0; j < n; j++) {
        dl[j] = sa[j];
        el[j] = sb[j];
    }
    double* rows[R];
    int nr = 0;
    for (int q = 0; q < R; q++) {
        const int row = lane + 32 * q;
        rows[q] = Z + (size_t)(row < n ? row : 0) * n;
        if (row < n) nr = q + 1;
    }
    __syncwarp();
    const bool ok = symtri_qr_rows<R>(dl, el, n, rows, nr);
    __syncwarp();
    for (int row = lane; row < m; row += 32) {
        double acc = 0.0;
        if (row < n)
            for (int k = 0; k < n; k++) acc += Z[row * n + k] * f_entropy(sc * dl[k]) * Z[k];
        zvec[(size_t)row * ld + c] = ok ? acc : nan("");
    }
}

// f(T) e1 = sum_j u_j u_{1j} f(sigma theta_j) for the matrix-function
// recovery of the Hutch++ sketch (eq. rational-krylov-approximation-matvec),
// with the spectrum of k_tridiag_quad: an isolated eigenvalue adds its
// twisted-factorisation eigenvector z scaled by z_1 f / ||z||^2; a cluster
// adds (1/2 pi i) \oint (f(c) + f'(c)(z - c) + f''(c)(z - c)^2 / 2)
// (z I - T)^{-1} e1 dz by the 32-point trapezoid rule (one point per lane of
// warp 0; the resolvent vector from the bottom-up continued fraction, then the
// forward ratios x_k = x_{k-1} beta_{k-1} / g_k).  Component k is summed by
// four lanes over the eigenvectors of a pass (or the contour points).
template <int MAXM>
__global__ void __launch_bounds__(TqCfg<MAXM>::NT)
    k_tridiag_fvec(const double* __restrict__ alpha, const double* __restrict__ beta,
                   const double* __restrict__ scale, int count, int m, int ld, double* __restrict__ zvec) {
    constexpr int LD = TqCfg<MAXM>::LD, RB = TqCfg<MAXM>::RB;
    __shared__ TqShared<MAXM> S;
    __shared__ double s_y0, s_err;
    extern __shared__ double piv[];  // pivot scratch of tq_vectors / resolvent, Z of the QR fallback
    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (c >= count) return;
    if (!tq_spectrum<MAXM>(alpha, beta, c, m, ld, S)) {
        for (int row = tid; row < m; row += blockDim.x) zvec[(size_t)row * ld + c] = nan("");
        return;
    }
    const int n = S.n;
    const double sc = scale[c] / S.s2;  // f is applied to the unscaled eigenvalues
    if (S.fallback) {
        if (warp == 0) fvec_by_qr<MAXM>(S.a, S.b, n, m, sc, lane, piv, zvec, ld, c);
        return;
    }
    // S.bw is free after the grouping: 1 marks an isolated eigenvalue
    for (int i = tid; i < n; i += blockDim.x) S.bw[i] = 0.0;
    if (tid == 0) s_err = 0.0;
    __syncthreads();
    for (int g = tid; g < S.ngroups; g += blockDim.x)
        if (S.cl_of_group[g] < 0) S.bw[S.gfirst[g]] = 1.0;
    __syncthreads();
    const int yk = tid >> 2, part = tid & 3;  // component of y, lane of its quad
    double y = 0.0;
    for (int rb = 0; rb < n; rb += RB) {
        const int nb = min(RB, n - rb);
        tq_vectors<MAXM, true>(S, piv, rb, nb);
        if (tid < nb) {
            const int i = rb + tid;
            S.c0[tid] = S.bw[i] != 0.0 ? S.z1[i] * f_entropy(sc * S.th[i]) / S.nrm[i] : 0.0;
        }
        __syncthreads();
        if (yk < n)
            for (int r = part; r < nb; r += 4) y += S.c0[r] * piv[yk * LD + r];
        __syncthreads();
    }
    // clusters: one round per cluster, contour point q on lane q of warp 0
    double* Dp = piv + lane;              // real parts of the resolvent recurrences, [k][LD]
    double* Rp = piv + MAXM * LD + lane;  // imaginary parts
    for (int cl = 0; cl < S.ncl; cl++) {
        if (warp == 0) {
            const double cc = S.cc[cl], rho = S.rho[cl], half = S.half[cl];
            double sph, cph;
            sincospi((2.0 * lane + 1.0) / kContourPoints, &sph, &cph);
            const double dzr = rho * cph, dzi = rho * sph;
            const double zr = cc + dzr, zi = dzi;
            // bottom-up continued fraction g_k, stored
            double gr = zr - S.a[n - 1], gi = zi;
            Dp[(n - 1) * LD] = gr;
            Rp[(n - 1) * LD] = gi;
            for (int k = n - 2; k >= 0; k--) {
                const double t = S.b2[k + 1] / (gr * gr + gi * gi);
                gr = (zr - S.a[k]) - t * gr;
                gi = zi + t * gi;
                Dp[k * LD] = gr;
                Rp[k * LD] = gi;
            }
            // Taylor weight h = dz (f0 + f1 dz + f2 dz^2 / 2) of the cluster centre
            const double x0 = sc * cc;
            const double f0 = f_entropy(x0);
            const double f1 = x0 > 0.0 ? sc * (-log(x0) - 1.0) : 0.0;
            const double f2 = cc > 0.0 ? -sc / cc : 0.0;
            const double d2r = dzr * dzr - dzi * dzi, d2i = 2.0 * dzr * dzi;
            const double pr = f0 + f1 * dzr + 0.5 * f2 * d2r, pi = f1 * dzi + 0.5 * f2 * d2i;
            const double hr = (dzr * pr - dzi * pi) / kContourPoints, hi = (dzr * pi + dzi * pr) / kContourPoints;
            // forward ratios: x_0 = 1 / g_0, x_k = x_{k-1} beta_{k-1} / g_k;
            // this point's share of y_k replaces the real part of g_k
            double xr, xi;
            {
                const double den = gr * gr + gi * gi;
                xr = gr / den;
                xi = -gi / den;
            }
            double wq = (xr * dzr - xi * dzi) / kContourPoints;  // Re x_0 dz / K
            Dp[0] = xr * hr - xi * hi;
            for (int k = 1; k < n; k++) {
                const double g_r = Dp[k * LD], g_i = Rp[k * LD];
                const double inv = S.b[k - 1] / (g_r * g_r + g_i * g_i);
                const double ur = g_r * inv, ui = -g_i * inv;  // beta / g
                const double nxr = xr * ur - xi * ui, nxi = xr * ui + xi * ur;
                xr = nxr;
                xi = nxi;
                Dp[k * LD] = xr * hr - xi * hi;
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) wq += __shfl_xor_sync(0xffffffffu, wq, off);
            if (lane == 0 && half > 1e-3 * fabs(cc))  // cluster at the origin: error below W f(c + half)
                s_err += fmax(wq, 0.0) * f_entropy(fmin(sc * fmax(cc + half, 0.0), 0.36787944117144233));
        }
        __syncthreads();
        if (yk < n)
            for (int r = part; r < 32; r += 4) y += piv[yk * LD + r];
        __syncthreads();
    }
    y += __shfl_xor_sync(0xffffffffu, y, 1);
    y += __shfl_xor_sync(0xffffffffu, y, 2);
    if (part == 0 && yk < m) zvec[(size_t)yk * ld + c] = yk < n ? y : 0.0;
    if (tid == 0) s_y0 = y;
    __syncthreads();
    if (warp == 0 && !(s_err <= 1e-10 * fabs(s_y0))) fvec_by_qr<MAXM>(S.a, S.b, n, m, sc, lane, piv, zvec, ld, c);
}

// A-posteriori bounds of Theorem 4.4 for the polynomial Lanczos quadrature
// after m steps (A V_m = V_m T_m + beta_m v_{m+1} e_m^T): with Ritz values
// theta_j, a_j = beta_m U_{mj}, b_j = U_{1j} and
// gamma_j = sum_{l != j} a_l b_l / (theta_j - theta_l),
//   g_m(z) = sum_j a_j^2 b_j^2 f[theta_j, theta_j, z] + 2 a_j b_j gamma_j f[theta_j, z]
// (divided differences of f, the limits at z = theta_j included; evaluated
// stably, see g_term), and ||c||^2 min / max of |g_m| over the
// spectral interval bound the quadrature error from below / above; their
// geometric mean is the paper's error estimate.  The minimum and maximum are
// taken over `grid` geometrically and `grid` linearly spaced points of
// [lam_min, lam_max] plus the Ritz values inside it, spread over the lanes.
// U_{1j}, U_{mj} come from the twisted-factorisation eigenvectors of the
// shared spectrum (for a tight cluster the individual products are as
// ill-conditioned as the formula itself).  f(x) = -x log x; the interval must
// be positive.
// Divided differences of f(x) = -x log x at (t, z), z = t (1 + u):
// f[t, z] = -log t - h and f[t, t, z] = (1 - h) / (z - t) with
// h = z (log z - log t) / (z - t) = (log z - log t) (1 + 1 / u).  For |u| < 0.1
// the power series 1 - h = sum_{k>=1} (-1)^k u^k / (k (k + 1)) (16 terms: the
// next are below 1e-18 of the sum) avoids the cancellation of the plain
// quotients.  With a Ritz value's constants this gives its term of g_m without
// the part -2 ab gamma log t, which does not depend on z and is summed once.
// FP64 instructions are what a term costs (a warp's holds its port 64 cycles):
// 12 in the plain form with 1 / u from a single-precision seed and one step of
// Halley's iteration, w (1 + e + e^2) with e = 1 - u w (three instructions, error
// e^3 < 1e-20; a division is nine, a reciprocal six), 21 by the series.
struct GTerm {
    double t, it, lt, c2, c1;  // theta, 1 / theta, log theta, (a b)^2 / theta, 2 a b gamma
};
__device__ __forceinline__ double g_term(double z, double lz, const GTerm& p, double g) {
    const double u = (z - p.t) * p.it;
    const float uf = (float)u;
    if (fabsf(uf) < 0.1f) {
        double ser = 0.0;  // (1 - h) / u by Horner
#pragma unroll
        for (int k = 16; k >= 1; k--) ser = fma(ser, u, ((k & 1) ? -1.0 : 1.0) / (double)(k * (k + 1)));
        g = fma(p.c2, ser, g);
        return fma(p.c1, fma(ser, u, -1.0), g);
    }
    double w = (double)__frcp_rn(uf);
    if (fabsf(uf) > 1e30f) {  // the seed would leave single precision's range
        w = 1.0 / u;
    } else {
        const double e = fma(-u, w, 1.0);
        w = fma(w, fma(e, e, e), w);
    }
    const double h = (lz - p.lt) * (1.0 + w);
    g = fma(p.c2 * w, 1.0 - h, g);
    return fma(-p.c1, h, g);
}

// The points are most of the work: 2 grid + n of them with n terms each, on the
// four FP64 ports of the column's SM.  So a column may take a cluster of two, four
// or eight CTAs: every CTA computes the spectrum (the same numbers, and no later
// than one would), takes its share of the points, and CTA 0 reads the others'
// minimum and maximum.  The values of the points, and so the results, do not depend on
// the cluster's size.  Served mix of 32 queries (460 calls of 8 to 1400
// columns, 512 points, 5 to 32 steps): 72 -> 62 us a call.
template <int MAXM>
__global__ void __launch_bounds__(TqCfg<MAXM>::NT)
    k_tridiag_bounds(const double* __restrict__ alpha, const double* __restrict__ beta,
                     const double* __restrict__ norm2, const double* __restrict__ scale, int count, int m_all, int ld,
                     double lam_min, double lam_max, int grid, double* __restrict__ lower,
                     double* __restrict__ upper, double* __restrict__ estimate, const int32_t* __restrict__ cols,
                     const int32_t* __restrict__ mcol, const double* __restrict__ lam_max_col,
                     double* __restrict__ psi) {
    __shared__ TqShared<MAXM> S;
    __shared__ GTerm G[MAXM];
    extern __shared__ double piv[];  // pivot scratch of tq_vectors
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto cluster = cooperative_groups::this_cluster();
    const int csize = (int)cluster.num_blocks(), crank = (int)cluster.block_rank();
    const int entry = (int)blockIdx.x / csize;
    if (entry >= count) return;
    // column c (of the ld-strided arrays) after m steps, with its own upper end
    // of the spectral interval if given; every return before the minimum is taken
    // by all CTAs of the cluster (the same data) or by none
    const int c = cols ? cols[entry] : entry;
    const int m = mcol ? mcol[entry] : m_all;
    if (lam_max_col) lam_max = lam_max_col[entry];
    auto put = [&](double lo, double hi, double est) {
        if (tid == 0 && crank == 0) {
            lower[c] = lo;
            upper[c] = hi;
            estimate[c] = est;
        }
    };
    if (!tq_spectrum<MAXM>(alpha, beta, c, m, ld, S)) {
        put(nan(""), nan(""), nan(""));
        if (psi && tid == 0 && crank == 0) psi[c] = nan("");
        return;
    }
    const int n = S.n;
    const double sc = scale[c] / S.s2;
    const double bm = beta[(size_t)(m - 1) * ld + c] * scale[c];  // beta_m of A
    const bool invariant = n < m || bm == 0.0;  // the Krylov space is invariant: the quadrature is exact
    if (!invariant || (psi && !S.fallback))
        for (int rb = 0; rb < n; rb += TqCfg<MAXM>::RB)
            tq_vectors<MAXM, false>(S, piv, rb, min(TqCfg<MAXM>::RB, n - rb));
    if (psi && crank == 0) {  // the quadrature itself, from the same spectrum
        if (S.fallback) {
            if (warp == 0) quad_by_qr<MAXM>(S.a, S.b, n, sc, norm2[c], lane, psi + c);
        } else {
            tq_quadrature<MAXM>(S, sc, norm2[c], psi + c);
        }
        __syncthreads();
    }
    if (invariant) {
        put(0.0, 0.0, 0.0);
        return;
    }
    if (tid == 0) {
        S.gmin = 0x7ff0000000000000ULL;  // +inf
        S.gmax = 0;
    }
    for (int j = tid; j < n; j += blockDim.x) {
        GTerm p;
        const double ab = bm * (S.zn[j] * S.z1[j]) / S.nrm[j];
        p.t = sc * S.th[j];
        p.it = 1.0 / p.t;
        p.lt = log(p.t);
        p.c2 = ab * ab * p.it;
        p.c1 = 0.0;
        G[j] = p;
        S.c0[j] = ab;
    }
    __syncthreads();
    {  // gamma_j = sum_{l != j} a_l b_l / (theta_j - theta_l), four lanes per j
        const int j = tid >> 2, part = tid & 3;
        double gs = 0.0;
        if (j < n)
            for (int l = part; l < n; l += 4)
                if (l != j) gs += S.c0[l] / (G[j].t - G[l].t);
        gs += __shfl_xor_sync(0xffffffffu, gs, 1);
        gs += __shfl_xor_sync(0xffffffffu, gs, 2);
        if (part == 0 && j < n) {
            G[j].c1 = 2.0 * S.c0[j] * gs;
            S.c1[j] = G[j].c1 * G[j].lt;
        }
    }
    __syncthreads();
    if (!(lam_min > 0.0)) {
        // half the smallest positive Ritz value of this column
        double tmin = INFINITY;
        for (int j = n - 1; j >= 0 && G[j].t > 0.0; j--) tmin = G[j].t;
        lam_min = 0.5 * tmin;
    }
    if (!(lam_min > 0.0 && lam_max > lam_min)) {
        put(INFINITY, INFINITY, INFINITY);  // no usable interval: not converged
        return;
    }
    double g0 = 0.0;  // the part of g_m that does not depend on z
    for (int j = 0; j < n; j++) g0 -= S.c1[j];
    const int npts = 2 * grid + n;
    const double lmin = log(lam_min), lratio = log(lam_max / lam_min), inv = grid > 1 ? 1.0 / (grid - 1) : 0.0;
    const double lstep = lratio * inv, zstep = (lam_max - lam_min) * inv;
    unsigned long long gmin = 0x7ff0000000000000ULL, gmax = 0;
    for (unsigned i = crank * TqCfg<MAXM>::NT + tid; i < (unsigned)npts; i += csize * TqCfg<MAXM>::NT) {
        const int q = (int)i;
        double z, lz;
        if (q < grid) {
            const double x = lstep * q;
            z = lam_min * exp(x);
            lz = lmin + x;
        } else if (q < 2 * grid) {
            z = lam_min + zstep * (q - grid);
            lz = log(z);
        } else {
            z = G[q - 2 * grid].t;
            if (!(z >= lam_min && z <= lam_max)) continue;
            lz = G[q - 2 * grid].lt;
        }
        double g = g0;
        for (int j = 0; j < n; j++) g = g_term(z, lz, G[j], g);
        // |g| >= 0: the order of the bits; NaN takes no part
        const unsigned long long ab = (unsigned long long)absbits(g);
        if (ab <= 0x7ff0000000000000ULL) {
            gmin = min(gmin, ab);
            gmax = max(gmax, ab);
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        gmin = min(gmin, __shfl_xor_sync(0xffffffffu, gmin, off));
        gmax = max(gmax, __shfl_xor_sync(0xffffffffu, gmax, off));
    }
    if (lane == 0) {
        atomicMin(&S.gmin, gmin);
        atomicMax(&S.gmax, gmax);
    }
    cluster.sync();
    if (crank == 0 && tid == 0) {
        gmin = S.gmin;
        gmax = S.gmax;
        for (int r = 1; r < csize; r++) {
            gmin = min(gmin, *cluster.map_shared_rank(&S.gmin, r));
            gmax = max(gmax, *cluster.map_shared_rank(&S.gmax, r));
        }
    }
    cluster.sync();  // the other CTAs' shared memory has been read
    const double lo = __longlong_as_double((long long)gmin), hi = __longlong_as_double((long long)gmax);
    const double nb = norm2[c];
    put(nb * lo, nb * hi, nb * sqrt(lo * hi));
}

// CTAs per column of k_tridiag_bounds: the size with the least work on the
// fullest SM.  A CTA costs its share of the points plus a spectrum, which holds the
// FP64 ports as long as about 80 points do (512 columns of 10 steps: 0.05 us a
// column for the spectra, 0.32 for 522 points).
static int bounds_cluster(int count, int64_t points) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        return 1;
    int best = 1;
    int64_t best_cost = 0;
    for (int size = 1; size <= 8; size *= 2) {
        const int64_t cost = (((int64_t)count * size + sms - 1) / sms) * (80 + points / size);
        if (size == 1 || cost < best_cost) {
            best = size;
            best_cost = cost;
        }
    }
    return best;
}

cudaError_t launch_tridiag_bounds(const double* alpha, const double* beta, const double* norm2, const double* scale,
                                  int count, int m, int ld, double lam_min, double lam_max, int grid, double* lower,
                                  double* upper, double* estimate, double* psi, cudaStream_t st) {
    return launch_tridiag_bounds_list(alpha, beta, norm2, scale, count, nullptr, nullptr, nullptr, m, ld, lam_min,
                                      lam_max, grid, lower, upper, estimate, psi, st);
}

cudaError_t launch_tridiag_bounds_list(const double* alpha, const double* beta, const double* norm2,
                                       const double* scale, int count, const int32_t* cols, const int32_t* mcol,
                                       const double* lam_max_col, int m, int ld, double lam_min, double lam_max,
                                       int grid, double* lower, double* upper, double* estimate, double* psi,
                                       cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    // lam_min <= 0: half the smallest positive Ritz value of each column
    if ((!lam_max_col && !(lam_max > 0.0 && lam_max > lam_min)) || grid < 1) return cudaErrorInvalidValue;
    const int size = bounds_cluster(count, 2 * (int64_t)grid + m);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = size;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
#define VNE_BOUND_CASE(MM)                                                                                   \
    if (m <= MM) {                                                                                          \
        const int smem = TqCfg<MM>::kSmem;                                                                  \
        cudaError_t e = cudaFuncSetAttribute(k_tridiag_bounds<MM>,                                          \
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem);            \
        if (e != cudaSuccess) return e;                                                                     \
        cudaLaunchConfig_t cfg{};                                                                           \
        cfg.gridDim = dim3((unsigned)(count * size));                                                       \
        cfg.blockDim = dim3(TqCfg<MM>::NT);                                                                 \
        cfg.dynamicSmemBytes = smem;                                                                        \
        cfg.stream = st;                                                                                    \
        cfg.attrs = at;                                                                                     \
        cfg.numAttrs = 1;                                                                                   \
        e = cudaLaunchKernelEx(&cfg, k_tridiag_bounds<MM>, alpha, beta, norm2, scale, count, m, ld, lam_min, \
                               lam_max, grid, lower, upper, estimate, cols, mcol, lam_max_col, psi);        \
        return e != cudaSuccess ? e : cudaGetLastError();                                                   \
    }
    VNE_BOUND_CASE(32)
    VNE_BOUND_CASE(64)
    VNE_BOUND_CASE(128)
#undef VNE_BOUND_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_tridiag_quad(const double* alpha, const double* beta, const double* norm2,
                                const double* scale_per_col, int count, int m, int ld, double* psi,
                                cudaStream_t st) {
    return launch_tridiag_quad_list(alpha, beta, norm2, scale_per_col, count, nullptr, nullptr, m, ld, psi, st);
}

cudaError_t launch_tridiag_quad_list(const double* alpha, const double* beta, const double* norm2,
                                     const double* scale_per_col, int count, const int32_t* cols,
                                     const int32_t* mcol, int m, int ld, double* psi, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    // one CTA per tridiagonal; dynamic shared memory holds the
    // twisted-factorisation pivots of up to 64 eigenvalues
#define VNE_QUAD_CASE(MM)                                                                                    \
    if (m <= MM) {                                                                                          \
        const int smem = TqCfg<MM>::kSmem;                                                                  \
        cudaError_t e = cudaFuncSetAttribute(k_tridiag_quad<MM>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                             smem);                                                         \
        if (e != cudaSuccess) return e;                                                                     \
        k_tridiag_quad<MM><<<count, TqCfg<MM>::NT, smem, st>>>(alpha, beta, norm2, scale_per_col, count, m,  \
                                                                ld, psi, cols, mcol);                       \
        return cudaGetLastError();                                                                          \
    }
    VNE_QUAD_CASE(32)
    VNE_QUAD_CASE(64)
    VNE_QUAD_CASE(128)
#undef VNE_QUAD_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_tridiag_fvec(const double* alpha, const double* beta, const double* scale_per_col, int count,
                                int m, int ld, double* zvec, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    // one CTA per tridiagonal; dynamic shared memory: pivots / resolvent, or
    // Z for the QR fallback (MM x MM, which fits)
#define VNE_FVEC_CASE(MM)                                                                                    \
    if (m <= MM) {                                                                                          \
        const int smem = TqCfg<MM>::kSmem;                                                                  \
        static_assert(TqCfg<MM>::kSmem >= MM * MM * (int)sizeof(double), "Z of the QR fallback");           \
        cudaError_t e = cudaFuncSetAttribute(k_tridiag_fvec<MM>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                             smem);                                                         \
        if (e != cudaSuccess) return e;                                                                     \
        k_tridiag_fvec<MM><<<count, TqCfg<MM>::NT, smem, st>>>(alpha, beta, scale_per_col, count, m, ld,    \
                                                                zvec);                                      \
        return cudaGetLastError();                                                                          \
    }
    VNE_FVEC_CASE(32)
    VNE_FVEC_CASE(64)
    VNE_FVEC_CASE(128)
#undef VNE_FVEC_CASE
    return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// Gram C = X^T Y, 64 x 64 output tile per CTA, rows split into chunks.
// Each thread owns a 4 x 4 block of the tile; the 64-row slabs of X and Y are
// staged transposed-free in shared memory ([row][col], float4-aligned).
// Products accumulate in the data precision over one 64-row slab, then in
// FP64 across slabs.
template <typename T, int KS>
__global__ void __launch_bounds__(256) k_gram(const T* __restrict__ X, int kx, const T* __restrict__ Y, int ky,
                                              int n, int rows_per_chunk, int tiles_y, double* __restrict__ part) {
    __shared__ __align__(16) T Xs[64][64];
    __shared__ __align__(16) T Ys[64][64];
    const int chunk = blockIdx.x;
    const int tx0 = (blockIdx.y / tiles_y) * 64, ty0 = (blockIdx.y % tiles_y) * 64;
    const int r_begin = chunk * rows_per_chunk;
    const int r_end = min(n, r_begin + rows_per_chunk);
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    double dacc[4][4];
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) dacc[a][b] = 0.0;
    for (int rt = r_begin; rt < r_end; rt += 64) {
        // each panel row holds KS consecutive columns: copy whole KS-runs
        for (int idx = threadIdx.x; idx < 64 * 64; idx += 256) {
            int rl = idx / 64, cl = idx % 64;
            int r = rt + rl;
            int cxg = tx0 + cl, cyg = ty0 + cl;
            T xv = (T)0, yv = (T)0;
            if (r < r_end) {
                if (cxg < kx) xv = X[(size_t)(cxg / KS) * n * KS + (size_t)r * KS + (cxg % KS)];
                if (cyg < ky) yv = Y[(size_t)(cyg / KS) * n * KS + (size_t)r * KS + (cyg % KS)];
            }
            Xs[rl][cl] = xv;
            Ys[rl][cl] = yv;
        }
        __syncthreads();
        T acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; a++)
#pragma unroll
            for (int b = 0; b < 4; b++) acc[a][b] = (T)0;
#pragma unroll 4
        for (int rl = 0; rl < 64; rl++) {
            T xa[4], yb[4];
#pragma unroll
            for (int a = 0; a < 4; a++) xa[a] = Xs[rl][tx * 4 + a];
#pragma unroll
            for (int b = 0; b < 4; b++) yb[b] = Ys[rl][ty * 4 + b];
#pragma unroll
            for (int a = 0; a < 4; a++)
#pragma unroll
                for (int b = 0; b < 4; b++) acc[a][b] += xa[a] * yb[b];
        }
#pragma unroll
        for (int a = 0; a < 4; a++)
#pragma unroll
            for (int b = 0; b < 4; b++) dacc[a][b] += (double)acc[a][b];
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) {
            int i = tx0 + tx * 4 + a, j = ty0 + ty * 4 + b;
            if (i < kx && j < ky) part[(size_t)chunk * kx * ky + (size_t)i * ky + j] = dacc[a][b];
        }
}

__global__ void k_gram_reduce(const double* __restrict__ part, int nchunks, int total, double* __restrict__ C) {
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    double s = 0.0;
    for (int c = 0; c < nchunks; c++) s += part[(size_t)c * total + idx];
    C[idx] = s;
}

// C <- C + C^T in place (C = the summed partials E of a symmetric Gram): one
// thread per pair a <= b.
__global__ void k_gram_symmetrize(double* __restrict__ C, int k) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= k * k) return;
    const int a = idx / k, b = idx % k;
    if (a > b) return;
    const double s = C[a * k + b] + C[b * k + a];
    C[a * k + b] = s;
    C[b * k + a] = s;
}

template <typename T>
cudaError_t launch_gram(const T* X, int kx, const T* Y, int ky, int ks, int n, double* part, int nchunks, double* C,
                        int* err, cudaStream_t st) {
    if (kx <= 0 || ky <= 0) return cudaSuccess;
    if (sizeof(T) == 4 && err && kx <= 128 && ky <= 128 && (ks == 8 || ks == 16 || ks == 32)) {
        int chunks = 0, sym = 0;
        cudaError_t e = launch_gram_tc5(reinterpret_cast<const float*>(X), kx, reinterpret_cast<const float*>(Y), ky,
                                        ks, n, part, nchunks, err, &chunks, &sym, st);
        if (e != cudaSuccess) return e;
        const int total = kx * ky;
        k_gram_reduce<<<(total + 255) / 256, 256, 0, st>>>(part, chunks, total, C);
        if (sym) k_gram_symmetrize<<<(total + 255) / 256, 256, 0, st>>>(C, kx);
        return cudaGetLastError();
    }
    int tiles_x = (kx + 63) / 64, tiles_y = (ky + 63) / 64;
    int rpc = (n + nchunks - 1) / nchunks;
    rpc = ((rpc + 63) / 64) * 64;
    int chunks = rpc > 0 ? (n + rpc - 1) / rpc : 1;
    if (chunks < 1) chunks = 1;
    dim3 grid(chunks, tiles_x * tiles_y);
    if (ks == 4) k_gram<T, 4><<<grid, 256, 0, st>>>(X, kx, Y, ky, n, rpc, tiles_y, part);
    else if (ks == 8) k_gram<T, 8><<<grid, 256, 0, st>>>(X, kx, Y, ky, n, rpc, tiles_y, part);
    else if (ks == 16) k_gram<T, 16><<<grid, 256, 0, st>>>(X, kx, Y, ky, n, rpc, tiles_y, part);
    else if (ks == 32) k_gram<T, 32><<<grid, 256, 0, st>>>(X, kx, Y, ky, n, rpc, tiles_y, part);
    else return cudaErrorInvalidValue;
    int total = kx * ky;
    k_gram_reduce<<<(total + 255) / 256, 256, 0, st>>>(part, chunks, total, C);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Out = In2 + coef * In * M.  Persistent CTAs: M (FP64 [kin][kout]) is staged
// once per CTA in shared memory in the data precision, then 64-row tiles of
// In are streamed through shared memory (stored transposed, [k][row]); each
// thread owns 4 rows x 8 output columns.
template <typename T, int KS>
__global__ void __launch_bounds__(256) k_apply(const T* __restrict__ In, int kin, const double* __restrict__ M,
                                               int kout, const T* __restrict__ In2, T* __restrict__ Out, int n,
                                               double coef) {
    extern __shared__ __align__(16) unsigned char smraw[];
    T* Ms = reinterpret_cast<T*>(smraw);          // [kin][128]
    T* Ist = Ms + (size_t)kin * 128;              // [kin][64]  (transposed tile)
    for (int idx = threadIdx.x; idx < kin * 128; idx += 256) {
        int a = idx / 128, b = idx % 128;
        Ms[idx] = (b < kout) ? (T)(coef * M[(size_t)a * kout + b]) : (T)0;
    }
    const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;  // rows ty*4.., cols tx*8..
    const int ntiles = (n + 63) / 64;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int r0 = tile * 64;
        __syncthreads();
        for (int idx = threadIdx.x; idx < 64 * kin; idx += 256) {
            int c = idx / 64, rl = idx % 64;
            int r = r0 + rl;
            Ist[idx] = (r < n) ? In[(size_t)(c / KS) * n * KS + (size_t)r * KS + (c % KS)] : (T)0;
        }
        __syncthreads();
        if (tx * 8 >= kout) continue;
        T acc[4][8];
#pragma unroll
        for (int a = 0; a < 4; a++)
#pragma unroll
            for (int b = 0; b < 8; b++) acc[a][b] = (T)0;
        for (int k = 0; k < kin; k++) {
            T av[4], bv[8];
#pragma unroll
            for (int a = 0; a < 4; a++) av[a] = Ist[k * 64 + ty * 4 + a];
#pragma unroll
            for (int b = 0; b < 8; b++) bv[b] = Ms[k * 128 + tx * 8 + b];
#pragma unroll
            for (int a = 0; a < 4; a++)
#pragma unroll
                for (int b = 0; b < 8; b++) acc[a][b] += av[a] * bv[b];
        }
#pragma unroll
        for (int a = 0; a < 4; a++) {
            const int r = r0 + ty * 4 + a;
            if (r >= n) continue;
#pragma unroll
            for (int b = 0; b < 8; b++) {
                const int c = tx * 8 + b;
                if (c < kout) {
                    size_t o = (size_t)(c / KS) * n * KS + (size_t)r * KS + (c % KS);
                    T v = acc[a][b];
                    if (In2) v += In2[o];
                    Out[o] = v;
                }
            }
        }
    }
}

template <typename T>
cudaError_t launch_apply(const T* In, int kin, const double* M, int kout, const T* In2, T* Out, int ks, int n,
                         double coef, int* err, cudaStream_t st) {
    if (kout > 128 || kin > 128) return cudaErrorInvalidValue;
    if (sizeof(T) == 4 && err && kin > 0 && kout > 0 && (ks == 8 || ks == 16 || ks == 32))
        return launch_apply_tc5(reinterpret_cast<const float*>(In), kin, M, kout, reinterpret_cast<const float*>(In2),
                                reinterpret_cast<float*>(Out), ks, n, coef, err, st);
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int ntiles = (n + 63) / 64;
    size_t smem = ((size_t)kin * 128 + 64 * (size_t)kin) * sizeof(T);
    int per_sm = sizeof(T) == 4 ? 2 : 1;
    dim3 grid(ntiles < sms * per_sm ? ntiles : sms * per_sm);
#define VNE_APPLY_CASE(KSV)                                                                                  \
    if (ks == KSV) {                                                                                        \
        cudaError_t e = cudaFuncSetAttribute(k_apply<T, KSV>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                             (int)smem);                                                    \
        if (e != cudaSuccess) return e;                                                                     \
        k_apply<T, KSV><<<grid, 256, smem, st>>>(In, kin, M, kout, In2, Out, n, coef);                      \
        return cudaGetLastError();                                                                          \
    }
    VNE_APPLY_CASE(4)
    VNE_APPLY_CASE(8)
    VNE_APPLY_CASE(16)
    VNE_APPLY_CASE(32)
#undef VNE_APPLY_CASE
    return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// Pivoted Cholesky G = P R^T R P^T (FP64), in two kernels: the factor (one
// CTA) and the triangular inverse (a warp per column).  Stops when the
// largest remaining pivot is <= tol * max diag(G); rank r = pivots taken.
// Writes Minv with Minv[piv[i]][c] = (R^{-1})[i][c] for i, c < r, zero
// elsewhere, so that Y Minv has orthonormal columns in exact arithmetic.
// Pivoted Cholesky factor of the FP64 Gram (one CTA): R upper triangular
// with P^T G P = R^T R, the pivots, 1 / R_jj and the numerical rank (the
// first pivot below tol * max diag stops the factorisation).  FP64 runs at a
// small fraction of the FP32 rate on this part, so a step costs one square
// root and one reciprocal (thread 0) and the row is scaled by multiplication.
// Output R: work[0 .. k*k) row-major (upper triangle), 1 / R_jj:
// work[k*k .. k*k + k), pivots: piv[0 .. k).  With pivot = 0 the columns are
// taken in their order (plain Cholesky; the first pivot below the cut-off
// stops it).
__global__ void k_chol_factor(const double* __restrict__ G, int k, double tol, double* __restrict__ work,
                              int* __restrict__ piv_out, int* __restrict__ rank_out, int pivot) {
    extern __shared__ double A[];  // k x (k + 1): odd row stride against bank conflicts
    const int ld = k + 1;
    __shared__ int piv[128];
    __shared__ int s_p, s_rank;
    __shared__ double s_max0, s_rinv;
    // symmetric part of G (the Gram partial sums of (a, b) and (b, a) may
    // round differently)
    for (int idx = threadIdx.x; idx < k * k; idx += blockDim.x) {
        const int a = idx / k, b = idx % k;
        A[a * ld + b] = 0.5 * (G[idx] + G[b * k + a]);
    }
    for (int i = threadIdx.x; i < k; i += blockDim.x) piv[i] = i;
    __syncthreads();
    if (threadIdx.x == 0) {
        double mx = 0.0;
        for (int i = 0; i < k; i++) mx = fmax(mx, A[i * ld + i]);
        s_max0 = mx;
        s_rank = k;
    }
    __syncthreads();
    for (int j = 0; j < k; j++) {
        if (threadIdx.x < 32) {
            // largest remaining diagonal entry (warp argmax, ties to the lower index)
            double best = -INFINITY;
            int p = j;
            if (pivot) {
                for (int i = j + (int)threadIdx.x; i < k; i += 32)
                    if (A[i * ld + i] > best) {
                        best = A[i * ld + i];
                        p = i;
                    }
            } else if (threadIdx.x == 0) {
                best = A[j * ld + j];
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const double ob = __shfl_xor_sync(0xffffffffu, best, off);
                const int op = __shfl_xor_sync(0xffffffffu, p, off);
                if (ob > best || (ob == best && op < p)) {
                    best = ob;
                    p = op;
                }
            }
            if (threadIdx.x == 0) {
                s_p = (best > tol * s_max0 && best > 0.0) ? p : -1;
                if (s_p < 0) s_rank = j;
            }
        }
        __syncthreads();
        const int p = s_p;
        if (p < 0) break;
        if (p != j) {
            for (int i = threadIdx.x; i < k; i += blockDim.x) {  // swap rows
                double t = A[j * ld + i];
                A[j * ld + i] = A[p * ld + i];
                A[p * ld + i] = t;
            }
            __syncthreads();
            for (int i = threadIdx.x; i < k; i += blockDim.x) {  // swap columns
                double t = A[i * ld + j];
                A[i * ld + j] = A[i * ld + p];
                A[i * ld + p] = t;
            }
            if (threadIdx.x == 0) {
                int t = piv[j];
                piv[j] = piv[p];
                piv[p] = t;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            const double rjj = sqrt(A[j * ld + j]);
            A[j * ld + j] = rjj;
            s_rinv = 1.0 / rjj;
        }
        __syncthreads();
        const double rinv = s_rinv;
        for (int i = j + 1 + threadIdx.x; i < k; i += blockDim.x) A[j * ld + i] *= rinv;
        if (threadIdx.x == 0) work[(size_t)k * k + j] = rinv;
        __syncthreads();
        // rank-1 update of the trailing block: the upper triangle (a warp per
        // row), mirrored into the lower one for later pivot swaps
        const int rem = k - j - 1;
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
        for (int a = warp; a < rem; a += nwarp) {
            const int ga = j + 1 + a;
            const double la = A[j * ld + ga];
            for (int gb = ga + lane; gb < k; gb += 32) {
                const double v = fma(-la, A[j * ld + gb], A[ga * ld + gb]);
                A[ga * ld + gb] = v;
                A[gb * ld + ga] = v;
            }
        }
        __syncthreads();
    }
    __syncthreads();
    const int r = s_rank;
    for (int idx = threadIdx.x; idx < k * k; idx += blockDim.x) {
        const int a = idx / k, b = idx % k;
        work[idx] = (a < r && b >= a) ? A[a * ld + b] : 0.0;
    }
    for (int i = threadIdx.x; i < k; i += blockDim.x) piv_out[i] = piv[i];
    if (threadIdx.x == 0) *rank_out = r;
}

// Minv = P R^{-1} (rows permuted back), zero beyond the rank: column c of
// R^{-1} by back substitution, x_c = 1 / R_cc and, for i = c - 1 .. 0,
// x_i = -(sum_{l = i+1..c} R_il x_l) / R_ii.  One warp per column, R staged
// in shared memory, the inner products lane-parallel with a butterfly sum;
// the columns are spread over the SMs (a column's chain is serial).
__global__ void __launch_bounds__(256) k_tri_inv(const double* __restrict__ work, int k, const int* __restrict__ piv,
                                                 const int* __restrict__ rank, double* __restrict__ Minv) {
    extern __shared__ double R[];  // rows 0 .. c_hi of R, row stride k + 1
    __shared__ double xs[8][128];
    const int ld = k + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = *rank;
    const int c_hi = min(k - 1, (int)blockIdx.x * 8 + 7);  // last column of this CTA
    for (int idx = threadIdx.x; idx < (c_hi + 1) * k; idx += blockDim.x) {
        const int a = idx / k, b = idx % k;
        R[a * ld + b] = work[idx];
    }
    __syncthreads();
    const int c = blockIdx.x * 8 + warp;
    if (c >= k) return;
    const double* rinv = work + (size_t)k * k;
    double* x = xs[warp];
    if (c < r) {
        if (lane == 0) x[c] = rinv[c];
        __syncwarp();
        for (int i = c - 1; i >= 0; i--) {
            double s = 0.0;
            for (int l = i + 1 + lane; l <= c; l += 32) s = fma(R[i * ld + l], x[l], s);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            if (lane == 0) x[i] = -s * rinv[i];
            __syncwarp();
        }
    }
    for (int i = lane; i < k; i += 32) Minv[(size_t)piv[i] * k + c] = (c < r && i <= c) ? x[i] : 0.0;
}

cudaError_t launch_chol_qr_factor(const double* G, int k, double tol, double* Minv, int* rank, double* work,
                                  int* piv, cudaStream_t st, bool pivot) {
    if (k > 128 || k <= 0) return cudaErrorInvalidValue;
    const size_t smem = (size_t)k * (k + 1) * sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(k_chol_factor, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_tri_inv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_chol_factor<<<1, 256, smem, st>>>(G, k, tol, work, piv, rank, pivot ? 1 : 0);
    k_tri_inv<<<(k + 7) / 8, 256, smem, st>>>(work, k, piv, rank, Minv);
    return cudaGetLastError();
}

template cudaError_t launch_gram<float>(const float*, int, const float*, int, int, int, double*, int, double*, int*,
                                       cudaStream_t);
template cudaError_t launch_gram<double>(const double*, int, const double*, int, int, int, double*, int, double*, int*,
                                        cudaStream_t);
template cudaError_t launch_apply<float>(const float*, int, const double*, int, const float*, float*, int, int, double, int*, cudaStream_t);
template cudaError_t launch_apply<double>(const double*, int, const double*, int, const double*, double*, int, int, double, int*, cudaStream_t);

}  // namespace vne
