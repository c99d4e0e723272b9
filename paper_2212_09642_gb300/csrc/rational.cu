// Rational Krylov quadrature with negative real poles (Sections 4, 4.2, 5.3)
// via a batched multi-shift conjugate gradient.
//
// For poles xi_s = -s_s (s_s > 0) and ell poles at infinity the rational
// Krylov space of eq. rational-krylov-subspace-definition is, by partial
// fractions, span{c, A c, .., A^ell c, x_1, .., x_S} with
// x_s = (A + s_s I)^{-1} c.  All S shifted systems are solved from one
// Krylov sequence: conjugate gradients run on the seed system (A + s_0 I),
// s_0 the smallest shift, and every shifted residual stays collinear with the
// seed residual, r_s = zeta_s r, which gives each shifted iterate from the
// seed's coefficients (Jegerlehner 1996; Frommer 2003).  A shift is retired
// once |zeta_s| ||r|| <= tol ||c||.
//
// Per CG iteration, for a block of K columns (panel-major, as in the
// Lanczos engine):
//   step kernel (shared with Lanczos)  q = (A + s_0 I) p,  d = p . q
//   k_cg_update      a = rho / d, r_{k+1} = r_k - a q into the next slot of a
//                    window of residuals, rho' = ||r_{k+1}||^2; the CTA that
//                    finishes a panel advances the panel's scalars: b =
//                    rho'/rho, zeta_s, a_s, b_s, convergence, and records
//                    zeta_s, a_s, b_s of the iteration
//   k_cg_direction   p = r + b p
// The shifted iterates are not touched per iteration.  With p_{s,k} =
// zeta_k r_k + b_{s,k-1} p_{s,k-1} and x_s += a_{s,k} p_{s,k}, a whole window
// of iterations adds to x_s and leaves in p_s fixed combinations of the
// window's residuals and of the p_s that entered it; their coefficients
// follow from the recorded scalars by a backward recurrence (k_cg_coefs), and
// one pass (k_cg_flush) reads every residual of the window once for all
// shifts.  An iteration then moves 6 vectors and a share of (window + 4 per
// live shift) / window instead of 6 + 4 per live shift.  Measured at n = 10^6,
// 22 columns, 8 shifts, FP32, per iteration: update 88 us and flush 46 us
// against 283 us for the update that touched every live x_s and p_s and 19 us
// for its scalar kernels (estimate 397 -> 278 ms; update 53 and flush 33 us, 183
// ms, with the shapes described at each kernel); FP64, n = 30,000, 12 columns:
// 23 + 10 us against 51 + 15 us (88 -> 59 ms; 41 ms now).
// Afterwards the basis W and A W are formed (A^j c by the step kernel,
// A x_s by the step kernel), their Gram matrices W^T W and W^T A W are
// accumulated per column in one pass over the vectors (k_multi_gram), and a per-column FP64 kernel orthonormalises W in
// pole order (Cholesky of the column-scaled Gram, dropping dependent
// columns; the first basis vector is c / ||c|| as in rational Arnoldi),
// applies that basis change to the vectors W and A W and repeats the
// orthonormalisation from the new Gram matrices (Cholesky-QR2, so the
// rounding error no longer grows with the square of the basis condition
// number), projects A, diagonalises the small matrix by cyclic Jacobi and
// returns psi = ||c||^2 e1^T f(A_m) e1.
#include <cooperative_groups.h>
#include <float.h>
#include <math.h>

#include "common.cuh"
#include "kernels.h"
#include "reduce.cuh"

namespace vne {

constexpr int kMaxBasis = 24;  // 1 + up to 15 polynomial directions + 8 poles

__device__ __forceinline__ double f_ent(double x) { return x > 0.0 ? -x * log(x) : 0.0; }

// r = p = c are set by copies; here the scalar state: rho = ||c||^2, zeta =
// zeta_prev = 1, a_prev = 1, b_prev = 0, all shifts active for non-zero
// columns.
__global__ void k_cg_init(CgState st, const double* norm2) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= st.K) return;
    const double n2 = norm2[c];
    st.rho[c] = n2;
    st.cnorm[c] = sqrt(n2);
    st.a_prev[c] = 1.0;
    st.b_prev[c] = 0.0;
    st.b[c] = 0.0;
    for (int s = 0; s < st.nshift; s++) {
        const size_t o = (size_t)s * st.K + c;
        st.zeta[o] = 1.0;
        st.zeta_prev[o] = 1.0;
        st.zeta_next[o] = 1.0;
        st.bstart[o] = 0.0;
        st.active[o] = n2 > 0.0 ? 1 : 0;
        st.iters[o] = 0;
        st.resid[o] = n2 > 0.0 ? 1.0 : 0.0;
    }
}

cudaError_t launch_cg_init(CgState st, const double* norm2, cudaStream_t s) {
    k_cg_init<<<(st.K + 63) / 64, 64, 0, s>>>(st, norm2);
    return cudaGetLastError();
}

// r_{k+1} = r_k - a q with a = rho / d (d from the step kernel as scale *
// (p . q)), rho' = ||r_{k+1}||^2 (runs of 16 rows in the data precision, FP64
// across runs and CTAs).  Each lane owns CPL consecutive columns of a row
// (16-byte vector accesses), four rows in flight.  A pure stream of three
// vectors.  The last CTA of a panel advances the panel's scalars, one thread
// per (shift, column): two single-warp kernels did that before, 19 us per
// iteration of dependent FP64 arithmetic that this tail spreads over a CTA.
// In FP32 a tile is short (two batches of four rows per thread), so what a CTA
// does before and after the rows counts: the first rows are loaded before the
// step lengths are formed, 64 registers keep four CTAs per SM (n = 10^6, 22
// columns: 70 us at three per SM; 62 so; loading the next rows ahead as well
// takes 96 registers and 80 us), and a CTA takes several tiles of a long panel
// (cg_update_ks).
// CLUSTER (FP64, few tiles): a thread-block cluster takes a tile, each CTA one
// run of 16 rows per thread, and CTA 0 adds the runs from distributed shared
// memory in the order in which one CTA would have added them (n = 30,000, 16
// columns: 32 tiles of 1888 rows, 23 us on 32 SMs; 18.6 in clusters of
// two).
template <typename T, int KS, bool CLUSTER>
__global__ void __launch_bounds__(VNE_THREADS, sizeof(T) == 8 ? 1 : 4)
    k_cg_update(CgVectors<T> v, CgState st, int wi, int it) {
    namespace cg = cooperative_groups;
    const int csize = CLUSTER ? (int)cg::this_cluster().num_blocks() : 1;
    const int crank = CLUSTER ? (int)cg::this_cluster().block_rank() : 0;
    const int cta = (int)blockIdx.x / csize;
    constexpr int CPL = LaneVec<T>::CPL;
    constexpr int LPR = KS / CPL;            // lanes per row
    constexpr int RPI = VNE_THREADS / LPR;   // rows per iteration
    constexpr int U = 4;
    // panels in reverse order: the step kernel walked them forwards, so the last
    // panel's q is still in L2 when this starts, and the direction pass begins
    // on the panel whose residual this wrote last
    const int tiles = (v.tiles_per_panel + v.group - 1) / v.group;  // CTAs per panel
    const int np = (int)gridDim.x / csize / tiles;
    const int panel = v.panel_base + np - 1 - cta / tiles, tile = cta % tiles;
    RowTile t = v.tiles[tile * v.group];
    t.row_end = v.tiles[min(v.tiles_per_panel, (tile + 1) * v.group) - 1].row_end;
    if (CLUSTER) {  // run crank of the tile
        t.row_begin += crank * 16 * RPI;
        t.row_end = min(t.row_end, t.row_begin + 16 * RPI);
    }
    const int sub = threadIdx.x % LPR, rs = threadIdx.x / LPR;
    const int cofs = sub * CPL;
    const size_t pofs = (size_t)panel * v.n * KS;
    const T* __restrict__ R = v.r + pofs;
    T* __restrict__ Rn = v.r_next + pofs;
    const T* __restrict__ Q = v.q + pofs;
    T rv[U][CPL], qv[U][CPL];
    auto fetch = [&](int r0, int re) {
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int r = r0 + u * RPI;
            if (r < re) {
                load_lane(R + (size_t)r * KS + cofs, rv[u]);
                load_lane_stream(Q + (size_t)r * KS + cofs, qv[u]);
            }
        }
    };
    // the first rows are on their way while the step lengths are formed (two
    // FP64 divisions behind two loads)
    int rb = t.row_begin + rs;
    if (rb < t.row_end) fetch(rb, min(t.row_end, rb + 16 * RPI));
    __shared__ double s_a[KS];
    if (threadIdx.x < KS) {
        const int c = panel * KS + threadIdx.x;
        const double d = st.dq[c] / st.scale, rho = st.rho[c];
        s_a[threadIdx.x] = (d > 0.0 && rho > 0.0) ? rho / d : 0.0;
    }
    __syncthreads();
    T a[CPL];
#pragma unroll
    for (int q = 0; q < CPL; q++) a[q] = (T)s_a[cofs + q];
    double acc[CPL];
    T accf[CPL];
#pragma unroll
    for (int q = 0; q < CPL; q++) {
        acc[q] = 0.0;
        accf[q] = (T)0;
    }
    // runs of 16 rows as a loop of its own: a flush under a condition would be a
    // predicated FP64 addition per iteration, which holds the FP64 port
    for (; rb < t.row_end; rb += 16 * RPI) {
        const int re = min(t.row_end, rb + 16 * RPI);
#pragma unroll 1
        for (int r0 = rb; r0 < re; r0 += U * RPI) {
            if (r0 != t.row_begin + rs) fetch(r0, re);
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int r = r0 + u * RPI;
                if (r < re) {
#pragma unroll
                    for (int q = 0; q < CPL; q++) {
                        rv[u][q] -= a[q] * qv[u][q];
                        accf[q] += rv[u][q] * rv[u][q];
                    }
                    store_lane(Rn + (size_t)r * KS + cofs, rv[u]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < CPL; q++) {
            acc[q] += (double)accf[q];
            accf[q] = (T)0;
        }
    }
    if (CLUSTER) {
        __shared__ double runs[CPL][VNE_THREADS];
#pragma unroll
        for (int q = 0; q < CPL; q++) runs[q][threadIdx.x] = acc[q];
        auto cl = cg::this_cluster();
        cl.sync();
        if (crank == 0)
            for (int k = 1; k < csize; k++) {
                const double* other = cl.map_shared_rank(&runs[0][0], k);
#pragma unroll
                for (int q = 0; q < CPL; q++) acc[q] += other[q * VNE_THREADS + threadIdx.x];
            }
        cl.sync();  // CTA 0 has read the runs
        if (crank != 0) return;
    }
    constexpr bool kSerial = sizeof(T) == 8;
    __shared__ double red[kSerial ? RPI : VNE_WARPS][KS];
    double tot;
    if (kSerial) cta_colsum_serial<KS, CPL>(acc, red, tot);
    else cta_colsum<KS, CPL>(acc, red, tot);
    if (threadIdx.x < KS) v.part[((size_t)panel * tiles + tile) * KS + threadIdx.x] = tot;
    __shared__ double s_rho[KS];
    if (kSerial) {
        __shared__ int s_last;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) s_last = (atomicAdd(v.counter + panel, 1u) == (unsigned)(tiles - 1));
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        if (threadIdx.x < KS) {
            double sum = 0.0;
            for (int i = 0; i < tiles; i++)
                sum += __ldcg(&v.part[((size_t)panel * tiles + i) * KS + threadIdx.x]);
            s_rho[threadIdx.x] = sum;
        }
        if (threadIdx.x == 0) v.counter[panel] = 0u;
        __syncthreads();
    } else if (!last_cta_reduce<KS>(v.part, v.counter + panel, panel, tiles, 0, tiles, s_rho)) {
        return;
    }
    int any = 0;
    for (int idx = threadIdx.x; idx < st.nshift * KS; idx += VNE_THREADS) {
        const int s = idx / KS, cc = idx % KS, c = panel * KS + cc;
        const size_t o = (size_t)s * st.K + c, h = ((size_t)wi * st.nshift + s) * st.K + c;
        if (!st.active[o]) {
            st.hz[h] = st.ha[h] = st.hb[h] = 0.0;
            continue;
        }
        // shifted step length from the collinear residuals
        const double aa = s_a[cc], rho = st.rho[c], rhon = s_rho[cc];
        const double zk = st.zeta[o];
        double zn = st.zeta_next[o], as = 0.0;
        if (aa != 0.0) {
            const double zkm1 = st.zeta_prev[o];
            const double ap = st.a_prev[c], bp = st.b_prev[c];
            const double delta = st.shift[s] - st.shift0;
            const double den = ap * zkm1 * (1.0 + delta * aa) + aa * bp * (zkm1 - zk);
            zn = (den != 0.0) ? zk * zkm1 * ap / den : 0.0;
            as = (zk != 0.0) ? aa * zn / zk : 0.0;
            st.zeta_next[o] = zn;
        }
        const double b = (rho > 0.0) ? rhon / rho : 0.0;
        const double ratio = (zk != 0.0) ? zn / zk : 0.0;
        st.hz[h] = zk;
        st.ha[h] = as;
        st.hb[h] = b * ratio * ratio;
        st.zeta_prev[o] = zk;
        st.zeta[o] = zn;
        st.iters[o] += 1;
        const double res = fabs(zn) * sqrt(rhon);
        st.resid[o] = res / st.cnorm[c];
        if (!(res > st.tol * st.cnorm[c])) st.active[o] = 0;  // converged (or breakdown)
        else any = 1;
    }
    any = __syncthreads_or(any);
    if (threadIdx.x < KS) {
        const int c = panel * KS + threadIdx.x;
        const double rho = st.rho[c], rhon = s_rho[threadIdx.x], aa = s_a[threadIdx.x];
        const double b = (rho > 0.0) ? rhon / rho : 0.0;
        st.a_prev[c] = aa;
        st.b_prev[c] = b;
        st.b[c] = b;
        st.rho[c] = rhon;
        if (st.ah && it < st.hist_rows) {
            st.ah[(size_t)it * st.K + c] = aa;
            st.bh[(size_t)it * st.K + c] = b;
        }
    }
    if (threadIdx.x == 0) st.any_active[panel] = any;
}

// p = r + b p
template <typename T, int KS>
__global__ void __launch_bounds__(VNE_THREADS) k_cg_direction(CgVectors<T> v, CgState st) {
    constexpr int CPL = LaneVec<T>::CPL;
    constexpr int LPR = KS / CPL;
    constexpr int RPI = VNE_THREADS / LPR;
    constexpr int U = 4;
    const int per = v.tiles_per_panel * v.sub;
    const int panel = v.panel_base + blockIdx.x / per;
    const int tile = (int)(blockIdx.x % per) / v.sub, piece = (int)(blockIdx.x % per) % v.sub;
    const RowTile t = v.tiles[tile];
    const int len = ((t.row_end - t.row_begin) + v.sub - 1) / v.sub;
    const int r_begin = t.row_begin + piece * len, r_end = min(t.row_end, r_begin + len);
    const int sub = threadIdx.x % LPR, rs = threadIdx.x / LPR;
    const int cofs = sub * CPL;
    const size_t pofs = (size_t)panel * v.n * KS;
    T b[CPL];
#pragma unroll
    for (int q = 0; q < CPL; q++) b[q] = (T)st.b[panel * KS + cofs + q];
    const T* __restrict__ R = v.r_next + pofs;
    T* __restrict__ Pp = v.p + pofs;
    for (int r0 = r_begin + rs; r0 < r_end; r0 += U * RPI) {
        T rv[U][CPL], pv[U][CPL];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int r = r0 + u * RPI;
            if (r < r_end) {
                load_lane(R + (size_t)r * KS + cofs, rv[u]);
                load_lane(Pp + (size_t)r * KS + cofs, pv[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int r = r0 + u * RPI;
            if (r < r_end) {
#pragma unroll
                for (int q = 0; q < CPL; q++) pv[u][q] = rv[u][q] + b[q] * pv[u][q];
                store_lane(Pp + (size_t)r * KS + cofs, pv[u]);
            }
        }
    }
}

// Coefficients of a window of `count` iterations, one thread per (shift,
// column), one CTA per panel.  With A_i = a_{s,i} + b_{s,i} A_{i+1} (A = 0
// after the last) and B_i = b_{s,i} B_{i+1} (B = 1 at the last):
//   x_s  += sum_i (zeta_i A_i) r_i + (b_start A_first) p_s
//   p_s   = sum_i (zeta_i B_i) r_i + (b_start B_first) p_s
// All factors are non-negative, and the residuals are orthogonal, so no term
// of x_s exceeds x_s itself.  An inactive iteration has zeta = a = b = 0.
template <typename T>
__global__ void __launch_bounds__(VNE_THREADS) k_cg_coefs(CgFlush<T> f, CgState st, int ks) {
    __shared__ int s_live;
    if (threadIdx.x == 0) s_live = f.first ? (1 << st.nshift) - 1 : 0;
    __syncthreads();
    const int panel = f.panel_base + blockIdx.x;
    for (int idx = threadIdx.x; idx < st.nshift * ks; idx += VNE_THREADS) {
        const int s = idx / ks, c = panel * ks + idx % ks;
        const size_t o = (size_t)s * st.K + c;
        double A = 0.0, B = 1.0;
        bool live = false;
        for (int i = f.count - 1; i >= 0; i--) {
            const size_t h = ((size_t)i * st.nshift + s) * st.K + c;
            const double z = st.hz[h], a = st.ha[h], b = st.hb[h];
            live = live || z != 0.0 || a != 0.0;
            A = fma(b, A, a);
            if (i != f.count - 1) B *= b;
            T* out = f.coef + ((size_t)i * st.nshift + s) * 2 * st.K + c;
            out[0] = (T)(z * A);
            out[st.K] = (T)(z * B);
        }
        const double bs = st.bstart[o];
        T* out = f.coef_p + (size_t)s * 2 * st.K + c;
        out[0] = (T)(bs * A);
        out[st.K] = (T)(bs * B);
        st.bstart[o] = st.hb[((size_t)(f.count - 1) * st.nshift + s) * st.K + c];
        if (live) atomicOr(&s_live, 1 << s);
    }
    __syncthreads();
    if (threadIdx.x == 0) f.live[panel] = s_live;
}

// x_s and p_s of the live shifts from a window of residuals: four shifts at a
// time in registers, two rows per lane (a coefficient read from shared memory
// serves both), every residual of the window read once per four live shifts.
// Bound by HBM: (count + 4 per live shift) vectors; FP64 by its multiply-adds
// (two per element, residual and live shift).
constexpr int kFlushShifts = 4;

template <typename T, int KS>
__global__ void __launch_bounds__(VNE_THREADS) k_cg_flush(CgFlush<T> f) {
    constexpr int CPL = LaneVec<T>::CPL;
    constexpr int LPR = KS / CPL;
    constexpr int RPI = VNE_THREADS / LPR;
    constexpr int G = kFlushShifts;
    extern __shared__ __align__(16) unsigned char fl_smem[];
    T* cf = reinterpret_cast<T*>(fl_smem);       // [count][G][2][KS]
    __shared__ __align__(16) T cp[G][2][KS];
    const int chunks = (f.n + f.rows - 1) / f.rows;
    const int panel = f.panel_base + blockIdx.x / chunks, chunk = blockIdx.x % chunks;
    const int r_begin = chunk * f.rows, r_end = min(f.n, r_begin + f.rows);
    const int sub = threadIdx.x % LPR, rs = threadIdx.x / LPR, cofs = sub * CPL;
    const size_t pofs = (size_t)panel * f.n * KS;
    unsigned live = (unsigned)f.live[panel];
    while (live) {
        int sh[G], ns = 0;
#pragma unroll
        for (int g = 0; g < G; g++) {
            sh[g] = -1;
            if (live) {
                sh[g] = __ffs(live) - 1;
                live &= live - 1;
                ns++;
            }
        }
        __syncthreads();  // the previous group's coefficients are no longer read
        for (int idx = threadIdx.x; idx < f.count * G * 2 * KS; idx += VNE_THREADS) {
            const int cc = idx % KS, w = (idx / KS) & 1, g = (idx / (2 * KS)) % G, i = idx / (2 * KS * G);
            const int s = sh[g];
            cf[idx] = s >= 0 ? f.coef[(((size_t)i * f.nshift + s) * 2 + w) * f.K + panel * KS + cc] : (T)0;
        }
        for (int idx = threadIdx.x; idx < G * 2 * KS; idx += VNE_THREADS) {
            const int cc = idx % KS, w = (idx / KS) & 1, g = idx / (2 * KS);
            cp[g][w][cc] = sh[g] >= 0 ? f.coef_p[((size_t)sh[g] * 2 + w) * f.K + panel * KS + cc] : (T)0;
        }
        __syncthreads();
        for (int r0 = r_begin + rs; r0 < r_end; r0 += 2 * RPI) {
            const bool two = r0 + RPI < r_end;
            const size_t o0 = pofs + (size_t)r0 * KS + cofs, o1 = two ? o0 + (size_t)RPI * KS : o0;
            T x[G][2][CPL], p[G][2][CPL];
#pragma unroll
            for (int g = 0; g < G; g++) {
                if (g < ns && !f.first) {
                    load_lane_stream(f.x[sh[g]] + o0, x[g][0]);
                    load_lane_stream(f.x[sh[g]] + o1, x[g][1]);
                    load_lane_stream(f.ps[sh[g]] + o0, p[g][0]);
                    load_lane_stream(f.ps[sh[g]] + o1, p[g][1]);
                } else {
#pragma unroll
                    for (int u = 0; u < 2; u++)
#pragma unroll
                        for (int q = 0; q < CPL; q++) x[g][u][q] = p[g][u][q] = (T)0;
                }
#pragma unroll
                for (int u = 0; u < 2; u++)
#pragma unroll
                    for (int q = 0; q < CPL; q++) {
                        x[g][u][q] += cp[g][0][cofs + q] * p[g][u][q];
                        p[g][u][q] *= cp[g][1][cofs + q];
                    }
            }
            int slot = f.slot0;
#pragma unroll 2
            for (int i = 0; i < f.count; i++) {
                T a[2][CPL];
                load_lane_stream(f.r + (size_t)slot * f.slot_stride + o0, a[0]);
                load_lane_stream(f.r + (size_t)slot * f.slot_stride + o1, a[1]);
                if (++slot == f.slots) slot = 0;
                const T* ci = cf + (size_t)i * G * 2 * KS + cofs;
#pragma unroll
                for (int g = 0; g < G; g++) {
                    if (g < ns) {
                        T cx[CPL], cq[CPL];
                        load_lane(ci + (g * 2) * KS, cx);
                        load_lane(ci + (g * 2 + 1) * KS, cq);
#pragma unroll
                        for (int u = 0; u < 2; u++)
#pragma unroll
                            for (int q = 0; q < CPL; q++) {
                                x[g][u][q] += cx[q] * a[u][q];
                                p[g][u][q] += cq[q] * a[u][q];
                            }
                    }
                }
            }
#pragma unroll
            for (int g = 0; g < G; g++)
                if (g < ns) {
                    store_lane_stream(f.x[sh[g]] + o0, x[g][0]);
                    if (two) store_lane_stream(f.x[sh[g]] + o1, x[g][1]);
                    if (!f.last) {
                        store_lane_stream(f.ps[sh[g]] + o0, p[g][0]);
                        if (two) store_lane_stream(f.ps[sh[g]] + o1, p[g][1]);
                    }
                }
        }
    }
}

// Per-column Cholesky of the column-scaled Gram matrix in pole order.  A
// column whose pivot (squared relative remainder) is <= drop is dependent on
// the kept ones and is dropped.  Returns the kept count; R (upper, kept
// columns) and D (column scales) are outputs.
__device__ int gram_cholesky(const double* Mg, int nb, int K, int c, double drop, double (&R)[kMaxBasis][kMaxBasis],
                             double (&D)[kMaxBasis], int (&keep)[kMaxBasis]) {
    for (int a = 0; a < nb; a++) {
        double maa = Mg[((size_t)a * nb + a) * K + c];
        D[a] = maa > 0.0 ? 1.0 / sqrt(maa) : 0.0;
    }
    int r = 0;
    for (int a = 0; a < nb; a++) {
        if (D[a] == 0.0) continue;
        double col[kMaxBasis];
        double s = 1.0;
        for (int i = 0; i < r; i++) {
            double v = Mg[((size_t)keep[i] * nb + a) * K + c] * D[keep[i]] * D[a];
            for (int l = 0; l < i; l++) v -= R[l][i] * col[l];
            col[i] = v / R[i][i];
            s -= col[i] * col[i];
        }
        if (s <= drop) continue;
        for (int i = 0; i < r; i++) R[i][r] = col[i];
        R[r][r] = sqrt(s);
        keep[r++] = a;
    }
    return r;
}

// Pass 1: X[c] = P D R^{-1} (nb x nb, rows by original column, zero for
// dropped ones) so that W X has orthonormal columns up to rounding; the
// second pass re-orthonormalises W X from its own Gram matrix (Cholesky-QR2).
__global__ void k_rational_pass1(const double* Mg, int nb, int K, double drop, double* X) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= K) return;
    double R[kMaxBasis][kMaxBasis], D[kMaxBasis];
    int keep[kMaxBasis];
    const int r = gram_cholesky(Mg, nb, K, c, drop, R, D, keep);
    for (int i = 0; i < nb * nb; i++) X[(size_t)i * K + c] = 0.0;
    for (int j = 0; j < r; j++) {
        // column j of R^{-1} (back substitution)
        double x[kMaxBasis];
        x[j] = 1.0 / R[j][j];
        for (int i = j - 1; i >= 0; i--) {
            double v = 0.0;
            for (int l = i + 1; l <= j; l++) v += R[i][l] * x[l];
            x[i] = -v / R[i][i];
        }
        for (int i = 0; i <= j; i++) X[((size_t)keep[i] * nb + j) * K + c] = D[keep[i]] * x[i];
    }
}

// Pass 2: orthonormalise the transformed basis, project A, diagonalise by
// Jacobi, psi = ||c||^2 sum_k z_{1k}^2 f(mu_k).  c2 = ||c||^2.  A warp per
// column with the matrices in shared memory (one thread per column before, its
// arrays in local memory: 2.8 ms for 12 columns of 11 vectors, 0.34 now):
// lanes share the rows of the triangular solves and products, and a Jacobi
// sweep takes its rotations in rounds of disjoint pairs (the circle method), a
// lane per rotation angle, since the angle's divisions and square roots are
// what a rotation costs.
__global__ void __launch_bounds__(32) k_rational_pass2(const double* Mg, const double* Kg, const double* c2v, int nb,
                                                       int K, double drop, double* psi, int* rank_out) {
    constexpr int N = kMaxBasis, LD = kMaxBasis + 1;
    __shared__ double R[N * LD], Ri[N * LD], T1[N * LD], Am[N * LD], Z[N * LD];
    __shared__ double D[N], s_c[N / 2], s_s[N / 2];
    __shared__ int keep[N], s_p[N / 2], s_q[N / 2];
    const int c = blockIdx.x, lane = threadIdx.x;
    const double c2 = c2v[c];
    if (!(c2 > 0.0)) {
        if (lane == 0) {
            psi[c] = 0.0;
            rank_out[c] = 0;
        }
        return;
    }
    if (lane < nb) {
        const double maa = Mg[((size_t)lane * nb + lane) * K + c];
        D[lane] = maa > 0.0 ? 1.0 / sqrt(maa) : 0.0;
    }
    __syncwarp();
    // Cholesky of the column-scaled Gram in basis order (gram_cholesky's rule):
    // lane i holds entry i of the new column
    int r = 0;
    for (int a = 0; a < nb; a++) {
        if (D[a] == 0.0) continue;
        double v = lane < r ? Mg[((size_t)keep[lane] * nb + a) * K + c] * D[keep[lane]] * D[a] : 0.0;
        double s = 1.0;
        for (int i = 0; i < r; i++) {
            const double ci = __shfl_sync(0xffffffffu, v, i) / R[i * LD + i];
            if (lane == i) v = ci;
            if (lane > i && lane < r) v -= R[i * LD + lane] * ci;
            s -= ci * ci;
        }
        if (s <= drop) continue;
        if (lane < r) R[lane * LD + r] = v;
        if (lane == 0) {
            R[r * LD + r] = sqrt(s);
            keep[r] = a;
        }
        r++;
        __syncwarp();
    }
    // R^{-1}, a lane per column
    if (lane < r) {
        for (int i = 0; i < r; i++) Ri[i * LD + lane] = 0.0;
        Ri[lane * LD + lane] = 1.0 / R[lane * LD + lane];
        for (int i = lane - 1; i >= 0; i--) {
            double v = 0.0;
            for (int l = i + 1; l <= lane; l++) v += R[i * LD + l] * Ri[l * LD + lane];
            Ri[i * LD + lane] = -v / R[i * LD + i];
        }
    }
    __syncwarp();
    // the scaled, symmetrised W^T A W on kept columns (in Z for now)
    for (int idx = lane; idx < r * r; idx += 32) {
        const int i = idx / r, l = idx % r, a = keep[i], b = keep[l];
        const double kab = 0.5 * (Kg[((size_t)a * nb + b) * K + c] + Kg[((size_t)b * nb + a) * K + c]);
        Z[i * LD + l] = kab * D[a] * D[b];
    }
    __syncwarp();
    for (int idx = lane; idx < r * r; idx += 32) {
        const int i = idx / r, j = idx % r;
        double v = 0.0;
        for (int l = 0; l <= j; l++) v += Z[i * LD + l] * Ri[l * LD + j];
        T1[i * LD + j] = v;
    }
    __syncwarp();
    for (int idx = lane; idx < r * r; idx += 32) {
        const int i = idx / r, j = idx % r;
        double v = 0.0;
        for (int l = 0; l <= i; l++) v += Ri[l * LD + i] * T1[l * LD + j];
        Am[i * LD + j] = v;
        Z[i * LD + j] = (i == j) ? 1.0 : 0.0;
    }
    __syncwarp();
    const int r2 = (r + 1) & ~1, half = r2 / 2;  // players of the circle method (an odd r sits one out)
    for (int sweep = 0; sweep < 30; sweep++) {
        double off = 0.0, tot = 0.0;
        for (int idx = lane; idx < r * r; idx += 32) {
            const double x = Am[(idx / r) * LD + idx % r];
            tot += x * x;
            if (idx / r != idx % r) off += x * x;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            off += __shfl_xor_sync(0xffffffffu, off, o);
            tot += __shfl_xor_sync(0xffffffffu, tot, o);
        }
        if (off <= 1e-30 * tot) break;
        for (int round = 0; round < r2 - 1; round++) {
            if (lane < half) {
                const int m = r2 - 1;
                int p = lane == 0 ? m : (round + lane) % m;
                int q = lane == 0 ? round : (round + m - lane) % m;
                if (p > q) {
                    const int x = p;
                    p = q;
                    q = x;
                }
                double cs = 1.0, sn = 0.0;
                if (q < r) {
                    const double apq = Am[p * LD + q];
                    if (apq != 0.0) {
                        const double theta = (Am[q * LD + q] - Am[p * LD + p]) / (2.0 * apq);
                        const double t = (theta >= 0.0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
                        cs = 1.0 / sqrt(t * t + 1.0);
                        sn = t * cs;
                    }
                }
                s_c[lane] = cs;
                s_s[lane] = sn;
                s_p[lane] = p;
                s_q[lane] = q;
            }
            __syncwarp();
            for (int idx = lane; idx < r * half; idx += 32) {  // columns of A and Z
                const int k = idx / half, h = idx % half, p = s_p[h], q = s_q[h];
                if (q >= r) continue;
                const double cs = s_c[h], sn = s_s[h];
                const double akp = Am[k * LD + p], akq = Am[k * LD + q];
                Am[k * LD + p] = cs * akp - sn * akq;
                Am[k * LD + q] = sn * akp + cs * akq;
                const double zkp = Z[k * LD + p], zkq = Z[k * LD + q];
                Z[k * LD + p] = cs * zkp - sn * zkq;
                Z[k * LD + q] = sn * zkp + cs * zkq;
            }
            __syncwarp();
            for (int idx = lane; idx < r * half; idx += 32) {  // rows of A
                const int k = idx % r, h = idx / r, p = s_p[h], q = s_q[h];
                if (q >= r) continue;
                const double cs = s_c[h], sn = s_s[h];
                const double apk = Am[p * LD + k], aqk = Am[q * LD + k];
                Am[p * LD + k] = cs * apk - sn * aqk;
                Am[q * LD + k] = sn * apk + cs * aqk;
            }
            __syncwarp();
        }
    }
    double s = 0.0;
    if (lane < r) s = Z[lane] * Z[lane] * f_ent(Am[lane * LD + lane]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
        psi[c] = c2 * s;
        rank_out[c] = r;
    }
}

template <typename T, int KS>
__global__ void __launch_bounds__(VNE_THREADS) k_cgs_scale(T* v, const double* orig2, const double* rem2,
                                                           double drop2, int n, int K, int tiles_per_panel,
                                                           const RowTile* tiles) {
    const int panel = blockIdx.x / tiles_per_panel, tile = blockIdx.x % tiles_per_panel;
    const RowTile t = tiles[tile];
    const int c = threadIdx.x % KS, rsub = threadIdx.x / KS;
    constexpr int RPI = VNE_THREADS / KS;
    const int col = panel * KS + c;
    const double r2 = rem2[col];
    const double s = (r2 > 0.0 && r2 > drop2 * orig2[col]) ? 1.0 / sqrt(r2) : 0.0;
    T* V = v + (size_t)panel * n * KS;
    for (int r = t.row_begin + rsub; r < t.row_end; r += RPI) V[(size_t)r * KS + c] = (T)(s * (double)V[(size_t)r * KS + c]);
}

template <typename T>
cudaError_t launch_cgs_scale(T* v, const double* orig2, const double* rem2, double drop, int n, int K, int ks,
                             int tiles_per_panel, const RowTile* tiles, cudaStream_t st) {
    dim3 grid((K / ks) * tiles_per_panel);
    const double d2 = drop * drop;
    if (ks == 4) k_cgs_scale<T, 4><<<grid, VNE_THREADS, 0, st>>>(v, orig2, rem2, d2, n, K, tiles_per_panel, tiles);
    else if (ks == 8) k_cgs_scale<T, 8><<<grid, VNE_THREADS, 0, st>>>(v, orig2, rem2, d2, n, K, tiles_per_panel, tiles);
    else if (ks == 16) k_cgs_scale<T, 16><<<grid, VNE_THREADS, 0, st>>>(v, orig2, rem2, d2, n, K, tiles_per_panel, tiles);
    else if (ks == 32) k_cgs_scale<T, 32><<<grid, VNE_THREADS, 0, st>>>(v, orig2, rem2, d2, n, K, tiles_per_panel, tiles);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}
template cudaError_t launch_cgs_scale<float>(float*, const double*, const double*, double, int, int, int, int,
                                             const RowTile*, cudaStream_t);
template cudaError_t launch_cgs_scale<double>(double*, const double*, const double*, double, int, int, int, int,
                                              const RowTile*, cudaStream_t);

// Per-column basis change: out_j = sum_i in_i X[i][j] (X per column, FP64,
// staged in shared memory in the data precision).
template <typename T, int KS>
__global__ void __launch_bounds__(VNE_THREADS) k_block_transform(BlockTransform<T> bt) {
    constexpr int RPI = VNE_THREADS / KS;
    const int panel = blockIdx.x / bt.tiles_per_panel, tile = blockIdx.x % bt.tiles_per_panel;
    const RowTile t = bt.tiles[tile];
    const int c = threadIdx.x % KS, rs = threadIdx.x / KS;
    const int col = panel * KS + c;
    extern __shared__ __align__(16) unsigned char bt_smem[];
    T(*sx)[KS] = reinterpret_cast<T(*)[KS]>(bt_smem);  // [nb * nb][KS]
    for (int idx = threadIdx.x; idx < bt.nb * bt.nb * KS; idx += VNE_THREADS) {
        const int e = idx / KS, cc = idx % KS;
        sx[e][cc] = (T)bt.X[(size_t)e * bt.K + panel * KS + cc];
    }
    __syncthreads();
    const size_t pofs = (size_t)panel * bt.n * KS;
    for (int r = t.row_begin + rs; r < t.row_end; r += RPI) {
        const size_t o = pofs + (size_t)r * KS + c;
        T v[kMaxBasis];
        for (int i = 0; i < bt.nb; i++) v[i] = bt.in[i][o];
        for (int j = 0; j < bt.nb; j++) {
            T acc = (T)0;
            for (int i = 0; i < bt.nb; i++) acc += v[i] * sx[i * bt.nb + j][c];
            bt.out[j][o] = acc;
        }
    }
    (void)col;
}

// ---------------------------------------------------------------------------
// Gram matrices W^T W and W^T (A W) per column in one pass over the vectors
// (a kernel per pair of vectors would read every vector about nb times).  A
// CTA takes a range of rows of one panel in tiles of kGramRows rows: all 2 nb
// vectors' tile rows go to shared memory, and each thread accumulates a
// fixed set of (pair, column) outputs; the outputs are split into groups of
// kGramOut so that a thread holds at most kGramPer of them.  Sums per tile in
// the data precision (16 rows, as the pairwise kernel), FP64 across tiles,
// FP64 fixed-order sum over the row ranges.
constexpr int kGramRows = 16;
constexpr int kGramPer = 16;
constexpr int kGramOut = VNE_THREADS * kGramPer;

template <typename T, int KS>
__global__ void __launch_bounds__(VNE_THREADS) k_multi_gram(MultiGram<T> g) {
    extern __shared__ __align__(16) unsigned char mg_smem[];
    T* sv = reinterpret_cast<T*>(mg_smem);  // [2 nb][kGramRows][KS]
    __shared__ unsigned char s_x[kGramOut / KS + 1], s_y[kGramOut / KS + 1];
    const int chunk = blockIdx.x, grp = blockIdx.y, panel = blockIdx.z;
    const int nb = g.nb, nu = nb * (nb + 1) / 2, npair = 2 * nu;
    const int o_begin = grp * kGramOut, o_end = min(npair * KS, o_begin + kGramOut);
    // pair -> (x vector, y vector) for this group's pairs; y >= nb is AW
    const int p_begin = o_begin / KS, p_end = (o_end + KS - 1) / KS;
    for (int pr = p_begin + threadIdx.x; pr < p_end; pr += VNE_THREADS) {
        const int half = pr >= nu, q = half ? pr - nu : pr;
        int a = 0, rem = q;
        while (rem >= nb - a) {
            rem -= nb - a;
            a++;
        }
        s_x[pr - p_begin] = (unsigned char)a;
        s_y[pr - p_begin] = (unsigned char)(a + rem + (half ? nb : 0));
    }
    const int rows_per = (g.n + g.chunks - 1) / g.chunks;
    const int r_begin = chunk * rows_per, r_end = min(g.n, r_begin + rows_per);
    const size_t pofs = (size_t)panel * g.n * KS;
    double acc[kGramPer];
#pragma unroll
    for (int j = 0; j < kGramPer; j++) acc[j] = 0.0;
    const int nvec = 2 * nb;
    for (int r0 = r_begin; r0 < r_end; r0 += kGramRows) {
        const int rows = min(kGramRows, r_end - r0);
        __syncthreads();
        for (int idx = threadIdx.x; idx < nvec * kGramRows * KS; idx += VNE_THREADS) {
            const int v = idx / (kGramRows * KS), e = idx % (kGramRows * KS), rr = e / KS;
            const T* src = v < nb ? g.w[v] : g.aw[v - nb];
            sv[idx] = rr < rows ? src[pofs + (size_t)(r0 + rr) * KS + (e % KS)] : (T)0;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kGramPer; j++) {
            const int o = o_begin + threadIdx.x + j * VNE_THREADS;
            if (o >= o_end) break;
            const int pr = o / KS, c = o % KS;
            const T* X = sv + (size_t)s_x[pr - p_begin] * kGramRows * KS + c;
            const T* Y = sv + (size_t)s_y[pr - p_begin] * kGramRows * KS + c;
            T t = (T)0;
#pragma unroll
            for (int rr = 0; rr < kGramRows; rr++) t += X[rr * KS] * Y[rr * KS];
            acc[j] += (double)t;
        }
    }
    const size_t gbase = (((size_t)panel * g.groups + grp) * g.chunks + chunk) * kGramOut;
#pragma unroll
    for (int j = 0; j < kGramPer; j++) {
        const int o = o_begin + threadIdx.x + j * VNE_THREADS;
        if (o < o_end) g.part[gbase + (o - o_begin)] = acc[j];
    }
}

// out[pair][panel * KS + c] = fixed-order sum over the row ranges
__global__ void k_multi_gram_reduce(const double* part, int panels, int groups, int chunks, int ks, int npair,
                                    double* out) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const int K = panels * ks;
    if (idx >= npair * K) return;
    const int pr = idx / K, col = idx % K, panel = col / ks, c = col % ks;
    const int o = pr * ks + c, grp = o / kGramOut, oo = o % kGramOut;
    double s = 0.0;
    for (int ch = 0; ch < chunks; ch++) s += part[(((size_t)panel * groups + grp) * chunks + ch) * kGramOut + oo];
    out[(size_t)pr * K + col] = s;
}

// Lanczos tridiagonal of A from the seed CG's scalars (the CG-Lanczos
// relation): with step lengths a_i and direction coefficients b_i of CG on
// A + s0 I, T_{i+1,i+1} = 1/a_i + b_{i-1}/a_{i-1} - s0 (no second term at
// i = 0) and T_{i+1,i+2} = sqrt(b_i)/a_i.  An off-diagonal at or below tau
// (the Lanczos breakdown threshold) is set to 0: the Krylov space is
// invariant there, and the rows after it are not used.  History rows
// [i][K], i < k.
__global__ void k_cg_tridiag(const double* ah, const double* bh, int K, int k, double s0, double tau,
                             double* diag, double* off) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= K) return;
    double prev = 0.0;  // b_{i-1} / a_{i-1}
    for (int i = 0; i < k; i++) {
        const double a = ah[(size_t)i * K + c], b = bh[(size_t)i * K + c];
        const double t = sqrt(b) / a;
        diag[(size_t)i * K + c] = 1.0 / a + prev - s0;
        off[(size_t)i * K + c] = t > tau ? t : 0.0;
        prev = b / a;
    }
}

// Full [nb][nb][K] Gram layout from its upper triangle, pairs (a <= b)
// numbered row by row.
__global__ void k_gram_mirror(const double* uniq, int nb, int K, double* full) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)nb * nb * K) return;
    const int c = (int)(idx % K), b = (int)((idx / K) % nb), a = (int)(idx / ((size_t)K * nb));
    const int lo = a < b ? a : b, hi = a < b ? b : a;
    const size_t pr = (size_t)lo * nb - (size_t)lo * (lo - 1) / 2 + (hi - lo);
    full[idx] = uniq[pr * K + c];
}

// ---------------------------------------------------------------------------

#define VNE_KS_SWITCH(T, ks, CALL)                                        \
    do {                                                                  \
        if ((ks) == 4) { constexpr int KS = 4; CALL; }                    \
        else if ((ks) == 8) { constexpr int KS = 8; CALL; }               \
        else if ((ks) == 16) { constexpr int KS = 16; CALL; }             \
        else if ((ks) == 32) { constexpr int KS = 32; CALL; }             \
        else return cudaErrorInvalidValue;                                \
    } while (0)

template <typename T, int KS>
cudaError_t cg_update_ks(CgVectors<T> v, const CgState& st, int panels, int wi, int it, cudaStream_t s) {
    constexpr int RPI = VNE_THREADS / (KS / LaneVec<T>::CPL);
    // three row tiles per CTA where that leaves the SMs more than one wave of four
    // (n = 10^6, 22 columns, per launch: 62 us with one, 57 with two, 53 with
    // three, 59 with four, 54 with five)
    v.group = sizeof(T) == 4 && (int64_t)panels * v.tiles_per_panel >= 16 * (int64_t)v.sm_count ? 3 : 1;
    const int ctas = panels * ((v.tiles_per_panel + v.group - 1) / v.group);
    if constexpr (sizeof(T) == 8) {
        // runs of 16 rows per thread in the largest tile; clusters pay while
        // the tiles alone do not fill the SMs twice
        const int runs = (v.max_tile_rows + 16 * RPI - 1) / (16 * RPI);
        if (runs > 1 && runs <= 8 && ctas < 2 * v.sm_count) {
            int size = 1;
            while (size < runs) size *= 2;
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3(ctas * size);
            cfg.blockDim = dim3(VNE_THREADS);
            cfg.stream = s;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = size;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            return cudaLaunchKernelEx(&cfg, k_cg_update<T, KS, true>, v, st, wi, it);
        }
    }
    k_cg_update<T, KS, false><<<ctas, VNE_THREADS, 0, s>>>(v, st, wi, it);
    return cudaSuccess;
}
template <typename T>
cudaError_t launch_cg_update(const CgVectors<T>& v, const CgState& st, int ks, int panels, int window_index,
                             int iteration, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    VNE_KS_SWITCH(T, ks, (e = cg_update_ks<T, KS>(v, st, panels, window_index, iteration, s)));
    return e != cudaSuccess ? e : cudaGetLastError();
}
template <typename T, int KS>
cudaError_t cg_flush_ks(CgFlush<T> f, cudaStream_t s) {
    // 1024 rows per CTA, 256 while that leaves SMs without one
    f.rows = (int64_t)f.panels * f.n >= 4 * 1024 * (int64_t)f.sm_count ? 1024 : 256;
    const size_t smem = (size_t)f.count * kFlushShifts * 2 * KS * sizeof(T);
    if (smem + 4096 > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_cg_flush<T, KS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
    }
    k_cg_flush<T, KS><<<f.panels * ((f.n + f.rows - 1) / f.rows), VNE_THREADS, smem, s>>>(f);
    return cudaSuccess;
}
template <typename T>
cudaError_t launch_cg_flush(const CgFlush<T>& f, const CgState& st, int ks, cudaStream_t s) {
    if (f.count <= 0) return cudaSuccess;
    k_cg_coefs<T><<<f.panels, VNE_THREADS, 0, s>>>(f, st, ks);
    cudaError_t e = cudaSuccess;
    VNE_KS_SWITCH(T, ks, (e = cg_flush_ks<T, KS>(f, s)));
    return e != cudaSuccess ? e : cudaGetLastError();
}
template <typename T>
cudaError_t launch_cg_direction(const CgVectors<T>& v, const CgState& st, int ks, int panels, cudaStream_t s) {
    VNE_KS_SWITCH(T, ks, (k_cg_direction<T, KS><<<panels * v.tiles_per_panel * v.sub, VNE_THREADS, 0, s>>>(v, st)));
    return cudaGetLastError();
}
template <typename T, int KS>
cudaError_t multi_gram_ks(const MultiGram<T>& g, cudaStream_t s) {
    const size_t smem = (size_t)2 * g.nb * kGramRows * KS * sizeof(T);
    // the static pair tables (about 2 KB) count against the 48 KB default too
    if (smem + 4096 > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_multi_gram<T, KS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
    }
    k_multi_gram<T, KS><<<dim3(g.chunks, g.groups, g.panels), VNE_THREADS, smem, s>>>(g);
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_multi_gram(MultiGram<T> g, double* out, cudaStream_t s) {
    if (g.nb < 1 || g.nb > 24) return cudaErrorInvalidValue;
    const int npair = g.nb * (g.nb + 1);
    g.groups = (npair * g.ks + kGramOut - 1) / kGramOut;
    cudaError_t e = cudaSuccess;
    VNE_KS_SWITCH(T, g.ks, (e = multi_gram_ks<T, KS>(g, s)));
    if (e != cudaSuccess) return e;
    const int K = g.panels * g.ks;
    k_multi_gram_reduce<<<(npair * K + 255) / 256, 256, 0, s>>>(g.part, g.panels, g.groups, g.chunks, g.ks, npair,
                                                                 out);
    return cudaGetLastError();
}
template cudaError_t launch_multi_gram<float>(MultiGram<float>, double*, cudaStream_t);
template cudaError_t launch_multi_gram<double>(MultiGram<double>, double*, cudaStream_t);

cudaError_t launch_cg_tridiag(const double* ah, const double* bh, int K, int k, double s0, double tau, double* diag,
                              double* off, cudaStream_t s) {
    if (k <= 0) return cudaSuccess;
    k_cg_tridiag<<<(K + 63) / 64, 64, 0, s>>>(ah, bh, K, k, s0, tau, diag, off);
    return cudaGetLastError();
}
cudaError_t launch_gram_mirror(const double* uniq, int nb, int K, double* full, cudaStream_t s) {
    const size_t total = (size_t)nb * nb * K;
    if (total == 0) return cudaSuccess;
    k_gram_mirror<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(uniq, nb, K, full);
    return cudaGetLastError();
}
cudaError_t launch_rational_pass1(const double* M, int nb, int K, double drop, double* X, cudaStream_t s) {
    if (nb > kMaxBasis) return cudaErrorInvalidValue;
    k_rational_pass1<<<(K + 31) / 32, 32, 0, s>>>(M, nb, K, drop, X);
    return cudaGetLastError();
}
cudaError_t launch_rational_pass2(const double* M, const double* Kmat, const double* c2, int nb, int K, double drop,
                                  double* psi, int* rank, cudaStream_t s) {
    if (nb > kMaxBasis) return cudaErrorInvalidValue;
    k_rational_pass2<<<K, 32, 0, s>>>(M, Kmat, c2, nb, K, drop, psi, rank);
    return cudaGetLastError();
}
// the basis-change matrix (nb^2 x KS values) lives in dynamic shared memory,
// beyond 48 KB for the largest bases
template <typename T, int KS>
cudaError_t block_transform_ks(const BlockTransform<T>& bt, int panels, size_t smem, cudaStream_t s) {
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_block_transform<T, KS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
    }
    k_block_transform<T, KS><<<panels * bt.tiles_per_panel, VNE_THREADS, smem, s>>>(bt);
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_block_transform(const BlockTransform<T>& bt, int ks, int panels, cudaStream_t s) {
    if (bt.nb > kMaxBasis) return cudaErrorInvalidValue;
    const size_t smem = (size_t)bt.nb * bt.nb * ks * sizeof(T);
    cudaError_t e = cudaSuccess;
    VNE_KS_SWITCH(T, ks, (e = block_transform_ks<T, KS>(bt, panels, smem, s)));
    return e != cudaSuccess ? e : cudaGetLastError();
}

template cudaError_t launch_cg_update<float>(const CgVectors<float>&, const CgState&, int, int, int, int, cudaStream_t);
template cudaError_t launch_cg_update<double>(const CgVectors<double>&, const CgState&, int, int, int, int,
                                              cudaStream_t);
template cudaError_t launch_cg_flush<float>(const CgFlush<float>&, const CgState&, int, cudaStream_t);
template cudaError_t launch_cg_flush<double>(const CgFlush<double>&, const CgState&, int, cudaStream_t);
template cudaError_t launch_cg_direction<float>(const CgVectors<float>&, const CgState&, int, int, cudaStream_t);
template cudaError_t launch_cg_direction<double>(const CgVectors<double>&, const CgState&, int, int, cudaStream_t);
template cudaError_t launch_block_transform<float>(const BlockTransform<float>&, int, int, cudaStream_t);
template cudaError_t launch_block_transform<double>(const BlockTransform<double>&, int, int, cudaStream_t);

}  // namespace vne
