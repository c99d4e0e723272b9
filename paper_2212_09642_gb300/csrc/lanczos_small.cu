// Lanczos recurrence of a small graph in one launch: a CTA per probe column.
//
// Columns are independent recurrences, so a graph whose vectors fit an SM's
// shared memory needs no communication between CTAs at all: the CTA keeps w_j
// and u (which overwrites w_{j-1}) in shared memory, gathers from there, and
// runs every step of the block.  The multi-CTA kernels spend two launches per
// step (nine with full reorthogonalisation), each a chain of launch, dependent
// loads, FP64 reductions and a last-CTA sum: 6 to 7 us per launch for a graph of
// 700 nodes whose arithmetic takes a fraction of one.  Here a step is a pass
// over the CTA's rows and two block reductions.
//
// What bounds it: without reorthogonalisation the gathers (nnz per column and
// step, indices from L1, values from shared memory) and 3.5 us per step of
// barriers, reductions and FP64 scalars; with it the FP64 port of the SM (4 j n
// multiply-adds at step j, 1.7 per cycle), which is why the rule that picks this
// kernel (small_lanczos_wins, with both sides' times) weighs K columns on K SMs
// against all columns on all SMs.  1024 threads, since one CTA has to hide its
// SM's latencies, and the step's scalars in warp 0 only (512 threads with the
// scalars in every warp took 0.47 against 0.30 ms for n = 5,000, one column, 20
// steps).  Only the two forms the rule picks are built: FP32
// without reorthogonalisation and FP64 with it.
#include "common.cuh"
#include "kernels.h"

namespace vne {

namespace {

constexpr int kSmallThreads = 1024;
constexpr int kSmallWarps = kSmallThreads / 32;

// Sum of one value per thread, fixed order; the result is valid in warp 0 only
// (an FP64 operation of all 32 warps holds the port for 32 x 16 cycles, so the
// scalars that follow are warp 0's too).  `pre`: 2^pre lanes are added in the
// data precision first, as far as FP32 sums of 16 products allow; a thread's own
// rows are one FP32 sum (up to 25 at the largest n that small_lanczos_wins
// admits, and up to eight long rows more in the step, each on lane 0).  Then
// 128 threads, a warp per sub-partition, add the rest in FP64, a shuffle tree and
// the four warps in order.  Contains two barriers.
template <typename T>
__device__ __forceinline__ double block_sum(T x, int pre, T* s_part, double* s_red) {
    for (int k = 0; k < pre; k++) x += __shfl_xor_sync(0xffffffffu, x, 1 << k);
    if ((threadIdx.x & ((1 << pre) - 1)) == 0) s_part[threadIdx.x >> pre] = x;
    __syncthreads();
    if (threadIdx.x < 128) {
        double t = 0.0;
        for (int i = threadIdx.x; i < (kSmallThreads >> pre); i += 128) t += (double)s_part[i];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = t;
    }
    __syncthreads();
    return threadIdx.x < 32 ? (s_red[0] + s_red[1]) + (s_red[2] + s_red[3]) : 0.0;
}

}  // namespace

template <typename T, bool VALUED, bool REORTH>  // REORTH: FP64 (its inner products are summed in T)
__global__ void __launch_bounds__(kSmallThreads, 1) k_lanczos_small(SmallLanczos<T> p) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    T* w = reinterpret_cast<T*>(sm_raw);  // w_j
    T* u = w + p.n;                       // w_{j-1}, then u, then w_{j+1}
    __shared__ T s_part[kSmallThreads];
    // scalars of the step, written by warp 0: alpha_j sigma_j, sigma_j and
    // beta_{j-1} sigma_{j-1} in the data precision; breakdown flag
    __shared__ T s_ta, s_ts, s_tc;
    __shared__ int s_stop;
    __shared__ double s_red[4], s_sig2[REORTH ? kSmallMaxSteps : 1];
    __shared__ T s_cf[REORTH ? kSmallMaxSteps : 1];
    const int c = blockIdx.x, n = p.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const size_t pofs = (size_t)(c / p.ks) * n * p.ks + c % p.ks;  // this column in the panel-major block
    for (int r = tid; r < n; r += kSmallThreads) w[r] = p.w1[pofs + (size_t)r * p.ks];
    const int rows_per = (n + kSmallThreads - 1) / kSmallThreads;
    const int pre = sizeof(T) == 8 ? 0 : (rows_per <= 2 ? 3 : (rows_per <= 4 ? 2 : (rows_per <= 8 ? 1 : 0)));
    double sig = p.sigma[c], cprev = 0.0;  // sigma_j, beta_{j-1} sigma_{j-1} (warp 0)
    if (tid == 0) {
        s_ts = (T)sig;
        s_tc = (T)0;
    }
    __syncthreads();
    for (int j = 1; j <= p.m; j++) {
        const size_t o = (size_t)(j - 1) * p.SK + c;
        T* basis = REORTH ? p.basis + ((size_t)c * p.m) * n : nullptr;  // this column's w_1 .. w_m
        if (REORTH) {
            for (int r = tid; r < n; r += kSmallThreads) basis[(size_t)(j - 1) * n + r] = w[r];
            if (tid == 0) s_sig2[j - 1] = sig * sig;
        }
        // u = sigma_j M w_j - beta_{j-1} sigma_{j-1} w_{j-1}, a thread per row;
        // rows longer than kSmallLongRow by whole warps afterwards
        const T ts = s_ts, tc = s_tc;
        T dot = (T)0;
        auto finish = [&](int r, T acc, int deg) {
            const T x = w[r];
            const T ax = VALUED ? acc : ((T)deg * x - acc);
            T v = ts * ax;
            if (j > 1) v -= tc * u[r];
            u[r] = v;
            dot += x * v;
        };
        for (int r = tid; r < n; r += kSmallThreads) {
            const int kb = p.rowptr[r], ke = p.rowptr[r + 1];
            if (ke - kb > kSmallLongRow) continue;
            T acc = (T)0;
            int k = kb;
            for (; k + 4 <= ke; k += 4) {
                int cc[4];
                T a[4];
#pragma unroll
                for (int q = 0; q < 4; q++) cc[q] = __ldg(p.col + k + q);
#pragma unroll
                for (int q = 0; q < 4; q++) a[q] = w[cc[q]];
                if (VALUED) {
#pragma unroll
                    for (int q = 0; q < 4; q++) acc += __ldg(p.vals + k + q) * a[q];
                } else {
                    acc += (a[0] + a[1]) + (a[2] + a[3]);
                }
            }
            for (; k < ke; k++) acc += VALUED ? __ldg(p.vals + k) * w[__ldg(p.col + k)] : w[__ldg(p.col + k)];
            finish(r, acc, ke - kb);
        }
        for (int i = warp; i < p.nlong; i += kSmallWarps) {
            const int r = p.long_rows[i], kb = p.rowptr[r], ke = p.rowptr[r + 1];
            T acc = (T)0;
            for (int k = kb + lane; k < ke; k += 32)
                acc += VALUED ? __ldg(p.vals + k) * w[__ldg(p.col + k)] : w[__ldg(p.col + k)];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if (lane == 0) finish(r, acc, ke - kb);
        }
        double alpha = block_sum<T>(dot, pre, s_part, s_red);
        if (warp == 0) {
            alpha *= sig;
            if (lane == 0) s_ta = (T)(alpha * sig);
        }
        __syncthreads();
        // w_{j+1} = u - alpha_j sigma_j w_j
        const T ta = s_ta;
        T nrm = (T)0;
        for (int r = tid; r < n; r += kSmallThreads) {
            const T v = u[r] - ta * w[r];
            u[r] = v;
            if (!REORTH) nrm += v * v;
        }
        if (REORTH) __syncthreads();
        if (REORTH) {
            // classical Gram-Schmidt twice against w_1 .. w_j: a warp per inner
            // product, then a thread per row
            for (int pass = 0; pass < 2; pass++) {
                for (int i = warp; i < j; i += kSmallWarps) {
                    const T* b = basis + (size_t)i * n;
                    T a0 = (T)0, a1 = (T)0, a2 = (T)0, a3 = (T)0;
                    int r = lane;
                    for (; r + 96 < n; r += 128) {
                        const T b0 = b[r], b1 = b[r + 32], b2 = b[r + 64], b3 = b[r + 96];
                        a0 += b0 * u[r];
                        a1 += b1 * u[r + 32];
                        a2 += b2 * u[r + 64];
                        a3 += b3 * u[r + 96];
                    }
                    for (; r < n; r += 32) a0 += b[r] * u[r];
                    double s = (double)((a0 + a1) + (a2 + a3));
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
                    if (lane == 0) s_cf[i] = (T)(s_sig2[i] * s);
                }
                __syncthreads();
                for (int r = tid; r < n; r += kSmallThreads) {
                    T v = u[r];
                    const T* b = basis + r;
                    int i = 0;
                    for (; i + 4 <= j; i += 4) {
                        const T b0 = b[(size_t)i * n], b1 = b[(size_t)(i + 1) * n], b2 = b[(size_t)(i + 2) * n],
                                b3 = b[(size_t)(i + 3) * n];
                        v -= s_cf[i] * b0;
                        v -= s_cf[i + 1] * b1;
                        v -= s_cf[i + 2] * b2;
                        v -= s_cf[i + 3] * b3;
                    }
                    for (; i < j; i++) v -= s_cf[i] * b[(size_t)i * n];
                    u[r] = v;
                }
                __syncthreads();
            }
            for (int r = tid; r < n; r += kSmallThreads) nrm += u[r] * u[r];
        }
        const double nrm2 = block_sum<T>(nrm, pre, s_part, s_red);
        if (warp == 0) {
            const double beta = sqrt(nrm2);
            const bool stop = !(beta > p.tau) || sig == 0.0;  // breakdown: the column is done
            const double snext = stop ? 0.0 : 1.0 / beta;
            cprev = beta * sig;
            if (lane == 0) {
                p.alpha[o] = alpha;
                p.beta[o] = stop ? 0.0 : beta;
                p.sigma[o + p.SK] = snext;
                s_ts = (T)snext;
                s_tc = (T)cprev;
                s_stop = stop;
            }
            sig = snext;
        }
        __syncthreads();
        if (s_stop) break;  // the later rows of alpha, beta and sigma are zero already
        T* t = w;
        w = u;
        u = t;
    }
}

size_t small_lanczos_smem(int n, bool fp64) { return (size_t)2 * n * (fp64 ? 8 : 4); }

template <typename T>
cudaError_t launch_lanczos_small(const SmallLanczos<T>& p, int cols, bool reorth, cudaStream_t st) {
    if (cols <= 0) return cudaSuccess;
    if (p.m > kSmallMaxSteps) return cudaErrorInvalidValue;
    const int smem = (int)small_lanczos_smem(p.n, sizeof(T) == 8);
    auto go = [&](auto kernel) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        kernel<<<cols, kSmallThreads, smem, st>>>(p);
        return cudaGetLastError();
    };
    constexpr bool R = sizeof(T) == 8;
    if (reorth != R) return cudaErrorInvalidValue;
    return p.vals ? go(k_lanczos_small<T, true, R>) : go(k_lanczos_small<T, false, R>);
}
template cudaError_t launch_lanczos_small<float>(const SmallLanczos<float>&, int, bool, cudaStream_t);
template cudaError_t launch_lanczos_small<double>(const SmallLanczos<double>&, int, bool, cudaStream_t);

}  // namespace vne
