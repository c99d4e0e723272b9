// Column sums of a CTA and their fixed-order combination across CTAs (not
// part of the public ABI).
//
// The FP64 additions of these tails are what they cost: GB300 issues one FP64
// instruction per warp and sub-partition in about 64 cycles whatever its
// independence, so a chain of 64 additions by KS threads alone takes 2 us and
// a butterfly that adds every column in every lane four times the slots of one
// that halves the columns a lane keeps at each stage.
#pragma once
#include "common.cuh"

namespace vne {

// Sum acc[] (CPL consecutive columns per lane, LPR = KS / CPL lanes per row,
// columns (lane % LPR) * CPL ..) over the CTA's VNE_THREADS threads.  Threads
// c < KS return column c's sum in tot (fixed order: lanes by a reduce-scatter
// tree, then warps in order).  Contains one barrier.
template <int KS, int CPL>
__device__ __forceinline__ void cta_colsum(double (&acc)[CPL], double (*red)[KS], double& tot) {
    constexpr int LPR = KS / CPL;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int col = (lane % LPR) * CPL;
    int width = CPL;  // compile-time after unrolling
#pragma unroll
    for (int off = LPR; off < 32; off <<= 1) {
        if (width > 1) {
            const int half = width / 2;
            const bool up = (lane & off) != 0;
#pragma unroll
            for (int i = 0; i < CPL / 2; i++)
                if (i < half) {
                    const double send = up ? acc[i] : acc[half + i];
                    const double keep = up ? acc[half + i] : acc[i];
                    acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
                }
            if (up) col += half;
            width = half;
        } else {
            acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], off);
        }
    }
    if (lane < KS) red[warp][col] = acc[0];
    __syncthreads();
    tot = 0.0;
    if (threadIdx.x < KS) {
#pragma unroll
        for (int w = 0; w < VNE_WARPS; w++) tot += red[w][threadIdx.x];
    }
}

// The same sum with one thread per column adding the rows' partials in row
// order.  FP64 conjugate gradients keep this order (with the serial order of
// last_cta_reduce): over hundreds of iterations the recurrence amplifies a
// change of rounding until a shift's iteration count moves by one.
template <int KS, int CPL>
__device__ __forceinline__ void cta_colsum_serial(const double (&acc)[CPL], double (*red)[KS], double& tot) {
    constexpr int LPR = KS / CPL, RPI = VNE_THREADS / LPR;
    const int sub = threadIdx.x % LPR, rs = threadIdx.x / LPR;
#pragma unroll
    for (int q = 0; q < CPL; q++) red[rs][sub * CPL + q] = acc[q];
    __syncthreads();
    tot = 0.0;
    if (threadIdx.x < KS)
        for (int q = 0; q < RPI; q++) tot += red[q][threadIdx.x];
}

// Fixed-order cross-CTA reduction: every CTA has written W partial values at
// part[(panel * nparts + idx) * W + c] and calls this; the CTA that arrives
// last for the counter sums the `count` partials starting at `begin` in a
// fixed order and returns true with the totals in s_out[0..W).  The counter is
// reset for the next launch.  SERIAL: a column's slots are added in slot order
// by one thread instead of by a tree (see cta_colsum_serial).
template <int W, bool SERIAL = false>
__device__ bool last_cta_reduce(const double* part, uint32_t* counter, int panel, int nparts, int begin, int count,
                                double* s_out) {
    static_assert(W <= 32 && 32 % W == 0, "a column's slots are whole lane strides");
    __shared__ int s_last;
    constexpr int NS = VNE_THREADS / W, NR = SERIAL ? NS : VNE_WARPS;
    __shared__ double red[NR][W];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned old = atomicAdd(counter, 1u);
        s_last = (old == (unsigned)(count - 1));
    }
    __syncthreads();
    if (!s_last) return false;
    __threadfence();
    const int c = threadIdx.x % W, s = threadIdx.x / W;
    // four independent accumulators, so that four loads are in flight at
    // once (the order of the additions is still fixed)
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const double* src = part + ((size_t)panel * nparts + begin) * W + c;
    int i = s;
    for (; i + 3 * NS < count; i += 4 * NS) {
#pragma unroll
        for (int u = 0; u < 4; u++) acc[u] += ld_cg(src + (size_t)(i + u * NS) * W);
    }
#pragma unroll
    for (int u = 0; u < 3; u++)
        if (i + u * NS < count) acc[u] += ld_cg(src + (size_t)(i + u * NS) * W);
    double t = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    if (SERIAL) {
        red[s][c] = t;
    } else {
#pragma unroll
        for (int off = W; off < 32; off <<= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        if ((threadIdx.x & 31) < W) red[threadIdx.x >> 5][c] = t;
    }
    __syncthreads();
    if (threadIdx.x < W) {
        double x = 0.0;
#pragma unroll
        for (int w = 0; w < NR; w++) x += red[w][threadIdx.x];
        s_out[threadIdx.x] = x;
    }
    if (threadIdx.x == 0) *counter = 0u;
    __syncthreads();
    return true;
}

}  // namespace vne
