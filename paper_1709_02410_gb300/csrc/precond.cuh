// Products with the body-block preconditioner's stored factors (precond.cu): the
// exact body-block saddle solve, shared by its own kernel and the one that ends a
// GMRES iteration.
#pragma once

#include <cuda_runtime.h>

#include "rpbd_internal.cuh"

namespace rpbd {

constexpr int PREC_MAX_M = 96;  // 3 * nper <= 96

// Rows of the stored factors' products, one CTA per body, entries read straight
// from global memory, every one once.  The threads split a row's columns into up
// to eight pieces, so a chain is ~m / 4 loads, issued eight at a time; with half
// the threads, the factor staged in shared memory first and loads one by one a
// 45-row product took 8.9 us of a call, now 4.6.  The FP64 pipe (one warp
// instruction in ~19 cycles of an SM) bounds the products of many bodies, so
// thread tid = q m + i takes piece q of row i: no lane is left out for a row count
// that is not a multiple of 32, and consecutive threads read consecutive entries.
constexpr int APPLY_THREADS = 256;
__host__ __device__ __forceinline__ int apply_parts(int m, int threads)
{
    const int p = threads / m;
    return p < 8 ? p : 8;
}

// s[c] summed over each group of G lanes (8, 16 or 32), c < 6: the lanes of a group
// halve the sums among them first, 5 + log2(G) - 2 additions instead of 6 log2(G).
// sum6_of(lane in the group) tells which sum the lane has (-1: a copy).
template <int G>
__device__ __forceinline__ double group_sum6(const double (&s)[6], int lane)
{
    double t[3];
    const bool u2 = lane & (G / 2), u4 = lane & (G / 4), u8 = lane & (G / 8);
#pragma unroll
    for (int c = 0; c < 3; ++c)
        t[c] = (u2 ? s[c + 3] : s[c]) + __shfl_xor_sync(0xffffffffu, u2 ? s[c] : s[c + 3], G / 2);
    const double a0 = (u4 ? t[2] : t[0]) + __shfl_xor_sync(0xffffffffu, u4 ? t[0] : t[2], G / 4);
    const double a1 = t[1] + __shfl_xor_sync(0xffffffffu, t[1], G / 4);
    double v = (u8 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, u8 ? a0 : a1, G / 8);
#pragma unroll
    for (int o = G / 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
template <int G>
__device__ __forceinline__ int sum6_of(int lane)
{
    const int l = lane & (G - 1);
    if (l & (G / 8 - 1)) return -1;
    const int b = (l & (G / 4)) ? ((l & (G / 8)) ? -4 : 2) : ((l & (G / 8)) ? 1 : 0);
    return b < 0 ? -1 : b + ((l & (G / 2)) ? 3 : 0);
}

struct PrecFactors {
    const double *Minv, *MinvK, *N;
};
inline PrecFactors prec_factors(const rpbd_handle* h)
{
    return PrecFactors{(const double*)h->buf[BUF_PREC_MINV], (const double*)h->buf[BUF_PREC_MINVK],
                       (const double*)h->buf[BUF_PREC_N]};
}

// [M(pp) -K_p; -K_p^T 0][lam; U] = [a; b] of body p, by the whole CTA:
//   t = (M^-1 K)^T a + b,  U = -N t,  lam = M^-1 a + (M^-1 K) U
// a(e), b(e): element e of the blob vector [3][n] and of the body vector [nb][6],
// each asked for once.  M^-1 a does not wait for U.  With t, U by their own warp,
// packed rows, and saddle products, norms and sums likewise thrifty with FP64
// instructions (krylov.cu), a GMRES iteration takes, beyond its matvec, at 1,920
// blobs 34 us (39 before), 3,840 38 (53), 7,680 41 (71), 16,380 60 (92), 65,535
// 142 (190).
template <class A, class B>
__device__ __forceinline__ void prec_saddle_body(int nper, int64_t n, const PrecFactors& M, int64_t p, A a, B b, double* lam,
                                                 double* U)
{
    __shared__ double va[PREC_MAX_M], part[APPLY_THREADS], t6[6], u6[6];
    constexpr int ROWS = APPLY_THREADS - 32;  // the last warp takes t and U
    const int m = 3 * nper;
    const int tid = threadIdx.x, lane = tid & 31;
    const int parts = apply_parts(m, ROWS);
    const double* Mi = M.Minv + p * m * m;      // column-major: (i, j) at j * m + i
    const double* MK = M.MinvK + p * 6 * m;     // (M^-1 K)^T rows: column c at c * m
    for (int e = tid; e < m; e += APPLY_THREADS) va[e] = a((e % 3) * n + p * nper + e / 3);
    __syncthreads();
    if (tid >= ROWS) {
        double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (int k = lane; k < m; k += 32) {
            const double x = va[k];
#pragma unroll
            for (int c = 0; c < 6; ++c) v[c] += MK[c * m + k] * x;
        }
        const double t = group_sum6<32>(v, lane);
        const int c = sum6_of<32>(lane);
        if (c >= 0) t6[c] = t + b(6 * p + c);
        __syncwarp();
        if (lane < 6) {
            double w = 0.0;
#pragma unroll
            for (int e = 0; e < 6; ++e) w -= M.N[p * 36 + e * 6 + lane] * t6[e];
            u6[lane] = w;
            U[6 * p + lane] = w;
        }
    } else if (tid < parts * m) {
        const int q = tid / m, i = tid - q * m;
        double v = 0.0;
#pragma unroll 8
        for (int j = q; j < m; j += parts) v += Mi[j * m + i] * va[j];
        part[tid] = v;
    }
    __syncthreads();
    if (tid < m) {
        double v = part[tid];
        for (int q2 = 1; q2 < parts; ++q2) v += part[q2 * m + tid];
#pragma unroll
        for (int c = 0; c < 6; ++c) v += MK[c * m + tid] * u6[c];
        lam[(tid % 3) * n + p * nper + tid / 3] = v;
    }
}

}  // namespace rpbd
