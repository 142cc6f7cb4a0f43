// Products with the body-block preconditioner's stored factors (precond.cu): the
// exact body-block saddle solve, shared by its own kernel and the one that ends a
// GMRES iteration.
#pragma once

#include <cuda_runtime.h>

#include "rpbd_internal.cuh"

namespace rpbd {

constexpr int PREC_MAX_M = 96;  // 3 * nper <= 96

// Rows of the stored factors' products, one CTA per body, entries read straight
// from global memory, every one once.  The threads split a row's columns into
// APPLY_THREADS / span pieces, so a chain is ~m / 4 loads, issued eight at a
// time; with half the threads, the factor staged in shared memory first and
// loads one by one a 45-row product took 8.9 us of a call, now 4.6.
constexpr int APPLY_THREADS = 256;

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
// each asked for once.  M^-1 a does not wait for U.
template <class A, class B>
__device__ __forceinline__ void prec_saddle_body(int nper, int64_t n, const PrecFactors& M, int64_t p, A a, B b, double* lam,
                                                 double* U)
{
    __shared__ double va[PREC_MAX_M], part[APPLY_THREADS], t6[6], u6[6];
    const int m = 3 * nper;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int span = (m + 31) & ~31, parts = APPLY_THREADS / span;
    const double* Mi = M.Minv + p * m * m;      // column-major: (i, j) at j * m + i
    const double* MK = M.MinvK + p * 6 * m;     // (M^-1 K)^T rows: column c at c * m
    for (int e = tid; e < m; e += APPLY_THREADS) va[e] = a((e % 3) * n + p * nper + e / 3);
    __syncthreads();
    if (warp < 6) {
        double v = 0.0;
        for (int k = lane; k < m; k += 32) v += MK[warp * m + k] * va[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) t6[warp] = v + b(6 * p + warp);
    }
    const int q = tid / span, i = tid % span;
    if (q < parts && i < m) {
        double v = 0.0;
#pragma unroll 8
        for (int j = q; j < m; j += parts) v += Mi[j * m + i] * va[j];
        part[q * span + i] = v;
    }
    __syncthreads();
    if (tid < 6) {
        double v = 0.0;
#pragma unroll
        for (int c = 0; c < 6; ++c) v -= M.N[p * 36 + c * 6 + tid] * t6[c];
        u6[tid] = v;
        U[6 * p + tid] = v;
    }
    __syncthreads();
    if (tid < m) {
        double v = part[tid];
        for (int q2 = 1; q2 < parts; ++q2) v += part[q2 * span + tid];
#pragma unroll
        for (int c = 0; c < 6; ++c) v += MK[c * m + tid] * u6[c];
        lam[(tid % 3) * n + p * nper + tid / 3] = v;
    }
}

}  // namespace rpbd
