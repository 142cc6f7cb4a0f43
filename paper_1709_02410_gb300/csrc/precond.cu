// Body-block-diagonal preconditioner (Sec. 2.2).
//
// Interactions between distinct bodies are dropped: M~(pq) = delta_pq M(pp),
// with M(pp) the dense FP64 blob mobility of body p's blobs alone (wall and
// overlap regularisation included).  One CTA per body builds, in shared
// memory:
//   L_p      Cholesky factor, M(pp) = L_p L_p^T      (Lanczos: L = M~^{1/2})
//   L_p^-1   its inverse (triangular)
//   M(pp)^-1 = L_p^-T L_p^-1
//   M(pp)^-1 K_p and N_p = (K_p^T M(pp)^-1 K_p)^-1  (exact body-block solve
//            of the saddle system, eqs. saddle and N_def per body)
// and stores them column-major (element (i, j) at j*m + i, m = 3 nper, blob-
// interleaved rows 3b + c).
#include <cuda_runtime.h>

#include "pair64.cuh"
#include "precond.cuh"
#include "rpbd_internal.cuh"

namespace rpbd {

constexpr int PREC_THREADS = 256;

// One CTA per body, bound by FP64 instructions (about 19 cycles a warp instruction
// per SM) and, for few bodies, by the chain of m pivots.  Pair blocks are formed
// once per unordered pair; factorisation and inversion advance together, one
// pivot at a time, on a 16 x 16 grid of threads that strides over the matrices
// (no index divisions), so a pivot costs one reciprocal root, a scaled column
// and one pass of independent updates; M^-1's lower half is summed and mirrored;
// K's structure (identity and [d]_x) replaces its products.  Before, a separate
// factorisation, a substitution per thread with m dependent divisions and a
// one-thread 6 x 6 inversion: 128 boomerangs 248 -> 93 us, 256 in the periodic
// cell 344 -> 145, 4,369 2,311 -> 1,095; 4,096 rollers 1,491 -> 685.
template <bool WALL, bool PER>
__global__ void __launch_bounds__(PREC_THREADS) prec_build_kernel(int nper, int64_t n, const double* __restrict__ r,
                                                                  const double* __restrict__ q, double a, double s_min,
                                                                  pair64::Const pc, double inv8pieta,
                                                                  double* __restrict__ gL, double* __restrict__ gLinv,
                                                                  double* __restrict__ gMinv, double* __restrict__ gMinvK,
                                                                  double* __restrict__ gN, int* __restrict__ err)
{
    extern __shared__ double sm[];
    const int m = 3 * nper;
    const int64_t p = blockIdx.x;
    const int tid = threadIdx.x, ti = tid & 15, tj = tid >> 4;
    double* A = sm;              // m*m: M(pp) -> L (lower) -> M^-1
    double* X = A + m * m;       // m*m: I -> L^-1 (lower)
    double* B = X + m * m;       // m*6: M^-1 K
    double* bx = B + 6 * m;      // nper * 7: x, y, zt, s, r - q
    __shared__ double S6[36];
    __shared__ double pivot[2];
    __shared__ int spd_fail;
    if (tid == 0) spd_fail = 0;
    const double q0 = q[3 * p], q1 = q[3 * p + 1], q2 = q[3 * p + 2];
    for (int b = tid; b < nper; b += PREC_THREADS) {
        const int64_t i = p * nper + b;
        const double x = r[i], y = r[n + i], z = r[2 * n + i];
        double zt = z, s = 1.0;
        if (WALL) {
            zt = z > a ? z : a;
            const double t = z / a;
            s = t >= 1.0 ? 1.0 : (t <= s_min ? s_min : t);
        }
        double* o = bx + 7 * b;
        o[0] = x;
        o[1] = y;
        o[2] = zt;
        o[3] = s;
        o[4] = x - q0;
        o[5] = y - q1;
        o[6] = z - q2;
    }
    for (int e = tid; e < m * m; e += PREC_THREADS) X[e] = 0.0;
    __syncthreads();
    // 1. dense M(pp): block (bi, bj), bj <= bi, fills both of its places
    for (int pr = tid; pr < nper * (nper + 1) / 2; pr += PREC_THREADS) {
        int bi = (int)((sqrtf(8.0f * (float)pr + 1.0f) - 1.0f) * 0.5f);
        if (bi * (bi + 1) / 2 > pr) --bi;
        if ((bi + 1) * (bi + 2) / 2 <= pr) ++bi;
        const int bj = pr - bi * (bi + 1) / 2;
        const double* vi = bx + 7 * bi;
        const double* vj = bx + 7 * bj;
        pair64::Block M;
        pair64::block<WALL, PER>(vi[0] - vj[0], vi[1] - vj[1], vi[2], vj[2], pc, M);
        const double sc = vi[3] * vj[3] * inv8pieta;
        const double v[3][3] = {{M.xx, M.xy, M.xz}, {M.xy, M.yy, M.yz}, {M.zx, M.zy, M.zz}};
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                A[(3 * bj + d) * m + 3 * bi + c] = sc * v[c][d];
                A[(3 * bi + c) * m + 3 * bj + d] = sc * v[c][d];
            }
    }
    for (int i = tid; i < m; i += PREC_THREADS) X[i * m + i] = 1.0;
    __syncthreads();
    // 2. pivot k: L's column k and L^-1's row k, then both updates (column-major; the column
    // of L stays unscaled in A until its own step, the updates use the scaled one in place)
    for (int k = 0; k < m; ++k) {
        if (tid == 0) {
            const double dkk = A[k * m + k];
            if (!(dkk > 0.0)) spd_fail = 1;
            const double d = dkk > 1e-290 ? dkk : 1e-290;
            pivot[0] = rsqrt3(d);
        }
        __syncthreads();
        const double inv = pivot[0];
        for (int i = k + tid; i < m; i += PREC_THREADS) A[k * m + i] *= inv;  // L(i, k)
        for (int j = tid; j <= k; j += PREC_THREADS) X[j * m + k] *= inv;     // L^-1(k, j)
        __syncthreads();
        for (int i0 = k + 1; i0 < m; i0 += 16) {
            const int i = i0 + ti;
            const double l = i < m ? A[k * m + i] : 0.0;
            for (int j = k + 1 + tj; j < min(i0 + 16, m); j += 16)
                if (i < m && j <= i) A[j * m + i] -= l * A[k * m + j];
            for (int j = tj; j <= k; j += 16)
                if (i < m) X[j * m + i] -= l * X[j * m + k];
        }
        __syncthreads();
    }
    // 3. store L (strict upper triangle zero) and L^-1; M^-1 = X^T X, its lower half mirrored
    double* L_out = gL + p * m * m;
    double* Li_out = gLinv + p * m * m;
    double* Mi_out = gMinv + p * m * m;
    for (int j = tj; j < m; j += 16)
        for (int i = ti; i < m; i += 16) {
            L_out[j * m + i] = i >= j ? A[j * m + i] : 0.0;
            Li_out[j * m + i] = X[j * m + i];
        }
    __syncthreads();
    for (int i0 = 0; i0 < m; i0 += 16) {
        const int i = i0 + ti;
        for (int j0 = 0; j0 <= i0; j0 += 16) {
            const int j = j0 + tj;
            if (i >= m || j > i) continue;
            double v0 = 0.0, v1 = 0.0;  // (X is zero above its diagonal: k from the tile's first row)
            int k = i0;
            for (; k + 1 < m; k += 2) {
                v0 = fma(X[i * m + k], X[j * m + k], v0);
                v1 = fma(X[i * m + k + 1], X[j * m + k + 1], v1);
            }
            if (k < m) v0 = fma(X[i * m + k], X[j * m + k], v0);
            A[j * m + i] = A[i * m + j] = v0 + v1;
        }
    }
    __syncthreads();
    for (int e = tid; e < m * m; e += PREC_THREADS) Mi_out[e] = A[e];
    // 4. B = M^-1 K, rows of K: 3b + c has e_c and row c of -[d_b]_x
    for (int e = tid; e < 6 * m; e += PREC_THREADS) {
        const int c = e / m, i = e - c * m, c3 = c % 3, u = (c3 + 1) % 3, w = (c3 + 2) % 3;
        double v = 0.0;
        if (c < 3)
            for (int b = 0; b < nper; ++b) v += A[(3 * b + c) * m + i];
        else  // omega_c: velocity omega x d has component w: +d_u, component u: -d_w
            for (int b = 0; b < nper; ++b) {
                const double* d = bx + 7 * b + 4;
                v = fma(A[(3 * b + w) * m + i], d[u], v);
                v = fma(-A[(3 * b + u) * m + i], d[w], v);
            }
        B[c * m + i] = v;
        gMinvK[p * 6 * m + e] = v;
    }
    __syncthreads();
    // 5. S6 = K^T M^-1 K
    if (tid < 36) {
        const int a6 = tid % 6, b6 = tid / 6, c3 = a6 % 3, u = (c3 + 1) % 3, w = (c3 + 2) % 3;
        const double* Bc = B + b6 * m;
        double v = 0.0;
        if (a6 < 3)
            for (int b = 0; b < nper; ++b) v += Bc[3 * b + a6];
        else
            for (int b = 0; b < nper; ++b) {
                const double* d = bx + 7 * b + 4;
                v = fma(Bc[3 * b + w], d[u], v);
                v = fma(-Bc[3 * b + u], d[w], v);
            }
        S6[tid] = v;
    }
    __syncthreads();
    // 6. N_p = S6^-1 (symmetric positive definite) by Gauss-Jordan, lane = column of [S6 | I]
    if (tid < 32) {
        double col[6];
#pragma unroll
        for (int i = 0; i < 6; ++i)
            col[i] = tid < 6 ? 0.5 * (S6[tid * 6 + i] + S6[i * 6 + tid]) : (i == tid - 6 ? 1.0 : 0.0);
        bool fail = false;
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            double f[6];
#pragma unroll
            for (int i = 0; i < 6; ++i) f[i] = __shfl_sync(0xffffffffu, col[i], c);
            if (!(fabs(f[c]) > 0.0)) {
                fail = true;
                continue;
            }
            col[c] /= f[c];
#pragma unroll
            for (int i = 0; i < 6; ++i)
                if (i != c) col[i] = fma(-f[i], col[c], col[i]);
        }
        if (tid >= 6 && tid < 12)
#pragma unroll
            for (int i = 0; i < 6; ++i) gN[p * 36 + (tid - 6) * 6 + i] = col[i];
        if (tid == 0 && (fail || spd_fail)) atomicExch(err, 2);
    }
}

// out = A_p x_p per body, A_p one of the stored factors.
// mode 0: L (lower), 1: L^-1 (lower), 2: L^-T, 3: M^-1.  With `active`
// (batches: systems at blob offsets off[0..n_sys]), bodies of inactive
// systems are skipped and their out left as it is.
__global__ void __launch_bounds__(APPLY_THREADS) prec_apply_kernel(int mode, int nper, int64_t n,
                                                                   const double* Mat, const double* x, double* out,
                                                                   const int* active, const int64_t* off, int n_sys)
{
    __shared__ double v[PREC_MAX_M], part[APPLY_THREADS];
    pdl_wait();
    pdl_trigger();
    const int m = 3 * nper;
    const int64_t p = blockIdx.x;
    if (active) {
        const int64_t i = p * nper;  // the body's first blob; bodies never straddle systems
        int lo = 0, hi = n_sys;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (off[mid] <= i) lo = mid;
            else hi = mid;
        }
        if (!active[lo]) return;
    }
    const double* A = Mat + p * m * m;
    const int tid = threadIdx.x;
    for (int e = tid; e < m; e += APPLY_THREADS) v[e] = x[(e % 3) * n + p * nper + e / 3];
    __syncthreads();
    const int parts = apply_parts(m, APPLY_THREADS);
    const int q = tid / m, i = tid - q * m;
    if (mode == 2) {  // (L^-1)^T: sum_j Linv(j, i) v_j, j >= i: through shared memory, rows of odd length
        extern __shared__ double sA[];
        const int ld = m | 1, lane = tid & 31;
        for (int c = tid >> 5; c < m; c += APPLY_THREADS / 32)
            for (int j = c + lane; j < m; j += 32) sA[c * ld + j] = A[c * m + j];
        __syncthreads();
        if (q < parts) {
            double acc = 0.0;
#pragma unroll 4
            for (int j = i + q; j < m; j += parts) acc += sA[i * ld + j] * v[j];
            part[tid] = acc;
        }
    } else if (q < parts) {  // M^-1, or lower triangular (j <= i): row i's columns j = q, q + parts, ...
        const int j1 = mode == 3 ? m : i + 1;
        double acc = 0.0;
#pragma unroll 8
        for (int j = q; j < j1; j += parts) acc += A[j * m + i] * v[j];
        part[tid] = acc;
    }
    __syncthreads();
    if (tid < m) {
        double acc = part[tid];
        for (int q2 = 1; q2 < parts; ++q2) acc += part[q2 * m + tid];
        out[(tid % 3) * n + p * nper + tid / 3] = acc;
    }
}

// for up to four vectors (blockIdx.y)
struct SaddleArgs {
    PrecSaddle p[4];
};
__global__ void __launch_bounds__(APPLY_THREADS) prec_saddle_kernel(int nper, int64_t n, PrecFactors M, SaddleArgs S)
{
    pdl_wait();
    pdl_trigger();
    const PrecSaddle P = S.p[blockIdx.y];
    prec_saddle_body(nper, n, M, blockIdx.x, [&](int64_t e) { return P.a ? P.a[e] : 0.0; },
                     [&](int64_t e) { return P.b ? P.b[e] : 0.0; }, P.lam, P.U);
}

int precond_build_impl(rpbd_handle* h, int64_t nb, int nper, const double* r, const double* q, cudaStream_t st)
{
    if (nb <= 0) return set_error(h, RPBD_BAD_ARG, "precond_build: no bodies");
    const int m = 3 * nper;
    if (nper <= 0 || m > PREC_MAX_M) return set_error(h, RPBD_BAD_ARG, "precond_build: need 1 <= nper <= 32");
    const int64_t n = nb * nper;
    double *L, *Li, *Mi, *MK, *N;
    RPBD_TRY(ensure_t(h, BUF_PREC_L, (size_t)nb * m * m, &L));
    RPBD_TRY(ensure_t(h, BUF_PREC_LINV, (size_t)nb * m * m, &Li));
    RPBD_TRY(ensure_t(h, BUF_PREC_MINV, (size_t)nb * m * m, &Mi));
    RPBD_TRY(ensure_t(h, BUF_PREC_MINVK, (size_t)nb * 6 * m, &MK));
    RPBD_TRY(ensure_t(h, BUF_PREC_N, (size_t)nb * 36, &N));
    const size_t smem = (size_t)(2 * m * m + 6 * m + 7 * nper) * sizeof(double);
    const double inv8pieta = 1.0 / (8.0 * 3.14159265358979323846 * h->p.eta);
    if (once_per_device(h, reinterpret_cast<const void*>(prec_build_kernel<true, false>))) {
        const int mx = (2 * PREC_MAX_M * PREC_MAX_M + 6 * PREC_MAX_M + 7 * 32) * (int)sizeof(double);
        RPBD_CU(h, cudaFuncSetAttribute(prec_build_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
        RPBD_CU(h, cudaFuncSetAttribute(prec_build_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
        RPBD_CU(h, cudaFuncSetAttribute(prec_build_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
    }
    if (once_per_device(h, reinterpret_cast<const void*>(prec_apply_kernel)))
        RPBD_CU(h, cudaFuncSetAttribute(prec_apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        PREC_MAX_M * (PREC_MAX_M | 1) * (int)sizeof(double)));
    RPBD_CU(h, cudaMemsetAsync(h->dev_flag, 0, sizeof(int), st));
    const pair64::Const pc = pair64::Const::make(h->p);
    if (h->p.Lx > 0.0)
        prec_build_kernel<true, true><<<(unsigned)nb, PREC_THREADS, smem, st>>>(nper, n, r, q, h->p.a, h->p.s_min, pc, inv8pieta, L, Li, Mi, MK, N, h->dev_flag);
    else if (h->p.wall)
        prec_build_kernel<true, false><<<(unsigned)nb, PREC_THREADS, smem, st>>>(nper, n, r, q, h->p.a, h->p.s_min, pc, inv8pieta, L, Li, Mi, MK, N, h->dev_flag);
    else
        prec_build_kernel<false, false><<<(unsigned)nb, PREC_THREADS, smem, st>>>(nper, n, r, q, h->p.a, h->p.s_min, pc, inv8pieta, L, Li, Mi, MK, N, h->dev_flag);
    count_launch();
    RPBD_LAUNCH_CHECK(h);
    h->prec_nb = nb;
    h->prec_nper = nper;
    h->prec_valid = true;
    return RPBD_OK;
}

int precond_apply_impl(rpbd_handle* h, int mode, const double* x, double* out, cudaStream_t st, const int* active,
                       const int64_t* off, int n_sys)
{
    if (!h->prec_valid) return set_error(h, RPBD_BAD_ARG, "preconditioner not built");
    if (mode < 0 || mode > 3 || !x || !out) return set_error(h, RPBD_BAD_ARG, "precond_apply: bad arguments");
    const double* Mat = mode == 0 ? (const double*)h->buf[BUF_PREC_L]
                        : mode == 3 ? (const double*)h->buf[BUF_PREC_MINV]
                                    : (const double*)h->buf[BUF_PREC_LINV];
    const int m = 3 * h->prec_nper;
    launch_pdl(prec_apply_kernel, (unsigned)h->prec_nb, APPLY_THREADS, mode == 2 ? sizeof(double) * m * (m | 1) : 0, st, mode, h->prec_nper,
               h->prec_nb * h->prec_nper, Mat, x, out, active, off, n_sys);
    count_launch();
    RPBD_LAUNCH_CHECK(h);
    return RPBD_OK;
}

int precond_saddle_impl(rpbd_handle* h, int np, const PrecSaddle* ps, cudaStream_t st)
{
    if (!h->prec_valid) return set_error(h, RPBD_BAD_ARG, "preconditioner not built");
    SaddleArgs S = {};
    for (int a = 0; a < np; ++a) S.p[a] = ps[a];
    launch_pdl(prec_saddle_kernel, dim3((unsigned)h->prec_nb, (unsigned)np), APPLY_THREADS, 0, st, h->prec_nper,
               h->prec_nb * h->prec_nper, prec_factors(h), S);
    count_launch();
    RPBD_LAUNCH_CHECK(h);
    return RPBD_OK;
}

}  // namespace rpbd

using namespace rpbd;

extern "C" {

int rpbd_precond_build(rpbd_handle* h, int64_t nb, int nper, const double* r, const double* q, void* stream)
{
    if (!h) return RPBD_BAD_ARG;
    if (!r || !q) return set_error(h, RPBD_BAD_ARG, "precond_build: null pointer");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    RPBD_TRY(precond_build_impl(h, nb, nper, r, q, st));
    int flag = 0;
    RPBD_CU(h, cudaMemcpyAsync(&flag, h->dev_flag, sizeof(int), cudaMemcpyDeviceToHost, st));
    RPBD_CU(h, cudaStreamSynchronize(st));
    if (flag) {
        h->prec_valid = false;
        return set_error(h, RPBD_BAD_INPUT, "precond_build: a body block is not positive definite");
    }
    return RPBD_OK;
}

int rpbd_precond_apply(rpbd_handle* h, int mode, const double* x, double* out, void* stream)
{
    if (!h) return RPBD_BAD_ARG;
    return precond_apply_impl(h, mode, x, out, reinterpret_cast<cudaStream_t>(stream));
}

}  // extern "C"
