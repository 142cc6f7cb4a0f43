// Krylov solvers of the hot path, FP64 vectors on the device:
//
//  Lanczos M^{1/2} W (Sec. 2.2): Lanczos on G = L^-1 M L^-T (L the block
//    Cholesky preconditioner) from v_1 = W/|W| with full (classical, twice)
//    reorthogonalisation; f(G) W ~ |W| V_m T_m^{1/2} e_1, T_m^{1/2} e_1 by one
//    warp (contour-integral quadrature, tridiag_sqrt.cuh); stop when |y_m - y_{m-1}| / |y_m| < tol (evaluated in the small space, V is
//    orthonormal); output L y_m.
//  GMRES (Sec. 2.1, eq. saddle): right-preconditioned restarted GMRES(m) on
//    [M -K; -K^T 0] with the exact body-block solve of Sec. 2.2 as
//    preconditioner; Arnoldi by classical Gram-Schmidt applied twice, Givens
//    rotations and the Hessenberg least-squares solve in a device kernel.
//
// The host drives the iteration and reads one FP64 scalar per iteration (the
// residual estimate or the Lanczos change, which the iteration's last kernel
// writes to pinned host memory) to decide whether to stop; every arithmetic
// step runs in the kernels below.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "ortho.cuh"
#include "precond.cuh"
#include "rpbd_internal.cuh"
#include "tridiag_sqrt.cuh"

namespace rpbd {

constexpr int DOT_BLOCKS = 256;
constexpr int LANCZOS_MAX = 80;

// ---------------------------------------------------------------------------
// vector kernels

// partial[i * gridDim.x + bx] = sum over the block's slice of V_i . w
__global__ void multidot_kernel(int64_t n, const double* __restrict__ V, int64_t ld, const double* __restrict__ w,
                                double* __restrict__ partial)
{
    const int i = blockIdx.y;
    const double* v = V + (int64_t)i * ld;
    double s = 0.0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        s += v[e] * w[e];
    __shared__ double red[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) partial[(int64_t)i * gridDim.x + blockIdx.x] = s;
    }
}

// out[i] = sum_b partial[i * nb + b]; one block per i
__global__ void reduce_partials_kernel(int nblocks, const double* __restrict__ partial, double* __restrict__ out)
{
    const int i = blockIdx.x;
    double s = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) s += partial[(int64_t)i * nblocks + b];
    __shared__ double red[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) out[i] = s;
    }
}

// out = scale * sum_i y[i] V_i
__global__ void lincomb_kernel(int64_t n, const double* __restrict__ V, int64_t ld, int nv,
                               const double* __restrict__ y, double scale, double* __restrict__ out)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int i = 0; i < nv; ++i) s += y[i] * V[(int64_t)i * ld + e];
        out[e] = scale * s;
    }
}

// out = x / sqrt(*nrm2)  (or 0 when the norm vanishes)
__global__ void normalize_kernel(int64_t n, const double* __restrict__ x, const double* __restrict__ nrm2,
                                 double* __restrict__ out)
{
    const double nv = sqrt(nrm2[0]);
    const double inv = nv > 0.0 ? 1.0 / nv : 0.0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        out[e] = x[e] * inv;
}

__global__ void add_kernel(int64_t n, const double* __restrict__ x, double* __restrict__ y)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        y[e] += x[e];
}

// Saddle products of up to four processes (blockIdx.y): w = [M lam - K U; -K^T lam]
// given M lam (Ml, which may be w itself).  G lanes per body, the smallest of 8,
// 16 and 32 that has one per blob: the FP64 pipe bounds it, at one warp per body
// and six separate sums 75 instructions a body of 15 blobs, now 26.
struct SaddleProd {
    const double *Ml, *lam, *U;
    double* w;
};
struct SaddleBatch {
    SaddleProd p[4];
};
constexpr int SADDLE_THREADS = 32;  // (few bodies: one warp per SM)
template <int G>
__global__ void saddle_kernel(int64_t nb, int nper, const double* r, const double* q, SaddleBatch B)
{
    pdl_wait();
    pdl_trigger();
    const int64_t bi = (blockIdx.x * (int64_t)SADDLE_THREADS + threadIdx.x) / G;
    const bool on = bi < nb;
    const int64_t b = on ? bi : nb - 1;
    const SaddleProd P = B.p[blockIdx.y];
    const int lane = threadIdx.x & 31;
    const int64_t n = nb * nper;
    const double q0 = q[3 * b], q1 = q[3 * b + 1], q2 = q[3 * b + 2];
    double u[6], s[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int c = 0; c < 6; ++c) u[c] = P.U[6 * b + c];
    for (int k = on ? lane % G : nper; k < nper; k += G) {
        const int64_t i = b * nper + k;
        const double d0 = r[i] - q0, d1 = r[n + i] - q1, d2 = r[2 * n + i] - q2;
        const double l0 = P.lam[i], l1 = P.lam[n + i], l2 = P.lam[2 * n + i];
        P.w[i] = P.Ml[i] - (u[0] + (u[4] * d2 - u[5] * d1));
        P.w[n + i] = P.Ml[n + i] - (u[1] + (u[5] * d0 - u[3] * d2));
        P.w[2 * n + i] = P.Ml[2 * n + i] - (u[2] + (u[3] * d1 - u[4] * d0));
        s[0] += l0;
        s[1] += l1;
        s[2] += l2;
        s[3] += d1 * l2 - d2 * l1;
        s[4] += d2 * l0 - d0 * l2;
        s[5] += d0 * l1 - d1 * l0;
    }
    const double v = group_sum6<G>(s, lane);
    const int c = sum6_of<G>(lane);
    if (on && c >= 0) P.w[3 * n + 6 * b + c] = -v;
}

static unsigned vgrid(int64_t n)
{
    int64_t g = (n + 255) / 256;
    if (g > 152 * 8) g = 152 * 8;
    return (unsigned)(g < 1 ? 1 : g);
}

// out[0..nv) = V^T w
static int multidot(rpbd_handle* h, int64_t n, const double* V, int64_t ld, int nv, const double* w, double* out,
                    double* partial, cudaStream_t st)
{
    multidot_kernel<<<dim3(DOT_BLOCKS, nv), 256, 0, st>>>(n, V, ld, w, partial); count_launch();
    reduce_partials_kernel<<<nv, 256, 0, st>>>(DOT_BLOCKS, partial, out); count_launch();
    RPBD_LAUNCH_CHECK(h);
    return RPBD_OK;
}

// ---------------------------------------------------------------------------
// Orthogonalisation of w against a Krylov basis V_0..V_{nv-1}: classical
// Gram-Schmidt twice, the norm, and v_nv = w / |w|, for up to four processes at
// once (blockIdx.y), in four kernels that start under each other's tail.  As
// separate dot, reduction, update, add, norm and normalisation launches the step
// was eleven launches, ~60 us of a ~140 us GMRES iteration at 1,920 blobs whose
// arithmetic takes ~3 us.  Each block keeps its slice of w in shared memory
// through an update and the dot products that follow it, and sums the previous
// kernel's per-block partials itself (the same fixed order in every block).
struct OrthoProc {
    const double* V;
    double *w, *part, *h, *vnext;  // part: ortho_part doubles; h: nv coefficients of both passes
    int nv;
    // GMRES: H column, rotations, residual; Lanczos: the tridiagonal's end
    double *H, *cs, *sn, *g, *sc, *zl, *zU;
    double *alpha, *beta, *c, *c_prev;
    double* host;  // two scalars for the host
};
struct OrthoBatch {
    OrthoProc p[4];
};

// blocks of w: 128 elements each while that does not fill two blocks per SM of
// this GPU's 152, at most 4,096 (the slice in shared memory)
static int ortho_blocks(int64_t len)
{
    const int64_t small = (len + 127) / 128;
    if (small <= 304) return (int)small;
    return (int)std::max<int64_t>(304, (len + 4095) / 4096);
}
static size_t ortho_part(int64_t len, int nv) { return (size_t)ortho_blocks(len) * (2 * nv + 1); }

// h[i] = sum of the blocks' partials of dot i, i < nv (shared memory, all threads)
__device__ __forceinline__ void ortho_gather(int nv, int nblk, const double* part, double* h)
{
    ortho_sums(nv, nblk, [&](int i, int b) { return part[(int64_t)i * nblk + b]; }, [&](int i, double s) { h[i] = s; });
    __syncthreads();
}

// PASS 0: partials of V^T w.  1: w -= V h with h from pass 0's partials, then
// partials of V^T w.  2: w -= V h with pass 1's, then the partials of |w|^2.
template <int PASS>
__global__ void ortho_kernel(int64_t len, int64_t ld, int slice, OrthoBatch B)
{
    extern __shared__ double sm[];
    double* ws = sm;           // slice
    double* h = sm + slice;    // nv
    pdl_wait();
    pdl_trigger();
    const OrthoProc P = B.p[blockIdx.y];
    const int nblk = gridDim.x;
    const int64_t e0 = (int64_t)blockIdx.x * slice;
    const int cnt = (int)max((int64_t)0, min((int64_t)slice, len - e0));
    const double* V = P.V + e0;
    double* in = P.part + (PASS == 2 ? (int64_t)P.nv * nblk : 0);
    double* out = P.part + (PASS == 0 ? 0 : PASS == 1 ? (int64_t)P.nv * nblk : 2 * (int64_t)P.nv * nblk);
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) ws[e] = P.w[e0 + e];
    if (PASS > 0) {
        ortho_gather(P.nv, nblk, in, h);
        if (blockIdx.x == 0)
            for (int i = threadIdx.x; i < P.nv; i += blockDim.x) P.h[i] = PASS == 1 ? h[i] : P.h[i] + h[i];
        for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
            double s4[4] = {0.0, 0.0, 0.0, 0.0};
            int i = 0;
            for (; i + 4 <= P.nv; i += 4)
#pragma unroll
                for (int u = 0; u < 4; ++u) s4[u] += h[i + u] * V[(int64_t)(i + u) * ld + e];
            for (; i < P.nv; ++i) s4[0] += h[i] * V[(int64_t)i * ld + e];
            const double s = ws[e] - ((s4[0] + s4[1]) + (s4[2] + s4[3]));
            ws[e] = s;
            P.w[e0 + e] = s;
        }
    }
    __syncthreads();
    if (PASS == 2)
        ortho_sums<1>(1, cnt, [&](int, int e) { return ws[e] * ws[e]; },
                      [&](int, double x) { out[blockIdx.x] = x; });
    else
        ortho_sums(P.nv, cnt, [&](int i, int e) { return V[(int64_t)i * ld + e] * ws[e]; },
                   [&](int i, double x) { out[(int64_t)i * nblk + blockIdx.x] = x; });
}

// h[0..2] = |w|^2 from the partials of pass 2, |w| and 1/|w| (0 when it vanishes):
// by one thread, a square root and a division in every one keep the FP64 pipe
// busy longer than the rest of the finishing kernels
__device__ __forceinline__ void ortho_norm(const OrthoProc& P, int nblk, double* h)
{
    const double* part = P.part + 2 * (int64_t)P.nv * nblk;
    ortho_sums<1>(1, nblk, [&](int, int b) { return part[b]; },
                  [&](int, double s) {
                      const double nv = sqrt(s);
                      h[0] = s;
                      h[1] = nv;
                      h[2] = nv > 0.0 ? 1.0 / nv : 0.0;
                  });
    __syncthreads();
}

// v_nv = w / |w| of the block's slice (0 when the norm vanishes)
__device__ __forceinline__ void ortho_normalize(const OrthoProc& P, int64_t len, int slice, double inv)
{
    const int64_t e0 = (int64_t)blockIdx.x * slice;
    const int cnt = (int)max((int64_t)0, min((int64_t)slice, len - e0));
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) P.vnext[e0 + e] = P.w[e0 + e] * inv;
}

// GMRES: v_{j+1} = w / |w| and at once z = P^-1 v_{j+1} for the next iteration (the
// body-block solve of precond.cuh, a block per body: two launches' work in one, and
// the residual is on its way to the host meanwhile); in one block more H's column
// j = nv - 1, the rotations and the residual estimate.  sc: [1] |b|, [2] residual
// estimate
__global__ void __launch_bounds__(APPLY_THREADS) gmres_finish_kernel(int nper, int64_t n, int nblk, int mdim, PrecFactors M,
                                                                     OrthoBatch B)
{
    extern __shared__ double sm[];  // 3 (mdim + 2)
    pdl_wait();
    pdl_trigger();
    const OrthoProc P = B.p[blockIdx.y];
    const int j = P.nv - 1;
    ortho_norm(P, nblk, sm);
    const double nv = sm[1], inv = sm[2];
    if (blockIdx.x + 1 < gridDim.x) {
        prec_saddle_body(nper, n, M, blockIdx.x,
                         [&](int64_t e) {
                             const double v = P.w[e] * inv;
                             P.vnext[e] = v;
                             return v;
                         },
                         [&](int64_t e) {
                             const double v = P.w[3 * n + e] * inv;
                             P.vnext[3 * n + e] = v;
                             return v;
                         },
                         P.zl, P.zU);
        return;
    }
    __syncthreads();
    double *col = sm, *cs = sm + mdim + 2, *sn = cs + mdim + 2;
    for (int i = threadIdx.x; i <= j; i += blockDim.x) {
        col[i] = P.h[i];
        cs[i] = P.cs[i];
        sn[i] = P.sn[i];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double last = nv, cur = col[0];  // rotate down the column
        for (int i = 0; i < j; ++i) {
            const double nx = col[i + 1];
            col[i] = cs[i] * cur + sn[i] * nx;
            cur = -sn[i] * cur + cs[i] * nx;
        }
        const double den = hypot(cur, last);
        const double c = den > 0.0 ? cur / den : 1.0, sv = den > 0.0 ? last / den : 0.0;
        P.cs[j] = c;
        P.sn[j] = sv;
        col[j] = den;
        const double gj = P.g[j], gn = -sv * gj;
        P.g[j + 1] = gn;
        P.g[j] = c * gj;
        const double res = fabs(gn) / P.sc[1];
        P.sc[2] = res;
        P.host[0] = P.sc[1];
        P.host[1] = res;
    }
    __syncthreads();
    double* H = P.H + (int64_t)j * (mdim + 1);
    for (int i = threadIdx.x; i <= j + 1; i += blockDim.x) H[i] = i <= j ? col[i] : 0.0;
}

// y = H(0:k,0:k)^-1 g(0:k), back substitution by columns: one block, the
// right-hand side in shared memory (k doubles)
__global__ void gmres_backsolve_kernel(int k, int mdim, const double* __restrict__ H, const double* __restrict__ g,
                                       double* __restrict__ y)
{
    extern __shared__ double s[];
    for (int i = threadIdx.x; i < k; i += blockDim.x) s[i] = g[i];
    __syncthreads();
    for (int i = k - 1; i >= 0; --i) {
        const double* col = H + (int64_t)i * (mdim + 1);
        const double d = col[i];
        const double v = d != 0.0 ? s[i] / d : 0.0;
        __syncthreads();
        for (int c = threadIdx.x; c < i; c += blockDim.x) s[c] -= col[c] * v;
        if (threadIdx.x == 0) y[i] = v;
        __syncthreads();
    }
}

// g = [sqrt(nrm2), 0, ...]; bnorm = sc[1] (when first) = sqrt(nrm2); sc[2] = sqrt(nrm2)/bnorm
__global__ void gmres_start_kernel(int mdim, const double* __restrict__ nrm2, double* __restrict__ g,
                                   double* __restrict__ sc, int first, double* __restrict__ host)
{
    const double b = sqrt(nrm2[0]);
    for (int i = threadIdx.x; i <= mdim; i += blockDim.x) g[i] = i == 0 ? b : 0.0;
    if (threadIdx.x == 0) {
        const double bn = first ? b : sc[1];
        sc[1] = bn;
        sc[2] = bn > 0.0 ? b / bn : 0.0;
        host[0] = bn;
        host[1] = sc[2];
    }
}

// ---------------------------------------------------------------------------
// Lanczos small kernels

// v_{m+1}, and in one block more alpha_m = h[m], beta_m = |w|, c = T^{1/2} e_1 of
// the (m+1) x (m+1) tridiagonal T (tridiag_sqrt.cuh, its shared memory) and the
// change |c - [c_prev; 0]| / |c|; nv = m + 1.  host: |w|^2, change
__global__ void lanczos_finish_kernel(int64_t len, int slice, const SqrtNode* nodes, OrthoBatch B)
{
    extern __shared__ double sm[];
    pdl_wait();
    pdl_trigger();
    const OrthoProc P = B.p[blockIdx.y];
    const int nblk = gridDim.x - 1, m1 = P.nv, lane = threadIdx.x & 31;
    ortho_norm(P, nblk, sm);
    const double nrm2 = sm[0], nv = sm[1], inv = sm[2];
    if ((int)blockIdx.x < nblk) {
        ortho_normalize(P, len, slice, inv);
        return;
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    if (lane == 0) {
        P.alpha[m1 - 1] = P.h[m1 - 1];
        P.beta[m1 - 1] = nv;
    }
    __syncwarp();
    tridiag_sqrt_e1(m1, nodes, P.alpha, P.beta, sm, P.c);
    double nc = 0.0, nd = 0.0;
    for (int i = lane; i < m1; i += 32) {
        const double v = P.c[i];
        const double prev = i < m1 - 1 ? P.c_prev[i] : 0.0;
        nc += v * v;
        nd += (v - prev) * (v - prev);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        nc += __shfl_xor_sync(0xffffffffu, nc, o);
        nd += __shfl_xor_sync(0xffffffffu, nd, o);
    }
    __syncwarp();
    for (int i = lane; i < m1; i += 32) P.c_prev[i] = P.c[i];
    if (lane == 0) {
        P.host[0] = nrm2;
        P.host[1] = nc > 0.0 ? sqrt(nd / nc) : 0.0;
    }
}

// ---------------------------------------------------------------------------
// host helpers

static int check_flag(rpbd_handle* h, cudaStream_t st)
{
    int flag = 0;
    RPBD_CU(h, cudaMemcpyAsync(&flag, h->dev_flag, sizeof(int), cudaMemcpyDeviceToHost, st));
    RPBD_CU(h, cudaStreamSynchronize(st));
    if (flag == 1) return set_error(h, RPBD_TIMEOUT, "a pair kernel's bounded wait expired");
    return RPBD_OK;
}

// small device scratch layout (doubles)
struct Small {
    double* base;
    int mdim;
    double* H() { return base; }                                   // (mdim+1) * mdim
    double* cs() { return H() + (int64_t)(mdim + 1) * mdim; }      // mdim
    double* sn() { return cs() + mdim; }                           // mdim
    double* g() { return sn() + mdim; }                            // mdim + 1
    double* y() { return g() + mdim + 1; }                         // mdim + 1
    double* hcol() { return y() + mdim + 1; }                      // mdim + 2
    double* scal() { return hcol() + mdim + 2; }                   // 8 scalars
    double* partial() { return scal() + 8; }                       // DOT_BLOCKS, or ortho_part(len, mdim)
    static size_t count(int mdim, int64_t len)
    {
        return (size_t)(mdim + 1) * mdim + 2 * mdim + 3 * (mdim + 1) + 1 + 8 +
               std::max<size_t>(DOT_BLOCKS, ortho_part(len, mdim));
    }
};

// orthogonalises the batch's np processes (the first three kernels; the caller
// launches the finishing one with the returned grid and slice)
struct OrthoGrid {
    int blocks, slice, threads;
};
static OrthoGrid launch_ortho(int64_t len, int np, const OrthoBatch& B, cudaStream_t st)
{
    OrthoGrid G;
    G.blocks = ortho_blocks(len);
    G.slice = (int)((len + G.blocks - 1) / G.blocks);
    G.threads = G.slice > 512 ? 512 : 256;
    int nv = 0;
    for (int a = 0; a < np; ++a) nv = std::max(nv, B.p[a].nv);
    const dim3 grid((unsigned)G.blocks, (unsigned)np);
    const size_t smem = (size_t)(G.slice + nv) * sizeof(double);
    launch_pdl(ortho_kernel<0>, grid, G.threads, smem, st, len, len, G.slice, B);
    count_launch();
    launch_pdl(ortho_kernel<1>, grid, G.threads, smem, st, len, len, G.slice, B);
    count_launch();
    launch_pdl(ortho_kernel<2>, grid, G.threads, smem, st, len, len, G.slice, B);
    count_launch();
    return G;
}

// ---------------------------------------------------------------------------
// Lanczos

// Several Lanczos processes (different W, same M and preconditioner) advance
// in lockstep: each iteration gathers the active processes' vectors into one
// multi-RHS matvec and reads every process's scalars with one
// synchronisation.  Each process keeps its own basis, tridiagonal matrix and
// stopping test, so the answers are those of separate runs.
struct LanczosProc {
    const double* W;
    double* out;
    double *V, *z, *y, *w, *alpha, *beta, *cvec, *cprev, *sc;  // sc: [0] |W|^2, [1] |w|^2, [2] change
    Small S{nullptr, 0};
    double W2 = 0.0, change = INFINITY;
    int m = 0, matvecs = 0, status = RPBD_NOT_CONVERGED;
    bool active = false;
};

int lanczos_multi_impl(rpbd_handle* h, int64_t n, const double* r, int nsys, const double* const* W,
                       double* const* out, double tol, int max_iter, int dtype, int use_precond, rpbd_stats* stats,
                       cudaStream_t st)
{
    if (n <= 0) return set_error(h, RPBD_BAD_ARG, "lanczos: n <= 0");
    if (nsys < 1 || nsys > 4) return set_error(h, RPBD_BAD_ARG, "lanczos: 1..4 vectors");
    if (max_iter < 1 || max_iter > LANCZOS_MAX) return set_error(h, RPBD_BAD_ARG, "lanczos: max_iter must be in 1..80");
    if (use_precond && (!h->prec_valid || h->prec_nb * h->prec_nper != n))
        return set_error(h, RPBD_BAD_ARG, "lanczos: preconditioner not built for these blobs");
    if (!r) return set_error(h, RPBD_BAD_ARG, "lanczos: null positions");
    RPBD_TRY(check_finite(h, 3 * n, r, st));
    const int64_t len = 3 * n;
    const int mdim = LANCZOS_MAX + 1;
    const size_t small_count = Small::count(mdim, len) + 4 * (size_t)mdim;
    double *Vall, *vall, *small, *mv = nullptr;
    RPBD_TRY(ensure_t(h, BUF_KRYLOV, (size_t)nsys * (max_iter + 1) * len, &Vall));
    RPBD_TRY(ensure_t(h, BUF_VEC, (size_t)nsys * 3 * len, &vall));
    RPBD_TRY(ensure_t(h, BUF_SMALL, (size_t)nsys * small_count, &small));
    if (nsys > 1) RPBD_TRY(ensure_t(h, BUF_GMRES_MV, (size_t)2 * nsys * len, &mv));
    if (once_per_device(h, reinterpret_cast<const void*>(lanczos_finish_kernel)))
        RPBD_CU(h, cudaFuncSetAttribute(lanczos_finish_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        tridiag_sqrt_smem_doubles(LANCZOS_MAX + 1) * (int)sizeof(double)));
    RPBD_CU(h, cudaMemsetAsync(h->dev_flag, 0, sizeof(int), st));
    const unsigned g = vgrid(len);
    LanczosProc P[4];
    for (int s = 0; s < nsys; ++s) {
        LanczosProc& p = P[s];
        if (!W[s] || !out[s]) return set_error(h, RPBD_BAD_ARG, "lanczos: null pointer");
        p.W = W[s];
        p.out = out[s];
        p.V = Vall + (int64_t)s * (max_iter + 1) * len;
        // z and y of all processes lie side by side: a k-RHS matvec takes them as they are
        p.z = vall + (int64_t)s * len;
        p.y = vall + (int64_t)(nsys + s) * len;
        p.w = vall + (int64_t)(2 * nsys + s) * len;
        p.S = Small{small + (int64_t)s * small_count, mdim};
        p.alpha = small + (int64_t)(s + 1) * small_count - 4 * (size_t)mdim;
        p.beta = p.alpha + mdim;
        p.cvec = p.beta + mdim;
        p.cprev = p.cvec + mdim;
        p.sc = p.S.scal();
        RPBD_CU(h, cudaMemsetAsync(p.cprev, 0, sizeof(double) * mdim, st));
        RPBD_TRY(multidot(h, len, p.W, 0, 1, p.W, &p.sc[0], p.S.partial(), st));
        normalize_kernel<<<g, 256, 0, st>>>(len, p.W, &p.sc[0], p.V); count_launch();
        RPBD_CU(h, cudaMemcpyAsync(h->host_small + s, &p.sc[0], sizeof(double), cudaMemcpyDeviceToHost, st));
    }
    RPBD_LAUNCH_CHECK(h);
    RPBD_CU(h, cudaStreamSynchronize(st));
    for (int s = 0; s < nsys; ++s) {
        P[s].W2 = h->host_small[s];
        if (P[s].W2 > 0.0) {
            P[s].active = true;
        } else {
            RPBD_CU(h, cudaMemsetAsync(P[s].out, 0, sizeof(double) * len, st));
            P[s].status = RPBD_OK;
        }
    }
    for (;;) {
        int act[4], k = 0;
        for (int s = 0; s < nsys; ++s)
            if (P[s].active) act[k++] = s;
        if (k == 0) break;
        // w = G v_m for every active process, one k-RHS matvec
        const bool side = act[k - 1] - act[0] == k - 1;  // their z and y are side by side
        for (int a = 0; a < k; ++a) {
            LanczosProc& p = P[act[a]];
            const double* vm = p.V + (int64_t)p.m * len;
            double* dst = side ? p.z : mv + (int64_t)a * len;
            if (use_precond) RPBD_TRY(precond_apply_impl(h, 2, vm, dst, st));
            else if (k > 1) RPBD_CU(h, cudaMemcpyAsync(dst, vm, sizeof(double) * len, cudaMemcpyDeviceToDevice, st));
        }
        LanczosProc& p0 = P[act[0]];
        const double* Fm = !use_precond && k == 1 ? p0.V + (int64_t)p0.m * len : side ? p0.z : mv;
        double* Um = !use_precond && k == 1 ? p0.w : side ? p0.y : mv + (int64_t)k * len;
        RPBD_TRY(mobility_apply_impl(h, n, r, Fm, Um, k, dtype, true, st));
        OrthoBatch B = {};
        int mmax = 0;
        for (int a = 0; a < k; ++a) {
            LanczosProc& p = P[act[a]];
            const double* my = Um + (int64_t)a * len;
            if (use_precond) RPBD_TRY(precond_apply_impl(h, 1, my, p.w, st));
            else if (k > 1) RPBD_CU(h, cudaMemcpyAsync(p.w, my, sizeof(double) * len, cudaMemcpyDeviceToDevice, st));
            ++p.matvecs;
            OrthoProc& o = B.p[a];
            o.V = p.V;
            o.w = p.w;
            o.part = p.S.partial();
            o.h = p.S.hcol();
            o.vnext = p.V + (int64_t)(p.m + 1) * len;
            o.nv = p.m + 1;
            o.alpha = p.alpha;
            o.beta = p.beta;
            o.c = p.cvec;
            o.c_prev = p.cprev;
            o.host = h->host_small + 2 * a;
            mmax = std::max(mmax, p.m + 1);
        }
        const OrthoGrid G = launch_ortho(len, k, B, st);
        launch_pdl(lanczos_finish_kernel, dim3((unsigned)G.blocks + 1, (unsigned)k), 256,
                   tridiag_sqrt_smem_doubles(mmax) * sizeof(double), st, len, G.slice,
                   (const SqrtNode*)h->sqrt_nodes, B);
        count_launch();
        RPBD_LAUNCH_CHECK(h);
        RPBD_CU(h, cudaStreamSynchronize(st));
        for (int a = 0; a < k; ++a) {
            LanczosProc& p = P[act[a]];
            const double w2 = h->host_small[2 * a], ch = h->host_small[2 * a + 1];
            bool stop = false;
            if (p.m >= 1) {
                p.change = ch;
                if (ch < tol) { p.status = RPBD_OK; stop = true; }
            }
            if (!stop && !(w2 > 1e-300 * p.W2)) { p.status = RPBD_OK; stop = true; }  // invariant subspace: exact
            if (!stop && p.m + 1 >= max_iter) stop = true;
            if (stop) {
                p.active = false;
                // y = |W| V c, out = L y
                const int nv = p.m + 1;
                lincomb_kernel<<<g, 256, 0, st>>>(len, p.V, len, nv, p.cvec, std::sqrt(p.W2),
                                                  use_precond ? p.y : p.out);
                count_launch();
                if (use_precond) RPBD_TRY(precond_apply_impl(h, 0, p.y, p.out, st));
            } else {
                ++p.m;
            }
        }
        RPBD_LAUNCH_CHECK(h);
    }
    RPBD_TRY(check_flag(h, st));
    bool all_ok = true;
    for (int s = 0; s < nsys; ++s) {
        const LanczosProc& p = P[s];
        if (stats)
            stats[s] = p.W2 > 0.0 ? rpbd_stats{p.m + 1, p.matvecs, p.m >= 1 ? p.change : 0.0, p.status}
                                  : rpbd_stats{0, 0, 0.0, RPBD_OK};
        all_ok = all_ok && p.status == RPBD_OK;
    }
    return all_ok ? RPBD_OK : RPBD_NOT_CONVERGED;
}

int lanczos_impl(rpbd_handle* h, int64_t n, const double* r, const double* W, double* out, double tol, int max_iter,
                 int dtype, int use_precond, rpbd_stats* stats, cudaStream_t st)
{
    return lanczos_multi_impl(h, n, r, 1, &W, &out, tol, max_iter, dtype, use_precond, stats, st);
}

// ---------------------------------------------------------------------------
// GMRES on the saddle system
//
// Each GMRES process is a small state machine; a driver advances several
// processes that share the positions (same M, K and preconditioner) in
// lockstep, so that their matvecs go out as one multi-RHS launch (k =
// number of processes needing one), and reads every process's residual with
// one host synchronisation per iteration.

struct GmresProc {
    GmresProblem pb;
    double *V, *x, *b, *w, *zl, *zU, *sc;
    Small S{nullptr, 0};
    enum Phase { NEED_RESID, NEED_ARNOLDI, READ_START, READ_ITER, DONE } phase = DONE;
    int j = 0, total = 0, matvecs = 0, status = RPBD_NOT_CONVERGED;
    double res = 1.0;
    const double *req_l = nullptr, *req_U = nullptr;  // vector whose saddle product is wanted
    bool z_ready = false;                             // z = P^-1 v_j already there
};

int gmres_multi_impl(rpbd_handle* h, int64_t nb, int nper, const double* r, const double* q, int nsys,
                     const GmresProblem* probs, int restart, int dtype, int build_precond, rpbd_stats* stats,
                     cudaStream_t st)
{
    if (nb <= 0 || nper <= 0) return set_error(h, RPBD_BAD_ARG, "gmres: no bodies");
    if (restart < 1 || restart > 200) return set_error(h, RPBD_BAD_ARG, "gmres: bad restart");
    if (nsys < 1 || nsys > 4) return set_error(h, RPBD_BAD_ARG, "gmres: 1..4 systems");
    for (int s = 0; s < nsys; ++s)
        if (probs[s].max_iter < 1 || !probs[s].lambda || !probs[s].U)
            return set_error(h, RPBD_BAD_ARG, "gmres: bad max_iter or null output");
    const int64_t n = nb * nper;
    if (!r || !q) return set_error(h, RPBD_BAD_ARG, "gmres: null positions");
    RPBD_TRY(check_finite(h, 3 * (int64_t)nb * nper, r, st));
    if (build_precond) RPBD_TRY(precond_build_impl(h, nb, nper, r, q, st));
    if (!h->prec_valid || h->prec_nb != nb || h->prec_nper != nper)
        return set_error(h, RPBD_BAD_ARG, "gmres: preconditioner not built for these bodies");
    const int64_t len = 3 * n + 6 * nb;
    const int mdim = restart;
    double *Vall, *vall, *small, *mv = nullptr;
    RPBD_TRY(ensure_t(h, BUF_KRYLOV, (size_t)nsys * (mdim + 1) * len, &Vall));
    RPBD_TRY(ensure_t(h, BUF_VEC, (size_t)nsys * 4 * len, &vall));
    const size_t small_count = Small::count(mdim, len);
    RPBD_TRY(ensure_t(h, BUF_SMALL, (size_t)nsys * small_count, &small));
    if (nsys > 1) RPBD_TRY(ensure_t(h, BUF_GMRES_MV, (size_t)2 * nsys * 3 * n, &mv));
    GmresProc P[4];
    const unsigned g = vgrid(len);
    RPBD_CU(h, cudaMemsetAsync(h->dev_flag, 0, sizeof(int), st));

    // r0 = w: |r0|, g, residual estimate, v_0 (first: |b| = |r0|)
    auto begin_cycle = [&](GmresProc& p, int first) -> int {
        RPBD_TRY(multidot(h, len, p.w, 0, 1, p.w, &p.sc[0], p.S.partial(), st));
        gmres_start_kernel<<<1, 64, 0, st>>>(mdim, &p.sc[0], p.S.g(), p.sc, first, h->host_small + 2 * (&p - P));
        count_launch();
        normalize_kernel<<<g, 256, 0, st>>>(len, p.w, &p.sc[0], p.V); count_launch();
        RPBD_LAUNCH_CHECK(h);
        p.phase = GmresProc::READ_START;
        return RPBD_OK;
    };
    // x += P^-1 V y over the cycle's jn Arnoldi vectors
    auto end_cycle = [&](GmresProc& p, int jn) -> int {
        gmres_backsolve_kernel<<<1, 64, jn * sizeof(double), st>>>(jn, mdim, p.S.H(), p.S.g(), p.S.y()); count_launch();
        lincomb_kernel<<<g, 256, 0, st>>>(len, p.V, len, jn, p.S.y(), 1.0, p.w); count_launch();
        const PrecSaddle ps{p.w, p.w + 3 * n, p.zl, p.zU};
        p.z_ready = false;
        RPBD_TRY(precond_saddle_impl(h, 1, &ps, st));
        add_kernel<<<g, 256, 0, st>>>(3 * n, p.zl, p.x); count_launch();
        add_kernel<<<vgrid(6 * nb), 256, 0, st>>>(6 * nb, p.zU, p.x + 3 * n); count_launch();
        RPBD_LAUNCH_CHECK(h);
        return RPBD_OK;
    };
    auto want_resid = [&](GmresProc& p) {  // the product with x
        p.req_l = p.x;
        p.req_U = p.x + 3 * n;
        p.phase = GmresProc::NEED_RESID;
    };

    for (int s = 0; s < nsys; ++s) {
        GmresProc& p = P[s];
        p.pb = probs[s];
        p.V = Vall + (int64_t)s * (mdim + 1) * len;
        p.x = vall + (int64_t)s * 3 * len;
        p.b = p.x + len;
        p.w = p.x + 2 * len;
        // the blob parts of all processes' z lie side by side: a k-RHS matvec takes them as they are
        p.zl = vall + (int64_t)nsys * 3 * len + (int64_t)s * 3 * n;
        p.zU = vall + (int64_t)nsys * (3 * len + 3 * n) + (int64_t)s * 6 * nb;
        p.S = Small{small + (int64_t)s * small_count, mdim};
        p.sc = p.S.scal();  // [0] |.|^2, [1] |b|, [2] residual estimate
        // b = [-slip; -FT]
        if (p.pb.slip) launch_scale_copy(3 * n, -1.0, p.pb.slip, p.b, st);
        else RPBD_CU(h, cudaMemsetAsync(p.b, 0, sizeof(double) * 3 * n, st));
        if (p.pb.FT) launch_scale_copy(6 * nb, -1.0, p.pb.FT, p.b + 3 * n, st);
        else RPBD_CU(h, cudaMemsetAsync(p.b + 3 * n, 0, sizeof(double) * 6 * nb, st));
        if (p.pb.warm) {
            // x0 = [lambda; U] as given; |b| is the scale of the stopping test, as for x0 = 0
            RPBD_CU(h, cudaMemcpyAsync(p.x, p.pb.lambda, sizeof(double) * 3 * n, cudaMemcpyDeviceToDevice, st));
            RPBD_CU(h, cudaMemcpyAsync(p.x + 3 * n, p.pb.U, sizeof(double) * 6 * nb, cudaMemcpyDeviceToDevice, st));
            RPBD_TRY(multidot(h, len, p.b, 0, 1, p.b, &p.sc[0], p.S.partial(), st));
            gmres_start_kernel<<<1, 64, 0, st>>>(mdim, &p.sc[0], p.S.g(), p.sc, 1, h->host_small + 2 * s); count_launch();
            want_resid(p);
        } else {
            RPBD_CU(h, cudaMemsetAsync(p.x, 0, sizeof(double) * len, st));
            launch_scale_copy(len, 1.0, p.b, p.w, st);
            RPBD_TRY(begin_cycle(p, 1));
        }
    }

    for (;;) {
        // residuals of every process waiting for one: one synchronisation
        bool read = false;
        for (int s = 0; s < nsys; ++s)
            read = read || P[s].phase == GmresProc::READ_START || P[s].phase == GmresProc::READ_ITER;
        if (read) RPBD_CU(h, cudaStreamSynchronize(st));
        PrecSaddle ps[4];
        int nps = 0;
        auto want_arnoldi = [&](GmresProc& p) {  // z = P^-1 v_j, and the product with it
            const double* v = p.V + (int64_t)p.j * len;
            if (!p.z_ready) ps[nps++] = PrecSaddle{v, v + 3 * n, p.zl, p.zU};
            p.z_ready = false;
            p.req_l = p.zl;
            p.req_U = p.zU;
            p.phase = GmresProc::NEED_ARNOLDI;
        };
        for (int s = 0; s < nsys; ++s) {
            GmresProc& p = P[s];
            const double bn = h->host_small[2 * s], res = h->host_small[2 * s + 1];
            if (p.phase == GmresProc::READ_START) {
                p.res = res;
                if (!(bn > 0.0)) {  // zero right-hand side: zero solution
                    RPBD_CU(h, cudaMemsetAsync(p.x, 0, sizeof(double) * len, st));
                    p.res = 0.0;
                    p.status = RPBD_OK;
                    p.phase = GmresProc::DONE;
                } else if (res <= p.pb.tol) {
                    p.status = RPBD_OK;
                    p.phase = GmresProc::DONE;
                } else if (p.total >= p.pb.max_iter) {
                    p.phase = GmresProc::DONE;
                } else {
                    p.j = 0;
                    want_arnoldi(p);
                }
            } else if (p.phase == GmresProc::READ_ITER) {
                p.res = res;
                ++p.total;
                const int jn = p.j + 1;
                if (res <= p.pb.tol || jn == mdim || p.total >= p.pb.max_iter) {
                    RPBD_TRY(end_cycle(p, jn));
                    if (res <= p.pb.tol) {
                        p.status = RPBD_OK;
                        p.phase = GmresProc::DONE;
                    } else if (p.total >= p.pb.max_iter) {
                        p.phase = GmresProc::DONE;
                    } else {
                        want_resid(p);  // restart: r0 = b - A x
                    }
                } else {
                    p.j = jn;
                    want_arnoldi(p);
                }
            }
        }
        if (nps) RPBD_TRY(precond_saddle_impl(h, nps, ps, st));
        // one matvec for every process that needs one
        int act[4], k = 0;
        for (int s = 0; s < nsys; ++s)
            if (P[s].phase == GmresProc::NEED_RESID || P[s].phase == GmresProc::NEED_ARNOLDI) act[k++] = s;
        if (k == 0) break;
        const double* Fm = P[act[0]].req_l;
        double* Um = k == 1 ? P[act[0]].w : mv;
        bool side = true;  // operands already side by side
        for (int a = 1; a < k; ++a) side = side && P[act[a]].req_l == Fm + (int64_t)a * 3 * n;
        if (!side) {
            for (int a = 0; a < k; ++a)
                RPBD_CU(h, cudaMemcpyAsync(mv + (int64_t)(k + a) * 3 * n, P[act[a]].req_l, sizeof(double) * 3 * n,
                                           cudaMemcpyDeviceToDevice, st));
            Fm = mv + (int64_t)k * 3 * n;
        }
        RPBD_TRY(mobility_apply_impl(h, n, r, Fm, Um, k, dtype, true, st));
        SaddleBatch SB = {};
        OrthoBatch B = {};
        int no = 0;
        for (int a = 0; a < k; ++a) {
            GmresProc& p = P[act[a]];
            SB.p[a] = SaddleProd{Um + (int64_t)a * 3 * n, p.req_l, p.req_U, p.w};
        }
        const int G = nper <= 8 ? 8 : nper <= 16 ? 16 : 32, per = SADDLE_THREADS / G;
        launch_pdl(G == 8 ? saddle_kernel<8> : G == 16 ? saddle_kernel<16> : saddle_kernel<32>,
                   dim3((unsigned)((nb + per - 1) / per), (unsigned)k), SADDLE_THREADS, 0, st, nb, nper, r, q, SB);
        count_launch();
        for (int a = 0; a < k; ++a) {
            GmresProc& p = P[act[a]];
            ++p.matvecs;
            if (p.phase == GmresProc::NEED_RESID) {
                launch_axpby(len, 1.0, p.b, -1.0, p.w, p.w, st);
                RPBD_TRY(begin_cycle(p, 0));
            } else {
                // Arnoldi: classical Gram-Schmidt twice, Givens, residual estimate
                OrthoProc& o = B.p[no++];
                o.V = p.V;
                o.w = p.w;
                o.part = p.S.partial();
                o.h = p.S.hcol();
                o.vnext = p.V + (int64_t)(p.j + 1) * len;
                o.nv = p.j + 1;
                o.H = p.S.H();
                o.cs = p.S.cs();
                o.sn = p.S.sn();
                o.g = p.S.g();
                o.sc = p.sc;
                o.zl = p.zl;
                o.zU = p.zU;
                p.z_ready = true;
                o.host = h->host_small + 2 * act[a];
                p.phase = GmresProc::READ_ITER;
            }
        }
        if (no) {
            const OrthoGrid G = launch_ortho(len, no, B, st);
            launch_pdl(gmres_finish_kernel, dim3((unsigned)nb + 1, (unsigned)no), APPLY_THREADS,
                       3 * (size_t)(mdim + 2) * sizeof(double), st, nper, n, G.blocks, mdim, prec_factors(h), B);
            count_launch();
            RPBD_LAUNCH_CHECK(h);
        }
    }
    RPBD_TRY(check_flag(h, st));
    bool all_ok = true;
    for (int s = 0; s < nsys; ++s) {
        GmresProc& p = P[s];
        RPBD_CU(h, cudaMemcpyAsync(p.pb.lambda, p.x, sizeof(double) * 3 * n, cudaMemcpyDeviceToDevice, st));
        RPBD_CU(h, cudaMemcpyAsync(p.pb.U, p.x + 3 * n, sizeof(double) * 6 * nb, cudaMemcpyDeviceToDevice, st));
        if (stats) stats[s] = rpbd_stats{p.total, p.matvecs, p.res, p.status};
        all_ok = all_ok && p.status == RPBD_OK;
    }
    return all_ok ? RPBD_OK : RPBD_NOT_CONVERGED;
}

int gmres_impl(rpbd_handle* h, int64_t nb, int nper, const double* r, const double* q, const double* slip,
               const double* FT, double* lambda, double* U, double tol, int max_iter, int restart, int dtype,
               int build_precond, int warm, rpbd_stats* stats, cudaStream_t st)
{
    const GmresProblem pb{slip, FT, lambda, U, tol, max_iter, warm};
    return gmres_multi_impl(h, nb, nper, r, q, 1, &pb, restart, dtype, build_precond, stats, st);
}

}  // namespace rpbd

using namespace rpbd;

extern "C" {

int rpbd_lanczos_sqrt_apply(rpbd_handle* h, int64_t n, const double* r, const double* W, double* out, double tol,
                            int max_iter, int dtype, int use_precond, rpbd_stats* stats, void* stream)
{
    if (!h) return RPBD_BAD_ARG;
    if (!r || !W || !out) return set_error(h, RPBD_BAD_ARG, "lanczos: null pointer");
    if (!(tol > 0)) return set_error(h, RPBD_BAD_ARG, "lanczos: tol must be > 0");
    if (dtype != RPBD_F32 && dtype != RPBD_F64) return set_error(h, RPBD_BAD_ARG, "lanczos: bad dtype");
    return lanczos_impl(h, n, r, W, out, tol, max_iter, dtype, use_precond, stats,
                        reinterpret_cast<cudaStream_t>(stream));
}

int rpbd_lanczos_sqrt_apply_multi(rpbd_handle* h, int64_t n, const double* r, int nsys, const double* const* W,
                                  double* const* out, double tol, int max_iter, int dtype, int use_precond,
                                  rpbd_stats* stats, void* stream)
{
    if (!h) return RPBD_BAD_ARG;
    if (!r || !W || !out) return set_error(h, RPBD_BAD_ARG, "lanczos_multi: null pointer");
    if (!(tol > 0)) return set_error(h, RPBD_BAD_ARG, "lanczos_multi: tol must be > 0");
    if (dtype != RPBD_F32 && dtype != RPBD_F64) return set_error(h, RPBD_BAD_ARG, "lanczos_multi: bad dtype");
    return lanczos_multi_impl(h, n, r, nsys, W, out, tol, max_iter, dtype, use_precond, stats,
                              reinterpret_cast<cudaStream_t>(stream));
}

int rpbd_gmres_rigid_solve_multi(rpbd_handle* h, int64_t nb, int nper, const double* r, const double* q, int nsys,
                                 const double* const* slip, const double* const* FT, double* const* lambda,
                                 double* const* U, double tol, int max_iter, int restart, int dtype,
                                 int build_precond, rpbd_stats* stats, void* stream)
{
    if (!h) return RPBD_BAD_ARG;
    if (!r || !q || nsys < 1 || nsys > 4 || !slip || !FT || !lambda || !U)
        return set_error(h, RPBD_BAD_ARG, "gmres_multi: bad arguments");
    if (!(tol > 0)) return set_error(h, RPBD_BAD_ARG, "gmres_multi: tol must be > 0");
    if (dtype != RPBD_F32 && dtype != RPBD_F64) return set_error(h, RPBD_BAD_ARG, "gmres_multi: bad dtype");
    GmresProblem pb[4];
    for (int s = 0; s < nsys; ++s) {
        if (!lambda[s] || !U[s]) return set_error(h, RPBD_BAD_ARG, "gmres_multi: null output");
        pb[s] = GmresProblem{slip[s], FT[s], lambda[s], U[s], tol, max_iter, 0};
    }
    return gmres_multi_impl(h, nb, nper, r, q, nsys, pb, restart, dtype, build_precond, stats,
                            reinterpret_cast<cudaStream_t>(stream));
}

int rpbd_gmres_rigid_solve(rpbd_handle* h, int64_t nb, int nper, const double* r, const double* q, const double* slip,
                           const double* FT, double* lambda, double* U, double tol, int max_iter, int restart,
                           int dtype, int build_precond, int warm_start, rpbd_stats* stats, void* stream)
{
    if (!h) return RPBD_BAD_ARG;
    if (!r || !q || !lambda || !U) return set_error(h, RPBD_BAD_ARG, "gmres: null pointer");
    if (!(tol > 0)) return set_error(h, RPBD_BAD_ARG, "gmres: tol must be > 0");
    if (dtype != RPBD_F32 && dtype != RPBD_F64) return set_error(h, RPBD_BAD_ARG, "gmres: bad dtype");
    return gmres_impl(h, nb, nper, r, q, slip, FT, lambda, U, tol, max_iter, restart, dtype, build_precond,
                      warm_start ? 1 : 0, stats, reinterpret_cast<cudaStream_t>(stream));
}

}  // extern "C"
