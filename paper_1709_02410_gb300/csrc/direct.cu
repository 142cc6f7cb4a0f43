// FP32 wall-RPY matvec of a small system in one launch (k <= 4, wall, open or
// periodic cell).
//
// Up to a couple of thousand blobs the packed symmetric matvec (sym.cu) is three
// short kernels whose starts, tails and chains cost several times its
// arithmetic.  Here every CTA converts all sources into shared memory itself
// (positions split into FP32 hi/lo by integer operations on the double's bits:
// the FP64 conversions and subtractions, ~12 per source at ~19 cycles a warp
// instruction, would be most of the kernel), the CTA's eight warps share one to
// eight pairs of targets, a warp's lanes striding over its share of the sources
// with both targets' blocks in packed two-wide FP32 (wall_rpy_x2.cuh), and the
// sums are added by shuffles and across warps in a fixed order: no packing kernel,
// no atomics, no reduction kernel, deterministic.  It does every block twice and
// converts every source in every CTA, so it stops paying off where that counts.
//
// What bounds it are the loads of the conversion (every thread has two to four
// sources in flight at once: with single ones where fewer are left 300 blobs took
// 5.9 us, now 4.6, 840 15.7, now 9.8) and the few FP64 instructions left.
//
// Device time of a call, sym.cu -> here, open cell, k = 1: 240 blobs 11.9 -> 3.8 us,
// 600 12.7 -> 6.6, 960 12.2 -> 10.2; k = 2: 13.4 -> 4.7, 14.1 -> 9.3, 14.3 -> 13.9;
// k = 4: 16.3 -> 7.1, 600 18.4 -> 14.4.  Periodic, against sym.cu's 25.5 (k = 1),
// 27.2 and 33.8 us at 1,080 blobs: 240 4.7, 5.7 and 7.9, 600 10.9, 13.7 and 19.0, 960
// 22.9 and 27.5.
#include <cuda_runtime.h>

#include "rpbd_internal.cuh"
#include "wall_rpy_x2.cuh"

namespace rpbd {
namespace direct {

constexpr int NT = 256;

// x = hi + lo to 2^-46: hi the leading 24 bits of x, lo the remaining 29 rounded
__device__ __forceinline__ void split(double x, float& hi, float& lo)
{
    const long long u = __double_as_longlong(x);
    const int e = (int)((u >> 52) & 0x7ff) - 896;  // FP32 exponent field
    if (e > 40 && e < 255) {  // (lo's exponent field stays normal)
        const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
        hi = __uint_as_float(sign | ((unsigned)e << 23) | ((unsigned)(u >> 29) & 0x7fffffu));
        const float l = (float)((int)u & 0x1fffffff);  // times 2^(e - 127 - 52)
        lo = __uint_as_float(__float_as_uint(l * __int_as_float((e - 52 + 12) << 23)) | sign) * 0x1p-12f;
    } else {  // tiny, zero, huge or not finite
        hi = (float)x;
        lo = e >= 255 ? hi - hi : (float)(x - (double)hi);
    }
}

template <int K, bool PER, class In, class Out>
__global__ void __launch_bounds__(NT) direct_kernel(int n, int k, int tp, const double* r, const In* F, double a, double ia,
                                                    double s_min, float Lx, float Ly, double inv8pieta, Out* U)
{
    extern __shared__ float sm[];  // fields x_hi, y_hi, x_lo, y_lo, z~/a, s F of [n]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_wait();
    pdl_trigger();
    float* f = sm + 5 * n;
    bool bad = false;
    constexpr int U4 = K == 1 ? 4 : 2;  // sources a thread has in flight, also at the end
    for (int i0 = tid; i0 < n; i0 += U4 * NT) {
        double x[U4], y[U4], zs[U4];
        In g[U4][3 * K];
#pragma unroll
        for (int u = 0; u < U4; ++u) {
            const int i = min(i0 + u * NT, n - 1);
            x[u] = r[i];
            y[u] = r[n + i];
            zs[u] = r[2 * n + i];
#pragma unroll
            for (int q = 0; q < 3 * K; ++q) g[u][q] = q < 3 * k ? F[(int64_t)q * n + i] : In(0);
        }
#pragma unroll
        for (int u = 0; u < U4; ++u) {
            const int i = i0 + u * NT;
            if (i >= n) break;
            float h, l;
            split(x[u], h, l);
            sm[i] = h;
            sm[2 * n + i] = l;
            split(y[u], h, l);
            sm[n + i] = h;
            sm[3 * n + i] = l;
            const double z = zs[u];
            const bool below = !(z >= a);  // overlaps the wall, or NaN (stays NaN)
            sm[4 * n + i] = (float)((below ? a : z) * ia);
            double s = 1.0;
            if (below) {
                const double t = z * ia;  // (an FP64 divide is ~40 instructions)
                s = t >= 1.0 ? 1.0 : (t <= s_min ? s_min : t);
            }
#pragma unroll
            for (int q = 0; q < 3 * K; ++q) {
                const float v = below ? (float)(s * (double)g[u][q]) : (float)g[u][q];
                bad = bad || !isfinite(v);
                f[q * n + i] = v;
            }
        }
    }
    bad = __syncthreads_or(bad);  // a force that is not finite: U is NaN everywhere, as in sym.cu
    const PairConstX2 pc = PairConstX2::make_unit();
    const float2 m1 = pc.m1, ia2 = bc2((float)ia);
    const int wp = NT / 32 / tp;                                     // warps per pair of targets
    const int t0 = ((int)blockIdx.x * tp + warp / wp) * 2, t1 = t0 + 1;
    const int c0 = min(t0, n - 1), c1 = min(t1, n - 1);
    const float2 xh = make_float2(sm[c0], sm[c1]), yh = make_float2(sm[n + c0], sm[n + c1]);
    const float2 xl = make_float2(sm[2 * n + c0], sm[2 * n + c1]), yl = make_float2(sm[3 * n + c0], sm[3 * n + c1]);
    const float2 zi = make_float2(sm[4 * n + c0], sm[4 * n + c1]);
    float2 acc[3 * K];
#pragma unroll
    for (int q = 0; q < 3 * K; ++q) acc[q] = make_float2(0.0f, 0.0f);
#pragma unroll(PER || K > 2 ? 1 : 2)
    for (int j = (warp % wp) * 32 + lane; j < n; j += 32 * wp) {
        const float2 zj = bc2(sm[4 * n + j]);
        float2 dx = add2(fma2(m1, bc2(sm[j]), xh), fma2(m1, bc2(sm[2 * n + j]), xl));
        float2 dy = add2(fma2(m1, bc2(sm[n + j]), yh), fma2(m1, bc2(sm[3 * n + j]), yl));
        const float2 dz = fma2(m1, zj, zi);
        dx = mul2(dx, ia2);
        dy = mul2(dy, ia2);
        if constexpr (PER) {
            const float iLx = 1.0f / Lx, iLy = 1.0f / Ly;
            dx = make_float2(dx.x - Lx * rintf(dx.x * iLx), dx.y - Lx * rintf(dx.y * iLx));
            dy = make_float2(dy.x - Ly * rintf(dy.x * iLy), dy.y - Ly * rintf(dy.y * iLy));
            ImageBlock2 M;
            pair_image_sum_x2<false>(dx, dy, dz, zi, zj, Lx, Ly, pc, M);
#pragma unroll
            for (int m = 0; m < K; ++m) {
                const float2 fx = bc2(f[3 * m * n + j]), fy = bc2(f[(3 * m + 1) * n + j]), fz = bc2(f[(3 * m + 2) * n + j]);
                acc[3 * m + 0] = fma2(M.xz, fz, fma2(M.xy, fy, fma2(M.xx, fx, acc[3 * m + 0])));
                acc[3 * m + 1] = fma2(M.yz, fz, fma2(M.yy, fy, fma2(M.xy, fx, acc[3 * m + 1])));
                acc[3 * m + 2] = fma2(M.zz, fz, fma2(M.zy, fy, fma2(M.zx, fx, acc[3 * m + 2])));
            }
        } else {
            float2 al, be, gx, gz, mzz;
            pair_factors_x2<false>(dx, dy, dz, zi, zj, pc, al, be, gx, gz, mzz);
#pragma unroll
            for (int m = 0; m < K; ++m) {
                const float2 fx = bc2(f[3 * m * n + j]), fy = bc2(f[(3 * m + 1) * n + j]), fz = bc2(f[(3 * m + 2) * n + j]);
                const float2 P = fma2(dy, fy, mul2(dx, fx));
                const float2 Q = fma2(be, P, mul2(gx, fz));
                acc[3 * m + 0] = fma2(dx, Q, fma2(al, fx, acc[3 * m + 0]));
                acc[3 * m + 1] = fma2(dy, Q, fma2(al, fy, acc[3 * m + 1]));
                acc[3 * m + 2] = fma2(mzz, fz, fma2(gz, P, acc[3 * m + 2]));
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 3 * K; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            acc[q].x += __shfl_xor_sync(0xffffffffu, acc[q].x, o);
            acc[q].y += __shfl_xor_sync(0xffffffffu, acc[q].y, o);
        }
    }
    // the pair's warps in order; thread (target of the CTA, component)
    __shared__ float part[NT / 32][3 * K][2];
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < 3 * K; ++q) {
            part[warp][q][0] = acc[q].x;
            part[warp][q][1] = acc[q].y;
        }
    __syncthreads();
    const int tl = tid / (3 * K), q = tid % (3 * K), t = (int)blockIdx.x * 2 * tp + tl;
    if (tl >= 2 * tp || t >= n || q >= 3 * k) return;
    float v = 0.0f;
    for (int w = 0; w < wp; ++w) v += part[(tl / 2) * wp + w][q][tl & 1];
    const double z = r[2 * (int64_t)n + t];
    double s = 1.0;
    if (!(z >= a)) {
        const double u = z * ia;
        s = u >= 1.0 ? 1.0 : (u <= s_min ? s_min : u);
    }
    U[(int64_t)q * n + t] = (Out)(bad || !isfinite(v) ? __longlong_as_double(0x7ff8000000000000LL) : s * inv8pieta * (double)v);
}

template <int K, bool PER, class In, class Out>
static int run(rpbd_handle* h, int n, const double* r, const In* F, Out* U, int k, cudaStream_t st)
{
    auto kern = direct_kernel<K, PER, In, Out>;
    const size_t smem = (size_t)(5 + 3 * K) * n * sizeof(float);  // (at most 43,520 bytes, see direct_takes)
    // pairs of targets per CTA: 1, 2, 4 or 8, about one CTA per SM
    int tp = 1;
    while (tp < 8 && n > 2 * tp * h->sm_count) tp *= 2;
    const double inv8pieta = 1.0 / (8.0 * 3.14159265358979323846 * h->p.eta * h->p.a);  // blocks in units of a
    if (h->profile) prof_begin(h, st);
    launch_pdl(kern, (unsigned)((n + 2 * tp - 1) / (2 * tp)), NT, smem, st, n, k, tp, r, F, h->p.a, 1.0 / h->p.a,
               h->p.s_min, (float)(h->p.Lx / h->p.a), (float)(h->p.Ly / h->p.a), inv8pieta, U);
    count_launch();
    if (h->profile) prof_end(h, st, PER ? 3 : 4, K, (double)n * (double)n);
    RPBD_LAUNCH_CHECK(h);
    return RPBD_OK;
}

template <class In, class Out>
static int dispatch(rpbd_handle* h, int n, const double* r, const In* F, Out* U, int k, cudaStream_t st)
{
    if (h->p.Lx > 0.0)
        return k == 1 ? run<1, true>(h, n, r, F, U, k, st) : k == 2 ? run<2, true>(h, n, r, F, U, k, st) : run<4, true>(h, n, r, F, U, k, st);
    return k == 1 ? run<1, false>(h, n, r, F, U, k, st) : k == 2 ? run<2, false>(h, n, r, F, U, k, st) : run<4, false>(h, n, r, F, U, k, st);
}

}  // namespace direct

// where the call is shorter this way (figures above): n <= 960, with three or
// four right-hand sides n <= 640
bool direct_takes(const rpbd_handle* h, int64_t n, int k)
{
    return h->p.wall && k <= 4 && n <= (k <= 2 ? 960 : 640);
}

int direct_apply_impl(rpbd_handle* h, int64_t n, const double* r, const void* F, void* U, int k, bool io_double, cudaStream_t st)
{
    if (io_double) return direct::dispatch(h, (int)n, r, (const double*)F, (double*)U, k, st);
    return direct::dispatch(h, (int)n, r, (const float*)F, (float*)U, k, st);
}

}  // namespace rpbd
