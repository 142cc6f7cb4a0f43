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
// lanes' sums (FP32, at most 32 terms) are added as compensated pairs (accum.cuh) by
// shuffles and across warps in a fixed order: no packing kernel, no atomics, no
// reduction kernel, deterministic, records and sums as precise as sym.cu's.  It does
// every block twice and converts every source in every CTA, so it stops paying off
// where that counts.
//
// What bounds it are the loads of the conversion (every thread has two to four
// sources in flight at once: with single ones where fewer are left 840 blobs took
// 15.7 us, now 10.2) and the few FP64 instructions left: x and y scaled by 1/a there
// and not in FP32 afterwards cost 0.1 us at 240 blobs and 0.3 at 960, the
// compensated sums 0.1.
//
// Device time of a call, sym.cu -> here, open cell, k = 1: 240 blobs 13.0 -> 4.3 us,
// 600 13.4 -> 7.4, 960 13.5 -> 11.1; k = 2: 14.4 -> 5.3, 15.1 -> 10.1, 15.1 -> 14.9;
// k = 4: 17.2 -> 7.3, 600 19.2 -> 15.1.  Periodic: 240 13.9 -> 5.2, 14.9 -> 6.2 and
// 17.2 -> 8.2, 600 18.2 -> 11.9, 19.6 -> 14.9 and 22.7 -> 19.8.
#include <cuda_runtime.h>

#include "accum.cuh"
#include "rpbd_internal.cuh"
#include "wall_rpy_x2.cuh"

namespace rpbd {
namespace direct {

constexpr int NT = 256;

// x = hi + lo, both rounded to nearest even, as (float)x and (float)(x - (double)hi)
__device__ __forceinline__ void split(double x, float& hi, float& lo)
{
    const long long u = __double_as_longlong(x);
    const int e = (int)((u >> 52) & 0x7ff) - 896;  // FP32 exponent field
    if (e > 60 && e < 254) {  // (lo is normal too; a carry leaves hi finite)
        const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
        const long long m = u & 0x7fffffffffffffffLL, h = (m + 0x0fffffff + ((m >> 29) & 1)) >> 29;
        hi = __uint_as_float(sign | ((unsigned)h - (896u << 23)));
        const float l = (float)(int)(m - (h << 29));  // times 2^(e - 127 - 52)
        lo = l * __uint_as_float(sign | ((unsigned)(e - 52) << 23));
    } else {  // tiny, zero, huge or not finite
        hi = (float)x;
        lo = (float)(x - (double)hi);
    }
}

// s + c += s2 + c2
__device__ __forceinline__ void two_sum_merge(float& s, float& c, float s2, float c2)
{
    two_sum_acc(s, c, s2);
    c = __fadd_rn(c, c2);
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
            split(x[u] * ia, h, l);
            sm[i] = h;
            sm[2 * n + i] = l;
            split(y[u] * ia, h, l);
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
    const float2 m1 = pc.m1;
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
    // the lanes' sums, as compensated pairs: halves of the sums (target, right-hand
    // side) to halves of the lanes down to three a lane, then those over the rest
    float v[6 * K], e[6 * K];
#pragma unroll
    for (int q = 0; q < 3 * K; ++q) {
        v[q] = acc[q].x;
        v[3 * K + q] = acc[q].y;
    }
#pragma unroll
    for (int q = 0; q < 6 * K; ++q) e[q] = 0.0f;
    int o = 16, g = 0;  // g: the lane's (target, right-hand side)
#pragma unroll
    for (int c = K; c > 0; c >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < 3 * c; ++i) {
            const float s2 = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[3 * c + i], o);
            const float e2 = __shfl_xor_sync(0xffffffffu, up ? e[i] : e[3 * c + i], o);
            v[i] = up ? v[3 * c + i] : v[i];
            e[i] = up ? e[3 * c + i] : e[i];
            two_sum_merge(v[i], e[i], s2, e2);
        }
        if (up) g += c;
    }
    const bool first = (lane & (2 * o - 1)) == 0;
#pragma unroll
    for (; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float s2 = __shfl_xor_sync(0xffffffffu, v[i], o), e2 = __shfl_xor_sync(0xffffffffu, e[i], o);
            two_sum_merge(v[i], e[i], s2, e2);
        }
    // the pair's warps in order; thread (target of the CTA, component)
    __shared__ float2 part[NT / 32][2][3 * K];
    if (first)
#pragma unroll
        for (int c = 0; c < 3; ++c) part[warp][g / K][g % K * 3 + c] = make_float2(v[c], e[c]);
    __syncthreads();
    const int tl = tid / (3 * K), q = tid % (3 * K), t = (int)blockIdx.x * 2 * tp + tl;
    if (tl >= 2 * tp || t >= n || q >= 3 * k) return;
    float sum = 0.0f, err = 0.0f;
    for (int w = 0; w < wp; ++w) {
        const float2 x = part[(tl / 2) * wp + w][tl & 1][q];
        two_sum_merge(sum, err, x.x, x.y);
    }
    const double z = r[2 * (int64_t)n + t];
    double s = 1.0;
    if (!(z >= a)) {
        const double u = z * ia;
        s = u >= 1.0 ? 1.0 : (u <= s_min ? s_min : u);
    }
    U[(int64_t)q * n + t] = (Out)(bad || !isfinite(sum) ? __longlong_as_double(0x7ff8000000000000LL) : s * inv8pieta * two_sum_value(sum, err));
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

// where the call is shorter this way: open cell n <= 960, with three or four
// right-hand sides 640; periodic cell, sym.cu -> here, k = 1 at 630 blobs 18.3 -> 17.1,
// at 690 18.3 -> 18.6, k = 2 and 4 at 600 as above, at 630 19.8 -> 20.5 and
// 22.7 -> 25.6 (beyond 608 a CTA has four pairs of targets instead of two)
bool direct_takes(const rpbd_handle* h, int64_t n, int k)
{
    if (!h->p.wall || k > 4) return false;
    return n <= (h->p.Lx > 0.0 ? (k == 1 ? 640 : 608) : (k <= 2 ? 960 : 640));
}

int direct_apply_impl(rpbd_handle* h, int64_t n, const double* r, const void* F, void* U, int k, bool io_double, cudaStream_t st)
{
    if (io_double) return direct::dispatch(h, (int)n, r, (const double*)F, (double*)U, k, st);
    return direct::dispatch(h, (int)n, r, (const float*)F, (float*)U, k, st);
}

}  // namespace rpbd
