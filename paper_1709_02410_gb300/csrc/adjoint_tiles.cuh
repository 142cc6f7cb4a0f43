// Symmetric gradient kernel: g_k = d(sum_m u_m^T M F_m)/d r_k.
//
// Every unordered pair is met once (adjoint_pair.cuh) and adds to both blobs:
// homes and visitors as in sym.cu -- home blobs in registers (one per lane in
// FP64, two in packed FP32), visitors in tiles of 32 through shared memory, lane
// l meets visitor (step + l) mod 32 and hands the visitor's running sums to lane
// l - 1 after every step.  Pairs inside a warp's own home blobs are done in the
// home direction only.  Sums of (dE/dx, dE/dy, dE/dz~, E) go to one partial row
// per (home tile, part) for the visitors and per (item, part) for the homes, added
// in a fixed order, so the result does not depend on the order of the CTAs.  FP64:
// by the last CTA to finish a blob tile (a ticket per tile, no CTA ever waits), in
// the same launch.  FP32, where the pairs are over sooner than one CTA has walked
// a tile's rows, by a kernel of its own (1,920 blobs 275 -> 49 us).
//
// Bound by arithmetic: the FP64 pipe, or packed FP32 issue (~160 operations per
// unordered pair).  Before, one thread per blob walked all sources with the block
// on dual numbers, so 1,920 blobs filled 15 of 152 SMs: FP64 gradient with its two
// matvecs 29.3 -> 1.30 ms at 1,920 blobs (FP64 pipe 85% busy); FP32 2.99 -> 0.78 ms
// at 16,380 (FMA pipe 78%).
//
// Cutting as in sym64.cu: CTAs of one warp for small n, four beyond, items of
// `chunk` visitor tiles, the 32 steps of a tile over `parts` items for very
// small n.  The partials stay under GROUP_BYTES (or MIN_ROWS rows, from 5 million
// blobs in FP64 and 11 in FP32): home tiles run in groups, for the visitors' rows;
// for the homes' rows, one per item, FP64 takes longer items and FP32, whose sums
// should not get longer, groups of items.  At 10^6 blobs the homes' rows alone
// would be 14.6 and 29 GiB.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "adjoint_pair.cuh"
#include "rpbd_internal.cuh"

namespace rpbd {
namespace adj {

constexpr int VT = 32;                            // visitor tile
constexpr double GROUP_BYTES = 4.0 * (1ull << 30);
constexpr int64_t MIN_ROWS = 24;  // 12 home tiles x 12 items a launch

// how one launch (a group of home tiles) is cut
struct Cut {
    int64_t n, n_pad;
    int nw, threads;   // warps with home blobs per CTA, threads per CTA
    int vpw, vph;      // visitor tiles per warp's home blobs, per home tile
    int tiles;         // visitor tiles
    int chunk, parts;  // visitor tiles per item (a power of two), items per tile's steps
    int h0, hg;        // first home tile, home tiles of the launch
    int i0, items;     // first item of every home tile, items of the launch
};

// one launch's outputs: G [4][n_pad] carries the sums between groups and passes
struct Out {
    double* G;
    int* ticket;          // one per home tile, zeroed before the launch
    double* grad;
    int first, last;      // first launch of the call (G not yet written), last pass
    double ig, ie;        // factors of dE/d(rt) and of E
};

template <class V>
struct Scalar { using S = double; };
template <>
struct Scalar<float2> { using S = float; };

// FP32 record of adjoint's pack kernel: x_hi, y_hi, x_lo, y_lo, z~, s F, s u, each
// duplicated, 16-byte chunk q of record j of a tile at (32 q + j)
template <int K>
struct Rec32 {
    static constexpr int NV = 5 + 6 * K, NCH = (NV + 1) / 2;
};

__device__ __forceinline__ double overlap_scale(double z, double a, double s_min)
{
    if (z >= a) return 1.0;
    const double t = z / a;  // NaN stays NaN
    return t >= 1.0 ? 1.0 : (t <= s_min ? s_min : t);
}

// g of blob i from its complete sums (q 0..3: dE/dx, dE/dy, dE/dz~, E); q 0, 1 or both of 2 and 3
__device__ __forceinline__ void write_xy(const Cut& c, const Out& o, int64_t i, int q, double s) { o.grad[q * c.n + i] = o.ig * s; }
__device__ __forceinline__ void write_z(const Cut& c, const Out& o, int64_t i, double sz, double se, const double* r, double a,
                                        int wall, double s_min)
{
    // z~ follows z from a upwards, s = z / a between s_min a and a
    const double z = r[2 * c.n + i];
    const bool above = !wall || z >= a, ramp = wall && z / a < 1.0 && z / a > s_min;
    const double dz = above || z != z ? o.ig * sz : 0.0;
    o.grad[2 * c.n + i] = dz + (ramp ? o.ie * se / z : 0.0);
}

// sum over rows e = e0, e0 + step, ... of one value, eight loads in flight
template <class S, class At>
__device__ __forceinline__ double sum_rows(int e0, int step, int rows, At at)
{
    double s = 0.0;
    int e = e0;
    for (; e + 7 * step < rows; e += 8 * step) {
        S v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldcg(at(e + u * step));
#pragma unroll
        for (int u = 0; u < 8; ++u) s += (double)v[u];
    }
    for (; e < rows; e += step) s += (double)__ldcg(at(e));
    return s;
}

// adds the rows of blob tile `home` (all threads of the CTA, one value each at a
// time), writes g when complete.  sm: 128 vph doubles of shared memory
template <class S>
__device__ void finish_tile(const Cut& c, const Out& o, int home, const S* partial, const double* r, double a, int wall,
                            double s_min, double* sm)
{
    const bool own = home >= c.h0 && home < c.h0 + c.hg;
    const int before = min(c.h0 + c.hg, home) - c.h0;  // home tiles of the group before this one
    const int nit = own ? (c.tiles - home * c.vph + c.chunk - 1) / c.chunk * c.parts : 0;
    const int ht = 32 * c.vph;
    for (int idx = threadIdx.x; idx < 4 * ht; idx += blockDim.x) {
        const int q = idx / ht, b = idx - q * ht;
        const int64_t i = (int64_t)home * ht + b;
        const int vis = (before + (own && b / 32 >= c.vpw ? 1 : 0)) * c.parts, shift = c.hg * c.parts - vis;
        const S* p = partial + q * c.n_pad + i;
        const int64_t ld = 4 * c.n_pad;
        double s = sum_rows<S>(0, 1, vis + nit, [&](int e) { return p + (e < vis ? e : e + shift) * ld; });
        if (!o.first) s += o.G[q * c.n_pad + i];
        if (!(own && o.last)) o.G[q * c.n_pad + i] = s;  // later groups' homes come after this tile
        sm[idx] = s;
    }
    __syncthreads();
    if (own && o.last)
        for (int idx = threadIdx.x; idx < 3 * ht; idx += blockDim.x) {
            const int q = idx / ht, b = idx - q * ht;
            const int64_t i = (int64_t)home * ht + b;
            if (i >= c.n) continue;
            if (q < 2) write_xy(c, o, i, q, sm[idx]);
            else write_z(c, o, i, sm[idx], sm[idx + ht], r, a, wall, s_min);
        }
    __syncthreads();
}

// the same for every tile, 32 blobs, one sum (blockIdx.y: x, y, z with E) and 8 row
// slices a block (the slices added in order)
constexpr int RS = 8;
template <class S>
__global__ void __launch_bounds__(32 * RS) adjoint_reduce_kernel(Cut c, Out o, const S* partial, const double* r, double a,
                                                                 int wall, double s_min)
{
    __shared__ double sm[2][RS][32];
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int vb = __ffs(c.vph) - 1, cb = __ffs(c.chunk) - 1;  // (powers of two)
    const int tile = blockIdx.x, home = tile >> vb, sub = tile - (home << vb), q0 = blockIdx.y, nq = q0 == 2 ? 2 : 1;
    if (home < c.h0) return;  // complete already
    const bool own = home < c.h0 + c.hg;
    const int64_t i = (int64_t)tile * VT + lane;
    // home tiles lo..hi of the launch met this tile in its items' range, the tile's own past its warps' own blobs
    const int beg = c.i0 << cb, end = beg + (c.items << cb);
    const int lo = max(c.h0, tile >= end ? ((tile - end) >> vb) + 1 : 0);
    int hi = min(c.h0 + c.hg - 1, own && sub >= c.vpw ? home : home - 1);
    hi = tile >= beg ? min(hi, (tile - beg) >> vb) : -1;
    const int vis = max(0, hi - lo + 1) * c.parts;
    const int its = (c.tiles - (home << vb) + c.chunk - 1) >> cb;
    const int rows = vis + (own ? max(0, min(its - c.i0, c.items)) * c.parts : 0);
    const int skip = (lo - c.h0) * c.parts, shift = c.hg * c.parts - vis;
    const int64_t ld = 4 * c.n_pad;
    for (int q = 0; q < nq; ++q) {
        const S* p = partial + (q0 + q) * c.n_pad + i;
        sm[q][y][lane] = sum_rows<S>(y, RS, rows, [&](int e) { return p + (e < vis ? e + skip : e + shift) * ld; });
    }
    __syncthreads();
    if (y || i >= c.n) return;
    double s[2] = {0.0, 0.0};
    for (int q = 0; q < nq; ++q) {
#pragma unroll
        for (int w = 0; w < RS; ++w) s[q] += sm[q][w][lane];
        double* G = o.G + (q0 + q) * c.n_pad + i;
        if (!o.first) s[q] += *G;
        if (!(own && o.last)) *G = s[q];
    }
    if (own && o.last) {
        if (q0 < 2) write_xy(c, o, i, q0, s[0]);
        else write_z(c, o, i, s[0], s[1], r, a, wall, s_min);
    }
}

// one visitor tile into shared memory.  FP64: fields x, y, z~, s F, s u of [32]
// doubles, straight from the caller's arrays; FP32: the packed records.
template <class V, int K>
__device__ __forceinline__ void load_tile(const Cut& c, int tile, int nr, const double* r, const double* u, const double* F,
                                          const float4* rec, double a, int wall, double s_min, void* st)
{
    if constexpr (std::is_same<V, double>::value) {
        double* o = static_cast<double*>(st);
        const int lane = threadIdx.x & 31;
        const int64_t i = (int64_t)tile * VT + lane;
        const bool real = i < c.n;
        const double z = real ? r[2 * c.n + i] : a;
        const double s = wall ? overlap_scale(z, a, s_min) : 1.0;
        for (int f = threadIdx.x >> 5; f < 3 + 6 * K; f += blockDim.x >> 5) {
            double v;
            if (f < 2) v = real ? r[f * c.n + i] : 1.0e7;  // padding: far away
            else if (f == 2) v = wall ? (z > a ? z : a) : z;
            else {
                const int q = f - 3, m = (q < 3 * K ? q : q - 3 * K);
                v = real && m < 3 * nr ? s * (q < 3 * K ? F : u)[(int64_t)m * c.n + i] : 0.0;
            }
            o[f * VT + lane] = v;
        }
    } else {
        constexpr int NCH = Rec32<K>::NCH;
        float4* o = static_cast<float4*>(st);
        const float4* src = rec + (int64_t)tile * VT * NCH;
        for (int e = threadIdx.x; e < VT * NCH; e += blockDim.x) o[e] = src[e];
    }
}

template <class V, int K, bool WALL, bool PER, class C>
__global__ void __launch_bounds__(128) adjoint_kernel(Cut c, int nr, const double* r, const double* u,
                                                      const double* F, const float4* rec, C k,
                                                      double a, double s_min, typename Scalar<V>::S Lx,
                                                      typename Scalar<V>::S Ly,
                                                      typename Scalar<V>::S* partial, Out out)
{
    using S = typename Scalar<V>::S;
    constexpr bool D = std::is_same<V, double>::value;
    constexpr int STAGE = D ? (3 + 6 * K) * VT * 8 : Rec32<K>::NCH * VT * 16;  // bytes
    extern __shared__ __align__(128) unsigned char smem_raw[];
    S* red = reinterpret_cast<S*>(smem_raw + 2 * STAGE);  // [2 buffers][nw][4][VT]
    const int home = c.h0 + blockIdx.x, item = blockIdx.y, part = blockIdx.z;
    const int tile0 = home * c.vph + (c.i0 + item) * c.chunk;  // visitors: the home tile's own blobs and all after them
    const int ntile = min(c.chunk, c.tiles - tile0);
    pdl_wait();
    pdl_trigger();
    if (ntile <= 0) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int s0 = VT / c.parts * part, s1 = s0 + VT / c.parts;

    load_tile<V, K>(c, tile0, nr, r, u, F, rec, a, WALL, s_min, smem_raw);
    // home blobs: 32 vpw per warp (warps past nw, in launches of few CTAs, only help to load and to add rows)
    const bool pairs = warp < c.nw;
    V hx, hy, hxl, hyl, hz, A[3 * K], B[3 * K];
    if constexpr (D) {
        const int64_t i = (int64_t)(home * c.vph + warp) * VT + lane;
        const bool real = pairs && i < c.n;
        const double z = real ? r[2 * c.n + i] : a, s = WALL ? overlap_scale(z, a, s_min) : 1.0;
        hx = real ? r[i] : 1.0e7;
        hy = real ? r[c.n + i] : 1.0e7;
        hz = WALL ? (z > a ? z : a) : z;
#pragma unroll
        for (int q = 0; q < 3 * K; ++q) {
            A[q] = real && q < 3 * nr ? s * u[(int64_t)q * c.n + i] : 0.0;
            B[q] = real && q < 3 * nr ? s * F[(int64_t)q * c.n + i] : 0.0;
        }
    } else {
        constexpr int NCH = Rec32<K>::NCH;
        const float4* p = rec + (int64_t)(home * c.vph + 2 * warp) * VT * NCH + lane;
        float2 v[2 * NCH];
#pragma unroll
        for (int q = 0; q < NCH; ++q) {
            const float4 x = p[q * VT], y = p[(NCH + q) * VT];
            v[2 * q] = make_float2(x.x, y.x);
            v[2 * q + 1] = make_float2(x.z, y.z);
        }
        hx = v[0]; hy = v[1]; hxl = v[2]; hyl = v[3]; hz = v[4];
#pragma unroll
        for (int q = 0; q < 3 * K; ++q) {
            B[q] = v[5 + q];
            A[q] = v[5 + 3 * K + q];
        }
    }
    const S iLx = PER ? S(1) / Lx : S(0), iLy = PER ? S(1) / Ly : S(0);
    (void)iLx;
    (void)iLy;
    const V zero = num_<V>(0.0);
    V acc[4] = {zero, zero, zero, zero};
    const int64_t row_v = ((int64_t)blockIdx.x * c.parts + part) * 4;
    for (int t = 0; t < ntile; ++t) {
        __syncthreads();  // tile t is in shared memory
        if (t + 1 < ntile)
            load_tile<V, K>(c, tile0 + t + 1, nr, r, u, F, rec, a, WALL, s_min, smem_raw + ((t + 1) & 1) * STAGE);
        const unsigned char* st = smem_raw + (t & 1) * STAGE;
        const int own = tile0 + t - home * c.vph;  // counted from the home tile's first
        S* rb = red + (t & 1) * (c.nw * 4 * VT);
        if (pairs && own >= warp * c.vpw) {
            const bool both = own >= (warp + 1) * c.vpw;
            V vacc[4] = {zero, zero, zero, zero};
#pragma unroll 1
            for (int step = s0; step < s1; ++step) {
                const int v = (step + lane) & (VT - 1);
                V dx, dy, zj;
                PairGrad<V> g;
                if constexpr (D) {
                    const double* p = reinterpret_cast<const double*>(st) + v;
                    dx = hx - p[0];
                    dy = hy - p[VT];
                    zj = p[2 * VT];
                    if constexpr (PER) {
                        dx -= Lx * rint(dx * iLx);
                        dy -= Ly * rint(dy * iLy);
                    }
                    pair_grad_images<WALL, PER, K>(dx, dy, hz, zj, k, Lx, Ly, A, B, [&](int q) { return p[(3 + q) * VT]; }, g);
                } else {
                    const float4* p = reinterpret_cast<const float4*>(st) + v;
                    const float4 p0 = p[0], p1 = p[VT], p2 = p[2 * VT];
                    const float2 m1 = bc2(-1.0f);
                    dx = add2(fma2(m1, make_float2(p0.x, p0.y), hx), fma2(m1, make_float2(p1.x, p1.y), hxl));
                    dy = add2(fma2(m1, make_float2(p0.z, p0.w), hy), fma2(m1, make_float2(p1.z, p1.w), hyl));
                    zj = make_float2(p2.x, p2.y);
                    if constexpr (PER) {
                        dx = make_float2(dx.x - Lx * rintf(dx.x * iLx), dx.y - Lx * rintf(dx.y * iLx));
                        dy = make_float2(dy.x - Ly * rintf(dy.x * iLy), dy.y - Ly * rintf(dy.y * iLy));
                    }
                    // value 5 + q sits in chunk (5 + q) / 2, lanes (0, 1) or (2, 3)
                    pair_grad_images<WALL, PER, K>(dx, dy, hz, zj, k, Lx, Ly, A, B, [&](int q) {
                        const float4 x = p[((5 + q) / 2) * VT];
                        return (5 + q) % 2 ? make_float2(x.z, x.w) : make_float2(x.x, x.y);
                    }, g);
                }
                acc[0] = add_(acc[0], g.x);
                acc[1] = add_(acc[1], g.y);
                acc[2] = add_(acc[2], g.zi);
                acc[3] = add_(acc[3], g.e);
                if (both) {
                    vacc[0] = sub_(vacc[0], g.x);
                    vacc[1] = sub_(vacc[1], g.y);
                    vacc[2] = add_(vacc[2], g.zj);
                    vacc[3] = add_(vacc[3], g.e);
                }
                // hand the visitor's sums to the lane that meets it next
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if constexpr (D) vacc[q] = __shfl_sync(0xffffffffu, vacc[q], (lane + 1) & 31);
                    else {
                        vacc[q].x = __shfl_sync(0xffffffffu, vacc[q].x, (lane + 1) & 31);
                        vacc[q].y = __shfl_sync(0xffffffffu, vacc[q].y, (lane + 1) & 31);
                    }
                }
            }
            // lane l holds the sums of visitor (l + s1) mod 32
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                S x;
                if constexpr (D) x = vacc[q];
                else x = vacc[q].x + vacc[q].y;
                rb[(warp * 4 + q) * VT + ((lane + s1) & (VT - 1))] = x;
            }
        }
        __syncthreads();
        if (own >= c.vpw) {  // warps that met this tile in both directions
            const int nm = min(own / c.vpw, c.nw);
            for (int e = tid; e < 4 * VT; e += blockDim.x) {
                const int q = e / VT, vl = e % VT;
                S sum = rb[q * VT + vl];
                for (int w = 1; w < nm; ++w) sum += rb[(w * 4 + q) * VT + vl];
                partial[(row_v + q) * c.n_pad + (int64_t)(tile0 + t) * VT + vl] = sum;
            }
        }
    }
    const int64_t row_h = ((int64_t)c.hg * c.parts + item * c.parts + part) * 4;
    const int64_t ib = (int64_t)(home * c.vph + warp * c.vpw) * VT + lane;
    if (pairs)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if constexpr (D) partial[(row_h + q) * c.n_pad + ib] = acc[q];
        else {
            partial[(row_h + q) * c.n_pad + ib] = acc[q].x;
            partial[(row_h + q) * c.n_pad + ib + VT] = acc[q].y;
        }
    }
    if constexpr (!D) return;  // (adjoint_reduce_kernel follows)
    // tickets of the blob tiles this item added to; the last one in finishes the tile
    __threadfence();
    __syncthreads();
    const int per_home = max(1, c.vph / c.chunk) * c.parts;  // items of one earlier home tile that meet a tile
    const int first = max(home + 1, tile0 / c.vph), last = (tile0 + ntile - 1) / c.vph;  // tiles visited past the home tile
    int* const ready = reinterpret_cast<int*>(red);
    for (int x = 0; x <= max(0, last - first + 1); ++x) {
        const int tile = x == 0 ? home : first + x - 1;
        __syncthreads();
        if (tid == 0) {
            const int homes = min(c.h0 + c.hg, tile) - c.h0;  // of this launch, before the tile
            const int own_items = tile < c.h0 + c.hg ? (c.tiles - tile * c.vph + c.chunk - 1) / c.chunk * c.parts : 0;
            *ready = atomicAdd(out.ticket + tile, 1) == homes * per_home + own_items - 1;
        }
        __syncthreads();
        const bool go = *ready != 0;
        __syncthreads();
        if (go) {
            __threadfence();
            finish_tile<S>(c, out, tile, partial, r, a, WALL, s_min, reinterpret_cast<double*>(red));
        }
    }
}

// cuts n blobs; vpw: visitor tiles per warp's home blobs (1: FP64, 2: packed FP32)
inline Cut cut(int64_t n, int vpw, int64_t small_n, int max_chunk, int sm_count)
{
    Cut c;
    c.n = n;
    c.nw = n <= small_n ? 1 : 4;
    c.vpw = vpw;
    c.vph = vpw * c.nw;
    const int64_t ht = 32 * c.vph;
    c.n_pad = (n + ht - 1) / ht * ht;
    c.tiles = (int)(c.n_pad / VT);
    const int T = c.tiles / c.vph;
    auto count = [&](int64_t ch) {
        int64_t m = 0;
        for (int64_t H = 0; H < T; ++H) m += (c.tiles - H * c.vph + ch - 1) / ch;
        return m;
    };
    c.chunk = max_chunk;
    while (c.chunk > 1 && count(c.chunk) < 16 * (int64_t)sm_count) c.chunk /= 2;
    c.parts = 1;
    while (c.parts < 4 && count(c.chunk) * c.parts < 16 * (int64_t)sm_count) c.parts *= 2;
    // few CTAs: help with the loads and sums, and steps over twice as many
    const bool few = count(c.chunk) * c.parts <= 4 * (int64_t)sm_count;
    if (few && vpw == 1) c.parts *= 2;
    c.threads = few && vpw == 1 ? 128 : 32 * c.nw;
    c.h0 = c.i0 = 0;
    c.hg = T;
    c.items = (c.tiles + c.chunk - 1) / c.chunk;
    return c;
}

// home tiles and items of a launch, half of the rows that fit for the items;
// longer: items may not be split into groups but take more visitor tiles
inline void group(Cut& c, int64_t rows, bool longer)
{
    const int T = c.tiles / c.vph;
    const int64_t most = std::min<int64_t>(65535, std::max(std::max<int64_t>(1, rows / 2), rows - T));
    if (longer)
        while ((c.tiles + c.chunk - 1) / c.chunk > most) c.chunk *= 2;
    c.items = (int)std::min<int64_t>((c.tiles + c.chunk - 1) / c.chunk, most);
    c.hg = (int)std::max<int64_t>(1, std::min<int64_t>(T, rows - c.items));
}

// all launches of one call: passes of up to four right-hand sides, groups of
// home tiles and of items.  pass(m0, kc): prepares pass m0 (FP32: packs its
// records); launch(c, kc, m0, out): one launch.
template <class S, class Pass, class Launch>
static int run_all(rpbd_handle* h, Cut c, int nr, double* grad, double ig, double ie, Pass pass, Launch launch, cudaStream_t st)
{
    constexpr bool tickets = sizeof(S) == 8;
    const int T = c.tiles / c.vph;
    unsigned char* base;
    const size_t g_bytes = sizeof(double) * 4 * c.n_pad, t_bytes = ((size_t)T * sizeof(int) + 15) / 16 * 16;
    const double row_bytes = 4.0 * sizeof(S) * (double)c.n_pad * c.parts;
    const Cut whole = c;
    double limit = GROUP_BYTES;
    for (;;) {  // smaller groups where device memory is short
        c = whole;
        group(c, std::max((int64_t)(limit / row_bytes), limit < GROUP_BYTES ? 2 : MIN_ROWS), tickets);
        const size_t part = (size_t)((int64_t)c.hg + c.items) * (size_t)row_bytes, bytes = part + g_bytes + t_bytes;
        const bool least = c.hg + c.items <= 2;
        if (least || worth_trying(h, BUF_PARTIAL, bytes, st)) {
            const int s = ensure_t(h, BUF_PARTIAL, bytes, &base);
            if (s == RPBD_OK) break;
            if (s != RPBD_NO_MEM || least) return s;
            cudaGetLastError();
        }
        limit = 0.5 * (double)part;
    }
    Out o;
    o.G = reinterpret_cast<double*>(base);
    o.ticket = reinterpret_cast<int*>(base + g_bytes);
    S* partial = reinterpret_cast<S*>(base + g_bytes + t_bytes);
    o.grad = grad;
    o.ig = ig;
    o.ie = ie;
    const int hg = c.hg, items = c.items;
    for (int m0 = 0; m0 < nr; m0 += 4) {
        const int kc = std::min(4, nr - m0);
        RPBD_TRY(pass(m0, kc));
        for (int h0 = 0; h0 < T; h0 += hg) {
            c.h0 = h0;
            c.hg = std::min(hg, T - h0);
            const int own = (c.tiles - h0 * c.vph + c.chunk - 1) / c.chunk;  // items of the first home tile, the most
            for (int i0 = 0; i0 < own; i0 += items) {
                if (tickets) RPBD_CU(h, cudaMemsetAsync(o.ticket, 0, t_bytes, st));
                c.i0 = i0;
                c.items = std::min(items, own - i0);
                o.first = m0 == 0 && h0 == 0 && i0 == 0;
                o.last = m0 + 4 >= nr && i0 + items >= own;
                RPBD_TRY(launch(c, kc, m0, partial, o));
                count_launch();
                RPBD_LAUNCH_CHECK(h);
            }
        }
    }
    return RPBD_OK;
}

}  // namespace adj
}  // namespace rpbd
