// Symmetric FP64 wall-RPY matvec (k <= 8 right-hand sides, up to four a pass).
//
// The FP64 pipe of this GPU starts a warp instruction about every 19 cycles per
// SM (1.05 TFLOP/s measured over the chip, 1/75 of FP32), so the kernel's time
// is its count of FP64 instructions, and everything here serves that count:
//  * M_ji = M_ij^T (Sec. 2.1): each unordered pair's block is formed once and
//    applied both ways in factored form -- 42 instructions for the block's five
//    scalars, 10 for its two reciprocal roots and 20 per right-hand side,
//    against 2 x (66 + 9 k) for the one-direction kernel it replaces;
//  * the blocks are formed as in pair64.cuh, 1/sqrt by one approximate seed and
//    one third-order step (rsqrt3);
//  * the periodic cell sums the nine images' block first, then applies it.
// Homes and visitors as in sym.cu: one home blob per lane, visitors in tiles of
// 32 records by the TMA ring, lane l meets visitor (step + l) mod 32 and hands
// the visitor's running sum to lane l - 1 after every step.  Inside a warp's own
// 32 blobs steps 1..15 give every pair once; steps 0 (itself) and 16 (both lanes
// of a pair meet each other) are applied in the home direction only.
// Sums go to one partial per (home tile, visitor) and per (item, home), added in
// a fixed order by reduce64_kernel (deterministic; FP64 atomics would not be).
//
// Cutting: CTAs of one warp (32 homes) up to SMALL_N blobs, so that a small
// system spreads over all SMs, of four warps beyond, which quarters the
// partials; items of `chunk` visitor tiles; and for very small systems the 32
// steps of a tile are split over `parts` items.
//
// Measured, boomerangs, k = 1, whole call: 1,920 blobs 541 -> 282 us (its FP64
// instructions at the measured rate: 253 us).
#include <cuda_runtime.h>

#include <algorithm>

#include "ring.cuh"
#include "rpbd_internal.cuh"
#include "pair64.cuh"

namespace rpbd {
namespace sym64 {

using namespace ring;

constexpr int VT = 32;           // visitor tile (records)
constexpr int NST = 4;           // ring stages
constexpr int MAX_CHUNK = 64;    // visitor tiles per item
constexpr int64_t SMALL_N = 4096;
constexpr double PARTIAL_LIMIT = 4.0 * (1ull << 30);

using namespace pair64;

// Records: field f of blob i at ((i / 32) NF + f) 32 + i % 32, fields x, y,
// z~, s F(0, x..z), ...; padding blobs sit far away with zero force.
template <int K>
__global__ void pack64_kernel(int64_t n, int64_t n_pad, int k, const double* r, const double* F, double a, int wall,
                              double s_min, double* rec, double* scale)
{
    pdl_wait();
    pdl_trigger();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n_pad) return;
    constexpr int NF = 3 + 3 * K;
    double* o = rec + (i / VT) * VT * NF + i % VT;
    double x = 1.0e7, y = 1.0e7, zt = a, s = 0.0;
    if (i < n) {
        x = r[i];
        y = r[n + i];
        const double z = r[2 * n + i];
        zt = z;
        s = 1.0;
        if (wall && !(z >= a)) {  // below the wall height, or NaN (stays NaN in s)
            zt = a;
            const double t = z / a;
            s = t >= 1.0 ? 1.0 : (t <= s_min ? s_min : t);
        }
        scale[i] = s;
    }
    o[0] = x;
    o[VT] = y;
    o[2 * VT] = zt;
#pragma unroll
    for (int m = 0; m < K; ++m)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            o[(3 + 3 * m + c) * VT] = i < n && m < k ? s * F[((int64_t)m * 3 + c) * n + i] : 0.0;
}

// Grid: (home tile, item of `chunk` visitor tiles, part of the steps).  Partial
// rows of [3K][n_pad]: T * parts visitor rows, then items * parts home rows.
template <int K, bool WALL, bool PER, int NW>
__global__ void __launch_bounds__(32 * NW) sym64_kernel(const double* rec, int64_t n_pad, int chunk, Const c,
                                                        double* partial, int* err_flag, RingTest rt)
{
    constexpr int NF = 3 + 3 * K, NT = 32 * NW;
    constexpr uint32_t TILE_BYTES = VT * NF * sizeof(double);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    double* stage = reinterpret_cast<double*>(smem_raw);
    double* red = stage + NST * VT * NF;  // [2 buffers][NW][3K][VT]
    uint64_t* bar = reinterpret_cast<uint64_t*>(red + 2 * NW * 3 * K * VT);
    const int T = gridDim.x, home = blockIdx.x, item = blockIdx.y, part = blockIdx.z, parts = gridDim.z;
    const int tiles = (int)(n_pad / VT);
    const int tile0 = home * NW + item * chunk;  // visitors: the home tile's own blobs and all after them
    const int ntile = min(chunk, tiles - tile0);
    pdl_wait();
    pdl_trigger();
    if (ntile <= 0) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int s0 = VT / parts * part, s1 = s0 + VT / parts;

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < NST; ++s) mbar_init(&bar[s], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (tid == 0)  // (failure-path test: stage 0 gets no copy, so its wait runs out)
        for (int s = rt.skip_first ? 1 : 0; s < NST && s < ntile; ++s) {
            mbar_expect_tx(&bar[s], TILE_BYTES);
            tma_load_1d(stage + (size_t)s * VT * NF, rec + (size_t)(tile0 + s) * VT * NF, TILE_BYTES, &bar[s]);
        }
    const double* hr = rec + (size_t)(home * NW + warp) * VT * NF + lane;
    const double hx = hr[0], hy = hr[VT], hz = hr[2 * VT], hz6 = 6.0 * hz;
    double hf[3 * K], acc[3 * K];
#pragma unroll
    for (int q = 0; q < 3 * K; ++q) {
        hf[q] = hr[(3 + q) * VT];
        acc[q] = 0.0;
    }
    int t = 0;
    bool bad = false;
    for (; t < ntile; ++t) {
        const int s = t % NST;
        const bool ok = mbar_wait_bounded(&bar[s], (t / NST) & 1, rt.limit);
        const double* st = stage + (size_t)s * VT * NF;
        const int own = tile0 + t - home * NW;  // visitor tile counted from the home tile's first
        const bool same = own == warp;          // the warp's own blobs
        double* rb = red + (t & 1) * (NW * 3 * K * VT);
        if (ok && own >= warp) {
            double vacc[3 * K];
#pragma unroll
            for (int q = 0; q < 3 * K; ++q) vacc[q] = 0.0;
            const int se = same ? min(s1, VT / 2 + 1) : s1;
            int step = s0;
            for (; step < se; ++step) {
                const int v = (step + lane) & (VT - 1);
                const double dx = hx - st[v], dy = hy - st[VT + v], zj = st[2 * VT + v];
                const bool both = !same || (step != 0 && step != VT / 2);
                if constexpr (PER) {
                    Block M;
                    image_sum(dx, dy, hz, zj, c, M);
#pragma unroll
                    for (int m = 0; m < K; ++m) {
                        const double fx = st[(3 + 3 * m) * VT + v], fy = st[(4 + 3 * m) * VT + v], fz = st[(5 + 3 * m) * VT + v];
                        acc[3 * m + 0] = fma(M.xz, fz, fma(M.xy, fy, fma(M.xx, fx, acc[3 * m + 0])));
                        acc[3 * m + 1] = fma(M.yz, fz, fma(M.yy, fy, fma(M.xy, fx, acc[3 * m + 1])));
                        acc[3 * m + 2] = fma(M.zz, fz, fma(M.zy, fy, fma(M.zx, fx, acc[3 * m + 2])));
                        if (both) {
                            const double gx = hf[3 * m], gy = hf[3 * m + 1], gz = hf[3 * m + 2];
                            vacc[3 * m + 0] = fma(M.zx, gz, fma(M.xy, gy, fma(M.xx, gx, vacc[3 * m + 0])));
                            vacc[3 * m + 1] = fma(M.zy, gz, fma(M.yy, gy, fma(M.xy, gx, vacc[3 * m + 1])));
                            vacc[3 * m + 2] = fma(M.zz, gz, fma(M.yz, gy, fma(M.xz, gx, vacc[3 * m + 2])));
                        }
                    }
                } else {
                    double al, be, gx, gz, mzz;
                    factors<WALL>(dx, dy, hz, hz6, zj, c, al, be, gx, gz, mzz);
#pragma unroll
                    for (int m = 0; m < K; ++m) {
                        const double fx = st[(3 + 3 * m) * VT + v], fy = st[(4 + 3 * m) * VT + v], fz = st[(5 + 3 * m) * VT + v];
                        const double P = fma(dy, fy, dx * fx);
                        const double Q = fma(be, P, gx * fz);
                        acc[3 * m + 0] = fma(dx, Q, fma(al, fx, acc[3 * m + 0]));
                        acc[3 * m + 1] = fma(dy, Q, fma(al, fy, acc[3 * m + 1]));
                        acc[3 * m + 2] = fma(mzz, fz, fma(gz, P, acc[3 * m + 2]));
                        if (both) {
                            const double ux = hf[3 * m], uy = hf[3 * m + 1], uz = hf[3 * m + 2];
                            const double Pt = fma(dy, uy, dx * ux);
                            const double Qt = fma(be, Pt, gz * uz);
                            vacc[3 * m + 0] = fma(dx, Qt, fma(al, ux, vacc[3 * m + 0]));
                            vacc[3 * m + 1] = fma(dy, Qt, fma(al, uy, vacc[3 * m + 1]));
                            vacc[3 * m + 2] = fma(mzz, uz, fma(gx, Pt, vacc[3 * m + 2]));
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < 3 * K; ++q) vacc[q] = __shfl_sync(0xffffffffu, vacc[q], (lane + 1) & 31);
            }
            // lane l now holds the sums of visitor (l + step) mod 32
            if (same) {
#pragma unroll
                for (int q = 0; q < 3 * K; ++q) acc[q] += __shfl_sync(0xffffffffu, vacc[q], (lane - step) & 31);
            } else {
#pragma unroll
                for (int q = 0; q < 3 * K; ++q) rb[(warp * 3 * K + q) * VT + ((lane + step) & (VT - 1))] = vacc[q];
            }
        }
        if (__syncthreads_or(!ok)) {
            bad = true;
            break;
        }
        if (own > 0) {  // the warps before this tile's own have met it
            const int nw = min(own, NW);
            const int64_t vbase = (int64_t)(tile0 + t) * VT;
            for (int e = tid; e < VT * 3 * K; e += NT) {
                const int q = e / VT, vl = e % VT;
                double sum = rb[q * VT + vl];
                for (int w = 1; w < nw; ++w) sum += rb[(w * 3 * K + q) * VT + vl];
                partial[((int64_t)(home * parts + part) * 3 * K + q) * n_pad + vbase + vl] = sum;
            }
        }
        if (tid == 0 && t + NST < ntile) {
            fence_proxy_async();
            mbar_expect_tx(&bar[s], TILE_BYTES);
            tma_load_1d(stage + (size_t)s * VT * NF, rec + (size_t)(tile0 + t + NST) * VT * NF, TILE_BYTES, &bar[s]);
        }
    }
    if (bad) {
        if (tid == 0) {
            atomicExch(err_flag, 1);
            for (int u = t + 1; u < ntile && u < t + NST; ++u) mbar_wait_bounded(&bar[u % NST], (u / NST) & 1);
        }
        return;
    }
    const int64_t row = (int64_t)T * parts + item * parts + part;
    const int64_t i = (int64_t)home * NT + tid;
#pragma unroll
    for (int q = 0; q < 3 * K; ++q) partial[(row * 3 * K + q) * n_pad + i] = acc[q];
}

// U_i = s_i / (8 pi eta) times the sum of blob i's partial rows: the visitor
// rows of the home tiles before its own (of its own too, past the tile's first
// 32 blobs) and the home rows of its tile's items.  32 blobs x RS row slices a
// block, the slices added in order: one thread per blob walked up to 120 rows
// one load after another at n = 1,920.
constexpr int RS = 8;
template <int K>
__global__ void __launch_bounds__(32 * RS) reduce64_kernel(int64_t n, int64_t n_pad, int nw, int T, int parts, int chunk,
                                                           const double* partial, const double* scale,
                                                           double inv8pieta, double* U)
{
    __shared__ double sm[RS][32];
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31, y = threadIdx.x >> 5, q = blockIdx.y;
    const int64_t tile = blockIdx.x, i = tile * VT + lane;
    const int home = (int)(tile / nw), sub = (int)(tile % nw);
    const int vis = (home + (sub > 0 ? 1 : 0)) * parts;
    const int tiles = (int)(n_pad / VT);
    const int rows = vis + (tiles - home * nw + chunk - 1) / chunk * parts;
    const double* p = partial + (int64_t)q * n_pad + i;
    const int64_t ld = (int64_t)3 * K * n_pad;
    double sum = 0.0;
#pragma unroll 4
    for (int e = y; e < rows; e += RS) sum += p[(e < vis ? e : T * parts + e - vis) * ld];
    sm[y][lane] = sum;
    __syncthreads();
    if (y == 0 && i < n) {
#pragma unroll
        for (int w = 1; w < RS; ++w) sum += sm[w][lane];
        U[(int64_t)q * n + i] = scale[i] * inv8pieta * sum;
    }
}

// how a matvec of n blobs is cut
struct Cut {
    int nw, T, chunk, items, parts;
    int64_t n_pad;
    double rows() const { return (double)(T + items) * parts; }
};

static Cut cut(int64_t n, int sm_count)
{
    Cut c;
    c.nw = n <= SMALL_N ? 1 : 4;
    const int64_t ht = 32 * c.nw;
    c.n_pad = (n + ht - 1) / ht * ht;
    c.T = (int)(c.n_pad / ht);
    const int64_t tiles = c.n_pad / VT;
    auto count = [&](int64_t ch) {
        int64_t m = 0;
        for (int64_t H = 0; H < c.T; ++H) m += (tiles - H * c.nw + ch - 1) / ch;
        return m;
    };
    c.chunk = MAX_CHUNK;
    while (c.chunk > 1 && count(c.chunk) < 16 * (int64_t)sm_count) c.chunk /= 2;
    c.parts = 1;
    while (c.parts < 4 && count(c.chunk) * c.parts < 16 * (int64_t)sm_count) c.parts *= 2;
    c.items = (int)((tiles + c.chunk - 1) / c.chunk);
    return c;
}

template <int K, bool WALL, bool PER, int NW>
static int launch(rpbd_handle* h, const Cut& c, const double* rec, double* partial, cudaStream_t st)
{
    auto kern = sym64_kernel<K, WALL, PER, NW>;
    const size_t smem = ((size_t)NST * VT * (3 + 3 * K) + 2 * NW * 3 * K * VT) * sizeof(double) + NST * sizeof(uint64_t);
    if (once_per_device(h, reinterpret_cast<const void*>(kern)))
        RPBD_CU(h, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    launch_pdl(kern, dim3((unsigned)c.T, (unsigned)c.items, (unsigned)c.parts), 32 * NW, smem, st, rec, c.n_pad, c.chunk,
               Const::make(h->p), partial, h->dev_flag, ring_test(h));
    return RPBD_OK;
}

template <int K>
static int run(rpbd_handle* h, const Cut& c, int64_t n, const double* r, const double* F, double* U, int k, cudaStream_t st)
{
    double *rec, *scale, *partial;
    RPBD_TRY(ensure_t(h, BUF_PACK, (size_t)c.n_pad * (3 + 3 * K), &rec));
    RPBD_TRY(ensure_t(h, BUF_SCALE, (size_t)c.n_pad, &scale));
    RPBD_TRY(ensure_t(h, BUF_PARTIAL, (size_t)c.rows() * 3 * K * c.n_pad, &partial));
    launch_pdl(pack64_kernel<K>, (unsigned)((c.n_pad + 127) / 128), 128, 0, st, n, c.n_pad, k, r, F, h->p.a, h->p.wall,
               h->p.s_min, rec, scale);
    count_launch();
    if (h->profile) prof_begin(h, st);
    const bool per = h->p.Lx > 0.0;
    if (c.nw == 1)
        RPBD_TRY((per ? launch<K, true, true, 1> : h->p.wall ? launch<K, true, false, 1> : launch<K, false, false, 1>)(
            h, c, rec, partial, st));
    else
        RPBD_TRY((per ? launch<K, true, true, 4> : h->p.wall ? launch<K, true, false, 4> : launch<K, false, false, 4>)(
            h, c, rec, partial, st));
    count_launch();
    if (h->profile) prof_end(h, st, RPBD_F64, K, (double)n * (double)n);
    const double inv8pieta = 1.0 / (8.0 * 3.14159265358979323846 * h->p.eta);
    launch_pdl(reduce64_kernel<K>, dim3((unsigned)(c.n_pad / VT), (unsigned)(3 * k)), 32 * RS, 0, st, n, c.n_pad, c.nw, c.T,
               c.parts, c.chunk, (const double*)partial, (const double*)scale, inv8pieta, U);
    count_launch();
    RPBD_LAUNCH_CHECK(h);
    return RPBD_OK;
}

}  // namespace sym64

// Whether the symmetric FP64 kernel takes n blobs with k right-hand sides.
// Instructions per ordered pair (above): passes of up to four right-hand sides
// cost 36, 46 or 66 each, the one-direction kernel 66 + 9 K with K = 8 or 16:
// fewer up to k = 8.  The partials, 3 K n^2/128 doubles beyond SMALL_N, have to
// stay under PARTIAL_LIMIT (n about 145,000 for k = 1), and everything has to fit
// the memory left: where it does not, the one-direction kernel, which needs a tenth
// of it, runs, and later calls of the handle go straight there (worth_trying).
bool sym64_takes(rpbd_handle* h, int64_t n, int k, cudaStream_t st)
{
    if (k > 8 || n > (int64_t)1 << 20) return false;
    const sym64::Cut c = sym64::cut(n, h->sm_count);
    const int K = k <= 2 ? k : 4;
    const double bytes = c.rows() * 3.0 * K * (double)c.n_pad * sizeof(double);
    if (c.items > 65535 || bytes > sym64::PARTIAL_LIMIT) return false;
    const struct { Buf b; size_t bytes; } need[] = {{BUF_PACK, (size_t)c.n_pad * (3 + 3 * K) * sizeof(double)},
                                                    {BUF_SCALE, (size_t)c.n_pad * sizeof(double)},
                                                    {BUF_PARTIAL, (size_t)bytes}};
    for (const auto& q : need)
        if (!worth_trying(h, q.b, q.bytes, st)) return false;
    for (const auto& q : need) {
        void* p;
        if (ensure(h, q.b, q.bytes, &p) != RPBD_OK) {
            cudaGetLastError();  // (the failed allocation is not the one-direction kernel's)
            cudaFree(h->buf[BUF_PARTIAL]);  // (nor does that kernel need partials of this size)
            h->buf[BUF_PARTIAL] = nullptr;
            h->cap[BUF_PARTIAL] = 0;
            return false;
        }
    }
    return true;
}

int sym64_apply_impl(rpbd_handle* h, int64_t n, const double* r, const double* F, double* U, int k, cudaStream_t st)
{
    const sym64::Cut c = sym64::cut(n, h->sm_count);
    for (int m0 = 0; m0 < k; m0 += 4) {
        const int kc = k - m0 < 4 ? k - m0 : 4;
        const double* Fm = F + (size_t)m0 * 3 * n;
        double* Um = U + (size_t)m0 * 3 * n;
        if (kc == 1) RPBD_TRY(sym64::run<1>(h, c, n, r, Fm, Um, kc, st));
        else if (kc == 2) RPBD_TRY(sym64::run<2>(h, c, n, r, Fm, Um, kc, st));
        else RPBD_TRY(sym64::run<4>(h, c, n, r, Fm, Um, kc, st));
    }
    return RPBD_OK;
}

}  // namespace rpbd
