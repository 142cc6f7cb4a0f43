// Derivatives of the wall-RPY mobility:
//
//  adjoint:    g_k = d(u^T M(r) F)/d r_k  (derivative of the matvec of
//              Sec. 2.1 with respect to blob positions): each unordered pair
//              once, derivatives in closed form (adjoint_pair.cuh,
//              adjoint_tiles.cuh); FP32 here, FP64 in adjoint64.cu
//  divergence: (div M)_i = sum_j d_{r_j} . M_ij  (the drift the RFD of
//              Sec. 3 estimates with B = M), FP64: the pair block on a
//              forward-mode dual number carrying the three partials with
//              respect to the TARGET blob's (regularised) position, and the
//              reciprocal symmetry M_ij(r_i, r_j) = M_ji(r_j, r_i)^T to turn
//              every source-side derivative into a target-side one, so each
//              thread owns one blob and no atomics are needed
//
// The regularisation M_ij = s_i s_j Mt(rt_i, rt_j), rt = (x, y, max(z, a)),
// s = clamp(z/a, s_min, 1) is differentiated with them.
#include <cuda_runtime.h>

#include "adjoint_tiles.cuh"
#include "rpbd_internal.cuh"
#include "wall_rpy.cuh"

namespace rpbd {

struct RegBlob {
    double x, y, zt, s, dzt, ds;
};

__device__ __forceinline__ RegBlob reg_blob(const double* r, int64_t n, int64_t i, double a, int wall, double s_min)
{
    RegBlob b;
    b.x = r[i];
    b.y = r[n + i];
    const double z = r[2 * n + i];
    if (wall) {
        if (z >= a) { b.zt = z; b.dzt = 1.0; } else { b.zt = a; b.dzt = 0.0; }
        const double t = z / a;
        if (t >= 1.0) { b.s = 1.0; b.ds = 0.0; }
        else if (t <= s_min) { b.s = s_min; b.ds = 0.0; }
        else { b.s = t; b.ds = 1.0 / a; }
    } else {
        b.zt = z; b.dzt = 1.0; b.s = 1.0; b.ds = 0.0;
    }
    return b;
}

// block of target t (dual: partials w.r.t. t's regularised coordinates) and
// source s, FP64; out[9] row-major
template <bool WALL, bool PER>
__device__ __forceinline__ void dual_block(const RegBlob& t, const RegBlob& s, const PairConst<double>& pc,
                                           Dual<3> M[9])
{
    using D3 = Dual<3>;
    D3 dx(t.x - s.x), dy(t.y - s.y), dz(t.zt - s.zt), zi(t.zt), zj(s.zt);
    dx.g[0] = 1.0;
    dy.g[1] = 1.0;
    dz.g[2] = 1.0;
    zi.g[2] = 1.0;
    D3 Mxx, Mxy, Mxz, Myy, Myz, Mzx, Mzy, Mzz;
    pair_block_images<D3, double, WALL, PER>(dx, dy, dz, zi, zj, pc, Mxx, Mxy, Mxz, Myy, Myz, Mzx, Mzy, Mzz);
    M[0] = Mxx; M[1] = Mxy; M[2] = Mxz;
    M[3] = Mxy; M[4] = Myy; M[5] = Myz;
    M[6] = Mzx; M[7] = Mzy; M[8] = Mzz;
}

// ---------------------------------------------------------------------------
// FP32 adjoint: records of one pass of up to four right-hand-side pairs (hi/lo
// split of x, y so that separations keep FP64-level accuracy; lengths in units
// of a), then the symmetric gradient kernel in packed two-wide FP32.  FP32 sums
// over an item (at most MAX_CHUNK visitor tiles), FP64 across them.
namespace adjf32 {

using adj::Rec32;
using adj::VT;

constexpr int64_t SMALL_N = 8192;
constexpr int MAX_CHUNK = 16;

// one thread per record, padding records far away with zero u, F
template <int K>
__global__ void pack_kernel(int64_t n, int64_t n_pad, int kc, const double* __restrict__ r, const double* __restrict__ u,
                            const double* __restrict__ F, double a, double ia, int wall, double s_min, float4* __restrict__ rec)
{
    pdl_trigger();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n_pad) return;
    constexpr int NCH = Rec32<K>::NCH;
    float v[2 * NCH];
#pragma unroll
    for (int q = 0; q < 2 * NCH; ++q) v[q] = 0.0f;
    const bool real = i < n;
    const double x = real ? r[i] * ia : 1.0e7, y = real ? r[n + i] * ia : 1.0e7, z = real ? r[2 * n + i] : a;
    const double s = wall ? adj::overlap_scale(z, a, s_min) : 1.0;
    v[0] = (float)x;
    v[1] = (float)y;
    v[2] = (float)(x - (double)v[0]);
    v[3] = (float)(y - (double)v[1]);
    v[4] = (float)((wall ? (z > a ? z : a) : z) * ia);
    if (real)
#pragma unroll
        for (int q = 0; q < 3 * K; ++q)
            if (q < 3 * kc) {
                v[5 + q] = (float)(s * F[(int64_t)q * n + i]);
                v[5 + 3 * K + q] = (float)(s * u[(int64_t)q * n + i]);
            }
    float4* o = rec + (i / VT) * VT * NCH + i % VT;
#pragma unroll
    for (int q = 0; q < NCH; ++q) o[q * VT] = make_float4(v[2 * q], v[2 * q], v[2 * q + 1], v[2 * q + 1]);
}

template <int K, bool WALL, bool PER>
static int launch(rpbd_handle* h, const adj::Cut& c, int kc, const double* r, const double* u, const double* F, const float4* rec,
                  float* partial, const adj::Out& o, cudaStream_t st)
{
    auto kern = adj::adjoint_kernel<float2, K, WALL, PER, adj::Unit>;
    const size_t smem = 2 * (size_t)Rec32<K>::NCH * VT * 16 + 2 * c.nw * 4 * VT * sizeof(float);
    const double ia = 1.0 / h->p.a;
    launch_pdl(kern, dim3((unsigned)c.hg, (unsigned)c.items, (unsigned)c.parts), 32 * c.nw, smem, st, c, kc, r, u, F, rec,
               adj::Unit{}, h->p.a, h->p.s_min, (float)(h->p.Lx * ia), (float)(h->p.Ly * ia), partial, o);
    count_launch();
    launch_pdl(adj::adjoint_reduce_kernel<float>, dim3((unsigned)c.tiles, 3), 32 * adj::RS, 0, st, c, o, (const float*)partial, r,
               h->p.a, (int)WALL, h->p.s_min);
    return RPBD_OK;
}

template <int K>
static int launch_any(rpbd_handle* h, const adj::Cut& c, int kc, const double* r, const double* u, const double* F,
                      const float4* rec, float* partial, const adj::Out& o, cudaStream_t st)
{
    return (h->p.Lx > 0.0 ? launch<K, true, true> : h->p.wall ? launch<K, true, false> : launch<K, false, false>)(
        h, c, kc, r, u, F, rec, partial, o, st);
}

template <int K>
static void pack(rpbd_handle* h, const adj::Cut& c, int kc, const double* r, const double* u, const double* F, float4* rec,
                 cudaStream_t st)
{
    pack_kernel<K><<<(unsigned)((c.n_pad + 127) / 128), 128, 0, st>>>(c.n, c.n_pad, kc, r, u, F, h->p.a, 1.0 / h->p.a,
                                                                      h->p.wall ? 1 : 0, h->p.s_min, rec);
    count_launch();
}

static int run(rpbd_handle* h, int64_t n, const double* r, const double* u, const double* F, int nr, double* grad,
               cudaStream_t st)
{
    const adj::Cut c = adj::cut(n, 2, SMALL_N, MAX_CHUNK, h->sm_count);
    float4* rec;
    RPBD_TRY(ensure_t(h, BUF_PACK, (size_t)c.n_pad * Rec32<4>::NCH, &rec));
    const double ie = 1.0 / (8.0 * 3.14159265358979323846 * h->p.eta * h->p.a), ig = ie / h->p.a;
    auto pass = [&](int m0, int kc) -> int {
        const double *um = u + (int64_t)m0 * 3 * n, *Fm = F + (int64_t)m0 * 3 * n;
        if (kc == 1) pack<1>(h, c, kc, r, um, Fm, rec, st);
        else if (kc == 2) pack<2>(h, c, kc, r, um, Fm, rec, st);
        else pack<4>(h, c, kc, r, um, Fm, rec, st);
        RPBD_LAUNCH_CHECK(h);
        return RPBD_OK;
    };
    auto launch = [&](const adj::Cut& g, int kc, int m0, float* partial, const adj::Out& o) -> int {
        const double *um = u + (int64_t)m0 * 3 * n, *Fm = F + (int64_t)m0 * 3 * n;
        return (kc == 1 ? launch_any<1> : kc == 2 ? launch_any<2> : launch_any<4>)(h, g, kc, r, um, Fm, rec, partial, o, st);
    };
    return adj::run_all<float>(h, c, nr, grad, ig, ie, pass, launch, st);
}

}  // namespace adjf32

template <bool WALL, bool PER>
__global__ void divergence_kernel(int64_t n, const double* __restrict__ r, double a, double s_min, double Lx,
                                  double Ly, double inv8pieta, double* __restrict__ div)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const PairConst<double> pc = PairConst<double>::make(a, Lx, Ly);
    const RegBlob bi = reg_blob(r, n, i, a, WALL, s_min);
    double acc[3] = {0.0, 0.0, 0.0};
    for (int64_t j = 0; j < n; ++j) {
        Dual<3> T[9];
        if (j == i) {
            dual_block<WALL, PER>(bi, bi, pc, T);
#pragma unroll
            for (int aa = 0; aa < 3; ++aa) {
                double v = 2.0 * bi.s * bi.ds * T[aa * 3 + 2].v;
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const double dzt = b == 2 ? bi.dzt : 1.0;
                    v += bi.s * bi.s * (T[aa * 3 + b].g[b] + T[b * 3 + aa].g[b]) * dzt;
                }
                acc[aa] += v;
            }
        } else {
            const RegBlob bj = reg_blob(r, n, j, a, WALL, s_min);
            dual_block<WALL, PER>(bj, bi, pc, T);  // target j, source i
#pragma unroll
            for (int aa = 0; aa < 3; ++aa) {
                double v = bi.s * bj.ds * T[2 * 3 + aa].v;
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const double dzt = b == 2 ? bj.dzt : 1.0;
                    v += bi.s * bj.s * T[b * 3 + aa].g[b] * dzt;
                }
                acc[aa] += v;
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) div[c * n + i] = inv8pieta * acc[c];
}

}  // namespace rpbd

using namespace rpbd;

extern "C" {

static int adjoint_entry(rpbd_handle* h, int64_t n, const double* r, const double* u, const double* F, int nr,
                         double* grad, void* stream, bool f32)
{
    if (!h) return RPBD_BAD_ARG;
    if (n < 0 || nr < 1 || nr > 16 || (n > 0 && (!r || !u || !F || !grad)))
        return set_error(h, RPBD_BAD_ARG, "adjoint: bad arguments (need n >= 0, 1 <= k <= 16, non-null pointers)");
    if (n == 0) return RPBD_OK;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    return f32 ? adjf32::run(h, n, r, u, F, nr, grad, st) : adjoint64_impl(h, n, r, u, F, nr, grad, st);
}

int rpbd_mobility_adjoint(rpbd_handle* h, int64_t n, const double* r, const double* u, const double* F, double* grad,
                          void* stream)
{
    return adjoint_entry(h, n, r, u, F, 1, grad, stream, false);
}

int rpbd_mobility_adjoint_f32(rpbd_handle* h, int64_t n, const double* r, const double* u, const double* F,
                              double* grad, void* stream)
{
    return adjoint_entry(h, n, r, u, F, 1, grad, stream, true);
}

int rpbd_mobility_adjoint_multi(rpbd_handle* h, int64_t n, const double* r, const double* u, const double* F, int k,
                                double* grad, int dtype, void* stream)
{
    if (h && dtype != RPBD_F32 && dtype != RPBD_F64) return set_error(h, RPBD_BAD_ARG, "adjoint: bad dtype");
    return adjoint_entry(h, n, r, u, F, k, grad, stream, dtype == RPBD_F32);
}

int rpbd_mobility_divergence(rpbd_handle* h, int64_t n, const double* r, double* div, void* stream)
{
    if (!h) return RPBD_BAD_ARG;
    if (n < 0 || (n > 0 && (!r || !div))) return set_error(h, RPBD_BAD_ARG, "divergence: bad arguments");
    if (n == 0) return RPBD_OK;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const double inv8pieta = 1.0 / (8.0 * 3.14159265358979323846 * h->p.eta);
    const unsigned grid = (unsigned)((n + 127) / 128);
    const double Lx = h->p.Lx, Ly = h->p.Ly;
    if (Lx > 0.0) divergence_kernel<true, true><<<grid, 128, 0, st>>>(n, r, h->p.a, h->p.s_min, Lx, Ly, inv8pieta, div);
    else if (h->p.wall) divergence_kernel<true, false><<<grid, 128, 0, st>>>(n, r, h->p.a, h->p.s_min, Lx, Ly, inv8pieta, div);
    else divergence_kernel<false, false><<<grid, 128, 0, st>>>(n, r, h->p.a, h->p.s_min, Lx, Ly, inv8pieta, div);
    count_launch();
    RPBD_LAUNCH_CHECK(h);
    return RPBD_OK;
}

}  // extern "C"
