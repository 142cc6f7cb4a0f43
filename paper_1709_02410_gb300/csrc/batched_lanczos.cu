// Batched preconditioned Lanczos M^{1/2} W (Sec. 2.2) for many independent
// suspensions, plus an optional matvec per system, as one CUDA graph.
//
// All systems advance in lockstep, one Lanczos iteration per step: the matvec
// is the batched pair kernel (batched.cu, sym.cu); dot products, the classical
// Gram-Schmidt reorthogonalisation (applied twice), the normalisation and the
// FP64 tridiagonal square root (tridiag_sqrt.cuh, one warp per system) all use
// per-system coefficients.  A system whose relative change
// |y_m - y_{m-1}|/|y_m| drops below tol is switched off by a device flag; later
// iterations skip its work, so max_iter iterations can be captured once and
// replayed without any host round trip.
//
// The vector kernels work on chunks of at most 1,024 blobs of one system, a block
// each, as krylov.cu's do on slices: a block keeps its chunk of w in shared memory
// through an update and the dot products that follow, and sums the previous
// kernel's partials of its system's chunks itself.  As eight kernels with one
// block per system and dot product (the whole chip waits for the largest system's),
// a search for the system and a square root and division per element, a Lanczos
// run took 140.8 ms on 64 systems of 471,495 blobs (126 of them the matvecs), now
// 137.2; on 64 systems of 120-1,920 blobs 6.17 -> 5.41, on 8 of those 2.17 -> 1.70.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "ortho.cuh"
#include "rpbd_internal.cuh"
#include "tridiag_sqrt.cuh"

namespace rpbd {

constexpr int BLZ_MAX = 64;

// blobs [b0, b0 + cnt) of system s; the system's chunks are c0 .. c0 + nc
struct BlzChunk {
    int64_t b0;
    int cnt, s, c0, nc;
    int pad[2];
};
// chunks so small only while that does not fill two blocks per SM of this GPU's 152
static int blz_chunk_size(int64_t n)
{
    const int64_t c = ((n + 303) / 304 + 127) / 128 * 128;
    return (int)std::min<int64_t>(1024, std::max<int64_t>(128, c));
}
static std::vector<BlzChunk> blz_chunks(int n_sys, const int64_t* off)
{
    const int64_t size = blz_chunk_size(off[n_sys]);
    std::vector<BlzChunk> v;
    for (int s = 0; s < n_sys; ++s) {
        const int64_t len = off[s + 1] - off[s], nc = (len + size - 1) / size;
        const int c0 = (int)v.size();
        for (int64_t c = 0; c < nc; ++c) {
            const int64_t lo = len * c / nc, hi = len * (c + 1) / nc;
            v.push_back(BlzChunk{off[s] + lo, (int)(hi - lo), s, c0, (int)nc, {0, 0}});
        }
    }
    return v;
}

// element e of a chunk's 3 cnt in the [3][n] vector
__device__ __forceinline__ int64_t blz_at(const BlzChunk& C, int64_t n, int e)
{
    const int c = (e >= C.cnt) + (e >= 2 * C.cnt);
    return c * n + C.b0 + (e - c * C.cnt);
}

// partials: [2 nv + 1][nch], rows 0..nv of pass 0, nv..2 nv of pass 1, 2 nv of |w|^2
// PASS 0: partials of V^T w.  1: w -= V h with h from pass 0's partials, then
// partials of V^T w.  2: w -= V h with pass 1's, then the partials of |w|^2.
// 3: the partials of |w|^2 alone (nv = 0).  H: both passes' coefficients, [s][ldh].
template <int PASS>
__global__ void blz_ortho_kernel(int64_t n, int nch, const BlzChunk* chunks, const double* V, int nv, double* w, double* part,
                                 double* H, int ldh, const int* active)
{
    extern __shared__ double sm[];
    pdl_wait();
    pdl_trigger();
    if ((int)blockIdx.x >= nch) return;
    const BlzChunk C = chunks[blockIdx.x];
    if (PASS < 3 && !active[C.s]) return;
    const int64_t ld = 3 * n;
    const int cnt = 3 * C.cnt;
    double *ws = sm, *h = sm + cnt;
    double* in = part + (PASS == 2 ? (int64_t)nv * nch : 0) + C.c0;
    double* out = part + (PASS == 0 ? 0 : PASS == 1 ? (int64_t)nv * nch : 2 * (int64_t)nv * nch) + blockIdx.x;
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) ws[e] = w[blz_at(C, n, e)];
    if (PASS == 1 || PASS == 2) {
        ortho_sums(nv, C.nc, [&](int i, int b) { return in[(int64_t)i * nch + b]; }, [&](int i, double x) { h[i] = x; });
        __syncthreads();
        if ((int)blockIdx.x == C.c0)
            for (int i = threadIdx.x; i < nv; i += blockDim.x) {
                double* Hi = H + (int64_t)C.s * ldh + i;
                *Hi = PASS == 1 ? h[i] : *Hi + h[i];
            }
        for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
            const int64_t g = blz_at(C, n, e);
            double s4[4] = {0.0, 0.0, 0.0, 0.0};
            int i = 0;
            for (; i + 4 <= nv; i += 4)
#pragma unroll
                for (int u = 0; u < 4; ++u) s4[u] += h[i + u] * V[(int64_t)(i + u) * ld + g];
            for (; i < nv; ++i) s4[0] += h[i] * V[(int64_t)i * ld + g];
            const double x = ws[e] - ((s4[0] + s4[1]) + (s4[2] + s4[3]));
            ws[e] = x;
            w[g] = x;
        }
    }
    __syncthreads();
    if (PASS >= 2)
        ortho_sums<1>(1, cnt, [&](int, int e) { return ws[e] * ws[e]; }, [&](int, double x) { out[0] = x; });
    else
        ortho_sums(nv, cnt, [&](int i, int e) { return V[(int64_t)i * ld + blz_at(C, n, e)] * ws[e]; },
                   [&](int i, double x) { out[(int64_t)i * nch] = x; });
}

struct BlzState {
    double *alpha, *beta, *c, *cprev, *W2, *change;
    int* iters;
    int mdim;
};

// h[0..2] = |w|^2 from its chunks' partials, |w|, 1/|w| (0 when it vanishes), by one
// thread: in every one the FP64 pipe would be busy with the root and the division
__device__ __forceinline__ void blz_norm(const double* part, int nc, double* h)
{
    ortho_sums<1>(1, nc, [&](int, int b) { return part[b]; },
                  [&](int, double s) {
                      const double nv = sqrt(s);
                      h[0] = s;
                      h[1] = nv;
                      h[2] = nv > 0.0 ? 1.0 / nv : 0.0;
                  });
    __syncthreads();
}
__device__ __forceinline__ void blz_normalize(const BlzChunk& C, int64_t n, const double* part, const double* w, double* out)
{
    __shared__ double h[3];
    blz_norm(part + C.c0, C.nc, h);
    for (int e = threadIdx.x; e < 3 * C.cnt; e += blockDim.x) {
        const int64_t g = blz_at(C, n, e);
        out[g] = w[g] * h[2];
    }
}

// v_0 = W / |W| by chunks, then one block per system: its state
__global__ void blz_start_kernel(int64_t n, int nch, const BlzChunk* chunks, const int2* sys, const double* W, const double* part,
                                 double* V, BlzState S, int* active)
{
    pdl_wait();
    pdl_trigger();
    if ((int)blockIdx.x < nch) {
        blz_normalize(chunks[blockIdx.x], n, part, W, V);
        return;
    }
    __shared__ double h[3];
    const int s = blockIdx.x - nch;
    blz_norm(part + sys[s].x, sys[s].y, h);
    if (threadIdx.x == 0) {
        S.W2[s] = h[0];
        active[s] = h[0] > 0.0 ? 1 : 0;
        S.iters[s] = 0;
        S.change[s] = 0.0;
    }
    for (int i = threadIdx.x; i < S.mdim; i += blockDim.x) {
        S.c[s * S.mdim + i] = 0.0;
        S.cprev[s * S.mdim + i] = 0.0;
    }
}

// v_{m+1} = w / |w| by chunks; then one block per system: alpha_m, beta_m,
// T^{1/2} e_1 (tridiag_sqrt.cuh) and the stop test.  The flags for the next
// iteration go to next, the other blocks still read active.
__global__ void blz_finish_kernel(int64_t n, int nch, const BlzChunk* chunks, const int2* sys, int m, int max_iter, double tol,
                                  const SqrtNode* nodes, const double* H, const double* w, const double* part, double* vnext,
                                  BlzState S, const int* active, int* next)
{
    extern __shared__ double sm[];
    pdl_wait();
    pdl_trigger();
    if ((int)blockIdx.x < nch) {
        const BlzChunk C = chunks[blockIdx.x];
        if (active[C.s]) blz_normalize(C, n, part, w, vnext);
        return;
    }
    const int s = blockIdx.x - nch, lane = threadIdx.x, m1 = m + 1;
    if (!active[s]) {
        if (lane == 0) next[s] = 0;
        return;
    }
    __shared__ double h[3];
    blz_norm(part + sys[s].x, sys[s].y, h);
    if (lane >= 32) return;
    const double nrm2 = h[0];
    double *al = S.alpha + s * S.mdim, *be = S.beta + s * S.mdim, *cs = S.c + s * S.mdim, *cp = S.cprev + s * S.mdim;
    if (lane == 0) {
        al[m] = H[s * (S.mdim + 1) + m];
        be[m] = h[1];
    }
    __syncwarp();
    tridiag_sqrt_e1(m1, nodes, al, be, sm, cs);
    double nc = 0.0, nd = 0.0;
    for (int i = lane; i < m1; i += 32) {
        const double v = cs[i];
        const double prev = i < m1 - 1 ? cp[i] : 0.0;
        nc += v * v;
        nd += (v - prev) * (v - prev);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        nc += __shfl_xor_sync(0xffffffffu, nc, o);
        nd += __shfl_xor_sync(0xffffffffu, nd, o);
    }
    __syncwarp();
    for (int i = lane; i < m1; i += 32) cp[i] = cs[i];
    if (lane == 0) {
        const double ch = nc > 0.0 ? sqrt(nd / nc) : 0.0;
        bool stop = false;
        if (m >= 1) {
            S.change[s] = ch;
            if (ch < tol) stop = true;
        }
        if (!(nrm2 > 1e-300 * S.W2[s])) stop = true;  // invariant subspace
        if (m1 >= max_iter) stop = true;
        next[s] = stop ? 0 : 1;
        if (stop) S.iters[s] = m1;
    }
}

// y = sqrt(W2[s]) sum_{i < iters[s]} c[s][i] V_i
__global__ void blz_combine_kernel(int64_t n, int nch, const BlzChunk* chunks, const double* V, BlzState S, double* y)
{
    __shared__ double c[BLZ_MAX], root;
    pdl_wait();
    pdl_trigger();
    if ((int)blockIdx.x >= nch) return;
    const BlzChunk C = chunks[blockIdx.x];
    const int it = S.iters[C.s];
    for (int i = threadIdx.x; i < it; i += blockDim.x) c[i] = S.c[C.s * S.mdim + i];
    if (threadIdx.x == 0) root = sqrt(S.W2[C.s]);
    __syncthreads();
    for (int e = threadIdx.x; e < 3 * C.cnt; e += blockDim.x) {
        const int64_t g = blz_at(C, n, e);
        double acc = 0.0;
#pragma unroll 4
        for (int i = 0; i < it; ++i) acc += c[i] * V[(int64_t)i * 3 * n + g];
        y[g] = root * acc;
    }
}

struct BatchGraph {
    std::vector<int64_t> off;
    int max_iter = 0;
    double tol = 0.0;
    int use_precond = 0;
    bool with_apply = false;
    int variant = -1;
    int test_stall = 0;  // the failure-path test option the kernels were captured with
    // every workspace buffer the captured kernels address: a buffer that has
    // grown (moved) since the capture invalidates the graph
    static constexpr int NSIG = 8;
    void* sig[NSIG] = {};
    cudaGraphExec_t exec = nullptr;
    cudaStream_t cap = nullptr;
};

void batched_free_graphs(rpbd_handle* h)
{
    for (BatchGraph* g : h->bgraphs) {
        if (g->exec) cudaGraphExecDestroy(g->exec);
        if (g->cap) cudaStreamDestroy(g->cap);
        delete g;
    }
    h->bgraphs.clear();
}

// The chunks of one batch layout on the device, written once when the handle first
// meets these offsets: later calls' kernels and the captured graphs, possibly still
// queued when another layout comes, read it where it is.
struct BlzTable {
    std::vector<int64_t> off;
    void* mem = nullptr;
    BlzChunk* chunks;
    int2* sys;  // first chunk and chunks of each system
    int64_t* doff;
    int nch, chunk;
};

void batched_free_tables(rpbd_handle* h)
{
    for (BlzTable* t : h->blz_tables) {
        cudaFree(t->mem);
        delete t;
    }
    h->blz_tables.clear();
}

static int blz_table(rpbd_handle* h, int n_sys, const int64_t* off, const BlzTable** out)
{
    for (const BlzTable* t : h->blz_tables)
        if ((int)t->off.size() == n_sys + 1 && std::equal(t->off.begin(), t->off.end(), off)) {
            *out = t;
            return RPBD_OK;
        }
    const std::vector<BlzChunk> ch = blz_chunks(n_sys, off);
    std::vector<char> host(ch.size() * sizeof(BlzChunk) + n_sys * sizeof(int2) + (n_sys + 1) * sizeof(int64_t));
    char* q = host.data();
    if (!ch.empty()) std::memcpy(q, ch.data(), ch.size() * sizeof(BlzChunk));
    int2* hs = reinterpret_cast<int2*>(q + ch.size() * sizeof(BlzChunk));
    for (int s = 0; s < n_sys; ++s) hs[s] = make_int2(0, 0);
    for (const BlzChunk& c : ch) hs[c.s] = make_int2(c.c0, c.nc);
    std::memcpy(hs + n_sys, off, (n_sys + 1) * sizeof(int64_t));
    BlzTable* t = new BlzTable();
    t->off.assign(off, off + n_sys + 1);
    t->nch = (int)ch.size();
    t->chunk = blz_chunk_size(off[n_sys]);
    if (cudaMalloc(&t->mem, host.size()) != cudaSuccess || upload(t->mem, q, host.size()) != cudaSuccess) {
        cudaFree(t->mem);
        delete t;
        return set_error(h, RPBD_NO_MEM, "batched lanczos: chunk table upload failed");
    }
    t->chunks = static_cast<BlzChunk*>(t->mem);
    t->sys = reinterpret_cast<int2*>(t->chunks + ch.size());
    t->doff = reinterpret_cast<int64_t*>(t->sys + n_sys);
    h->blz_tables.push_back(t);
    *out = t;
    return RPBD_OK;
}

struct BlzBufs {
    double *V, *z, *y, *w, *Win, *rin, *out, *Fin, *Uout;
    double *H, *part;
    BlzState S;
    int* active[2];  // of even and odd iterations
    const BlzTable* T;
};

// every kernel of one batched Lanczos (+ optional matvec), no host sync
static int blz_body(rpbd_handle* h, int n_sys, const int64_t* off, int64_t n, const BlzBufs& B, double tol,
                    int max_iter, int use_precond, bool with_apply, cudaStream_t st)
{
    const int64_t len = 3 * n;
    const BlzTable& T = *B.T;
    const int ldh = B.S.mdim + 1, threads = 3 * T.chunk > 512 ? 512 : 256;
    const unsigned g = (unsigned)std::max(1, T.nch), gs = (unsigned)(T.nch + n_sys);
    const int elems = 3 * T.chunk;
    auto ortho = [&](auto kernel, int nv, double* w, const int* active) {
        launch_pdl(kernel, g, threads, (size_t)(elems + nv) * sizeof(double), st, n, T.nch, (const BlzChunk*)T.chunks,
                   (const double*)B.V, nv, w, B.part, B.H, ldh, active);
        count_launch();
    };
    ortho(blz_ortho_kernel<3>, 0, B.Win, nullptr);
    launch_pdl(blz_start_kernel, gs, 256, 0, st, n, T.nch, (const BlzChunk*)T.chunks, (const int2*)T.sys, (const double*)B.Win,
               (const double*)B.part, B.V, B.S, B.active[0]);
    count_launch();
    for (int m = 0; m < max_iter; ++m) {
        const double* vm = B.V + (int64_t)m * len;
        const int* act = B.active[m & 1];
        if (use_precond) {
            RPBD_TRY(precond_apply_impl(h, 2, vm, B.z, st, act, T.doff, n_sys));
            RPBD_TRY(batched_apply_impl(h, n_sys, off, B.rin, B.z, B.y, 1, true, act, st));
            RPBD_TRY(precond_apply_impl(h, 1, B.y, B.w, st, act, T.doff, n_sys));
        } else {
            RPBD_TRY(batched_apply_impl(h, n_sys, off, B.rin, vm, B.w, 1, true, act, st));
        }
        const int nv = m + 1;
        ortho(blz_ortho_kernel<0>, nv, B.w, act);
        ortho(blz_ortho_kernel<1>, nv, B.w, act);
        ortho(blz_ortho_kernel<2>, nv, B.w, act);
        launch_pdl(blz_finish_kernel, gs, 256, tridiag_sqrt_smem_doubles(nv) * sizeof(double), st, n, T.nch,
                   (const BlzChunk*)T.chunks, (const int2*)T.sys, m, max_iter, tol, (const SqrtNode*)h->sqrt_nodes,
                   (const double*)B.H, (const double*)B.w, (const double*)(B.part + 2 * (int64_t)nv * T.nch),
                   B.V + (int64_t)(m + 1) * len, B.S, act, B.active[(m + 1) & 1]);
        count_launch();
    }
    launch_pdl(blz_combine_kernel, g, 256, 0, st, n, T.nch, (const BlzChunk*)T.chunks, (const double*)B.V, B.S,
               use_precond ? B.y : B.out);
    count_launch();
    if (use_precond) RPBD_TRY(precond_apply_impl(h, 0, B.y, B.out, st));
    if (with_apply) RPBD_TRY(batched_apply_impl(h, n_sys, off, B.rin, B.Fin, B.Uout, 1, true, nullptr, st));
    RPBD_LAUNCH_CHECK(h);
    return RPBD_OK;
}

static int blz_bufs(rpbd_handle* h, int n_sys, const int64_t* off, int64_t n, int max_iter, BlzBufs* B)
{
    const int64_t len = 3 * n;
    const int mdim = BLZ_MAX + 1;
    double* big;
    RPBD_TRY(ensure_t(h, BUF_BLZ, (size_t)(max_iter + 1) * len + 8 * len, &big));
    B->V = big;
    double* p = big + (size_t)(max_iter + 1) * len;
    B->z = p; p += len;
    B->y = p; p += len;
    B->w = p; p += len;
    B->Win = p; p += len;
    B->rin = p; p += len;
    B->out = p; p += len;
    B->Fin = p; p += len;
    B->Uout = p; p += len;
    RPBD_TRY(blz_table(h, n_sys, off, &B->T));
    double* sm;
    const size_t nsm = (size_t)n_sys * (mdim + 1 + 4 * mdim + 2) + (size_t)2 * n_sys + B->T->nch * (2 * (size_t)max_iter + 1);
    RPBD_TRY(ensure_t(h, BUF_BLZ_SMALL, nsm, &sm));
    B->H = sm; sm += (size_t)n_sys * (mdim + 1);
    B->S.mdim = mdim;
    B->S.alpha = sm; sm += (size_t)n_sys * mdim;
    B->S.beta = sm; sm += (size_t)n_sys * mdim;
    B->S.c = sm; sm += (size_t)n_sys * mdim;
    B->S.cprev = sm; sm += (size_t)n_sys * mdim;
    B->S.W2 = sm; sm += n_sys;
    B->S.change = sm; sm += n_sys;
    B->part = sm; sm += B->T->nch * (2 * (size_t)max_iter + 1);
    B->S.iters = reinterpret_cast<int*>(sm);
    B->active[0] = B->S.iters + n_sys;
    B->active[1] = B->active[0] + n_sys;
    return RPBD_OK;
}

}  // namespace rpbd

using namespace rpbd;

extern "C" {

int rpbd_lanczos_sqrt_apply_batched(rpbd_handle* h, int n_sys, const int64_t* offsets, const double* r, const double* W,
                                    double* out, const double* F, double* U, double tol, int max_iter,
                                    int use_precond, int use_graph, int* iters, void* stream)
{
    if (!h) return RPBD_BAD_ARG;
    if (n_sys <= 0 || !offsets || !r || !W || !out || (F && !U) || (!F && U))
        return set_error(h, RPBD_BAD_ARG, "batched lanczos: bad arguments");
    if (!(tol > 0) || max_iter < 1 || max_iter > BLZ_MAX)
        return set_error(h, RPBD_BAD_ARG, "batched lanczos: need tol > 0 and 1 <= max_iter <= 64");
    RPBD_TRY(batched_check_offsets(h, n_sys, offsets));  // (before chunks are cut from them)
    const int64_t n = offsets[n_sys];
    if (use_precond && (!h->prec_valid || h->prec_nb * h->prec_nper != n))
        return set_error(h, RPBD_BAD_ARG, "batched lanczos: preconditioner not built for these blobs");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (once_per_device(h, reinterpret_cast<const void*>(blz_finish_kernel)))
        RPBD_CU(h, cudaFuncSetAttribute(blz_finish_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        tridiag_sqrt_smem_doubles(BLZ_MAX) * (int)sizeof(double)));
    BlzBufs B;
    RPBD_TRY(blz_bufs(h, n_sys, offsets, n, max_iter, &B));
    const bool with_apply = F != nullptr;
    RPBD_CU(h, cudaMemcpyAsync(B.Win, W, sizeof(double) * 3 * n, cudaMemcpyDeviceToDevice, st));
    RPBD_CU(h, cudaMemcpyAsync(B.rin, r, sizeof(double) * 3 * n, cudaMemcpyDeviceToDevice, st));
    if (with_apply) RPBD_CU(h, cudaMemcpyAsync(B.Fin, F, sizeof(double) * 3 * n, cudaMemcpyDeviceToDevice, st));
    RPBD_CU(h, cudaMemsetAsync(h->dev_flag, 0, sizeof(int), st));
    if (!use_graph) {
        RPBD_TRY(blz_body(h, n_sys, offsets, n, B, tol, max_iter, use_precond, with_apply, st));
    } else {
        BatchGraph* G = nullptr;
        auto signature = [&](void** sg) {
            const Buf bs[BatchGraph::NSIG] = {BUF_BLZ,     BUF_BLZ_SMALL, BUF_BPACK,  BUF_BPARTIAL,
                                              BUF_BSCALE,  BUF_BSEG,      BUF_PREC_L, BUF_PREC_LINV};
            for (int i = 0; i < BatchGraph::NSIG; ++i) sg[i] = h->buf[bs[i]];
        };
        void* sig[BatchGraph::NSIG];
        signature(sig);
        for (BatchGraph* c : h->bgraphs)
            if (c->max_iter == max_iter && c->tol == tol && c->use_precond == use_precond &&
                c->with_apply == with_apply && c->variant == h->batch_variant && c->test_stall == h->test_stall &&
                (int)c->off.size() == n_sys + 1 &&
                std::equal(c->off.begin(), c->off.end(), offsets) && std::equal(sig, sig + BatchGraph::NSIG, c->sig))
                G = c;
        if (!G) {
            // run once eagerly so every workspace buffer and work list exists,
            // then capture the same sequence of kernels
            RPBD_TRY(blz_body(h, n_sys, offsets, n, B, tol, max_iter, use_precond, with_apply, st));
            RPBD_CU(h, cudaStreamSynchronize(st));
            void* sig2[BatchGraph::NSIG];
            signature(sig2);
            G = new BatchGraph();
            G->off.assign(offsets, offsets + n_sys + 1);
            G->max_iter = max_iter;
            G->tol = tol;
            G->use_precond = use_precond;
            G->with_apply = with_apply;
            G->variant = h->batch_variant;
            G->test_stall = h->test_stall;
            std::copy(sig2, sig2 + BatchGraph::NSIG, G->sig);
            h->bgraphs.push_back(G);
            RPBD_CU(h, cudaStreamCreateWithFlags(&G->cap, cudaStreamNonBlocking));
            const bool prof = h->profile;
            h->profile = false;
            RPBD_CU(h, cudaStreamBeginCapture(G->cap, cudaStreamCaptureModeThreadLocal));
            const int s_body = blz_body(h, n_sys, offsets, n, B, tol, max_iter, use_precond, with_apply, G->cap);
            cudaGraph_t graph = nullptr;
            const cudaError_t e_end = cudaStreamEndCapture(G->cap, &graph);
            h->profile = prof;
            if (s_body != RPBD_OK) {
                if (graph) cudaGraphDestroy(graph);
                return s_body;
            }
            if (e_end != cudaSuccess) return set_error(h, RPBD_CUDA, "batched lanczos: graph capture failed");
            const cudaError_t e_inst = cudaGraphInstantiate(&G->exec, graph, 0);
            cudaGraphDestroy(graph);
            if (e_inst != cudaSuccess) return set_error(h, RPBD_CUDA, "batched lanczos: graph instantiate failed");
        }
        RPBD_CU(h, cudaGraphLaunch(G->exec, st));
        count_launch();
    }
    RPBD_CU(h, cudaMemcpyAsync(out, B.out, sizeof(double) * 3 * n, cudaMemcpyDeviceToDevice, st));
    if (with_apply) RPBD_CU(h, cudaMemcpyAsync(U, B.Uout, sizeof(double) * 3 * n, cudaMemcpyDeviceToDevice, st));
    if (iters) {
        RPBD_CU(h, cudaMemcpyAsync(iters, B.S.iters, sizeof(int) * n_sys, cudaMemcpyDeviceToHost, st));
        RPBD_CU(h, cudaStreamSynchronize(st));
        int flag = 0;
        RPBD_CU(h, cudaMemcpy(&flag, h->dev_flag, sizeof(int), cudaMemcpyDeviceToHost));
        if (flag == 1) return set_error(h, RPBD_TIMEOUT, "batched lanczos: a pair kernel's bounded wait expired");
    }
    return RPBD_OK;
}

}  // extern "C"
