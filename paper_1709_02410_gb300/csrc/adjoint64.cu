// FP64 adjoint: the symmetric gradient kernel (adjoint_tiles.cuh) in FP64, one
// launch per pass of up to four right-hand-side pairs.
#include <cuda_runtime.h>

#include "adjoint_tiles.cuh"

namespace rpbd {
namespace adj64 {

constexpr int64_t SMALL_N = 4096;
constexpr int MAX_CHUNK = 64;

template <int K, bool WALL, bool PER>
static int launch(rpbd_handle* h, const adj::Cut& c, int kc, const double* r, const double* u, const double* F, double* partial,
                  const adj::Out& o, cudaStream_t st)
{
    const size_t smem = 2 * (size_t)(3 + 6 * K) * adj::VT * 8 + 2 * c.nw * 4 * adj::VT * sizeof(double);
    adj::adjoint_kernel<double, K, WALL, PER, adj::Radius>
        <<<dim3((unsigned)c.hg, (unsigned)c.items, (unsigned)c.parts), c.threads, smem, st>>>(
            c, kc, r, u, F, nullptr, adj::Radius::make(h->p.a), h->p.a, h->p.s_min, h->p.Lx, h->p.Ly, partial, o);
    return RPBD_OK;
}

template <int K>
static int launch_any(rpbd_handle* h, const adj::Cut& c, int kc, const double* r, const double* u, const double* F,
                      double* partial, const adj::Out& o, cudaStream_t st)
{
    return (h->p.Lx > 0.0 ? launch<K, true, true> : h->p.wall ? launch<K, true, false> : launch<K, false, false>)(
        h, c, kc, r, u, F, partial, o, st);
}

}  // namespace adj64

int adjoint64_impl(rpbd_handle* h, int64_t n, const double* r, const double* u, const double* F, int nr, double* grad,
                   cudaStream_t st)
{
    using namespace adj64;
    const adj::Cut c = adj::cut(n, 1, SMALL_N, MAX_CHUNK, h->sm_count);
    const double i8 = 1.0 / (8.0 * 3.14159265358979323846 * h->p.eta);
    auto launch = [&](const adj::Cut& g, int kc, int m0, double* partial, const adj::Out& o) -> int {
        const double *um = u + (int64_t)m0 * 3 * n, *Fm = F + (int64_t)m0 * 3 * n;
        return (kc == 1 ? launch_any<1> : kc == 2 ? launch_any<2> : launch_any<4>)(h, g, kc, r, um, Fm, partial, o, st);
    };
    return adj::run_all<double>(h, c, nr, grad, i8, i8, [](int, int) { return RPBD_OK; }, launch, st);
}

}  // namespace rpbd
