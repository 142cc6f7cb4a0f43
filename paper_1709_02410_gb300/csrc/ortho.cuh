// Many dot products in one CTA, for the Gram-Schmidt kernels of the Krylov methods.
#pragma once

#include <cuda_runtime.h>

namespace rpbd {

// d[i] = sum_e at(i, e), i < nd, e < cnt, by the block's warps, U sums at a time
// each (independent chains: one FP64 addition takes tens of cycles here)
template <int U, class At, class Put>
__device__ __forceinline__ void ortho_sums(int nd, int cnt, At at, Put put)
{
    const int lane = threadIdx.x & 31;
    for (int i0 = (threadIdx.x >> 5) * U; i0 < nd; i0 += (blockDim.x >> 5) * U) {
        double s[U];
#pragma unroll
        for (int u = 0; u < U; ++u) s[u] = 0.0;
#pragma unroll 4
        for (int e = lane; e < cnt; e += 32)
#pragma unroll
            for (int u = 0; u < U; ++u) s[u] += at(min(i0 + u, nd - 1), e);
        // half of the sums to each half of the lanes while there are several
        int o = 16, mine = 0;
#pragma unroll
        for (int c = U / 2; c > 0; c >>= 1, o >>= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int u = 0; u < c; ++u)
                s[u] = (up ? s[u + c] : s[u]) + __shfl_xor_sync(0xffffffffu, up ? s[u] : s[u + c], o);
            if (up) mine += c;
        }
        const int first = 2 * o - 1;
#pragma unroll
        for (; o > 0; o >>= 1) s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
        if ((lane & first) == 0 && i0 + mine < nd) put(i0 + mine, s[0]);
    }
}
template <class At, class Put>
__device__ __forceinline__ void ortho_sums(int nd, int cnt, At at, Put put)
{
    const int nw = blockDim.x >> 5;
    if (nd <= nw) ortho_sums<1>(nd, cnt, at, put);
    else if (nd <= 2 * nw) ortho_sums<2>(nd, cnt, at, put);
    else ortho_sums<4>(nd, cnt, at, put);
}

}  // namespace rpbd
