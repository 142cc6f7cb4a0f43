// T^{1/2} e_1 for the Lanczos square root (Sec. 2.2), T_m symmetric tridiagonal
// (diagonal alpha, off-diagonal beta), by one warp.
//
// Positive definite T (every Lanczos run on an SPD mobility): the contour-
// integral quadrature of Hale, Higham & Trefethen (SIAM J. Numer. Anal. 46,
// 2008, method 3 for the square root).  From
//   T^{1/2} = (2/pi) int_0^inf T (T + t^2)^{-1} dt,  t = sqrt(lo) sc(u | k'),
// the midpoint rule in u over (0, K') with N nodes converges as
// exp(-2 pi^2 N / (log(hi/lo) + 3)) for a spectrum in [lo, hi]: N = 32, one node
// per lane, is below 1e-16 up to hi/lo = 1e6, and 64, two per lane, up to 1e12.
// Each node is one tridiagonal solve (T + t^2) z = T e_1 (no cancellation), so the
// chain is ~2 m steps; Jacobi needs 5-6 sweeps of ~m dependent rounds (129 us per
// call, mean over the iterations of a time step, against 39 for the quadrature
// with everything on the device, and 1e-15 instead of 1e-16 off at condition 1e4).
// hi is Gershgorin's bound; lo the largest of 32 trial shifts hi 2^{-47 j/32} with
// T - shift positive definite.  The shifts' and weights' ratios to hi and sqrt(hi)
// depend on j alone: a table of 33 KB that the host fills once (sqrt_nodes), since
// one FP64 operation after another takes the warp ~0.04 us (with the elliptic
// functions on the device 21.6 us of a Lanczos iteration at 7 vectors, now 10.3).
//
// Otherwise (an eigenvalue below ~1e-14 of the largest, or negative) T is
// diagonalised by cyclic Jacobi, T = Q diag(lambda) Q^T, and
//   c = T^{1/2} e_1 = Q diag(sqrt(max(lambda, 0))) Q^T e_1.
// The rotations of one sweep are ordered as a round-robin tournament: in each
// of the N - 1 rounds (N = m1 rounded up to even) the indices form N/2
// disjoint pairs, so the round's rotations commute and are applied together
// (all column updates, then all row updates, the lanes splitting the
// entries).  A sweep therefore costs N - 1 dependent steps instead of
// m1 (m1 - 1) / 2.  Each pair's 2x2 block is then set from the closed form
// (diagonal app - t apq, aqq + t apq, off-diagonal exactly zero).
#pragma once

#include <cuda_runtime.h>

#include <cmath>

#include "wall_rpy.cuh"

namespace rpbd {

constexpr int TRIDIAG_MAX_PAIRS = 48;

// shared memory (doubles) the routine needs for order m1
__host__ __device__ inline int tridiag_sqrt_smem_doubles(int m1)
{
    const int jacobi = 2 * m1 * m1 + 6 * TRIDIAG_MAX_PAIRS, quad = 66 * m1;
    return jacobi > quad ? jacobi : quad;
}

constexpr int SQRT_TRIALS = 32, SQRT_NODES = 64;
struct SqrtNode {
    double shift, weight;  // over hi, over sqrt(hi)
};
// lo / hi of trial j; with 32 nodes from this ratio on, below it with 64
__host__ __device__ constexpr bool sqrt_32_nodes(double ratio) { return ratio >= 1e-6; }

// SQRT_TRIALS rows of SQRT_NODES nodes, then one of the trials' ratios (as shifts).
// The elliptic functions sc, dn for modulus k', k = sqrt(lo / hi), from the
// arithmetic-geometric mean and Gauss' transformation (Abramowitz & Stegun 16.12,
// 17.6), nodes beyond K'/2 from those below by sc(K' - u) = 1 / (k sc(u)).
constexpr int SQRT_TABLE = (SQRT_TRIALS + 1) * SQRT_NODES;
inline void sqrt_nodes(SqrtNode* t)
{
    for (int i = 0; i < SQRT_TABLE; ++i) t[i] = SqrtNode{0.0, 0.0};
    const double pi = 3.14159265358979323846;
    for (int j = 0; j < SQRT_TRIALS; ++j) {
        const double ratio = std::exp2(-47.0 / SQRT_TRIALS * (SQRT_TRIALS - j)), k = std::sqrt(ratio);
        t[SQRT_TRIALS * SQRT_NODES + j].shift = ratio;
        double a = 1.0, b = k, km[12], kc[12];  // modulus after n + 1 steps, and one minus it
        int steps = 0;
        while (steps < 12 && a - b > 1e-15 * a) {
            const double an = 0.5 * (a + b), cn = 0.5 * (a - b);
            km[steps] = cn / an;
            kc[steps++] = b / an;
            b = std::sqrt(a * b);
            a = an;
        }
        const double Kp = 0.5 * pi / a;
        const int N = sqrt_32_nodes(ratio) ? 32 : 64;
        for (int i = 0; i < N; ++i) {
            const int ii = i < N / 2 ? i : N - 1 - i;
            const double u = (ii + 0.5) * Kp / N;
            double sn = std::sin(u * a), cn = std::cos(u * a), dn = 1.0;  // a = the mean: u divided by every 1 + km
            for (int n = steps - 1; n >= 0; --n) {
                const double q = 1.0 + km[n] * sn * sn, p = kc[n] + km[n] * cn * cn;  // p = 2 - q, without the cancellation
                cn = cn * dn / q;
                sn = (1.0 + km[n]) * sn / q;
                dn = p / q;
            }
            double sc = sn / cn, w = dn / (cn * cn);
            if (i != ii) {
                w /= k * sc * sc;
                sc = 1.0 / (k * sc);
            }
            t[j * SQRT_NODES + i] = SqrtNode{ratio * sc * sc, w * 2.0 * Kp * k / (pi * N)};
        }
    }
}

// the quadrature; false (nothing written) when T is not safely positive definite
__device__ inline bool tridiag_sqrt_quadrature(int m1, const SqrtNode* __restrict__ nodes,
                                               const double* __restrict__ alpha, const double* __restrict__ beta, double* sm, double* __restrict__ c)
{
    const int lane = threadIdx.x & 31;
    double* al = sm;            // m1
    double* be = al + m1;       // m1 (m1 - 1 used)
    double* dinv = be + m1;     // [m1][32]: 1 / pivot of each lane's node
    double* y = dinv + 32 * m1; // [m1][32]
    for (int i = lane; i < m1; i += 32) {
        al[i] = alpha[i];
        be[i] = i + 1 < m1 ? beta[i] : 0.0;
    }
    __syncwarp();
    double hi = 0.0;
    bool fine = true;
    for (int i = lane; i < m1; i += 32) {
        const double g = al[i] + fabs(be[i]) + (i ? fabs(be[i - 1]) : 0.0);
        fine = fine && g > 0.0 && g < 1e300;
        hi = fmax(hi, g);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    if (!__all_sync(0xffffffffu, fine)) return false;
    // T - x positive definite? (pivots of L D L^T)
    const double ratio = nodes[SQRT_TRIALS * SQRT_NODES + lane].shift, x = hi * ratio;
    {
        double d = al[0] - x;
        bool pos = d > 1e-280;
        for (int i = 1; i < m1; ++i) {
            d = fma(-(be[i - 1] * be[i - 1]), rcp3(d), al[i] - x);  // (0, tiny or NaN pivots: not positive)
            pos = pos && d > 1e-280 && d < 1e300;
        }
        const unsigned ok = __ballot_sync(0xffffffffu, pos);
        if (!(ok & 1u)) return false;
        hi = __shfl_sync(0xffffffffu, hi, 0);
        const int best = __popc(ok & ~(ok + 1u)) - 1;  // last of the leading run of lanes
        const int N = sqrt_32_nodes(__shfl_sync(0xffffffffu, ratio, best)) ? 32 : 64;
        double ci = 0.0, cj = 0.0, ck = 0.0;  // components lane, lane + 32, lane + 64
        for (int half = 0; half < N / 32; ++half) {
            const SqrtNode nd = nodes[best * SQRT_NODES + 32 * half + lane];
            const double sig = hi * nd.shift, w = sqrt(hi) * nd.weight;
            // (T + sig) z = T e_1
            double di = rcp3(al[0] + sig), yi = al[0];
            dinv[lane] = di;
            y[lane] = yi;
            for (int i = 1; i < m1; ++i) {
                const double bb = be[i - 1], l = bb * di;
                di = rcp3(fma(-(bb * bb), di, al[i] + sig));
                yi = (i == 1 ? bb : 0.0) - l * yi;
                dinv[i * 32 + lane] = di;
                y[i * 32 + lane] = yi;
            }
            double z = 0.0;
            for (int i = m1 - 1; i >= 0; --i) {
                z = (y[i * 32 + lane] - be[i] * z) * dinv[i * 32 + lane];
                y[i * 32 + lane] = w * z;
            }
            __syncwarp();
            for (int s = 0; s < 32; ++s) {  // (rotated: every lane its own bank)
                const int q = (lane + s) & 31;
                if (lane < m1) ci += y[lane * 32 + q];
                if (lane + 32 < m1) cj += y[(lane + 32) * 32 + q];
                if (lane + 64 < m1) ck += y[(lane + 64) * 32 + q];
            }
            __syncwarp();
        }
        if (lane < m1) c[lane] = ci;
        if (lane + 32 < m1) c[lane + 32] = cj;
        if (lane + 64 < m1) c[lane + 64] = ck;
    }
    __syncwarp();
    return true;
}

// One warp (all 32 lanes call it).  nodes: the table of sqrt_nodes(); sm: tridiag_sqrt_smem_doubles(m1)
// doubles of shared memory; m1 <= 2 * TRIDIAG_MAX_PAIRS.  On return c[i]
// (global or shared, i < m1) holds T^{1/2} e_1; the return value is valid
// in every lane.
__device__ inline void tridiag_sqrt_e1(int m1, const SqrtNode* __restrict__ nodes, const double* __restrict__ alpha,
                                       const double* __restrict__ beta, double* sm, double* __restrict__ c)
{
    const int lane = threadIdx.x & 31;
    if (tridiag_sqrt_quadrature(m1, nodes, alpha, beta, sm, c)) return;
    double* A = sm;                    // m1 x m1, row-major
    double* Q = A + m1 * m1;           // eigenvectors (columns)
    double* rc = Q + m1 * m1;          // per pair: cos, sin, t, apq, app, aqq
    double* rs = rc + TRIDIAG_MAX_PAIRS;
    double* rt = rs + TRIDIAG_MAX_PAIRS;
    double* rpq = rt + TRIDIAG_MAX_PAIRS;
    double* rpp = rpq + TRIDIAG_MAX_PAIRS;
    double* rqq = rpp + TRIDIAG_MAX_PAIRS;
    for (int e = lane; e < m1 * m1; e += 32) {
        const int i = e / m1, j = e % m1;
        double v = 0.0;
        if (i == j) v = alpha[i];
        else if (j == i + 1) v = beta[i];
        else if (i == j + 1) v = beta[j];
        A[e] = v;
        Q[e] = (i == j) ? 1.0 : 0.0;
    }
    __syncwarp();
    double fro = 0.0;
    for (int e = lane; e < m1 * m1; e += 32) fro += A[e] * A[e];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) fro += __shfl_xor_sync(0xffffffffu, fro, o);
    const int N = (m1 + 1) & ~1;  // even number of slots; slot m1 (odd m1) sits out
    const int np = N / 2;
    // pair p of round r: slot N-1 against r, then (r + p, r - p) mod (N - 1)
    auto pair_of = [&](int r, int p, int& i, int& j) {
        int a, b;
        if (p == 0) {
            a = N - 1;
            b = r;
        } else {
            a = (r + p) % (N - 1);
            b = (r - p + (N - 1)) % (N - 1);
        }
        i = a < b ? a : b;
        j = a < b ? b : a;
    };
    for (int sweep = 0; sweep < 60 && m1 > 1; ++sweep) {
        double off = 0.0;
        for (int e = lane; e < m1 * m1; e += 32)
            if (e / m1 != e % m1) off += A[e] * A[e];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) off += __shfl_xor_sync(0xffffffffu, off, o);
        if (off <= 1e-32 * fro) break;
        for (int r = 0; r < N - 1; ++r) {
            // 1: one lane per pair computes its rotation (identity when skipped)
            for (int p = lane; p < np; p += 32) {
                int i, j;
                pair_of(r, p, i, j);
                double cc = 1.0, sn = 0.0, t = 0.0, apq = 0.0, app = 0.0, aqq = 0.0;
                if (j < m1) {
                    apq = A[i * m1 + j];
                    app = A[i * m1 + i];
                    aqq = A[j * m1 + j];
                    if (fabs(apq) > 1e-300 && !(fabs(apq) < 1e-19 * sqrt(fabs(app * aqq)))) {
                        const double tau = (aqq - app) / (2.0 * apq);
                        t = tau != 0.0 ? copysign(1.0, tau) / (fabs(tau) + sqrt(1.0 + tau * tau)) : 1.0;
                        cc = 1.0 / sqrt(1.0 + t * t);
                        sn = t * cc;
                    }
                }
                rc[p] = cc;
                rs[p] = sn;
                rt[p] = t;
                rpq[p] = apq;
                rpp[p] = app;
                rqq[p] = aqq;
            }
            __syncwarp();
            // 2: columns of A and Q: X <- X J
            for (int e = lane; e < np * m1; e += 32) {
                const int p = e / m1, k = e % m1;
                if (rs[p] == 0.0) continue;
                int i, j;
                pair_of(r, p, i, j);
                const double cc = rc[p], sn = rs[p];
                const double aki = A[k * m1 + i], akj = A[k * m1 + j];
                A[k * m1 + i] = cc * aki - sn * akj;
                A[k * m1 + j] = sn * aki + cc * akj;
                const double qki = Q[k * m1 + i], qkj = Q[k * m1 + j];
                Q[k * m1 + i] = cc * qki - sn * qkj;
                Q[k * m1 + j] = sn * qki + cc * qkj;
            }
            __syncwarp();
            // 3: rows of A: A <- J^T A
            for (int e = lane; e < np * m1; e += 32) {
                const int p = e / m1, k = e % m1;
                if (rs[p] == 0.0) continue;
                int i, j;
                pair_of(r, p, i, j);
                const double cc = rc[p], sn = rs[p];
                const double aik = A[i * m1 + k], ajk = A[j * m1 + k];
                A[i * m1 + k] = cc * aik - sn * ajk;
                A[j * m1 + k] = sn * aik + cc * ajk;
            }
            __syncwarp();
            // 4: each rotated pair's 2x2 block from the closed form
            for (int p = lane; p < np; p += 32) {
                if (rs[p] == 0.0) continue;
                int i, j;
                pair_of(r, p, i, j);
                A[i * m1 + i] = rpp[p] - rt[p] * rpq[p];
                A[j * m1 + j] = rqq[p] + rt[p] * rpq[p];
                A[i * m1 + j] = 0.0;
                A[j * m1 + i] = 0.0;
            }
            __syncwarp();
        }
    }
    __syncwarp();
    for (int i = lane; i < m1; i += 32) {
        double v = 0.0;
        for (int k = 0; k < m1; ++k) {
            const double lam = A[k * m1 + k];
            v += Q[i * m1 + k] * sqrt(lam > 0.0 ? lam : 0.0) * Q[k];  // Q[0][k]
        }
        c[i] = v;
    }
    __syncwarp();
}

}  // namespace rpbd
