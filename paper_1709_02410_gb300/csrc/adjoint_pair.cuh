// Gradient of one pair's share of sum_m u_m^T M F_m, for either arithmetic.
//
// With home blob i, visitor j, a = s_i u_i, b = s_i F_i, c = s_j F_j, e = s_j u_j
// (per right-hand side) and M_ji = M_ij^T, the unordered pair contributes
//   E = sum_m a^T Mt c + b^T Mt e,   Mt = Mt(rt_i, rt_j),
// which the block's factored form (wall_rpy.cuh) reduces to
//   E = c1 A + c2 C - A/R + v (W - C),
//   A = S1 + S3, C = Q + dz (G + dz S3), W = iA A + h1 X - 20/3 a^4 w^2 Rz D + S3 (...)
// with the contractions S1 = a.c + b.e (x, y), S3 (z), Q = (a.d)(c.d) + (b.d)(e.d),
// G and D the sum and difference of the two mixed ones, X = w (Q + Rz D) - y S3, and
// iA, h1 the polynomials of wall_rpy_x2.cuh in w = 1/|R|^2, y = e_z^2, u = zi zj.  The
// derivatives follow by hand from this form: E depends on dx, dy through rho^2 and
// the contractions, on the heights through dz, Rz and u.  ~160 operations give all
// of dE/d(rt_i, rt_j) and E -- against ~400 per ORDERED pair for the block on dual
// numbers with three partials (checked against the oracle's gradient, and against
// finite differences of the matvec).
//
// V: double, or float2 for two pairs in packed FP32 (lengths in units of a).
#pragma once

#include <cuda_runtime.h>

#include "wall_rpy_x2.cuh"

namespace rpbd {
namespace adj {

__device__ __forceinline__ double add_(double a, double b) { return a + b; }
__device__ __forceinline__ double sub_(double a, double b) { return a - b; }
__device__ __forceinline__ double mul_(double a, double b) { return a * b; }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float2 add_(float2 a, float2 b) { return add2(a, b); }
__device__ __forceinline__ float2 sub_(float2 a, float2 b) { return fma2(bc2(-1.0f), b, a); }
__device__ __forceinline__ float2 mul_(float2 a, float2 b) { return mul2(a, b); }
__device__ __forceinline__ float2 fma_(float2 a, float2 b, float2 c) { return fma2(a, b, c); }
__device__ __forceinline__ double neg_(double a) { return -a; }
__device__ __forceinline__ float2 neg_(float2 a) { return make_float2(-a.x, -a.y); }
template <class V>
__device__ __forceinline__ V num_(double x);
template <>
__device__ __forceinline__ double num_<double>(double x) { return x; }
template <>
__device__ __forceinline__ float2 num_<float2>(double x) { return bc2((float)x); }
__device__ __forceinline__ double bc_(double x) { return x; }
__device__ __forceinline__ float2 bc_(float x) { return bc2(x); }
__device__ __forceinline__ double rsq_(double x) { return rsqrt3(x); }
__device__ __forceinline__ float2 rsq_(float2 x) { return make_float2(rsqrtf(x.x), rsqrtf(x.y)); }

// Constants of the pair: a number times a power of the blob radius.  Radius
// holds them for any a (kernel parameters, read as constant operands), Unit is
// a = 1, immediates.
enum Coef { C23, CM2, CM1, C5, H0, HY, A0, Z0, FOUR, HWY, HW0, AW0, ZL, ZW, PW, KSELF, KOVL, I8, NCOEF };
__host__ __device__ constexpr double coef(int i)
{
    return i == C23 ? 2.0 / 3.0 : i == CM2 ? -2.0 : i == CM1 ? -1.0 : i == C5 ? 5.0 : i == H0 ? 2.0 : i == HY ? -10.0
         : i == A0 ? -2.0 / 3.0 : i == Z0 ? -4.0 : i == FOUR ? 4.0 : i == HWY ? 70.0 / 3.0 : i == HW0 ? -10.0 / 3.0
         : i == AW0 ? 2.0 / 3.0 : i == ZL ? -8.0 / 3.0 : i == ZW ? 20.0 : i == PW ? -20.0 / 3.0 : i == KSELF ? 4.0 / 3.0
         : i == KOVL ? 3.0 / 8.0 : 1.0 / 8.0;
}
struct Radius {
    double v[NCOEF];
    static Radius make(double a)
    {
        Radius r;
        for (int i = 0; i < NCOEF; ++i)
            r.v[i] = coef(i) * (i <= FOUR ? a * a : i <= PW ? a * a * a * a : i == KSELF ? 1.0 / a : 1.0 / (a * a));
        return r;
    }
    template <int I, class V> __device__ __forceinline__ V get() const { return v[I]; }
};
struct Unit {
    template <int I, class V> __device__ __forceinline__ V get() const
    {
        constexpr double x = coef(I);
        return num_<V>(x);
    }
};
template <>
__device__ __forceinline__ float num_<float>(double x) { return (float)x; }

// c1, c2 and their derivatives with respect to r^2 where blobs overlap (r < 2a) or coincide
template <class S, class C>
__device__ __forceinline__ void overlap(S r2, S ri, const C& c, S& c1, S& c2, S& c1p, S& c2p)
{
    if (r2 < c.template get<FOUR, S>()) {
        const S ks = c.template get<KSELF, S>(), ko = c.template get<KOVL, S>(), i8 = c.template get<I8, S>();
        const bool apart = r2 > (sizeof(S) == 8 ? S(1e-200) : S(4e-26));  // (r^-3 finite; closer: coincident)
        c1 = apart ? ks - ko * (r2 * ri) : ks;
        c2 = apart ? ri * i8 : S(0);
        c1p = apart ? S(-0.5) * ko * ri : S(0);
        c2p = apart ? S(-0.5) * i8 * (ri * ri * ri) : S(0);
    }
}
// (closer than 1e-90 r^-3 would overflow: the gradient depends on the direction of the
// separation only, which a factor 2^200 keeps)
template <class C>
__device__ __forceinline__ void overlap_(double r2, double ri, const C& c, double& dx, double& dy, double& dz, double& c1,
                                         double& c2, double& c1p, double& c2p)
{
    if (r2 < c.template get<FOUR, double>()) {
        if (r2 < 1e-180) {
            dx *= 0x1p200;
            dy *= 0x1p200;
            dz *= 0x1p200;
            r2 = fma(dz, dz, fma(dy, dy, dx * dx));
            ri = rsq_(r2);
        }
        overlap<double>(r2, ri, c, c1, c2, c1p, c2p);
    }
}
template <class C>
__device__ __forceinline__ void overlap_(float2 r2, float2 ri, const C& c, float2&, float2&, float2&, float2& c1, float2& c2,
                                         float2& c1p, float2& c2p)
{
    if (r2.x < 4.0f || r2.y < 4.0f) {
        overlap<float>(r2.x, ri.x, c, c1.x, c2.x, c1p.x, c2p.x);
        overlap<float>(r2.y, ri.y, c, c1.y, c2.y, c1p.y, c2p.y);
    }
}

// dE/dx_i, dE/dy_i (minus those of j), dE/dz_i, dE/dz_j and E
template <class V>
struct PairGrad {
    V x, y, zi, zj, e;
};

// A, B: a, b of the home blob, [3 K]; ce(q): q < 3 K the visitor's c, else its e
template <bool WALL, int K, class V, class C, class Src>
__device__ __forceinline__ void pair_grad(V dx, V dy, V zi, V zj, const C& c, const V* A, const V* B, Src ce, PairGrad<V>& g)
{
    V dz = sub_(zi, zj);
    const V rho2 = fma_(dy, dy, mul_(dx, dx));
    const V r2 = fma_(dz, dz, rho2);
    const V ri = rsq_(r2), ri2 = mul_(ri, ri), ri3 = mul_(ri, ri2);
    V c1 = fma_(c.template get<C23, V>(), ri3, ri);
    V c2 = mul_(ri3, fma_(c.template get<CM2, V>(), ri2, num_<V>(1.0)));
    V c1p = mul_(ri3, fma_(c.template get<CM1, V>(), ri2, num_<V>(-0.5)));
    V c2p = mul_(mul_(ri3, ri2), fma_(c.template get<C5, V>(), ri2, num_<V>(-1.5)));
    overlap_(r2, ri, c, dx, dy, dz, c1, c2, c1p, c2p);
    // contractions, summed over the right-hand sides
    V S1, S3, Q, R, Z, T1x, T1y, T2x, T2y, qx, qy;
#pragma unroll
    for (int m = 0; m < K; ++m) {
        const V ax = A[3 * m], ay = A[3 * m + 1], az = A[3 * m + 2], bx = B[3 * m], by = B[3 * m + 1], bz = B[3 * m + 2];
        const V cx = ce(3 * m), cy = ce(3 * m + 1), cz = ce(3 * m + 2);
        const V ex = ce(3 * K + 3 * m), ey = ce(3 * K + 3 * m + 1), ez = ce(3 * K + 3 * m + 2);
        const V P1 = fma_(ay, dy, mul_(ax, dx)), P2 = fma_(by, dy, mul_(bx, dx));
        const V D1 = fma_(cy, dy, mul_(cx, dx)), D2 = fma_(ey, dy, mul_(ex, dx));
        S1 = fma_(ay, cy, m ? fma_(ax, cx, S1) : mul_(ax, cx));
        S1 = fma_(by, ey, fma_(bx, ex, S1));
        S3 = fma_(bz, ez, m ? fma_(az, cz, S3) : mul_(az, cz));
        Q = fma_(P2, D2, m ? fma_(P1, D1, Q) : mul_(P1, D1));
        R = fma_(ez, P2, m ? fma_(cz, P1, R) : mul_(cz, P1));
        Z = fma_(bz, D2, m ? fma_(az, D1, Z) : mul_(az, D1));
        T1x = fma_(bz, ex, m ? fma_(az, cx, T1x) : mul_(az, cx));
        T1y = fma_(bz, ey, m ? fma_(az, cy, T1y) : mul_(az, cy));
        T2x = fma_(ez, bx, m ? fma_(cz, ax, T2x) : mul_(cz, ax));
        T2y = fma_(ez, by, m ? fma_(cz, ay, T2y) : mul_(cz, ay));
        qx = fma_(cx, P1, m ? fma_(ax, D1, qx) : mul_(ax, D1));
        qx = fma_(ex, P2, fma_(bx, D2, qx));
        qy = fma_(cy, P1, m ? fma_(ay, D1, qy) : mul_(ay, D1));
        qy = fma_(ey, P2, fma_(by, D2, qy));
    }
    const V A1 = add_(S1, S3), G = add_(R, Z), dS = mul_(dz, S3);
    const V Cc = fma_(dz, add_(G, dS), Q);                // C
    const V gC = fma_(num_<V>(2.0), dS, G);               // dC/dz
    const V Ef = fma_(Cc, c2p, mul_(A1, c1p));            // free-space dE/d(r^2)
    const V two = num_<V>(2.0);
    if constexpr (!WALL) {
        const V k = add_(Ef, Ef), base = mul_(dz, c2);
        g.x = fma_(k, dx, fma_(c2, qx, mul_(base, add_(T1x, T2x))));
        g.y = fma_(k, dy, fma_(c2, qy, mul_(base, add_(T1y, T2y))));
        g.zi = fma_(k, dz, mul_(c2, gC));
        g.zj = neg_(g.zi);
        g.e = fma_(c1, A1, mul_(c2, Cc));
        return;
    }
    const V Rz = add_(zi, zj);
    const V Ri = rsq_(fma_(Rz, Rz, rho2)), w = mul_(Ri, Ri), v = mul_(Ri, w);
    const V t = mul_(Rz, Ri), y = mul_(t, t);
    const V b1 = fma_(c.template get<HWY, V>(), y, c.template get<HW0, V>());     // dh1/dw
    const V d1 = fma_(c.template get<HWY, V>(), w, c.template get<HY, V>());           // dh1/dy
    const V h1 = fma_(w, b1, fma_(c.template get<HY, V>(), y, fma_(mul_(num_<V>(6.0), zi), zj, c.template get<H0, V>())));
    const V aw = fma_(c.template get<HW0, V>(), y, c.template get<AW0, V>());      // diA/dw
    const V ay = fma_(c.template get<HW0, V>(), w, c.template get<H0, V>());            // diA/dy
    const V iA = fma_(w, aw, fma_(mul_(num_<V>(-2.0), zi), zj, fma_(c.template get<H0, V>(), y, c.template get<A0, V>())));
    const V D = sub_(Z, R), RD = mul_(Rz, D), QD = add_(Q, RD);
    const V X = fma_(w, QD, neg_(mul_(y, S3)));                                            // dW/dh1
    const V tz = fma_(c.template get<ZW, V>(), w, c.template get<Z0, V>());
    const V pw = mul_(c.template get<PW, V>(), w), pRD = mul_(pw, RD);
    const V zl = c.template get<ZL, V>();
    const V W = fma_(iA, A1, fma_(h1, X, fma_(w, pRD, mul_(S3, fma_(y, tz, mul_(zl, w))))));
    const V Ww = fma_(b1, X, fma_(h1, QD, fma_(aw, A1, fma_(two, pRD, mul_(S3, fma_(c.template get<ZW, V>(), y, zl))))));
    const V Wy = fma_(A1, ay, fma_(d1, X, mul_(S3, sub_(tz, h1))));
    const V Wu = fma_(num_<V>(6.0), X, mul_(num_<V>(-2.0), A1));
    const V vw = mul_(v, w);
    // dE/d(|R|^2)
    const V in = fma_(num_<V>(1.5), sub_(Cc, W), neg_(fma_(w, Ww, mul_(y, Wy))));
    const V Ew = fma_(vw, in, mul_(mul_(num_<V>(0.5), v), A1));
    const V Pn = mul_(w, add_(h1, pw));                                                    // -P
    const V Rz2 = add_(Rz, Rz);
    const V eR = fma_(v, fma_(Pn, D, mul_(mul_(Rz2, w), Wy)), mul_(Rz2, Ew));              // dE/d(Rz)
    const V c2v = sub_(c2, v), be = fma_(vw, h1, c2v), base = mul_(dz, c2v), vp = mul_(mul_(v, Rz), Pn);
    const V gz = add_(base, vp), gx = sub_(base, vp);
    const V k = mul_(two, add_(Ef, Ew));
    g.x = fma_(k, dx, fma_(be, qx, fma_(gz, T1x, mul_(gx, T2x))));
    g.y = fma_(k, dy, fma_(be, qy, fma_(gz, T1y, mul_(gx, T2y))));
    const V zd = fma_(mul_(two, dz), Ef, mul_(c2v, gC)), vu = mul_(v, Wu);
    g.zi = add_(zd, fma_(vu, zj, eR));
    g.zj = sub_(fma_(vu, zi, eR), zd);
    g.e = fma_(sub_(c1, Ri), A1, fma_(c2v, Cc, mul_(v, W)));
}

// pair_grad, or its sum over the minimum image and the eight nearest ones
template <bool WALL, bool PER, int K, class V, class C, class S, class Src>
__device__ __forceinline__ void pair_grad_images(V dx, V dy, V zi, V zj, const C& c, S Lx, S Ly, const V* A,
                                                 const V* B, Src ce, PairGrad<V>& g)
{
    if constexpr (!PER) {
        pair_grad<WALL, K>(dx, dy, zi, zj, c, A, B, ce, g);
    } else {
        const V zero = num_<V>(0.0);
        g = PairGrad<V>{zero, zero, zero, zero, zero};
#pragma unroll 1
        for (int s = 0; s < 9; ++s) {
            const V sx = bc_(S(s / 3 - 1) * Lx), sy = bc_(S(s % 3 - 1) * Ly);
            PairGrad<V> o;
            pair_grad<WALL, K>(add_(dx, sx), add_(dy, sy), zi, zj, c, A, B, ce, o);
            g = PairGrad<V>{add_(g.x, o.x), add_(g.y, o.y), add_(g.zi, o.zi), add_(g.zj, o.zj), add_(g.e, o.e)};
        }
    }
}

}  // namespace adj
}  // namespace rpbd
