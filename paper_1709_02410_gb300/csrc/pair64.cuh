// The wall-RPY pair block in FP64 (8 pi eta M_ij, heights clamped): the Horner form
// of wall_rpy_x2.cuh with a folded into the constants (lengths stay the caller's:
// scaling x, y by 1/a would round them, at 1e-16 of the box instead of the
// separation).  42 FP64 instructions for the five block scalars and 10 for their
// two reciprocal roots.
#pragma once

#include <cuda_runtime.h>

#include "rpbd_internal.cuh"
#include "wall_rpy.cuh"

namespace rpbd {
namespace pair64 {

// constants of the Horner form for blob radius a (wall_rpy.cuh has the formulas)
struct Const {
    double c23, m2, k_self, k_ovl, i8;       // free space: 2a^2/3, -2a^2, 4/(3a), 3/(8a^2), 1/(8a^2)
    double h0, hy, hw0, hwy;                 // h1 = 6 zi zj + h0 + hy y + w (hw0 + hwy y)
    double a0, ay, aw0, awy;                 // iA = -2 zi zj + a0 + ay y + w (aw0 + awy y)
    double pw, zw, z0, zl;                   // P: -20/3 a^4; Z: 20 a^4, 4 a^2, -8/3 a^4
    long long four_a2;                       // bits of 4 a^2 (non-negative doubles order like their bits)
    double Lx, Ly, iLx, iLy;
    static Const make(const rpbd_params& p)
    {
        Const c;
        const double a2 = p.a * p.a, a4 = a2 * a2;
        c.c23 = 2.0 * a2 / 3.0;
        c.m2 = -2.0 * a2;
        c.k_self = 4.0 / (3.0 * p.a);
        c.k_ovl = 3.0 / (8.0 * a2);
        c.i8 = 1.0 / (8.0 * a2);
        c.h0 = 2.0 * a2;
        c.hy = -10.0 * a2;
        c.hw0 = -10.0 / 3.0 * a4;
        c.hwy = 70.0 / 3.0 * a4;
        c.a0 = -2.0 / 3.0 * a2;
        c.ay = 2.0 * a2;
        c.aw0 = 2.0 / 3.0 * a4;
        c.awy = -10.0 / 3.0 * a4;
        c.pw = -20.0 / 3.0 * a4;
        c.zw = 20.0 * a4;
        c.z0 = 4.0 * a2;
        c.zl = -8.0 / 3.0 * a4;
        const double f = 4.0 * a2;
        static_assert(sizeof(f) == sizeof(c.four_a2), "bits of a double");
        __builtin_memcpy(&c.four_a2, &f, sizeof(f));
        c.Lx = p.Lx;
        c.Ly = p.Ly;
        c.iLx = p.Lx > 0.0 ? 1.0 / p.Lx : 0.0;
        c.iLy = p.Ly > 0.0 ? 1.0 / p.Ly : 0.0;
        return c;
    }
};

// reciprocal distance and free-space c1, g with c2 = g / r^3
__device__ __forceinline__ void free_space(double r2, const Const& c, double& rinv, double& rinv3, double& c1, double& g)
{
    rinv = rsqrt3(r2);
    const double rinv2 = rinv * rinv;
    rinv3 = rinv * rinv2;
    c1 = fma(c.c23, rinv3, rinv);
    g = fma(c.m2, rinv2, 1.0);
    if (__double_as_longlong(r2) < c.four_a2) {  // overlapping or self: rare
        if (r2 > 1e-180) {  // (r^-3 is finite)
            c1 = c.k_self - c.k_ovl * (r2 * rinv);
            g = r2 * c.i8;
        } else {  // (closer than 1e-90: the self block to rounding)
            c1 = c.k_self;
            rinv3 = g = 0.0;
        }
    }
}

// the five block scalars of one pair in the open cell (8 pi eta M, wall_rpy.cuh)
template <bool WALL>
__device__ __forceinline__ void factors(double dx, double dy, double zi, double zi6, double zj, const Const& c, double& al,
                                        double& be, double& gx, double& gz, double& mzz)
{
    const double dz = zi - zj;
    const double rho2 = fma(dy, dy, dx * dx);
    double rinv, rinv3, c1, g;
    free_space(fma(dz, dz, rho2), c, rinv, rinv3, c1, g);
    if (!WALL) {
        be = rinv3 * g;
        al = c1;
        gx = gz = be * dz;
        mzz = fma(dz, gx, c1);
        return;
    }
    const double Rz = zi + zj;
    const double Rinv = rsqrt3(fma(Rz, Rz, rho2));
    const double w = Rinv * Rinv, v = Rinv * w;
    const double t = Rz * Rinv, y = t * t;
    const double c2v = fma(rinv3, g, -v);
    const double h1 = fma(w, fma(c.hwy, y, c.hw0), fma(c.hy, y, fma(zi6, zj, c.h0)));
    const double iA = fma(w, fma(c.awy, y, c.aw0), fma(-2.0 * zi, zj, fma(c.ay, y, c.a0)));
    const double tz = fma(c.zw, w, -(h1 + c.z0));
    const double iZ = fma(y, tz, c.zl * w);
    al = fma(v, iA, c1 - Rinv);
    be = fma(v, w * h1, c2v);
    const double base = dz * c2v;
    const double vp = (t * w) * (w * fma(c.pw, w, h1));  // -v Rz P
    gx = base - vp;
    gz = base + vp;
    mzz = fma(v, iZ, fma(dz, base, al));
}

struct Block {
    double xx, xy, xz, yy, yz, zx, zy, zz;
};

// block summed over the minimum image and its eight neighbours (the scalar
// form of pair_image_sum_x2 in wall_rpy_x2.cuh)
__device__ __forceinline__ void image_sum(double dx0, double dy0, double zi, double zj, const Const& c, Block& M)
{
    const double dz = zi - zj, Rz = zi + zj, dz2 = dz * dz, q = Rz * Rz, u = zi * zj;
    const double hu = fma(6.0, u, c.h0), au = fma(-2.0, u, c.a0);
    dx0 -= c.Lx * rint(dx0 * c.iLx);
    dy0 -= c.Ly * rint(dy0 * c.iLy);
    double al = 0.0, cs = 0.0, zs = 0.0, bxx = 0.0, bxy = 0.0, byy = 0.0, cx = 0.0, cy = 0.0, px = 0.0, py = 0.0;
#pragma unroll 1
    for (int a = -1; a <= 1; ++a) {
        const double dx = fma((double)a, c.Lx, dx0), dxx = dx * dx;
        double rb = 0.0, rby = 0.0, rc = 0.0, rp = 0.0;
#pragma unroll
        for (int b = -1; b <= 1; ++b) {
            const double dy = b == 0 ? dy0 : (b < 0 ? dy0 - c.Ly : dy0 + c.Ly), dyy = dy * dy;
            const double rho2 = dxx + dyy;
            double rinv, rinv3, c1, g;
            free_space(rho2 + dz2, c, rinv, rinv3, c1, g);
            const double Rinv = rsqrt3(rho2 + q);
            const double w = Rinv * Rinv, v = Rinv * w, y = q * w;
            const double c2v = fma(rinv3, g, -v);
            const double h1 = fma(w, fma(c.hwy, y, c.hw0), fma(c.hy, y, hu));
            const double iA = fma(w, fma(c.awy, y, c.aw0), fma(c.ay, y, au));
            const double iZ = fma(y, fma(c.zw, w, -(h1 + c.z0)), c.zl * w);
            const double vP = v * (w * fma(c.pw, w, h1));
            const double be = fma(v, w * h1, c2v);
            al += fma(v, iA, c1 - Rinv);
            zs = fma(v, iZ, zs);
            rb += be;
            rby = fma(be, dy, rby);
            byy = fma(be, dyy, byy);
            rc += c2v;
            cy = fma(c2v, dy, cy);
            rp += vP;
            py = fma(vP, dy, py);
        }
        bxx = fma(rb, dxx, bxx);
        bxy = fma(rby, dx, bxy);
        cx = fma(rc, dx, cx);
        cs += rc;
        px = fma(rp, dx, px);
    }
    M.xx = al + bxx;
    M.xy = bxy;
    M.yy = al + byy;
    M.xz = fma(dz, cx, -(Rz * px));
    M.yz = fma(dz, cy, -(Rz * py));
    M.zx = fma(dz, cx, Rz * px);
    M.zy = fma(dz, cy, Rz * py);
    M.zz = fma(dz2, cs, al) + zs;
}

// the block's entries, or its sum over the images
template <bool WALL, bool PER>
__device__ __forceinline__ void block(double dx, double dy, double zi, double zj, const Const& c, Block& M)
{
    if constexpr (PER) {
        image_sum(dx, dy, zi, zj, c, M);
    } else {
        double al, be, gx, gz;
        factors<WALL>(dx, dy, zi, 6.0 * zi, zj, c, al, be, gx, gz, M.zz);
        const double bx = be * dx, by = be * dy;
        M.xx = fma(bx, dx, al);
        M.xy = bx * dy;
        M.yy = fma(by, dy, al);
        M.xz = dx * gx;
        M.yz = dy * gx;
        M.zx = dx * gz;
        M.zy = dy * gz;
    }
}

}  // namespace pair64
}  // namespace rpbd
