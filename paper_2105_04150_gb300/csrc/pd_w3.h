// Three-word FP32 node records and the double-word bond arithmetic on them
// (device code only), for kernels whose results have to be FP64-grade.
//
// A value v (a position or displacement component in units of a power of two U
// no smaller than the longest bond of the model) is split into
//   h  v rounded to FP32, to a multiple of a grid 2^g
//   m  the remainder v - h rounded to a multiple of 2^(g - 23)
//   t  what is left, |t| <= 1.25 2^(g - 24)
// Positions have one grid for the whole model (each instance of a batch), that of
// its largest |x|; t is kept as an 11-bit integer (in units of 2^(g - 33)).
// Displacements have g = -22 below 4 and their own FP32 grid above; t is kept to 13
// bits.  So h + m + t holds 57 bits of the largest position and 2^-59 U of a
// displacement, or every bit of an FP64 displacement above 4 U.
// The words of two bonded nodes lie on grids at most a factor 2 apart, so their
// differences dh and dm are exact FP32 operations (|dh| <= 2.02 = the largest
// component difference of a bond that is stretched by less than kW3XMax, and
// |dm| <= 1.75 2^g), and dh + dm + dt, renormalised with one fast two-sum (dh is
// zero or its exponent no smaller than dm's), is the difference of the two values.
// The difference of two plain double-words costs more (a two-sum for the leading
// words, whose grids differ) and keeps only 2^-48 of |v|.
//
// Record: two 32-byte sectors, each one 256-bit load
//   {xh.x, xh.y, xh.z, uh.x | uh.y, uh.z, t.x, t.y}
//   {xm.x, xm.y, xm.z, um.x | um.y, um.z, t.z, 0}
// word t.c holds the integer t of x_c, biased, in its low 11 bits and above them
// the leading 21 bits of the t of u_c, an FP32 number.
#pragma once

#include <cuda_runtime.h>

#include "pd_dw.h"
#include "pd_internal.h"

namespace pd {
namespace w3 {

using dwa::Dw;
using dwa::Rec;
using dwa::dw_add;
using dwa::dw_mul;
using dwa::two_sum;

// Bonds with |x| = ||y|^2 / |xi|^2 - 1| past kW3XMax (a stretch of 0.78 %) are left
// to the literal FP64 evaluation of Eq. 4, which has the smaller error there: its
// stretch carries an absolute rounding error of about 3e-16, i.e. 3e-16 / s of the
// bond's force, against the 1e-14 of bond_w3.

struct Own {
    float xh[3], xm[3], xk[3], uh[3], um[3], ut[3];
};

// 2^23 + the integer t of a packed word's position
__device__ __forceinline__ float k_of(float w)
{
    return __uint_as_float((__float_as_uint(w) & 0x7ffu) | 0x4b000000u);
}

// the t of a packed word's displacement
__device__ __forceinline__ float ut_of(float w)
{
    return __uint_as_float(__float_as_uint(w) & ~0x7ffu);
}

__device__ __forceinline__ Own own_words(const Rec& r)
{
    Own o;
    o.xh[0] = r.a0.x; o.xh[1] = r.a0.y; o.xh[2] = r.a0.z;
    o.uh[0] = r.a0.w; o.uh[1] = r.a1.x; o.uh[2] = r.a1.y;
    o.xm[0] = r.b0.x; o.xm[1] = r.b0.y; o.xm[2] = r.b0.z;
    o.um[0] = r.b0.w; o.um[1] = r.b1.x; o.um[2] = r.b1.y;
    const float t[3] = {r.a1.z, r.a1.w, r.b1.z};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        o.xk[c] = k_of(t[c]);
        o.ut[c] = ut_of(t[c]);
    }
    return o;
}

__device__ __forceinline__ float pow2(int e) { return __uint_as_float((uint32_t)(127 + e) << 23); }

// v = h + m + t (see above); g: the grid's exponent, or the smallest one
__device__ __forceinline__ void split3(double v, int g, float& h, float& m, float& t)
{
    h = rintf((float)v * pow2(-g)) * pow2(g);  // beyond 2^(g + 23): v's own FP32 grid
    const double r = v - (double)h;
    g = max((int)((__float_as_uint(h) >> 23) & 0xffu) - 127 - 23, g);
    // (an overflowing v makes h or r non-finite, and the literal evaluation takes over)
    g = min(max(g, -100), 100);
    m = rintf((float)r * pow2(23 - g)) * pow2(g - 23);
    t = (float)(r - (double)m);
}

// the biased integer t of a position (grid exponent g)
__device__ __forceinline__ uint32_t t_int(float xt, int g)
{
    return (uint32_t)min(max((int)rintf(xt * pow2(24 - g) * 512.0f) + 1024, 0), 2047);
}

// the packed third words of one component
__device__ __forceinline__ float pack_t(uint32_t k, float ut)
{
    return __uint_as_float(((__float_as_uint(ut) + 0x400u) & ~0x7ffu) | k);
}

// the difference j - i of one component as a double-word: dh + dm + dt ts
__device__ __forceinline__ Dw diff3(float jh, float jm, float ih, float im, float dt, float ts)
{
    const float dh = jh - ih, dm = jm - im;
    const float s = dh + dm;
    return {s, fmaf(dt, ts, dm - (s - dh))};
}

// One bond of the lane's node (in units of U).
struct Geo {
    Dw xi[3], et[3];  // xi = x_j - x_i, eta = u_j - u_i
    Dw y[3];          // xi + eta
    Dw x;             // |y|^2 / |xi|^2 - 1
    Dw z;             // |xi| / |y| - 1
};

// il: the slot's U / |xi| as a double-word; ts: the unit of the positions' t.
// num = eta . (2 xi + eta) = |y|^2 - |xi|^2 without cancellation, x = num / |xi|^2,
// and with r = sqrt(1 + x) = |y| / |xi|: s / |y| = (1 - 1/r) / |xi|.  z = 1/r - 1 is
// a small number, so it is formed by itself: seeded in FP32 as -x / (r (1 + r))
// and corrected by one Newton step on f(z) = (1 + z)^2 (1 + x) - 1 whose residual
// (2z + z^2 + x) + x (2z + z^2) is taken in double-word arithmetic (its leading
// terms cancel exactly).  23 operations, against 45 for the double-word square
// root, reciprocal and quotient of the direct form; relative error < 2^-44.
__device__ __forceinline__ Geo bond_geo(const Own& o, const Rec& j, const float2 il, float ts)
{
    const float jxh[3] = {j.a0.x, j.a0.y, j.a0.z}, juh[3] = {j.a0.w, j.a1.x, j.a1.y};
    const float jxm[3] = {j.b0.x, j.b0.y, j.b0.z}, jum[3] = {j.b0.w, j.b1.x, j.b1.y};
    const float jt[3] = {j.a1.z, j.a1.w, j.b1.z};
    Geo out;
    Dw nm[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        out.xi[c] = diff3(jxh[c], jxm[c], o.xh[c], o.xm[c], k_of(jt[c]) - o.xk[c], ts);
        out.et[c] = diff3(juh[c], jum[c], o.uh[c], o.um[c], ut_of(jt[c]) - o.ut[c], 1.0f);
        out.y[c] = dw_add(out.xi[c], out.et[c]);
        nm[c] = dw_mul(out.et[c], dw_add(out.xi[c], out.y[c]));  // eta_c (2 xi_c + eta_c)
    }
    Dw num = two_sum(nm[0].h, nm[1].h);
    num.l += nm[0].l + nm[1].l;
    num = dw_add(num, nm[2]);
    const Dw iL{il.x, il.y};
    const Dw x = dw_mul(dw_mul(num, iL), iL);
    const float x1 = 1.0f + x.h;
    const float r = x1 * dwa::rsqrt_seed(x1);
    const float z0 = -x.h * dwa::rcp_seed(fmaf(r, r, r));
    // p = 2 z0 + z0^2 as a double-word
    const float zz = z0 * z0, ph = fmaf(2.0f, z0, zz);
    const Dw p{ph, (zz - fmaf(-2.0f, z0, ph)) + fmaf(z0, z0, -zz)};
    const Dw xp = dw_mul(x, p);
    const float R = ((ph + x.h) + xp.h) + ((p.l + x.l) + xp.l);
    out.x = x;
    out.z = Dw{z0, R * fmaf(z0, -0.5f, -0.5f)};
    return out;
}

struct Bond {
    Dw x;     // |y|^2 / |xi|^2 - 1
    Dw coef;  // -s / |y| (in 1 / U)
    Dw y[3];  // deformed bond vector (in U)
};

__device__ __forceinline__ Bond bond_w3(const Own& o, const Rec& j, const float2 il, float ts)
{
    const Geo g = bond_geo(o, j, il, ts);
    return {g.x, dw_mul(g.z, Dw{il.x, il.y}), {g.y[0], g.y[1], g.y[2]}};
}

}  // namespace w3
}  // namespace pd
