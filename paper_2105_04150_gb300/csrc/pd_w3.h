// Three-word FP32 node records and the double-word bond arithmetic on them
// (device code only), for kernels whose results have to be FP64-grade.
//
// A value v (a position or displacement component in units of a power of two U
// no smaller than the longest bond of the model) is split into
//   h  v rounded to FP32, to a multiple of a grid 2^g
//   m  the remainder v - h rounded to a multiple of 2^(g - 23)
//   t  what is left, |t| <= 1.25 2^(g - 24)
// Positions, counted along each axis from the body's near end where it lies away from the
// origin (an exact difference), have one grid for the whole model (each instance of a
// batch), that of its largest |x|; t is kept as an 11-bit integer (in units of 2^(g - 33)).
// Displacements have g = -22 below 4 and their own FP32 grid above; t is kept to 13
// bits.  So h + m + t holds 57 bits of the largest position and 2^-59 U of a
// displacement, or every bit of an FP64 displacement above 4 U.
// The words of two bonded nodes lie on grids at most a factor 2 apart, so their
// differences dh and dm are exact FP32 operations (|dh| <= 2.23, the largest component of
// eta of a bond with |y|^2 <= 1.5 |xi|^2 however it turned, below the 4 that 24 bits of a
// grid of 2^-22 hold, and |dm| <= 1.75 2^g), and dh + dm + dt, renormalised with one fast two-sum (dh is
// zero or its exponent no smaller than dm's), is the difference of the two values.
// The difference of two plain double-words costs more (a two-sum for the leading
// words, whose grids differ) and keeps only 2^-48 of |v|.
//
// Record: two 32-byte sectors, each one 256-bit load
//   {xh.x, xh.y, uh.x, uh.y | xh.z, uh.z, t.x, t.y}
//   {xm.x, xm.y, um.x, um.y | xm.z, um.z, t.z, 0}
// word t.c holds the integer t of x_c, biased, in its low 11 bits and above them
// the leading 21 bits of the t of u_c, an FP32 number.
//
// Paired arithmetic: sm_103a's paired FP32 instructions do two operations in one
// issue slot.  A bond's (x, y) components, and z of xi and of eta, are adjacent in the
// record for that; from num on the two bonds of a chunk are a pair (the slots'
// U / |xi| are stored by pairs of slots).  Each half is rounded as the scalar operation.
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

// Range of the arithmetic: |x| = ||y|^2 / |xi|^2 - 1| <= 1/2 (kW3XWide: there the leading
// terms of the Newton residuals cancel exactly), the whole of it on PD_PREC_DW handles,
// whose contract is about 1e-13 of the bond's force.  (Up to 0.78 % only, the bonds past it
// in FP64, a step of a body at 2 % strain took 6.7 times as long: 220k nodes 1621 instead
// of 242 us, state-based 4280 / 488.)
// FP64 handles leave the double-word form where the literal FP64 evaluation of Eq. 4 has the
// smaller error.  That one rounds s at an absolute 1.1e-16 rms at any stretch and rotation;
// this one has a relative error, of the bond and of the force sum (renormalised with every
// pair of bonds), that reaches it at a stretch of 0.5 % (force of an irregular body against
// the exact sum, in the literal form's rms error: 0.66 at 0.4 %, 1.04 at 0.6 %) and, the
// state-based force having the coherent error of the dilation, at 0.35 %: kW3XMax and
// kW3XMaxOsb.  And num = eta . (2 xi + eta) cancels when a bond turns: its terms of size
// |eta| |xi| carry 2^-47 each, so s an absolute error (rms, on random lattice bonds) of
// 2.4e-17, 1.2e-16, 7e-16 and 4.2e-15 at 0.01, 0.05, 0.3 and pi/2 rad.  So bonds with a
// component of eta past kW3EtaMax |xi| (about 1 to 1.5 degrees) are literal too.
// PD_PREC_DW, about 1e-13 of the force and no less than 46 bits of |y|, has no such bounds.
// The positions' grid adds 1.4 2^(g - 33) of s, nothing that shows while the largest position
// is below 512 U; in longer bodies, near whose origin FP64 coordinates are finer than the
// grid, the bounds of FP64 handles shrink with it (w3_s_grid: without that a line of 66,000
// horizons had 50 times the literal form's error there at a stretch of 0.7 %).

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
    o.xh[0] = r.a0.x; o.xh[1] = r.a0.y; o.xh[2] = r.a1.x;
    o.uh[0] = r.a0.z; o.uh[1] = r.a0.w; o.uh[2] = r.a1.y;
    o.xm[0] = r.b0.x; o.xm[1] = r.b0.y; o.xm[2] = r.b1.x;
    o.um[0] = r.b0.z; o.um[1] = r.b0.w; o.um[2] = r.b1.y;
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

// the same number with |l| at most half an ulp of h (fast two-sum)
__device__ __forceinline__ Dw renorm(Dw a)
{
    const float s = __fadd_rn(a.h, a.l);
    return {s, __fsub_rn(a.l, __fsub_rn(s, a.h))};
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
    float x;          // |y|^2 / |xi|^2 - 1
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
    const float jxh[3] = {j.a0.x, j.a0.y, j.a1.x}, juh[3] = {j.a0.z, j.a0.w, j.a1.y};
    const float jxm[3] = {j.b0.x, j.b0.y, j.b1.x}, jum[3] = {j.b0.z, j.b0.w, j.b1.y};
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
    const float xs = x.h + x.l;  // (see stretch2)
    const float x1 = 1.0f + xs;
    const float r = x1 * dwa::rsqrt_seed(x1);
    const float z0 = -xs * dwa::rcp_seed(fmaf(r, r, r));
    // p = 2 z0 + z0^2 as a double-word
    const float zz = __fmul_rn(z0, z0), ph = fmaf(2.0f, z0, zz);
    const Dw p{ph, (zz - fmaf(-2.0f, z0, ph)) + fmaf(z0, z0, -zz)};
    const Dw xp = dw_mul(x, p);
    const float R = __fadd_rn(__fadd_rn(ph, x.h), xp.h) + ((p.l + x.l) + xp.l);
    out.x = xs;
    out.z = Dw{z0, R * fmaf(z0, -0.5f, -0.5f)};
    return out;
}

// ---- two bonds at a time ----------------------------------------------------

// two double-words, one per half
struct Dw2 {
    float2 h, l;
};
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }
// a - b (a product by -1 is exact, so this is one rounding)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, both(-1.0f), a); }

__device__ __forceinline__ Dw2 two_sum2(float2 a, float2 b)
{
    const float2 s = add2(a, b);
    const float2 bb = sub2(s, a);
    return {s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ Dw2 dw_add2(Dw2 a, Dw2 b)
{
    Dw2 t = two_sum2(a.h, b.h);
    t.l = add2(t.l, add2(a.l, b.l));
    return t;
}
__device__ __forceinline__ Dw2 dw_mul2(Dw2 a, Dw2 b)
{
    const float2 p = mul2(a.h, b.h);
    const float2 e = make_float2(fmaf(a.h.x, b.h.x, -p.x), fmaf(a.h.y, b.h.y, -p.y));
    return {p, fma2(a.h, b.l, fma2(a.l, b.h, e))};
}
// the same numbers with |l| at most half an ulp of h (fast two-sum)
__device__ __forceinline__ Dw2 renorm2(Dw2 a)
{
    const float2 s = add2(a.h, a.l);
    return {s, sub2(a.l, sub2(s, a.h))};
}
// the difference of two records' pairs, as diff3
__device__ __forceinline__ Dw2 diff3_2(float2 jh, float2 jm, float2 nh, float2 nm, float2 dt,
                                       float2 ts)
{
    const float2 dh = add2(jh, nh), dm = add2(jm, nm);
    const float2 s = add2(dh, dm);
    return {s, fma2(dt, ts, sub2(dm, sub2(s, dh)))};
}

// The lane's own words, negated, in the pairs of the record.
struct Own2 {
    float2 xh, uh, zh, xm, um, zm;  // (x, y) of x and u; (x_z, u_z)
    float2 xk, ut, zt;              // the third words likewise
};
__device__ __forceinline__ Own2 own_pairs(const Rec& r)
{
    Own2 o;
    o.xh = make_float2(-r.a0.x, -r.a0.y);
    o.uh = make_float2(-r.a0.z, -r.a0.w);
    o.zh = make_float2(-r.a1.x, -r.a1.y);
    o.xm = make_float2(-r.b0.x, -r.b0.y);
    o.um = make_float2(-r.b0.z, -r.b0.w);
    o.zm = make_float2(-r.b1.x, -r.b1.y);
    o.xk = make_float2(-k_of(r.a1.z), -k_of(r.a1.w));
    o.ut = make_float2(-ut_of(r.a1.z), -ut_of(r.a1.w));
    o.zt = make_float2(-k_of(r.b1.z), -ut_of(r.b1.z));
    return o;
}

// xi and eta of one bond: the (x, y) components and z
struct Pair {
    Dw2 xi, et;
    Dw xz, ez;
};
__device__ __forceinline__ Pair pair_of(const Own2& o, const Rec& j, float2 ts2, float2 tsz)
{
    Pair p;
    p.xi = diff3_2(make_float2(j.a0.x, j.a0.y), make_float2(j.b0.x, j.b0.y), o.xh, o.xm,
                   add2(make_float2(k_of(j.a1.z), k_of(j.a1.w)), o.xk), ts2);
    const float2 dt = add2(make_float2(ut_of(j.a1.z), ut_of(j.a1.w)), o.ut);
    {
        const float2 dh = add2(make_float2(j.a0.z, j.a0.w), o.uh);
        const float2 dm = add2(make_float2(j.b0.z, j.b0.w), o.um);
        const float2 s = add2(dh, dm);
        p.et = Dw2{s, add2(dt, sub2(dm, sub2(s, dh)))};
    }
    const Dw2 zz = diff3_2(make_float2(j.a1.x, j.a1.y), make_float2(j.b1.x, j.b1.y), o.zh, o.zm,
                           add2(make_float2(k_of(j.b1.z), ut_of(j.b1.z)), o.zt), tsz);
    p.xz = Dw{zz.h.x, zz.l.x};
    p.ez = Dw{zz.h.y, zz.l.y};
    return p;
}

// eta . v
__device__ __forceinline__ Dw eta_dot(const Pair& p, Dw2 v, Dw vz)
{
    const Dw2 n2 = dw_mul2(p.et, v);
    const Dw nz = dw_mul(p.ez, vz);
    Dw num = two_sum(n2.h.x, n2.h.y);
    num.l += n2.l.x + n2.l.y;
    return dw_add(num, nz);
}

// the largest |component| of eta
__device__ __forceinline__ float eta_max(const Pair& p)
{
    return fmaxf(fmaxf(fabsf(p.et.h.x), fabsf(p.et.h.y)), fabsf(p.ez.h));
}

// y = xi + eta and num = eta . (2 xi + eta) of one bond
struct Kin {
    Dw2 y;   // x, y components
    Dw yz;
    Dw num;
    float e;  // eta_max
};
__device__ __forceinline__ Kin kin(const Own2& o, const Rec& j, float2 ts2, float2 tsz)
{
    const Pair p = pair_of(o, j, ts2, tsz);
    Kin k;
    k.y = dw_add2(p.xi, p.et);
    k.yz = dw_add(p.xz, p.ez);
    k.num = eta_dot(p, dw_add2(p.xi, k.y), dw_add(p.xz, k.yz));
    k.e = eta_max(p);
    return k;
}

// num alone: without y, 24 operations less
struct KinNum {
    Dw num;
    float e;
};
__device__ __forceinline__ KinNum kin_num(const Own2& o, const Rec& j, float2 ts2, float2 tsz)
{
    const Pair p = pair_of(o, j, ts2, tsz);
    const Dw2 x2{add2(p.xi.h, p.xi.h), add2(p.xi.l, p.xi.l)};
    return {eta_dot(p, dw_add2(x2, p.et), dw_add(Dw{p.xz.h + p.xz.h, p.xz.l + p.xz.l}, p.ez)),
            eta_max(p)};
}

// x = |y|^2 / |xi|^2 - 1 and z = |xi| / |y| - 1 of two bonds (see bond_geo).  x is the sum of
// both words: in a turned bond num's low word is 2^-24 of terms that cancel, so its leading
// word alone misses num by 1e-5 of it at one degree and a stretch of 1e-4, and by more at
// more, past the margin of the comparison with x_hi (bonds above s_c did not break).  As the
// seed of z too the sum lengthens the chain (242 -> 245 us a step); Newton's step does not
// need it.
struct Stretch2 {
    float2 x;
    Dw2 z;
};
__device__ __forceinline__ Stretch2 stretch2(Dw2 num, const float4 il)
{
    const Dw2 iL{make_float2(il.x, il.y), make_float2(il.z, il.w)};
    const Dw2 x = dw_mul2(dw_mul2(num, iL), iL);
    const float2 x1 = add2(both(1.0f), x.h);
    const float2 r = mul2(x1, make_float2(dwa::rsqrt_seed(x1.x), dwa::rsqrt_seed(x1.y)));
    const float2 den = fma2(r, r, r);
    const float2 nx = mul2(x.h, both(-1.0f));
    const float2 z0 = mul2(nx, make_float2(dwa::rcp_seed(den.x), dwa::rcp_seed(den.y)));
    const float2 zz = mul2(z0, z0), ph = fma2(both(2.0f), z0, zz);
    const float2 e = make_float2(fmaf(z0.x, z0.x, -zz.x), fmaf(z0.y, z0.y, -zz.y));
    const Dw2 p{ph, add2(sub2(zz, fma2(both(-2.0f), z0, ph)), e)};
    const Dw2 xp = dw_mul2(x, p);
    const float2 R = add2(add2(add2(ph, x.h), xp.h), add2(add2(p.l, x.l), xp.l));
    return {add2(x.h, x.l), Dw2{z0, mul2(R, fma2(z0, both(-0.5f), both(-0.5f)))}};
}

// eta past eta_max |xi| (il: the slot's U / |xi|)
__device__ __forceinline__ bool turned(float e, float il, float eta_max) { return e * il >= eta_max; }

// Which of two live bonds are to be evaluated literally: near or past s_c or past x_max
// (x_hi), past -x_max, or not a number.  (Turned bonds of FP64 handles: elsewhere.)
__device__ __forceinline__ uint32_t literal_of(float2 x, float x_hi, float x_max, uint32_t live)
{
    const bool A = !(x.x < x_hi) || !(x.x > -x_max);
    const bool B = !(x.y < x_hi) || !(x.y > -x_max);
    return ((A ? 1u : 0u) | (B ? 2u : 0u)) & live;
}

// x of two bonds and (1 / |xi|) z = -s / |y|
struct Coef2 {
    float2 x;
    Dw2 c;
};
__device__ __forceinline__ Coef2 coef2(Dw a, Dw b, const float4 il)
{
    const Stretch2 t = stretch2(Dw2{make_float2(a.h, b.h), make_float2(a.l, b.l)}, il);
    return {t.x, dw_mul2(t.z, Dw2{make_float2(il.x, il.y), make_float2(il.z, il.w)})};
}

}  // namespace w3
}  // namespace pd
