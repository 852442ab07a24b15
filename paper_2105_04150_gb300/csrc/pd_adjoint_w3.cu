// Reverse step of the adjoint with most of its work off the FP64 pipe (sm_103a); it
// computes what k_adj_step (pd_adjoint.cu) computes:
//
//   ubar^n_m = ubar_m + (dt/rho) sum_j c_mj K_mj d_mj,  d_mj = V_m w_j - V_j w_m
//   vbar^n_m = (1 - dt eta/rho) w_m
//   dL/dc[m->j] += (dt/rho) s V_j (y/|y|).w_m
//
// with K = (1/L - 1/|y|) I + y y^T / |y|^3.  k_adj_step spends about 60 FP64
// operations on a bond, each in the time of 64 FP32 ones: 1.14 ms per reverse step of
// a 100k-node plate.  Written about the undeformed bond, with z = L/|y| - 1 and
// q = (1 + z)^3,
//
//   K d = e (e.d),  e = xi / L^(3/2)                        (FP64: 9 operations)
//       + [xi (B + (q - 1)(A + B)) + eta q (A + B)] / L^3 - (z / L) d,
//   A = xi.d, B = eta.d,
//
// e is a constant of the slot, stored (24 bytes streamed cost less than the five
// operations that form it: 0.34 ms a step of the 100k plate with xi and 1 / L^3, 0.31 so,
// the FP64 pipe 69 % busy).  The second line is smaller than the first by |eta| / L, 1e-4 to 1e-2, so the
// double-word arithmetic of pd_w3.h (relative 1e-14) gives it to FP64's rounding
// of the whole; it runs on the FP32 pipe beside the FP64 one.  dL/dc needs the
// stretch, which is more accurate in double-words than in the literal FP64 form
// (whose s has an absolute error of 3e-16).  Bonds with |eta| / L past kW3EtaMax or past
// kW3XMax, or whose w differ in bucket, are evaluated literally in FP64: 0.35 ms
// a step of a 16k plate at 2 % strain, 0.08 at rest (all of it literal before: 0.60).  The
// per-slot sums of dL/dc over the steps are FP64: two additions a bond.
//
// PD_PREC_DW handles (F64 false) take K d = y q (A + B) / L^3 - (z / L) d in double-word
// arithmetic as a whole, to 2^-44 of each bond's term: no FP64 operation but the two of
// dL/dc and no e, and the whole range of pd_w3.h, at any rotation.
//
// The FP64 pipe needs few warps and a model of this use is small (the recorded run
// is kept in memory), so a slice is shared by a block of four warps, each taking
// every fourth slot; their sums are added in a fixed order.
#include <cuda_runtime.h>

#include "pd_internal.h"
#include "pd_w3.h"

namespace pd {
namespace {

using namespace w3;

constexpr int kTeam = 4;

int grid_of(int64_t work)
{
    const int64_t b = (work + 255) / 256;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 16));
}

// four FP64 words of a node's record in one 256-bit load
struct D4 {
    double x, y, z, w;
};
__device__ __forceinline__ D4 ld_d4(const double* p)
{
    D4 r;
    asm volatile("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];"
                 : "=d"(r.x), "=d"(r.y), "=d"(r.z), "=d"(r.w)
                 : "l"(p));
    return r;
}

// Largest |component| of the seeds as they enter w = vbar + dt ubar, into *out
// (zeroed before; the bits of non-negative doubles are ordered like integers).
__global__ void k_adj_scale(const double* __restrict__ ub, const double* __restrict__ vb, int64_t n3,
                            double dt, unsigned long long* __restrict__ out)
{
    double m = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n3;
         e += (int64_t)gridDim.x * blockDim.x)
        m = fmax(m, fmax(fabs(vb[e]), dt * fabs(ub[e])));
    if (m > 0.0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// power of two that brings that component to [1, 2), as far as it is a finite number (1
// without seeds)
__device__ __forceinline__ double unit_scale(const unsigned long long* m)
{
    const double v = __longlong_as_double((long long)*m);
    return v > 0.0 && v < 1e300 ? scalbn(1.0, min(-ilogb(v), 1000)) : 1.0;
}

// Far from a local seed w is smaller by any number of orders of magnitude, over most of the
// body for as long as no wave has reached it.  So a node's double-words are in a unit of its
// own, 2^(-104 B) of that one, its bucket B chosen so that its largest component lies above
// 2^-64 in it, where FP32 holds its products with s / |y|, low words included (in buckets
// past 0 up to 2^40, well inside FP32).  Bonds between buckets are evaluated literally.
// (All bonds of nodes past bucket 0 literally: 1313 ms for the gradient of 2000 steps of a
// 100k plate with a loss of two nodes, 1192 so; 1160 without regard to the range.)
// The record holds the bucket as the float whose bits are (896 - 104 B) << 20, the exponent
// offset from FP32 to FP64 of such a word (wide_of), and not-a-number, which equals no
// bucket, past bucket 8.
__device__ __forceinline__ float w_bucket(double w_max)
{
    const int e = (int)((uint32_t)__double2hiint(w_max) >> 20) - 1023;
    const int B = e >= -63 || w_max == 0.0 ? 0 : 1 + (-64 - e) / 104;
    return __uint_as_float(B <= 8 ? (896u - 104u * (uint32_t)B) << 20 : 0x7fc00000u);
}
// 2^(104 B) and its reciprocal
__device__ __forceinline__ double bucket_up(float b)
{
    return __hiloint2double((int)(((1023u + 896u) << 20) - __float_as_uint(b)), 0);
}
__device__ __forceinline__ double bucket_down(float b)
{
    return __hiloint2double((int)(((1023u - 896u) << 20) + __float_as_uint(b)), 0);
}

// The records of a reverse step for node p, from its ubar, vbar and u^n: w = ws (vbar + dt
// ubar) with the controlled components of ubar and vbar zeroed (as k_adj_mask), the
// three-word record of x (its words from `fwd`) and u^n, w in FP64 ({w, 0}) and w as
// double-words in units of 2^(-104 B) / unit_scale ({wh, wl.x} {wl.y, wl.z, B, 0}).
__device__ __forceinline__ void adj_records(const AdjW3Args& a, int64_t p, uint32_t mask,
                                            const double (&ub)[3], const double (&vb)[3],
                                            const double* un, double dt, double ws, double us,
                                            const Rec& fwd, float4* rec, double* w64, float4* wdw)
{
    const float tin[3] = {fwd.a1.z, fwd.a1.w, fwd.b1.z};
    float uh[3], um[3], t[3], wh[3], wl[3];
    double w[3];
    for (int k = 0; k < 3; ++k) {
        const bool ctl = (mask >> k) & 1u;
        const double u = ctl ? 0.0 : ub[k];
        const double v = ctl ? 0.0 : vb[k];
        w[k] = ws * (v + dt * u);
        a.ubm[3 * p + k] = u;
        float ut;
        split3(un[3 * p + k] * a.scale, kW3UGrid, uh[k], um[k], ut);
        t[k] = pack_t(__float_as_uint(tin[k]) & 0x7ffu, ut);
    }
    const double w_max = fmax(fabs(w[0]), fmax(fabs(w[1]), fabs(w[2]))), v_max = w_max * us;
    float bucket = w_bucket(v_max);
    if (v_max == 0.0 && w_max > 0.0) bucket = __uint_as_float(0x7fc00000u);
    const double up = bucket == bucket ? bucket_up(bucket) : 1.0;
    for (int k = 0; k < 3; ++k) {
        const double v1 = w[k] * us * up;
        wh[k] = (float)v1;
        wl[k] = (float)(v1 - (double)wh[k]);
    }
    double2* wr = reinterpret_cast<double2*>(w64 + 4 * p);
    wr[0] = make_double2(w[0], w[1]);
    wr[1] = make_double2(w[2], 0.0);
    dwa::st_rec(rec + 4 * p, make_float4(fwd.a0.x, fwd.a0.y, uh[0], uh[1]),
                make_float4(fwd.a1.x, uh[2], t[0], t[1]));
    dwa::st_rec(rec + 4 * p + 2, make_float4(fwd.b0.x, fwd.b0.y, um[0], um[1]),
                make_float4(fwd.b1.x, um[2], t[2], 0.0f));
    dwa::st_rec(wdw + 2 * p, make_float4(wh[0], wh[1], wh[2], wl[0]),
                make_float4(wl[1], wl[2], bucket, 0.0f));
}

__global__ void k_adj_prep_w3(const __grid_constant__ AdjW3Args a, double dt, double ws, int64_t n_pad)
{
    const double us = unit_scale(a.wmax);
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n_pad;
         p += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t cls = a.bcc[p];
        Rec f;
        f.a0 = a.fwd[4 * p];
        f.a1 = a.fwd[4 * p + 1];
        f.b0 = a.fwd[4 * p + 2];
        f.b1 = a.fwd[4 * p + 3];
        const double ub[3] = {a.ub[3 * p], a.ub[3 * p + 1], a.ub[3 * p + 2]};
        const double vb[3] = {a.vb[3 * p], a.vb[3 * p + 1], a.vb[3 * p + 2]};
        adj_records(a, p, cls ? a.bct[cls].mask : 0u, ub, vb, a.un, dt, ws, us, f, a.rec, a.w64,
                    a.wdw);
    }
}

// One bond literally in FP64: K d (without V_ref and c_ij) into f, and
// (s / |y|) y.w_m (times V_j / V_ref) as the return value.
__device__ __noinline__ double literal_adj(const AdjW3Args& a, int64_t m, int64_t j, int64_t slot,
                                           double* f)
{
    double y[3], d[3], y2 = 0.0, yd = 0.0, yw = 0.0;
    const double vm = a.uniform_w ? 1.0 : a.vol[m] * a.inv_vref, vj = a.uniform_w ? 1.0 : a.vol[j] * a.inv_vref;
    for (int k = 0; k < 3; ++k) {
        y[k] = (a.x64[8 * j + k] - a.x64[8 * m + k]) + (a.un[3 * j + k] - a.un[3 * m + k]);
        d[k] = vm * a.w64[4 * j + k] - vj * a.w64[4 * m + k];
        y2 += y[k] * y[k];
        yd += y[k] * d[k];
        yw += y[k] * a.w64[4 * m + k];
    }
    const double iL = a.ilen[slot], ir = rsqrt_nr(y2);
    const double s = fma(y2 * ir, iL, -1.0);
    const double k1 = iL - ir, k2 = yd * (ir * ir * ir);
    for (int k = 0; k < 3; ++k) f[k] = k1 * d[k] + y[k] * k2;
    return s * vj * yw * ir;
}

__device__ __forceinline__ Dw dot3(const Dw (&a)[3], const Dw (&b)[3])
{
    Dw s = dw_mul(a[0], b[0]);
    s = dw_add(s, dw_mul(a[1], b[1]));
    return dw_add(s, dw_mul(a[2], b[2]));
}

// v 2^(-104 B) in FP64 by integer operations: a conversion instruction takes a turn of the
// FP64 pipe (2 % of the sweep of a 100k plate).  Denormal numbers become 0.
__device__ __forceinline__ double wide_of(float v, float bucket)
{
    const uint32_t b = __float_as_uint(v);
    const uint32_t hi = (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + __float_as_uint(bucket));
    return (b & 0x7f800000u) != 0u ? __hiloint2double((int)hi, (int)(b << 29)) : 0.0;
}

template <bool UW, bool F64>
__global__ void __launch_bounds__(32 * kTeam, 4) k_adj_step_w3(const __grid_constant__ AdjW3Args a)
{
    __shared__ double sd[kTeam][3][32];
    __shared__ float sf[kTeam][6][32];
    const int lane = threadIdx.x & 31, rank = threadIdx.x >> 5;
    const int Q = a.Q;
    const int64_t g = blockIdx.x;
    pdl_begin();
    const int64_t m = (g << 5) + lane;
    const int Wg = a.sw[g];
    const int64_t slot0 = g * 32LL * Q * 32 + lane;
    const int32_t* __restrict__ col = a.nbr + slot0;
    const double us = unit_scale(a.wmax);
    const float ts = pow2(a.x_grid - 33);

    Rec me;
    dwa::ld_rec(a.rec + 4 * m, me.a0, me.a1);
    dwa::ld_rec(a.rec + 4 * m + 2, me.b0, me.b1);
    const Own own = own_words(me);
    const D4 wm = ld_d4(a.w64 + 4 * m);
    float4 w0, w1;
    dwa::ld_rec(a.wdw + 2 * m, w0, w1);
    const Dw wd[3] = {{w0.x, w0.w}, {w0.y, w1.x}, {w0.z, w1.y}};
    const float bucket = w1.z;
    float2 rm = make_float2(1.0f, 0.0f);
    if (!UW) rm = __ldg(a.wrel + m);
    const double vm = UW ? 1.0 : (double)rm.x + (double)rm.y;

    double acc[3] = {0.0, 0.0, 0.0};
    Dw cor[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    // Software-pipelined as the forward walk: a bond's loads go out when the previous one's
    // words are consumed.
    struct In {
        Rec nb;
        D4 wj;
        float4 v0, v1;
        float4 il2;
        double e0, e1, e2;
        double gc;  // the sum of the steps before (FP64 handles load it where it is used: held
                    // from here, the registers run out, 507 instead of 451 us a step)
    } in;
    auto load = [&](int b, int64_t j) {
        const int64_t row = g * 32LL * Q + b;  // of 32 slots
        dwa::ld_rec(a.rec + 4 * j, in.nb.a0, in.nb.a1);
        dwa::ld_rec(a.rec + 4 * j + 2, in.nb.b0, in.nb.b1);
        dwa::ld_rec(a.wdw + 2 * j, in.v0, in.v1);
        if (F64) in.wj = ld_d4(a.w64 + 4 * j);
        in.il2 = __ldg(a.il + (row >> 1) * 32 + lane);
        if (F64) {
            const double* ep = a.e + row * 96 + lane;  // x, y, z rows
            in.e0 = __ldg(ep);
            in.e1 = __ldg(ep + 32);
            in.e2 = __ldg(ep + 64);
        }
        if (!F64) in.gc = a.gc[row * 32 + lane];
    };
    uint32_t word = 0u;
    int32_t jc = 0, jn = 0;
    if (rank < Wg) {
        jc = __ldg(col + rank * 32);
        if (rank + kTeam < Wg) jn = __ldg(col + (rank + kTeam) * 32);
        load(rank, jc);
        word = a.bits[g * Q * 32 + lane];
    }
    for (int b = rank; b < Wg; b += kTeam) {
        const bool alive = (word >> (b & 31)) & 1u;
        const int64_t j = jc, slot = slot0 + b * 32;
        const float2 il = b & 1 ? make_float2(in.il2.y, in.il2.w) : make_float2(in.il2.x, in.il2.z);
        const double old = in.gc;
        float2 rj = make_float2(1.0f, 0.0f);
        if (!UW) rj = __ldg(a.wrel + j);
        const Geo geo = bond_geo(own, in.nb, il, ts);
        const Dw wn[3] = {{in.v0.x, in.v0.w}, {in.v0.y, in.v1.x}, {in.v0.z, in.v1.y}};
        const bool same = in.v1.z == bucket;
        Dw d[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (UW) {
                d[k] = two_sum(wn[k].h, -wd[k].h);
                d[k].l += wn[k].l - wd[k].l;
            } else {
                const Dw p = dw_mul(Dw{rm.x, rm.y}, wn[k]), q = dw_mul(Dw{rj.x, rj.y}, wd[k]);
                d[k] = dw_add(p, Dw{-q.h, -q.l});
            }
        }
        // the undeformed part in FP64
        double e0 = 0.0, e1 = 0.0, e2 = 0.0, ed = 0.0;
        if (F64) {
            double d0, d1, d2;
            if (UW) {
                d0 = in.wj.x - wm.x;
                d1 = in.wj.y - wm.y;
                d2 = in.wj.z - wm.z;
            } else {
                const double vj = (double)rj.x + (double)rj.y;
                d0 = vm * in.wj.x - vj * wm.x;
                d1 = vm * in.wj.y - vj * wm.y;
                d2 = vm * in.wj.z - vj * wm.z;
            }
            e0 = in.e0;
            e1 = in.e1;
            e2 = in.e2;
            ed = fma(e0, d0, fma(e1, d1, e2 * d2));
        }
        if (b + kTeam < Wg) {
            load(b + kTeam, jn);
            jc = jn;
            if (((b + kTeam) & 31) < kTeam) word = a.bits[(g * Q + ((b + kTeam) >> 5)) * 32 + lane];
            if (b + 2 * kTeam < Wg) jn = __ldg(col + (b + 2 * kTeam) * 32);
        }
        Dw B{0.0f, 0.0f}, AB;
        if (F64) {
            B = dot3(geo.et, d);
            AB = dw_add(dot3(geo.xi, d), B);
        } else {
            AB = dot3(geo.y, d);
        }
        const float eta = fmaxf(fmaxf(fabsf(geo.et[0].h), fabsf(geo.et[1].h)), fabsf(geo.et[2].h));
        const bool ok = fabsf(geo.x) < a.x_max && (!F64 || eta * il.x < a.eta_max) && fabsf(AB.h) < 1e30f && same;
        if (!alive) continue;
        if (ok) {
            const Dw iL{il.x, il.y};
            const Dw zL = dw_mul(geo.z, iL);
            // q - 1 = z (3 + 3z + z^2); the low word of z, 2^-22 of it, enters z^2 too
            const float p = __fmul_rn(3.0f, geo.z.h), zz = __fmul_rn(geo.z.h, geo.z.h);
            const float s1 = __fadd_rn(3.0f, p), s2 = __fadd_rn(s1, zz);
            const Dw t3{s2, ((p - (s1 - 3.0f)) + (zz - (s2 - s1))) +
                                fmaf(fmaf(2.0f, geo.z.h, 3.0f), geo.z.l, fmaf(3.0f, geo.z.h, -p)) +
                                fmaf(geo.z.h, geo.z.h, -zz)};
            const Dw qAB = dw_mul(dw_mul(geo.z, t3), AB);
            Dw i3 = dw_mul(iL, dw_mul(iL, iL));
            Dw zc = zL;
            const Dw yw = dot3(geo.y, wd);
            Dw gs = dw_mul(zL, yw);  // -dL/dc of the bond in units of V_ref / unit_scale
            if (!UW) gs = dw_mul(gs, Dw{rj.x, rj.y});
            a.gc[slot] = (F64 ? a.gc[slot] : old) + (wide_of(-gs.h, bucket) + wide_of(-gs.l, bucket));
            if (a.cbond != nullptr) {  // per-bond stiffness (a uniform branch)
                const float2 cv = __ldg(a.cb + slot);
                i3 = dw_mul(i3, Dw{cv.x, cv.y});
                zc = dw_mul(zc, Dw{cv.x, cv.y});
                if (F64) ed *= __ldg(a.cbond + slot);
            }
            const Dw be = dw_mul(dw_add(AB, qAB), i3);
            Dw al{0.0f, 0.0f};
            if (F64) {
                acc[0] = fma(ed, e0, acc[0]);
                acc[1] = fma(ed, e1, acc[1]);
                acc[2] = fma(ed, e2, acc[2]);
                al = dw_mul(dw_add(B, qAB), i3);
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Dw zd = dw_mul(zc, d[k]);
                const Dw v = F64 ? dw_add(dw_mul(geo.xi[k], al), dw_mul(geo.et[k], be))
                                 : dw_mul(geo.y[k], be);
                const Dw f = dw_add(v, Dw{-zd.h, -zd.l});
                cor[k] = renorm(dw_add(cor[k], f));
            }
        } else {
            double f[3];
            a.gc[slot] = (F64 ? a.gc[slot] : old) + literal_adj(a, m, j, slot, f) * us;
            const double cij = a.cbond != nullptr ? __ldg(a.cbond + slot) : 1.0;
            acc[0] += cij * f[0];
            acc[1] += cij * f[1];
            acc[2] += cij * f[2];
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        sd[rank][k][lane] = acc[k];
        sf[rank][2 * k][lane] = cor[k].h;
        sf[rank][2 * k + 1][lane] = cor[k].l;
    }
    __syncthreads();
    if (rank == 0 && m < a.n) {
        const double w3[3] = {wm.x, wm.y, wm.z};
        double ub[3], vb[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            double s = 0.0;
            Dw c{0.f, 0.f};
            for (int r = 0; r < kTeam; ++r) {
                s += sd[r][k][lane];
                c = dw_add(c, Dw{sf[r][2 * k][lane], sf[r][2 * k + 1][lane]});
            }
            // (a node past the buckets has nothing in c)
            const double unit = bucket == bucket ? (a.scale / us) * bucket_down(bucket) : 0.0;
            s = fma(s, a.inv_c_ref, ((double)c.h + (double)c.l) * unit);
            ub[k] = a.ubm[3 * m + k] + (a.dt_rho * a.w_ref) * s;
            vb[k] = a.damp * w3[k];
            a.ub_out[3 * m + k] = ub[k];
            a.vb_out[3 * m + k] = vb[k];
        }
        const uint32_t cls = a.bcc[m];
        uint32_t mask = 0u;
        if (cls) {
            const BcClass& bc = a.bct[cls];
            mask = bc.mask;
            a.gl[m] += bc.force[0] * w3[0] + bc.force[1] * w3[1] + bc.force[2] * w3[2];
        }
        // the next reverse step's records: everything they need is this node's
        if (a.next_un != nullptr)
            adj_records(a, m, mask, ub, vb, a.next_un, a.next_dt, a.next_ws, us, me, a.next_rec,
                        a.next_w64, a.next_wdw);
    }
}

// FP64 pairs h + l (products through fused multiply-add, Knuth's two-sum)
struct Dd {
    double h, l;
};
__device__ __forceinline__ Dd dd_sum(double a, double b)
{
    const double s = a + b, bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ Dd dd_mul(Dd a, Dd b)
{
    const double p = a.h * b.h;
    return {p, fma(a.h, b.l, fma(a.l, b.h, fma(a.h, b.h, -p)))};
}

// e = xi / L^(3/2) of every slot, to rounding: t = L2^(-3/4) in FP64, corrected by one
// Newton step on t^4 L2^3 = 1 with the residual in FP64 pairs
__global__ void k_adj_e(const double* __restrict__ x64, const int32_t* __restrict__ nbr,
                        int64_t n_slices, int Q, double* __restrict__ e)
{
    const int64_t W = 32LL * Q;
    const int lane = threadIdx.x & 31;
    const int64_t rows = n_slices * W;
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < rows;
         r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int64_t p = (r / W) * 32 + lane, j = nbr[r * 32 + lane];
        double out[3] = {0.0, 0.0, 0.0};
        if (j != p) {
            double xi[3];
            Dd L2{0.0, 0.0};
            for (int k = 0; k < 3; ++k) {
                xi[k] = x64[8 * j + k] - x64[8 * p + k];
                const double q = xi[k] * xi[k];
                const Dd s = dd_sum(L2.h, q);
                L2 = Dd{s.h, L2.l + s.l + fma(xi[k], xi[k], -q)};
            }
            const double i1 = 1.0 / sqrt(L2.h), t = i1 * sqrt(i1);
            const Dd tt = dd_mul(Dd{t, 0.0}, Dd{t, 0.0});
            const Dd P = dd_mul(dd_mul(tt, tt), dd_mul(L2, dd_mul(L2, L2)));
            const double tl = 0.25 * t * ((1.0 - P.h) - P.l);
            for (int k = 0; k < 3; ++k) {
                const double h = xi[k] * t;
                out[k] = h + fma(xi[k], tl, fma(xi[k], t, -h));
            }
        }
        for (int k = 0; k < 3; ++k) e[(r * 3 + k) * 32 + lane] = out[k];
    }
}

// the per-slot sums times scale / unit_scale
__global__ void k_adj_merge_w3(double* gc, int64_t count, double scale,
                               const unsigned long long* __restrict__ wmax)
{
    const double s = scale / unit_scale(wmax);
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count;
         e += (int64_t)gridDim.x * blockDim.x)
        gc[e] *= s;
}

}  // namespace

cudaError_t launch_adj_scale_w3(const double* ub, const double* vb, int64_t n3, double dt,
                                unsigned long long* wmax, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(wmax, 0, 8, s);
    if (e != cudaSuccess) return e;
    k_adj_scale<<<grid_of(n3), 256, 0, s>>>(ub, vb, n3, dt, wmax);
    return cudaGetLastError();
}

cudaError_t launch_adj_e(const double* x64, const int32_t* nbr, int64_t n_slices, int Q, double* e,
                         cudaStream_t s)
{
    k_adj_e<<<grid_of(n_slices * 32 * Q * 32), 256, 0, s>>>(x64, nbr, n_slices, Q, e);
    return cudaGetLastError();
}

cudaError_t launch_adj_prep_w3(const AdjW3Args& a, double dt, double ws, int64_t n_pad,
                               cudaStream_t s)
{
    k_adj_prep_w3<<<grid_of(n_pad), 256, 0, s>>>(a, dt, ws, n_pad);
    return cudaGetLastError();
}

cudaError_t launch_adj_step_w3(const AdjW3Args& a, cudaStream_t s)
{
    const void* fn = a.e != nullptr
                         ? a.uniform_w ? (const void*)k_adj_step_w3<true, true>
                                       : (const void*)k_adj_step_w3<false, true>
                     : a.uniform_w ? (const void*)k_adj_step_w3<true, false>
                                   : (const void*)k_adj_step_w3<false, false>;
    void* args[] = {const_cast<AdjW3Args*>(&a)};
    return launch_pdl(fn, dim3((unsigned)((a.n + 31) / 32)), dim3(32 * kTeam), args, 0, s);
}

cudaError_t launch_adj_merge_w3(double* gc, int64_t count, double scale,
                                const unsigned long long* wmax, cudaStream_t s)
{
    k_adj_merge_w3<<<grid_of(count), 256, 0, s>>>(gc, count, scale, wmax);
    return cudaGetLastError();
}

}  // namespace pd
