// What the bond-based and the state-based steps on three-word records share (device
// code only): the hashed critical stretch, the force sum, and the end of a node's step.
#pragma once

#include <cuda_runtime.h>

#include "pd_internal.h"
#include "pd_w3.h"

namespace pd {
namespace w3 {

__device__ __forceinline__ uint64_t splitmix_out(uint64_t seed, uint64_t m)
{
    uint64_t z = seed + m * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ double sc_draw(uint64_t seed, double lo, double hi, int32_t gi,
                                          int32_t gj)
{
    const uint64_t a = (uint64_t)(uint32_t)min(gi, gj);
    const uint64_t b = (uint64_t)(uint32_t)max(gi, gj);
    const uint64_t h = splitmix_out(seed, ((a << 32) | b) + 1ull);
    return lo + (hi - lo) * ((double)(h >> 11) * 0x1.0p-53);
}

__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// The lane's force sum: (x, y) and z.
struct Force {
    Dw2 xy;
    Dw z;
};

// F += c y when `ok` (a select: whatever a masked slot computed, including a
// non-finite value, is dropped)
__device__ __forceinline__ void add_force(Force& F, float ch, float cl, const Kin& b, bool ok)
{
    ch = ok ? ch : 0.0f;
    cl = ok ? cl : 0.0f;
    const Dw2 f = dw_mul2(Dw2{both(ch), both(cl)}, b.y);
    const Dw fz = dw_mul(Dw{ch, cl}, b.yz);
    const Dw2 t = two_sum2(F.xy.h, f.h);
    F.xy = Dw2{t.h, add2(F.xy.l, add2(t.l, f.l))};
    const Dw tz = two_sum(F.z.h, fz.h);
    F.z = Dw{tz.h, F.z.l + (tz.l + fz.l)};
}

// What the end of a node's step reads, loaded before the team's barrier.
struct Node {
    double2 u01, u2_;
    double v[3];
    double phi0;
    uint32_t cls;
    int fam;  // bonds of the intact family
};
__device__ __forceinline__ Node load_node(const StepArgsF64& a, const W3Args& d, int cur, int64_t i)
{
    const double2* __restrict__ rin = reinterpret_cast<const double2*>(a.rec[cur]);
    Node n;
    n.u01 = __ldg(rin + 4 * i + 2);
    n.u2_ = __ldg(rin + 4 * i + 3);
#pragma unroll
    for (int c = 0; c < 3; ++c) n.v[c] = a.v[3 * i + c];
    n.phi0 = __ldg(d.phi0 + i);
    n.cls = a.bcc[i];
    n.fam = __ldg(d.fam + i);
    return n;
}

// Integration of the lane's node (damped Euler-Cromer, Eq. 11, or damped
// velocity-Verlet), BCs, damage, and the records its neighbours read next.
__device__ __forceinline__ void finish_node(const StepArgsF64& a, const W3Args& d, int cur,
                                            int64_t step, const Rec& me, const Node& nd,
                                            double scale, int64_t i, const double (&T)[3], int alive)
{
    double2* __restrict__ rout = reinterpret_cast<double2*>(const_cast<double*>(a.rec[cur ^ 1]));
    float4* __restrict__ Rout = const_cast<float4*>(d.rec[cur ^ 1]);
    const bool first = a.vv && step == a.step_ctr[1];  // velocity-Verlet: a^n formed afresh
    uint32_t mask = 0u;
    double gdisp[3] = {0.0, 0.0, 0.0};
    double F[3] = {T[0], T[1], T[2]};
    if (nd.cls != 0u) {
        const BcClass& bc = a.bct[nd.cls];
        mask = bc.mask;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            gdisp[c] = bc.disp[c];
            F[c] += a.load * bc.force[c];
        }
    }
    const double uo[3] = {nd.u01.x, nd.u01.y, nd.u2_.x};
    double un[3];
    float uh[3], um[3], tw[3];
    const float tin[3] = {me.a1.z, me.a1.w, me.b1.z};
    bool finite = true;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        // stored velocity: v^n (Euler-Cromer) or, for velocity-Verlet, the
        // half-step velocity v^{n-1} + dt/2 a^{n-1} (v^n right after a set state)
        const double vi = nd.v[c];
        const double adt = (F[c] - a.eta * vi) * d.dt_rho;  // dt a
        double vn, vfull;
        if (a.vv) {
            vfull = first ? vi : fma(0.5, adt, vi);
            vn = fma(0.5, adt, vfull);
        } else {
            vn = vi + adt;
            vfull = vn;
        }
        double u = fma(a.dt, vn, uo[c]);
        if (mask & (1u << c)) {
            const double2 uv = bc_controlled(a.disp_rate, a.ramp_steps, a.dt, gdisp[c], step);
            u = uv.x;
            vn = uv.y;
            vfull = vi;
        }
        finite = finite && isfinite(u);
        un[c] = u;
        if (a.peek)
            a.vout[3 * i + c] = vfull;
        else
            a.v[3 * i + c] = vn;
        float ut;
        split3(u * scale, kW3UGrid, uh[c], um[c], ut);
        tw[c] = pack_t(__float_as_uint(tin[c]) & 0x7ffu, ut);
    }
    if (a.peek) return;
    rout[4 * i + 2] = make_double2(un[0], un[1]);  // (positions and weights: in both buffers)
    rout[4 * i + 3] = make_double2(un[2], 0.0);
    if (a.uout != nullptr)  // the adjoint's recomputed segment
        for (int c = 0; c < 3; ++c) a.uout[3 * i + c] = un[c];
    dwa::st_rec(Rout + 4 * i, make_float4(me.a0.x, me.a0.y, uh[0], uh[1]),
                make_float4(me.a1.x, uh[2], tw[0], tw[1]));
    dwa::st_rec(Rout + 4 * i + 2, make_float4(me.b0.x, me.b0.y, um[0], um[1]),
                make_float4(me.b1.x, um[2], tw[2], 0.0f));
    double phi = nd.phi0;
    if (alive != nd.fam)
        phi = d.uniform_w != 0
                  ? damage_ratio(nd.fam, alive)
                  : damage_lost(false, a.rec[cur], a.nbr, a.bits, a.bits0, a.wsum_inv[i], nd.phi0,
                                i >> 5, (int)(i & 31), a.Q);
    a.damage[i] = phi;
    if (!finite) atomicOr(a.err, PD_DEVERR_NONFINITE);
}

}  // namespace w3
}  // namespace pd
