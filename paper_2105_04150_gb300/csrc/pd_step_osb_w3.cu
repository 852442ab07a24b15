// Ordinary state-based peridynamics (linear peridynamic solid, constant influence
// function) on FP64 and double-word handles (sm_103a): the two loops per step of the
// paper's "State-based Peridynamics" section as two lane-per-node kernels over the
// sliced family layout of the bond-based step.
//
//   k_osb_w3_dilation  per node: bonds past s_c break (Eq. 6, s = e / |xi|), then
//                      theta_i = (3 / m_i) sum_j mu_ij |xi| e_ij V_j, e = |y| - |xi|
//   k_osb_w3_force     per node: F_i = sum_j mu_ij (t_ij + t_ji) V_j y / |y| with
//                      t_ij = alpha_i |xi| + beta_i e, beta_i = 15 G / m_i,
//                      alpha_i = 3 K theta_i / m_i - beta_i theta_i / 3; then the
//                      update, boundary conditions and damage of the bond-based step
//
// m_i = sum_j |xi|^2 V_j over the family after the initial cuts, computed once.
// Formed literally in FP64 (57 operations a bond in both loops) the step is bound by the
// FP64 pipe, 14.7 ms on the 1M-node notched beam.  The bonds are evaluated as in
// pd_step_f64.cu instead, from exact differences of three-word records in double-word
// arithmetic, with z = |xi| / |y| - 1 and num = |y|^2 - |xi|^2:
//   |xi| e = num (1 + z) / (2 + z) = (num + num w) / 2,  w = z / (2 + z),
//   t |y|^-1 = (alpha_i + alpha_j) + (gamma_i + gamma_j) z,  gamma = alpha - beta,
// so neither loop needs |xi|, a root or a division of its own.  alpha and gamma are
// published per node as double-words in units of (K + G) / (V_ref U^2).  Bonds past
// kW3XMaxOsb or turned past kW3EtaMax (on PD_PREC_DW handles: past kW3XWide), and in the
// dilation loop those in or above the band below the smallest s_c, are evaluated (and
// decided) literally in FP64 after their flag word.
#include <algorithm>

#include <cuda_runtime.h>

#include "pd_internal.h"
#include "pd_w3.h"
#include "pd_w3_node.h"

namespace pd {
namespace {

using namespace w3;

// A bond literally in FP64, from the slot's 1 / |xi|: |xi| e is s |xi|^2, so no root is
// taken.  Bound by the FP64 pipe: 220k nodes at 2 % strain, where every bond is literal,
// take 3214 us a step (4285 with roots; 3255 fully literal with |xi| stored per slot).  The
// lane's own record is read again for every bond: a function that holds it costs the walk,
// whose registers are all taken, 90 bytes of spills, and a step at rest 546 instead of 475 us.
struct OsbBond {
    double y[3], x2, r, ir, s;
};
__device__ __forceinline__ OsbBond osb_bond(const double* __restrict__ rin, int64_t i, int64_t j,
                                            double iL)
{
    OsbBond b;
    double q = 0.0;
    b.x2 = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double xi = __ldg(rin + 8 * j + c) - __ldg(rin + 8 * i + c);
        b.y[c] = xi + (__ldg(rin + 8 * j + 4 + c) - __ldg(rin + 8 * i + 4 + c));
        b.x2 += xi * xi;
        q += b.y[c] * b.y[c];
    }
    b.ir = rsqrt_nr_int(q);
    b.r = q * b.ir;
    b.s = fma(b.r, iL, -1.0);
    return b;
}

__device__ __forceinline__ double bond_sc(const StepArgsF64& a, int64_t i, int64_t j)
{
    if (a.inst != nullptr) {  // batch: the instance's parameters, instance-local ids as keys
        const InstParams& ip = a.itab[a.inst[i]];
        return ip.sc_mode == 1 ? sc_draw(ip.sc_seed, ip.sc_lo, ip.sc_hi, a.hid[i], a.hid[j]) : ip.sc;
    }
    return a.sc_mode == 1 ? sc_draw(a.sc_seed, a.sc_lo, a.sc_hi, a.gid[i], a.gid[j]) : a.sc;
}

// High word of a stretch below which no bond of the node breaks, with room for rounding.
__device__ __forceinline__ int near_hi(const StepArgsF64& a, int64_t i)
{
    return __double2hiint(a.inst != nullptr ? a.itab[a.inst[i]].sc_lo : a.sc_lo) - 2;
}

// e / |xi| >= s_c.  s is within a few 2^-53 of e / |xi|, so their high words (2^-20 of
// either) decide, without a root, unless they meet or s_c is below 1e-8; not a number: no.
__device__ __forceinline__ bool past_sc(const StepArgsF64& a, int64_t i, int64_t j, const OsbBond& b,
                                        double iL)
{
    const double sc = bond_sc(a, i, j);
    const int hs = __double2hiint(b.s), hc = __double2hiint(sc);
    if (abs(hs - hc) > 1 && hc > 0x3e500000 && hs <= 0x7ff00000) return hs > hc;
    return (b.r - sqrt(b.x2)) * iL >= sc;
}

__global__ void k_osb_w3_volume(const StepArgsF64 a, const OsbW3Args o,
                                const double* __restrict__ x64)
{
    const int64_t W = 32LL * a.Q;
    const int64_t total = ((a.n + 31) >> 5) << 5;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < total;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = p >> 5;
        const int lane = (int)(p & 31);
        double acc = 0.0;
        for (int m = 0; m < a.sw[g]; ++m) {
            if (!((a.bits[(g * a.Q + (m >> 5)) * 32 + lane] >> (m & 31)) & 1u)) continue;
            const int64_t j = a.nbr[(g * W + m) * 32 + lane];
            double q = 0.0;
            for (int c = 0; c < 3; ++c) {
                const double e = x64[3 * j + c] - x64[3 * p + c];
                q += e * e;
            }
            acc += q * o.vol[j];
        }
        o.mvol[p] = acc;
    }
}

// The slots of one slice, two at a time, the next chunk's loads in flight while the
// current one is evaluated (as in pd_step_f64.cu).  `geo` forms a bond's geometry (kin or
// kin_num); `bond` gets the two bonds' neighbours,
// geometry, U / |xi| and flags, and returns which of the live ones are to be evaluated
// literally; `word_end(q, word, pend)` is called after each flag word.
template <class Geo, class Bond, class WordEnd>
__device__ __forceinline__ void osb_walk(const StepArgsF64& a, const W3Args& d, int cur,
                                         const Own2& own, float ts, int64_t g, int Wg, Geo geo, Bond bond,
                                         WordEnd word_end)
{
    const int lane = threadIdx.x & 31;
    const int Q = a.Q;
    const float4* __restrict__ R = d.rec[cur];
    const int32_t* __restrict__ col = a.nbr + g * 32LL * Q * 32 + lane;
    const float4* __restrict__ ilp = d.il + g * 16LL * Q * 32 + lane;
    const uint32_t* const bw = a.bits + g * Q * 32 + lane;
    if (Wg <= 0) return;
    int32_t j0 = __ldg(col), j1 = __ldg(col + 32);
    int32_t n0 = 0, n1 = 0;
    if (2 < Wg) {
        n0 = __ldg(col + 64);
        n1 = __ldg(col + 96);
    }
    Rec A, B;
    dwa::ld_rec(R + 4 * (int64_t)j0, A.a0, A.a1);
    dwa::ld_rec(R + 4 * (int64_t)j0 + 2, A.b0, A.b1);
    dwa::ld_rec(R + 4 * (int64_t)j1, B.a0, B.a1);
    dwa::ld_rec(R + 4 * (int64_t)j1 + 2, B.b0, B.b1);
    float4 il = __ldg(ilp);
    uint32_t word = 0u, pend = 0u;
    for (int m = 0; m < Wg; m += 2) {
        const bool more = m + 2 < Wg;
        const int b = m & 31;
        if (b == 0) {
            word = bw[(m >> 5) * 32];
            pend = 0u;
        }
        const auto kA = geo(own, A, both(ts), make_float2(ts, 1.0f));
        if (more) {
            dwa::ld_rec(R + 4 * (int64_t)n0, A.a0, A.a1);
            dwa::ld_rec(R + 4 * (int64_t)n0 + 2, A.b0, A.b1);
        }
        const auto kB = geo(own, B, both(ts), make_float2(ts, 1.0f));
        const float4 ilc = il;
        const int32_t c0 = j0, c1 = j1;
        if (more) {
            dwa::ld_rec(R + 4 * (int64_t)n1, B.a0, B.a1);
            dwa::ld_rec(R + 4 * (int64_t)n1 + 2, B.b0, B.b1);
            il = __ldg(ilp + (m + 2) * 16);
            j0 = n0;
            j1 = n1;
            if (m + 4 < Wg) {
                n0 = __ldg(col + (m + 4) * 32);
                n1 = __ldg(col + (m + 5) * 32);
            }
        }
        pend |= bond(c0, c1, kA, kB, ilc, (word >> b) & 3u) << b;
        if (b == 30 || !more) word_end(m >> 5, word, pend);
    }
}

// x and w = z / (2 + z) of two bonds: seeded as -x / (1 + r)^2, r = sqrt(1 + x), and
// corrected by one Newton step on f(w) = x (1 + w)^2 + 4 w = 0, f' = 4 r, whose leading
// terms cancel exactly for |x| <= 1/2.
__device__ __forceinline__ Stretch2 w_of(Dw2 num, const float4 il)
{
    const Dw2 iL{make_float2(il.x, il.y), make_float2(il.z, il.w)};
    const Dw2 x = dw_mul2(dw_mul2(num, iL), iL);
    const float2 x1 = add2(both(1.0f), x.h);
    const float2 ir = make_float2(dwa::rsqrt_seed(x1.x), dwa::rsqrt_seed(x1.y));
    const float2 r1 = fma2(x1, ir, both(1.0f));
    const float2 den = mul2(r1, r1), nx = mul2(x.h, both(-1.0f));
    const float2 w0 = mul2(nx, make_float2(dwa::rcp_seed(den.x), dwa::rcp_seed(den.y)));
    const float2 ww = mul2(w0, w0), ph = fma2(both(2.0f), w0, ww);
    const float2 e = make_float2(fmaf(w0.x, w0.x, -ww.x), fmaf(w0.y, w0.y, -ww.y));
    const Dw2 p{ph, add2(sub2(ww, fma2(both(-2.0f), w0, ph)), e)};
    const Dw2 xp = dw_mul2(x, p);
    const float2 R = add2(add2(fma2(both(4.0f), w0, x.h), xp.h), add2(x.l, xp.l));
    return {add2(x.h, x.l) /* see stretch2 */, Dw2{w0, mul2(R, mul2(ir, both(-0.25f)))}};
}

// literal_of with the turned bonds of FP64 handles (here the infinite x of pd_step_f64.cu
// is the slower form: 494 against 473 us a step of 220k nodes)
template <bool WIDE>
__device__ __forceinline__ uint32_t literal_or_turned(float2 x, float eA, float eB, const float4 il,
                                                      float x_hi, const W3Args& d, uint32_t live)
{
    uint32_t lit = literal_of(x, x_hi, d.x_max, live);
    if (!WIDE) {
        const float2 t = mul2(make_float2(eA, eB), make_float2(il.x, il.y));
        lit |= ((t.x < d.eta_max ? 0u : 1u) | (t.y < d.eta_max ? 0u : 2u)) & live;
    }
    return lit;
}

// The unit, grid and weight of the slice's node (batches: its instance's)
struct Unit {
    double w_ref, scale;
    float x_hi, ts;
};
__device__ __forceinline__ Unit unit_of(const StepArgsF64& a, const W3Args& d, int64_t i)
{
    Unit u{d.w_ref, d.scale, d.x_hi, pow2(d.x_grid - 33)};
    if (a.inst != nullptr) {
        const InstParams& ip = a.itab[a.inst[i]];
        u.w_ref = ip.w_ref;
        u.scale = ip.w3_scale;
        u.x_hi = a.frozen ? d.x_hi : ip.w3_x_hi;
        u.ts = pow2(ip.w3_x_grid - 33);
    }
    return u;
}

// The bonds `pend` of a flag word literally: breaks (cleared from the word in memory),
// and |xi| e V_j of the others
__device__ __noinline__ double literal_dilation(const StepArgsF64& a, const OsbW3Args& o, int cur,
                                                int64_t i, const int32_t* col, uint32_t pend,
                                                uint32_t* bw)
{
    double sum = 0.0;
    uint32_t gone = 0u;
    for (; pend; pend &= pend - 1u) {
        const int b = __ffs(pend) - 1;
        const int64_t j = col[b * 32];
        const double iL = __ldg(a.ilen + (col - a.nbr) + b * 32);
        const OsbBond bd = osb_bond(a.rec[cur], i, j, iL);
        bool brk = !a.frozen && __double2hiint(bd.s) >= near_hi(a, i) && past_sc(a, i, j, bd, iL);
        if (brk && a.has_nofail) brk = ((a.bct[a.bcc[i]].mask | a.bct[a.bcc[j]].mask) & 8u) == 0u;
        if (brk)
            gone |= 1u << b;
        else
            sum += bd.s * bd.x2 * o.vol[j];
    }
    if (gone) *bw &= ~gone;
    return sum;
}

template <bool UW, bool WIDE>
__global__ void __launch_bounds__(256, 2)
    k_osb_w3_dilation(const __grid_constant__ StepArgsF64 a, const __grid_constant__ W3Args d,
                      const __grid_constant__ OsbW3Args o)
{
    const int lane = threadIdx.x & 31;
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    pdl_begin();
    const int64_t step = a.step_ctr[0] + a.k;
    const int cur = (int)(step & 1);
    const float4* __restrict__ R = d.rec[cur];
    const int64_t nslices = (a.n + 31) >> 5;
    for (int64_t g = wid; g < nslices; g += nwarps) {
        const int64_t i = (g << 5) + lane;
        Rec me;
        dwa::ld_rec(R + 4 * i, me.a0, me.a1);
        dwa::ld_rec(R + 4 * i + 2, me.b0, me.b1);
        const Unit un = unit_of(a, d, i);
        const int32_t* col = a.nbr + g * 32LL * a.Q * 32 + lane;
        // sums of |xi| e V_j / V_ref over the even and the odd slots, in units of U^2
        Dw2 acc{both(0.0f), both(0.0f)};
        double lit = 0.0;
        osb_walk(
            a, d, cur, own_pairs(me), un.ts, g, a.sw[g], kin_num,
            [&](int32_t c0, int32_t c1, const KinNum& A, const KinNum& B, const float4 il, uint32_t live) {
                const Dw2 num{make_float2(A.num.h, B.num.h), make_float2(A.num.l, B.num.l)};
                const Stretch2 t = w_of(num, il);
                const uint32_t pend = literal_or_turned<WIDE>(t.x, A.e, B.e, il, un.x_hi, d, live);
                const Dw2 hn{mul2(num.h, both(0.5f)), mul2(num.l, both(0.5f))};
                Dw2 e = dw_add2(hn, dw_mul2(hn, t.z));
                if (!UW) {
                    const float2 wA = __ldg(d.wrel + c0), wB = __ldg(d.wrel + c1);
                    e = dw_mul2(e, Dw2{make_float2(wA.x, wB.x), make_float2(wA.y, wB.y)});
                }
                const uint32_t ok = live & ~pend;
                const bool kA = ok & 1u, kB = ok & 2u;
                acc = dw_add2(acc, Dw2{make_float2(kA ? e.h.x : 0.0f, kB ? e.h.y : 0.0f),
                                       make_float2(kA ? e.l.x : 0.0f, kB ? e.l.y : 0.0f)});
                return pend;
            },
            [&](int q, uint32_t, uint32_t pend) {
                if (pend)
                    lit += literal_dilation(a, o, cur, i, col + (int64_t)q * 32 * 32, pend,
                                            a.bits + (g * a.Q + q) * 32 + lane);
            });
        if (i >= a.n) continue;
        const double u2 = un.w_ref / (un.scale * un.scale);  // V_ref U^2
        const double m = o.mvol[i];
        double th = 0.0, al = 0.0, be = 0.0;
        if (m > 0.0) {
            const double s = ((double)acc.h.x + (double)acc.l.x) + ((double)acc.h.y + (double)acc.l.y);
            th = 3.0 * fma(s, u2, lit) / m;
            be = 15.0 * o.G / m;
            al = 3.0 * o.K * th / m - be * th / 3.0;
        }
        o.ab64[i] = make_double2(al, be);
        const double sg = u2 / (o.K + o.G);
        const double as = al * sg, gs = (al - be) * sg;
        const float ah = (float)as, gh = (float)gs;
        o.ab[i] = make_float4(ah, (float)(as - (double)ah), gh, (float)(gs - (double)gh));
    }
}

// The bonds `pend` of a flag word literally: their force into f
__device__ __noinline__ void literal_force(const StepArgsF64& a, const OsbW3Args& o, int cur,
                                           int64_t i, const int32_t* col, uint32_t pend, double* f)
{
    const double2 abi = o.ab64[i];
    for (; pend; pend &= pend - 1u) {
        const int b = __ffs(pend) - 1;
        const int64_t j = col[b * 32];
        const double iL = __ldg(a.ilen + (col - a.nbr) + b * 32);
        const OsbBond bd = osb_bond(a.rec[cur], i, j, iL);
        const double2 abj = o.ab64[j];
        // (t_ij + t_ji) / |xi|
        const double t = fma(abi.y + abj.y, bd.s, abi.x + abj.x);
        const double c = t * (bd.x2 * iL) * o.vol[j] * bd.ir;
        for (int k = 0; k < 3; ++k) f[k] += c * bd.y[k];
    }
}

template <bool UW, bool WIDE>
__global__ void __launch_bounds__(256, 2)
    k_osb_w3_force(const __grid_constant__ StepArgsF64 a, const __grid_constant__ W3Args d,
                   const __grid_constant__ OsbW3Args o)
{
    const int lane = threadIdx.x & 31;
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    pdl_begin();
    const int64_t step = a.step_ctr[0] + a.k;
    const int cur = (int)(step & 1);
    const float4* __restrict__ R = d.rec[cur];
    const int64_t nslices = (a.n + 31) >> 5;
    for (int64_t g = wid; g < nslices; g += nwarps) {
        const int64_t i = (g << 5) + lane;
        Rec me;  // (read again for the epilogue: the walk's registers are all taken)
        dwa::ld_rec(R + 4 * i, me.a0, me.a1);
        dwa::ld_rec(R + 4 * i + 2, me.b0, me.b1);
        const float ts = unit_of(a, d, i).ts;
        const float4 own_ab = o.ab[i];
        const int32_t* col = a.nbr + g * 32LL * a.Q * 32 + lane;
        Force F{Dw2{both(0.0f), both(0.0f)}, Dw{0.0f, 0.0f}};
        double lit[3] = {0.0, 0.0, 0.0};
        int alive = 0;
        osb_walk(
            a, d, cur, own_pairs(me), ts, g, a.sw[g], kin,
            [&](int32_t c0, int32_t c1, const Kin& A, const Kin& B, const float4 il,
                uint32_t live) {
                // (behind the geometry: the stretch hides most of their latency)
                const float4 p0 = __ldg(o.ab + c0), p1 = __ldg(o.ab + c1);
                const Stretch2 t = stretch2(
                    Dw2{make_float2(A.num.h, B.num.h), make_float2(A.num.l, B.num.l)}, il);
                const uint32_t pend = literal_or_turned<WIDE>(t.x, A.e, B.e, il, d.x_max, d, live);
                const Dw2 al = dw_add2(Dw2{both(own_ab.x), both(own_ab.y)},
                                       Dw2{make_float2(p0.x, p1.x), make_float2(p0.y, p1.y)});
                const Dw2 ga = dw_add2(Dw2{both(own_ab.z), both(own_ab.w)},
                                       Dw2{make_float2(p0.z, p1.z), make_float2(p0.w, p1.w)});
                Dw2 c = dw_add2(al, dw_mul2(ga, t.z));
                if (!UW) {
                    const float2 wA = __ldg(d.wrel + c0), wB = __ldg(d.wrel + c1);
                    c = dw_mul2(c, Dw2{make_float2(wA.x, wB.x), make_float2(wA.y, wB.y)});
                }
                const uint32_t ok = live & ~pend;
                add_force(F, c.h.x, c.l.x, A, ok & 1u);
                add_force(F, c.h.y, c.l.y, B, ok & 2u);
                F.xy = renorm2(F.xy);  // (472 -> 475 us; a third of the error at 0.6 %)
                F.z = renorm(F.z);
                return pend;
            },
            [&](int q, uint32_t word, uint32_t pend) {
                alive += __popc(word);
                if (pend) literal_force(a, o, cur, i, col + (int64_t)q * 32 * 32, pend, lit);
            });
        if (i >= a.n) continue;
        const Node nd = load_node(a, d, cur, i);
        dwa::ld_rec(R + 4 * i, me.a0, me.a1);
        dwa::ld_rec(R + 4 * i + 2, me.b0, me.b1);
        const Unit un = unit_of(a, d, i);
        const double fs = (o.K + o.G) * un.scale;
        const Dw Fk[3] = {{F.xy.h.x, F.xy.l.x}, {F.xy.h.y, F.xy.l.y}, F.z};
        double T[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) T[k] = fma((double)Fk[k].h + (double)Fk[k].l, fs, lit[k]);
        finish_node(a, d, cur, step, me, nd, un.scale, i, T, alive);
    }
}

}  // namespace

cudaError_t launch_osb_w3_setup(const StepArgsF64& a, const OsbW3Args& o, const double* x64,
                                cudaStream_t s)
{
    const int64_t b = ((((a.n + 31) >> 5) << 5) + 255) / 256;
    k_osb_w3_volume<<<(int)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 16)), 256, 0, s>>>(a, o, x64);
    return cudaGetLastError();
}

cudaError_t launch_osb_w3_step(const StepArgsF64& a, const W3Args& d, const OsbW3Args& o, int grid,
                               int block, cudaStream_t s)
{
    void* args[] = {const_cast<StepArgsF64*>(&a), const_cast<W3Args*>(&d), const_cast<OsbW3Args*>(&o)};
    static const void* const dil_k[4] = {
        (const void*)k_osb_w3_dilation<false, false>, (const void*)k_osb_w3_dilation<true, false>,
        (const void*)k_osb_w3_dilation<false, true>, (const void*)k_osb_w3_dilation<true, true>};
    const void* dil = dil_k[(d.wide ? 2 : 0) + (d.uniform_w ? 1 : 0)];
    const cudaError_t e = launch_pdl(dil, dim3(grid), dim3(block), args, 0, s);
    return e != cudaSuccess
               ? e
               : launch_pdl(osb_w3_force_kernel(d.uniform_w != 0, d.wide != 0), dim3(grid), dim3(block), args, 0, s);
}

const void* osb_w3_force_kernel(bool uniform_w, bool wide)
{
    static const void* const k[4] = {
        (const void*)k_osb_w3_force<false, false>, (const void*)k_osb_w3_force<true, false>,
        (const void*)k_osb_w3_force<false, true>, (const void*)k_osb_w3_force<true, true>};
    return k[(wide ? 2 : 0) + (uniform_w ? 1 : 0)];
}

}  // namespace pd
