// Fused FP64 peridynamic step kernel for sm_103a (the parity path).
//
// Same decomposition as the other step kernels (lane per node over the sliced
// family layout, double-buffered displacement, bond flags as the lane's own bit
// words, integration and damage in the same pass).  Node state and integration
// are FP64.  GB300 issues one FP64 operation in the time of 64 FP32 ones, so a
// kernel that forms Eq. 4 literally in FP64 (about 41 FP64 operations a bond) is
// bound by that pipe: 1.88 ms per step of a 180x35x35 notched beam, and 0.29 ms of a
// 4000-node bar, whose 125 warps each walk a whole family alone.  With the arithmetic
// and the split below they take 0.25 and 0.0125 ms, 202 warp instructions a bond (277
// without the paired instructions, 0.285 ms), 59 % of the issue slots with the FMA
// pipe occupied twice by each pair and 16 warps per SM (128 registers).
// Here the FP64 differences x_j - x_i and u_j - u_i come exactly from three-word
// FP32 records, and the stretch without cancellation in double-word arithmetic
// (pd_w3.h): no FP64 operation on the bonds of the bulk.  The literal form rounds
// s = |y| / |xi| - 1 at an absolute 3e-16, 3e-12 of the force at a stretch of
// 1e-4; this one has a relative error of about 1e-14 of the force, so it is the more
// accurate of the two up to stretches of about 0.5 % (velocities of the beam after 5
// steps: 6e-13 relative to the exact step instead of 1.2e-11).  The other bonds are decided and
// evaluated literally in FP64 after their segment (literal_bond): those past kW3XMax,
// turned past kW3EtaMax or far shorter than U (a body all of whose bonds are takes 1.63
// ms, 1.71 in the kernel it replaced; on PD_PREC_DW handles, WIDE, only those past kW3XWide
// are) and those in or above the band below the smallest s_c, so that every break is an
// FP64 decision on Eq. 4.  Models with softening take the literal kernel of
// pd_step_f64_soft.cu for every bond.
//
// Work split: a family is walked in segments of 16 slots whose force sums are
// added up in segment order, so the result does not depend on which warp walks
// which segment.  A model with few slices gives each slice to a team of warps
// (TEAM), which take its segments in turn and add their sums through shared memory.
#include <algorithm>

#include <cuda_runtime.h>

#include "pd_internal.h"
#include "pd_w3.h"
#include "pd_w3_node.h"

namespace pd {
namespace {

using namespace w3;

constexpr int kSeg = kW3Seg;  // slots per segment

// One bond literally in FP64: s = |y| / |xi| - 1 (1/|xi| stored per slot, 1/|y| from
// the Newton-refined reciprocal square root), the break test against the bond's s_c,
// the no-fail rule, and the force, added to f.  True when it breaks.
__device__ __forceinline__ bool literal_bond(const StepArgsF64& a, int cur, int64_t i, int64_t j,
                                          int64_t slot, double* f)
{
    const double2* __restrict__ rin = reinterpret_cast<const double2*>(a.rec[cur]);
    const double2 x01 = __ldg(rin + 4 * i), x2w = __ldg(rin + 4 * i + 1);
    const double2 u01 = __ldg(rin + 4 * i + 2), u2_ = __ldg(rin + 4 * i + 3);
    const double2 X01 = __ldg(rin + 4 * j), X2w = __ldg(rin + 4 * j + 1);
    const double2 U01 = __ldg(rin + 4 * j + 2), U2_ = __ldg(rin + 4 * j + 3);
    const double yx = (X01.x - x01.x) + (U01.x - u01.x);
    const double yy = (X01.y - x01.y) + (U01.y - u01.y);
    const double yz = (X2w.x - x2w.x) + (U2_.x - u2_.x);
    const double y2 = yx * yx + yy * yy + yz * yz;
    const double ir = rsqrt_nr(y2);
    const double s = fma(y2 * ir, __ldg(a.ilen + slot), -1.0);
    double sc = a.sc;
    if (a.inst != nullptr) {  // batch: instance parameters, local ids as keys
        const InstParams& ip = a.itab[a.inst[i]];
        sc = ip.sc_mode == 1 ? sc_draw(ip.sc_seed, ip.sc_lo, ip.sc_hi, a.hid[i], a.hid[j]) : ip.sc;
    } else if (a.sc_mode == 1) {
        sc = sc_draw(a.sc_seed, a.sc_lo, a.sc_hi, a.gid[i], a.gid[j]);
    }
    bool brk = !a.frozen && s >= sc;
    if (brk && a.has_nofail) brk = ((a.bct[a.bcc[i]].mask | a.bct[a.bcc[j]].mask) & 8u) == 0u;
    if (brk) return true;
    double w = X2w.y;
    if (a.cbond != nullptr) w *= __ldg(a.cbond + slot);
    const double c = w * s * ir;
    f[0] += c * yx;
    f[1] += c * yy;
    f[2] += c * yz;
    return false;
}

// The sums of a segment, or of a whole family, of the 32 nodes of a slice, in shared
// memory (the walk's registers are all taken).
struct __align__(16) Sums {
    float F[6][32];   // sum of -s y / |y| (times w_j / w_ref and c_ij), leading and low words
    double lit[3][32];  // force density of the literally evaluated bonds
    int info[32];       // intact bonds, + kLit if lit is not zero
};
constexpr int kLit = 1 << 16;

// The segment's bonds `pend` literally: their breaks and their forces, in slot order.
// Returns the broken ones.
__device__ __noinline__ uint32_t literal_segment(const StepArgsF64& a, int cur, int64_t i, int64_t g,
                                             int m_lo, uint32_t pend, uint32_t* bw, Sums& S)
{
    const int lane = threadIdx.x & 31;
    const int64_t slot0 = (g * 32LL * a.Q + m_lo) * 32 + lane;
    uint32_t gone = 0u;
    double lit[3] = {0.0, 0.0, 0.0};
    for (; pend; pend &= pend - 1u) {
        const int b = __ffs(pend) - 1;
        const int64_t slot = slot0 + (int64_t)b * 32;
        if (literal_bond(a, cur, i, a.nbr[slot], slot, lit)) gone |= 1u << b;
    }
    // another warp of the team may own the other half of the flag word
    if (gone) atomicAnd(bw + (m_lo >> 5) * 32, ~(gone << (m_lo & 31)));
    for (int k = 0; k < 3; ++k) S.lit[k][lane] += lit[k];
    return gone;
}

// The segments of a family that the warp takes, `rank`, rank + team, ...: into their
// entries of S (TEAM), or added up in it.  The neighbours' records come from L2 as
// often as from L1 and nothing else hides that latency (16 warps per SM, and a
// prefetch to L1 has no effect), so the walk is software-pipelined across segments:
// a record's registers are free after kin(), and the next chunk's loads go out
// there, behind them the coefficients and forces of the current one.
template <bool UW, bool TEAM, bool WIDE>
__device__ __forceinline__ void walk(const StepArgsF64& a, const W3Args& d, int cur,
                                     const Own2& own, float x_hi, float ts, int64_t i, int64_t g,
                                     int rank, int team, int Wg, Sums* S)
{
    const int lane = threadIdx.x & 31;
    const int Q = a.Q;
    const float4* __restrict__ R = d.rec[cur];
    const int32_t* __restrict__ col = a.nbr + g * 32LL * Q * 32 + lane;
    const float4* __restrict__ ilp = d.il + g * 16LL * Q * 32 + lane;
    uint32_t* const bw = a.bits + g * Q * 32 + lane;
    // first slot of the chunk after the one at m: within a segment, then the team's next
    auto after = [&](int m) { return ((m + 2) & (kSeg - 1)) ? m + 2 : m + 2 + (team - 1) * kSeg; };

    int m = rank * kSeg;
    if (m >= Wg) return;
    int mn = after(m);
    int32_t j0 = __ldg(col + m * 32), j1 = __ldg(col + m * 32 + 32);
    int32_t n0 = 0, n1 = 0;  // the next chunk's neighbours
    if (mn < Wg) {
        n0 = __ldg(col + mn * 32);
        n1 = __ldg(col + mn * 32 + 32);
    }
    Rec A, B;
    dwa::ld_rec(R + 4 * (int64_t)j0, A.a0, A.a1);
    dwa::ld_rec(R + 4 * (int64_t)j0 + 2, A.b0, A.b1);
    dwa::ld_rec(R + 4 * (int64_t)j1, B.a0, B.a1);
    dwa::ld_rec(R + 4 * (int64_t)j1 + 2, B.b0, B.b1);
    float4 il = __ldg(ilp + m * 16);
    uint32_t word = 0u, pend = 0u;
    Force F{Dw2{both(0.0f), both(0.0f)}, Dw{0.0f, 0.0f}};
    while (true) {
        const bool more = mn < Wg;
        const int b = m & (kSeg - 1);
        if (b == 0) word = (bw[(m >> 5) * 32] >> (m & 31)) & ((1u << kSeg) - 1u);
        // (a turned bond's x becomes infinite; held until literal_of as one more word, its
        // eta costs a 220k-node step 253 instead of 241 us, 237 without the bound)
        Kin bA = kin(own, A, both(ts), make_float2(ts, 1.0f));
        if (!WIDE && turned(bA.e, il.x, d.eta_max)) bA.num.h = INFINITY;
        if (more) {
            dwa::ld_rec(R + 4 * (int64_t)n0, A.a0, A.a1);
            dwa::ld_rec(R + 4 * (int64_t)n0 + 2, A.b0, A.b1);
        }
        Kin bB = kin(own, B, both(ts), make_float2(ts, 1.0f));
        if (!WIDE && turned(bB.e, il.y, d.eta_max)) bB.num.h = INFINITY;
        const float4 ilc = il;
        const int32_t c0 = j0, c1 = j1;
        const int mc = m;
        if (more) {
            dwa::ld_rec(R + 4 * (int64_t)n1, B.a0, B.a1);
            dwa::ld_rec(R + 4 * (int64_t)n1 + 2, B.b0, B.b1);
            il = __ldg(ilp + mn * 16);
            m = mn;
            mn = after(m);
            if (!UW) {
                j0 = n0;
                j1 = n1;
            }
            if (mn < Wg) {
                n0 = __ldg(col + mn * 32);
                n1 = __ldg(col + mn * 32 + 32);
            }
        }
        Coef2 cf = coef2(bA.num, bB.num, ilc);
        const uint32_t live = (word >> b) & 3u;
        const uint32_t lit = literal_of(cf.x, x_hi, d.x_max, live);
        if (d.cb != nullptr) {  // per-bond stiffness (a uniform branch)
            const float2* cb = d.cb + (g * 32LL * Q + mc) * 32 + lane;
            const float2 cA = __ldg(cb), cB = __ldg(cb + 32);
            cf.c = dw_mul2(cf.c, Dw2{make_float2(cA.x, cB.x), make_float2(cA.y, cB.y)});
        }
        if (!UW) {
            const float2 wA = __ldg(d.wrel + c0), wB = __ldg(d.wrel + c1);
            cf.c = dw_mul2(cf.c, Dw2{make_float2(wA.x, wB.x), make_float2(wA.y, wB.y)});
        }
        pend |= lit << b;
        add_force(F, cf.c.h.x, cf.c.l.x, bA, (live & ~lit) & 1u);
        add_force(F, cf.c.h.y, cf.c.l.y, bB, (live & ~lit) & 2u);
        F.xy = renorm2(F.xy);  // (240 -> 242 us a step; without it 1.6 times the error at 0.6 %)
        F.z = renorm(F.z);

        if (b == kSeg - 2 || !more) {  // the segment's end
            const int m_lo = mc & ~(kSeg - 1);
            Sums& T = S[TEAM ? m_lo / kSeg : 0];
            const Dw Fk[3] = {{F.xy.h.x, F.xy.l.x}, {F.xy.h.y, F.xy.l.y}, F.z};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Dw t = TEAM ? Fk[k] : dw_add(Dw{T.F[2 * k][lane], T.F[2 * k + 1][lane]}, Fk[k]);
                T.F[2 * k][lane] = t.h;
                T.F[2 * k + 1][lane] = t.l;
            }
            F = Force{Dw2{both(0.0f), both(0.0f)}, Dw{0.0f, 0.0f}};
            int info = TEAM ? 0 : T.info[lane];
            if (pend) {
                if (TEAM)
                    for (int k = 0; k < 3; ++k) T.lit[k][lane] = 0.0;
                word &= ~literal_segment(a, cur, i, g, m_lo, pend, bw, T);
                info |= kLit;
                pend = 0u;
            }
            T.info[lane] = info + __popc(word);
        }
        if (!more) break;
    }
}

template <bool UW, bool TEAM, bool WIDE>
__global__ void __launch_bounds__(256, 2)
    k_step_f64(const __grid_constant__ StepArgsF64 a, const __grid_constant__ W3Args d)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    const int team = TEAM ? d.team : 1;       // warps per slice (a power of two)
    const int sh = TEAM ? __ffs(team) - 1 : 0;
    const int tpb = wpb >> sh;                // slices per block at a time
    const int tm = (int)(threadIdx.x >> 5) >> sh;
    const int rank = (int)(threadIdx.x >> 5) & (team - 1);
    // the slice's sums: one entry, or one per segment for a team
    Sums* const S = reinterpret_cast<Sums*>(smem) + (TEAM ? tm * d.max_seg : tm);
    const int64_t nslices = (a.n + 31) >> 5;

    // before the previous kernel is done (programmatic launch): nothing it writes is read
    if (lane == 0 && rank == 0 && (int64_t)blockIdx.x * tpb + tm < nslices) {
        const int64_t g = (int64_t)blockIdx.x * tpb + tm;
        const int Wg = a.sw[g];
        prefetch_l2(a.nbr + g * 32LL * a.Q * 32, (uint32_t)(((Wg + 3) & ~3) * 128));
        if (TEAM) prefetch_l2(d.il + g * 16LL * a.Q * 32, (uint32_t)(((Wg + 3) & ~3) * 256));
    }
    pdl_begin(TEAM);
    const int64_t step = a.step_ctr[0] + a.k;
    const int cur = (int)(step & 1);
    const float4* __restrict__ R = d.rec[cur];

    // (every warp of a block makes the same number of rounds: teams synchronise)
    for (int64_t g0 = (int64_t)blockIdx.x * tpb; g0 < nslices; g0 += (int64_t)gridDim.x * tpb) {
        const int64_t g = g0 + tm;
        const bool have = g < nslices;
        if (!TEAM && !have) continue;
        const int64_t i = (g << 5) + lane;
        Rec me{};
        Node nd{};
        int nseg = 0;
        double w_ref = d.w_ref, scale = d.scale;
        if (have) {
            const int Wg = a.sw[g];
            nseg = (Wg + kSeg - 1) / kSeg;
            if (lane == 0 && rank == 0 && g0 != (int64_t)blockIdx.x * tpb)
                prefetch_l2(a.nbr + g * 32LL * a.Q * 32, (uint32_t)(((Wg + 3) & ~3) * 128));
            dwa::ld_rec(R + 4 * i, me.a0, me.a1);
            dwa::ld_rec(R + 4 * i + 2, me.b0, me.b1);
            const Own2 own = own_pairs(me);
            float x_hi = d.x_hi;
            int grid = d.x_grid;
            if (a.inst != nullptr) {  // batch: the instance's own band, weight and unit
                const InstParams& ip = a.itab[a.inst[i]];
                w_ref = ip.w_ref;
                scale = ip.w3_scale;
                if (!a.frozen) x_hi = ip.w3_x_hi;
                grid = ip.w3_x_grid;
            }
            const float ts = pow2(grid - 33);
            if (!TEAM) {
#pragma unroll
                for (int k = 0; k < 6; ++k) S->F[k][lane] = 0.0f;
#pragma unroll
                for (int k = 0; k < 3; ++k) S->lit[k][lane] = 0.0;
                S->info[lane] = 0;
            }
            walk<UW, TEAM, WIDE>(a, d, cur, own, x_hi, ts, i, g, rank, team, Wg, S);
            if (rank == 0) nd = load_node(a, d, cur, i);  // (node arrays are padded)
        }
        if (TEAM) __syncthreads();
        if (have && rank == 0 && i < a.n) {
            // the segments' sums in their order, whichever warps formed them
            Dw F[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
            double T[3] = {0.0, 0.0, 0.0};
            int alive = 0;
            for (int e = 0; e < (TEAM ? nseg : 1); ++e) {
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    F[k] = dw_add(F[k], Dw{S[e].F[2 * k][lane], S[e].F[2 * k + 1][lane]});
                const int info = S[e].info[lane];
                alive += info & (kLit - 1);
                if (info >= kLit) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) T[k] += S[e].lit[k][lane];
                }
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) T[k] = fma(-((double)F[k].h + (double)F[k].l), w_ref, T[k]);
            finish_node(a, d, cur, step, me, nd, scale, i, T, alive);
        }
        if (TEAM) __syncthreads();  // the sums' memory is free again
    }
}

// Records of every node from its FP64 record
__global__ void k_w3_publish(const double* __restrict__ rec64, float4* __restrict__ rec,
                             int64_t n_pad, double scale, int x_grid, double3 origin,
                             const int32_t* __restrict__ inst, const InstParams* __restrict__ itab)
{
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n_pad;
         p += (int64_t)gridDim.x * blockDim.x) {
        const double* r = rec64 + 8 * p;
        const double sc = inst != nullptr ? itab[inst[p]].w3_scale : scale;
        const int g = inst != nullptr ? itab[inst[p]].w3_x_grid : x_grid;
        const double3 o = inst != nullptr ? itab[inst[p]].w3_origin : origin;
        const double o3[3] = {o.x, o.y, o.z};
        float xh[3], xm[3], uh[3], um[3], t[3];
        for (int k = 0; k < 3; ++k) {
            float xt, ut;
            split3((r[k] - o3[k]) * sc, g, xh[k], xm[k], xt);
            split3(r[4 + k] * sc, kW3UGrid, uh[k], um[k], ut);
            t[k] = pack_t(t_int(xt, g), ut);
        }
        rec[4 * p] = make_float4(xh[0], xh[1], uh[0], uh[1]);
        rec[4 * p + 1] = make_float4(xh[2], uh[2], t[0], t[1]);
        rec[4 * p + 2] = make_float4(xm[0], xm[1], um[0], um[1]);
        rec[4 * p + 3] = make_float4(xm[2], um[2], t[2], 0.0f);
    }
}

// U / |xi| of every slot as a double-word (1 where there is no bond, not a number past il_max,
// so that x is not and the bond literal), by pairs of slots: {h, h', l, l'} of slots m and m + 1
__global__ void k_w3_ilen(const double* __restrict__ ilen, const int32_t* __restrict__ nbr,
                          const int32_t* __restrict__ sw, int64_t n, int Q, double scale,
                          float il_max, const int32_t* __restrict__ inst,
                          const InstParams* __restrict__ itab, float4* __restrict__ il)
{
    const int64_t W = 32LL * Q;
    const int64_t total = ((n + 31) >> 5) << 5;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < total;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = p >> 5;
        const double U = 1.0 / (inst != nullptr ? itab[inst[p]].w3_scale : scale);  // a power of two
        const float top = inst != nullptr ? itab[inst[p]].w3_il_max : il_max;
        for (int m = 0; m < W; m += 2) {
            float h[2], l[2];
            for (int k = 0; k < 2; ++k) {
                const int64_t slot = (g * W + m + k) * 32 + (p & 31);
                const double v = m + k < sw[g] && nbr[slot] != p ? ilen[slot] * U : 1.0;
                h[k] = v <= (double)top ? (float)v : __uint_as_float(0x7fc00000u);
                l[k] = (float)(v - (double)h[k]);
            }
            il[(g * W / 2 + m / 2) * 32 + (p & 31)] = make_float4(h[0], h[1], l[0], l[1]);
        }
    }
}

int grid_of(int64_t work)
{
    const int64_t b = (work + 255) / 256;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 16));
}

}  // namespace

size_t step_f64_smem(int team, int max_seg, int block)
{
    return (size_t)(block / 32 / team) * (team > 1 ? max_seg : 1) * sizeof(Sums);
}

size_t step_f64_smem_max() { return step_f64_smem(2, kW3TeamSegs, 256); }

// Percent of the unified L1/shared array (228 KB) that the sums of 16 resident warps
// take; the rest is the records' L1.
int step_f64_carveout(int team, int max_seg, int block)
{
    const size_t resident = (size_t)(512 / block) * (step_f64_smem(team, max_seg, block) + 1024);
    return (int)std::min<size_t>(100, 1 + 100 * resident / (228 << 10));
}

const void* step_f64_kernel(bool uniform_w, bool team, bool wide)
{
    static const void* const k[8] = {
        (const void*)k_step_f64<false, false, false>, (const void*)k_step_f64<false, true, false>,
        (const void*)k_step_f64<true, false, false>,  (const void*)k_step_f64<true, true, false>,
        (const void*)k_step_f64<false, false, true>,  (const void*)k_step_f64<false, true, true>,
        (const void*)k_step_f64<true, false, true>,   (const void*)k_step_f64<true, true, true>};
    return k[(wide ? 4 : 0) + (uniform_w ? 2 : 0) + (team ? 1 : 0)];
}

cudaError_t launch_step_f64(const StepArgsF64& a, const W3Args& d, int grid, int block,
                            cudaStream_t s)
{
    const void* fn = step_f64_kernel(d.uniform_w != 0, d.team > 1, d.wide != 0);
    void* args[] = {const_cast<StepArgsF64*>(&a), const_cast<W3Args*>(&d)};
    return launch_pdl(fn, dim3(grid), dim3(block), args, step_f64_smem(d.team, d.max_seg, block), s,
                      step_f64_carveout(d.team, d.max_seg, block));
}

cudaError_t launch_w3_publish(const double* rec64, float4* rec, int64_t n_pad, double scale,
                              int x_grid, double3 origin, const int32_t* inst,
                              const InstParams* itab, cudaStream_t s)
{
    k_w3_publish<<<grid_of(n_pad), 256, 0, s>>>(rec64, rec, n_pad, scale, x_grid, origin, inst, itab);
    return cudaGetLastError();
}

cudaError_t launch_w3_ilen(const double* ilen, const int32_t* nbr, const int32_t* sw, int64_t n,
                           int Q, double scale, float il_max, const int32_t* inst,
                           const InstParams* itab, float4* il, cudaStream_t s)
{
    k_w3_ilen<<<grid_of(((n + 31) >> 5) << 5), 256, 0, s>>>(ilen, nbr, sw, n, Q, scale, il_max, inst,
                                                            itab, il);
    return cudaGetLastError();
}

}  // namespace pd
