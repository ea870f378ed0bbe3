// tctile.cuh -- what the two tensor-core summations (tcsum.cu, tcsum64.cu) share: tile records, the
// fixed-point phases and the warpgroup barrier.
#pragma once

#include "fewsum_internal.h"
#include "launch.cuh"
#include "phase_eval.cuh"
#include "tcgen05.cuh"

namespace fewsum {

// A pointer into the plan, for a plan that may be read elsewhere than at its device address (from the
// kernel parameters).
template <typename T>
__device__ __forceinline__ const T *tc_local(const PlanHdr &h, const T *p)
{
    return reinterpret_cast<const T *>(reinterpret_cast<const unsigned char *>(&h) +
                                       (reinterpret_cast<const unsigned char *>(p) - h.self));
}
__device__ __forceinline__ const WaveDev &tc_wave(const PlanHdr &h, int w) { return tc_local(h, h.waves)[w]; }

// The last block writes a plan that came in the parameters to its device address (after pdl_wait).
__device__ __forceinline__ void tc_store_plan(const PlanParam &plan)
{
    if (blockIdx.x + 1 != gridDim.x) return;
    const uint4 *src = reinterpret_cast<const uint4 *>(plan.bytes);
    for (int i = threadIdx.x; i < (plan.n + 15) / 16; i += blockDim.x)
        reinterpret_cast<uint4 *>(plan.dev)[i] = src[i];
}

// A value in turns as 2^-64 turn units modulo one turn.
__device__ __forceinline__ long long turns_fixed(double y)
{
    return __double2ll_rn((y - rint(y)) * 18446744073709551616.0);
}

// Pairs hi + lo of doubles (106 bits) for the FP64 plans' records: one anchor stands for 128 samples,
// so its rounding would be common to them; formed in pairs it stays far below FP64's own.
struct Dd {
    double h, l;
};
__device__ __forceinline__ Dd dd_sum(double a, double b)
{
    const double s = a + b, v = s - a;
    return Dd{s, (a - (s - v)) + (b - v)};
}
__device__ __forceinline__ Dd dd_prod(double a, double b)
{
    const double p = a * b;
    return Dd{p, fma(a, b, -p)};
}
__device__ __forceinline__ Dd dd_add(const Dd &a, const Dd &b)
{
    const Dd s = dd_sum(a.h, b.h);
    return dd_sum(s.h, s.l + (a.l + b.l));
}
__device__ __forceinline__ Dd dd_mul(const Dd &a, const Dd &b)
{
    const Dd p = dd_prod(a.h, b.h);
    return dd_sum(p.h, p.l + fma(a.h, b.l, a.l * b.h));
}
__device__ __forceinline__ Dd dd_scale(const Dd &a, double x) { return dd_mul(a, Dd{x, 0.0}); }
__device__ __forceinline__ Dd dd_div(const Dd &a, double b)
{
    const double q = a.h / b;
    return dd_sum(q, (fma(-q, b, a.h) + a.l) / b);
}
__device__ __forceinline__ long long dd_turns_fixed(const Dd &a)
{
    return (long long)((unsigned long long)__double2ll_rn((a.h - rint(a.h)) * 18446744073709551616.0) +
                       (unsigned long long)__double2ll_rn(a.l * 18446744073709551616.0));
}

// The Taylor coefficients (turns per sample^k, fixed point) of one phase spline about time x after the
// segment's first knot, from its Hermite data (values y0, y1, slopes s0, s1, width h) in pairs; offset
// added to the phase.  v^3 reaches 2^21, so the cubic coefficient also gets its next 32 bits (lo3, units
// of 2^-96 turn).
__device__ inline void dd_phase_taylor(const double *c, double h, const Dd &x, double dt, double offset,
                                       long long (&out)[4], int &lo3)
{
    const Dd inv2pi{0.15915494309189535, -9.8393400450386e-18};  // 1/(2 pi)
    const Dd a = dd_prod(h, c[2]), b = dd_prod(h, c[3]), D = dd_sum(c[1], -c[0]);
    const Dd p1 = dd_add(dd_scale(D, 3.0), dd_add(dd_scale(a, -2.0), Dd{-b.h, -b.l}));
    const Dd p2 = dd_add(dd_add(a, b), dd_scale(D, -2.0));
    const Dd u = dd_div(x, h), du = dd_mul(dd_div(Dd{dt, 0.0}, h), inv2pi), w = dd_div(Dd{dt, 0.0}, h);
    const Dd v0 = dd_mul(dd_add(dd_mul(dd_add(dd_mul(p2, u), p1), u), a), u);
    out[0] = dd_turns_fixed(dd_mul(dd_add(v0, dd_sum(c[0], offset)), inv2pi));
    const Dd q = dd_add(dd_scale(dd_mul(p2, u), 3.0), p1);                                // Phi''/2
    const Dd d1 = dd_add(dd_mul(dd_add(dd_scale(dd_mul(p2, u), 3.0), dd_scale(p1, 2.0)), u), a);  // Phi'
    out[1] = dd_turns_fixed(dd_mul(d1, du));
    out[2] = dd_turns_fixed(dd_mul(dd_mul(q, w), du));
    const Dd c3 = dd_mul(dd_mul(dd_mul(p2, w), w), du);
    const double x3 = (c3.h - rint(c3.h)) * 18446744073709551616.0;
    out[3] = __double2ll_rn(x3);
    const double rest = (x3 - (double)out[3]) + c3.l * 18446744073709551616.0;
    lo3 = __double2int_rn(rest * 4294967296.0);
}

__device__ __forceinline__ int tc_wave_of_seg(const PlanHdr &h, int g)
{
    int lo = 0, hi = h.n_waves - 1;
    while (lo < hi) {  // largest w with seg_begin <= g
        const int mid = (lo + hi + 1) >> 1;
        if (tc_wave(h, mid).seg_begin <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Record of tile T: its segment, the phases at its first sample and their Taylor expansion (FP64;
// pairs of FP64 for the FP64 plans).
__device__ inline void tc_fill_record(const PlanHdr &h, int T, bool fp64)
{
    int lo = 0, hi = h.n_waves - 1;
    while (lo < hi) {  // largest w with tile_begin <= T
        const int mid = (lo + hi + 1) >> 1;
        if (tc_wave(h, mid).tile_begin <= T) lo = mid; else hi = mid - 1;
    }
    const WaveDev &W = tc_wave(h, lo);
    const TrajDev &tr = W.tr;
    const int *tile_off = tc_local(h, W.tile_off), *seg_start = tc_local(h, W.seg_start);
    const int t = T - W.tile_begin;
    int s = 0, e = tr.S - 1;
    while (s < e) {  // largest s with tile_off[s] <= t: the segment that holds tile t
        const int mid = (s + e + 1) >> 1;
        if (tile_off[mid] <= t) s = mid; else e = mid - 1;
    }
    TileRec r;
    r.s0 = seg_start[s];
    r.s1 = seg_start[s + 1];
    r.i0 = (r.s0 / kTcTile + (t - tile_off[s])) * kTcTile;
    r.tile_end = W.tile_begin + tile_off[s + 1];
    const SegPhase sp = seg_phase(tr, s, W.dphi_phi, W.dphi_r);
    const double kInv2Pi = 0.15915494309189533577;
    const double u = (fma((double)max(r.i0, r.s0), W.dt, W.t0) - sp.tk) * sp.ih, du = W.dt * sp.ih;
    double all = 0.0;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const double *p = k ? sp.pr : sp.pphi;
        long long *c = k ? r.r : r.phi;
        const double f0 = fma(fma(fma(p[2], u, p[1]), u, p[0]), u, k ? sp.c0r : sp.c0phi) * kInv2Pi;
        c[0] = turns_fixed(f0);
        c[1] = turns_fixed(fma(fma(3.0 * p[2], u, 2.0 * p[1]), u, p[0]) * du * kInv2Pi);
        c[2] = turns_fixed(fma(3.0 * p[2], u, p[1]) * du * du * kInv2Pi);
        c[3] = turns_fixed(p[2] * du * du * du * kInv2Pi);
        all += f0;
    }
    // integers cannot carry a NaN: non-finite phases (latched by the build) reach the output here
    // (FP64: in the segment's factor)
    r.u0 = (float)((fma((double)r.s0, W.dt, W.t0) - sp.tk) * sp.ih) + (float)(all - all);
    r.du = (float)du;
    if (fp64) {
        const double *c = tr.coef + (size_t)s * tr.J * 4;
        const Dd x = dd_add(dd_prod((double)max(r.i0, r.s0), W.dt), dd_sum(W.t0, -sp.tk));
        int lo_phi, lo_r;
        dd_phase_taylor(c, tr.h[s], x, W.dt, W.dphi_phi, r.phi, lo_phi);
        dd_phase_taylor(c + 4, tr.h[s], x, W.dt, W.dphi_r, r.r, lo_r);
        r.u0 = __int_as_float(lo_phi);
        r.du = __int_as_float(lo_r);
    }
    r.seg = fp64 ? (const void *)(W.seg64 + s) : (const void *)(W.tab_inv + s);
    r.tab = W.tab + (size_t)s * (fp64 ? tc64_table_bytes(tr.tc_pairs, tr.tc_ks)
                                      : tc_table_bytes(tr.tc_pairs, tr.tc_ks));
    r.out = W.out;
    r.pairs = tr.tc_pairs;
    r.ks = tr.tc_ks;
    r.n_mid = tr.n_mid;
    r.c64 = W.out_c64;
    h.recs[T] = r;
}

// c0 + c1 v + c2 v^2 + c3 v^3 in 64-bit wrap-around arithmetic (modulo one turn).
__device__ __forceinline__ unsigned long long phase_fixed(const long long *c, uint32_t v)
{
    const longlong2 a = reinterpret_cast<const longlong2 *>(c)[0];
    const longlong2 b = reinterpret_cast<const longlong2 *>(c)[1];
    unsigned long long p = (unsigned long long)b.y;
    p = p * v + (unsigned long long)b.x;
    p = p * v + (unsigned long long)a.y;
    return p * v + (unsigned long long)a.x;
}

// Barrier of one warpgroup that also tells every thread whether any of them failed.
__device__ __forceinline__ bool wg_any(int id, bool bad)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred q, %2, 128, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)bad), "r"(id)
        : "memory");
    return r != 0;
}

}  // namespace fewsum
