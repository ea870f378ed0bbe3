// tctile.cuh -- what the two tensor-core summations (tcsum.cu, tcsum64.cu) share: tile records, the
// fixed-point phases and the warpgroup barrier.
#pragma once

#include <type_traits>

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

// A value in turns as 2^-64 turn units modulo one turn (0 if not finite): the significand shifted into
// place.  (Four FP64 instructions would do it too, of 64 cycles each for a scheduler's warp.)
__device__ __forceinline__ long long turns_fixed(double y)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(y);
    const int e = (int)(b >> 52) & 2047, sh = e - 1011;  // significand 2^(e - 1075) = units 2^sh
    const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
    unsigned long long v = 0;
    if (sh >= 0) {
        if (sh < 64) v = m << sh;
    } else if (sh > -55) {
        v = ((m >> (-sh - 1)) + 1) >> 1;
    }
    return (long long)((long long)b < 0 ? 0ull - v : v);
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
    return (long long)((unsigned long long)turns_fixed(a.h) + (unsigned long long)turns_fixed(a.l));
}

// The same with the next 32 bits (units of 2^-96 turn).
__device__ __forceinline__ long long tc_fixed96(const Dd &a, int &lo)
{
    const double x = (a.h - rint(a.h)) * 18446744073709551616.0, y = a.l * 18446744073709551616.0;
    const long long cx = __double2ll_rn(x), cy = __double2ll_rn(y);
    const double r = (x - (double)cx) + (y - (double)cy), k = rint(r);
    lo = __double2int_rn((r - k) * 4294967296.0);
    return (long long)((unsigned long long)cx + (unsigned long long)cy + (unsigned long long)(long long)k);
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

// Tile records.  A record holds the Taylor expansion of its segment's phases about the tile's first
// sample: polynomials in u = (t - t_k)/h of the phase and of its derivatives per sample, in turns, whose
// coefficients are the segment's.  A lane a segment forms those for 32 segments at a time in shared
// memory, and a thread a tile only evaluates them: FP64 arithmetic bounds the fill (16 cycles a warp
// instruction and SM), and every tile forming its own coefficients took four times as many.
struct PhaseFill {  // the phase c, its derivative per sample d, half the second one q, a sixth of the third
    double c[4], d[3], q[2];
    long long c3;
};
struct PhaseFill64 {  // the same in pairs; v^3 reaches 2^21, so c3 also has its next 32 bits (2^-96 turn; c2: tc_fixed96)
    Dd c[4], d[3], q[2];
    long long c3;
    int lo3;
};
template <bool FP64>
struct SegFill {
    std::conditional_t<FP64, PhaseFill64, PhaseFill> p[2];
    double tk, t0, dt;
    Dd ih;
    const void *seg, *tab;
    void *out;
    float u0, du;
    int first, end;  // tiles
    int s0, s1;
    int pairs, ks, n_mid, c64;
};

// x modulo 2 pi (2 pi in two parts; see reduce_2pi).
__device__ __forceinline__ double tc_reduce(double x)
{
    const double k = rint(x * 0.15915494309189533577);
    return fma(-k, 2.4492935982947064e-16, fma(-k, 6.283185307179586232, x));
}

// Every product that is added to something is an explicit fma or an explicit product, so that the two
// places this is inlined in round alike.
__device__ inline void tc_phase_fill(const double *y, double h, Dd ih, double dt, double offset,
                                     PhaseFill &o)
{
    const double kInv2Pi = 0.15915494309189533577;
    const double D = y[1] - y[0], a = __dmul_rn(h, y[2]), b = __dmul_rn(h, y[3]);  // (hermite_to_power)
    const double c2 = fma(-2.0, a, fma(3.0, D, -b)), c3 = fma(-2.0, D, a + b);
    const double w = dt * ih.h, w2 = w * w, t = 3.0 * c3 * kInv2Pi;
    o.c[0] = (tc_reduce(y[0]) + tc_reduce(offset)) * kInv2Pi;
    o.c[1] = a * kInv2Pi;
    o.c[2] = c2 * kInv2Pi;
    o.c[3] = c3 * kInv2Pi;
    o.d[0] = o.c[1] * w;
    o.d[1] = __dmul_rn(o.c[2], 2.0 * w);
    o.d[2] = t * w;
    o.q[0] = o.c[2] * w2;
    o.q[1] = t * w2;
    o.c3 = turns_fixed(o.c[3] * w * w2);
}

__device__ inline void tc_phase_fill(const double *y, double h, Dd ih, double dt, double offset,
                                     PhaseFill64 &o)
{
    const Dd inv2pi{0.15915494309189535, -9.8393400450386e-18};  // 1/(2 pi)
    const Dd a = dd_prod(h, y[2]), b = dd_prod(h, y[3]), D = dd_sum(y[1], -y[0]);
    const Dd p1 = dd_add(dd_scale(D, 3.0), dd_add(dd_scale(a, -2.0), Dd{-b.h, -b.l}));
    const Dd p2 = dd_add(dd_add(a, b), dd_scale(D, -2.0));
    const Dd w = dd_scale(ih, dt);
    o.c[0] = dd_mul(dd_sum(y[0], offset), inv2pi);
    o.c[1] = dd_mul(a, inv2pi);
    o.c[2] = dd_mul(p1, inv2pi);
    o.c[3] = dd_mul(p2, inv2pi);
    o.d[0] = dd_mul(o.c[1], w);
    o.q[0] = dd_mul(o.c[2], w);
    const Dd c3 = dd_mul(o.c[3], w);
    o.d[1] = Dd{2.0 * o.q[0].h, 2.0 * o.q[0].l};
    o.d[2] = dd_scale(c3, 3.0);
    o.q[0] = dd_mul(o.q[0], w);
    o.q[1] = dd_mul(o.d[2], w);
    o.c3 = tc_fixed96(dd_mul(dd_mul(c3, w), w), o.lo3);
}

__device__ __forceinline__ double tc_u(const SegFill<false> &S, int i)
{
    return (fma((double)i, S.dt, S.t0) - S.tk) * S.ih.h;
}
__device__ __forceinline__ Dd tc_u(const SegFill<true> &S, int i)
{
    return dd_mul(dd_add(dd_prod((double)i, S.dt), dd_sum(S.t0, -S.tk)), S.ih);
}
// The expansion about u; returns whether the phase is finite.
__device__ __forceinline__ bool tc_phase_at(const PhaseFill &p, double u, long long (&o)[4])
{
    const double f = fma(fma(fma(p.c[3], u, p.c[2]), u, p.c[1]), u, p.c[0]);
    o[0] = turns_fixed(f);
    o[1] = turns_fixed(fma(fma(p.d[2], u, p.d[1]), u, p.d[0]));
    o[2] = turns_fixed(fma(p.q[1], u, p.q[0]));
    o[3] = p.c3;
    return (__double2hiint(f) & 0x7ff00000) != 0x7ff00000;
}
// lo2: c2's next 32 bits.  v^2 reaches 2^14: rounded to 2^-64 turn, c2 alone was wrong by up to 3e-15 rad at a
// tile's end, n times that in the n-th power, which showed wherever the phases themselves are small.
__device__ __forceinline__ void tc_phase_at(const PhaseFill64 &p, const Dd &u, long long (&o)[4], int &lo2)
{
    o[0] = dd_turns_fixed(
        dd_add(dd_mul(dd_add(dd_mul(dd_add(dd_mul(p.c[3], u), p.c[2]), u), p.c[1]), u), p.c[0]));
    o[1] = dd_turns_fixed(dd_add(dd_mul(dd_add(dd_mul(p.d[2], u), p.d[1]), u), p.d[0]));
    o[2] = tc_fixed96(dd_add(dd_mul(p.q[1], u), p.q[0]), lo2);
    o[3] = p.c3;
}

template <bool FP64>
__device__ __forceinline__ Dd tc_seg_ih(const WaveDev &W, int s)
{
    if constexpr (FP64) return dd_div(Dd{1.0, 0.0}, W.tr.h[s]);
    return Dd{W.tr.inv_h[s], 0.0};
}
// Phase p (0 Phi_phi, 1 Phi_r) of segment s.
template <bool FP64>
__device__ __forceinline__ void tc_seg_phase(const WaveDev &W, int s, int p, Dd ih, SegFill<FP64> &o)
{
    tc_phase_fill(W.tr.coef + (size_t)s * W.tr.J * 4 + 4 * p, W.tr.h[s], ih, W.dt, p ? W.dphi_r : W.dphi_phi, o.p[p]);
}
// The rest of segment s.
template <bool FP64>
__device__ inline void tc_seg_fill(const PlanHdr &h, const WaveDev &W, int s, Dd ih, SegFill<FP64> &o)
{
    const TrajDev &tr = W.tr;
    const int *tile_off = tc_local(h, W.tile_off), *seg_start = tc_local(h, W.seg_start);
    o.first = W.tile_begin + tile_off[s];
    o.end = W.tile_begin + tile_off[s + 1];
    o.s0 = seg_start[s];
    o.s1 = seg_start[s + 1];
    o.tk = tr.t[s];
    o.t0 = W.t0;
    o.dt = W.dt;
    o.ih = ih;
    o.u0 = (float)((fma((double)o.s0, W.dt, W.t0) - o.tk) * ih.h);
    o.du = (float)(W.dt * ih.h);
    o.seg = FP64 ? (const void *)(W.seg64 + s) : (const void *)(W.tab_inv + s);
    o.tab = W.tab + (size_t)s * (FP64 ? tc64_table_bytes(tr.tc_pairs, tr.tc_ks)
                                      : tc_table_bytes(tr.tc_pairs, tr.tc_ks));
    o.out = W.out;
    o.pairs = tr.tc_pairs;
    o.ks = tr.tc_ks;
    o.n_mid = tr.n_mid;
    o.c64 = W.out_c64;
}

// Segments g0 .. of the plan for a block's cache; past the last one: no tiles.  FP64: a phase a thread (the
// second phases in another warp, on another scheduler's share of the FP64 pipe).
template <bool FP64>
__device__ inline void tc_cache_segs(const PlanHdr &h, int g0, SegFill<FP64> *seg)
{
    constexpr int kThreads = FP64 ? 2 * kTcFillSegs : kTcFillSegs;
    if (threadIdx.x >= kThreads) return;
    const int k = threadIdx.x % kTcFillSegs, p = threadIdx.x / kTcFillSegs, g = g0 + k;
    if (g >= h.total_segs) {
        if (p == 0) seg[k].first = seg[k].end = h.total_tiles;
        return;
    }
    const WaveDev &W = tc_wave(h, tc_wave_of_seg(h, g));
    const int s = g - W.seg_begin;
    const Dd ih = tc_seg_ih<FP64>(W, s);
    tc_seg_phase<FP64>(W, s, p, ih, seg[k]);
    if (!FP64) tc_seg_phase<FP64>(W, s, 1, ih, seg[k]);
    if (p == 0) tc_seg_fill<FP64>(h, W, s, ih, seg[k]);
}

// The segment s of wave W that holds tile T.
__device__ inline const WaveDev &tc_find_tile(const PlanHdr &h, int T, int &s)
{
    int lo = 0, hi = h.n_waves - 1;
    while (lo < hi) {  // largest w with tile_begin <= T
        const int mid = (lo + hi + 1) >> 1;
        if (tc_wave(h, mid).tile_begin <= T) lo = mid; else hi = mid - 1;
    }
    const WaveDev &W = tc_wave(h, lo);
    const int *tile_off = tc_local(h, W.tile_off);
    int e = W.tr.S - 1;
    s = 0;
    while (s < e) {  // largest s with tile_off[s] <= t: the segment that holds tile T
        const int mid = (s + e + 1) >> 1;
        if (tile_off[mid] <= T - W.tile_begin) s = mid; else e = mid - 1;
    }
    return W;
}

// What a record holds beside the phases.  fin: the phases are finite.
template <bool FP64>
__device__ __forceinline__ void tc_record_rest(const SegFill<FP64> &S, int t, bool fin, TileRec &r)
{
    r.i0 = (S.s0 / kTcTile + (t - S.first)) * kTcTile;
    r.s0 = S.s0;
    r.s1 = S.s1;
    r.tile_end = S.end;
    if constexpr (FP64) {  // non-finite data reach the output through the segment's factor
        r.u0 = __int_as_float(S.p[0].lo3);
        r.du = __int_as_float(S.p[1].lo3);
    } else {  // integers cannot carry a NaN: non-finite phases (latched by the build) go here
        r.u0 = fin ? S.u0 : __int_as_float(0x7fffffff);
        r.du = S.du;
    }
    r.seg = S.seg;
    r.tab = static_cast<const unsigned char *>(S.tab);
    r.out = S.out;
    r.pairs = S.pairs;
    r.ks = S.ks;
    r.n_mid = S.n_mid;
    r.c64 = S.c64;
}

template <bool FP64>
__device__ __forceinline__ auto tc_tile_u(const SegFill<FP64> &S, int t)
{
    return tc_u(S, max((S.s0 / kTcTile + (t - S.first)) * kTcTile, S.s0));
}

__device__ __forceinline__ void tc_store_record(const PlanHdr &h, const SegFill<false> &S, int t)
{
    TileRec r;
    const double u = tc_tile_u(S, t);
    bool fin = tc_phase_at(S.p[0], u, r.phi);
    fin = tc_phase_at(S.p[1], u, r.r) && fin;
    tc_record_rest(S, t, fin, r);
    h.recs[t] = r;
}

// FP64: phase p of a record, and with the first one the rest.
__device__ __forceinline__ void tc_store_record(const PlanHdr &h, const SegFill<true> &S, int t, int p)
{
    TileRec r, &dst = h.recs[t];
    int lo2;
    tc_phase_at(S.p[p], tc_tile_u(S, t), r.phi, lo2);
    longlong2 *c = reinterpret_cast<longlong2 *>(dst.phi) + 2 * p;
    c[0] = make_longlong2(r.phi[0], r.phi[1]);
    c[1] = make_longlong2(r.phi[2], r.phi[3]);
    (p ? dst.c64 : dst.ks) = lo2;
    if (p > 0) return;
    tc_record_rest(S, t, true, r);
#pragma unroll
    for (int q = 4; q < 7; ++q) reinterpret_cast<int4 *>(&dst)[q] = reinterpret_cast<const int4 *>(&r)[q];
    dst.pairs = tc64_shape(r.pairs, r.ks, r.c64);
    dst.n_mid = r.n_mid;
}

// The records of a block after the segments' (an even share of the tiles; seg: kTcFillSegs entries in
// shared memory).  Shares of one tile a thread form their segments' coefficients themselves (mixed): one
// chain of latencies instead of two, 1.5 us of a one-week waveform's 25; with more tiles the cache wins:
// records and fold of a four-year one 190 -> 74 us.
template <bool FP64>
__device__ inline void tc_fill_records(const PlanHdr &h, SegFill<FP64> *seg)
{
    const int blocks = (int)gridDim.x - h.total_segs, share = (h.total_tiles + blocks - 1) / blocks;
    int T = ((int)blockIdx.x - h.total_segs) * share;
    const int T1 = min(h.total_tiles, T + share);
    if (!FP64 && share <= kTcRecTiles) {
        T += threadIdx.x;
        if (T >= T1) return;
        int s;
        const WaveDev &W = tc_find_tile(h, T, s);
        SegFill<false> S;
        const Dd ih = tc_seg_ih<false>(W, s);
        tc_seg_phase<false>(W, s, 0, ih, S);
        tc_seg_phase<false>(W, s, 1, ih, S);
        tc_seg_fill<false>(h, W, s, ih, S);
        tc_store_record(h, S, T);
        return;
    }
    while (T < T1) {  // uniform
        int s;
        const WaveDev &W = tc_find_tile(h, T, s);
        tc_cache_segs<FP64>(h, W.seg_begin + s, seg);
        __syncthreads();
        const int Te = min(T1, seg[kTcFillSegs - 1].end);
        for (int i = threadIdx.x; i < (FP64 ? 2 : 1) * (Te - T); i += blockDim.x) {
            const int p = i >= Te - T, t = T + i - p * (Te - T);
            int k = 0, ke = kTcFillSegs - 1;
            while (k < ke) {  // largest k with first <= t
                const int mid = (k + ke + 1) >> 1;
                if (seg[mid].first <= t) k = mid; else ke = mid - 1;
            }
            if constexpr (FP64)
                tc_store_record(h, seg[k], t, p);
            else
                tc_store_record(h, seg[k], t);
        }
        __syncthreads();
        T = Te;
    }
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
