// tcsum.cu -- the mixed-precision mode sum on the tensor cores (arXiv:2104.04582 Sec. 3.C, Sec. 4).
//
// With K_{m,n}(u) = sum_d c_{m,n,d} u^d the folded cubic of a signed frequency (fold_tc.cuh),
// n = n_mid + b and theta = Phi_r, the sum over n of one row m is, degree by degree,
//     sum_n c_{m,n,d} e^{-i n theta} = e^{-i n_mid theta} [ sum_{b >= 0} X_{m,b,d} cos(b theta)
//                                                        + Y_{m,b,d} sin(b theta) ],
//     X = c_{+b} + c_{-b},  Y = -i (c_{+b} - c_{-b})   (b = 0: X = c_0, Y = 0):
// a real contraction over at most 64 basis values per sample, with 8 real columns (two components,
// four degrees) per row, whose right-hand side is the same for every sample of a segment.  That
// is a matrix product, [samples x 64] [64 x 8 rows], and it runs on tcgen05; what is left per
// sample is the basis (powers of z = e^{i theta}), one cubic in u per row and Horner's rule in
// z_phi over the rows: ~600 FP32 operations instead of the ~12,800 of the scalar chain (sum.cu) on
// the 21 x 61 grid.
//
// Precision: both operands are split in two fp16 parts, x = hi + lo (11 significant bits each;
// the table after exact power-of-two scaling of the segment's largest entry into [2^14, 2^15)),
// and the products lo.hi, hi.lo, hi.hi are accumulated in FP32 in tensor memory; the dropped
// lo.lo is below 2^-24 of the term.  Phases are 64-bit fixed-point turns: a cubic in the sample
// number whose coefficients (the FP64 Taylor expansion of the phase splines at the tile's first
// sample) are in units of 2^-64 turn, so that wrap-around arithmetic is the exact reduction modulo
// one turn and z_r^8 and z_r^{n_mid} come from exact integer multiples of the
// phases instead of powers of rounded exponentials.  Measured error against a 64-bit restatement
// over the one-year 3843-mode waveform: 1.7e-7 to 2.9e-7 over seeds (the scalar chain: 2.3e-6).
//
// Work decomposition: tiles of 128 samples (one per tensor-memory lane) that start at multiples of
// 128 within a segment; a persistent CTA per SM takes a contiguous run of tiles.  Four warpgroups
// take its tiles in turn on two slots of accumulator and operand columns in tensor memory.  The
// operand tables of this and the next segment sit in shared memory (bulk copies, two buffers,
// refilled by the last warpgroup to release one).
#include <type_traits>

#include <cuda_fp16.h>

#include "fewsum_internal.h"
#include "convert.cuh"
#include "fold_tc.cuh"
#include "harmonics.cuh"
#include "tctile.cuh"

namespace fewsum {

namespace {

constexpr int kTcGroups = 4;                        // warpgroups
constexpr int kTcThreads = 128 * kTcGroups;
constexpr int kTcDrain = 6;                         // row pairs in registers while draining
constexpr int kTcMaxKs = (kTcMaxHalf + 8) / 8;
constexpr int kTcMaxLm = 31 * kTcMaxPairs;  // (l, m) pairs: 2 <= l <= 32, m <= 10
constexpr int kTcMaxTable = 1024 * kTcMaxPairs * kTcMaxKs;
constexpr uint32_t kTcDStride = 192, kTcECol = 384, kTcEStride = 64, kTcELo = 32;  // tmem columns

__device__ __forceinline__ float pow2(int e) { return __uint_as_float((uint32_t)(127 + e) << 23); }

}  // namespace

// Operand tables and tile records.  Block g < total_segs: segment g's table.  The block computes the
// harmonics (252 of them for l <= 10; they need nothing of the spline build before it), forms the
// cubics, scales by the power of two that brings the table's largest entry into [2^14, 2^15) and packs
// high and low fp16 parts as the MMA reads them (K-major without swizzle: 8 x 16 B core matrices,
// 128 B apart along K; column 16 p + 2 x + e of the product is row 16 p + 2 x + e of the cubics, basis
// value 2 b is cos(b theta), 2 b + 1 sin(b theta)).  The blocks after that fill the tile records (FP64
// work beside the fold's gathers).
// wait: the plan is in the parameters (at a device address it is read after pdl_wait).
__device__ __forceinline__ void fold_tc_block(const PlanHdr &h, bool wait)
{
    extern __shared__ __align__(16) float tcf[];  // cubics, then harmonics
    __shared__ float s_max[kTcFoldThreads / 32];
    const int tid = threadIdx.x;
    if ((int)blockIdx.x >= h.total_segs) {
        if (wait) pdl_wait();
        tc_fill_records<false>(h, reinterpret_cast<SegFill<false> *>(tcf));
        return;
    }
    const WaveDev &W = tc_wave(h, tc_wave_of_seg(h, blockIdx.x));
    const TrajDev &tr = W.tr;
    const int s = (int)blockIdx.x - W.seg_begin;
    const int *tile_off = tc_local(h, W.tile_off);
    const bool any = s < tr.S && tile_off[s] < tile_off[s + 1];  // samples in this segment
    const int P = tr.tc_pairs, ks = tr.tc_ks, ld = fold_stride(ks, sizeof(float));
    float2 *Y = reinterpret_cast<float2 *>(tcf + 16 * P * ld);
    if (any) {
        for (int t = tid; t < 2 * tr.n_pairs; t += blockDim.x) {
            const double2 y = wave_harmonic<float>(W, tr.pair_lm[t >> 1], t & 1);
            Y[t] = make_float2(f64_to_f32_fast(y.x), f64_to_f32_fast(y.y));
        }
    }
    if (wait) pdl_wait();
    if (!any) return;
    __syncthreads();
    fold_rows<float>(tr, s, W.scale, Y, tcf);
    __syncthreads();
    float mx = 0.0f;
    for (int it = tid; it < 16 * P * 8 * ks; it += blockDim.x) {
        float X, Z;
        fold_basis(tcf, ks, it / (8 * ks), it % (8 * ks), X, Z);
        mx = fmaxf(mx, fmaxf(fabsf(X), fabsf(Z)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((tid & 31) == 0) s_max[tid >> 5] = mx;
    __syncthreads();
    mx = 0.0f;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) mx = fmaxf(mx, s_max[w]);
    int e = 0;
    if (mx > 0.0f) e = 14 + 127 - (int)(__float_as_uint(mx) >> 23);
    e = max(-126, min(126, e));
    const float f = pow2(e);
    if (tid == 0) W.tab_inv[s] = pow2(-e);
    unsigned char *hi_dst = W.tab + (size_t)s * tc_table_bytes(P, ks);
    unsigned char *lo_dst = hi_dst + tc_table_bytes(P, ks) / 2;
    const int c8n = 2 * ks;
    for (int id = tid; id < 16 * P * c8n; id += blockDim.x) {  // 16-byte chunks in memory order
        const int r8 = id & 7, g = id >> 3, c8 = g % c8n, r = (g / c8n) * 8 + r8;
        uint32_t wh[4], wl[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float x0, x1;
            fold_basis(tcf, ks, r, 4 * c8 + k, x0, x1);
            x0 *= f;
            x1 *= f;
            const __half2 hi = __floats2half2_rn(x0, x1);
            const float2 hf = __half22float2(hi);
            const __half2 lo = __floats2half2_rn(x0 - hf.x, x1 - hf.y);
            wh[k] = *reinterpret_cast<const uint32_t *>(&hi);
            wl[k] = *reinterpret_cast<const uint32_t *>(&lo);
        }
        reinterpret_cast<uint4 *>(hi_dst)[id] = make_uint4(wh[0], wh[1], wh[2], wh[3]);
        reinterpret_cast<uint4 *>(lo_dst)[id] = make_uint4(wl[0], wl[1], wl[2], wl[3]);
    }
}

__global__ void __launch_bounds__(kTcFoldThreads) k_fold_tc(const PlanHdr *hp)
{
    pdl_wait();
    pdl_launch_dependents();
    fold_tc_block(*hp, false);
}

// The plan in the parameters; the last block copies it to the device for the summation.
__global__ void __launch_bounds__(kTcFoldThreads) k_fold_tc_param(const __grid_constant__ PlanParam plan)
{
    pdl_launch_dependents();
    fold_tc_block(*reinterpret_cast<const PlanHdr *>(plan.bytes), true);
    tc_store_plan(plan);
}

namespace {

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }

// cos and sin of 2 pi f 2^-32, f a 32-bit fixed-point turn: the quadrant is split off exactly, so
// the rest, |t| <= 1/8 turn, is rounded once (2^-28 turn at most); Taylor polynomials in t to t^10
// and t^9 (truncation below 2e-9), the linear coefficient 2 pi in two parts.
__device__ __forceinline__ void sincos_fixed(uint32_t f, float &s, float &c)
{
    const uint32_t q = f + 0x20000000u;
    const float t = (float)(int)(f - (q & 0xc0000000u)) * 2.3283064365386963e-10f;  // 2^-32
    const float t2 = t * t;
    float ps = fmaf(t2, 42.058693f, -76.70586f);
    ps = fmaf(ps, t2, 81.60525f);
    ps = fmaf(ps, t2, -41.3417f);
    ps = fmaf(ps, t2, -1.7484556e-7f);
    ps = fmaf(t, 6.2831855f, ps * t);
    float pc = fmaf(t2, -26.426256f, 60.24464f);
    pc = fmaf(pc, t2, -85.45682f);
    pc = fmaf(pc, t2, 64.93939f);
    pc = fmaf(pc, t2, -19.739208f);
    pc = fmaf(pc, t2, 1.0f);
    const bool swap = (q & 0x40000000u) != 0;
    const float a = swap ? pc : ps, b = swap ? ps : pc;
    s = __uint_as_float(__float_as_uint(a) ^ (q & 0x80000000u));
    c = __uint_as_float(__float_as_uint(b) ^ ((q + 0x40000000u) & 0x80000000u));
}

// Eight powers (cos, sin), two to a float2, as packed fp16 high and low parts: word k holds
// (cos, sin) of power k.
__device__ __forceinline__ void split_powers(const float2 (&c)[4], const float2 (&s)[4],
                                             uint32_t (&vh)[8], uint32_t (&vl)[8])
{
    const float2 neg = both(-1.0f);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const __half2 h0 = __floats2half2_rn(c[k].x, s[k].x), h1 = __floats2half2_rn(c[k].y, s[k].y);
        const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
        const float2 lc = fma2(make_float2(f0.x, f1.x), neg, c[k]);
        const float2 ls = fma2(make_float2(f0.y, f1.y), neg, s[k]);
        const __half2 l0 = __floats2half2_rn(lc.x, ls.x), l1 = __floats2half2_rn(lc.y, ls.y);
        vh[2 * k] = *reinterpret_cast<const uint32_t *>(&h0);
        vh[2 * k + 1] = *reinterpret_cast<const uint32_t *>(&h1);
        vl[2 * k] = *reinterpret_cast<const uint32_t *>(&l0);
        vl[2 * k + 1] = *reinterpret_cast<const uint32_t *>(&l1);
    }
}

// (c, s) <- (ac, as) (bc, bs), two complex products at once.
__device__ __forceinline__ void cmul2(float2 ac, float2 as, float2 bc, float2 bs, float2 &c, float2 &s)
{
    const float2 nbs = make_float2(-bs.x, -bs.y);
    c = fma2(ac, bc, mul2(as, nbs));
    s = fma2(ac, bs, mul2(as, bc));
}

// Powers 0 .. 7 of z = e^{2 pi i f}, f the top 32 bits of a fixed-point phase.
__device__ __forceinline__ void first_powers(unsigned long long f, float2 (&c)[4], float2 (&s)[4])
{
    float s1, c1;
    sincos_fixed((uint32_t)(f >> 32), s1, c1);
    const float c2 = fmaf(c1, c1, -s1 * s1), s2 = 2.0f * (c1 * s1);
    c[0] = make_float2(1.0f, c1);
    s[0] = make_float2(0.0f, s1);
    cmul2(c[0], s[0], both(c2), both(s2), c[1], s[1]);              // 2, 3
    const float c4 = fmaf(c2, c2, -s2 * s2), s4 = 2.0f * (c2 * s2);
    cmul2(c[0], s[0], both(c4), both(s4), c[2], s[2]);              // 4, 5
    cmul2(c[1], s[1], both(c4), both(s4), c[3], s[3]);              // 6, 7
}

}  // namespace

// Starts the copy of table `n` of the CTA's run (first tile T) into its buffer (one thread).
__device__ __forceinline__ void load_table(const TileRec *recs, int T, int n,
                                           unsigned char *buf, uint64_t *full)
{
    const TileRec *r = recs + T;
    const uint32_t bytes = (uint32_t)tc_table_bytes(r->pairs, r->ks);
    const unsigned char *src = r->tab;
    mbar_arrive_expect_tx(&full[n & 1], bytes);
    for (uint32_t o = 0; o < bytes; o += 16384u)
        bulk_g2s(buf + (n & 1) * kTcMaxTable + o, src + o, min(16384u, bytes - o), &full[n & 1]);
}

// Warpgroup k takes every fourth tile of the CTA's run, on slot k & 1 of tensor memory (operand and
// accumulator columns).  A tile's operand columns are free when the slot's previous MMAs have
// completed, its accumulator when the slot's previous tile has been drained; a warpgroup forms
// its basis in registers while the slot's other warpgroup waits for its MMAs, and stores it while
// that one drains them.
// KS: K steps of the plan's widest n range (a wave with fewer uses the first of them).
// One year, 3843 modes: 109-111 us a launch, 104 from the first CTA's start to the last one's end (the scalar
// chain 1,417), 1,154 cycles a tile = twelve N = 176 MMAs of 96,
// the tensor cores 90 % active.  Sets of fewer rows run at 430 to 700 ns a tile whatever their size:
// there the chain of a slot bounds it (issue ~900 cycles, the MMAs' tail ~440, loads to the release
// of the accumulator ~500, wake-up ~350).  Six warpgroups of 80 registers: 133 us; factors before
// the issue: 122; MMAs in tile order by a token: 114.
template <int KS>
__global__ void __launch_bounds__(kTcThreads, 1) k_sum_tc(const PlanHdr *hp)
{
    extern __shared__ __align__(128) unsigned char tcs[];  // two operand tables
    __shared__ __align__(8) uint64_t b_full[2], d_full[2], d_free[2];
    __shared__ int b_left[2];  // warpgroups that still need the table in the buffer
    __shared__ int s_loaded;   // tables whose copies have been started
    __shared__ __align__(16) uint32_t s_rec[4 * kTcGroups][32];  // each warp's tile record
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_abort;
    pdl_wait();
    pdl_launch_dependents();
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform
    const TileRec *recs = hp->recs;
    const int T0 = hp->tile_cta[blockIdx.x], T1 = hp->tile_cta[blockIdx.x + 1];
    if (T0 >= T1) return;  // uniform across the CTA: no work
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_slot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 32) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&b_full[b], 1);
            mbar_init(&d_full[b], 1);
            mbar_init(&d_free[b], 4);
            b_left[b] = kTcGroups;
        }
        fence_mbar_init();
        s_abort = 0;
        load_table(recs, T0, 0, tcs, b_full);
        const int next = recs[T0].tile_end;
        if (next < T1) load_table(recs, next, 1, tcs, b_full);
        s_loaded = next < T1 ? 2 : 1;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const int group = warp >> 2, slot = group & 1, lane = tid & 127;
    const bool lead = lane == 0;
    const uint32_t quarter = (uint32_t)(32 * (warp & 3)) << 16;
    const uint32_t d_col = tmem + (uint32_t)slot * kTcDStride;
    const uint32_t e_col = tmem + kTcECol + (uint32_t)slot * kTcEStride;
    int j = 0, tend = recs[T0].tile_end;  // table of the current tile, and where it ends
    bool bad = false;
    // This warpgroup's MMAs on table j have completed: release it (lead), and let the last of the
    // warpgroups refill its buffer.  A table is released only once it has landed (also one that the
    // warpgroup had no tile in): its buffer's previous table has then been released by every
    // warpgroup, so neither the count nor a parity wait can be taken for the previous table's.
    auto release_table = [&]() {
        const int next = recs[tend].tile_end;  // end of table j + 1, first tile of j + 2
        if (lead && !bad) {
            if (!mbar_wait_bounded(&b_full[j & 1], (j >> 1) & 1)) {
                bad = true;
            } else if (__threadfence_block(), atomicSub(&b_left[j & 1], 1) == 1) {
                __threadfence_block();
                b_left[j & 1] = kTcGroups;
                if (next < T1) {
                    s_loaded = j + 3;
                    load_table(recs, next, j, tcs, b_full);  // table j + 2, the same buffer
                }
            }
        }
        ++j;
        tend = next;
    };
    // a warp fetches the next tile's record a word a lane while its MMAs run, and reads it from its
    // own line of shared memory
    const TileRec *rp = reinterpret_cast<const TileRec *>(s_rec[warp]);
    uint32_t next_word = 0;
    if (T0 + group < T1) next_word = reinterpret_cast<const uint32_t *>(recs + T0 + group)[tid & 31];
#pragma unroll 1
    for (int T = T0 + group; T < T1; T += kTcGroups) {
        s_rec[warp][tid & 31] = next_word;
        while (T >= tend) release_table();
        __syncwarp();
        const uint32_t use = (uint32_t)(T - T0) >> 1;  // of the slot
        const int4 span = *reinterpret_cast<const int4 *>(&rp->i0);      // i0, s0, s1
        const int4 shape = *reinterpret_cast<const int4 *>(&rp->pairs);  // pairs, ks, n_mid, c64
        const int pairs = shape.x, ks = shape.y;
        const int i = span.x + lane;
        const uint32_t v = (uint32_t)max(i - max(span.x, span.y), 0);
        const unsigned long long fr = phase_fixed(rp->r, v), fphi = phase_fixed(rp->phi, v);
        // the basis: powers 0 .. 8 ks - 1, eight at a time, z and z^8 from the phase itself, held
        // in registers until the slot's operand columns are free
        uint32_t vh[KS][8], vl[KS][8];
        {
            float2 c[4], s[4];
            first_powers(fr, c, s);
            split_powers(c, s, vh[0], vl[0]);
            if (KS > 1) {
                float bs, bc;
                sincos_fixed((uint32_t)((8 * fr) >> 32), bs, bc);
                const float2 BC = both(bc), BS = both(bs);
                float2 gc = BC, gs = BS;  // z^(8 a), in both halves
#pragma unroll
                for (int a = 1; a < KS; ++a) {
                    float2 pc[4], ps[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) cmul2(c[k], s[k], gc, gs, pc[k], ps[k]);
                    split_powers(pc, ps, vh[a], vl[a]);
                    if (a + 1 < KS) {
                        float2 nc, ns;
                        cmul2(gc, gs, BC, BS, nc, ns);
                        gc = nc;
                        gs = ns;
                    }
                }
            }
        }
        if (use > 0 && !mbar_wait_bounded(&d_full[slot], (use - 1) & 1)) bad = true;
        __syncwarp();
        tc_fence_after();
#pragma unroll
        for (int a = 0; a < KS; ++a) {
            tc_st8(e_col + quarter + 8 * a, vh[a]);
            tc_st8(e_col + quarter + kTcELo + 8 * a, vl[a]);
        }
        tc_wait_st();
        tc_fence_before();
        bad = wg_any(1 + group, bad);
        if (bad) break;
        if ((warp & 3) == 0) {  // the warpgroup's first warp issues the MMAs
            const bool ok = (use == 0 || mbar_wait_bounded(&d_free[slot], (use - 1) & 1)) &&
                            mbar_wait_bounded(&b_full[j & 1], (j >> 1) & 1);
            if (__all_sync(0xffffffffu, ok)) {
                tc_fence_after();
                const int up = __shfl_sync(0xffffffffu, pairs, 0), uk = __shfl_sync(0xffffffffu, ks, 0);
                const uint32_t b_hi = smem_u32(tcs) + (uint32_t)(j & 1) * kTcMaxTable;
                const uint32_t b_lo = b_hi + (uint32_t)tc_table_bytes(up, uk) / 2;
                const uint32_t idesc =
                    (1u << 4) | ((uint32_t)(2 * up) << 17) | ((uint32_t)(kTcTile >> 4) << 24);
                const uint64_t d_hi = smem_desc(b_hi, 128, 256u * (uint32_t)uk);
                const uint64_t d_lo = smem_desc(b_lo, 128, 256u * (uint32_t)uk);
                if (elect_one()) {
                    for (int a = 0; a < uk; ++a) {  // the small products first; 256 B per K step
                        tc_mma_ta(d_col, e_col + kTcELo + 8 * a, d_hi + 16 * a, idesc, a != 0);
                        tc_mma_ta(d_col, e_col + 8 * a, d_lo + 16 * a, idesc, 1);
                    }
                    for (int a = 0; a < uk; ++a) tc_mma_ta(d_col, e_col + 8 * a, d_hi + 16 * a, idesc, 1);
                    tc_commit(&d_full[slot]);
                }
                __syncwarp();
            } else {
                s_abort = 1;
            }
        }
        // while the MMAs run: this sample's factors
        const float2 uu = *reinterpret_cast<const float2 *>(&rp->u0);
        const float inv = *static_cast<const float *>(rp->seg);
        void *out = rp->out;
        if (T + kTcGroups < T1)
            next_word = reinterpret_cast<const uint32_t *>(recs + T + kTcGroups)[tid & 31];
        const float u = fmaf((float)(i - span.y), uu.y, uu.x);
        float zs, zc;
        sincos_fixed((uint32_t)(fphi >> 32), zs, zc);
        float fs = 0.0f, fc = inv;  // z_r^{n_mid} over the table's scale
        if (shape.z != 0) {
            sincos_fixed((uint32_t)(((unsigned long long)(long long)shape.z * fr) >> 32), fs, fc);
            fs *= inv;
            fc *= inv;
        }
        const float2 U = both(u), U2 = both(u * u);
        // rows m = m_top - p and p - m_top: Horner in z_phi and in its conjugate
        const float2 WR = both(zc), WI = make_float2(-zs, zs), NWI = make_float2(zs, -zs);
        float2 tr = both(0.0f), ti = tr;
        if (!mbar_wait_bounded(&d_full[slot], use & 1)) {
            s_abort = 1;
            bad = true;
        }
        __syncwarp();
        tc_fence_after();
        auto row_pair = [&](const float(&d)[16]) {
            const float2 *k = reinterpret_cast<const float2 *>(d);
            const float2 kr = fma2(fma2(k[3], U, k[2]), U2, fma2(k[1], U, k[0]));
            const float2 ki = fma2(fma2(k[7], U, k[6]), U2, fma2(k[5], U, k[4]));
            const float2 nr = fma2(ti, NWI, fma2(tr, WR, kr));
            const float2 ni = fma2(ti, WR, fma2(tr, WI, ki));
            tr = nr;
            ti = ni;
        };
        // six row pairs' loads in flight, then each pair's registers reloaded once it is used, so
        // that the accumulator is free before the second half is computed (columns past the last
        // pair belong to the slot and are not used)
        const uint32_t d_lane = d_col + quarter;
        auto drain = [&](auto full) {  // full: every pair of the accumulator is in use
            float d[kTcDrain][16];
#pragma unroll
            for (int q = 0; q < kTcDrain; ++q) tc_ld16(d_lane + 16 * q, d[q]);
            tc_wait_ld16(d[0]);
#pragma unroll
            for (int q = 1; q < kTcDrain; ++q) tc_landed16(d[q]);
#pragma unroll
            for (int q = 0; q < kTcDrain; ++q) {
                if (decltype(full)::value || q < pairs) row_pair(d[q]);
                if (q + kTcDrain < kTcMaxPairs) tc_ld16(d_lane + 16 * (q + kTcDrain), d[q]);
            }
            tc_wait_ld16(d[0]);
#pragma unroll
            for (int q = 1; q < kTcMaxPairs - kTcDrain; ++q) tc_landed16(d[q]);
            tc_fence_before();
            __syncwarp();
            if ((tid & 31) == 0) mbar_arrive(&d_free[slot]);
#pragma unroll
            for (int q = kTcDrain; q < kTcMaxPairs; ++q)
                if (decltype(full)::value || q < pairs) row_pair(d[q - kTcDrain]);
        };
        if (pairs == kTcMaxPairs)
            drain(std::true_type());
        else
            drain(std::false_type());
        if (i >= span.y && i < span.z) {
            const float hr = tr.x + tr.y, hi = ti.x + ti.y;
            const float yr = fmaf(hr, fc, hi * fs), yi = fmaf(hi, fc, -hr * fs);
            if (shape.w)
                reinterpret_cast<float2 *>(out)[i] = make_float2(yr, yi);
            else
                reinterpret_cast<double2 *>(out)[i] = make_double2((double)yr, (double)yi);
        }
    }
    while (tend < T1 && !bad) release_table();  // tables that only other warpgroups still need
    if (lead && bad) s_abort = 1;
    __syncthreads();
    if (tid == 0 && s_abort) {
        atomicOr(hp->err, ERRBIT_TIMEOUT);
        // no copy may land after the CTA's shared memory is gone
        for (int n = max(s_loaded - 2, 0); n < s_loaded; ++n) mbar_wait_bounded(&b_full[n & 1], (n >> 1) & 1);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

namespace {
using TcKernel = void (*)(const PlanHdr *);
// cubics and harmonics of a fold block
constexpr int kFoldSmem =
    (16 * kTcMaxPairs * fold_stride(kTcMaxKs, sizeof(float)) + 4 * kTcMaxLm) * (int)sizeof(float);
const TcKernel kTcKernels[kTcMaxKs] = {k_sum_tc<1>, k_sum_tc<2>, k_sum_tc<3>, k_sum_tc<4>};
}  // namespace

cudaError_t tc_configure()
{
    for (TcKernel k : kTcKernels) {
        const cudaError_t e =
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kTcMaxTable);
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = cudaFuncSetAttribute(k_fold_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kFoldSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_fold_tc_param, cudaFuncAttributeMaxDynamicSharedMemorySize, kFoldSmem);
    return e;
}

cudaError_t launch_fold_tc(const PlanHdr *hdr_dev, const PlanParam *plan, int total_segs, int total_tiles,
                           int sm_count, cudaStream_t st)
{
    if (total_tiles <= 0) return cudaSuccess;
    const unsigned grid = total_segs + tc_record_blocks(total_tiles, 0, sm_count);
    // More segments than multiprocessors: blocks of half the threads, two a multiprocessor, so that one
    // loads while the other packs (24 uneven waveforms, 2,400 segments: 3.17 -> 2.99 ms with the records'
    // share of that); else a thread a frequency, for the latency of the one block.
    const unsigned threads = total_segs > sm_count ? kTcFoldThreads / 2 : kTcFoldThreads;
    if (plan) return launch_pdl(k_fold_tc_param, grid, threads, kFoldSmem, st, *plan);
    return launch_pdl(k_fold_tc, grid, threads, kFoldSmem, st, hdr_dev);
}

cudaError_t launch_sum_tc(const PlanHdr *hdr_dev, int grid, int ks, cudaStream_t st)
{
    if (grid <= 0) return cudaSuccess;
    if (ks < 1 || ks > kTcMaxKs) return cudaErrorInvalidValue;
    return launch_pdl(kTcKernels[ks - 1], grid, kTcThreads, 2 * kTcMaxTable, st, hdr_dev);
}

}  // namespace fewsum
