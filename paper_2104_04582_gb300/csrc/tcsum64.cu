// tcsum64.cu -- the FP64 mode sum on the tensor cores, in exact integer arithmetic (arXiv:2104.04582
// Sec. 3.C, Sec. 4).
//
// The contraction is the one of tcsum.cu: per segment a real product [samples x 16 ks] [16 ks x 8
// columns per row] of the basis cos(b theta), sin(b theta) with the folded cubics' coefficients.
// The chip's FP64 pipe does two FMA a cycle and SM, 1/2000 of the tensor cores' rate, and bounded the
// scalar chain (10 FMA per slot and sample); here it evaluates u and scales the output only.
//
// Both operands are fixed-point numbers of 7 signed 8-bit digits (units of 2^-54; the table scaled
// by the power of two that brings its largest entry into [1/2, 1)), held as fp16 integers.  The
// products of digits i and j with i + j = o <= 6 are summed in accumulator o: at most 63 x 98304
// < 2^23 (order_bound), so the FP32 accumulators are exact integers.  What is left out (o >= 7) and the operands'
// rounding are below 2^-50 of the table's largest entry, as is FP64's own rounding of such a sum.
// The accumulators are put together as 64-bit integers, and the cubic in u and Horner's rules in
// z_phi and its conjugate run in 64-bit fixed point too (a product costs ~6 instructions; an FP64
// operation holds a scheduler's share of the pipe for 64 cycles).  Powers of z_r and sincos are 62-bit fixed point
// (Taylor series); phases as in tcsum.cu.
//
// Work decomposition: as tcsum.cu, tiles of 128 samples, a persistent CTA per SM.  The segment's
// table (up to 158 KB) stays in shared memory.  Tensor memory holds one tile's basis digits (7 x 32
// columns) and two accumulator sets of one row pair (7 x 16 columns each): the MMAs of one pair run
// while the previous pair's sums are formed.  Two warpgroups take the tiles in turn; one prepares its
// exponentials while the other's MMAs run.
// One year, 3843 modes: 1.89 ms (the scalar chain 66.6), ~22,000 cycles a tile: 13,000 of MMAs (tensor cores
// 44 % active), the rest the forming of sums, ~1,700 a row pair by one warp a scheduler (issue 47 %).
// Both warpgroups on every tile (half of the rows each): 2.03 ms.  Error against 64-bit phases 1.6e-13
// to 2.4e-13 over seeds (the scalar chain 3.5e-13 to 4.0e-13).
#include <cuda_fp16.h>

#include "fewsum_internal.h"
#include "fold_tc.cuh"
#include "tctile.cuh"

namespace fewsum {

namespace {

constexpr int kT64FoldThreads = 352;  // FP64 fold: registers for a thread's two cubics
constexpr int kT64Groups = 2, kT64Issuers = 2;
constexpr int kT64Threads = 128 * kT64Groups + 32 * kT64Issuers;  // and the MMAs' warps
constexpr int kT64MaxKs = (kTcMaxHalf + 8) / 8;
constexpr int kT64MaxTable = 512 * kTc64Slices * kTcMaxPairs * kT64MaxKs;
constexpr uint32_t kT64EStride = 32;                    // tensor-memory columns of a digit slice
constexpr uint32_t kT64DCol = kTc64Slices * kT64EStride;  // two accumulator sets follow the digits
constexpr uint32_t kT64DStride = 16 * kTc64Slices;

__device__ __forceinline__ double pow2d(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// The 7 digits of x (a multiple of 2^-54, |x| <= 1) as unsigned bytes digit + 128, least
// significant first.
__device__ __forceinline__ unsigned long long digit_bytes(long long x)
{
    return (unsigned long long)x + 0x0080808080808080ull;
}

// fp16 integer digits of two numbers from byte k of each: (0x64 byte) is 1024 + byte.
__device__ __forceinline__ uint32_t digit_pair(uint32_t word, uint32_t sel)
{
    const uint32_t w = __byte_perm(word, 0x64646464u, sel);
    const __half2 d = __hsub2(*reinterpret_cast<const __half2 *>(&w), __floats2half2_rn(1152.0f, 1152.0f));
    return *reinterpret_cast<const uint32_t *>(&d);
}

}  // namespace

// Operand tables (block per segment) and tile records, as fold_tc_block, in FP64 (the harmonics by
// k_ylm: in FP64 their latency is too long to be repeated in every block).  Chunk p of a table is row
// pair p: 7 digit slices (most significant first) of 16 rows each.
__device__ __forceinline__ void fold_tc64_block(const PlanHdr &h)
{
    extern __shared__ __align__(16) double tcf64[];
    __shared__ double s_max[kT64FoldThreads / 32], s_sum[kT64FoldThreads / 32];
    const int tid = threadIdx.x;
    pdl_wait();
    if ((int)blockIdx.x >= h.total_segs) {
        tc_fill_records<true>(h, reinterpret_cast<SegFill<true> *>(tcf64));
        return;
    }
    const WaveDev &W = tc_wave(h, tc_wave_of_seg(h, blockIdx.x));
    const TrajDev &tr = W.tr;
    const int s = (int)blockIdx.x - W.seg_begin;
    const int *tile_off = tc_local(h, W.tile_off);
    if (s >= tr.S || tile_off[s] == tile_off[s + 1]) return;  // no sample in this segment
    const int P = tr.tc_pairs, ks = tr.tc_ks;
    const double *cs = tr.coef + (size_t)s * tr.J * 4;
    fold_rows<double>(tr, s, W.scale, W.ylm, tcf64);
    __syncthreads();
    double mx = 0.0, sum = 0.0;
    for (int it = tid; it < 16 * P * 8 * ks; it += blockDim.x) {
        double X, Z;
        fold_basis(tcf64, ks, it / (8 * ks), it % (8 * ks), X, Z);
        X = fabs(X);
        Z = fabs(Z);
        mx = fmax(mx, fmax(X, Z));
        sum += 9.5367431640625e-7 * (X + Z);  // 2^-20: no overflow
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    if ((tid & 31) == 0) {
        s_max[tid >> 5] = mx;
        s_sum[tid >> 5] = sum;
    }
    __syncthreads();
    mx = sum = 0.0;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) {
        mx = fmax(mx, s_max[w]);
        sum += s_sum[w];
    }
    // e: mx 2^e in [1/2, 1); 2^e in two factors, each a normal number
    int e = 0;
    if (mx > 0.0) e = 1022 - (int)((unsigned)__double2hiint(mx) >> 20);
    const double f1 = pow2d(e / 2), f2 = pow2d(e - e / 2);
    if (tid == 0) {
        TcSeg64 g;
        // the digit sums come out in units of 2^-52 of the scaled table; every partial sum of a
        // sample is at most l1
        const double l1 = sum * f1 * f2 * 1048576.0;
        int up = 14;  // l1 < 2^up (sums too small to be added up: as many entries as there are)
        if (l1 >= 0.5) up = (int)((unsigned)__double2hiint(l1) >> 20) - 1022;
        // (sums of one row have two guard bits, 2^-54, and stay below 2^62; the rows' total is kept
        // below 2^61)
        g.shift = max(0, min(32, up - 7));
        const int x = -e - 54 + g.shift;  // 2^x: one unit of the shifted sums
        g.inv1 = pow2d(x / 2);
        // non-finite data (latched by the build) reach the output
        double all = sum - sum;
        for (int k = 0; k < 8; ++k) all += cs[k] - cs[k];  // the two phases
        g.inv1 += all;
        g.inv2 = pow2d(x - x / 2);
        g.tk = tr.t[s];
        g.ih = tr.inv_h[s];
        g.t0 = W.t0;
        g.dt = W.dt;
        W.seg64[s] = g;
    }
    unsigned char *tab = W.tab + (size_t)s * tc64_table_bytes(P, ks);
    const int c8n = 2 * ks, slice = 512 * ks;  // bytes of one slice of one pair
    for (int id = tid; id < 16 * P * c8n; id += blockDim.x) {  // 16-byte chunks in memory order
        const int r8 = id & 7, g = id >> 3, c8 = g % c8n, r = (g / c8n) * 8 + r8;  // row 0 .. 16 P - 1
        unsigned long long v[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            double X, Z;
            fold_basis(tcf64, ks, r, 4 * c8 + k, X, Z);
            v[2 * k] = digit_bytes(__double2ll_rn(X * f1 * f2 * 18014398509481984.0));
            v[2 * k + 1] = digit_bytes(__double2ll_rn(Z * f1 * f2 * 18014398509481984.0));
        }
        unsigned char *dst = tab + (size_t)(r >> 4) * kTc64Slices * slice + ((r >> 3) & 1) * 256 * ks +
                             c8 * 128 + r8 * 16;
#pragma unroll
        for (int q = 0; q < kTc64Slices; ++q) {  // slice q: byte 6 - q
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t b0 = (uint32_t)(v[2 * k] >> (8 * (6 - q))) & 255u;
                const uint32_t b1 = (uint32_t)(v[2 * k + 1] >> (8 * (6 - q))) & 255u;
                w[k] = digit_pair(b0 | (b1 << 8), 0x4140);
            }
            *reinterpret_cast<uint4 *>(dst + (size_t)q * slice) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

__global__ void __launch_bounds__(kT64FoldThreads) k_fold_tc64(const PlanHdr *hp)
{
    pdl_launch_dependents();
    fold_tc64_block(*hp);
}

namespace {

// 62-bit fixed point in balanced halves: value = h 2^32 + l, l signed.  A product then takes three
// 32 x 32 -> 64-bit multiply-adds (the low halves' product, below half a unit of 2^-60, is left
// out), against ~25 instructions for a 128-bit product.
struct Q62 {
    int h, l;
};
__device__ __forceinline__ Q62 q62(long long v)
{
    const int l = (int)v;
    return Q62{(int)(v >> 32) - (l >> 31), l};
}
__device__ __forceinline__ long long value(const Q62 &a) { return ((long long)a.h << 32) + a.l; }
// a b + c, one instruction (written out: from C++ the products came out unsigned with corrections)
__device__ __forceinline__ long long wide(int a, int b, long long c)
{
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}

// a b 2^-64, rounded; |a|, |b| <= 2^62.
__device__ __forceinline__ long long mul_hi(const Q62 &a, const Q62 &b)
{
    const long long t = wide(a.h, b.l, wide(a.l, b.h, 0x80000000ll));
    return wide(a.h, b.h, t >> 32);
}
__device__ __forceinline__ long long mul62(const Q62 &a, const Q62 &b) { return mul_hi(a, b) << 2; }

struct Cq {  // complex
    Q62 c, s;
};

// (c, s) of a b in 62-bit fixed point, |a| = |b| = 1.
__device__ __forceinline__ Cq cmul(const Cq &a, const Cq &b)
{
    const long long t = wide(a.c.h, b.c.l, wide(a.c.l, b.c.h, 0x80000000ll));
    const long long v = wide(a.s.h, b.s.l, wide(a.s.l, b.s.h, 0));
    const long long re = wide(a.c.h, b.c.h, (t - v) >> 32) - wide(a.s.h, b.s.h, 0);
    const long long w = wide(a.c.h, b.s.l, wide(a.c.l, b.s.h, wide(a.s.h, b.c.l, wide(a.s.l, b.c.h, 0x80000000ll))));
    const long long im = wide(a.c.h, b.s.h, wide(a.s.h, b.c.h, w >> 32));
    return Cq{q62(re << 2), q62(im << 2)};
}

// cos and sin of 2 pi f 2^-64 in 62-bit fixed point: quadrant split off exactly, Taylor series to
// x^16 and x^17 on |x| <= pi/4 (truncation 2e-18).
__device__ __forceinline__ Cq sincos62(unsigned long long f)
{
    const unsigned long long q = f + 0x2000000000000000ull;
    const long long r = (long long)(f - (q & 0xc000000000000000ull));
    const long long one = 1ll << 62;
    const Q62 x = q62(mul62(q62(r), q62(7244019458077122842ll)));  // pi/2 2^62: r 2 pi 2^-64 in 2^-62
    const Q62 x2 = q62(mul62(x, x));
    auto step = [&](long long p, long long k) { return mul62(x2, q62(p)) + k; };
    // 2^62 / n!, rounded
    long long p = step(12966ll, -3526632ll);     // 17!, 15!
    p = step(p, 740592679ll);                    // 13!
    p = step(p, -115532457973ll);                // 11!
    p = step(p, 12708570377060ll);               // 9!
    p = step(p, -915017067148291ll);             // 7!
    p = step(p, 38430716820228233ll);            // 5!
    p = step(p, -768614336404564651ll);          // 3!
    const long long sn = value(x) + mul62(x, q62(mul62(x2, q62(p))));
    long long c = step(220414ll, -52899477ll);   // 16!, 14!
    c = step(c, 9627704831ll);                   // 12!
    c = step(c, -1270857037706ll);               // 10!
    c = step(c, 114377133393536ll);              // 8!
    c = step(c, -6405119470038039ll);            // 6!
    c = step(c, 192153584101141163ll);           // 4!
    c = step(c, -(one >> 1));                    // 2!
    const long long cs = one + mul62(x2, q62(c));
    const bool swap = (q >> 62) & 1;
    const long long a = swap ? cs : sn, b = swap ? sn : cs;
    const bool ns = (q >> 63) & 1, nc = ((q + 0x4000000000000000ull) >> 63) & 1;
    return Cq{q62(nc ? -b : b), q62(ns ? -a : a)};
}

// The digits of one power into column `col` of every slice (this thread's lane).
__device__ __forceinline__ void digit_words(const Cq &z, uint32_t (&w)[kTc64Slices])
{
    // 62-bit -> multiples of 2^-54, rounded
    const unsigned long long c = digit_bytes((value(z.c) + 128) >> 8), s = digit_bytes((value(z.s) + 128) >> 8);
    const uint32_t cl = (uint32_t)c, ch = (uint32_t)(c >> 32), sl = (uint32_t)s, sh = (uint32_t)(s >> 32);
    const uint32_t a = __byte_perm(cl, sl, 0x5140), b = __byte_perm(cl, sl, 0x7362);  // bytes 0 1, 2 3
    const uint32_t d = __byte_perm(ch, sh, 0x5140), g = __byte_perm(ch, sh, 0x7362);  // bytes 4 5, 6
    w[6] = digit_pair(a, 0x4140);
    w[5] = digit_pair(a, 0x4342);
    w[4] = digit_pair(b, 0x4140);
    w[3] = digit_pair(b, 0x4342);
    w[2] = digit_pair(d, 0x4140);
    w[1] = digit_pair(d, 0x4342);
    w[0] = digit_pair(g, 0x4140);
}

__device__ __forceinline__ void store_digits(uint32_t e_addr, const Cq (&z)[8])
{
    uint32_t w[kTc64Slices][8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        uint32_t v[kTc64Slices];
        digit_words(z[k], v);
#pragma unroll
        for (int q = 0; q < kTc64Slices; ++q) w[q][k] = v[q];
    }
#pragma unroll
    for (int q = 0; q < kTc64Slices; ++q) tc_st8(e_addr + kT64EStride * q, w[q]);
}

// Largest magnitude of accumulator o: the basis has 2 kTcMaxHalf + 1 values (sin 0 is left out), digits are at most
// 128, and the top ones at most 64, because neither operand exceeds 1 = 64 x 2^48 units of 2^-54 (the table by
// its scale, the basis as a cosine or sine).  join_orders relies on both bounds; the first holds by 1.6 %.
constexpr int order_bound(int o)
{
    return (2 * kTcMaxHalf + 1) * (o == 0 ? 64 * 64 : 2 * 64 * 128 + (o - 1) * 128 * 128);
}
static_assert(kTc64Slices == 7 && order_bound(4) < 1 << 22, "orders 0 .. 4 stay in 1.5 2^23's low mantissa bits");
static_assert(order_bound(kTc64Slices - 1) < 1 << 23, "the FP32 accumulators are exact integers");

// The sums of one column pair (even, odd row), orders 0 .. 6, as 64-bit integers 4 sum_o S_o
// 2^(40 - 8 o) (two guard bits): orders 0 .. 4 exact (|S_o| < 2^22: the 1.5 2^23 addition leaves the
// integer in the low mantissa bits), orders 5 and 6 to a unit.  S: orders 16 columns apart.
__device__ __forceinline__ void join_orders(const float2 (&S)[kTc64Slices], long long (&v)[2])
{
    const float2 kM = make_float2(12582912.0f, 12582912.0f), kNM = make_float2(-12582912.0f, -12582912.0f);
    const float2 k256 = make_float2(0.00390625f, 0.00390625f), kN256 = make_float2(-256.0f, -256.0f);
    const uint32_t kMi = 0x4b400000u;
    // (an opaque copy: from __float_as_uint of the packed sums nvcc 13.0 drops the shift of n4c below
    // for the even column)
    auto bits = [](float x) {
        uint32_t u;
        asm("mov.b32 %0, %1;" : "=r"(u) : "f"(x));
        return u;
    };
    const float2 t = __ffma2_rn(S[6], k256, S[5]);
    const float2 cm = __ffma2_rn(t, k256, kM);
    const float2 rest = __fadd2_rn(__ffma2_rn(__fadd2_rn(cm, kNM), kN256, t), kM);
    const float2 n0 = __fadd2_rn(S[0], kM), n1 = __fadd2_rn(S[1], kM), n2 = __fadd2_rn(S[2], kM);
    const float2 n3 = __fadd2_rn(S[3], kM), n4 = __fadd2_rn(S[4], kM);
    auto join = [&](float a0, float a1, float a2, float a3, float a4, float c, float a5) {
        const uint32_t p1 = (bits(a0) << 8) + (bits(a1) - (kMi << 8) - kMi);
        const uint32_t p2 = (bits(a2) << 8) + (bits(a3) - (kMi << 8) - kMi);
        const uint32_t n4c = bits(a4) - kMi + (bits(c) - kMi);
        const uint32_t p3 = (n4c << 8) + (bits(a5) - kMi);
        return wide((int)p2, 1 << 18, wide((int)p3, 4, (long long)((unsigned long long)p1 << 34)));
    };
    v[0] = join(n0.x, n1.x, n2.x, n3.x, n4.x, cm.x, rest.x);
    v[1] = join(n0.y, n1.y, n2.y, n3.y, n4.y, cm.y, rest.y);
}

__device__ __forceinline__ bool warp_ok(bool ok) { return __all_sync(0xffffffffu, ok); }

// Half of the MMAs of one row pair (one elected thread): accumulator o sums the products of digits q
// of the basis and o - q of the table.  Issuer 0 takes orders 1 .. 4, issuer 1 orders 0, 5 and 6 (14
// products each): one warp issues an N = 16 MMA every ~13 cycles, two together one every 10.6.
// Everything but three bases is a compile-time offset: with run-time loops the uniform datapath's
// address arithmetic took ~50 cycles an MMA.
template <int KS, int ISSUER>
__device__ __forceinline__ void issue_half(uint32_t d, uint32_t e, uint64_t desc)
{
    constexpr uint32_t idesc = (1u << 4) | (2u << 17) | ((uint32_t)(kTcTile >> 4) << 24);
    constexpr uint32_t slice = 512u * KS;
#pragma unroll
    for (int o = 0; o < kTc64Slices; ++o) {
        if ((o >= 1 && o <= 4) != (ISSUER == 0)) continue;
#pragma unroll
        for (int q = 0; q <= o; ++q) {
#pragma unroll
            for (int a = 0; a < KS; ++a)
                tc_mma_ta(d + 16 * o, e + kT64EStride * q + 8 * a,
                          desc + (uint64_t)((o - q) * (slice >> 4) + 16 * a), idesc, (q | a) != 0);
        }
    }
}
template <int KS>
__device__ __forceinline__ void issue_pair(int issuer, uint32_t d, uint32_t e, uint64_t desc)
{
    if (issuer == 0)
        issue_half<KS, 0>(d, e, desc);
    else
        issue_half<KS, 1>(d, e, desc);
}

}  // namespace

// Warps 0 - 7: two warpgroups, every other tile of the CTA's run each.  Warps 8 and 9 issue the MMAs,
// tile by tile and row pair by row pair (half of each), warp 8 loads the tables.  Barriers (chunk = row pair, counted over
// the run): e_full[g] the basis of group g's tile is stored; done[g] its MMAs have completed (the
// operand columns are free); d_full[b], d_empty[b] accumulator set b = chunk & 1.
template <int KS>
__global__ void __launch_bounds__(kT64Threads, 1) k_sum_tc64(const PlanHdr *hp)
{
    extern __shared__ __align__(128) unsigned char tcs64[];  // the operand table
    __shared__ __align__(8) uint64_t b_full, d_full[2], d_empty[2], e_full[kT64Groups], done[kT64Groups];
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
        mbar_init(&b_full, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&d_full[b], kT64Issuers);
            mbar_init(&d_empty[b], 4);
        }
        for (int g = 0; g < kT64Groups; ++g) {
            mbar_init(&e_full[g], 4);
            mbar_init(&done[g], kT64Issuers);
        }
        fence_mbar_init();
        s_abort = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp >= 4 * kT64Groups) {
        const int issuer = warp - 4 * kT64Groups;
        int tend = T0, table = -1;
        uint32_t chunk = 0;
        bool ok = true;
        for (int T = T0; T < T1 && ok; ++T) {
            const int shape = __shfl_sync(0xffffffffu, recs[T].pairs, 0), pairs = shape & 255, ks = shape >> 8 & 255;
            const int g = (T - T0) & 1;
            if (T == tend) {  // the table's first tile: the previous one's MMAs must have completed
                tend = recs[T].tile_end;
                ++table;
                if (T > T0) ok = warp_ok(mbar_wait_bounded(&done[g ^ 1], (uint32_t)(T - 1 - T0) >> 1 & 1u));
                if (ok && issuer == 0 && (tid & 31) == 0) {
                    const uint32_t bytes = (uint32_t)tc64_table_bytes(pairs, ks);
                    const unsigned char *src = recs[T].tab;
                    mbar_arrive_expect_tx(&b_full, bytes);
                    for (uint32_t o = 0; o < bytes; o += 16384u)
                        bulk_g2s(tcs64 + o, src + o, min(16384u, bytes - o), &b_full);
                }
                __syncwarp();
                ok = ok && warp_ok(mbar_wait_bounded(&b_full, (uint32_t)table & 1u));
            }
            ok = ok && warp_ok(mbar_wait_bounded(&e_full[g], (uint32_t)(T - T0) >> 1 & 1u));
            for (int p = 0; p < pairs && ok; ++p, ++chunk) {
                const uint32_t b = chunk & 1u;
                if (chunk >= 2) ok = warp_ok(mbar_wait_bounded(&d_empty[b], ((chunk >> 1) - 1u) & 1u));
                if (!ok) break;
                tc_fence_after();
                const uint32_t d = tmem + kT64DCol + b * kT64DStride;
                const uint64_t desc = smem_desc(
                    smem_u32(tcs64) + (uint32_t)(p * kTc64Slices * ks) * 512u, 128, 256u * (uint32_t)ks);
                if (elect_one()) {
                    if (ks == KS) {
                        issue_pair<KS>(issuer, d, tmem, desc);
                    } else {  // a wave with fewer K steps than the plan's widest
                        if (KS > 1 && ks == 1) issue_pair<1>(issuer, d, tmem, desc);
                        if (KS > 2 && ks == 2) issue_pair<2>(issuer, d, tmem, desc);
                        if (KS > 3 && ks == 3) issue_pair<3>(issuer, d, tmem, desc);
                    }
                    tc_commit(&d_full[b]);
                    if (p + 1 == pairs) tc_commit(&done[g]);
                }
                __syncwarp();
            }
        }
        if (!ok && (tid & 31) == 0) {
            s_abort = 1;
            // no copy may land after the CTA's shared memory is gone
            if (table >= 0) mbar_wait_bounded(&b_full, (uint32_t)table & 1u);
        }
        __syncwarp();
    } else {
        const int group = warp >> 2, other = group ^ 1, lane = tid & 127;
        const uint32_t quarter = (uint32_t)(32 * (warp & 3)) << 16;
        uint32_t chunk = 0;  // first chunk of this group's tile
        int counted = T0;    // tiles whose chunks are counted
        bool bad = false;
#pragma unroll 1
        for (int T = T0 + group; T < T1; T += kT64Groups) {
            const TileRec *rp = recs + T;
            const int4 span = *reinterpret_cast<const int4 *>(&rp->i0);      // i0, s0, s1, tile_end
            const int4 shape = *reinterpret_cast<const int4 *>(&rp->pairs);  // tc64_shape, c2's (phi), n_mid, c2's (r)
            const int pairs = shape.x & 255;
            for (; counted < T; ++counted) chunk += (uint32_t)(recs[counted].pairs & 255);
            const int i = span.x + lane;
            const uint32_t v = (uint32_t)max(i - max(span.x, span.y), 0);
            TileRec ph;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                reinterpret_cast<int4 *>(&ph)[k] = reinterpret_cast<const int4 *>(rp)[k];
            const int2 lo3 = *reinterpret_cast<const int2 *>(&rp->u0);  // of c3: phi, r
            const long long v2 = (long long)(v * v), v3 = (long long)(v * v * v);
            const unsigned long long fr = phase_fixed(ph.r, v) + (unsigned long long)((lo3.y * v3 + shape.w * v2) >> 32);
            const unsigned long long fphi = phase_fixed(ph.phi, v) + (unsigned long long)((lo3.x * v3 + shape.y * v2) >> 32);
            const TcSeg64 *sg = static_cast<const TcSeg64 *>(rp->seg);
            // (lanes outside the segment take its first or last sample's u: sums stay in range)
            const double u = (fma((double)min(max(i, span.y), span.z - 1), sg->dt, sg->t0) - sg->tk) * sg->ih;
            const Q62 U = q62(__double2ll_rn(u * 4611686018427387904.0));
            const Cq zphi = sincos62(fphi);
            Cq z[8];  // e^{i k theta}
            z[0] = Cq{q62(1ll << 62), q62(0)};
            z[1] = sincos62(fr);
            z[2] = cmul(z[1], z[1]);
            z[3] = cmul(z[2], z[1]);
            z[4] = cmul(z[2], z[2]);
            z[5] = cmul(z[4], z[1]);
            z[6] = cmul(z[4], z[2]);
            z[7] = cmul(z[4], z[3]);
            const Cq z8 = KS > 1 ? sincos62(8 * fr) : z[0];
            // the operand columns are free once the previous tile's MMAs have completed; the waits on
            // its last accumulators (complete by then) keep this group's parities in step
            if (T > T0) {
                if (!mbar_wait_bounded(&done[other], (uint32_t)(T - 1 - T0) >> 1 & 1u)) bad = true;
                for (uint32_t k = chunk > 1 ? 2 : 1; k >= 1 && !bad; --k)
                    if (!mbar_wait_bounded(&d_full[(chunk - k) & 1u], (chunk - k) >> 1 & 1u)) bad = true;
            }
            __syncwarp();
            tc_fence_after();
            store_digits(tmem + quarter, z);
            if (KS > 1) {
                Cq g = z8;
#pragma unroll 1
                for (int a = 1; a < KS; ++a) {
                    Cq p[8];
                    p[0] = g;
#pragma unroll
                    for (int k = 1; k < 8; ++k) p[k] = cmul(g, z[k]);
                    store_digits(tmem + quarter + 8 * a, p);
                    g = cmul(g, z8);
                }
            }
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (s_abort) bad = true;
            if (__any_sync(0xffffffffu, bad)) {
                bad = true;
                break;
            }
            if ((tid & 31) == 0) mbar_arrive(&e_full[group]);
            const int shift = sg->shift;
            const long long round = (1ll << shift) >> 1;
            Q62 t0r{0, 0}, t0i{0, 0}, t1r{0, 0}, t1i{0, 0};  // rows m >= 0 in z_phi^-1, rows m < 0 in z_phi
#pragma unroll 1
            for (int p = 0; p < pairs; ++p) {
                const uint32_t ch = chunk + (uint32_t)p, b = ch & 1u;
                if (!mbar_wait_bounded(&d_full[b], (ch >> 1) & 1u)) bad = true;
                __syncwarp();
                if (__any_sync(0xffffffffu, bad)) {
                    bad = true;
                    break;
                }
                tc_fence_after();
                const uint32_t d = tmem + kT64DCol + b * kT64DStride + quarter;
                float S[kTc64Slices][16];
#pragma unroll
                for (int o = 0; o < kTc64Slices; ++o) tc_ld16(d + 16 * o, S[o]);
                tc_wait_ld16(S[0]);
#pragma unroll
                for (int o = 1; o < kTc64Slices; ++o) tc_landed16(S[o]);
                tc_fence_before();
                __syncwarp();
                if ((tid & 31) == 0) mbar_arrive(&d_empty[b]);
                // rows m = m_top - p (even columns) and p - m_top (odd): the cubics, then Horner's step
                long long a[2][2];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    long long acc[2];
#pragma unroll
                    for (int dg = 3; dg >= 0; --dg) {
                        float2 w[kTc64Slices];
                        long long k[2];
#pragma unroll
                        for (int o = 0; o < kTc64Slices; ++o)
                            w[o] = reinterpret_cast<const float2 *>(S[o])[4 * c + dg];
                        join_orders(w, k);
#pragma unroll
                        for (int e = 0; e < 2; ++e) acc[e] = dg == 3 ? k[e] : mul62(q62(acc[e]), U) + k[e];
                    }
                    a[0][c] = (acc[0] + round) >> shift;
                    a[1][c] = (acc[1] + round) >> shift;
                }
                // z_phi = e^{-i Phi_phi} = (c, -s)
                const long long n0r = mul62(t0r, zphi.c) + mul62(t0i, zphi.s) + a[0][0];
                const long long n0i = mul62(t0i, zphi.c) - mul62(t0r, zphi.s) + a[0][1];
                const long long n1r = mul62(t1r, zphi.c) - mul62(t1i, zphi.s) + a[1][0];
                const long long n1i = mul62(t1i, zphi.c) + mul62(t1r, zphi.s) + a[1][1];
                t0r = q62(n0r);
                t0i = q62(n0i);
                t1r = q62(n1r);
                t1i = q62(n1i);
            }
            if (bad) break;
            if (i >= span.y && i < span.z) {
                const double hr = (double)(value(t0r) + value(t1r)), hi = (double)(value(t0i) + value(t1i));
                const double inv = sg->inv1;
                double fc = inv, fs = 0.0;
                if (shape.z != 0) {  // z_r^{n_mid}
                    const Cq w = sincos62((unsigned long long)(long long)shape.z * fr);
                    fc = (double)value(w.c) * 2.168404344971008868e-19 * inv;  // 2^-62
                    fs = (double)value(w.s) * 2.168404344971008868e-19 * inv;
                }
                const double yr = fma(hr, fc, hi * fs) * sg->inv2, yi = fma(hi, fc, -hr * fs) * sg->inv2;
                void *out = rp->out;
                if (shape.x >> 16)
                    reinterpret_cast<float2 *>(out)[i] = make_float2((float)yr, (float)yi);
                else
                    reinterpret_cast<double2 *>(out)[i] = make_double2(yr, yi);
            }
        }
        if (bad) s_abort = 1;
    }
    __syncthreads();
    if (tid == 0 && s_abort) atomicOr(hp->err, ERRBIT_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

namespace {
using Tc64Kernel = void (*)(const PlanHdr *);
const Tc64Kernel kTc64Kernels[kT64MaxKs] = {k_sum_tc64<1>, k_sum_tc64<2>, k_sum_tc64<3>, k_sum_tc64<4>};
constexpr int kFold64Smem = 16 * kTcMaxPairs * fold_stride(kT64MaxKs, sizeof(double)) * (int)sizeof(double);
}  // namespace

cudaError_t tc64_configure()
{
    for (Tc64Kernel k : kTc64Kernels) {
        const cudaError_t e =
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kT64MaxTable);
        if (e != cudaSuccess) return e;
    }
    return cudaFuncSetAttribute(k_fold_tc64, cudaFuncAttributeMaxDynamicSharedMemorySize, kFold64Smem);
}

cudaError_t launch_fold_tc64(const PlanHdr *hdr_dev, int total_segs, int total_tiles, int sm_count,
                             cudaStream_t st)
{
    if (total_tiles <= 0) return cudaSuccess;
    const unsigned grid = total_segs + tc_record_blocks(total_tiles, total_segs, sm_count);
    return launch_pdl(k_fold_tc64, grid, kT64FoldThreads, kFold64Smem, st, hdr_dev);
}

cudaError_t launch_sum_tc64(const PlanHdr *hdr_dev, int grid, int ks, cudaStream_t st)
{
    if (grid <= 0) return cudaSuccess;
    if (ks < 1 || ks > kT64MaxKs) return cudaErrorInvalidValue;
    return launch_pdl(kTc64Kernels[ks - 1], grid, kT64Threads, kT64MaxTable, st, hdr_dev);
}

}  // namespace fewsum
