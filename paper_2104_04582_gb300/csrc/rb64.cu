// rb64.cu -- FP64 reduced-basis amplitudes on the tensor cores, in exact integer arithmetic (arXiv:2104.04582
// Sec. 3.E; the product and its scale: rb.cu).
//
// A_k,i = s_k sum_j alpha_k,j B_j,i is a real product of depth 2 Nb (rb.cu), and the chip's FP64 pipe (two
// FMA a cycle and SM) bounds it.  Here both operands are fixed-point numbers of 8 signed 8-bit digits, held
// as fp16 integers: a knot's coefficients and a mode's basis column, each scaled by the power of two that
// brings its largest entry into [1/2, 1), in units of 2^-62.  The products of digits i and j with i + j = o
// <= 7 (36 of them) are summed in accumulator o.  The top digits are at most 64, so with at most 204
// columns to a sum the FP32 accumulators of orders 0 .. 5 are exact integers (below 2^24); orders 6 and 7,
// in units of 2^-60 and 2^-68, may be rounded by a unit.  Deeper bases are summed in parts of 192 columns.
// What is left out (o >= 8) is near 2^-58 of the two scales, so the result is as good as FP64's own
// rounding, 2^-53 of sum |alpha B| and more, unless that sum is far below the product of the largest
// entries.  That is checked for every output: a ninth product, of the top digits' magnitudes, bounds the
// sum of magnitudes, and an output where it is below 2^-5, or whose row or column has entries that
// are not finite or not within 2^+-400, is computed by an FP64 chain in the product's own epilogue.
//
// A CTA forms one tile of 64 modes (128 real columns: tensor-memory lanes) x up to 64 knots (an even share
// of them): eight accumulators of 64 columns fill tensor memory.  The operands' digits of 16 columns (48 KB) are one stage of a ring
// filled by bulk copies.  Shared memory bounds the products (an MMA reads 6 KB: 48 cycles), then the
// conversions of the sums.  100 knots x 99 vectors x 3843 modes, whole call: 305 us with the
// FP64 chain, 51 us here, and 6.4e-16 -> 1.0e-16 from quadruple precision; 374 x 170 x 3843 1808 -> 257 us,
// 100 x 20 x 200 35 -> 29 us, so k_rb_fp64 (rb.cu) is left only where there is no memory for the
// slices.
#include <cuda_fp16.h>

#include "async.cuh"
#include "fewsum_internal.h"
#include "launch.cuh"
#include "rb_scale.cuh"
#include "tcgen05.cuh"

namespace fewsum {

namespace {

constexpr int kDigits = 8, kRows = 128, kKnots = 64;       // slices; tile
constexpr int kA = kRows * 32, kB = kKnots * 32;            // bytes of one slice of 16 columns
constexpr int kStages = 4, kStage = kDigits * (kA + kB);     // 48 KB
constexpr int kSumSteps = 12, kSumColumns = 204;              // K steps of a part; columns that need no parts
constexpr int kEpiWarps = 8, kThreads = 32 * (kEpiWarps + 2);  // and producer, MMAs
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(kKnots >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);
constexpr float kSmall = 128.0f;                             // 2^-5 in units of the top digits' products

__device__ __forceinline__ double pow2_64(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// Two bytes digit + 128 as fp16 integers: 0x64 byte is 1024 + byte.
__device__ __forceinline__ uint32_t digits2(uint32_t b0, uint32_t b1)
{
    const uint32_t w = 0x64006400u | b0 | b1 << 16;
    const __half2 d = __hsub2(*reinterpret_cast<const __half2 *>(&w), __floats2half2_rn(1152.0f, 1152.0f));
    return *reinterpret_cast<const uint32_t *>(&d);
}

// The digit slices of 8 consecutive columns x[0 .. 7] of one row (each scaled by f to units of 2^-62), at
// `dst` and every `step` bytes after, most significant first, and the top digits' magnitudes at `top`.
__device__ __forceinline__ void store_slices(const double (&x)[8], double f, unsigned char *dst, int step,
                                             unsigned char *top)
{
    unsigned long long v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = (unsigned long long)__double2ll_rn(x[k] * f) + 0x8080808080808080ull;
#pragma unroll
    for (int q = 0; q < kDigits; ++q) {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            w[k] = digits2((uint32_t)(v[2 * k] >> (56 - 8 * q)) & 255u, (uint32_t)(v[2 * k + 1] >> (56 - 8 * q)) & 255u);
        *reinterpret_cast<uint4 *>(dst + (size_t)q * step) = make_uint4(w[0], w[1], w[2], w[3]);
        if (q == 0)
            *reinterpret_cast<uint4 *>(top) = make_uint4(w[0] & 0x7fff7fffu, w[1] & 0x7fff7fffu, w[2] & 0x7fff7fffu,
                                                         w[3] & 0x7fff7fffu);
    }
}

// Place of row r, columns 8 c .. 8 c + 7 (c = 0, 1) in a slice of 16 columns.
__host__ __device__ constexpr int core64(int r, int c) { return (r >> 3) * 256 + c * 128 + (r & 7) * 16; }

}  // namespace

// Scaling exponents of each mode's basis column: for the mixed product's split (bexp) and for the digit
// slices (bexp64, or null); 0 past the last mode.  Eight warps share the basis vectors of 32 modes (a thread
// a mode left the chip idle: 45 us for 3843 modes of 99 vectors, 5 so).
constexpr int kColWarps = 8;

__global__ void __launch_bounds__(32 * kColWarps)
k_rb_col_exp(const double *__restrict__ bre, const double *__restrict__ bim, int Nb, int N, int n_exp, int n_exp64,
             int *__restrict__ bexp, int *__restrict__ bexp64)
{
    __shared__ double s_max[kColWarps][32];
    __shared__ unsigned long long s_mag[kColWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    double m = 0.0;
    unsigned long long g = 0;
    if (i < N) {
#pragma unroll 4
        for (int j = w; j < Nb; j += kColWarps) {
            const double x = bre[(size_t)j * N + i], y = bim[(size_t)j * N + i];
            m = fmax(m, fmax(fabs(x), fabs(y)));
            g = max(g, max(mag(x), mag(y)));
        }
    }
    s_max[w][lane] = m;
    s_mag[w][lane] = g;
    __syncthreads();
    if (w > 0) return;
#pragma unroll
    for (int k = 1; k < kColWarps; ++k) {
        m = fmax(m, s_max[k][lane]);
        g = max(g, s_mag[k][lane]);
    }
    if (i < n_exp) bexp[i] = scale_exp((float)m);
    if (bexp64 && i < n_exp64) bexp64[i] = scale_exp64(__longlong_as_double((long long)g));
}

// Basis slices: tile t holds [steps][8][4 KB], then the magnitudes [steps][4 KB].  Row r is the real (r < 64)
// or imaginary output column of mode 64 t + r % 64 (Bhat of rb.cu).
__global__ void k_rb64_pack_b(const double *__restrict__ bre, const double *__restrict__ bim, int Nb, int N,
                              int steps, int tiles, const int *__restrict__ bexp, unsigned char *__restrict__ pack)
{
    const long long chunks = (long long)tiles * steps * 2 * kRows;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < chunks; t += (long long)gridDim.x * blockDim.x) {
        const int r = (int)(t % kRows), c8 = (int)(t / kRows % (2 * steps)), tile = (int)(t / kRows / (2 * steps));
        const int i = tile * 64 + r % 64, e = bexp[i];
        const double f = e == kPlain ? 0.0 : pow2_64(e + 62);
        double x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int q = 8 * c8 + k, j = q < Nb ? q : q - Nb;
            x[k] = 0.0;
            if (i < N && q < 2 * Nb && e != kPlain) {
                const bool im = (q >= Nb) != (r >= 64);  // of B
                x[k] = (im ? bim : bre)[(size_t)j * N + i];
                if (q >= Nb && r < 64) x[k] = -x[k];
            }
        }
        unsigned char *p = pack + (size_t)tile * steps * (kDigits + 1) * kA;
        const int s = c8 >> 1, at = core64(r, c8 & 1);
        store_slices(x, f, p + (size_t)s * kDigits * kA + at, kA, p + ((size_t)steps * kDigits + s) * kA + at);
    }
}

// Coefficient slices, one warp a row: tile t, of `per` knots on 64 rows, holds [steps][8][2 KB], then
// [steps][2 KB].
__global__ void __launch_bounds__(128)
k_rb64_pack_a(const double *__restrict__ are, const double *__restrict__ aim, int M, int Nb, int steps, int per,
              unsigned char *__restrict__ pack, int *__restrict__ aexp)
{
    pdl_launch_dependents();  // the product
    const int lane = threadIdx.x & 31, row = blockIdx.x * 4 + (threadIdx.x >> 5);
    const int k = row / kKnots * per + row % kKnots;
    {
        const bool live = row % kKnots < per && k < M;
        const double *xr = are + (size_t)k * Nb, *xi = aim + (size_t)k * Nb;
        unsigned long long m = 0;
        if (live)
            for (int j = lane; j < Nb; j += 32) m = max(m, max(mag(xr[j]), mag(xi[j])));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        const int e = scale_exp64(__longlong_as_double((long long)m));
        if (lane == 0) aexp[row] = e;
        const double f = e == kPlain ? 0.0 : pow2_64(e + 62);
        unsigned char *p = pack + (size_t)(row / kKnots) * steps * (kDigits + 1) * kB;
        for (int c8 = lane; c8 < 2 * steps; c8 += 32) {
            double x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int q = 8 * c8 + i;
                x[i] = live && q < 2 * Nb && e != kPlain ? (q < Nb ? xr[q] : xi[q - Nb]) : 0.0;
            }
            const int s = c8 >> 1, at = core64(row % kKnots, c8 & 1);
            store_slices(x, f, p + (size_t)s * kDigits * kB + at, kB, p + ((size_t)steps * kDigits + s) * kB + at);
        }
    }
    pdl_wait();  // the scale's kernel: the product waits for this one alone
}

// Warps 0 - 7 convert the sums (warp w: lanes 32 (w % 4) .. + 31, half w / 4 of the knots), warp 8 fills the
// ring, warp 9 issues the MMAs.  Sums in turn: the magnitudes, then each part of the columns; tfull: a
// sum has been formed; tempty: it has been read.
__global__ void __launch_bounds__(kThreads, 1) k_rb64_mma(Rb64Args a)
{
    extern __shared__ __align__(128) unsigned char rb64_smem[];
    __shared__ __align__(8) uint64_t full[kStages], empty[kStages], tfull, tempty;
    __shared__ int s_e[kKnots];      // the rows' exponents
    __shared__ double s_s[kKnots];   // s_k
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_abort;
    __shared__ int s_issued, s_taken;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int tile = blockIdx.x % a.tiles, kt = blockIdx.x / a.tiles, k0 = kt * a.per;
    const int steps = a.steps, parts = 2 * a.Nb <= kSumColumns ? 1 : (steps + kSumSteps - 1) / kSumSteps;
    const int tops = (steps + kDigits - 1) / kDigits;  // stages of magnitudes, eight K steps each
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 32 * kEpiWarps) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&tfull, 1);
        mbar_init(&tempty, kEpiWarps);
        fence_mbar_init();
        s_abort = 0;
        s_issued = s_taken = 0;
    }
    pdl_wait();
    if (tid < kKnots) {
        s_e[tid] = a.aexp[kt * kKnots + tid];
        s_s[tid] = a.scale && k0 + tid < a.M ? a.scale[k0 + tid] : 1.0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == kEpiWarps) {
        if (lane == 0) {
            const unsigned char *ga = a.bpack + (size_t)tile * steps * (kDigits + 1) * kA;
            const unsigned char *gb = a.apack + (size_t)kt * steps * (kDigits + 1) * kB;
            for (int g = 0; g < tops + steps; ++g) {
                const int s = g % kStages;
                unsigned char *st = rb64_smem + s * kStage;
                if (g >= kStages && !mbar_wait_bounded(&empty[s], (g / kStages - 1) & 1)) {
                    s_abort = 1;
                    break;
                }
                // slices of eight K steps' magnitudes, or the eight of one K step: alike in size and place
                const int first = g < tops ? steps * kDigits + g * kDigits : (g - tops) * kDigits;
                const int n = g < tops ? min(kDigits, steps - g * kDigits) : kDigits;
                mbar_arrive_expect_tx(&full[s], (uint32_t)n * (kA + kB));
                bulk_g2s(st, ga + (size_t)first * kA, (uint32_t)n * kA, &full[s]);
                bulk_g2s(st + kDigits * kA, gb + (size_t)first * kB, (uint32_t)n * kB, &full[s]);
                s_issued = g + 1;
            }
        }
        __syncwarp();
    } else if (warp == kEpiWarps + 1) {
        int g = 0;
        bool ok = true;
        for (int part = -1; part < parts && ok; ++part) {  // -1: the magnitudes
            if (part >= 0) ok = __all_sync(0xffffffffu, mbar_wait_bounded(&tempty, part & 1));
            if (!ok) break;
            tc_fence_after();
            const int g0 = g;
            const int g1 = part < 0 ? tops : part + 1 < parts ? tops + (part + 1) * kSumSteps : tops + steps;
            for (; g < g1 && ok; ++g) {
                const int s = g % kStages;
                ok = __all_sync(0xffffffffu, mbar_wait_bounded(&full[s], (g / kStages) & 1));
                if (!ok) break;
                tc_fence_after();
                const uint32_t base = smem_u32(rb64_smem + s * kStage);
                const uint64_t da = smem_desc(base, 128, 256), db = smem_desc(base + kDigits * kA, 128, 256);
                const int n = part < 0 ? min(kDigits, steps - g * kDigits) : 0;
                if (elect_one()) {
                    if (part < 0) {
                        for (int q = 0; q < n; ++q)
                            tc_mma(tmem, da + q * (kA >> 4), db + q * (kB >> 4), kIdesc, (g | q) != 0);
                    } else {
#pragma unroll
                        for (int o = 0; o < kDigits; ++o)
#pragma unroll
                            for (int q = 0; q <= o; ++q)
                                tc_mma(tmem + kKnots * o, da + q * (kA >> 4), db + (o - q) * (kB >> 4), kIdesc,
                                       g != g0 || q != 0);
                    }
                    tc_commit(&empty[s]);
                    if (g + 1 == g1) tc_commit(&tfull);
                }
                __syncwarp();
            }
        }
        if (!ok) s_abort = 1;
        if (lane == 0) s_taken = g;
        __syncwarp();
    } else {
        const int qd = warp & 3, half = (a.per + 1) / 2, col0 = half * (warp >> 2);
        const uint32_t t_lane = tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)col0;
        const int mode = tile * 64 + (qd & 1) * 32 + lane;
        const bool imag = qd >= 2, live = mode < a.N;
        const int eb = a.bexp[mode];
        double *out = (imag ? a.out_im : a.out_re) + (size_t)(k0 + col0) * a.N + mode;
        const int rows = min(half, min(a.per, a.M - k0) - col0);
        uint32_t plain = 0;  // of the 32 knots
        bool ok = true;
        for (int part = -1; part < parts; ++part) {
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(&tfull, (part + 1) & 1));
            if (!ok) break;
            tc_fence_after();
            if (part < 0) {
                uint32_t v[32];
                tc_ld32(t_lane, v);
#pragma unroll
                for (int c = 0; c < 32; ++c)
                    if (!(__uint_as_float(v[c]) >= kSmall) || s_e[col0 + c] == kPlain) plain |= 1u << c;
                if (eb == kPlain) plain = 0xffffffffu;
            } else {
#pragma unroll 1
                for (int h = 0; 16 * h < rows; ++h) {
                    float S[kDigits][16];
#pragma unroll
                    for (int o = 0; o < kDigits; ++o) tc_ld16(t_lane + kKnots * o + 16 * h, S[o]);
                    tc_wait_ld16(S[0]);
#pragma unroll
                    for (int o = 1; o < kDigits; ++o) tc_landed16(S[o]);
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        // orders 0, 1 in units of 2^-20; 2 .. 6 and the rounded 7 in units of 2^-60
                        const int hi = (__float2int_rn(S[0][c]) << 8) + __float2int_rn(S[1][c]);
                        long long lo = (long long)__float2int_rn(S[2][c]) * 16777216ll + (long long)__float2int_rn(S[3][c]) * 65536;
                        lo = (lo + (long long)__float2int_rn(S[4][c]) * 256 + __float2int_rn(S[5][c])) * 256 +
                             __float2int_rn(fmaf(S[7][c], 0.00390625f, S[6][c]));
                        const double d = fma((double)hi, 1099511627776.0, (double)lo);
                        const int row = 16 * h + c;
                        // times 2^-(60 + e_k + e_i): into the exponent (neither bound of it is near)
                        double x = d == 0.0 ? 0.0
                                            : __hiloint2double(__double2hiint(d) - ((60 + s_e[col0 + row] + eb) << 20),
                                                               __double2loint(d));
                        x *= s_s[col0 + row];
                        if (row < rows && live) {
                            double *dst = out + (size_t)row * a.N;
                            if (part > 0) x += *dst;
                            *dst = x;
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty);
        }
        if (!ok) s_abort = 1;
        // The outputs left to the plain chain: the rows that any lane of the warp needs, eight at a time (eight
        // chains in flight, broadcast coefficients, one pair of basis loads for all), or each lane its own rows
        // one after another (scattered loads, ~1.2 times as long a row) where its lanes need few and different ones.
        // 400 knots of 3843 modes and 99 vectors: localised basis and decaying coefficients 2,606 us by the second
        // form alone, 1,440 so; unit vectors and even coefficients 870; by the plain chain of every output 1,705.
        if (rows < 32) plain &= rows > 0 ? (1u << rows) - 1u : 0u;
        if (!live || !ok) plain = 0;
        const int col = min(mode, a.N - 1);
        uint32_t any = __reduce_or_sync(0xffffffffu, plain);
        if (5u * __reduce_max_sync(0xffffffffu, (unsigned)__popc(plain)) < 4u * (unsigned)__popc(any)) {
            for (; plain; plain &= plain - 1u) {
                const int row = __ffs(plain) - 1;
                const double *xr = a.are + (size_t)(k0 + col0 + row) * a.Nb, *xi = a.aim + (size_t)(k0 + col0 + row) * a.Nb;
                double acc = 0.0;
                for (int j = 0; j < a.Nb; ++j) {
                    const double br = __ldg(a.bre + (size_t)j * a.N + col), bi = __ldg(a.bim + (size_t)j * a.N + col);
                    acc = fma(__ldg(xr + j), imag ? bi : br, fma(__ldg(xi + j), imag ? br : -bi, acc));
                }
                out[(size_t)row * a.N] = s_s[col0 + row] * acc;
            }
            any = 0;
        }
        while (any) {
            constexpr int R = 8;
            int row[R];
            const double *xr[R], *xi[R];
            double acc[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                row[r] = any ? __ffs(any) - 1 : row[r - 1];
                any &= any - 1u;
                xr[r] = a.are + (size_t)(k0 + col0 + row[r]) * a.Nb;
                xi[r] = a.aim + (size_t)(k0 + col0 + row[r]) * a.Nb;
                acc[r] = 0.0;
            }
#pragma unroll 2
            for (int j = 0; j < a.Nb; ++j) {
                const double br = __ldg(a.bre + (size_t)j * a.N + col), bi = __ldg(a.bim + (size_t)j * a.N + col);
                const double y0 = imag ? bi : br, y1 = imag ? br : -bi;
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r] = fma(__ldg(xr[r] + j), y0, fma(__ldg(xi[r] + j), y1, acc[r]));
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (plain >> row[r] & 1u) out[(size_t)row[r] * a.N] = s_s[col0 + row[r]] * acc[r];
        }
    }
    __syncthreads();
    if (tid == 0 && s_abort) {
        atomicOr(a.err, ERRBIT_TIMEOUT);
        // copies and MMAs in flight end before shared and tensor memory are given back
        for (int g = s_taken; g < s_issued; ++g) mbar_wait_bounded(&full[g % kStages], (g / kStages) & 1);
        for (int g = max(0, s_taken - kStages); g < s_taken; ++g) mbar_wait_bounded(&empty[g % kStages], (g / kStages) & 1);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

size_t rb64_basis_bytes(int Nb, int N)
{
    return (size_t)((N + 63) / 64) * ((2 * Nb + 15) / 16) * (kDigits + 1) * kA;
}
size_t rb64_coef_bytes(int Nb, int M)
{
    return (size_t)((M + kKnots - 1) / kKnots) * ((2 * Nb + 15) / 16) * (kDigits + 1) * kB;
}
int rb64_rows(int M) { return (M + kKnots - 1) / kKnots * kKnots; }
int rb64_modes(int N) { return (N + 63) / 64 * 64; }

cudaError_t rb64_configure()
{
    return cudaFuncSetAttribute(k_rb64_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, kStages * kStage);
}

cudaError_t launch_rb_exponents(const double *bre, const double *bim, int Nb, int N, int n_exp, int *bexp, int *bexp64,
                                cudaStream_t st)
{
    const int modes = rb64_modes(N), most = n_exp > modes ? n_exp : modes;
    k_rb_col_exp<<<(most + 31) / 32, 32 * kColWarps, 0, st>>>(bre, bim, Nb, N, n_exp, modes, bexp, bexp64);
    return cudaGetLastError();
}

cudaError_t launch_rb64_basis(const double *bre, const double *bim, int Nb, int N, const int *bexp, unsigned char *pack,
                              int sm_count, cudaStream_t st)
{
    const int modes = rb64_modes(N);
    k_rb64_pack_b<<<sm_count * 8, 256, 0, st>>>(bre, bim, Nb, N, (2 * Nb + 15) / 16, modes / 64, bexp, pack);
    return cudaGetLastError();
}

cudaError_t launch_rb64(Rb64Args a, unsigned char *apack, int *aexp, bool after_scale, cudaStream_t st)
{
    const int rows = rb64_rows(a.M), tiles = rows / kKnots;
    a.per = (a.M + tiles - 1) / tiles;
    a.steps = (2 * a.Nb + 15) / 16;
    a.tiles = rb64_modes(a.N) / 64;
    a.apack = apack;
    a.aexp = aexp;
    cudaError_t e;
    if (after_scale) {  // beside the scale's kernel, whose plain launch it leans on (launch.cuh)
        e = launch_pdl(k_rb64_pack_a, (unsigned)(rows / 4), 128u, (size_t)0, st, a.are, a.aim, a.M, a.Nb, a.steps,
                       a.per, apack, aexp);
    } else {
        k_rb64_pack_a<<<rows / 4, 128, 0, st>>>(a.are, a.aim, a.M, a.Nb, a.steps, a.per, apack, aexp);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    return launch_pdl(k_rb64_mma, (unsigned)(tiles * a.tiles), (unsigned)kThreads, (size_t)(kStages * kStage), st, a);
}

}  // namespace fewsum
