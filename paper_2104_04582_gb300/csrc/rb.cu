// rb.cu -- mode amplitudes from reduced-basis coefficients (arXiv:2104.04582 Sec. 3.E).
//
// Each knot k carries Nb complex coefficients alpha_k; its N mode amplitudes are
//     A_k,i = s_k sum_j alpha_k,j B_j,i,
// with s_k = nu_k / ||alpha_k B|| when target norms nu_k are given (the renormalisation of the
// network's output to the trajectory's norm spline), else s_k = 1.  The norm comes from the
// basis Gram matrix, ||alpha B||^2 = sum_jl alpha_j conj(alpha_l) G_jl with G = B B^H, so the
// scale is known before the product and no second pass over the output is needed.
//
// FP64 path: exact integer digit slices on the tensor cores (rb64.cu); on the FP64 pipe (k_rb_fp64) in a
// context without room for the slices.
// Mixed path: the complex product as one real GEMM on the tcgen05 tensor cores,
//     [Re A_i, Im A_i] = s sum_q a_q Bhat_q,(2i, 2i+1),  a = [Re alpha | Im alpha] (2 Nb),
//     Bhat_q,2i = (Re B_qi | -Im B_qi),  Bhat_q,2i+1 = (Im B_qi | Re B_qi),
// in fp16 with FP32 accumulation in tensor memory.  To keep near-FP32 accuracy every operand is
// split into two fp16 parts x = hi + lo (11 significant bits each) and the three products of
// order <= 2^-11 (hi.hi, hi.lo, lo.hi) are laid side by side along K, so one GEMM of depth
// 3 x 2 Nb sums them all.  fp16's narrow exponent range is handled by exact power-of-two
// scaling: each knot's coefficient row and each mode's basis column are scaled so that their
// largest magnitude lies in [2^14, 2^15) before the split, and the epilogue multiplies the
// accumulator back by both inverse powers and by the knot's renormalisation s (so the scale's kernels run
// beside the coefficient pack: as dependent launches up to 128 vectors, on a second stream above, and end
// before the product).  An entry far below its row or column maximum keeps an absolute error near 2^-24 of
// that maximum.
//
// The product is computed transposed, A^T = Bhat^T a^T: the MMA's M side (tensor-memory lanes)
// is 128 real output columns of two groups of 32 modes (rows 0-63 the real parts, 64-127 the
// imaginary parts)
// and its N side (tensor-memory columns) 256 knots.  A lane of the accumulator then holds one
// output column for consecutive knots, so for each knot a warp stores 32 consecutive modes (256
// contiguous bytes) straight from registers.  With N not a multiple of four the rows start at any of
// four places in a 32-byte sector; groups then overlap by four modes, and a warp stores the 28 of
// its 32 that fill whole sectors (written in parts by two warps, the sectors held the stores to
// 4.8 TB/s, whole they reach 6.1: see k_rb_mma).  Operands are packed once into the canonical K-major
// layout without swizzle that the tensor core's shared-memory descriptors read: 8 x 8 fp16 "core
// matrices" of 16-byte rows, core matrices adjacent in K 128 bytes apart, 8-row groups 1024
// bytes apart.  A k-block of 64 columns of a 128-row basis tile or a 256-row coefficient tile is
// one contiguous 16 / 32 KB block in global memory, so each pipeline stage is filled by two bulk
// asynchronous copies.
#include <type_traits>

#include <cuda_fp16.h>

#include "async.cuh"
#include "convert.cuh"
#include "fewsum_internal.h"
#include "launch.cuh"
#include "rb_scale.cuh"
#include "tcgen05.cuh"

namespace fewsum {

constexpr int kRbTileM = 128;   // MMA M, tensor-memory lanes: real output columns of 64 modes
constexpr int kRbTileN = 256;   // MMA N, tensor-memory columns: knots per coefficient tile
constexpr int kRbTileK = 64;    // fp16 columns per k-block: 128 bytes per row
constexpr int kRbStages = 4;    // shared-memory pipeline depth
constexpr int kRbParts = 3;     // split products laid along K
constexpr uint32_t kRbABytes = kRbTileM * kRbTileK * 2;  // 16 KB: basis (A operand)
constexpr uint32_t kRbBBytes = kRbTileN * kRbTileK * 2;  // 32 KB: coefficients (B operand)
constexpr uint32_t kRbStageBytes = kRbABytes + kRbBBytes;

// Which fp16 part of the A (coefficient) and B (basis) operand each K segment g < kRbParts
// holds (0 = hi, 1 = lo): the segments multiply hi x hi, hi x lo and lo x hi.  Arithmetic, not a
// table, so lanes at different segments need no divergent constant-memory reads.
__host__ __device__ constexpr int part_a(int g) { return g == 2 ? 1 : 0; }
__host__ __device__ constexpr int part_b(int g) { return g == 1 ? 1 : 0; }
__host__ __device__ constexpr uint32_t core_offset(int r, int c)
{
    return (uint32_t)(r >> 3) * 1024u + (uint32_t)(c >> 3) * 128u + (uint32_t)(r & 7) * 16u +
           (uint32_t)(c & 7) * 2u;
}

__device__ __forceinline__ __half split_part(float x, int part)
{
    const __half hi = __float2half_rn(x);
    if (part == 0) return hi;
    return __float2half_rn(x - __half2float(hi));  // the difference is exact in FP32
}

__device__ __forceinline__ uint32_t pack2(__half a, __half b)
{
    return (uint32_t)__half_as_ushort(a) | ((uint32_t)__half_as_ushort(b) << 16);
}

// 2^e as a float, |e| <= kRbMaxExp.
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((uint32_t)(127 + e) << 23); }

// ---- basis set-up -------------------------------------------------------------------------

// Gram matrix G_jl = sum_i B_ji conj(B_li), stored transposed (gt[l][j] = G_jl) so that the
// lanes of a warp, one per j, read consecutive entries; FP64 and an FP32 copy.
__global__ void k_rb_gram(const double *__restrict__ bre, const double *__restrict__ bim, int Nb,
                          int N, double2 *__restrict__ gt64, float2 *__restrict__ gt32)
{
    const int j = blockIdx.x % Nb, l = blockIdx.x / Nb;
    double sr = 0.0, si = 0.0;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const double ar = bre[(size_t)j * N + i], ai = bim[(size_t)j * N + i];
        const double cr = bre[(size_t)l * N + i], ci = bim[(size_t)l * N + i];
        sr += ar * cr + ai * ci;  // B_ji conj(B_li)
        si += ai * cr - ar * ci;
    }
    __shared__ double red[2][32];
    for (int o = 16; o > 0; o >>= 1) {
        sr += __shfl_down_sync(0xffffffffu, sr, o);
        si += __shfl_down_sync(0xffffffffu, si, o);
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (lane == 0) { red[0][w] = sr; red[1][w] = si; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double tr = 0.0, ti = 0.0;
        for (int k = 0; k < nw; ++k) { tr += red[0][k]; ti += red[1][k]; }
        gt64[(size_t)l * Nb + j] = make_double2(tr, ti);
        gt32[(size_t)l * Nb + j] = make_float2((float)tr, (float)ti);
    }
}

// Basis operand (the MMA's A side), scaled, split and packed: row r of basis tile b is the real
// (r < 64) or imaginary (r >= 64) output column of mode r mod 32 of group 2 b + (r mod 64) / 32, whose
// first mode is `step` times its number; column c = g 2Nb + q
// holds part part_b(g) of 2^bexp[mode] Bhat for that column.  Modes past N and columns past
// 3 x 2Nb are zero.
__global__ void k_rb_pack_b(const double *__restrict__ bre, const double *__restrict__ bim, int Nb,
                            int N, int n_kb, int n_tiles, int step, const int *__restrict__ bexp,
                            unsigned char *__restrict__ bpack)
{
    const long long chunks = (long long)n_tiles * kRbTileM * n_kb * (kRbTileK / 8);
    const int Kr = 2 * Nb;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < chunks;
         t += (long long)gridDim.x * blockDim.x) {
        const int q8 = (int)(t % (n_kb * (kRbTileK / 8)));
        const int row = (int)(t / (n_kb * (kRbTileK / 8)));
        const int c0 = q8 * 8;
        const int rr = row % kRbTileM, i = ((row / kRbTileM) * 2 + (rr / 32) % 2) * step + rr % 32;
        const bool imag_out = rr >= kRbTileM / 2;
        uint32_t w[4];
        for (int e = 0; e < 8; e += 2) {
            __half v[2];
            for (int h = 0; h < 2; ++h) {
                const int c = c0 + e + h, g = c / Kr, q = c % Kr;
                float x = 0.0f;
                int part = 0;
                if (g < kRbParts && i < N) {
                    const int j = q % Nb;
                    const bool from_im = q >= Nb;
                    const double br = bre[(size_t)j * N + i], bi = bim[(size_t)j * N + i];
                    const double v = imag_out ? (from_im ? br : bi) : (from_im ? -bi : br);
                    x = (float)ldexp(v, bexp[i]);
                    part = part_b(g);
                }
                v[h] = split_part(x, part);
            }
            w[e / 2] = pack2(v[0], v[1]);
        }
        const int tile = row / kRbTileM, kb = c0 / kRbTileK;
        unsigned char *blk = bpack + ((size_t)tile * n_kb + kb) * kRbABytes;
        *reinterpret_cast<uint4 *>(blk + core_offset(rr, c0 % kRbTileK)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// ---- per call -----------------------------------------------------------------------------

// Quadratic form q_k = ||alpha_k B||^2 = sum_j Re(alpha_j t_j), t_j = sum_l G_jl conj(alpha_l), in
// FP32, as a small register-blocked product: a block takes 32 knots
// and 64 values of j, l advancing in chunks of 64 staged in (dynamic) shared memory; a thread owns
// 4 knots x 2 values of j (j and j + 32), so 6 shared-memory reads feed 16 complex multiply-adds.
// Partial sums over j are reduced per warp and added to q (FP64, zeroed beforehand); k_rb_norm
// then forms s_k.  Used for bases of more than 128 vectors.
constexpr int kQRows = 32, kQJ = 64, kQL = 64, kQThreads = 256, kQPer = 4;

constexpr int kQSmem = (kQL * kQJ + kQRows * kQL) * (int)sizeof(float2);

__global__ void __launch_bounds__(kQThreads)
k_rb_quad(const double *__restrict__ are, const double *__restrict__ aim, int M, int Nb,
          const float2 *__restrict__ gt, double *__restrict__ q)
{
    extern __shared__ __align__(16) unsigned char rb_quad_smem_raw[];
    float2(*sg)[kQJ] = reinterpret_cast<float2(*)[kQJ]>(rb_quad_smem_raw);                       // G_jl [l][j]
    float2(*sa)[kQL] = reinterpret_cast<float2(*)[kQL]>(rb_quad_smem_raw + kQL * kQJ * sizeof(float2));  // alpha
    const int tid = threadIdx.x, jl = tid & 31, rg = tid >> 5;  // rg: knots 4 rg .. 4 rg + 3
    const int j0 = blockIdx.x * kQJ + jl, k0 = blockIdx.y * kQRows;
    float tr[kQPer][2], ti[kQPer][2];
#pragma unroll
    for (int i = 0; i < kQPer; ++i) tr[i][0] = tr[i][1] = ti[i][0] = ti[i][1] = 0;
    for (int l0 = 0; l0 < Nb; l0 += kQL) {
        const int lc = Nb - l0 < kQL ? Nb - l0 : kQL;
        __syncthreads();
        for (int e = tid; e < lc * kQJ; e += kQThreads) {
            const int l = l0 + e / kQJ, jx = blockIdx.x * kQJ + e % kQJ;
            sg[e / kQJ][e % kQJ] = jx < Nb ? gt[(size_t)l * Nb + jx] : float2{};
        }
        for (int e = tid; e < kQRows * lc; e += kQThreads) {
            const int r = e / lc, l = l0 + e % lc, k = k0 + r;
            float2 v{};
            if (k < M) {
                v.x = (float)are[(size_t)k * Nb + l];
                v.y = (float)aim[(size_t)k * Nb + l];
            }
            sa[r][e % lc] = v;
        }
        __syncthreads();
#pragma unroll 2
        for (int l = 0; l < lc; ++l) {
            const float2 g0 = sg[l][jl], g1 = sg[l][jl + 32];
#pragma unroll
            for (int i = 0; i < kQPer; ++i) {
                const float2 x = sa[rg * kQPer + i][l];
                tr[i][0] += g0.x * x.x + g0.y * x.y;  // G_jl conj(alpha_l)
                ti[i][0] += g0.y * x.x - g0.x * x.y;
                tr[i][1] += g1.x * x.x + g1.y * x.y;
                ti[i][1] += g1.y * x.x - g1.x * x.y;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < kQPer; ++i) {
        const int k = k0 + rg * kQPer + i;
        float c = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = j0 + 32 * h;
            if (k < M && j < Nb)
                c += (float)are[(size_t)k * Nb + j] * tr[i][h] - (float)aim[(size_t)k * Nb + j] * ti[i][h];
        }
        for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
        if (jl == 0 && k < M) atomicAdd(q + k, (double)c);
    }
}

// Mixed path, Nb <= 128: the renormalisation scale in one kernel.  A block takes kTRows knots; their FP32
// coefficients and the whole FP32 Gram matrix (j padded to a multiple of 16) sit in shared memory.  The sum over l is
// split among kTParts thread groups (l = part mod kTParts);
// within a group thread (rg, jg) owns knots 4 rg .. 4 rg + 3 and j = jg + 16 t, t < T = ceil(Nb / 16),
// so 12 shared-memory reads (half of them broadcasts) feed 128 multiply-adds per l (T = 8).  The 16 threads of
// a knot group share a half-warp and reduce their partial q_k by shuffles; the groups' partials
// are added in group order and s_k = nu_k / sqrt(q_k) written directly (0 for q_k = 0; a
// non-finite or negative nu_k latches ERRBIT_NONFINITE).  A block needs most of a multiprocessor's shared memory at
// 128 vectors, so one is resident: 44 rows are what 528 threads take by fours, and leave 6,400 knots in one wave of
// 152 (146 blocks; 48 rows would be 134 of 9 % more work).  Any number of knots runs in such waves.
constexpr int kTRows = 44, kTGroup = (kTRows / 4) * 16, kTParts = 3;
constexpr int kTThreads = kTGroup * kTParts;
constexpr int kTMaxBasis = 128;

template <int T>
__global__ void __launch_bounds__(kTThreads)
k_rb_scale_tile(const double *__restrict__ are, const double *__restrict__ aim, int M, int Nb,
                const float2 *__restrict__ gt, const double *__restrict__ nu,
                double *__restrict__ scale, unsigned *__restrict__ err)
{
    constexpr int kTJ = 16 * T;
    pdl_launch_dependents();  // the pack
    extern __shared__ __align__(16) float2 rb_tile_smem[];
    float2 *as = rb_tile_smem;                 // [kTRows][Nb] alpha
    float2 *gs = rb_tile_smem + kTRows * Nb;   // [Nb][kTJ] G_jl stored [l][j], zero for j >= Nb
    __shared__ float q_part[kTParts][kTRows];
    const int tid = threadIdx.x, part = tid / kTGroup, local = tid - part * kTGroup;
    const int jg = local & 15, rg = local >> 4;
    const int k0 = blockIdx.x * kTRows;
    // staging: the Gram matrix by asynchronous copies, all in flight, while the coefficients (9 loads of
    // each array in flight a thread: 44 rows of up to 108 vectors in one round) pass through registers
    for (int l = tid / 16; l < Nb; l += kTThreads / 16) {
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const int j = (tid & 15) + 16 * t;
            if (j < Nb)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(gs + l * kTJ + j)),
                             "l"(gt + (size_t)l * Nb + j)
                             : "memory");
            else
                gs[l * kTJ + j] = make_float2(0.f, 0.f);
        }
    }
    constexpr int kU = 9;
    const int live = min(kTRows, M - k0) * Nb;
    const double *pr = are + (size_t)k0 * Nb, *pi = aim + (size_t)k0 * Nb;  // rows k0 .. are contiguous
    for (int e0 = tid; e0 < kTRows * Nb; e0 += kTThreads * kU) {
        double vr[kU], vi[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int e = e0 + u * kTThreads;
            vr[u] = e < live ? pr[e] : 0.0;
            vi[u] = e < live ? pi[e] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int e = e0 + u * kTThreads;
            if (e < kTRows * Nb) as[e] = make_float2(f64_to_f32(vr[u]), f64_to_f32(vi[u]));
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    float tr[4][T], ti[4][T];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int t = 0; t < T; ++t) tr[r][t] = ti[r][t] = 0.f;
    for (int l = part; l < Nb; l += kTParts) {
        float2 x[4], g[T];
#pragma unroll
        for (int r = 0; r < 4; ++r) x[r] = as[(rg * 4 + r) * Nb + l];
#pragma unroll
        for (int t = 0; t < T; ++t) g[t] = gs[l * kTJ + jg + 16 * t];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int t = 0; t < T; ++t) {
                tr[r][t] += g[t].x * x[r].x + g[t].y * x[r].y;  // G_jl conj(alpha_l)
                ti[r][t] += g[t].y * x[r].x - g[t].x * x[r].y;
            }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int row = rg * 4 + r;
        float q = 0.f;
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const int j = jg + 16 * t;
            if (j < Nb) {
                const float2 a = as[row * Nb + j];
                q += a.x * tr[r][t] - a.y * ti[r][t];  // Re(alpha_j t_j)
            }
        }
        const unsigned half = 0xffffu << (tid & 16);  // (the block's last warp is a half one)
        for (int o = 8; o > 0; o >>= 1) q += __shfl_xor_sync(half, q, o);
        if (jg == 0) q_part[part][row] = q;
    }
    __syncthreads();
    if (tid < kTRows && k0 + tid < M) {
        const int k = k0 + tid;
        float q = q_part[0][tid];
#pragma unroll
        for (int p = 1; p < kTParts; ++p) q += q_part[p][tid];
        const double v = nu[k];
        if (!(v >= 0.0) || !isfinite(v)) atomicOr(err, ERRBIT_NONFINITE);
        scale[k] = q > 0.f ? v / sqrt((double)q) : 0.0;
    }
}

// s_k = nu_k / sqrt(q_k) (0 when q_k = 0, i.e. alpha_k B = 0).  A non-finite or negative target
// norm latches ERRBIT_NONFINITE.
__global__ void k_rb_norm(const double *__restrict__ q, const double *__restrict__ nu, int M,
                          double *__restrict__ scale, unsigned *__restrict__ err)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M) return;
    const double v = nu[k], qk = q[k];
    if (!(v >= 0.0) || !isfinite(v)) atomicOr(err, ERRBIT_NONFINITE);
    scale[k] = qk > 0.0 ? v / sqrt(qk) : 0.0;
}

// Coefficient operand (the MMA's B side), one warp per row: row k of tile k/256, column
// c = g * 2Nb + q holds part part_a(g) of 2^aexp[k] x_q, x_q = alpha_k,q (real parts for q < Nb,
// imaginary parts after; the renormalisation s_k is applied by the product's epilogue, so this
// pack does not wait for it).  The row's x_q are converted once (on the integer pipe) into shared
// memory, its largest magnitude sets aexp[k], then the lanes write its 16-byte chunks.  Rows past
// M are zero.
constexpr int kRbPackWarps = 8;

__global__ void __launch_bounds__(kRbPackWarps * 32)
k_rb_pack_a(const double *__restrict__ are, const double *__restrict__ aim, int M, int Nb, int n_kb,
            int m_tiles, unsigned char *__restrict__ apack, int *__restrict__ aexp)
{
    pdl_launch_dependents();  // the product
    __shared__ float xs[kRbPackWarps][2 * FEW_MAX_BASIS];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, Kr = 2 * Nb;
    float *x = xs[w];
    const int rows = m_tiles * kRbTileN, chunks = n_kb * (kRbTileK / 8);
    for (int row = blockIdx.x * kRbPackWarps + w; row < rows; row += gridDim.x * kRbPackWarps) {
        const bool live = row < M;
        float mx = 0.0f;
        for (int q = lane; q < Kr; q += 32) {
            x[q] = live ? f64_to_f32(q < Nb ? are[(size_t)row * Nb + q] : aim[(size_t)row * Nb + q - Nb])
                        : 0.0f;
            mx = fmaxf(mx, fabsf(x[q]));
        }
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const int e = scale_exp(mx);
        const float f = pow2f(e);
        if (lane == 0) aexp[row] = e;
        __syncwarp();
        unsigned char *tile = apack + (size_t)(row / kRbTileN) * n_kb * kRbBBytes;
        for (int q8 = lane; q8 < chunks; q8 += 32) {
            const int c0 = q8 * 8;
            int g = c0 / Kr, q = c0 - g * Kr;  // segment and column of c0, then stepped
            uint32_t wv[4];
#pragma unroll
            for (int e2 = 0; e2 < 8; e2 += 2) {
                __half v[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    v[h] = g < kRbParts ? split_part(x[q] * f, part_a(g)) : __float2half_rn(0.0f);
                    if (++q == Kr) { q = 0; ++g; }
                }
                wv[e2 / 2] = pack2(v[0], v[1]);
            }
            *reinterpret_cast<uint4 *>(tile + (size_t)(c0 / kRbTileK) * kRbBBytes +
                                       core_offset(row % kRbTileN, c0 % kRbTileK)) =
                make_uint4(wv[0], wv[1], wv[2], wv[3]);
        }
        __syncwarp();
    }
    pdl_wait();  // the scale's kernel: the product waits for this one alone
}

// ---- tensor-core GEMM ---------------------------------------------------------------------

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), fp16 A and B (bits 7-9
// and 10-12 = 0), both K-major (bits 15, 16 = 0), M >> 4 at bits 24-28 (N >> 3 goes to bits 17-22).
constexpr uint32_t kRbIdesc = (1u << 4) | ((uint32_t)(kRbTileM >> 4) << 24);

struct RbMmaArgs {
    const unsigned char *apack;  // coefficients: [m_tiles][n_kb] blocks of kRbBBytes (B operand)
    const unsigned char *bpack;  // basis: [n_tiles][n_kb] blocks of kRbABytes (A operand)
    double *out_re, *out_im;     // [M][N]
    const int *aexp, *bexp;      // scaling exponents of the coefficient rows and basis columns
    const double *scale;         // [M] renormalisation s_k, applied in the epilogue (or null)
    int M, N, n_kb, m_tiles, n_tiles, groups, step;
    int k16_last;                // K = 16 steps of the last k-block holding real columns
    unsigned *err;
};

constexpr int kRbEpiWarps = 16;  // four per tensor-memory lane quarter, every fourth 32-column chunk
constexpr int kRbEpiPerQuarter = kRbEpiWarps / 4;
constexpr int kRbMmaThreads = 64 + 32 * kRbEpiWarps;  // producer warp, MMA warp, epilogue warps
constexpr uint32_t kRbTmemCols = 2 * kRbTileN;         // two accumulator buffers

__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity)
{
    return __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity));
}

// Persistent: CTA b takes items of an equal share (see `item`; tile t = knot tile t / n_tiles, basis tile
// t % n_tiles: neighbours write neighbouring parts of the same rows at about the same time; with each
// CTA on one basis tile the stores alone took 76 us instead of 65).  Warp 0 (one lane) streams each tile's k-blocks through a kRbStages ring of
// shared-memory stages with bulk copies; warp 1 (one lane) issues the MMAs of a tile into one of
// two tensor-memory accumulators of 256 columns and commits; warps 2.. drain the other
// accumulator meanwhile: warp w reads lanes 32 (w % 4) .. + 31 (32 output columns: real parts
// for w % 4 < 2, imaginary parts otherwise) and one in kRbEpiPerQuarter chunks of 32 knots, and
// for each knot stores its columns' FP64 values, 28 modes in seven whole sectors (or 32, see rb_layout),
// from registers.  Bound by the stores and, nearly as much, by shared memory (an MMA reads 12 KB, and as
// much is filled for it: 190 cycles for the tensor core's 128).  6400 knots of 3843 modes and 99 basis
// vectors, the stores alone: 81 us with 256 bytes a warp across nine sectors, 65 as whole sectors;
// the whole call 130 -> 121 us (28 of 32 columns used cost 13 % more tiles, so the conversion to FP64
// takes four instructions instead of ~15, the factors come from shared memory instead of by shuffles,
// and CTAs get equal shares: 12 tiles for each had been 11.4 on average).
// Every wait is bounded; a timeout latches ERRBIT_TIMEOUT and the CTA waits for its copies and MMAs in
// flight before it frees tensor memory.
__global__ void __launch_bounds__(kRbMmaThreads, 1) k_rb_mma(RbMmaArgs a)
{
    extern __shared__ unsigned char rb_mma_smem[];
    __shared__ __align__(8) uint64_t full[kRbStages], empty[kRbStages], tfull[2], tempty[2], drain;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_abort;
    __shared__ uint32_t s_issued, s_consumed;
    __shared__ __align__(16) float s_fa[kRbEpiWarps][32];  // a warp's 32 knots' factors
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // Item u of this CTA: rows k0 .. k0 + nn - 1 (nn a multiple of 16) of basis tile nt.  What is left
    // over of the tiles after as many for every CTA is cut in up to eight parts that come first: the
    // stores start after a small product, and no CTA has a whole tile more than another.
    const int grid = gridDim.x, whole = a.m_tiles * a.n_tiles / grid, left = a.m_tiles * a.n_tiles - whole * grid;
    int cut = 8;
    while (cut > 1 && left * cut > grid) cut >>= 1;
    const int parts = (left * cut + grid - 1) / grid;  // (0 or 1)
    auto item = [&](int u, int &nt, int &k0, int &nn) {
        int t = (u - parts) * grid + (int)blockIdx.x, n = kRbTileN, n0 = 0;
        if (u < parts) {
            const bool mine = (int)blockIdx.x < left * cut;
            n = mine ? kRbTileN / cut : 0;
            n0 = ((int)blockIdx.x % cut) * n;
            t = mine ? whole * grid + (int)blockIdx.x / cut : 0;
        }
        nt = t % a.n_tiles;
        k0 = (t / a.n_tiles) * kRbTileN + n0;
        nn = min(n, (a.M - k0 + 15) & ~15);
    };
    const int items = parts + whole;
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(rb_mma_smem) + 127) & ~(uintptr_t)127);
    unsigned char *sA = base, *sB = base + kRbStages * kRbABytes;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_slot)),
                     "r"(kRbTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < kRbStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], kRbEpiWarps);
        }
        mbar_init(&drain, 1);
        fence_mbar_init();
        s_abort = 0;
        s_issued = s_consumed = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_wait();

    if (warp == 0) {
        if (lane == 0) {  // producer
            const uint64_t keep = l2_evict_last_policy();  // operands are re-read by other CTAs
            uint32_t g = 0;
            for (int w = 0; w < items && !s_abort; ++w) {
                int nt, k0, nn;
                item(w, nt, k0, nn);
                if (nn <= 0) continue;
                const unsigned char *ga = a.bpack + (size_t)nt * a.n_kb * kRbABytes;  // basis
                const unsigned char *gb = a.apack + (size_t)(k0 / kRbTileN) * a.n_kb * kRbBBytes +
                                          (size_t)(k0 % kRbTileN) * (kRbTileK * 2);  // coefficients
                const uint32_t b_bytes = (uint32_t)nn * (kRbTileK * 2);
                for (int kb = 0; kb < a.n_kb; ++kb, ++g) {
                    const int s = g % kRbStages;
                    if (!mbar_wait_bounded(&empty[s], ((g / kRbStages) & 1) ^ 1)) { s_abort = 1; break; }
                    mbar_arrive_expect_tx(&full[s], kRbABytes + b_bytes);
                    bulk_g2s_hint(sA + s * kRbABytes, ga + (size_t)kb * kRbABytes, kRbABytes, &full[s], keep);
                    bulk_g2s_hint(sB + s * kRbBBytes, gb + (size_t)kb * kRbBBytes, b_bytes, &full[s], keep);
                }
            }
            s_issued = g;
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {  // MMA issuer
            uint32_t g = 0;
            int u = 0;
            for (int w = 0; w < items && !s_abort; ++w) {
                int nt, k0, nn;
                item(w, nt, k0, nn);
                if (nn <= 0) continue;
                const uint32_t idesc = kRbIdesc | ((uint32_t)(nn >> 3) << 17);
                const int b = u & 1;
                if (!mbar_wait_bounded(&tempty[b], ((u >> 1) & 1) ^ 1)) { s_abort = 1; break; }
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(b * kRbTileN);
                bool ok = true;
                for (int kb = 0; kb < a.n_kb; ++kb, ++g) {
                    const int s = g % kRbStages;
                    if (!mbar_wait_bounded(&full[s], (g / kRbStages) & 1)) { s_abort = 1; ok = false; break; }
                    tc_fence_after();
                    const uint32_t a0 = smem_u32(sA + s * kRbABytes), b0 = smem_u32(sB + s * kRbBBytes);
                    // the last k-block's columns past 3 x 2 Nb are zero: their MMAs are skipped
                    const int nk = kb + 1 < a.n_kb ? kRbTileK / 16 : a.k16_last;
#pragma unroll
                    for (int k = 0; k < kRbTileK / 16; ++k)  // K = 16 per MMA: two core matrices
                        if (k < nk)
                            tc_mma(d, smem_desc(a0 + k * 256, 128, 1024),
                                   smem_desc(b0 + k * 256, 128, 1024), idesc,
                                   (uint32_t)((kb | k) != 0));
                    tc_commit(&empty[s]);
                }
                if (!ok) break;
                tc_commit(&tfull[b]);
                ++u;
            }
            s_consumed = g;
            tc_commit(&drain);  // arrives once every MMA issued above has completed
        }
        __syncwarp();
    } else {  // epilogue
        const int e = warp - 2, qd = warp & 3;  // a warp reads tensor-memory lanes 32 (warp % 4) ..
        const int c_first = e / 4;              // and chunks c_first + kRbEpiPerQuarter i
        int u = 0;
        for (int w = 0; w < items && !__any_sync(0xffffffffu, s_abort != 0); ++w) {
            int nt, k0, nn;
            item(w, nt, k0, nn);
            if (nn <= 0) continue;
            const int b = u & 1;
            if (!warp_wait(&tfull[b], (u >> 1) & 1)) { s_abort = 1; break; }
            tc_fence_after();
            const int group = nt * 2 + (qd & 1), m0 = group * a.step, mode = m0 + lane;
            double *dst = qd < 2 ? a.out_re : a.out_im;
            // the lanes whose modes fill whole 32-byte sectors of the row, and the row's two ends
            const bool overlap = a.step < 32, first = group == 0, last = group >= a.groups - 1;
            const bool live = group < a.groups && mode < a.N;
            const unsigned at0 = (unsigned)(reinterpret_cast<uintptr_t>(dst) >> 3) + (unsigned)m0;  // modulo 2^32
            const float fb = pow2f(-a.bexp[mode]);  // undo the column scaling (exact)
            for (int c = c_first; c < (nn + 31) / 32; c += kRbEpiPerQuarter) {
                float v[32];
                tc_ld32(tmem + (uint32_t)(b * kRbTileN) + ((uint32_t)(32 * qd) << 16) + (uint32_t)(32 * c),
                        reinterpret_cast<uint32_t(&)[32]>(v));
                const int kc = k0 + 32 * c;
                // knot kc + lane's row scaling (exact) times its renormalisation s_k, for the other lanes
                float fa_lane = pow2f(-a.aexp[kc + lane]);
                if (a.scale && kc + lane < a.M) fa_lane *= (float)a.scale[kc + lane];
                s_fa[e][lane] = fa_lane;
                __syncwarp();
                bool on[4];  // of knots kc + j, by j mod 4
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int off = overlap ? (int)(0u - (at0 + (unsigned)(kc + j) * (unsigned)a.N) & 3u) : 0;
                    on[j] = live && (first || lane >= off) && (last || lane < off + a.step);
                }
                double *row = dst + (size_t)kc * a.N + mode;
                auto store = [&](auto whole) {  // every knot of the chunk is one of the call's
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        const float4 fa = *reinterpret_cast<const float4 *>(&s_fa[e][j]);
                        const float2 fb2 = make_float2(fb, fb);
                        const float2 y0 = __fmul2_rn(__fmul2_rn(make_float2(v[j], v[j + 1]), fb2), make_float2(fa.x, fa.y));
                        const float2 y1 = __fmul2_rn(__fmul2_rn(make_float2(v[j + 2], v[j + 3]), fb2), make_float2(fa.z, fa.w));
                        const float y[4] = {y0.x, y0.y, y1.x, y1.y};
                        double w[4];
                        bool odd = false;  // not a normal number
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            w[i] = f32_normal_to_f64(y[i]);
                            odd |= !f32_is_normal(y[i]);
                        }
                        if (odd) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) w[i] = f32_to_f64(y[i]);
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) {  // streamed once: evict-first
                            if (on[i] && (decltype(whole)::value || kc + j + i < a.M)) __stcs(row, w[i]);
                            row += a.N;
                        }
                    }
                };
                if (kc + 32 <= a.M)
                    store(std::true_type());
                else
                    store(std::false_type());
                __syncwarp();  // s_fa is rewritten
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[b]);
            ++u;
        }
    }

    __syncthreads();
    if (!warp_wait(&drain, 0)) s_abort = 1;  // no MMA of this CTA still running
    if (tid == 0 && s_abort) {
        atomicOr(a.err, ERRBIT_TIMEOUT);
        for (uint32_t g = s_consumed; g < s_issued; ++g)  // let copies in flight land
            mbar_wait_bounded(&full[g % kRbStages], (g / kRbStages) & 1);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kRbTmemCols)
                     : "memory");
}

// ---- FP64 GEMM ----------------------------------------------------------------------------

// The FP64 pipe is the bound (two FMA a cycle and SM), so all that matters is that every SM gets the
// same share of the multiply-adds and none is spent on padding: a warp takes at most 8 knots (the
// knots spread evenly over the groups) x 32 modes, one mode a lane, straight from L1 (coalesced
// basis loads, broadcast coefficients), one warp to a block.  The tiled form
// before it (32 knots x 64 modes a block) left 100 knots x 3843 modes in 1.6 waves with 28 % of its
// rows padding.
constexpr int kRb64Max = 8, kRb64Threads = 32;

template <int R>
__device__ __forceinline__ void rb64_rows(const double *__restrict__ are, const double *__restrict__ aim,
                                          const double *__restrict__ bre, const double *__restrict__ bim,
                                          int k0, int i, int Nb, int N, const double *__restrict__ scale,
                                          double *__restrict__ ore, double *__restrict__ oim)
{
    double ar[R], ai[R];
#pragma unroll
    for (int r = 0; r < R; ++r) ar[r] = ai[r] = 0.0;
    const int col = min(i, N - 1);  // a lane past the end computes the last column and stores nothing
    const double *xr = are + (size_t)k0 * Nb, *xi = aim + (size_t)k0 * Nb;
#pragma unroll 2
    for (int j = 0; j < Nb; ++j) {
        const double br = __ldg(bre + (size_t)j * N + col), bi = __ldg(bim + (size_t)j * N + col);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double cr = __ldg(xr + (size_t)r * Nb + j), ci = __ldg(xi + (size_t)r * Nb + j);
            ar[r] = fma(cr, br, fma(-ci, bi, ar[r]));
            ai[r] = fma(cr, bi, fma(ci, br, ai[r]));
        }
    }
    if (i >= N) return;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const double s = scale ? scale[k0 + r] : 1.0;
        ore[(size_t)(k0 + r) * N + i] = s * ar[r];
        oim[(size_t)(k0 + r) * N + i] = s * ai[r];
    }
}

__global__ void __launch_bounds__(kRb64Threads)
k_rb_fp64(const double *__restrict__ are, const double *__restrict__ aim, const double *__restrict__ bre,
          const double *__restrict__ bim, int M, int Nb, int N, const double *__restrict__ scale,
          double *__restrict__ ore, double *__restrict__ oim)
{
    const int cols = (N + kRb64Threads - 1) / kRb64Threads, groups = (M + kRb64Max - 1) / kRb64Max;
    const int g = blockIdx.x / cols, i = (blockIdx.x % cols) * kRb64Threads + threadIdx.x;
    if ((i & ~31) >= N) return;  // a whole warp past the last mode
    const int k0 = (int)((long long)M * g / groups), rows = (int)((long long)M * (g + 1) / groups) - k0;
    switch (rows) {
    case 1: rb64_rows<1>(are, aim, bre, bim, k0, i, Nb, N, scale, ore, oim); break;
    case 2: rb64_rows<2>(are, aim, bre, bim, k0, i, Nb, N, scale, ore, oim); break;
    case 3: rb64_rows<3>(are, aim, bre, bim, k0, i, Nb, N, scale, ore, oim); break;
    case 4: rb64_rows<4>(are, aim, bre, bim, k0, i, Nb, N, scale, ore, oim); break;
    case 5: rb64_rows<5>(are, aim, bre, bim, k0, i, Nb, N, scale, ore, oim); break;
    case 6: rb64_rows<6>(are, aim, bre, bim, k0, i, Nb, N, scale, ore, oim); break;
    case 7: rb64_rows<7>(are, aim, bre, bim, k0, i, Nb, N, scale, ore, oim); break;
    case 8: rb64_rows<8>(are, aim, bre, bim, k0, i, Nb, N, scale, ore, oim); break;
    default: break;
    }
}

// The renormalisation of the FP64 path, one block per knot: q_k = sum_jl Re(alpha_j G_jl conj(alpha_l)), s_k =
// nu_k / sqrt(q_k).  G is Hermitian: with the rows in groups of at most 32, a warp a group, a group's
// square of G counts once and what is left of it twice.  Four sets of warps share the columns, for
// loads in flight; partial sums are added in order.  (FP64 pipe: 100 knots of 99 vectors 35 us as one
// set over whole rows, bound by the loads' latency; 19 us so.)
constexpr int kScaleSets = 4;

__global__ void __launch_bounds__(FEW_MAX_BASIS * kScaleSets)
k_rb_scale64(const double *__restrict__ are, const double *__restrict__ aim, int Nb, int groups,
             const double2 *__restrict__ gt, const double *__restrict__ nu,
             double *__restrict__ scale, unsigned *__restrict__ err)
{
    __shared__ double2 a[FEW_MAX_BASIS];
    __shared__ double part[FEW_MAX_BASIS / 32 * kScaleSets];
    pdl_launch_dependents();  // the pack, if it is launched so
    const int k = blockIdx.x, tid = threadIdx.x, w = tid >> 5, group = w % groups, set = w / groups;
    for (int j = tid; j < Nb; j += blockDim.x) a[j] = make_double2(are[(size_t)k * Nb + j], aim[(size_t)k * Nb + j]);
    __syncthreads();
    const int rows = (Nb + groups - 1) / groups, first = group * rows, end = min(first + rows, Nb);
    const int j = first + (tid & 31), jj = min(j, Nb - 1);
    double q = 0.0;
#pragma unroll
    for (int twice = 1; twice >= 0; --twice) {  // the columns before the group's own, then those
        const int l1 = twice ? first : end;
        double tr[2] = {0.0, 0.0}, ti[2] = {0.0, 0.0};
#pragma unroll 4
        for (int l = (twice ? 0 : first) + set, i = 0; l < l1; l += kScaleSets, ++i) {
            const double2 g = __ldg(gt + (size_t)l * Nb + jj), x = a[l];
            tr[i & 1] = fma(g.x, x.x, fma(g.y, x.y, tr[i & 1]));
            ti[i & 1] = fma(g.y, x.x, fma(-g.x, x.y, ti[i & 1]));
        }
        if (j < end) {
            const double p = a[j].x * (tr[0] + tr[1]) - a[j].y * (ti[0] + ti[1]);
            q += twice ? 2.0 * p : p;
        }
    }
    for (int o = 16; o > 0; o >>= 1) q += __shfl_down_sync(0xffffffffu, q, o);
    if ((tid & 31) == 0) part[w] = q;
    __syncthreads();
    if (tid == 0) {
        q = 0.0;
        for (int i = 0; i < (int)blockDim.x / 32; ++i) q += part[i];
        const double v = nu[k];
        if (!(v >= 0.0) || !isfinite(v)) atomicOr(err, ERRBIT_NONFINITE);
        scale[k] = q > 0.0 ? v / sqrt(q) : 0.0;
    }
}

// ---- launchers ----------------------------------------------------------------------------

RbLayout rb_layout(int Nb, int N, int M)
{
    RbLayout L;
    L.n_kb = (kRbParts * 2 * Nb + kRbTileK - 1) / kRbTileK;
    // whole sectors: 28 modes of each group (N a multiple of four: every row is aligned alike, all 32)
    L.step = N % 4 ? 28 : 32;
    L.groups = N <= 32 ? 1 : (N - (32 - L.step) + L.step - 1) / L.step;
    L.n_tiles = (L.groups + 1) / 2;
    L.m_tiles = (M + kRbTileN - 1) / kRbTileN;
    L.modes_padded = (2 * L.n_tiles - 1) * L.step + 32;
    L.rows_padded = L.m_tiles * kRbTileN;
    L.bpack_bytes = (size_t)L.n_tiles * L.n_kb * kRbABytes;
    L.apack_bytes = (size_t)L.m_tiles * L.n_kb * kRbBBytes;
    return L;
}

cudaError_t launch_rb_basis(const double *bre, const double *bim, int Nb, int N, double2 *gt64,
                            float2 *gt32, const int *bexp, unsigned char *bpack, int sm_count, cudaStream_t st)
{
    const RbLayout L = rb_layout(Nb, N, 0);
    k_rb_gram<<<Nb * Nb, 128, 0, st>>>(bre, bim, Nb, N, gt64, gt32);
    k_rb_pack_b<<<sm_count * 8, 256, 0, st>>>(bre, bim, Nb, N, L.n_kb, L.n_tiles, L.step, bexp, bpack);
    return cudaGetLastError();
}

cudaError_t launch_rb(const double *are, const double *aim, int M, int Nb, int N, const double *nu,
                      bool fp64, const double *bre, const double *bim, const double2 *gt64,
                      const float2 *gt32, const int *bexp, const unsigned char *bpack, double *scale,
                      int *aexp, unsigned char *apack, const int *bexp64, const unsigned char *bpack64,
                      double *ore, double *oim, unsigned *err,
                      int sm_count, cudaStream_t st, cudaStream_t side, cudaEvent_t fork_ev,
                      cudaEvent_t join_ev)
{
    if (M == 0) return cudaSuccess;
    const RbLayout L = rb_layout(Nb, N, M);
    cudaError_t e;
    const double *sc = nullptr;
    // mixed path: the scale is applied in the product's epilogue, so its kernels run beside the
    // coefficient pack: the one-kernel form (Nb <= 128) lets the pack start with it and the product
    // with the pack's end (dependent launches; 1,486 knots of 60 vectors and 279 modes 37.6 -> 21.5 us
    // without the side stream's two events), the longer one runs on a side stream
    const bool tile = nu && !fp64 && Nb <= kTMaxBasis;
    const bool fork = nu && !fp64 && !tile && side;
    cudaStream_t ss = fork ? side : st;
    if (fork) {
        if ((e = cudaEventRecord(fork_ev, st)) != cudaSuccess) return e;
        if ((e = cudaStreamWaitEvent(side, fork_ev, 0)) != cudaSuccess) return e;
    }
    // a failure after the fork waits for the side stream, so nothing of it outlives the call's
    // scratch, which the caller releases on `st`
    auto fail = [&](cudaError_t err) {
        if (fork) cudaStreamSynchronize(side);
        return err;
    };
    if (tile) {
        using Kernel = void (*)(const double *, const double *, int, int, const float2 *, const double *, double *,
                                unsigned *);
        static const Kernel kernels[8] = {k_rb_scale_tile<1>, k_rb_scale_tile<2>, k_rb_scale_tile<3>,
                                          k_rb_scale_tile<4>, k_rb_scale_tile<5>, k_rb_scale_tile<6>,
                                          k_rb_scale_tile<7>, k_rb_scale_tile<8>};
        const int T = (Nb + 15) / 16, smem = (kTRows * Nb + Nb * 16 * T) * (int)sizeof(float2);
        const Kernel k = kernels[T - 1];
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (kTRows + kTMaxBasis) * kTMaxBasis * (int)sizeof(float2));
        if (e != cudaSuccess) return e;
        k<<<(M + kTRows - 1) / kTRows, kTThreads, smem, st>>>(are, aim, M, Nb, gt32, nu, scale, err);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        sc = scale;
    } else if (nu && fp64) {
        const int groups = (Nb + 31) / 32;
        k_rb_scale64<<<M, 32 * groups * kScaleSets, 0, ss>>>(are, aim, Nb, groups, gt64, nu, scale, err);
        // (launch_rb64's pack leans on this launch: see launch.cuh)
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        sc = scale;
    } else if (nu) {
        double *q = scale + M;  // the caller's scratch holds scale [M] then q [M]
        e = cudaMemsetAsync(q, 0, sizeof(double) * (size_t)M, ss);
        if (e != cudaSuccess) return fail(e);
        const dim3 grid((Nb + kQJ - 1) / kQJ, (M + kQRows - 1) / kQRows);
        e = cudaFuncSetAttribute(k_rb_quad, cudaFuncAttributeMaxDynamicSharedMemorySize, kQSmem);
        if (e != cudaSuccess) return fail(e);
        k_rb_quad<<<grid, kQThreads, kQSmem, ss>>>(are, aim, M, Nb, gt32, q);
        k_rb_norm<<<(M + 255) / 256, 256, 0, ss>>>(q, nu, M, scale, err);
        if ((e = cudaGetLastError()) != cudaSuccess) return fail(e);
        sc = scale;
    }
    if (fork && (e = cudaEventRecord(join_ev, side)) != cudaSuccess) return fail(e);
    if (fp64 && bpack64) {  // (the plain chain: a context without room for the digits)
        Rb64Args a{};
        a.bpack = bpack64;
        a.bexp = bexp64;
        a.are = are;
        a.aim = aim;
        a.bre = bre;
        a.bim = bim;
        a.out_re = ore;
        a.out_im = oim;
        a.M = M;
        a.N = N;
        a.Nb = Nb;
        a.err = err;
        a.scale = sc;
        return launch_rb64(a, apack, aexp, sc != nullptr, st);
    }
    if (fp64) {
        const unsigned grid = (unsigned)((N + kRb64Threads - 1) / kRb64Threads) *
                              (unsigned)((M + kRb64Max - 1) / kRb64Max);
        k_rb_fp64<<<grid, kRb64Threads, 0, st>>>(are, aim, bre, bim, M, Nb, N, sc, ore, oim);
        return cudaGetLastError();
    }
    const int rows = L.m_tiles * kRbTileN;
    const int pgrid = (rows + kRbPackWarps - 1) / kRbPackWarps;
    const unsigned pblocks = pgrid < sm_count * 8 ? pgrid : sm_count * 8;
    if (tile) {  // beside the scale's kernel, whose plain launch it leans on (launch.cuh)
        e = launch_pdl(k_rb_pack_a, pblocks, kRbPackWarps * 32, 0, st, are, aim, M, Nb, L.n_kb, L.m_tiles, apack,
                       aexp);
    } else {
        k_rb_pack_a<<<pblocks, kRbPackWarps * 32, 0, st>>>(are, aim, M, Nb, L.n_kb, L.m_tiles, apack, aexp);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return fail(e);
    if (fork && (e = cudaStreamWaitEvent(st, join_ev, 0)) != cudaSuccess) return fail(e);
    const int smem = kRbStages * (int)kRbStageBytes + 128;
    e = cudaFuncSetAttribute(k_rb_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const int tiles = L.m_tiles * L.n_tiles;
    const int k_last = kRbParts * 2 * Nb - (L.n_kb - 1) * kRbTileK;  // real columns, last block
    RbMmaArgs args{apack, bpack, ore, oim, aexp, bexp, sc, M, N, L.n_kb, L.m_tiles, L.n_tiles, L.groups, L.step,
                   (k_last + 15) / 16, err};
    // (small calls: a CTA for each part of a tile)
    const int blocks = tiles * 8 < sm_count ? tiles * 8 : sm_count;
    if (!fork) return launch_pdl(k_rb_mma, blocks, kRbMmaThreads, smem, st, args);
    k_rb_mma<<<blocks, kRbMmaThreads, smem, st>>>(args);
    return cudaGetLastError();
}

}  // namespace fewsum
