// direct.cu -- direct (non-interpolated) mode summation (arXiv:2104.04582 Sec. 3.C).
//
// The "more basic" summation of the paper: the phases and every mode's amplitude are given at
// the output's own sample density, so there is no spline; at each sample i
//     h_i = scale * sum_modes [ A_i Y+ e^{-i Phi_mn,i} + (m > 0) conj(A_i) Y- e^{+i Phi_mn,i} ],
// Phi_mn,i = m Phi_phi,i + n Phi_r,i, Y+ = -2Y_lm, Y- = (-1)^l -2Y_{l,-m}  (Eq. amp_symmetry).
//
// Each mode-sample reads 16 bytes of FP64 amplitude and nothing is reused across samples, so in
// mixed precision the kernel is bound by HBM bandwidth (FP64 arithmetic throughout is bound by
// the FP64 pipe instead).  One warp per sample: lanes stride over the modes (coalesced reads of
// the [sample][mode] arrays, several loads in flight per lane), each lane forms its modes'
// exponentials from the sample's reduced phases (FP64 reduction of Phi_phi and Phi_r modulo 2 pi,
// then the sine and cosine of the reduced integer combination), and the warp reduces its partial
// sums with shuffles.
#include <type_traits>

#include <cuda_fp16.h>

#include "async.cuh"
#include "fewsum_internal.h"
#include "launch.cuh"
#include "harmonics.cuh"
#include "phase_eval.cuh"
#include "convert.cuh"

namespace fewsum {

// Per-mode constants in the arithmetic type of the path.  With Y+ = -2Y_lm and
// Y- = (-1)^l -2Y_{l,-m} (zero for m = 0), a mode contributes
//     A Y+ e^{-i Phi} + conj(A) Y- e^{+i Phi}
//   = Re A [ (a c + b s) + i (g c - d s) ] + Im A [ (a s - b c) + i (d c + g s) ],
// c = cos Phi, s = sin Phi, with a = Re(Y+ + Y-), b = Im(Y+ - Y-), g = Im(Y+ + Y-),
// d = Re(Y+ - Y-).  The record is 16-byte aligned so a lane fetches it in wide loads.
template <typename T>
struct alignas(16) ModeConst {
    T a, b, g, d;
    T m, n;
};

template <typename T>
__global__ void k_mode_consts(const int *__restrict__ l, const int *__restrict__ m,
                              const int *__restrict__ n, int N, double theta, double phi,
                              ModeConst<T> *__restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double2 yp = swsh_m2(l[i], m[i], theta, phi);
    double2 ym = make_double2(0.0, 0.0);
    if (m[i] > 0) {
        ym = swsh_m2(l[i], -m[i], theta, phi);
        if (l[i] & 1) ym = make_double2(-ym.x, -ym.y);
    }
    ModeConst<T> c;
    c.a = (T)(yp.x + ym.x); c.b = (T)(yp.y - ym.y);
    c.g = (T)(yp.y + ym.y); c.d = (T)(yp.x - ym.x);
    c.m = (T)m[i]; c.n = (T)n[i];
    out[i] = c;
}

// Amplitude conversion of the arithmetic path: the mixed path uses the branchless integer-pipe
// conversion (ties away from zero, below 2^-126 flushed, from 2^128 up given as infinity): the
// exact even-tie conversion costs about 15 integer operations per value and bounded this kernel.
__device__ __forceinline__ double to_t(double v, double) { return v; }
__device__ __forceinline__ float to_t(double v, float) { return f64_to_f32_fast(v); }

// Nearest integer of |x| < 2^22 by the 1.5 * 2^23 addition (FP32 add pipe); FP64 uses rint.
__device__ __forceinline__ float round_near(float x)
{
    const float k = 12582912.0f;
    return (x + k) - k;
}
__device__ __forceinline__ double round_near(double x) { return rint(x); }

// Exponential of the reduced phase ph (turns, |ph| <= 1/2): FP64 sincospi for the plain path;
// for the mixed path the SFU sine and cosine of 2 pi ph (|x| <= pi, absolute error below 1e-6).
__device__ __forceinline__ void expi_turns(double ph, double *s, double *c) { sincospi(2.0 * ph, s, c); }
__device__ __forceinline__ void expi_turns(float ph, float *s, float *c)
{
    __sincosf(6.283185307179586f * ph, s, c);
}

constexpr int kDirectUnroll = 8;  // amplitude loads in flight per lane before any arithmetic

template <typename T>
__global__ void __launch_bounds__(256)
k_direct(const double *__restrict__ pphi, const double *__restrict__ pr,
         const double *__restrict__ are, const double *__restrict__ aim, long long ns, int N,
         const ModeConst<T> *__restrict__ mc, double scale, void *__restrict__ out, int out_c64)
{
    const double kInv2Pi = 0.15915494309189533577;
    const int lane = threadIdx.x & 31;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long i = warp; i < ns; i += nwarps) {
        const double xp = reduce_2pi(pphi[i]) * kInv2Pi, xr = reduce_2pi(pr[i]) * kInv2Pi;
        const T fphi = (T)(xp - rint(xp)), fr = (T)(xr - rint(xr));
        const double *ar = are + (size_t)i * N, *ai = aim + (size_t)i * N;
        T hr = 0, hi = 0;
        for (int j0 = lane; j0 < N; j0 += 32 * kDirectUnroll) {
            double vr[kDirectUnroll], vi[kDirectUnroll];
#pragma unroll
            for (int u = 0; u < kDirectUnroll; ++u) {
                const int j = j0 + 32 * u;
                vr[u] = j < N ? __ldcs(ar + j) : 0.0;  // streamed once: evict-first
                vi[u] = j < N ? __ldcs(ai + j) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < kDirectUnroll; ++u) {
                const int j = j0 + 32 * u;
                if (j >= N) break;
                const ModeConst<T> c = mc[j];
                const T Ar = to_t(vr[u], T()), Ai = to_t(vi[u], T());
                T ph = c.m * fphi + c.n * fr;
                ph -= round_near(ph);
                T s, co;
                expi_turns(ph, &s, &co);
                hr += Ar * (c.a * co + c.b * s) + Ai * (c.a * s - c.b * co);
                hi += Ar * (c.g * co - c.d * s) + Ai * (c.d * co + c.g * s);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            hr += __shfl_down_sync(0xffffffffu, hr, o);
            hi += __shfl_down_sync(0xffffffffu, hi, o);
        }
        if (lane == 0) {
            const double vr0 = (double)hr * scale, vi0 = (double)hi * scale;
            if (out_c64)
                reinterpret_cast<float2 *>(out)[i] = make_float2((float)vr0, (float)vi0);
            else
                reinterpret_cast<double2 *>(out)[i] = make_double2(vr0, vi0);
        }
    }
}

// FP64 with exponential tables.  The plain path is bound by the FP64 pipe, and sincospi per mode
// and sample was most of it (~60 of ~75 FP64 operations).  A mode list has few distinct m and n
// (11 + 31 against 1953 modes on the |n| <= 15 grid), so each warp first fills a table of
// e^{i m Phi_phi} (m = 0 .. m_top) and e^{i n Phi_r} (n_lo .. n_hi) for its sample in shared
// memory, and a mode costs 12 FP64 operations: e^{i Phi} = the product of two entries, w = A
// e^{-i Phi}, and
//     h += w Y+ + conj(w) Y- = [a Re w - b Im w] + i [g Re w + d Im w]   (a, b, g, d as above).
// kPairs: the factor of (l, m) is formed once per sample too, in a table over (l, m): with v = A e^{-i n
// Phi_r}, c = cos m Phi_phi, s = sin m Phi_phi,
//     h += [(a c + b s) Re v - (b c - a s) Im v] + i [(g c - d s) Re v + (d c + g s) Im v],
// and a mode costs 8 operations.
// Small blocks (4 samples), so that the last wave is spread evenly.  4001 samples x 1953 modes: 814 us
// with sincospi per mode, 245 with the exponentials' tables, 182 with kPairs.
constexpr int kTabThreads = 128;
constexpr int kTabMaxBytes = 12 * 1024;  // a warp, with kPairs
constexpr int kTabMaxEntries = 512;  // (m_top + 1) + (n_hi - n_lo + 1): 8 KB a warp

struct alignas(16) ModeConstTab {
    double a, b, g, d;
    int m, n, pad[2];  // table entries of m and n
};
struct alignas(16) PairConst64 {
    double a, b, g, d;
};

__global__ void k_mode_consts_tab(const int *__restrict__ l, const int *__restrict__ m,
                                  const int *__restrict__ n, int N, double theta, double phi,
                                  int m_top, int n_lo, ModeConstTab *__restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double2 yp = swsh_m2(l[i], m[i], theta, phi);
    double2 ym = make_double2(0.0, 0.0);
    if (m[i] > 0) {
        ym = swsh_m2(l[i], -m[i], theta, phi);
        if (l[i] & 1) ym = make_double2(-ym.x, -ym.y);
    }
    out[i] = ModeConstTab{yp.x + ym.x, yp.y - ym.y, yp.y + ym.y, yp.x - ym.x,
                          m[i], m_top + 1 + n[i] - n_lo, {0, 0}};
}

// kPairs: the constants of every (l, m), record (l - 2) (m_top + 1) + m, and each mode's record and n.
__global__ void k_pair_consts(const int *__restrict__ l, const int *__restrict__ m, const int *__restrict__ n, int N,
                              double theta, double phi, int l_top, int m_top, int n_lo, int2 *__restrict__ modes,
                              PairConst64 *__restrict__ pairs)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) modes[i] = make_int2((l[i] - 2) * (m_top + 1) + m[i], m_top + 1 + n[i] - n_lo);
    if (i >= (l_top - 1) * (m_top + 1)) return;
    const int li = 2 + i / (m_top + 1), mi = i % (m_top + 1);
    if (mi > li) {  // no such mode
        pairs[i] = PairConst64{};
        return;
    }
    const double2 yp = swsh_m2(li, mi, theta, phi);
    double2 ym = make_double2(0.0, 0.0);
    if (mi > 0) {
        ym = swsh_m2(li, -mi, theta, phi);
        if (li & 1) ym = make_double2(-ym.x, -ym.y);
    }
    pairs[i] = PairConst64{yp.x + ym.x, yp.y - ym.y, yp.y + ym.y, yp.x - ym.x};
}

// The n from which the table's exponentials are computed up (0: and mirrored), and how many there are.
__host__ __device__ inline int tab_first(int n_lo, int n_hi) { return n_lo < 0 && n_hi > 0 ? 0 : n_lo; }
__host__ __device__ inline int tab_count(int m_top, int n_lo, int n_hi)
{
    const int a0 = tab_first(n_lo, n_hi), a1 = a0 == 0 && -n_lo > n_hi ? -n_lo : n_hi;
    return m_top + 2 + a1 - a0;
}

// tables: the modes' ModeConstTab, or (kPairs) n_pairs PairConst64, then int2 per mode.
template <bool kPairs>
__global__ void __launch_bounds__(kTabThreads)
k_direct_tab(const double *__restrict__ pphi, const double *__restrict__ pr,
             const double *__restrict__ are, const double *__restrict__ aim, long long ns, int N,
             const void *__restrict__ tables, int n_pairs, int m_top, int n_lo, int entries, double scale,
             void *__restrict__ out, int out_c64)
{
    extern __shared__ __align__(16) double2 dir_tab[];
    const double kInv2Pi = 0.15915494309189533577;
    const int lane = threadIdx.x & 31;
    const long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;  // sample
    if (i >= ns) return;  // a whole warp
    double2 *tab = dir_tab + (threadIdx.x >> 5) * (entries + (kPairs ? 2 * n_pairs : 0));
    const double xp = reduce_2pi(pphi[i]) * kInv2Pi, xr = reduce_2pi(pr[i]) * kInv2Pi;
    const double fphi = xp - rint(xp), fr = xr - rint(xr);
    // (of n and -n one is computed: the table of a range about zero takes half the sincospi; lanes past the end
    // repeat the last entry: lanes a pass apart went through the unrolled loop one group after the other, 64
    // modes of 33 exponentials, 60,000 samples: 580 us, 458 so)
    const int n_hi = n_lo + entries - m_top - 2, a0 = tab_first(n_lo, n_hi), count = tab_count(m_top, n_lo, n_hi);
    for (int e0 = 0; e0 < count; e0 += 32) {
        const int e = min(e0 + lane, count - 1), a = a0 + e - m_top - 1;
        const double x = e <= m_top ? e * fphi : (double)a * fr;
        double s, c;
        sincospi(2.0 * (x - rint(x)), &s, &c);
        if (e <= m_top || a <= n_hi) tab[e <= m_top ? e : m_top + 1 + a - n_lo] = make_double2(c, s);
        if (e > m_top && a0 == 0 && -a >= n_lo) tab[m_top + 1 - a - n_lo] = make_double2(c, -s);
    }
    __syncwarp();
    const double *ar = are + (size_t)i * N, *ai = aim + (size_t)i * N;
    double hr = 0.0, hi = 0.0;
    if constexpr (kPairs) {
        const PairConst64 *pc = static_cast<const PairConst64 *>(tables);
        const int2 *md = reinterpret_cast<const int2 *>(pc + n_pairs);
        double2 *fac = tab + entries;
        for (int p = lane; p < n_pairs; p += 32) {
            const PairConst64 y = pc[p];
            const double2 e = tab[p % (m_top + 1)];
            fac[2 * p] = make_double2(fma(y.a, e.x, y.b * e.y), fma(y.b, e.x, -y.a * e.y));
            fac[2 * p + 1] = make_double2(fma(y.g, e.x, -y.d * e.y), fma(y.d, e.x, y.g * e.y));
        }
        __syncwarp();
#pragma unroll 4
        for (int j = lane; j < N; j += 32) {
            const double vr = __ldcs(ar + j), vi = __ldcs(ai + j);
            const int2 k = md[j];
            const double2 q = tab[k.y], f = fac[2 * k.x], g = fac[2 * k.x + 1];
            const double wr = fma(vr, q.x, vi * q.y), wi = fma(vi, q.x, -vr * q.y);
            hr = fma(wr, f.x, fma(-wi, f.y, hr));
            hi = fma(wr, g.x, fma(wi, g.y, hi));
        }
    } else {
        const ModeConstTab *mc = static_cast<const ModeConstTab *>(tables);
#pragma unroll 4
        for (int j = lane; j < N; j += 32) {
            const double vr = __ldcs(ar + j), vi = __ldcs(ai + j);
            const double2 y0 = *reinterpret_cast<const double2 *>(&mc[j].a);
            const double2 y1 = *reinterpret_cast<const double2 *>(&mc[j].g);
            const int2 mn = *reinterpret_cast<const int2 *>(&mc[j].m);
            const double2 p = tab[mn.x], q = tab[mn.y];
            const double co = fma(p.x, q.x, -p.y * q.y), s = fma(p.y, q.x, p.x * q.y);
            const double wr = fma(vr, co, vi * s), wi = fma(vi, co, -vr * s);
            hr = fma(wr, y0.x, fma(-wi, y0.y, hr));
            hi = fma(wr, y1.x, fma(wi, y1.y, hi));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        hr += __shfl_down_sync(0xffffffffu, hr, o);
        hi += __shfl_down_sync(0xffffffffu, hi, o);
    }
    if (lane == 0) {
        if (out_c64)
            reinterpret_cast<float2 *>(out)[i] = make_float2((float)(hr * scale), (float)(hi * scale));
        else
            reinterpret_cast<double2 *>(out)[i] = make_double2(hr * scale, hi * scale);
    }
}

// Mixed precision with the amplitudes streamed through shared memory.  The kernel is bound by HBM, and a
// warp of k_direct that holds its loads in registers has none in flight while it computes.  Here every
// warp keeps a ring of three chunks (256 modes of one sample, 4 KB) filled by bulk copies, two of them on
// the way while it works on the third: 130 KB in flight on each multiprocessor, no barrier between
// warps.  The ring leaves L1 too small for 32 bytes of constants per mode (four times the amplitudes'
// bytes), but Y+ and Y- belong to (l, m), not to n: a word per mode (its (l, m), n) and a record per
// (l, m), which a warp's 32 modes mostly share, fit in shared memory beside the ring.
// A copy starts and ends on 16-byte boundaries, so it may take a neighbouring element with it; a chunk
// for which that would lie outside the arrays is read directly.  At four warps a scheduler instruction
// issue comes next: amplitudes that are normal FP32 numbers take a four-instruction conversion, a mode
// 36 instructions, and a lane forms the phases of one of the next 32 samples (FP64 work that every lane
// did for every sample: half the time of 132-mode calls).
// 100,000 samples x 3843 modes: see launch_direct for both sides.
constexpr int kRingWarps = 16, kRingStages = 3, kRingModes = 256;
constexpr int kRingRow = (kRingModes + 2) * (int)sizeof(double);  // one component of a chunk
constexpr int kRingBytes = kRingWarps * kRingStages * 2 * kRingRow;
constexpr int kRingTables = 32 * 1024;  // words and records beside the ring

struct alignas(16) PairConst {
    float a, b, g, d;  // as ModeConst
    float m, pad[3];
};

__host__ __device__ inline int ring_table_bytes(int N, int pairs)
{
    return ((N * (int)sizeof(unsigned) + 15) & ~15) + pairs * (int)sizeof(PairConst);
}

// The tables: (l, m) is record (l - 2) (m_top + 1) + m; a word is the record's place in bytes (later its address) and n in fp16
// (exact: |n| <= 1024).
__global__ void k_mode_words(const int *__restrict__ l, const int *__restrict__ m, const int *__restrict__ n, int N,
                             double theta, double phi, int l_top, int m_top, unsigned *__restrict__ words,
                             PairConst *__restrict__ pairs)
{
    pdl_launch_dependents();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N)
        words[i] = (unsigned)(((l[i] - 2) * (m_top + 1) + m[i]) * (int)sizeof(PairConst)) |
                   (unsigned)__half_as_ushort(__int2half_rn(n[i])) << 16;
    if (i >= (l_top - 1) * (m_top + 1)) return;
    const int li = 2 + i / (m_top + 1), mi = i % (m_top + 1);
    if (mi > li) return;  // no such mode
    const double2 yp = swsh_m2(li, mi, theta, phi);
    double2 ym = make_double2(0.0, 0.0);
    if (mi > 0) {
        ym = swsh_m2(li, -mi, theta, phi);
        if (li & 1) ym = make_double2(-ym.x, -ym.y);
    }
    pairs[i] = PairConst{(float)(yp.x + ym.x), (float)(yp.y - ym.y), (float)(yp.y + ym.y), (float)(yp.x - ym.x),
                         (float)mi, {}};
}

__global__ void __launch_bounds__(32 * kRingWarps, 1)
k_direct_ring(const double *__restrict__ pphi, const double *__restrict__ pr, const double *__restrict__ are,
              const double *__restrict__ aim, long long ns, int N, const uint4 *tables, int table_bytes,
              double scale, void *__restrict__ out, int out_c64, unsigned *__restrict__ err)
{
    extern __shared__ __align__(16) unsigned char ring_smem[];
    __shared__ __align__(8) uint64_t full[kRingWarps][kRingStages];
    const double kInv2Pi = 0.15915494309189533577;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the tables (a word's record as its address in shared memory), then the warps' rings
    const int word_uints = (N + 3) & ~3;
    const unsigned recs = smem_u32(ring_smem) + 4u * word_uints;
    unsigned char *ring = ring_smem + table_bytes + warp * kRingStages * 2 * kRingRow;
    uint64_t *bar = full[warp];
    if (lane == 0) {
        for (int s = 0; s < kRingStages; ++s) mbar_init(&bar[s], 1);
        fence_mbar_init();
    }
    // this warp's samples, spread over the multiprocessors first
    const long long first = (long long)warp * gridDim.x + blockIdx.x, step = (long long)kRingWarps * gridDim.x;
    const int chunks = (N + kRingModes - 1) / kRingModes, tail = N - (chunks - 1) * kRingModes;
    const long long items = first < ns ? ((ns - 1 - first) / step + 1) * chunks : 0;
    // an item is copied unless its 16-byte units reach before the arrays' start or past their end
    const uintptr_t end = sizeof(double) * (uintptr_t)ns * (uintptr_t)N;
    const bool skip0 = first == 0 && ((reinterpret_cast<uintptr_t>(are) | reinterpret_cast<uintptr_t>(aim)) & 8);
    const bool skip1 = (ns - 1 - first) % step == 0 &&
                       (((reinterpret_cast<uintptr_t>(are) + end) | (reinterpret_cast<uintptr_t>(aim) + end)) & 8);
    auto copied = [&](long long it) { return !(it == 0 && skip0) && !(it + 1 == items && skip1); };
    const uint64_t once = l2_evict_first_policy();
    // the next item to fill (one lane): address of its first elements and its chunk
    const long long row0 = sizeof(double) * first * N;
    uintptr_t fa = reinterpret_cast<uintptr_t>(are) + row0;
    const intptr_t other = reinterpret_cast<intptr_t>(aim) - reinterpret_cast<intptr_t>(are);
    const long long next_row = (long long)sizeof(double) * (step * N - (long long)(chunks - 1) * kRingModes);
    long long filled = 0;
    int fc = 0;
    auto fill = [&](int s) {
        if (filled == items) return;
        const bool last = ++fc == chunks;
        if (copied(filled)) {
            const uint32_t len = (uint32_t)(last ? tail : kRingModes) * 8u;
            const uintptr_t sa = fa & ~(uintptr_t)15, sb = (fa + other) & ~(uintptr_t)15;
            const uint32_t la = (uint32_t)(fa & 8) + len + 15 & ~15u, lb = (uint32_t)((fa + other) & 8) + len + 15 & ~15u;
            mbar_arrive_expect_tx(&bar[s], la + lb);
            bulk_g2s_hint(ring + 2 * s * kRingRow, reinterpret_cast<const void *>(sa), la, &bar[s], once);
            bulk_g2s_hint(ring + (2 * s + 1) * kRingRow, reinterpret_cast<const void *>(sb), lb, &bar[s], once);
        } else {
            mbar_arrive(&bar[s]);
        }
        fa += last ? next_row : (long long)(8 * kRingModes);
        if (last) fc = 0;
        ++filled;
    };
    if (lane == 0)
        for (int s = 0; s < kRingStages; ++s) fill(s);
    pdl_wait();  // the tables (the amplitudes were there before their kernel)
    for (int i = threadIdx.x; i < table_bytes / 16; i += blockDim.x) {
        uint4 v = tables[i];
        if (4 * i < word_uints) {
            v.x += recs;
            v.y += recs;
            v.z += recs;
            v.w += recs;
        }
        reinterpret_cast<uint4 *>(ring_smem)[i] = v;
    }
    __syncthreads();
    if (items == 0) return;
    long long i = first;
    int c = 0, s = 0;
    uint32_t parity = 0;
    float fphi = 0.0f, fr = 0.0f, hr = 0.0f, hi = 0.0f;
    float vphi = 0.0f, vr = 0.0f;  // phases of 32 samples, one a lane
    int ahead = 0;                 // of them, used
    bool ok = true;
    for (long long it = 0; it < items; ++it) {
        if (c == 0) {
            if (ahead == 0) {
                const long long mine = i + lane * step;
                const double xp = reduce_2pi(pphi[mine < ns ? mine : i]) * kInv2Pi;
                const double xr = reduce_2pi(pr[mine < ns ? mine : i]) * kInv2Pi;
                vphi = (float)(xp - rint(xp));
                vr = (float)(xr - rint(xr));
            }
            fphi = __shfl_sync(0xffffffffu, vphi, ahead);
            fr = __shfl_sync(0xffffffffu, vr, ahead);
            ahead = (ahead + 1) & 31;
            hr = hi = 0.0f;
        }
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(&bar[s], parity));
        if (!ok) break;
        const size_t at = (size_t)i * N + (size_t)c * kRingModes;
        const int left = N - c * kRingModes - lane;  // modes of the chunk from this lane's first on
        const unsigned *wp = reinterpret_cast<const unsigned *>(ring_smem) + c * kRingModes + lane;
        constexpr int U = kRingModes / 32;
        auto sum = [&](auto whole, const double *ra, const double *rb) {
            constexpr bool kWhole = decltype(whole)::value;  // every lane has all its modes
            double va[U], vb[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                va[u] = kWhole || 32 * u < left ? ra[32 * u] : 1.0;
                vb[u] = kWhole || 32 * u < left ? rb[32 * u] : 1.0;
            }
            float xa[U], xb[U];
            bool odd = false;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                xa[u] = f64_normal_to_f32(va[u]);
                xb[u] = f64_normal_to_f32(vb[u]);
                odd |= !f64_is_f32_normal(va[u]);
                odd |= !f64_is_f32_normal(vb[u]);
            }
            if (odd) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    xa[u] = f64_to_f32_fast(va[u]);
                    xb[u] = f64_to_f32_fast(vb[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (!kWhole && 32 * u >= left) break;
                const unsigned w = wp[32 * u];
                float ka, kb, kg, kd, km;  // the record
                asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(ka), "=f"(kb), "=f"(kg), "=f"(kd) : "r"(w & 0xffffu));
                asm("ld.shared.f32 %0, [%1 + 16];" : "=f"(km) : "r"(w & 0xffffu));
                const float n = __half2float(__ushort_as_half((unsigned short)(w >> 16)));
                float ph = fmaf(n, fr, km * fphi);
                ph -= round_near(ph);
                float sn, co;
                expi_turns(ph, &sn, &co);
                // A e^{-i Phi}
                const float wr = fmaf(xb[u], sn, xa[u] * co), wi = fmaf(xb[u], co, -xa[u] * sn);
                hr += fmaf(ka, wr, -(kb * wi));  // (one rounding at the sum's size)
                hi += fmaf(kg, wr, kd * wi);
            }
        };
        if (copied(it)) {
            const uintptr_t pa = reinterpret_cast<uintptr_t>(are) + 8 * at, pb = reinterpret_cast<uintptr_t>(aim) + 8 * at;
            const double *ra = reinterpret_cast<const double *>(ring + 2 * s * kRingRow + (pa & 8)) + lane;
            const double *rb = reinterpret_cast<const double *>(ring + (2 * s + 1) * kRingRow + (pb & 8)) + lane;
            if (c + 1 < chunks || tail == kRingModes)
                sum(std::true_type(), ra, rb);
            else
                sum(std::false_type(), ra, rb);
        } else {
            sum(std::false_type(), are + at + lane, aim + at + lane);
        }
        __syncwarp();  // the chunk has been read
        if (lane == 0) fill(s);
        __syncwarp();
        if (++s == kRingStages) {
            s = 0;
            parity ^= 1u;
        }
        if (++c < chunks) continue;
        c = 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            hr += __shfl_down_sync(0xffffffffu, hr, o);
            hi += __shfl_down_sync(0xffffffffu, hi, o);
        }
        if (lane == 0) {
            const double vr0 = (double)hr * scale, vi0 = (double)hi * scale;
            if (out_c64)
                reinterpret_cast<float2 *>(out)[i] = make_float2((float)vr0, (float)vi0);
            else
                reinterpret_cast<double2 *>(out)[i] = make_double2(vr0, vi0);
        }
        i += step;
    }
    if (!ok && lane == 0) {
        atomicOr(err, ERRBIT_TIMEOUT);
        // no copy may land after the block's shared memory is gone: this round's stages from s on, the
        // next one's before it (those that were filled)
        for (int q = s; q < s + kRingStages; ++q)
            mbar_wait_bounded(&bar[q % kRingStages], q < kRingStages ? parity : parity ^ 1u);
    }
}

cudaError_t direct_configure()
{
    return cudaFuncSetAttribute(k_direct_ring, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kRingBytes + kRingTables);
}

cudaError_t launch_direct(const double *pphi, const double *pr, const double *are,
                          const double *aim, long long ns, const int *l, const int *m, const int *n,
                          int N, double theta, double phi, double scale, bool fp64, void *out,
                          int out_c64, void *mode_consts, int l_top, int m_top, int n_lo, int n_hi, int sm_count,
                          unsigned *err, cudaStream_t st)
{
    // mixed precision: through the ring while the mode tables fit beside it and in the caller's scratch
    // (100,000 samples: 3843 modes 1,095 -> 875 us, reading them alone takes 835; 78,314 samples of 132
    // modes 163 -> 87 us a call), else a warp a sample from registers
    const int pairs = (l_top - 1) * (m_top + 1), table = ring_table_bytes(N, pairs);
    if (!fp64 && ns > 0 && table <= kRingTables && (size_t)table <= direct_mode_const_bytes(N)) {
        auto *words = static_cast<unsigned *>(mode_consts);
        auto *recs = reinterpret_cast<PairConst *>(static_cast<unsigned char *>(mode_consts) + table) - pairs;
        const int n_thr = N > pairs ? N : pairs;
        k_mode_words<<<(n_thr + 63) / 64, 64, 0, st>>>(l, m, n, N, theta, phi, l_top, m_top, words, recs);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        // (reads the caller's arrays beside the plain launch above: launch.cuh)
        return launch_pdl(k_direct_ring, (unsigned)(ns < sm_count ? ns : sm_count), 32 * kRingWarps,
                          (size_t)(kRingBytes + table), st, pphi, pr, are, aim, ns, N,
                          static_cast<const uint4 *>(mode_consts), table, scale, out, out_c64, err);
    }
    // The tables pay where a warp fills them in fewer passes than the modes take (60,000 samples, 33 to 64 modes:
    // one pass 447 -> 340 us, two 447 -> 458), and in as many for few samples, by blocks of four instead of eight
    // (4,000: 12 modes 39 -> 38, 250 modes and 225 exponentials 127 -> 119; 16,000: 96 -> 99, 402 -> 403 and more).
    const int entries = m_top + 1 + n_hi - n_lo + 1, passes = (tab_count(m_top, n_lo, n_hi) + 31) / 32;
    if (fp64 && entries <= kTabMaxEntries && entries < N && (passes < (N + 31) / 32 || ns <= 32ll * sm_count) && ns > 0) {
        const int per = kTabThreads / 32;
        const unsigned blocks = (unsigned)((ns + per - 1) / per);
        // factors of (l, m): eight operations a pair and sample save four a mode, where there are more
        // than twice as many modes (and the tables stay within 12 KB a sample and the caller's scratch)
        const int bytes = (entries + 2 * pairs) * (int)sizeof(double2);
        if (N > 2 * pairs && bytes <= kTabMaxBytes &&
            sizeof(PairConst64) * pairs + sizeof(int2) * (size_t)N <= direct_mode_const_bytes(N)) {
            auto *pc = static_cast<PairConst64 *>(mode_consts);
            const int n_thr = N > pairs ? N : pairs;
            k_pair_consts<<<(n_thr + 63) / 64, 64, 0, st>>>(l, m, n, N, theta, phi, l_top, m_top, n_lo,
                                                            reinterpret_cast<int2 *>(pc + pairs), pc);
            k_direct_tab<true><<<blocks, kTabThreads, per * bytes, st>>>(pphi, pr, are, aim, ns, N, pc, pairs, m_top,
                                                                       n_lo, entries, scale, out, out_c64);
            return cudaGetLastError();
        }
        auto *mc = static_cast<ModeConstTab *>(mode_consts);
        k_mode_consts_tab<<<(N + 63) / 64, 64, 0, st>>>(l, m, n, N, theta, phi, m_top, n_lo, mc);
        k_direct_tab<false><<<blocks, kTabThreads, per * entries * (int)sizeof(double2), st>>>(
            pphi, pr, are, aim, ns, N, mc, 0, m_top, n_lo, entries, scale, out, out_c64);
        return cudaGetLastError();
    }
    // one wave of resident blocks (8 warps, i.e. 8 samples, per block per round)
    static int resident[2] = {0, 0};
    int &rb = resident[fp64 ? 1 : 0];
    if (rb == 0) {
        const cudaError_t e = fp64 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                         &rb, k_direct<double>, 256, 0)
                                   : cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                         &rb, k_direct<float>, 256, 0);
        if (e != cudaSuccess) return e;
        if (rb < 1) rb = 1;
    }
    const long long want = (ns + 7) / 8, cap = (long long)sm_count * rb;
    const int grid = (int)(want < cap ? want : cap);
    if (fp64) {
        auto *mc = static_cast<ModeConst<double> *>(mode_consts);
        k_mode_consts<double><<<(N + 63) / 64, 64, 0, st>>>(l, m, n, N, theta, phi, mc);
        if (ns > 0)
            k_direct<double><<<grid, 256, 0, st>>>(pphi, pr, are, aim, ns, N, mc, scale, out, out_c64);
    } else {
        auto *mc = static_cast<ModeConst<float> *>(mode_consts);
        k_mode_consts<float><<<(N + 63) / 64, 64, 0, st>>>(l, m, n, N, theta, phi, mc);
        if (ns > 0)
            k_direct<float><<<grid, 256, 0, st>>>(pphi, pr, are, aim, ns, N, mc, scale, out, out_c64);
    }
    return cudaGetLastError();
}

static_assert(kMaxAbsN <= 2048 && kRingTables + 4096 <= 65536, "a word: n in fp16, a record's address");
static_assert(sizeof(ModeConstTab) == sizeof(ModeConst<double>), "one scratch size for both");
size_t direct_mode_const_bytes(int N) { return sizeof(ModeConst<double>) * (size_t)N; }

}  // namespace fewsum
