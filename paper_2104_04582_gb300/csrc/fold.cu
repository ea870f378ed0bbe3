// fold.cu -- per-request harmonics and fold of the harmonics into the spline coefficients.
//
// Sec. 4 sum: h = scale * sum_{lmn} A_lmn(t) -2Y_lm(theta, phi) e^{-i Phi_mn}, with the m < 0
// modes given by Eq. (amp_symmetry), k = 0: A_{l,-m,-n} = (-1)^l conj(A_lmn).  Grouping every
// term by its signed frequency (m, n) gives
//     h = sum_{(m,n) signed} K_{m,n}(u) e^{-i (m Phi_phi + n Phi_r)},
//     K_{m,n}   = scale * sum_l A_lmn(u) Y+_lm                        (m >= 0 entries),
//     K_{-m,-n} = scale * sum_l conj(A_lmn(u)) Y-_lm,  Y- = (-1)^l -2Y_{l,-m}   (m > 0),
// and each K is again a complex cubic in u per segment (a fixed linear combination of the
// amplitude splines).  k_fold forms these "slot" cubics for one request; the summation kernel
// then evaluates sum K z_phi^m z_r^n by Horner's rule.  This is exact algebra on the
// coefficients (only the rounding order differs from summing mode by mode).
//
// Spin-weighted harmonics (the paper lists them as a utility, Sec. 3.D, without a formula):
//     sY_lm(theta, phi) = (-1)^s sqrt((2l+1)/(4 pi)) d^l_{m,-s}(theta) e^{i m phi},  s = -2,
// with the Wigner small-d evaluated through its Jacobi-polynomial form
//     d^l_{m',m}(b) = xi sqrt(k! (k+mu+nu)! / ((k+mu)! (k+nu)!)) sin^mu(b/2) cos^nu(b/2)
//                      P_k^{(mu,nu)}(cos b),
//     mu = |m - m'|, nu = |m + m'|, k = l - (mu+nu)/2, xi = 1 if m >= m' else (-1)^(m-m'),
// and the Jacobi polynomial by its three-term recurrence in the degree.
#include "fewsum_internal.h"
#include "harmonics.cuh"
#include "convert.cuh"
#include "tctile.cuh"

namespace fewsum {

__device__ __forceinline__ int wave_of(const WaveDev *waves, int n, int g, bool by_pair)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        const int b = by_pair ? waves[mid].pair_begin : waves[mid].fold_begin;
        if (b <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Two threads per (wave, (l, m) pair): one computes Y+, the other Y- (halves the dependency
// chain each thread waits on).  FP64 plans evaluate the harmonics in FP64; mixed plans, whose
// folded coefficients are FP32, evaluate them in FP32 (relative error near 1e-7, far below the
// path's 1e-6 mismatch budget) and stay off GB300's narrow FP64 pipe.
// One instantiation per arithmetic type keeps each kernel's code small (it runs cold, once).
template <bool FP64>
__device__ __forceinline__ void ylm_thread(const PlanHdr &h, bool wait)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int g = t >> 1, which = t & 1;
    double2 y = make_double2(0.0, 0.0);
    double2 *dst = nullptr;
    if (g < h.total_pairs) {
        const WaveDev *waves = tc_local(h, h.waves);
        const WaveDev &W = waves[wave_of(waves, h.n_waves, g, true)];
        const int p = g - W.pair_begin;
        if (p < W.tr.n_pairs) {
            const int2 lm = W.tr.pair_lm[p];
            y = FP64 ? wave_harmonic<double>(W, lm, which) : wave_harmonic<float>(W, lm, which);
            dst = W.ylm + 2 * p + which;
        } else {
            atomicOr(h.err, ERRBIT_INTERNAL);
        }
    }
    if (wait) pdl_wait();
    if (dst) *dst = y;
}

template <bool FP64>
__global__ void __launch_bounds__(kYlmThreads) k_ylm(const PlanHdr *hp)
{
    pdl_wait();
    pdl_launch_dependents();
    ylm_thread<FP64>(*hp, false);
}

// The plan in the parameters: the harmonics need nothing of an earlier kernel, only their store waits;
// the last block copies the plan to the device for the kernels that follow.
__global__ void __launch_bounds__(kYlmThreads) k_ylm_param(const __grid_constant__ PlanParam plan)
{
    pdl_launch_dependents();
    ylm_thread<true>(*reinterpret_cast<const PlanHdr *>(plan.bytes), true);
    tc_store_plan(plan);
}

cudaError_t launch_ylm(const PlanHdr *hdr_dev, const PlanParam *plan, int total_pairs, bool fp64,
                       cudaStream_t st)
{
    if (total_pairs <= 0) return cudaSuccess;
    const int threads = 2 * total_pairs, grid = (threads + kYlmThreads - 1) / kYlmThreads;
    if (plan) return launch_pdl(k_ylm_param, grid, kYlmThreads, 0, st, *plan);
    return launch_pdl(fp64 ? k_ylm<true> : k_ylm<false>, grid, kYlmThreads, 0, st, hdr_dev);
}

__device__ __forceinline__ double cvt(double v, double) { return v; }
__device__ __forceinline__ float cvt(double v, float) { return f64_to_f32_fast(v); }

template <typename T> struct Slot8;
template <> struct Slot8<double> {
    __device__ static void store(double *dst, const double (&re)[4], const double (&im)[4])
    {
        double2 *d = reinterpret_cast<double2 *>(dst);
        d[0] = make_double2(re[0], re[1]);
        d[1] = make_double2(re[2], re[3]);
        d[2] = make_double2(im[0], im[1]);
        d[3] = make_double2(im[2], im[3]);
    }
};
template <> struct Slot8<float> {
    __device__ static void store(float *dst, const float (&re)[4], const float (&im)[4])
    {
        float4 *d = reinterpret_cast<float4 *>(dst);
        d[0] = make_float4(re[0], re[1], re[2], re[3]);
        d[1] = make_float4(im[0], im[1], im[2], im[3]);
    }
};

// One thread per (wave, segment, slot): K_slot = scale * sum of its contributions, summed on the
// splines' Hermite data (values and slopes at the segment's two knots) and turned into power
// coefficients in u once.
// T is the arithmetic and storage type of the folded coefficients (double for FEW_FP64,
// float for FEW_MIXED, whose amplitudes are FP32 by design).
template <typename T>
__global__ void __launch_bounds__(kFoldThreads) k_fold(const PlanHdr *__restrict__ hp)
{
    const PlanHdr h = *hp;
    const int b = blockIdx.x;
    const int w = wave_of(h.waves, h.n_waves, b, false);
    const WaveDev &W = h.waves[w];
    const int local = b - W.fold_begin;
    const int s = local / W.fold_blocks_per_seg;
    const int slot = (local % W.fold_blocks_per_seg) * kFoldThreads + threadIdx.x;
    const TrajDev &tr = W.tr;
    if (s >= tr.S || slot >= tr.n_slots) return;
    T re[4] = {0, 0, 0, 0}, im[4] = {0, 0, 0, 0};
    const int c0 = tr.slot_ptr[slot], c1 = tr.slot_ptr[slot + 1];
    const double *__restrict__ cs = tr.coef + (size_t)s * tr.J * 4;
    for (int c = c0; c < c1; ++c) {
        const int2 code = tr.contrib[c];  // (mode * 2 + kind, harmonic-table index)
        const int i = code.x >> 1, kind = code.x & 1;
        const double2 Yd = W.ylm[code.y];
        const T yr = cvt(Yd.x, T()), yi = cvt(Yd.y, T());
        const double2 *ca = reinterpret_cast<const double2 *>(cs + (size_t)(2 + 2 * i) * 4);
        const double2 r01 = ca[0], r23 = ca[1], i01 = ca[2], i23 = ca[3];
        const T ar[4] = {cvt(r01.x, T()), cvt(r01.y, T()), cvt(r23.x, T()), cvt(r23.y, T())};
        T ai[4] = {cvt(i01.x, T()), cvt(i01.y, T()), cvt(i23.x, T()), cvt(i23.y, T())};
        if (kind) {
#pragma unroll
            for (int q = 0; q < 4; ++q) ai[q] = -ai[q];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            re[q] += ar[q] * yr - ai[q] * yi;
            im[q] += ar[q] * yi + ai[q] * yr;
        }
    }
    // the folded values are Hermite data (the fold is linear in them): power coefficients in u
    // once per (segment, slot)
    const T hk = cvt(tr.h[s], T()), sc = cvt(W.scale, T());
    T pre[4], pim[4];
    hermite_to_power(re[0], re[1], re[2], re[3], hk, pre);
    hermite_to_power(im[0], im[1], im[2], im[3], hk, pim);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        pre[q] *= sc;
        pim[q] *= sc;
    }
    T *dst = reinterpret_cast<T *>(W.fcoef) + ((size_t)s * tr.n_slots + slot) * 8;
    Slot8<T>::store(dst, pre, pim);
}

cudaError_t launch_fold(const PlanHdr *hdr_dev, int total_fold_blocks, bool fp64, cudaStream_t st)
{
    if (total_fold_blocks <= 0) return cudaSuccess;
    if (fp64)
        k_fold<double><<<total_fold_blocks, kFoldThreads, 0, st>>>(hdr_dev);
    else
        k_fold<float><<<total_fold_blocks, kFoldThreads, 0, st>>>(hdr_dev);
    return cudaGetLastError();
}

}  // namespace fewsum
