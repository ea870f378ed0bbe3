// fold_slot.cuh -- one harmonic slot of one segment: the fold shared by the summation variants.
#pragma once

#include "convert.cuh"
#include "fewsum_internal.h"

namespace fewsum {

__device__ __forceinline__ double cvt(double v, double) { return v; }
__device__ __forceinline__ float cvt(double v, float) { return f64_to_f32_fast(v); }

// K_slot = scale * sum of the slot's contributions (A Y+ or conj(A) Y-), summed on the splines'
// Hermite data `cs` of the segment (values and slopes at its two knots; the fold is linear in
// them) and turned into power coefficients in u once.
template <typename T>
__device__ __forceinline__ void fold_slot(const TrajDev &tr, const double2 *__restrict__ ylm,
                                          const double *__restrict__ cs, int slot, double h,
                                          double scale, T (&pre)[4], T (&pim)[4])
{
    T re[4] = {0, 0, 0, 0}, im[4] = {0, 0, 0, 0};
    const int c0 = tr.slot_ptr[slot], c1 = tr.slot_ptr[slot + 1];
    for (int c = c0; c < c1; ++c) {
        const int2 code = tr.contrib[c];  // (mode * 2 + kind, harmonic-table index)
        const int i = code.x >> 1, kind = code.x & 1;
        const double2 Yd = ylm[code.y];
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
    const T hk = cvt(h, T()), sc = cvt(scale, T());
    hermite_to_power(re[0], re[1], re[2], re[3], hk, pre);
    hermite_to_power(im[0], im[1], im[2], im[3], hk, pim);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        pre[q] *= sc;
        pim[q] *= sc;
    }
}

}  // namespace fewsum
