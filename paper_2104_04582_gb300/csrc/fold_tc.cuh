// fold_tc.cuh -- the fold of the tensor-core summations (tcsum.cu, tcsum64.cu): one block forms the cubics
// of every signed frequency of one segment in shared memory.
//
// A mode (l, m, n) with m > 0 feeds two frequencies, (m, n) through Y+ and (-m, -n) through Y-, so one
// thread takes a frequency with m >= 0 and forms both cubics from one read of the splines' Hermite
// data (the loads of three modes in flight).  Per segment of the one-year 3843-mode waveform that is
// 246 KB of data read once instead of twice.
#pragma once

#include "convert.cuh"
#include "fewsum_internal.h"

namespace fewsum {

__device__ __forceinline__ double fold_cvt(double v, double) { return v; }
__device__ __forceinline__ float fold_cvt(double v, float) { return f64_to_f32_fast(v); }
template <typename T> struct Pair2;
template <> struct Pair2<float> { using type = float2; };
template <> struct Pair2<double> { using type = double2; };

// Row stride of the cubics in shared memory (elements): column half + n - n_mid of row 16 p + 2 x + e
// is coefficient x = 4 component + degree of frequency n in the row of m = m_top - p (e = 0) or
// p - m_top (e = 1; zero for m = 0).  half = 8 ks - 1; the padding keeps the packing's reads of 8
// consecutive rows on different banks.
__host__ __device__ constexpr int fold_stride(int ks, size_t size) { return 16 * ks + (size == 4 ? 4 : 2); }

// Y: [n_pairs][2] harmonics Y+, Y- in the arithmetic type.  Needs a barrier before kc is read.
template <typename T>
__device__ __forceinline__ void fold_rows(const TrajDev &tr, int s, double scale,
                                          const typename Pair2<T>::type *Y, T *__restrict__ kc)
{
    const int ks = tr.tc_ks, half = 8 * ks - 1, width = 2 * half + 1, ld = fold_stride(ks, sizeof(T));
    const double *cs = tr.coef + (size_t)s * tr.J * 4;
    const T hk = fold_cvt(tr.h[s], T()), sc = fold_cvt(scale, T());
    for (int it = threadIdx.x; it < tr.tc_pairs * width; it += blockDim.x) {
        const int p = it / width, off = it - p * width - half, m = tr.m_top - p;
        const int4 rs = tr.row_slot[p];  // first slot, n = rs.y .. rs.z
        const int n = tr.n_mid + off;
        T a[8], b[8];  // Hermite data of (m, n) and (-m, -n): 4 real, 4 imaginary
#pragma unroll
        for (int q = 0; q < 8; ++q) a[q] = b[q] = (T)0;
        if (n <= rs.y && n >= rs.z) {
            const int slot = rs.x + rs.y - n;
            const int c0 = tr.slot_ptr[slot], c1 = tr.slot_ptr[slot + 1];
            constexpr int U = 3;
            for (int c = c0; c < c1; c += U) {
                double2 v[U][4];
                int pair[U];
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    const int2 code = tr.contrib[min(c + k, c1 - 1)];  // (mode * 2, 2 * pair)
                    pair[k] = code.y;
                    const double2 *ca = reinterpret_cast<const double2 *>(cs + (size_t)(2 + code.x) * 4);
#pragma unroll
                    for (int q = 0; q < 4; ++q) v[k][q] = ca[q];
                }
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    if (c + k >= c1) break;
                    const auto yp = Y[pair[k]], ym = Y[pair[k] + 1];
                    const T re[4] = {fold_cvt(v[k][0].x, T()), fold_cvt(v[k][0].y, T()),
                                     fold_cvt(v[k][1].x, T()), fold_cvt(v[k][1].y, T())};
                    const T im[4] = {fold_cvt(v[k][2].x, T()), fold_cvt(v[k][2].y, T()),
                                     fold_cvt(v[k][3].x, T()), fold_cvt(v[k][3].y, T())};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        a[q] += re[q] * yp.x - im[q] * yp.y;
                        a[4 + q] += re[q] * yp.y + im[q] * yp.x;
                        if (m > 0) {  // conj(A) Y-
                            b[q] += re[q] * ym.x + im[q] * ym.y;
                            b[4 + q] += re[q] * ym.y - im[q] * ym.x;
                        }
                    }
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            T *dst = kc + (16 * p + e) * ld + half + (e ? -off : off);
            const T(&g)[8] = e ? b : a;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                T w[4];
                hermite_to_power(g[4 * c], g[4 * c + 1], g[4 * c + 2], g[4 * c + 3], hk, w);
#pragma unroll
                for (int d = 0; d < 4; ++d) dst[2 * (4 * c + d) * ld] = w[d] * sc;
            }
        }
    }
}

// Basis coefficients of row r and power b: X of cos(b theta) = c_+ + c_-, Y of sin(b theta) = -i (c_+ -
// c_-) (b = 0: c_0 and 0).
template <typename T>
__device__ __forceinline__ void fold_basis(const T *__restrict__ kc, int ks, int r, int b, T &X, T &Y)
{
    const int half = 8 * ks - 1, ld = fold_stride(ks, sizeof(T));
    const T *row = kc + r * ld + half, *other = kc + (r ^ 8) * ld + half;  // the other component
    if (b == 0) {
        X = row[0];
        Y = (T)0;
        return;
    }
    X = row[b] + row[-b];
    const T d = other[b] - other[-b];
    Y = (r & 8) ? -d : d;
}

}  // namespace fewsum
