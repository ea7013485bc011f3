// Twiddles of the band kernels whose radices and strides are known at compile time (band_pow2.cu, band_smooth.cuh); append_twiddle_rows
// in api.cu writes the rows.
#pragma once
#include "static_fft.cuh"

namespace cqt {

__host__ __device__ constexpr int twiddle_rows(int r) { return r <= 1 ? 0 : 1 + twiddle_rows((r + 1) / 2); }   // powers 1, 2, 4 ... below r

// Twiddles w, w^2, w^4, w^8 of one butterfly: rows of s entries, in the order in which consecutive butterflies read them; the
// other powers are products of at most three of those (raising one rounded w to the q-th power would multiply its error by q).
template <int R>
struct TwiddleRows {
    static constexpr int N = twiddle_rows(R);
    float2 w[N];
    __device__ __forceinline__ void load(const float2 *__restrict__ rows, int s, int np) {
#pragma unroll
        for (int i = 0; i < N; ++i) w[i] = __ldg(rows + i * s + np);
    }
    template <int SIGN>
    __device__ __forceinline__ void apply(float (&re)[R], float (&im)[R]) const {
        float wr[R], wi[R];
#pragma unroll
        for (int q = 1; q < R; ++q) {
            const int hi = q >= 8 ? 3 : (q >= 4 ? 2 : (q >= 2 ? 1 : 0)), hb = 1 << hi, lo = q - hb;
            if (lo == 0) {
                wr[q] = w[hi].x;
                wi[q] = SIGN > 0 ? -w[hi].y : w[hi].y;
            } else {
                wr[q] = fmaf(wr[hb], wr[lo], -wi[hb] * wi[lo]);
                wi[q] = fmaf(wr[hb], wi[lo], wi[hb] * wr[lo]);
            }
            const float x = re[q], y = im[q];
            re[q] = fmaf(x, wr[q], -y * wi[q]);
            im[q] = fmaf(x, wi[q], y * wr[q]);
        }
    }
};

}  // namespace cqt
