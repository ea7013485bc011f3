// Shapes of the two-pass long FFT and what its passes share (long_fft_forward.cu, long_fft_inverse.cu).
#pragma once
#include "long_common.cuh"
#include "static_fft.cuh"

namespace cqt {

// Lp = A B with B = 2^ceil(log2(Lp) / 2), at most 1024: every split that occurs, N = 2^14 ... 2^22
#define CQT_LONG_SPLITS(X) X(64, 128) X(128, 128) X(128, 256) X(256, 256) X(256, 512) X(512, 512) X(512, 1024) X(1024, 1024) X(2048, 1024)

// Columns: 16 of them make 128-byte runs of the signal and of T; 8 where 16 would not leave room for two CTAs.
// Rows: 8 + 8 mirror rows (4 + 4), runs of 64 (32) bytes of X, for the same reason.
// Radices: few stages; at most two butterflies' worth of registers per thread; radix 8 (4) where the untangle
// (overlap-add) of two butterflies' operands shares a thread with them.
template <int LEN> struct ColsForwardT;
template <> struct ColsForwardT<64> { using S = TileShape<64, 8, 8, 1, 16, kPlain>; };
template <> struct ColsForwardT<128> { using S = TileShape<128, 16, 8, 1, 16, kPlain>; };
template <> struct ColsForwardT<256> { using S = TileShape<256, 16, 16, 1, 16, kPlain>; };
template <> struct ColsForwardT<512> { using S = TileShape<512, 8, 8, 8, 16, kPlain>; };
template <> struct ColsForwardT<1024> { using S = TileShape<1024, 16, 8, 8, 8, kPlain>; };
template <> struct ColsForwardT<2048> { using S = TileShape<2048, 16, 16, 8, 8, kPlain>; };
template <int LEN> using ColsForward = typename ColsForwardT<LEN>::S;

// inverse columns: loads run along the column, hence the odd pitch
template <int LEN> struct ColsInverseT;
template <> struct ColsInverseT<64> { using S = TileShape<64, 8, 8, 1, 16, kOddPitch>; };
template <> struct ColsInverseT<128> { using S = TileShape<128, 16, 8, 1, 16, kOddPitch>; };
template <> struct ColsInverseT<256> { using S = TileShape<256, 16, 16, 1, 16, kOddPitch>; };
template <> struct ColsInverseT<512> { using S = TileShape<512, 8, 8, 8, 16, kOddPitch>; };
template <> struct ColsInverseT<1024> { using S = TileShape<1024, 16, 8, 8, 8, kOddPitch>; };
template <> struct ColsInverseT<2048> { using S = TileShape<2048, 16, 16, 8, 8, kOddPitch>; };
template <int LEN> using ColsInverse = typename ColsInverseT<LEN>::S;

template <int LEN> struct RowsForwardT;
template <> struct RowsForwardT<128> { using S = TileShape<128, 16, 8, 1, 16, kOddPitch>; };
template <> struct RowsForwardT<256> { using S = TileShape<256, 8, 4, 8, 16, kOddPitch>; };
template <> struct RowsForwardT<512> { using S = TileShape<512, 8, 8, 8, 16, kOddPitch>; };
template <> struct RowsForwardT<1024> { using S = TileShape<1024, 16, 8, 8, 8, kOddPitch>; };
template <int LEN> using RowsForward = typename RowsForwardT<LEN>::S;

template <int LEN> struct RowsInverseT;
template <> struct RowsInverseT<128> { using S = TileShape<128, 4, 4, 8, 16, kSwizzle>; };
template <> struct RowsInverseT<256> { using S = TileShape<256, 4, 8, 8, 16, kSwizzle>; };
template <> struct RowsInverseT<512> { using S = TileShape<512, 4, 8, 16, 16, kSwizzle>; };
template <> struct RowsInverseT<1024> { using S = TileShape<1024, 4, 16, 16, 8, kSwizzle>; };
template <int LEN> using RowsInverse = typename RowsInverseT<LEN>::S;

// entry y of a two-level table of n entries
template <int64_t n>
__device__ __forceinline__ float2 two_level(const float2 *tab, uint32_t y) {
    constexpr int C = low_bits(n);
    return cmul(tab[y & ((1u << C) - 1)], tab[(1 << C) + (y >> C)]);
}

// Rows of CTA t of the row passes, column r of its tile: r < TW is row TW t + 1 + r, r >= TW its mirror
// A - (TW t + 1 + (r - TW)).  Eq. untangle pairs row k1 with row A - k1, so both operands of every output are in
// the tile.  The last tile's row A/2 is its own mirror; the column that would repeat it holds row 0, which pairs
// with itself too: every row sits in exactly one tile and nothing is transformed twice.
template <int A, int TW>
__device__ __forceinline__ int row_of(int t, int r) {
    const int k1 = r < TW ? TW * t + 1 + r : A - (TW * t + 1 + (r - TW));
    return (r >= TW && 2 * k1 == A) ? 0 : k1;
}

inline cudaError_t launch_long(const void *fn, int tiles, int64_t batch, int threads, size_t smem, LongArgs &a, cudaStream_t st) {
    void *args[] = {&a};
    return launch_kernel(fn, dim3((unsigned)tiles, (unsigned)batch), dim3((unsigned)threads), args, smem, st);
}

}  // namespace cqt
