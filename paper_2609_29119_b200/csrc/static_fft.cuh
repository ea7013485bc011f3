// Tile transforms with every radix, stride and column count known at compile time: LEN = R0 R1 R2 points (R2 = 1: two
// stages) on NC interleaved columns in shared memory, T threads with 16 elements each.  In-place decimation in
// frequency: stage 0 has butterflies over positions b + q LEN/R0, the last stage leaves frequency
// k0 + R0 k1 (+ R0 R1 q) in butterfly b = k0 R1 + k1, element q.  The kernels fuse their loads into stage 0 and their
// stores into the last stage, both on registers.
#pragma once
#include "engine.cuh"

namespace cqt {

enum { kPlain = 0, kOddPitch = 1, kSwizzle = 2 };   // shared-memory layouts of a tile

template <int LEN_, int R0_, int R1_, int R2_, int NC_, int LAYOUT_>
struct TileShape {
    static constexpr int LEN = LEN_, R0 = R0_, R1 = R1_, R2 = R2_, NC = NC_, LAYOUT = LAYOUT_;
    static constexpr int S0 = LEN / R0, RL = R2 > 1 ? R2 : R1, NL = LEN / RL;   // NL: butterflies of the last stage
    static constexpr int T = LEN * NC / 16;
    // kOddPitch: consecutive positions of one column lie in different banks; kSwizzle: half-tiles (8 + 8 or 4 + 4
    // columns) of consecutive positions do
    static constexpr int PITCH = LAYOUT == kOddPitch ? NC + 1 : NC;
    static constexpr int ELEMS = LEN * PITCH;
    static_assert(R0 * R1 * R2 == LEN, "radices");
    static __device__ __forceinline__ int at(int p, int col) {
        if constexpr (LAYOUT == kSwizzle) return p * NC + (col ^ (NC == 16 ? (p & 1) << 3 : ((p >> 1) & 1) << 2));
        else return p * PITCH + col;
    }
    // position of frequency k
    static __device__ __forceinline__ int position(int k) {
        if constexpr (R2 > 1) return ((k % R0) * R1 + (k / R0) % R1) * R2 + k / (R0 * R1);
        else return (k % R0) * R1 + k / R0;
    }
    // lowest frequency of butterfly b of the last stage
    static __device__ __forceinline__ int low(int b) { return R2 > 1 ? b / R1 + R0 * (b % R1) : b; }
};

template <int R, int SIGN>
__device__ __forceinline__ void dft(float (&re)[R], float (&im)[R]) {
    if (SIGN < 0) Codelet<R>::run(re, im); else Codelet<R>::run(im, re);
}

// end of stage 0 for one butterfly: twiddles, store.  twf: full table of W_LEN
template <class S, int SIGN>
__device__ __forceinline__ void finish_first(float2 *buf, const float2 *twf, int b, int col, float (&re)[S::R0], float (&im)[S::R0]) {
    dft<S::R0, SIGN>(re, im);
    apply_twiddle_direct<S::R0, SIGN>(twf, (uint32_t)b, re, im);
#pragma unroll
    for (int q = 0; q < S::R0; ++q) buf[S::at(b + q * S::S0, col)] = make_float2(re[q], im[q]);
}

// the stage between first and last, in shared memory
template <class S, int SIGN>
__device__ __forceinline__ void tile_middle(float2 *buf, const float2 *twf, int tid) {
    if constexpr (S::R2 > 1) {
        constexpr int R1 = S::R1, R2 = S::R2, units = S::LEN / R1 * S::NC / S::T;
        static_assert(units * S::T * R1 == S::LEN * S::NC, "whole rounds");
#pragma unroll 1
        for (int u = 0; u < units; ++u) {
            const int w = tid + u * S::T, col = w % S::NC, b = w / S::NC, np = b % R2, p = (b / R2) * S::S0 + np;
            float re[R1], im[R1];
#pragma unroll
            for (int q = 0; q < R1; ++q) {
                const float2 v = buf[S::at(p + q * R2, col)];
                re[q] = v.x; im[q] = v.y;
            }
            dft<R1, SIGN>(re, im);
            apply_twiddle_direct<R1, SIGN>(twf, (uint32_t)(np * S::R0), re, im);
#pragma unroll
            for (int q = 0; q < R1; ++q) buf[S::at(p + q * R2, col)] = make_float2(re[q], im[q]);
        }
        __syncthreads();
    }
}

// butterfly b of the last stage of column col into registers
template <class S, int SIGN>
__device__ __forceinline__ void last_butterfly(const float2 *buf, int b, int col, float (&re)[S::RL], float (&im)[S::RL]) {
#pragma unroll
    for (int q = 0; q < S::RL; ++q) {
        const float2 v = buf[S::at(b * S::RL + q, col)];
        re[q] = v.x; im[q] = v.y;
    }
    dft<S::RL, SIGN>(re, im);
}

}  // namespace cqt
