// What the long-FFT kernels share: arguments, packed signal access, twiddle staging, overlap-add and Eq. retangle.
#pragma once
#include "engine.cuh"
#include "internal.hpp"

namespace cqt {

struct LongArgs {
    const float2 *tw;
    int tw_full_A, tw_full_B;    // full tables of W_A, W_B
    int tw_u, tw_v;              // twiddles between the passes: U[low][i], V[q][i] (long_fft_forward.cu)
    int tw_n, log_n_c, n_n;      // two-level table of W_N
    int valid_len;
    int aligned;           // signal rows allow float2 access
    long long x_stride;
    const float *x_in;
    float *x_out;
    float2 *T;
    long long t_pitch;
    float2 *X;             // half spectrum rows (forward)
    long long x_pitch;
    const float2 *Y;       // weighted-bin planes (inverse)
    long long y_pitch;     // per signal
    long long y_plane;     // per plane
    int planes;
    const int32_t *cover;
    int *dbg;
    // sliced source (forward column pass of the streaming form, see SliceSource)
    float *ring;
    const float *slice_win;
    int ring_len, ring_base;      // position of the first slice's sample 0 in the ring
    int lead;                     // samples of the first slice before the start of the stream
    int hop, channels, slices;
    const float *fresh;
    long long fresh_stride;
    int fresh_at, keep_at;        // sample of the first slice / of the last slice where the fresh / the kept ones begin
    int fresh_pairs;              // fresh samples can be read in pairs
};

__device__ __forceinline__ float2 load_packed(const float *row, int j, int valid_len, int aligned) {
    const int i = 2 * j;
    if (i + 1 < valid_len) {
        if (aligned) return __ldcs(reinterpret_cast<const float2 *>(row + i));   // read once: streaming
        return make_float2(__ldcs(row + i), __ldcs(row + i + 1));
    }
    if (i < valid_len) return make_float2(__ldcs(row + i), 0.f);
    return make_float2(0.f, 0.f);
}

__device__ __forceinline__ void store_packed(float *row, int j, float2 v, int valid_len, int aligned) {
    const int i = 2 * j;
    if (i + 1 < valid_len) {
        if (aligned) __stcs(reinterpret_cast<float2 *>(row + i), v);
        else { __stcs(row + i, v.x); __stcs(row + i + 1, v.y); }
    } else if (i < valid_len) {
        __stcs(row + i, v.x);
    }
}

// copies N entries of a table into shared memory on T threads, the first `scaled` of them times `scale`: all loads of a
// thread are issued before any is stored, one trip to the L2 instead of one per round
template <int N, int T>
__device__ __forceinline__ void stage_table(float2 *dst, const float2 *__restrict__ src, int tid, int scaled = 0, float scale = 1.f) {
    constexpr int rounds = (N + T - 1) / T;
    float2 v[rounds];
#pragma unroll
    for (int i = 0; i < rounds; ++i)
        if (tid + i * T < N) v[i] = __ldg(src + tid + i * T);
#pragma unroll
    for (int i = 0; i < rounds; ++i) {
        const int e = tid + i * T;
        if (e < scaled) { v[i].x *= scale; v[i].y *= scale; }
        if (e < N) dst[e] = v[i];
    }
}

// log2 of the low part of a two-level table of n = 2^m entries (see append_twiddles in api.cu), and its entry count
__host__ __device__ constexpr int low_bits(int64_t n) {
    int l = 0;
    while ((1ll << (2 * l)) < n) ++l;
    return l;
}
__host__ __device__ constexpr int two_level_entries(int64_t n) { return (int)((1ll << low_bits(n)) + (n >> low_bits(n))); }

// ---------------------------------------------------------------- inverse: overlap-add
// Sum of the planes that hold bin k.  MASK (at most 31 planes): the cover word is a bit mask of them; else it is
// (plane of the first covering band << 8) | number of covering bands, band i of the range in plane (first + i) mod
// planes.  The order is fixed either way.  plane_first: three of them (the lowest three planes), without a branch, so
// that the loads of several bins are in flight together; plane_rest adds the others (bins of the lowest bands, where
// the minimum width makes many overlap).
template <bool MASK>
__device__ __forceinline__ float2 plane_first(const LongArgs &a, const float2 *Y, int k, int32_t cover) {
    float2 v[3];
    const int n = cover & 255;
    int plane = cover >> 8;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if constexpr (MASK) v[i] = (cover >> i) & 1 ? ld_data(Y + i * a.y_plane + k) : make_float2(0.f, 0.f);
        else {
            v[i] = i < n && CQT_CHK(a.dbg, 206, n, a.planes + 1) ? ld_data(Y + plane * a.y_plane + k) : make_float2(0.f, 0.f);
            if (++plane >= a.planes) plane -= a.planes;
        }
    }
    return make_float2(v[0].x + v[1].x + v[2].x, v[0].y + v[1].y + v[2].y);
}
template <bool MASK>
__device__ __forceinline__ void plane_rest(const LongArgs &a, const float2 *Y, int k, int32_t cover, float2 &acc) {
    int left = MASK ? cover >> 3 : (cover & 255) - 3, plane = MASK ? 3 : (cover >> 8) + 3;
    while (left > 0) {
        float2 w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (!MASK && plane >= a.planes) plane -= a.planes;
            w[j] = (MASK ? left & 1 : left > 0) && CQT_CHK(a.dbg, 207, plane, a.planes) ? ld_data(Y + plane * a.y_plane + k) : make_float2(0.f, 0.f);
            ++plane;
            left = MASK ? left >> 1 : left - 1;
        }
        acc.x += (w[0].x + w[1].x) + (w[2].x + w[3].x);
        acc.y += (w[0].y + w[1].y) + (w[2].y + w[3].y);
    }
}
template <bool MASK>
__device__ __forceinline__ float2 plane_sum(const LongArgs &a, const float2 *Y, int k, int32_t cover) {
    float2 acc = plane_first<MASK>(a, Y, k, cover);
    plane_rest<MASK>(a, Y, k, cover, acc);
    return acc;
}

// One pair (q, m = Lp - q) of packed bins from the half-spectrum bins X_q, X_m (Eq. retangle, w_{Lp-q} = -conj w_q):
// Z_q = s [E + i conj(w) O], Z_m = s conj[E - i conj(w) O], E = X_q + conj X_m, O = X_q - conj X_m,
// w = exp(-2 pi i q / N), s = 1 / (2 Lp), a power of two; sw = s w
__device__ __forceinline__ void retangle(float2 xq, float2 xm, float2 sw, float s, float2 &zq, float2 &zm) {
    const float ex = xq.x + xm.x, ey = xq.y - xm.y, ox = xq.x - xm.x, oy = xq.y + xm.y;
    const float px = sw.y * ox - sw.x * oy, py = sw.x * ox + sw.y * oy;
    zq = make_float2(fmaf(s, ex, px), fmaf(s, ey, py));
    zm = make_float2(fmaf(s, ex, -px), py - s * ey);
}

// ---------------------------------------------------------------- host side
inline LongArgs base_args(const cqt_plan &p, int64_t valid_len, int64_t x_stride, const void *xptr) {
    LongArgs a{};
    a.tw = p.d.tw;
    a.tw_full_A = p.ffts[(size_t)p.lf.fft_A].tw_full_off;
    a.tw_full_B = p.ffts[(size_t)p.lf.fft_B].tw_full_off;
    a.tw_n = p.lf.tw_n;
    a.log_n_c = p.lf.log_n_c;
    a.n_n = p.lf.n_n;
    a.valid_len = (int)valid_len;
    a.x_stride = x_stride;
    a.aligned = ((reinterpret_cast<uintptr_t>(xptr) & 7) == 0 && (x_stride & 1) == 0) ? 1 : 0;
    a.t_pitch = p.lf.Lp;
    a.x_pitch = p.lf.x_pitch;
    a.y_pitch = p.y_pitch;
    a.y_plane = p.y_plane;
    a.planes = p.y_planes;
    a.cover = p.d.cover;
    a.dbg = p.d.dbg;
    return a;
}

// one-pass real FFTs of short signals (short_fft.cu)
cudaError_t launch_short_rfft_forward(const cqt_plan &p, LongArgs &a, int64_t batch, cudaStream_t st);
cudaError_t launch_short_rfft_inverse(const cqt_plan &p, LongArgs &a, int64_t batch, cudaStream_t st);

}  // namespace cqt
