// What the long-FFT kernels share: arguments, packed signal access, twiddle staging, overlap-add and Eq. retangle.
#pragma once
#include "engine.cuh"
#include "internal.hpp"

namespace cqt {

extern __shared__ float2 smem_long[];

struct LongArgs {
    const FftPlan *ffts;
    const float2 *tw;
    int fft_A, fft_B;
    int A, B, Lp;
    int tw_lp, log_lp_c, n_lp;   // two-level table of W_Lp and its entry count
    int tw_n, log_n_c, n_n;      // two-level table of W_N
    int tw_cols, tw_rows;
    int valid_len;
    int aligned;           // signal rows allow float2 access
    long long x_stride;
    const float *x_in;
    float *x_out;
    float2 *T;
    long long t_pitch;
    float2 *X;             // half spectrum rows (forward)
    long long x_pitch;
    // inverse: overlap-add + retangle in the prologue of the row pass
    int log_b, log_own;    // log2 B, log2 (2 TWr)
    const float2 *Y;
    long long y_pitch;     // per signal
    long long y_plane;     // per plane
    int planes;
    const int32_t *cover;
    float scale;
    uint32_t cols_magic, rows_magic;
    int *dbg;
    // sliced source (forward column pass of the streaming form): row r is slice r / channels of channel r % channels,
    // its sample i is slice_win[i] * ring[channel][(slice_first + (r / channels) * hop + i) mod ring_len], zero
    // before the start of the stream
    const float *ring;
    const float *slice_win;
    long long ring_len, slice_first, hop;
    int channels;
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

// copies the full twiddle table of a power-of-two plan into shared memory
__device__ __forceinline__ void stage_full(float2 *dst, const float2 *__restrict__ tw_base, const FftPlan &fp, int tid, int nthr) {
    const float2 *src = tw_base + fp.tw_full_off;
    for (int i = tid; i < fp.M; i += nthr) dst[i] = __ldg(src + i);
}

__device__ __forceinline__ void stage_table(float2 *dst, const float2 *__restrict__ src, int n, int tid, int nthr) {
    for (int i = tid; i < n; i += nthr) dst[i] = __ldg(src + i);
}

// ---------------------------------------------------------------- inverse: overlap-add + retangle
// sum over the bands covering bin k, in band order
// Sum over the bands covering bin k, in band order.  The cover word is (plane of the first covering band << 8) | number
// of covering bands; band i of the range sits in plane (first + i) mod planes.  The first kUnroll plane values are loaded
// unconditionally-predicated before any is used, so that their latencies overlap; absent terms add +0.
constexpr int kGatherUnroll = 3;
struct GatherLoads {
    float2 v[kGatherUnroll];
    int n, off, plane_len, wrap;
};
__device__ __forceinline__ GatherLoads gather_issue(const LongArgs &a, const float2 *__restrict__ Y, int k, int32_t cv) {
    GatherLoads g;
    g.n = cv & 255;
    g.plane_len = (int)a.y_plane;
    g.wrap = a.planes * g.plane_len;
    g.off = (cv >> 8) * g.plane_len + k;
    if (!CQT_CHK(a.dbg, 206, g.n, a.planes + 1)) g.n = 0;
#pragma unroll
    for (int i = 0; i < kGatherUnroll; ++i) {
        g.v[i] = i < g.n ? __ldg(Y + g.off) : make_float2(0.f, 0.f);
        g.off += g.plane_len;
        if (g.off >= g.wrap) g.off -= g.wrap;
    }
    return g;
}
__device__ __forceinline__ float2 gather_finish(const float2 *__restrict__ Y, GatherLoads &g) {
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < kGatherUnroll; ++i) { acc.x += g.v[i].x; acc.y += g.v[i].y; }
    for (int i = kGatherUnroll; i < g.n; ++i) {
        const float2 v = __ldg(Y + g.off);
        acc.x += v.x;
        acc.y += v.y;
        g.off += g.plane_len;
        if (g.off >= g.wrap) g.off -= g.wrap;
    }
    return acc;
}

// One pair (q, m = Lp - q) of packed bins: both half-spectrum bins are summed once (bands in fixed order) and both
// packed bins follow from the same two values (Eq. retangle with w_{Lp-q} = -conj w_q):
//   Z_q      = s [ (X_q + conj X_m) + i conj(w) (X_q - conj X_m) ]
//   Z_{Lp-q} = s [ (X_m + conj X_q) - i w (X_m - conj X_q) ],   w = exp(-2 pi i q / N), s = 1/(2 Lp)
// wn: two-level table of W_N (shared memory).
__device__ __forceinline__ void retangle_finish(const LongArgs &a, const float2 *__restrict__ Y, const float2 *wn, int q,
                                                GatherLoads &gq, GatherLoads &gm, float2 &zq, float2 &zm) {
    float2 xq = gather_finish(Y, gq);
    float2 xm = gather_finish(Y, gm);
    if (q == 0) { xq.y = 0.f; xm.y = 0.f; }   // bins 0 and N/2 are made real
    const float2 w = twiddle_s(wn, a.log_n_c, (uint32_t)q);
    {
        const float2 ev = make_float2(xq.x + xm.x, xq.y - xm.y);   // X_q + conj X_m
        const float2 od = make_float2(xq.x - xm.x, xq.y + xm.y);   // X_q - conj X_m
        const float2 rot = cmul(make_float2(w.y, w.x), od);        // i conj(w) = (w.y, w.x)
        zq = make_float2(a.scale * (ev.x + rot.x), a.scale * (ev.y + rot.y));
    }
    {
        const float2 ev = make_float2(xm.x + xq.x, xm.y - xq.y);   // X_m + conj X_q
        const float2 od = make_float2(xm.x - xq.x, xm.y + xq.y);   // X_m - conj X_q
        const float2 rot = cmul(make_float2(w.y, -w.x), od);       // -i w = (w.y, -w.x)
        zm = make_float2(a.scale * (ev.x + rot.x), a.scale * (ev.y + rot.y));
    }
}
__device__ __forceinline__ void retangle_pair(const LongArgs &a, const float2 *__restrict__ Y, const float2 *wn, int q, int m,
                                              float2 &zq, float2 &zm) {
    const int32_t cvq = __ldg(a.cover + q), cvm = __ldg(a.cover + m);
    GatherLoads gq = gather_issue(a, Y, q, cvq), gm = gather_issue(a, Y, m, cvm);
    retangle_finish(a, Y, wn, q, gq, gm, zq, zm);
}

// ---------------------------------------------------------------- host side
inline uint32_t magic_of(uint32_t d) { return d <= 1 ? 0u : (uint32_t)(((1ull << 32) + d - 1) / d); }

inline LongArgs base_args(const cqt_plan &p, int64_t valid_len, int64_t x_stride, const void *xptr) {
    LongArgs a{};
    a.ffts = p.d.ffts;
    a.tw = p.d.tw;
    a.fft_A = p.lf.fft_A;
    a.fft_B = p.lf.fft_B;
    a.A = (int)p.lf.A;
    a.B = (int)p.lf.B;
    a.Lp = (int)p.lf.Lp;
    a.tw_lp = p.lf.tw_lp;
    a.log_lp_c = p.lf.log_lp_c;
    a.n_lp = p.lf.n_lp;
    a.tw_n = p.lf.tw_n;
    a.log_n_c = p.lf.log_n_c;
    a.n_n = p.lf.n_n;
    a.tw_cols = p.lf.tw_cols;
    a.tw_rows = p.lf.tw_rows;
    a.valid_len = (int)valid_len;
    a.x_stride = x_stride;
    a.aligned = ((reinterpret_cast<uintptr_t>(xptr) & 7) == 0 && (x_stride & 1) == 0) ? 1 : 0;
    a.t_pitch = p.lf.Lp;
    a.x_pitch = p.lf.x_pitch;
    a.y_pitch = p.y_pitch;
    a.y_plane = p.y_plane;
    a.planes = p.y_planes;
    a.cover = p.d.cover;
    a.cols_magic = magic_of(a.tw_cols);
    a.dbg = p.d.dbg;
    a.log_b = 0;
    while ((1ll << a.log_b) < p.lf.B) ++a.log_b;
    a.log_own = 0;
    while ((1 << a.log_own) < 2 * p.lf.tw_rows) ++a.log_own;
    return a;
}

// one-pass real FFTs of short signals (short_fft.cu)
cudaError_t launch_short_rfft_forward(const cqt_plan &p, LongArgs &a, int64_t batch, cudaStream_t st);
cudaError_t launch_short_rfft_inverse(const cqt_plan &p, LongArgs &a, int64_t batch, cudaStream_t st);
cudaError_t configure_short_fft_kernels(const cqt_plan &p);

}  // namespace cqt
