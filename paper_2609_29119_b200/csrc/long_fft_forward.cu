// Packed real FFT of length N through a complex FFT of length Lp = N/2 = A * B (Eq. pack), two passes, with the
// conjugate-symmetric fold (Eq. untangle) in the epilogue of the second.  One-pass lengths: short_fft.cu.
//
// Index split: sample index j = j1 * B + j2, bin index k = k1 + A * k2 (j1, k1 < A; j2, k2 < B).
//   pass C ("columns"): for 16 (8) adjacent j2, A-point DFT over j1, times W_Lp^{j2 k1}, written to T[k1][j2].  First
//                       stage on registers straight from the signal (packing on load), last stage straight to T.
//   pass R ("rows"):    a CTA transforms 8 (4) rows k1 and their mirror rows A - k1 (row_of), B points each, and writes
//                       the half spectrum X[0 .. Lp].  Both operands of Eq. untangle, Z_k and Z_{Lp-k}, come out of
//                       two butterflies that one thread runs, so the fold happens in its registers.
// Bounds: issue slots; both passes move 8 bytes in and out per point, and instructions, not memory, set the time.
// Lengths, radices, tile widths and strides are compile-time (A and B follow from N), a thread keeps its 16 loads in
// flight before the first butterfly, and there is one exchange through shared memory per stage and none for the fold.
// 32 signals of N = 2^19 (A = B = 512) before, with run-time strides and the fold through shared memory: 45 us + 50 us.
#include <algorithm>

#include "long_passes.cuh"

namespace cqt {

extern __shared__ float2 smem_long[];

// ---------------------------------------------------------------- pass C
// SLICED: the rows are slices cut from a ring buffer of the stream and multiplied by the slice window on load (the
// slice cut of the sliced transform, fused into this pass: no staged copy of the windowed slices)
template <int A, int B, bool SLICED>
__global__ void __launch_bounds__(ColsForward<A>::T, 1024 / ColsForward<A>::T) rfft_cols_fwd_kernel(LongArgs a) {
    using S = ColsForward<A>;
    pdl_launch_dependents();
    const int tid = threadIdx.x, col = tid % S::NC, j2 = blockIdx.x * S::NC + col, ch = blockIdx.y;
    float2 *buf = smem_long, *tws = buf + S::ELEMS;
    stage_table<A, S::T>(tws, a.tw + a.tw_full_A, tid);
    constexpr int R0 = S::R0, units = S::S0 * S::NC / S::T, step = S::T / S::NC;
    float re[units][R0], im[units][R0];
    if constexpr (SLICED) {
#pragma unroll
        for (int u = 0; u < units; ++u)
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                const float2 w = __ldg(reinterpret_cast<const float2 *>(a.slice_win) + (tid / S::NC + u * step + q * S::S0) * B + j2);
                re[u][q] = w.x; im[u][q] = w.y;
            }
    }
    pdl_wait();   // the tables above belong to the plan; what follows reads the predecessor's output
    auto load_all = [&](auto load) {
#pragma unroll
        for (int u = 0; u < units; ++u)
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                const float2 v = load(tid / S::NC + u * step + q * S::S0);
                re[u][q] = v.x; im[u][q] = v.y;
            }
    };
    if constexpr (SLICED) {
        // re, im hold the window; it is constant for the stream's life and was fetched before the wait
        const int s_rel = ch / a.channels, chan = ch - s_rel * a.channels, R = a.ring_len;
        int base = a.ring_base + s_rel * a.hop;       // one wrap at most: the ring is longer than the slices of a call
        if (base >= R) base -= R;
        const int lead = a.lead - s_rel * a.hop, fresh_at = a.fresh_at - s_rel * a.hop;
        const int keep = s_rel == a.slices - 1 ? max(a.keep_at, fresh_at) : 1 << 30;
        float *ring = a.ring + (long long)chan * R;
        const float *fresh = a.fresh + (long long)chan * a.fresh_stride - fresh_at;
        auto sample = [&](int i) -> float {
            if (i < lead || (i >= fresh_at && !a.fresh)) return 0.f;
            int p = base + i;
            if (p >= R) p -= R;
            if (!CQT_CHK(a.dbg, 212, p, R)) return 0.f;
            return i >= fresh_at ? __ldcs(fresh + i) : __ldcs(ring + p);
        };
#pragma unroll
        for (int u = 0; u < units; ++u)
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                const int i = 2 * ((tid / S::NC + u * step + q * S::S0) * B + j2);
                int p = base + i;
                if (p >= R) p -= R;
                float2 v;
                // hops, ring lengths and the start of the stream are even: only fresh samples may come unpaired
                if (i >= lead && i + 1 < fresh_at && CQT_CHK(a.dbg, 213, p + 1, R)) v = ld_data(reinterpret_cast<const float2 *>(ring + p));
                else if (i >= fresh_at && a.fresh_pairs) v = __ldcs(reinterpret_cast<const float2 *>(fresh + i));
                else v = make_float2(sample(i), sample(i + 1));
                if (i + 1 >= keep && CQT_CHK(a.dbg, 214, p + 1, R)) {
                    if (i >= keep) ring[p] = v.x;
                    ring[p + 1] = v.y;
                }
                re[u][q] *= v.x; im[u][q] *= v.y;
            }
    } else {
        const float *row = a.x_in + (long long)ch * a.x_stride + 2 * j2;
        const int left = a.valid_len - 2 * j2;   // samples of this column pair's row run that exist
        if (a.aligned) {
            const int whole = left < 2 ? 0 : (left - 2) / (2 * B) + 1;   // rows j1 whose two samples exist
            load_all([&](int j1) -> float2 {
                if (j1 < whole) return __ldcs(reinterpret_cast<const float2 *>(row + (long long)j1 * (2 * B)));   // read once: streaming
                return make_float2(left - j1 * 2 * B == 1 ? __ldcs(row + (long long)j1 * (2 * B)) : 0.f, 0.f);
            });
        } else {
            load_all([&](int j1) -> float2 {
                const float *p = row + (long long)j1 * (2 * B);
                const int n = left - j1 * 2 * B;
                return make_float2(n > 0 ? __ldcs(p) : 0.f, n > 1 ? __ldcs(p + 1) : 0.f);
            });
        }
    }
    __syncthreads();   // the staged tables
#pragma unroll
    for (int u = 0; u < units; ++u) finish_first<S, -1>(buf, tws, tid / S::NC + u * step, col, re[u], im[u]);
    __syncthreads();
    tile_middle<S, -1>(buf, tws, tid);
    float2 *T = a.T + (long long)ch * a.t_pitch + j2;
    // W_Lp^{j2 k1}, k1 = low + q NL, as U[low][j2] V[q][j2]: neighbouring columns read neighbouring entries (a two-level table
    // indexed by the product j2 k1 cost two conflicting shared loads per element), a thread's U is one load
    const float2 *U = a.tw + a.tw_u + j2, *V = a.tw + a.tw_v + j2;
    constexpr int last = S::NL * S::NC / S::T;
#pragma unroll 1
    for (int u = 0; u < last; ++u) {
        const int b = tid / S::NC + u * step, low = S::low(b);
        const float2 wu = __ldg(U + low * B);
        float x[S::RL], y[S::RL];
        last_butterfly<S, -1>(buf, b, col, x, y);
#pragma unroll
        for (int q = 0; q < S::RL; ++q) {
            const int k1 = low + q * S::NL;
            const float2 w = cmul(wu, __ldg(V + q * B));
            if (CQT_CHK(a.dbg, 201, k1 * B + j2, A * B)) T[k1 * B] = cmul(make_float2(x[q], y[q]), w);
        }
    }
}

// ---------------------------------------------------------------- pass R (+ untangle)
// X_k = 1/2 (1 - i w) Z_k + 1/2 (1 + i w) conj Z_{Lp-k}, w = exp(-2 pi i k / N), half_w = w / 2; with z = Z_k,
// zp = Z_{Lp-k}: E = (z + conj zp) / 2, P = -i w (z - conj zp) / 2, X_k = E + P, X_{Lp-k} = conj(E - P)
__device__ __forceinline__ void untangle(float2 z, float2 zp, float2 half_w, float2 &xk, float2 &xm) {
    const float sx = z.x + zp.x, sy = z.y - zp.y, ox = z.x - zp.x, oy = z.y + zp.y;
    const float px = half_w.y * ox + half_w.x * oy, py = half_w.y * oy - half_w.x * ox;
    xk = make_float2(fmaf(0.5f, sx, px), fmaf(0.5f, sy, py));
    xm = make_float2(fmaf(0.5f, sx, -px), py - 0.5f * sy);
}

template <int A, int B>
__global__ void __launch_bounds__(RowsForward<B>::T, 1024 / RowsForward<B>::T) rfft_rows_fwd_kernel(LongArgs a) {
    using S = RowsForward<B>;
    constexpr int TW = S::NC / 2, N = 2 * A * B, Lp = A * B;
    pdl_launch_dependents();
    const int tid = threadIdx.x, ch = blockIdx.y, t = blockIdx.x;
    float2 *buf = smem_long, *tws = buf + S::ELEMS, *wn = tws + B;
    stage_table<B, S::T>(tws, a.tw + a.tw_full_B, tid);
    // the low part of the table of W_N halved: the fold needs w / 2
    stage_table<two_level_entries(N), S::T>(wn, a.tw + a.tw_n, tid, 1 << low_bits(N), 0.5f);
    pdl_wait();   // the tables above belong to the plan; what follows reads the predecessor's output
    {
        const float2 *T = a.T + (long long)ch * a.t_pitch;
        constexpr int R0 = S::R0, units = S::S0 * S::NC / S::T;
        float re[units][R0], im[units][R0];
#pragma unroll
        for (int u = 0; u < units; ++u) {
            const int w = tid + u * S::T, b = w % S::S0, row = row_of<A, TW>(t, w / S::S0);
            const float2 *src = T + row * B + b;
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                const float2 v = CQT_CHK(a.dbg, 202, row * B + b + q * S::S0, Lp) ? ld_data(src + q * S::S0) : make_float2(0.f, 0.f);
                re[u][q] = v.x; im[u][q] = v.y;
            }
        }
        __syncthreads();   // the staged tables
#pragma unroll
        for (int u = 0; u < units; ++u) finish_first<S, -1>(buf, tws, (tid + u * S::T) % S::S0, (tid + u * S::T) / S::S0, re[u], im[u]);
    }
    __syncthreads();
    tile_middle<S, -1>(buf, tws, tid);
    // row r and its mirror, column r + TW: frequency k2 of the one pairs with B - 1 - k2 of the other, that is butterfly
    // b, element q with butterfly NL - 1 - b, element RL - 1 - q
    float2 *X = a.X + (long long)ch * a.x_pitch;
    constexpr int RL = S::RL, C = low_bits(N);
    static_assert(S::NL * TW == S::T, "one pair of butterflies per thread");
    static_assert((A * S::NL) % (1 << C) == 0, "the low part of the table index does not depend on q");
    const bool last_tile = 2 * TW * (t + 1) == A;
    const int r = tid % TW, b = tid / TW;
    float x[RL], y[RL], xm[RL], ym[RL];
    last_butterfly<S, -1>(buf, b, r, x, y);
    last_butterfly<S, -1>(buf, S::NL - 1 - b, r + TW, xm, ym);
    if (last_tile && r == TW - 1) {
        // rows A/2 and 0 pair with themselves: their fold goes through shared memory below
#pragma unroll
        for (int q = 0; q < RL; ++q) {
            buf[S::at(b * RL + q, r)] = make_float2(x[q], y[q]);
            buf[S::at((S::NL - 1 - b) * RL + q, r + TW)] = make_float2(xm[q], ym[q]);
        }
    } else {
        const int k0 = TW * t + 1 + r + A * S::low(b);
        const float2 wlo = wn[k0 & ((1 << C) - 1)];
        const float2 *whi = wn + (1 << C) + (k0 >> C);
#pragma unroll
        for (int q = 0; q < RL; ++q) {
            const int k = k0 + q * (A * S::NL);
            float2 xk, xk_m;
            untangle(make_float2(x[q], y[q]), make_float2(xm[RL - 1 - q], ym[RL - 1 - q]), cmul(wlo, whi[q * ((A * S::NL) >> C)]), xk, xk_m);
            if (!CQT_CHK(a.dbg, 203, k, Lp) || !CQT_CHK(a.dbg, 204, Lp - k, Lp)) continue;
            X[k] = xk;
            X[Lp - k] = xk_m;
        }
    }
    if (!last_tile) return;
    __syncthreads();
    for (int i = tid; i < 2 * (B / 2) + 1; i += S::T) {
        // i < B/2: row A/2, k2 = i with B - 1 - i; else row 0, k2 = i - B/2 with (B - k2) mod B, 0 <= k2 <= B/2
        const bool zero = i >= B / 2;
        const int k2 = zero ? i - B / 2 : i, k2p = zero ? (B - k2) % B : B - 1 - k2, c = zero ? 2 * TW - 1 : TW - 1;
        const float2 z = buf[S::at(S::position(k2), c)], zp = buf[S::at(S::position(k2p), c)];
        const int k = (zero ? 0 : A / 2) + A * k2;
        float2 xk, xk_m;
        untangle(z, zp, two_level<N>(wn, (uint32_t)k), xk, xk_m);
        if (!CQT_CHK(a.dbg, 209, k, Lp)) continue;
        X[k] = xk;
        if (2 * k != Lp) X[Lp - k] = xk_m;   // k = 0: X[Lp]
    }
}

// ---------------------------------------------------------------- host side
template <int A, int B>
struct Forward {
    static const void *cols(bool sliced) {
        return sliced ? (const void *)rfft_cols_fwd_kernel<A, B, true> : (const void *)rfft_cols_fwd_kernel<A, B, false>;
    }
    static const void *rows() { return (const void *)rfft_rows_fwd_kernel<A, B>; }
};

struct ForwardKernels {
    const void *cols = nullptr, *cols_sliced = nullptr, *rows = nullptr;
    int cols_threads = 0, rows_threads = 0, cols_tiles = 0, rows_tiles = 0;
    size_t cols_smem = 0, rows_smem = 0;
};

static ForwardKernels forward_kernels(const cqt_plan &p) {
    ForwardKernels k;
#define X(A_, B_)                                                                                    \
    if (p.lf.A == A_ && p.lf.B == B_) {                                                              \
        using C = ColsForward<A_>;                                                                   \
        using R = RowsForward<B_>;                                                                   \
        k.cols = Forward<A_, B_>::cols(false); k.cols_sliced = Forward<A_, B_>::cols(true); k.rows = Forward<A_, B_>::rows(); \
        k.cols_threads = C::T; k.rows_threads = R::T;                                                \
        k.cols_tiles = B_ / C::NC; k.rows_tiles = A_ / R::NC;                                        \
        k.cols_smem = sizeof(float2) * ((size_t)C::ELEMS + A_);                                     \
        k.rows_smem = sizeof(float2) * ((size_t)R::ELEMS + B_ + p.lf.n_n);                           \
    }
    CQT_LONG_SPLITS(X)
#undef X
    return k;
}

cudaError_t launch_rfft_forward(const cqt_plan &p, const float *x, int64_t x_stride, int64_t batch, int64_t valid_len,
                                float2 *T, float2 *X, cudaStream_t st, const SliceSource *src) {
    LongArgs a = base_args(p, valid_len, x_stride, x);
    a.x_in = x;
    a.T = T;
    a.X = X;
    a.tw_u = p.lf.tw_fwd_u;
    a.tw_v = p.lf.tw_fwd_v;
    if (p.lf.A == 1) {
        if (src) return cudaErrorInvalidValue;
        cudaError_t e = launch_short_rfft_forward(p, a, batch, st);
        note_launch(p, "rfft_rows_fwd", st);
        return e;
    }
    if (src) {
        const long long R = src->ring_len, last = src->first + (src->slices - 1) * src->hop;
        if (src->channels <= 0 || R < p.N + (src->slices - 1) * src->hop || R > INT32_MAX / 2 || (R & 1) || (src->first & 1) || (src->hop & 1))
            return cudaErrorInvalidValue;
        auto clamp = [](long long v) { return (int)std::max<long long>(-(1 << 30), std::min<long long>(1 << 30, v)); };
        a.ring = src->ring; a.slice_win = src->win;
        a.ring_len = (int)R;
        a.ring_base = (int)(((src->first % R) + R) % R);
        a.lead = clamp(-src->first);
        a.hop = (int)src->hop; a.channels = src->channels; a.slices = src->slices;
        a.fresh = src->fresh; a.fresh_stride = src->fresh_stride;
        a.fresh_at = clamp(src->new_first - src->first);
        a.keep_at = clamp(src->keep_from - last);
        a.fresh_pairs = src->fresh && (a.fresh_at & 1) == 0 && (reinterpret_cast<uintptr_t>(src->fresh) & 7) == 0 && (src->fresh_stride & 1) == 0;
    }
    const ForwardKernels k = forward_kernels(p);
    cudaError_t e = launch_long(src ? k.cols_sliced : k.cols, k.cols_tiles, batch, k.cols_threads, k.cols_smem, a, st);
    note_launch(p, "rfft_cols_fwd", st);
    if (e != cudaSuccess) return e;
    e = launch_long(k.rows, k.rows_tiles, batch, k.rows_threads, k.rows_smem, a, st);
    note_launch(p, "rfft_rows_fwd", st);
    return e;
}

int long_cols_last_radix(int64_t A) {
#define X(A_, B_) if (A == A_) return ColsForward<A_>::RL;
    CQT_LONG_SPLITS(X)
#undef X
    return 1;
}

cudaError_t configure_long_forward_kernels(const cqt_plan &p) {
    const ForwardKernels k = forward_kernels(p);
    if (!k.cols) return cudaErrorInvalidDeviceFunction;
    for (const void *fn : {k.cols, k.cols_sliced}) {
        cudaError_t e = allow_dynamic_smem(fn, k.cols_smem, p);
        if (e != cudaSuccess) return e;
    }
    return allow_dynamic_smem(k.rows, k.rows_smem, p);
}

}  // namespace cqt
