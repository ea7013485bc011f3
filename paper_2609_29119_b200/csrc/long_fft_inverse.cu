// Packed inverse real FFT of length N, two passes; the mirror image of long_fft_forward.cu (index split, tiles, rows).
//   pass R': a CTA owns the same rows as in the forward pass R; per bin pair (q, Lp - q) it forms X^_q = sum over the
//            covering bands once and Z_q, Z_{Lp-q} by Eq. retangle, then the inverse B-point DFT over q2, times
//            conj W_Lp^{j2 q1}, written transposed to Tinv[j2][q1].
//   pass C': inverse A-point DFT over q1, unpacked to x[2j], x[2j+1]; only valid_len samples are written.
//
// Weighted-bin scratch: P planes of Lp+1 bins per signal, P the largest number of bands covering one bin.  A band writes the
// lowest plane that is free at its first bin (interval colouring at plan creation; with more than 31 planes band b writes plane
// b mod P), so two bands of one plane never share a bin and the sum over the bands covering bin k reads their planes at
// index k: coalesced, in fixed order, no atomics.
//
// Bounds: issue slots and, in pass R', the latency of a chain of loads (cover word, planes).  The two operands of every
// fold feed two butterflies of one thread, so sums and fold stay in its registers and the tile is written once; cover
// words belong to the plan and are fetched before the predecessor kernel is waited for; up to 31 planes the word is a
// bit mask of the planes that hold the bin (MASK).  The last stage stores straight to Tinv.  32 signals of
// N = 2^19 before (fold, transform and transposition through shared memory, run-time strides): 88 us + 35 us.
#include "long_passes.cuh"

namespace cqt {

extern __shared__ float2 smem_long[];

template <int A, int B, bool MASK>
__global__ void __launch_bounds__(RowsInverse<B>::T, 1024 / RowsInverse<B>::T) irfft_rows_kernel(LongArgs a) {
    using S = RowsInverse<B>;
    constexpr int TW = S::NC / 2, N = 2 * A * B, Lp = A * B, R0 = S::R0, S0 = S::S0, C = low_bits(N);
    constexpr int units = S0 * TW / S::T, step = S::T / TW;
    static_assert(units * S::T == S0 * TW && S::T % TW == 0, "whole rounds");
    static_assert((A * S0) % (1 << C) == 0, "the low part of the table index does not depend on q");
    constexpr float s = 0.5f / (float)Lp;    // a power of two
    pdl_launch_dependents();
    const int tid = threadIdx.x, ch = blockIdx.y, t = blockIdx.x;
    float2 *buf = smem_long, *tws = buf + S::ELEMS, *wn = tws + B;
    stage_table<B, S::T>(tws, a.tw + a.tw_full_B, tid);
    // the low part of the table of W_N times s
    stage_table<two_level_entries(N), S::T>(wn, a.tw + a.tw_n, tid, 1 << C, s);
    // thread: column r and its mirror r + TW; unit u: butterfly b = b0 + u step of the one, S0 - 1 - b of the other, whose
    // operands are the bins k = k0 + A (u step + q S0) and Lp - k
    const int r = tid % TW, b0 = tid / TW;
    const bool last_tile = 2 * TW * (t + 1) == A, spare = last_tile && r == TW - 1;
    const int k0 = TW * t + 1 + r + A * b0;
    int32_t cq[units][R0], cm[units][R0];
#pragma unroll
    for (int u = 0; u < units; ++u)
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            const int k = k0 + A * (u * step + q * S0);
            cq[u][q] = __ldg(a.cover + k);
            cm[u][q] = __ldg(a.cover + (Lp - k));
        }
    __syncthreads();   // the staged tables
    pdl_wait();        // they belong to the plan; what follows reads the predecessor's output
    const float2 *Y = a.Y + (long long)ch * a.y_pitch;
    if (last_tile) {
        // rows A/2 (column TW - 1) and 0 (column 2 TW - 1) pair with themselves: their inputs go through shared memory.
        // i < B/2: row A/2, q2 = i with B - 1 - i; else row 0, q2 = i - B/2 with (B - q2) mod B, 0 <= q2 <= B/2
        for (int i = tid; i < 2 * (B / 2) + 1; i += S::T) {
            const bool zero = i >= B / 2;
            const int q2 = zero ? i - B / 2 : i, q2m = zero ? B - q2 : B - 1 - q2, col = zero ? 2 * TW - 1 : TW - 1;
            const int q = (zero ? 0 : A / 2) + A * q2;
            float2 xq = plane_sum<MASK>(a, Y, q, __ldg(a.cover + q)), xm = plane_sum<MASK>(a, Y, Lp - q, __ldg(a.cover + (Lp - q)));
            if (q == 0) { xq.y = 0.f; xm.y = 0.f; }   // bins 0 and N/2 are made real
            float2 zq, zm;
            retangle(xq, xm, two_level<N>(wn, (uint32_t)q), s, zq, zm);
            buf[S::at(q2, col)] = zq;
            if (q2m < B && q2m != q2) buf[S::at(q2m, col)] = zm;
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < units; ++u) {
        const int b = b0 + u * step;
        float x[R0], y[R0], xm[R0], ym[R0];
        if (spare) {
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                const float2 v = buf[S::at(b + q * S0, r)], w = buf[S::at(S0 - 1 - b + q * S0, r + TW)];
                x[q] = v.x; y[q] = v.y; xm[q] = w.x; ym[q] = w.y;
            }
        } else {
            const int k = k0 + A * u * step;
            const float2 wlo = wn[k & ((1 << C) - 1)];
            const float2 *whi = wn + (1 << C) + (k >> C);
            float2 vq[R0], vm[R0];
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                const int kq = k + q * (A * S0);
                vq[q] = plane_first<MASK>(a, Y, kq, cq[u][q]);
                vm[q] = plane_first<MASK>(a, Y, Lp - kq, cm[u][q]);
            }
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                const int kq = k + q * (A * S0);
                plane_rest<MASK>(a, Y, kq, cq[u][q], vq[q]);
                plane_rest<MASK>(a, Y, Lp - kq, cm[u][q], vm[q]);
                float2 zq, zm;
                retangle(vq[q], vm[q], cmul(wlo, whi[q * ((A * S0) >> C)]), s, zq, zm);
                x[q] = zq.x; y[q] = zq.y;
                xm[R0 - 1 - q] = zm.x; ym[R0 - 1 - q] = zm.y;
            }
        }
        finish_first<S, +1>(buf, tws, b, r, x, y);
        finish_first<S, +1>(buf, tws, S0 - 1 - b, r + TW, xm, ym);
    }
    __syncthreads();
    tile_middle<S, +1>(buf, tws, tid);
    // transposed intermediate Tinv[j2][q1]: consecutive threads take consecutive columns, runs of TW rows
    const int col = tid % S::NC, q1 = row_of<A, TW>(t, col);
    float2 *T = a.T + (long long)ch * a.t_pitch + q1;
    const float2 *U = a.tw + a.tw_u + q1, *V = a.tw + a.tw_v + q1;   // W_Lp^{j2 q1} = U[low][q1] V[q][q1], j2 = low + q NL
    constexpr int last = S::NL * S::NC / S::T;
#pragma unroll 1
    for (int u = 0; u < last; ++u) {
        const int b = tid / S::NC + u * (S::T / S::NC), low = S::low(b);
        const float2 wu = __ldg(U + low * A);
        float x[S::RL], y[S::RL];
        last_butterfly<S, +1>(buf, b, col, x, y);
#pragma unroll
        for (int q = 0; q < S::RL; ++q) {
            const int j2 = low + q * S::NL;
            const float2 w = cmul(wu, __ldg(V + q * A));
            if (CQT_CHK(a.dbg, 207, j2 * A + q1, Lp)) T[j2 * A] = cmul(make_float2(x[q], y[q]), cconj(w));
        }
    }
}

template <int A, int B>
__global__ void __launch_bounds__(ColsInverse<A>::T, 1024 / ColsInverse<A>::T) irfft_cols_kernel(LongArgs a) {
    using S = ColsInverse<A>;
    pdl_launch_dependents();
    const int tid = threadIdx.x, j2_0 = blockIdx.x * S::NC, ch = blockIdx.y;
    float2 *buf = smem_long, *tws = buf + S::ELEMS;
    stage_table<A, S::T>(tws, a.tw + a.tw_full_A, tid);
    pdl_wait();   // the table belongs to the plan; what follows reads the predecessor's output
    {
        // a column of Tinv[j2][q1] is a contiguous run: consecutive threads take consecutive q1
        const float2 *T = a.T + (long long)ch * a.t_pitch + (long long)j2_0 * A;
        constexpr int R0 = S::R0, units = S::S0 * S::NC / S::T;
        float re[units][R0], im[units][R0];
#pragma unroll
        for (int u = 0; u < units; ++u) {
            const int w = tid + u * S::T, i = (w / S::S0) * A + w % S::S0;
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                const float2 v = CQT_CHK(a.dbg, 208, (long long)j2_0 * A + i + q * S::S0, A * B) ? ld_data(T + i + q * S::S0) : make_float2(0.f, 0.f);
                re[u][q] = v.x; im[u][q] = v.y;
            }
        }
        __syncthreads();   // the staged table
#pragma unroll
        for (int u = 0; u < units; ++u) finish_first<S, +1>(buf, tws, (tid + u * S::T) % S::S0, (tid + u * S::T) / S::S0, re[u], im[u]);
    }
    __syncthreads();
    tile_middle<S, +1>(buf, tws, tid);
    const int col = tid % S::NC, j2 = j2_0 + col, left = a.valid_len - 2 * j2;
    float *row = a.x_out + (long long)ch * a.x_stride + 2 * j2;
    constexpr int last = S::NL * S::NC / S::T;
#pragma unroll 1
    for (int u = 0; u < last; ++u) {
        const int b = tid / S::NC + u * (S::T / S::NC), low = S::low(b);
        float x[S::RL], y[S::RL];
        last_butterfly<S, +1>(buf, b, col, x, y);
#pragma unroll
        for (int q = 0; q < S::RL; ++q) {
            const int j1 = low + q * S::NL, n = left - j1 * (2 * B);   // samples of the pair that exist
            float *d = row + (long long)j1 * (2 * B);
            if (n > 1 && a.aligned) __stcs(reinterpret_cast<float2 *>(d), make_float2(x[q], y[q]));
            else {
                if (n > 0) __stcs(d, x[q]);
                if (n > 1) __stcs(d + 1, y[q]);
            }
        }
    }
}

// ---------------------------------------------------------------- host side
struct InverseKernels {
    const void *rows = nullptr, *cols = nullptr;
    int rows_threads = 0, cols_threads = 0, rows_tiles = 0, cols_tiles = 0;
    size_t rows_smem = 0, cols_smem = 0;
};

static InverseKernels inverse_kernels(const cqt_plan &p) {
    InverseKernels k;
#define X(A_, B_)                                                                                                  \
    if (p.lf.A == A_ && p.lf.B == B_) {                                                                            \
        using R = RowsInverse<B_>;                                                                                 \
        using C = ColsInverse<A_>;                                                                                 \
        k.rows = cover_is_mask(p) ? (const void *)irfft_rows_kernel<A_, B_, true> : (const void *)irfft_rows_kernel<A_, B_, false>; \
        k.cols = (const void *)irfft_cols_kernel<A_, B_>;                                                          \
        k.rows_threads = R::T; k.cols_threads = C::T;                                                              \
        k.rows_tiles = A_ / R::NC; k.cols_tiles = B_ / C::NC;                                                      \
        k.rows_smem = sizeof(float2) * ((size_t)R::ELEMS + B_ + p.lf.n_n);                                         \
        k.cols_smem = sizeof(float2) * ((size_t)C::ELEMS + A_);                                                    \
    }
    CQT_LONG_SPLITS(X)
#undef X
    return k;
}

cudaError_t launch_rfft_inverse(const cqt_plan &p, const float2 *Y, float2 *T, float *x, int64_t x_stride,
                                int64_t batch, int64_t valid_len, cudaStream_t st) {
    LongArgs a = base_args(p, valid_len, x_stride, x);
    a.x_out = x;
    a.T = T;
    a.Y = Y;
    a.tw_u = p.lf.tw_inv_u;
    a.tw_v = p.lf.tw_inv_v;
    if (p.lf.A == 1) {
        cudaError_t e = launch_short_rfft_inverse(p, a, batch, st);
        note_launch(p, "irfft_rows", st);
        return e;
    }
    const InverseKernels k = inverse_kernels(p);
    cudaError_t e = launch_long(k.rows, k.rows_tiles, batch, k.rows_threads, k.rows_smem, a, st);
    note_launch(p, "irfft_rows", st);
    if (e != cudaSuccess) return e;
    e = launch_long(k.cols, k.cols_tiles, batch, k.cols_threads, k.cols_smem, a, st);
    note_launch(p, "irfft_cols", st);
    return e;
}

int long_rows_inverse_last_radix(int64_t B) {
#define X(A_, B_) if (B == B_) return RowsInverse<B_>::RL;
    CQT_LONG_SPLITS(X)
#undef X
    return 1;
}

cudaError_t configure_long_inverse_kernels(const cqt_plan &p) {
    const InverseKernels k = inverse_kernels(p);
    if (!k.rows) return cudaErrorInvalidDeviceFunction;
    cudaError_t e = allow_dynamic_smem(k.rows, k.rows_smem, p);
    return e != cudaSuccess ? e : allow_dynamic_smem(k.cols, k.cols_smem, p);
}

}  // namespace cqt
