// Packed real FFT of a short signal (Lp = N/2 <= 4096) in one kernel, one CTA per signal: the whole transform lies in
// shared memory, with Eq. pack on load and Eq. untangle in the epilogue (forward), overlap-add and Eq. retangle in the
// prologue and unpack on store (inverse).
//
// Bounds: a call with few signals is a chain of latencies (table staging, one round of loads, three butterfly stages,
// one round of stores), so each of these is one round of independent accesses per thread: Lp / 8 threads, compile-time
// radices, the spectrum brought into natural order before the epilogue (the digit-reversed positions of consecutive bins
// sit in one bank), the cover words of all of a thread's bins fetched before the predecessor kernel is waited for.
// With N = 8192 and three signals the run-time planned engine on this path took 18.5 us forward and 38 us inverse.
// A CTA walks several signals when there are more than fit the device, so that the staged tables are read once.
#include <algorithm>

#include "long_common.cuh"

namespace cqt {

extern __shared__ float2 smem_short[];

// Lp = R0 R1 R2 points (R2 = 1: two stages) on T threads
template <int R0_, int R1_, int R2_, int T_>
struct ShortShape {
    static constexpr int R0 = R0_, R1 = R1_, R2 = R2_, T = T_;
    static constexpr int Lp = R0 * R1 * R2, S0 = R1 * R2;
    static constexpr int RL = R2 > 1 ? R2 : R1;     // radix of the last stage
    // one element skipped per last-stage block, one more per first-stage chunk: the last stage reads one position of
    // consecutive chunks, whose distance must be odd
    static constexpr int CHUNK = R2 > 1 ? S0 + R1 + (R1 % 2 == 0 ? 1 : 0) : S0 + 1;
    static constexpr int BUF = R0 * CHUNK;          // elements of the padded buffer (>= Lp)
    static __device__ __forceinline__ int chunk_at(int p) { return R2 > 1 ? p + p / R2 : p; }   // position inside a chunk
};

// Runs the transform; load(j) yields input j, the results of the last stage stay in the thread's registers: butterfly t
// holds frequencies t + q Lp / RL.  The caller's tables become visible at the first barrier.  Returns whether the
// thread has a butterfly.
template <class S, int SIGN, class Load>
__device__ __forceinline__ bool short_fft(float2 *buf, const float2 *twf, Load load, int tid, float (&re)[S::RL], float (&im)[S::RL]) {
    constexpr int R0 = S::R0, R1 = S::R1, R2 = S::R2, S0 = S::S0;
    {
        const bool active = tid < S0;
        float a[R0], b[R0];
        static_assert(S0 <= S::T || S0 % S::T == 0, "one or several full rounds");
        constexpr int rounds = S0 > S::T ? S0 / S::T : 1;
#pragma unroll
        for (int r = 0; r < rounds; ++r) {
            const int p = tid + r * S::T;
            if (active) {
#pragma unroll
                for (int q = 0; q < R0; ++q) {
                    const float2 v = load(p + q * S0);
                    a[q] = v.x; b[q] = v.y;
                }
            }
            if (r == 0) __syncthreads();
            if (active) {
                if (SIGN < 0) Codelet<R0>::run(a, b); else Codelet<R0>::run(b, a);
                apply_twiddle_direct<R0, SIGN>(twf, (uint32_t)p, a, b);
                float2 *d = buf + S::chunk_at(p);
#pragma unroll
                for (int q = 0; q < R0; ++q) d[q * S::CHUNK] = make_float2(a[q], b[q]);
            }
        }
    }
    __syncthreads();
    if constexpr (R2 > 1) {
        constexpr int total = R0 * R2;
        for (int w = tid; w < total; w += S::T) {
            const int k0 = w / R2, np = w % R2;
            float2 *d = buf + k0 * S::CHUNK + np;
            float a[R1], b[R1];
#pragma unroll
            for (int q = 0; q < R1; ++q) {
                const float2 v = d[q * (R2 + 1)];
                a[q] = v.x; b[q] = v.y;
            }
            if (SIGN < 0) Codelet<R1>::run(a, b); else Codelet<R1>::run(b, a);
            apply_twiddle_direct<R1, SIGN>(twf, (uint32_t)(np * R0), a, b);
#pragma unroll
            for (int q = 0; q < R1; ++q) d[q * (R2 + 1)] = make_float2(a[q], b[q]);
        }
        __syncthreads();
    }
    constexpr int total = S::Lp / S::RL;
    static_assert(total <= S::T, "one butterfly per thread in the last stage");
    if (tid >= total) return false;
    // butterfly tid = k0 + R0 k1: its frequencies are tid + q total
    const float2 *d = R2 > 1 ? buf + (tid % R0) * S::CHUNK + (tid / R0) * (R2 + 1) : buf + tid * S::CHUNK;
#pragma unroll
    for (int q = 0; q < S::RL; ++q) {
        const float2 v = d[q];
        re[q] = v.x; im[q] = v.y;
    }
    if (SIGN < 0) Codelet<S::RL>::run(re, im); else Codelet<S::RL>::run(im, re);
    return true;
}

template <class S>
__global__ void __launch_bounds__(S::T, S::T >= 512 ? 2 : 4) short_rfft_forward_kernel(LongArgs a, int batch) {
    pdl_launch_dependents();
    const int tid = threadIdx.x;
    float2 *buf = smem_short, *twf = buf + S::BUF, *wn = twf + S::Lp;
    stage_table<S::Lp, S::T>(twf, a.tw + a.tw_full_B, tid);
    stage_table<two_level_entries(2 * S::Lp), S::T>(wn, a.tw + a.tw_n, tid);
    pdl_wait();
    constexpr int NB = S::Lp / S::RL;
    for (int ch = blockIdx.x; ch < batch; ch += gridDim.x) {
        const float *row = a.x_in + (long long)ch * a.x_stride;
        float re[S::RL], im[S::RL];
        const bool have = short_fft<S, -1>(buf, twf, [&](int j) { return load_packed(row, j, a.valid_len, a.aligned); }, tid, re, im);
        __syncthreads();
        if (have) {
#pragma unroll
            for (int q = 0; q < S::RL; ++q) buf[tid + q * NB] = make_float2(re[q], im[q]);
        }
        __syncthreads();
        float2 *X = a.X + (long long)ch * a.x_pitch;
        // X_k = 1/2 (1 - i w) Z_k + 1/2 (1 + i w) conj Z_{Lp-k},  w = exp(-2 pi i k / N)
#pragma unroll 4
        for (int k = tid; k < S::Lp; k += S::T) {
            const float2 z = buf[k], zp = buf[(S::Lp - k) & (S::Lp - 1)];
            const float2 w = twiddle_s(wn, a.log_n_c, (uint32_t)k);
            const float2 ev = make_float2(0.5f * (z.x + zp.x), 0.5f * (z.y - zp.y));
            const float2 od = make_float2(0.5f * (z.x - zp.x), 0.5f * (z.y + zp.y));
            X[k] = make_float2(ev.x + (w.y * od.x + w.x * od.y), ev.y + (w.y * od.y - w.x * od.x));
            if (k == 0) X[S::Lp] = make_float2(z.x - z.y, 0.f);
        }
        __syncthreads();   // buf is rewritten by the next signal's first stage
    }
}

template <class S, bool MASK>
__global__ void __launch_bounds__(S::T, S::T >= 512 ? 2 : 4) short_rfft_inverse_kernel(LongArgs a, int batch) {
    pdl_launch_dependents();
    const int tid = threadIdx.x;
    float2 *buf = smem_short, *twf = buf + S::BUF, *wn = twf + S::Lp, *nat = wn + a.n_n;
    stage_table<S::Lp, S::T>(twf, a.tw + a.tw_full_B, tid);
    constexpr float s = 0.5f / (float)S::Lp;
    // the low part of the table of W_N times s
    stage_table<two_level_entries(2 * S::Lp), S::T>(wn, a.tw + a.tw_n, tid, 1 << low_bits(2 * S::Lp), s);
    // bin pairs (q, Lp - q): q = tid + u T for q <= Lp/2
    constexpr int NP = S::Lp / 2 / S::T > 0 ? S::Lp / 2 / S::T : 1;
    int32_t cq[NP], cm[NP];
#pragma unroll
    for (int u = 0; u < NP; ++u) {
        const int q = tid + u * S::T;
        const bool ok = q <= S::Lp / 2;
        cq[u] = ok ? __ldg(a.cover + q) : 0;
        cm[u] = ok ? __ldg(a.cover + (S::Lp - q)) : 0;
    }
    __syncthreads();   // the table of W_N is staged
    pdl_wait();
    for (int ch = blockIdx.x; ch < batch; ch += gridDim.x) {
        const float2 *Y = a.Y + (long long)ch * a.y_pitch;
        float2 vq[NP], vm[NP];
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int q = min(tid + u * S::T, S::Lp / 2);
            vq[u] = plane_first<MASK>(a, Y, q, cq[u]);
            vm[u] = plane_first<MASK>(a, Y, S::Lp - q, cm[u]);
        }
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int q = tid + u * S::T, m = S::Lp - q;
            if (q > S::Lp / 2) break;
            plane_rest<MASK>(a, Y, q, cq[u], vq[u]);
            plane_rest<MASK>(a, Y, m, cm[u], vm[u]);
            if (q == 0) { vq[u].y = 0.f; vm[u].y = 0.f; }   // bins 0 and N/2 are made real
            float2 zq, zm;
            retangle(vq[u], vm[u], twiddle_s(wn, a.log_n_c, (uint32_t)q), s, zq, zm);
            nat[q] = zq;
            if (q != 0 && m != q) nat[m] = zm;
        }
        if (tid == 0 && NP * S::T <= S::Lp / 2) {   // the pair of the middle bin with itself
            constexpr int q = S::Lp / 2;
            const float2 xq = plane_sum<MASK>(a, Y, q, __ldg(a.cover + q));
            float2 zq, zm;
            retangle(xq, xq, twiddle_s(wn, a.log_n_c, (uint32_t)q), s, zq, zm);
            nat[q] = zq;
        }
        __syncthreads();
        float re[S::RL], im[S::RL];
        const bool have = short_fft<S, +1>(buf, twf, [&](int q) { return nat[q]; }, tid, re, im);
        constexpr int NB = S::Lp / S::RL;
        float *row = a.x_out + (long long)ch * a.x_stride;
        if (have) {
#pragma unroll
            for (int q = 0; q < S::RL; ++q) store_packed(row, tid + q * NB, make_float2(re[q], im[q]), a.valid_len, a.aligned);
        }
        // nat is next written after every thread has passed the barriers of this transform; buf after the barrier below
    }
}

using S4096 = ShortShape<16, 16, 16, 512>;
using S2048 = ShortShape<16, 16, 8, 256>;
using S1024 = ShortShape<16, 8, 8, 128>;
using S512 = ShortShape<8, 8, 8, 64>;
using S256 = ShortShape<16, 16, 1, 32>;
using S128 = ShortShape<16, 8, 1, 32>;
using S64 = ShortShape<8, 8, 1, 32>;
using S32 = ShortShape<8, 4, 1, 32>;
#define CQT_SHORT_SHAPES(X) X(S4096) X(S2048) X(S1024) X(S512) X(S256) X(S128) X(S64) X(S32)

struct ShortKernel {
    const void *fn = nullptr;
    int threads = 0;
    size_t smem = 0;
};

static ShortKernel short_kernel(const cqt_plan &p, bool forward) {
    const FftPlan &fp = p.ffts[p.lf.fft_B];
    ShortKernel k;
#define X(S)                                                                                                             \
    if (p.lf.Lp == S::Lp && fp.st[0].radix == S::R0 && fp.st[1].radix == S::R1) {                                         \
        k.fn = forward ? (const void *)short_rfft_forward_kernel<S> : (cover_is_mask(p) ? (const void *)short_rfft_inverse_kernel<S, true> : (const void *)short_rfft_inverse_kernel<S, false>);         \
        k.threads = S::T;                                                                                                 \
        k.smem = sizeof(float2) * ((size_t)S::BUF + S::Lp + p.lf.n_n + (forward ? 0 : S::Lp));                            \
    }
    CQT_SHORT_SHAPES(X)
#undef X
    return k;
}

static cudaError_t launch_short(const cqt_plan &p, LongArgs &a, int64_t batch, bool forward, cudaStream_t st) {
    const ShortKernel k = short_kernel(p, forward);
    if (!k.fn) return cudaErrorInvalidDeviceFunction;
    // as many CTAs as are resident at once
    const int64_t per_sm = std::min<int64_t>({(int64_t)((p.max_smem_optin + 1024) / (k.smem + 1024)), (int64_t)1024 / k.threads, (int64_t)16});
    int n = (int)batch;
    void *args[] = {&a, &n};
    return launch_kernel(k.fn, dim3((unsigned)std::min<int64_t>(batch, std::max<int64_t>(1, per_sm) * p.sm_count)), dim3((unsigned)k.threads), args, k.smem, st);
}
cudaError_t launch_short_rfft_forward(const cqt_plan &p, LongArgs &a, int64_t batch, cudaStream_t st) { return launch_short(p, a, batch, true, st); }
cudaError_t launch_short_rfft_inverse(const cqt_plan &p, LongArgs &a, int64_t batch, cudaStream_t st) { return launch_short(p, a, batch, false, st); }

cudaError_t configure_short_fft_kernels(const cqt_plan &p) {
    for (bool forward : {true, false}) {
        const ShortKernel k = short_kernel(p, forward);
        if (!k.fn) return cudaErrorInvalidDeviceFunction;
        cudaError_t e = allow_dynamic_smem(k.fn, k.smem, p);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace cqt
