// Bands whose length has a prime factor above 5 (the multiple-of-4 length policy makes them), M = 4 m with m > 32.
//
// One radix-4 step, taken on load, turns the M-point DFT into four independent m-point ones,
//   X[k0 + 4 k'] = sum_n' W_m^{n' k'} y_k0[n'],   y_k0[n'] = W_M^{n' k0} sum_q W_4^{q k0} x[n' + q m],
// and each of them is a chirp-z (Bluestein) transform,
//   X[k0 + 4 k'] = c[k'] sum_n' (y_k0[n'] c[n']) conj(c[k' - n']),   c[n] = exp(-i pi n^2 / m),
// the convolution through two power-of-two transforms of length L >= 2 m - 1 in shared memory.  A positive exponent is
// the same on conjugated input and output.
//
// Bounds: latency.  Such bands come in single signals more than in batches, and one M-point chirp-z with L >= 2 M - 1
// on the run-time planned engine was 31 - 52 us of a 65 us analysis (M up to 5,000, nine passes through shared memory).
// Four sub-transforms have a quarter of the points each and go to CTAs of their own when they are long; radices are
// compile-time; the last forward stage, the product with the filter's spectrum and the first inverse stage act on the
// same elements and stay in registers, so a sub-transform of up to 4,096 points is five passes.  The price is that
// every input is read by four work items, from the L2.
#include <algorithm>

#include "band_common.cuh"

namespace cqt {

// L = R0 R1 R2 R3 (trailing ones: fewer stages); T threads per sub-transform
template <int R0_, int R1_, int R2_, int R3_>
struct ChirpShape {
    static constexpr int R0 = R0_, R1 = R1_, R2 = R2_, R3 = R3_;
    static constexpr int L = R0 * R1 * R2 * R3, S0 = L / R0;
    static constexpr int RL = R3 > 1 ? R3 : (R2 > 1 ? R2 : R1);
    static constexpr int T = L / 16 < kChirpThreads ? L / 16 : kChirpThreads;
    static constexpr int PER_CTA = kChirpThreads / T;
    // one element skipped per RL positions, an odd number of elements between first-stage chunks (bank spread)
    static __device__ __host__ constexpr int at(int p) { return L > R0 * RL ? p + p / RL : p; }
    static constexpr int CHUNK = (at(S0 - 1) + 1) | 1;
    static constexpr int BUF = R0 * CHUNK;
};
using C128 = ChirpShape<16, 8, 1, 1>;
using C256 = ChirpShape<16, 16, 1, 1>;
using C512 = ChirpShape<8, 8, 8, 1>;
using C1024 = ChirpShape<16, 8, 8, 1>;
using C2048 = ChirpShape<16, 16, 8, 1>;
using C4096 = ChirpShape<16, 16, 16, 1>;
using C8192 = ChirpShape<16, 8, 8, 8>;
#define CQT_CHIRP_SHAPES(X) X(C8192) X(C4096) X(C2048) X(C1024) X(C512) X(C256) X(C128)

extern __shared__ float2 smem_chirp[];

// A butterfly of a stage between the first and the last, in place; forward: butterfly, then twiddles W^{np q}; inverse:
// conjugate twiddles, then the inverse butterfly.
template <int R, int SIGN>
__device__ __forceinline__ void chirp_stage(float2 *d, int step, const float2 *twf, uint32_t y) {
    float re[R], im[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const float2 v = d[q * step];
        re[q] = v.x; im[q] = v.y;
    }
    if (SIGN > 0) apply_twiddle_direct<R, +1>(twf, y, re, im);
    if (SIGN < 0) Codelet<R>::run(re, im); else Codelet<R>::run(im, re);
    if (SIGN < 0) apply_twiddle_direct<R, -1>(twf, y, re, im);
#pragma unroll
    for (int q = 0; q < R; ++q) d[q * step] = make_float2(re[q], im[q]);
}

// stage with sub-transforms of length n, radix R (stride n / R), tmul = L / n; every sub-transform's positions lie in
// one first-stage chunk
template <class S, int R, int N_CUR, int SIGN>
__device__ __forceinline__ void chirp_middle(float2 *buf, const float2 *twf, int t) {
    constexpr int s = N_CUR / R, blocks = S::S0 / N_CUR;
    for (int w = t; w < S::L / R; w += S::T) {
        const int np = w % s, blk = w / s, k0 = blk / blocks, in = (blk % blocks) * N_CUR + np;
        static_assert(s % S::RL == 0, "the skipped elements lie at multiples of the stride");
        chirp_stage<R, SIGN>(buf + k0 * S::CHUNK + S::at(in), S::at(s), twf, (uint32_t)(np * (S::L / N_CUR)));
    }
    __syncthreads();
}

// The convolution of one sub-transform on T threads.  load(n), n < m: chirped input; filter: spectrum of the conjugate
// chirp over L, natural order; store(n, v), n < m: convolution.
template <class S, class Load, class Store>
__device__ __forceinline__ void chirp_convolve(float2 *buf, const float2 *twf, const float2 *__restrict__ filter, int m, bool active, int t,
                                               Load load, Store store) {
    constexpr int R0 = S::R0, S0 = S::S0, RL = S::RL;
    constexpr int N1 = S0;                    // length of the sub-transforms of the second stage
    for (int b = t; b < S0; b += S::T) {
        float re[R0], im[R0];
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            const int n = b + q * S0;
            // m <= L / 2: the upper half of the inputs is zero
            const float2 v = q < (R0 + 1) / 2 && active && n < m ? load(n) : make_float2(0.f, 0.f);
            re[q] = v.x; im[q] = v.y;
        }
        Codelet<R0>::run(re, im);
        if (b == t) __syncthreads();          // the staged twiddle table
        apply_twiddle_direct<R0, -1>(twf, (uint32_t)b, re, im);
        float2 *d = buf + S::at(b);
#pragma unroll
        for (int q = 0; q < R0; ++q) d[q * S::CHUNK] = make_float2(re[q], im[q]);
    }
    __syncthreads();
    if constexpr (S::R2 > 1) chirp_middle<S, S::R1, N1, -1>(buf, twf, t);
    if constexpr (S::R3 > 1) chirp_middle<S, S::R2, N1 / S::R1, -1>(buf, twf, t);
    // last forward stage, filter, first inverse stage: butterfly w holds frequencies w + q L / RL
    for (int w = t; w < S::L / RL; w += S::T) {
        // w = k0 + R0 (k1 + R1 (k2 ...)), position ((k0 R1 + k1) R2 + ...) RL
        int in;
        if constexpr (S::R3 > 1) in = ((w / R0) % S::R1) * (S::R2 * RL) + (w / (R0 * S::R1)) * RL;
        else if constexpr (S::R2 > 1) in = (w / R0) * RL;
        else in = 0;
        float2 *d = buf + (w % R0) * S::CHUNK + S::at(in);
        float re[RL], im[RL];
#pragma unroll
        for (int q = 0; q < RL; ++q) {
            const float2 v = d[q];
            re[q] = v.x; im[q] = v.y;
        }
        Codelet<RL>::run(re, im);
#pragma unroll
        for (int q = 0; q < RL; ++q) {
            const float2 f = __ldg(filter + w + q * (S::L / RL));
            const float2 v = cmul(make_float2(re[q], im[q]), f);
            re[q] = v.x; im[q] = v.y;
        }
        Codelet<RL>::run(im, re);
#pragma unroll
        for (int q = 0; q < RL; ++q) d[q] = make_float2(re[q], im[q]);
    }
    __syncthreads();
    if constexpr (S::R3 > 1) chirp_middle<S, S::R2, N1 / S::R1, +1>(buf, twf, t);
    if constexpr (S::R2 > 1) chirp_middle<S, S::R1, N1, +1>(buf, twf, t);
    for (int b = t; b < S0; b += S::T) {
        float re[R0], im[R0];
        const float2 *d = buf + S::at(b);
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            const float2 v = d[q * S::CHUNK];
            re[q] = v.x; im[q] = v.y;
        }
        apply_twiddle_direct<R0, +1>(twf, (uint32_t)b, re, im);
        Codelet<R0>::run(im, re);
#pragma unroll
        for (int q = 0; q < R0; ++q)
            if (q < (R0 + 1) / 2 && active && b + q * S0 < m) store(b + q * S0, make_float2(re[q], im[q]));
    }
}

struct ChirpArgs {
    BandArgs b;
    const ChirpRec *recs;
    ChirpSegment seg[kChirpLengths];   // by length, longest first
};

template <bool ANALYSIS, class S>
__device__ __forceinline__ void chirp_cta(const ChirpArgs &a, const ChirpSegment &sg) {
    const int g = (int)threadIdx.x / S::T, t = (int)threadIdx.x % S::T;
    float2 *twf = smem_chirp, *buf = smem_chirp + S::L + g * S::BUF;
    // sub-transform index: k0 fastest (the four read the same input), then signal, then band
    const int idx = ((int)blockIdx.x - sg.cta0) * S::PER_CTA + g;
    const int k0 = idx & 3, item = idx >> 2;
    const bool active = item < sg.n_bands * a.b.batch;
    const int band = active ? item / a.b.batch : 0, ch = active ? item - band * a.b.batch : 0;
    const ChirpRec &cr = a.recs[sg.first_band + band];
    const BandRec br = cr.br;
    const int m = br.M >> 2;
    const float2 *pre = a.b.tw + cr.pre_off + k0 * m, *post = a.b.tw + cr.pre_off, *filter = a.b.tw + cr.filter_off;
    for (int i = threadIdx.x; i < S::L; i += kChirpThreads) twf[i] = __ldg(a.b.tw + cr.tw_full_off + i);
    chain_begin(a.b);
    const float *tab = a.b.table + br.tab_off;
    // W_4^{q k0}: even k0: (x0 + x2) +- (x1 + x3), odd: (x0 - x2) -+ i (x1 - x3); then W_M^{n k0} and the chirp
    auto combine = [&](float2 x0, float2 x1, float2 x2, float2 x3, int n) -> float2 {
        const float s = (k0 & 1) ? -1.f : 1.f;
        const float2 e = make_float2(fmaf(s, x2.x, x0.x), fmaf(s, x2.y, x0.y)), o = make_float2(fmaf(s, x3.x, x1.x), fmaf(s, x3.y, x1.y));
        const float u = (k0 & 2) ? -1.f : 1.f;
        // k0 = 1: e - i o, k0 = 3: e + i o
        const float2 v = (k0 & 1) ? make_float2(fmaf(u, o.y, e.x), fmaf(-u, o.x, e.y)) : make_float2(fmaf(u, o.x, e.x), fmaf(u, o.y, e.y));
        return cmul(v, __ldg(pre + n));
    };
    if constexpr (ANALYSIS) {
        const float2 *X = a.b.spec + (long long)ch * a.b.spec_pitch;
        float2 *out = a.b.coef + coef_row(a.b.row0, a.b.rows, ch) * a.b.coeff_count + br.coeff_off;
        auto in = [&](int n) { return cconj(slot_value<true>(br, tab, X, a.b.N, n, a.b.dbg)); };
        chirp_convolve<S>(buf, twf, filter, m, active, t, [&](int n) { return combine(in(n), in(n + m), in(n + 2 * m), in(n + 3 * m), n); },
                          [&](int n, float2 v) { out[k0 + 4 * n] = cconj(cmul(v, __ldg(post + n))); });
    } else {
        const float2 *c = a.b.coef + coef_row(a.b.row0, a.b.rows, ch) * a.b.coeff_count + br.coeff_off;
        float2 *Y = a.b.Y + (long long)ch * a.b.y_pitch + br.y_off;
        const bool fold = a.b.fold && br.side != 0;
        auto in = [&](int n) {
            const float2 v = ld_chained(c + n);
            return fold ? make_float2(2.f * v.x, 0.f) : v;
        };
        chirp_convolve<S>(buf, twf, filter, m, active, t, [&](int n) { return combine(in(n), in(n + m), in(n + 2 * m), in(n + 3 * m), n); },
                          [&](int n, float2 v) { slot_store(br, tab, Y, a.b.N, k0 + 4 * n, cmul(v, __ldg(post + n))); });
    }
}

template <bool ANALYSIS>
__global__ void __launch_bounds__(kChirpThreads, 2) chirp_bands_kernel(ChirpArgs a) {
    chain_enter(a.b);
    int i = 0;
#define X(S)                                                                                               \
    if ((int)blockIdx.x >= a.seg[i].cta0 && (int)blockIdx.x < a.seg[i].cta0 + a.seg[i].n_cta) chirp_cta<ANALYSIS, S>(a, a.seg[i]); \
    ++i;
    CQT_CHIRP_SHAPES(X)
#undef X
    chain_end(a.b);
}

static const int kChirpL[kChirpLengths] = {8192, 4096, 2048, 1024, 512, 256, 128};

size_t chirp_smem(const cqt_plan &p) {
    size_t most = 0;
    int i = 0;
#define X(S)                                                                                                              \
    static_assert(S::L >= 128 && S::L <= 8192, "kChirpL");                                                                \
    if (p.chirp.n_bands[i]) most = std::max(most, sizeof(float2) * ((size_t)S::L + (size_t)S::PER_CTA * S::BUF));         \
    ++i;
    CQT_CHIRP_SHAPES(X)
#undef X
    return most;
}

int chirp_grid(const cqt_plan &p, int64_t batch, ChirpSegment *seg) {
    int64_t grid = 0;
    int band = 0;
    for (int i = 0; i < kChirpLengths; ++i) {
        const int per_cta = std::max(1, kChirpThreads * 16 / kChirpL[i]);
        const int64_t ctas = (4 * (int64_t)p.chirp.n_bands[i] * batch + per_cta - 1) / per_cta;
        if (seg) seg[i] = ChirpSegment{(int)grid, (int)ctas, band, p.chirp.n_bands[i]};
        band += p.chirp.n_bands[i];
        grid += ctas;
    }
    return (int)std::min<int64_t>(grid, INT32_MAX);
}

// position of a sub-transform length in the plan's length list, -1 if there is none
int chirp_length_index(int64_t m) {
    for (int i = kChirpLengths - 1; i >= 0; --i)
        if (m > kChirpL[kChirpLengths - 1] / 4 && kChirpL[i] >= 2 * m - 1) return i;
    return -1;
}
int chirp_length(int index) { return kChirpL[index]; }

cudaError_t launch_chirp(const cqt_plan &p, bool analysis, const BandArgs &b, cudaStream_t st) {
    ChirpArgs a{};
    a.b = b;
    a.recs = p.chirp.d_recs;
    const int grid = chirp_grid(p, b.batch, a.seg);
    void *args[] = {&a};
    const void *fn = analysis ? (const void *)chirp_bands_kernel<true> : (const void *)chirp_bands_kernel<false>;
    cudaError_t e = launch_kernel(fn, dim3((unsigned)grid), dim3(kChirpThreads), args, chirp_smem(p), st);
    note_launch(p, analysis ? "bands_from_spectrum/chirp" : "bands_to_spectrum/chirp", st);
    return e;
}

cudaError_t configure_chirp_kernels(const cqt_plan &p) {
    if (p.chirp.recs.empty()) return cudaSuccess;
    cudaError_t e = allow_dynamic_smem((const void *)chirp_bands_kernel<true>, chirp_smem(p), p);
    return e != cudaSuccess ? e : allow_dynamic_smem((const void *)chirp_bands_kernel<false>, chirp_smem(p), p);
}

}  // namespace cqt
