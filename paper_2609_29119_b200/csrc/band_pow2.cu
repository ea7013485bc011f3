// Bands of 256 ... 16,384 coefficients in plans whose longer bands all have power-of-two lengths (the power-of-two length
// policy, one length per octave).
//
// Bounds: issue slots.  On the run-time planned engine such a band costs 34 instructions per element and radix stage
// (strides, digit loops and two-level twiddle look-ups at run time) and 4 - 5 stages.  Here radices and strides are
// compile-time: 16 elements per thread, at most radix 16, 2 - 4 stages.  A stage's twiddles are rows w, w^2, w^4, w^8 in
// the order in which the threads read them: coalesced loads from the L1, none from shared memory, no table to stage, no
// bank conflicts; the other powers are products of at most three of those.  Short bands share a CTA (the same number
// of threads for each), and all lengths go in one launch (8,192 and 16,384 in a second one), longest first.
// Multi-resolution layout, 128 signals of 2^16 samples: 129 us of band kernels in analysis and 123 us in synthesis before.
#include <algorithm>

#include "band_common.cuh"
#include "twiddle_rows.cuh"

namespace cqt {

// L = R0 R1 R2 R3 (trailing ones: fewer stages) on T threads of a CTA of THREADS
template <int R0_, int R1_, int R2_, int R3_, int THREADS_>
struct Pow2Shape {
    static constexpr int R0 = R0_, R1 = R1_, R2 = R2_, R3 = R3_, THREADS = THREADS_;
    static constexpr int L = R0 * R1 * R2 * R3, S0 = L / R0, S1 = S0 / R1, S2 = S1 / R2;
    static constexpr int RL = R3 > 1 ? R3 : (R2 > 1 ? R2 : R1), NL = L / RL;
    static constexpr int T = L / 16 < THREADS ? L / 16 : THREADS, PER_CTA = THREADS / T;
    // one element skipped per RL positions, an odd number of elements between first-stage chunks (bank spread)
    static __host__ __device__ constexpr int at(int p) { return R2 > 1 ? p + p / RL : p; }
    static constexpr int CHUNK = (at(S0 - 1) + 1) | 1, BUF = R0 * CHUNK;
    // twiddle rows of the stages before the last, one after another
    static constexpr int TW1 = twiddle_rows(R0) * S0, TW2 = TW1 + (R2 > 1 ? twiddle_rows(R1) * S1 : 0), TW_COUNT = TW2 + (R3 > 1 ? twiddle_rows(R2) * S2 : 0);
};
using P256 = Pow2Shape<16, 16, 1, 1, 256>;
using P512 = Pow2Shape<8, 8, 8, 1, 256>;
using P1024 = Pow2Shape<16, 8, 8, 1, 256>;
using P2048 = Pow2Shape<16, 16, 8, 1, 256>;
using P4096 = Pow2Shape<16, 16, 16, 1, 256>;
using P8192 = Pow2Shape<16, 8, 8, 8, 512>;
using P16384 = Pow2Shape<16, 16, 8, 8, 512>;
// longest first
#define CQT_POW2_LONG(X) X(P16384) X(P8192)
#define CQT_POW2_SHORT(X) X(P4096) X(P2048) X(P1024) X(P512) X(P256)

template <int T, int THREADS>
__device__ __forceinline__ void group_sync() {
    if constexpr (T <= 32) __syncwarp();
    else if constexpr (T == THREADS) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / T), "n"(T) : "memory");
}

// stage of radix R on sub-transforms of length R * STRIDE, each inside one first-stage chunk
template <class S, int R, int STRIDE, int SIGN>
__device__ __forceinline__ void pow2_middle(float2 *buf, const float2 *rows, int t) {
    constexpr int blocks = S::S0 / (R * STRIDE);
    static_assert(STRIDE % S::RL == 0, "the skipped elements lie at multiples of the stride");
#pragma unroll 1
    for (int w = t; w < S::L / R; w += S::T) {
        const int np = w % STRIDE, blk = w / STRIDE, k0 = blk / blocks;
        float2 *d = buf + k0 * S::CHUNK + S::at((blk % blocks) * (R * STRIDE) + np);
        TwiddleRows<R> tw;
        tw.load(rows, STRIDE, np);
        float re[R], im[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const float2 v = d[q * S::at(STRIDE)];
            re[q] = v.x; im[q] = v.y;
        }
        dft<R, SIGN>(re, im);
        tw.template apply<SIGN>(re, im);
#pragma unroll
        for (int q = 0; q < R; ++q) d[q * S::at(STRIDE)] = make_float2(re[q], im[q]);
    }
    group_sync<S::T, S::THREADS>();
}

// load(b, re, im): operands b + q S0 of a first-stage butterfly; pre(w): whatever the store needs from global memory;
// store(w, re, im, pre): results w + q NL
template <class S, int SIGN, class Load, class Pre, class Store>
__device__ __forceinline__ void pow2_fft(float2 *buf, const float2 *rows, int t, Load load, Pre pre, Store store) {
    constexpr int R0 = S::R0, RL = S::RL;
#pragma unroll 1
    for (int b = t; b < S::S0; b += S::T) {
        float re[R0], im[R0];
        TwiddleRows<R0> tw;
        tw.load(rows, S::S0, b);
        load(b, re, im);
        dft<R0, SIGN>(re, im);
        tw.template apply<SIGN>(re, im);
        float2 *d = buf + S::at(b);
#pragma unroll
        for (int q = 0; q < R0; ++q) d[q * S::CHUNK] = make_float2(re[q], im[q]);
    }
    group_sync<S::T, S::THREADS>();
    if constexpr (S::R2 > 1) pow2_middle<S, S::R1, S::S1, SIGN>(buf, rows + S::TW1, t);
    if constexpr (S::R3 > 1) pow2_middle<S, S::R2, S::S2, SIGN>(buf, rows + S::TW2, t);
#pragma unroll 1
    for (int w = t; w < S::NL; w += S::T) {
        // w = k0 + R0 (k1 + R1 k2), position ((k0 R1 + k1) R2 + k2) RL
        int in = 0;
        if constexpr (S::R3 > 1) in = ((w / R0) % S::R1) * (S::R2 * RL) + (w / (R0 * S::R1)) * RL;
        else if constexpr (S::R2 > 1) in = (w / R0) * RL;
        const float2 *d = buf + (w % R0) * S::CHUNK + S::at(in);
        const auto fetched = pre(w);
        float re[RL], im[RL];
#pragma unroll
        for (int q = 0; q < RL; ++q) {
            const float2 v = d[q];
            re[q] = v.x; im[q] = v.y;
        }
        dft<RL, SIGN>(re, im);
        store(w, re, im, fetched);
    }
}

extern __shared__ float2 smem_pow2[];

struct Pow2Segment {
    int cta0, n_cta, first_band, n_bands;
};
struct Pow2Args {
    BandArgs b;
    const Pow2Rec *recs;
    Pow2Segment seg[kPow2Lengths];   // by length, longest first; the launch's own lengths only
};

template <bool ANALYSIS, class S>
__device__ __forceinline__ void pow2_cta(const Pow2Args &a, const Pow2Segment &sg) {
    const int g = (int)threadIdx.x / S::T, t = (int)threadIdx.x % S::T;
    const int last = sg.n_bands * a.b.batch - 1, idx = ((int)blockIdx.x - sg.cta0) * S::PER_CTA + g;
    const bool active = idx <= last;          // idle groups repeat the last item and store nothing
    const int item = active ? idx : last, band = item / a.b.batch, ch = item - band * a.b.batch;
    const Pow2Rec *rec = a.recs + sg.first_band + band;
    const BandRec br = rec->br;
    const float2 *rows = a.b.tw + rec->tw_off;
    float2 *buf = smem_pow2 + g * S::BUF;
    const float *tab = a.b.table + br.tab_off;
    constexpr int M = S::L;
    chain_begin(a.b);   // the record belongs to the plan; what follows touches the predecessor's output
    float2 *c = a.b.coef + coef_row(a.b.row0, a.b.rows, ch) * a.b.coeff_count + br.coeff_off;
    const int last_pos = br.d0 + br.S - 1, first_neg = M + br.d0;
    // support entry of slot m, -1: none
    auto entry = [&](int m) { return m <= last_pos ? m - br.d0 : (m >= first_neg ? m - first_neg : -1); };
    if constexpr (ANALYSIS) {
        const float2 *X = a.b.spec + (long long)ch * a.b.spec_pitch;
        auto load = [&](int b, float (&re)[S::R0], float (&im)[S::R0]) {
            if (br.side == 0) {
                // all loads are issued before the first product
                const float2 *Xs = X + (br.kc + br.d0);
#pragma unroll
                for (int q = 0; q < S::R0; ++q) {
                    const int j = entry(b + q * S::S0);
                    const float2 v = j >= 0 && CQT_CHK(a.b.dbg, 701, j, br.S) ? ld_chained(Xs + j) : make_float2(0.f, 0.f);
                    re[q] = v.x; im[q] = v.y;
                }
#pragma unroll
                for (int q = 0; q < S::R0; ++q) {
                    const int j = entry(b + q * S::S0);
                    const float h = j >= 0 ? __ldg(tab + j) : 0.f;
                    re[q] *= h; im[q] *= h;
                }
            } else {
#pragma unroll
                for (int q = 0; q < S::R0; ++q) {
                    const float2 v = slot_value<true>(br, tab, X, a.b.N, b + q * S::S0, a.b.dbg);
                    re[q] = v.x; im[q] = v.y;
                }
            }
        };
        // coefficients are written once and not read again by this call: streaming stores keep the L2 for the spectrum
        auto store = [&](int w, float (&re)[S::RL], float (&im)[S::RL], int) {
            if (!active) return;
#pragma unroll
            for (int q = 0; q < S::RL; ++q) __stcs(c + w + q * S::NL, make_float2(re[q], im[q]));
        };
        pow2_fft<S, +1>(buf, rows, t, load, [](int) { return 0; }, store);
    } else {
        const bool fold = a.b.fold && br.side != 0;
        auto load = [&](int b, float (&re)[S::R0], float (&im)[S::R0]) {
#pragma unroll
            for (int q = 0; q < S::R0; ++q) {
                const float2 v = ld_chained(c + b + q * S::S0);   // read once
                re[q] = v.x; im[q] = v.y;
            }
            if (fold) {
#pragma unroll
                for (int q = 0; q < S::R0; ++q) { re[q] *= 2.f; im[q] = 0.f; }
            }
        };
        // support entries outside bins 0..N/2 (sidebands) are dropped
        const int k0 = br.kc + br.d0, lo = max(0, -k0), hi = min(br.S, (a.b.N >> 1) + 1 - k0);
        float2 *Ys = a.b.Y + (long long)ch * a.b.y_pitch + br.y_off + k0;
        struct Window { float h[S::RL]; };
        auto pre = [&](int w) {
            Window f;
#pragma unroll
            for (int q = 0; q < S::RL; ++q) {
                const int j = entry(w + q * S::NL);
                f.h[q] = j >= 0 ? __ldg(tab + j) : 0.f;
            }
            return f;
        };
        auto store = [&](int w, float (&re)[S::RL], float (&im)[S::RL], const Window &f) {
            if (!active) return;
#pragma unroll
            for (int q = 0; q < S::RL; ++q) {
                const int j = entry(w + q * S::NL);
                if (j >= lo && j < hi && CQT_CHK(a.b.dbg, 702, (long long)br.y_off + k0 + j, a.b.y_pitch)) Ys[j] = make_float2(f.h[q] * re[q], f.h[q] * im[q]);
            }
        };
        pow2_fft<S, -1>(buf, rows, t, load, pre, store);
    }
}

template <bool ANALYSIS, bool LONG>
__global__ void __launch_bounds__(LONG ? 512 : 256, LONG ? 2 : 4) pow2_bands_kernel(Pow2Args a) {
    chain_enter(a.b);
    int i = 0;
#define X(S)                                                                                                                        \
    if ((int)blockIdx.x >= a.seg[i].cta0 && (int)blockIdx.x < a.seg[i].cta0 + a.seg[i].n_cta) pow2_cta<ANALYSIS, S>(a, a.seg[i]);  \
    ++i;
    if constexpr (LONG) { CQT_POW2_LONG(X) }
    else { CQT_POW2_SHORT(X) }
#undef X
    chain_end(a.b);
}

// ---------------------------------------------------------------- host side
int pow2_length_index(int64_t M) {
    int i = 0;
#define X(S) if (M == S::L) return i; ++i;
    CQT_POW2_LONG(X) CQT_POW2_SHORT(X)
#undef X
    return -1;
}

void pow2_radices(int index, int (&r)[5]) {
    int i = 0;
#define X(S) if (i++ == index) { r[0] = S::R0; r[1] = S::R1; r[2] = S::R2; r[3] = S::R3; r[4] = 1; }
    CQT_POW2_LONG(X) CQT_POW2_SHORT(X)
#undef X
}

struct Pow2Launch {
    Pow2Segment seg[kPow2Lengths] = {};
    int grid = 0;
    size_t smem = 0;
};

static Pow2Launch pow2_shape(const cqt_plan &p, int64_t batch, bool long_ones) {
    Pow2Launch l;
    int64_t grid = 0;
    int band = 0, all = 0, i = 0;
#define X(S)                                                                                        \
    {                                                                                               \
        const int n = p.pow2.n_bands[all++];                                                        \
        if ((S::THREADS == 512) == long_ones) {                                                     \
            const int64_t ctas = (n * batch + S::PER_CTA - 1) / S::PER_CTA;                         \
            l.seg[i++] = Pow2Segment{(int)grid, (int)ctas, band, n};                                \
            grid += ctas;                                                                           \
            if (n) l.smem = std::max(l.smem, sizeof(float2) * (size_t)(S::PER_CTA * S::BUF));       \
        }                                                                                           \
        band += n;                                                                                  \
    }
    CQT_POW2_LONG(X) CQT_POW2_SHORT(X)
#undef X
    l.grid = (int)grid;
    return l;
}

static const void *pow2_kernel(bool analysis, bool long_ones) {
    if (long_ones) return analysis ? (const void *)pow2_bands_kernel<true, true> : (const void *)pow2_bands_kernel<false, true>;
    return analysis ? (const void *)pow2_bands_kernel<true, false> : (const void *)pow2_bands_kernel<false, false>;
}

bool pow2_has(const cqt_plan &p, bool long_ones) { return pow2_shape(p, 1, long_ones).grid > 0; }

cudaError_t launch_pow2(const cqt_plan &p, bool analysis, bool long_ones, const BandArgs &b, cudaStream_t st) {
    const Pow2Launch l = pow2_shape(p, b.batch, long_ones);
    Pow2Args a{};
    a.b = b;
    a.recs = p.pow2.d_recs;
    std::copy(l.seg, l.seg + kPow2Lengths, a.seg);
    void *args[] = {&a};
    cudaError_t e = launch_kernel(pow2_kernel(analysis, long_ones), dim3((unsigned)l.grid), dim3(long_ones ? 512 : 256), args, l.smem, st);
    note_launch(p, analysis ? (long_ones ? "bands_from_spectrum/pow2_long" : "bands_from_spectrum/pow2")
                            : (long_ones ? "bands_to_spectrum/pow2_long" : "bands_to_spectrum/pow2"), st);
    return e;
}

cudaError_t configure_pow2_kernels(const cqt_plan &p) {
    if (p.pow2.recs.empty()) return cudaSuccess;
    for (bool long_ones : {false, true})
        for (bool analysis : {false, true}) {
            cudaError_t e = allow_dynamic_smem(pow2_kernel(analysis, long_ones), pow2_shape(p, 1, long_ones).smem, p);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

}  // namespace cqt
