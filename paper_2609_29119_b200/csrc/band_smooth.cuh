// Bands whose length has no prime factor above 5, every length a transform of its own: radices, strides, threads and the layout
// of the buffer are known at compile time (band_shapes.cuh, chosen by choose_shapes.py).
//
// Bounds: instructions, their fetch included.  Thread instructions per coefficient, on the run-time planned kernels and here: analysis
// of class 1 151 and 106, of class 2 153 and 114 (3.2 and 3.9 stages on average), of class 4 143 and 119, its synthesis 141 and 125 (16
// signals of 2^19 samples); a band of at most 128 coefficients takes two stages instead of up to three.  The code of one length (4 - 20 KB)
// does not stay in an SM's instruction cache from one length to the next: a CTA's first pass over it waits for the cache that
// the SMs of a GPC share (first stage of a 960-coefficient item 13,000 cycles, the same stage again 4,900).  Hence the order of
// the grid, equal lengths adjacent, so that all SMs fetch the same code at about the same time (persistent CTAs that each walk a
// length of their own: 51 us where this order takes 37), and several units per CTA where a call has many (launch_smooth).
// All kernels have 64 registers per thread, so that 1024 threads share an SM, and most lengths spill (bytes of spill stores per thread,
// the lengths that do, the most): analysis of class 0 11 of 19, 52; class 1 30 of 33, 32; class 2 33 of 35, 176; class 4 31 of 31, 184;
// synthesis of class 0 9 of 19, 220; class 4 31 of 31, 392 (16,000 = 10 10 10 16, whose last butterflies hold 16 values and 16 window entries).
#pragma once
#include "band_common.cuh"
#include "band_shapes.cuh"
#include "twiddle_rows.cuh"

namespace cqt {

template <int M_, int R0_, int R1_, int R2_, int R3_, int R4_, int T_, int PER_, int THREADS_, int PAD_, int CHUNK_, int MAP1_, int MAP2_, int MAP3_>
struct SmoothShape {
    static constexpr int M = M_, R0 = R0_, R1 = R1_, R2 = R2_, R3 = R3_, R4 = R4_, T = T_, PER = PER_, THREADS = THREADS_, CHUNK = CHUNK_;
    static constexpr int MAP1 = MAP1_, MAP2 = MAP2_, MAP3 = MAP3_;
    static constexpr int S0 = M / R0, S1 = S0 / R1, S2 = S1 / R2, S3 = S2 / R3;
    static constexpr int STAGES = R4 > 1 ? 5 : (R3 > 1 ? 4 : (R2 > 1 ? 3 : 2));
    static constexpr int RL = STAGES == 5 ? R4 : (STAGES == 4 ? R3 : (STAGES == 3 ? R2 : R1)), NL = M / RL;
    // one element skipped per PAD positions of a first-stage chunk
    static __host__ __device__ constexpr int at(int p) { return PAD_ ? p + p / (PAD_ ? PAD_ : 1) : p; }
    static constexpr int BUF = R0 * CHUNK;
    // barrier of the T threads of an item: a warp's, the CTA's, or a named one (1 ... PER)
    static constexpr bool WARP_SYNC = T <= 32, CTA_SYNC = !WARP_SYNC && PER == 1;
    // twiddle rows of the stages before the last, one after another
    static constexpr int TW1 = twiddle_rows(R0) * S0, TW2 = TW1 + twiddle_rows(R1) * S1, TW3 = TW2 + twiddle_rows(R2) * S2;
    static_assert(R0 * R1 * R2 * R3 * R4 == M && at(S0 - 1) < CHUNK, "shape");
    static_assert(T * PER == THREADS && (WARP_SYNC ? 32 % T == 0 : T % 32 == 0 && PER < 16), "every thread of a barrier belongs to the item");
    static_assert(PAD_ == 0 || PAD_ == RL, "the skipped elements lie at multiples of every stride");
};

template <class S>
__device__ __forceinline__ void smooth_sync() {
    if constexpr (S::WARP_SYNC) __syncwarp();
    else if constexpr (S::CTA_SYNC) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / S::T), "n"(S::T) : "memory");
}

// Stage of radix R on sub-transforms of length R * STRIDE, each inside one first-stage chunk.  Starts with the barrier that
// ends the stage before; the first round's twiddles are fetched ahead of it.
template <class S, int R, int STRIDE, int MAP, int SIGN>
__device__ __forceinline__ void smooth_middle(float2 *buf, const float2 *rows, int t, int *dbg) {
    constexpr int blocks = S::S0 / (R * STRIDE), units = S::M / R;
    auto place = [](int w, int &np) {
        if constexpr (MAP) {   // short strides: neighbouring threads on neighbouring chunks, which lie in different banks
            const int x = w / S::R0;
            np = x % STRIDE;
            return (w % S::R0) * S::CHUNK + S::at((x / STRIDE) * (R * STRIDE) + np);
        } else {
            const int x = w / STRIDE;
            np = w % STRIDE;
            return (x / blocks) * S::CHUNK + S::at((x % blocks) * (R * STRIDE) + np);
        }
    };
    int w = t, np = 0, at = 0;
    TwiddleRows<R> tw;
    if (w < units) {
        at = place(w, np);
        tw.load(rows, STRIDE, np);
    }
    smooth_sync<S>();
    while (w < units) {
        float2 *d = buf + at;
        float re[R], im[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const float2 v = CQT_CHK(dbg, 808, at + q * S::at(STRIDE), S::BUF) ? d[q * S::at(STRIDE)] : make_float2(0.f, 0.f);
            re[q] = v.x; im[q] = v.y;
        }
        dft<R, SIGN>(re, im);
        tw.template apply<SIGN>(re, im);
#pragma unroll
        for (int q = 0; q < R; ++q)
            if (CQT_CHK(dbg, 808, at + q * S::at(STRIDE), S::BUF)) d[q * S::at(STRIDE)] = make_float2(re[q], im[q]);
        w += S::T;
        if (w < units) {
            at = place(w, np);
            tw.load(rows, STRIDE, np);
        }
    }
}

// load(b, re, im): operands b + q S0 of a first-stage butterfly; pre(w): whatever the store needs from global memory;
// store(w, re, im, pre): results w + q NL.  again: the buffer holds the item before, whose last stage some threads may still read;
// the others are on with this item's loads and first butterflies meanwhile.
template <class S, int SIGN, class Load, class Pre, class Store>
__device__ __forceinline__ void smooth_fft(float2 *buf, const float2 *rows, int t, bool again, int *dbg, Load load, Pre pre, Store store) {
    constexpr int R0 = S::R0, RL = S::RL;
    constexpr int rounds = (S::S0 + S::T - 1) / S::T;
#pragma unroll 1
    for (int r = 0; r < rounds; ++r) {
        const int b = t + r * S::T;
        float re[R0], im[R0];
        if (b < S::S0) {
            TwiddleRows<R0> tw;
            tw.load(rows, S::S0, b);
            load(b, re, im);
            dft<R0, SIGN>(re, im);
            tw.template apply<SIGN>(re, im);
        }
        if (again && r == 0) smooth_sync<S>();
        if (b < S::S0) {
            float2 *d = buf + S::at(b);
#pragma unroll
            for (int q = 0; q < R0; ++q)
                if (CQT_CHK(dbg, 807, S::at(b) + q * S::CHUNK, S::BUF)) d[q * S::CHUNK] = make_float2(re[q], im[q]);
        }
    }
    if constexpr (S::STAGES > 2) smooth_middle<S, S::R1, S::S1, S::MAP1, SIGN>(buf, rows + S::TW1, t, dbg);
    if constexpr (S::STAGES > 3) smooth_middle<S, S::R2, S::S2, S::MAP2, SIGN>(buf, rows + S::TW2, t, dbg);
    if constexpr (S::STAGES > 4) smooth_middle<S, S::R3, S::S3, S::MAP3, SIGN>(buf, rows + S::TW3, t, dbg);
    int w = t;
    decltype(pre(0)) fetched{};
    if (w < S::NL) fetched = pre(w);
    smooth_sync<S>();
#pragma unroll 1
    while (w < S::NL) {
        // w = k0 + R0 (k1 + R1 (k2 + ...)), at position k1 S1 + k2 S2 + ... of chunk k0
        int in = 0;
        if constexpr (S::STAGES == 3) in = (w / R0) * S::S1;
        if constexpr (S::STAGES == 4) in = ((w / R0) % S::R1) * S::S1 + (w / (R0 * S::R1)) * S::S2;
        if constexpr (S::STAGES == 5) in = ((w / R0) % S::R1) * S::S1 + ((w / (R0 * S::R1)) % S::R2) * S::S2 + (w / (R0 * S::R1 * S::R2)) * S::S3;
        const int at = (w % R0) * S::CHUNK + S::at(in);
        const float2 *d = buf + at;
        float re[RL], im[RL];
#pragma unroll
        for (int q = 0; q < RL; ++q) {
            const float2 v = CQT_CHK(dbg, 809, at + q, S::BUF) ? d[q] : make_float2(0.f, 0.f);
            re[q] = v.x; im[q] = v.y;
        }
        dft<RL, SIGN>(re, im);
        store(w, re, im, fetched);
        w += S::T;
        if (w < S::NL) fetched = pre(w);
    }
}

constexpr int smooth_threads(int cls) { return cls == 4 ? 1024 : 256; }   // of a CTA; 1024 threads of 64 registers share an SM

// Bands of one length, from CTA cta0 of the launch on.  A unit is PER work items of them, one per group of T threads; a CTA takes
// `repeat` units one after another.
struct SmoothSegment {
    int cta0, first_band, n_bands, shape;
};
struct SmoothArgs {
    BandArgs b;
    const SmoothRec *recs;
    int repeat;
    int n;                                 // segments
    SmoothSegment seg[kSmoothLengths];
};

extern __shared__ float2 smem_smooth[];

// CHAINED: the launch may be a member of a chain (band_common.cuh); only class 0 is ever in one.
template <bool ANALYSIS, bool CHAINED, class S>
__device__ __noinline__ void smooth_units(const SmoothArgs &a, int seg) {
    const SmoothSegment sg = a.seg[seg];
    const int per = S::M <= 128 ? (int)blockDim.x / S::T : S::PER;   // class 0 also runs in narrower CTAs
    const int g = S::PER > 1 ? (int)threadIdx.x / S::T : 0;
    const int t = (int)threadIdx.x - g * S::T;
    const int batch = a.b.batch, last = sg.n_bands * batch - 1;
    const int u0 = ((int)blockIdx.x - sg.cta0) * a.repeat, u1 = min(u0 + a.repeat, last / per + 1);
    const SmoothRec *recs = a.recs + sg.first_band;
    const float2 *rows = a.b.tw + recs->tw_off;
    float2 *buf = smem_smooth + g * S::BUF;
    constexpr int M = S::M;
#pragma unroll 1
    for (int u = u0; u < u1; ++u) {
        const int idx = u * per + g;
        const bool active = idx <= last;   // groups beyond the last item repeat it and store nothing
        const int item = active ? idx : last, band = item / batch, ch = item - band * batch;
        const BandRec br = recs[band].br;
        const float *tab = a.b.table + br.tab_off;
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
                        const bool in = j >= 0 && CQT_CHK(a.b.dbg, 801, j, br.S) && CQT_CHK(a.b.dbg, 802, br.kc + br.d0 + j, (a.b.N >> 1) + 1);
                        const float2 v = in ? ld_spectrum<CHAINED>(Xs + j) : make_float2(0.f, 0.f);
                        re[q] = v.x; im[q] = v.y;
                    }
#pragma unroll
                    for (int q = 0; q < S::R0; ++q) {
                        const int j = entry(b + q * S::S0);
                        const float h = j >= 0 && CQT_CHK(a.b.dbg, 803, br.tab_off + j, a.b.table_len) ? __ldg(tab + j) : 0.f;
                        re[q] *= h; im[q] *= h;
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < S::R0; ++q) {
                        const float2 v = slot_value<CHAINED>(br, tab, X, a.b.N, b + q * S::S0, a.b.dbg);
                        re[q] = v.x; im[q] = v.y;
                    }
                }
            };
            // coefficients are written once and not read again by this call: streaming stores keep the L2 for the spectrum
            auto store = [&](int w, float (&re)[S::RL], float (&im)[S::RL], int) {
                if (!active) return;
#pragma unroll
                for (int q = 0; q < S::RL; ++q)
                    if (CQT_CHK(a.b.dbg, 804, w + q * S::NL, M)) __stcs(c + w + q * S::NL, make_float2(re[q], im[q]));
            };
            smooth_fft<S, +1>(buf, rows, t, u > u0, a.b.dbg, load, [](int) { return 0; }, store);
        } else {
            const bool fold = a.b.fold && br.side != 0;
            auto load = [&](int b, float (&re)[S::R0], float (&im)[S::R0]) {
#pragma unroll
                for (int q = 0; q < S::R0; ++q) {
                    const float2 v = CQT_CHK(a.b.dbg, 805, b + q * S::S0, M) ? ld_coefficient<CHAINED>(c + b + q * S::S0) : make_float2(0.f, 0.f);   // read once
                    re[q] = v.x; im[q] = v.y;
                }
                if (fold) {
#pragma unroll
                    for (int q = 0; q < S::R0; ++q) { re[q] *= 2.f; im[q] = 0.f; }
                }
            };
            // support entries outside bins 0..N/2 (sidebands) are dropped
            const int k0 = br.kc + br.d0, last_in = min(last_pos, (a.b.N >> 1) - br.kc), first_in = first_neg + max(0, -k0);
            auto kept = [&](int m) { return m <= last_in ? m - br.d0 : (m >= first_in ? m - first_neg : -1); };
            float2 *Ys = a.b.Y + (long long)ch * a.b.y_pitch + br.y_off + k0;
            struct Window { float h[S::RL]; };
            auto pre = [&](int w) {
                Window f;
#pragma unroll
                for (int q = 0; q < S::RL; ++q) {
                    const int j = kept(w + q * S::NL);
                    f.h[q] = j >= 0 && CQT_CHK(a.b.dbg, 803, br.tab_off + j, a.b.table_len) ? __ldg(tab + j) : 0.f;
                }
                return f;
            };
            auto store = [&](int w, float (&re)[S::RL], float (&im)[S::RL], const Window &f) {
                if (!active) return;
#pragma unroll
                for (int q = 0; q < S::RL; ++q) {
                    const int j = kept(w + q * S::NL);
                    if (j >= 0 && CQT_CHK(a.b.dbg, 806, (long long)br.y_off + k0 + j, a.b.y_pitch)) Ys[j] = make_float2(f.h[q] * re[q], f.h[q] * im[q]);
                }
            };
            smooth_fft<S, -1>(buf, rows, t, u > u0, a.b.dbg, load, pre, store);
        }
    }
}

// segment of this CTA
__device__ __forceinline__ int smooth_segment(const SmoothArgs &a) {
    int lo = 0, hi = a.n;   // cta0[lo] <= blockIdx.x < cta0[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if ((int)blockIdx.x >= a.seg[mid].cta0) lo = mid; else hi = mid;
    }
    return lo;
}

// One kernel per class, direction and kind of launch, each compiled by itself (band_smooth_kernel.cu; the list is that of build.py)
template <bool ANALYSIS, int CLASS, bool CHAINED>
struct SmoothKernel {
    static const void *get();
};
#define CQT_SMOOTH_KERNELS(X) \
    X(0, false, false) X(0, false, true) X(0, true, false) X(0, true, true) X(1, true, false) X(2, true, false) X(4, false, false) X(4, true, false)

}  // namespace cqt
