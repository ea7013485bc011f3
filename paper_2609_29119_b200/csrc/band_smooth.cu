// Host side of the kernels of 5-smooth lengths (band_smooth.cuh).
#include <algorithm>

#include "band_smooth.cuh"

namespace cqt {

namespace {

const SmoothInfo kShapes[] = {   // longest first
#define X(M, R0, R1, R2, R3, R4, T, PER, THREADS, PAD, CHUNK, ...) {M, PER, R0 * CHUNK, {R0, R1, R2, R3, R4}},
    CQT_SHAPES_4(X) CQT_SHAPES_2(X) CQT_SHAPES_1(X) CQT_SHAPES_0(X)
#undef X
};

const void *kernel_of(bool analysis, int cls, bool chained) {
#define X(C, A, H) if (cls == C && analysis == A && chained == H) return SmoothKernel<A, C, H>::get();
    CQT_SMOOTH_KERNELS(X)
#undef X
    return nullptr;
}

}  // namespace

const SmoothInfo *smooth_info(int64_t M) {
    const SmoothInfo *end = kShapes + sizeof(kShapes) / sizeof(kShapes[0]);
    const SmoothInfo *s = std::lower_bound(kShapes, end, M, [](const SmoothInfo &a, int64_t m) { return a.M > m; });
    return s != end && s->M == M ? s : nullptr;
}

// names of the launches: the class's, as in the other kernels of the class, and this kernel's mark
const char *const kNames[2][kNumClasses] = {
    {"bands_to_spectrum/class0/smooth", "bands_to_spectrum/class1/smooth", "bands_to_spectrum/class2/smooth", "bands_to_spectrum/class3/smooth", "bands_to_spectrum/class4/smooth"},
    {"bands_from_spectrum/class0/smooth", "bands_from_spectrum/class1/smooth", "bands_from_spectrum/class2/smooth", "bands_from_spectrum/class3/smooth", "bands_from_spectrum/class4/smooth"}};

bool has_smooth(const cqt_plan &p, bool analysis, int cls) { return !p.smooth[cls].recs.empty() && kernel_of(analysis, cls, false); }

// A CTA takes `repeat` units of one length one after another: the code of the length is fetched once for them, and warps that
// are done with one are on with the loads of the next.  More of them leave fewer CTAs to even out the end of the launch.
// Two from 1.5 rounds of the resident CTAs on and four from 8, but two only from 3 rounds (class 0) or 2 (the others) where the class has at
// least half of the coefficients: nothing beside it then fills the SMs that its last round leaves idle.  Whole transform with one / two:
//   class 0, 56 % or more: 1.9 rounds 36.3 / 41.8 us, 2.5 47.9 / 51.3, 4 65.8 / 63.6 (2^13 samples, 24 bands per octave, synthesis); 2.5 26.9 / 28.7,
//   3 29.0 / 29.1, 4 33.0 / 31.7 (2^14, 96); round trips: 1.2 43.6 / 57.7, 2.5 50.3 / 60.5 (2^13, 48), the other way 2.5 78.4 / 76.2 (2^12, 12)
//   class 0, 28 %: 1.75 40.6 / 40.9, 2 43.4 / 43.0 (2^15, 48, analysis); 14 %: 1.8 81.9 / 79.8 (2^15, 24)
//   class 1, 82 %: 1.75 44.9 / 49.7, 2 48.8 / 52.3, 2.5 59.4 / 58.0 (2^15, 24); 47 %: 1.5 72.2 / 70.7, 2 89.7 / 87.3 (2^17, 48)
//   class 2, 46 %: 1.5 58.0 / 58.9, 2 76.7 / 73.6 (2^17, 48); 40 %: 1.25 72.3 / 70.9, 2 109.2 / 105.0 (2^18, 24)
// and with two / four: class 0 at 8 rounds 174 / 169 (2^15, 48), class 1 at 6 126 / 122.
cudaError_t launch_smooth(const cqt_plan &p, bool analysis, int cls, const BandArgs &b, cudaStream_t st, int threads) {
    if (threads == 0) threads = smooth_threads(cls);
    const SmoothBands &s = p.smooth[cls];
    SmoothArgs a;
    a.b = b;
    a.recs = s.d_recs;
    a.n = (int)s.lengths.size();
    const int part = smooth_threads(cls) / threads;   // narrower CTAs have so much fewer items and shared memory
    const size_t smem = s.smem / part;
    const int64_t resident = p.sm_count * std::min<int64_t>(1024 / threads, (p.max_smem_optin + 1024) / ((int64_t)smem + 1024));
    int64_t units = 0;
    for (const SmoothBands::Length &l : s.lengths) units += ((int64_t)l.n_bands * b.batch + l.per / part - 1) / (l.per / part);
    int64_t coefficients = 0;
    for (const SmoothBands::Length &l : s.lengths) coefficients += (int64_t)l.M * l.n_bands;
    const int64_t halves = 2 * coefficients < p.lay.coeff_count ? 3 : (cls == 0 ? 6 : 4);   // half rounds
    a.repeat = 2 * units < halves * resident ? 1 : (units < 8 * resident ? 2 : 4);
    int64_t grid = 0;
    for (int i = 0; i < a.n; ++i) {
        const SmoothBands::Length &l = s.lengths[(size_t)i];
        const int64_t per_cta = (int64_t)(l.per / part) * a.repeat;
        a.seg[i] = SmoothSegment{(int)grid, l.first_band, l.n_bands, l.M};
        grid += ((int64_t)l.n_bands * b.batch + per_cta - 1) / per_cta;
    }
    void *args[] = {&a};
    const void *fn = kernel_of(analysis, cls, b.chain == kChainMember);   // the head of a chain waits for itself
    if (!fn) return cudaErrorInvalidDeviceFunction;
    cudaError_t e = launch_kernel(fn, dim3((unsigned)grid), dim3((unsigned)threads), args, smem, st);
    note_launch(p, kNames[analysis][cls], st);
    return e;
}

cudaError_t configure_smooth_kernels(const cqt_plan &p) {
    for (int c = 0; c < kNumClasses; ++c)
        for (bool analysis : {false, true}) {
            if (!has_smooth(p, analysis, c)) continue;
            for (bool chained : {false, true}) {
                const void *fn = kernel_of(analysis, c, chained);
                if (!fn) continue;
                cudaError_t e = allow_dynamic_smem(fn, p.smooth[c].smem, p);
                if (e != cudaSuccess) return e;
            }
        }
    return cudaSuccess;
}

}  // namespace cqt
