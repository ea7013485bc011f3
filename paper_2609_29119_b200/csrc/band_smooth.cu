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
// are done with one are on with the loads of the next.  More of them leave fewer CTAs to even out the end of the launch:
// twice where the launch is at least 1.5 rounds of the resident CTAs, four times from 8 rounds on.
cudaError_t launch_smooth(const cqt_plan &p, bool analysis, int cls, const BandArgs &b, cudaStream_t st, int threads) {
    if (threads == 0) threads = kSmoothThreads[cls];
    const SmoothBands &s = p.smooth[cls];
    SmoothArgs a;
    a.b = b;
    a.recs = s.d_recs;
    a.n = (int)s.lengths.size();
    const int part = kSmoothThreads[cls] / threads;   // narrower CTAs have so much fewer items and shared memory
    const size_t smem = s.smem / part;
    const int64_t resident = p.sm_count * std::min<int64_t>(1024 / threads, (p.max_smem_optin + 1024) / ((int64_t)smem + 1024));
    int64_t units = 0;
    for (const SmoothBands::Length &l : s.lengths) units += ((int64_t)l.n_bands * b.batch + l.per / part - 1) / (l.per / part);
    a.repeat = 2 * units < 3 * resident ? 1 : (units < 8 * resident ? 2 : 4);
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
