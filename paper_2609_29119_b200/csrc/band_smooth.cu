// Host side of the kernels of 5-smooth lengths (band_smooth.cuh).
#include <algorithm>

#include "band_smooth.cuh"

namespace cqt {

namespace {

struct ShapeInfo {
    int M, per, buf, r[5];
};
const ShapeInfo kShapes[] = {   // longest first
#define X(M, R0, R1, R2, R3, R4, T, PER, THREADS, PAD, CHUNK, ...) {M, PER, R0 * CHUNK, {R0, R1, R2, R3, R4}},
    CQT_SHAPES_4(X) CQT_SHAPES_2(X) CQT_SHAPES_1(X) CQT_SHAPES_0(X)
#undef X
};

const ShapeInfo *shape_of(int64_t M) {
    const ShapeInfo *end = kShapes + sizeof(kShapes) / sizeof(kShapes[0]);
    const ShapeInfo *s = std::lower_bound(kShapes, end, M, [](const ShapeInfo &a, int64_t m) { return a.M > m; });
    return s != end && s->M == M ? s : nullptr;
}

const void *kernel_of(bool analysis, int cls) {
#define X(C, A) if (cls == C && analysis == A) return SmoothKernel<A, C>::get();
    CQT_SMOOTH_KERNELS(X)
#undef X
    return nullptr;
}

// Items of a unit: fewer in narrower CTAs of class 0
int items_per_unit(const ShapeInfo &s, int cls, int threads) { return s.per * threads / kSmoothThreads[cls]; }

size_t smem_of(const SmoothBands &s, int cls, int threads) {
    size_t most = 0;
    for (const SmoothBands::Length &l : s.lengths) {
        const ShapeInfo &sh = *shape_of(l.M);
        most = std::max(most, sizeof(float2) * (size_t)(items_per_unit(sh, cls, threads) * sh.buf));
    }
    return most;
}

}  // namespace

bool smooth_radices(int64_t M, int (&r)[5]) {
    const ShapeInfo *s = shape_of(M);
    if (s) std::copy(s->r, s->r + 5, r);
    return s != nullptr;
}

bool has_smooth(const cqt_plan &p, bool analysis, int cls) { return !p.smooth[cls].recs.empty() && kernel_of(analysis, cls); }

// A CTA takes `repeat` units of one length one after another: the code of the length is fetched once for them, and warps that
// are done with one are on with the loads of the next.  More of them leave fewer CTAs to even out the end of the launch:
// twice where the launch is at least 1.5 rounds of the resident CTAs, four times from 8 rounds on.
cudaError_t launch_smooth(const cqt_plan &p, bool analysis, int cls, const char *name, const BandArgs &b, cudaStream_t st, int threads) {
    if (threads == 0) threads = kSmoothThreads[cls];
    const SmoothBands &s = p.smooth[cls];
    SmoothArgs a{};
    a.b = b;
    a.recs = s.d_recs;
    const size_t smem = smem_of(s, cls, threads);
    const int64_t resident = p.sm_count * std::min<int64_t>(1024 / threads, (p.max_smem_optin + 1024) / ((int64_t)smem + 1024));
    int64_t units = 0;
    for (const SmoothBands::Length &l : s.lengths) {
        const int per = items_per_unit(*shape_of(l.M), cls, threads);
        units += ((int64_t)l.n_bands * b.batch + per - 1) / per;
    }
    a.repeat = 2 * units < 3 * resident ? 1 : (units < 8 * resident ? 2 : 4);
    int64_t grid = 0;
    for (const SmoothBands::Length &l : s.lengths) {
        const int64_t per_cta = (int64_t)items_per_unit(*shape_of(l.M), cls, threads) * a.repeat;
        a.seg[a.n++] = SmoothSegment{(int)grid, l.first_band, l.n_bands, l.M};
        grid += ((int64_t)l.n_bands * b.batch + per_cta - 1) / per_cta;
    }
    void *args[] = {&a};
    cudaError_t e = launch_kernel(kernel_of(analysis, cls), dim3((unsigned)grid), dim3((unsigned)threads), args, smem, st);
    note_launch(p, name, st);
    return e;
}

cudaError_t configure_smooth_kernels(const cqt_plan &p) {
    for (int c = 0; c < kNumClasses; ++c)
        for (bool analysis : {false, true}) {
            if (!has_smooth(p, analysis, c)) continue;
            cudaError_t e = allow_dynamic_smem(kernel_of(analysis, c), smem_of(p.smooth[c], c, kSmoothThreads[c]), p);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

}  // namespace cqt
