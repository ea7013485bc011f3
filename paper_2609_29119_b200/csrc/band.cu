// Host side of the fused band kernels: per-class launches on the caller's stream and the plan's helper streams.
#include <algorithm>

#include "band_common.cuh"

namespace cqt {

static BandArgs make_args(const cqt_plan &p, const BandClass &c, const float *table, int64_t batch) {
    BandArgs a{};
    a.items = c.d_items;
    a.tw = p.d.tw;
    a.table = table;
    a.n_work = c.n_bands;
    a.batch = (int)batch;
    a.N = (int)p.N;
    a.max_elems = c.max_elems;
    a.coeff_count = p.lay.coeff_count;
    a.y_pitch = p.y_pitch;
    a.table_len = p.lay.table_len;
    a.dbg = p.d.dbg;
    return a;
}

static void set_rows(BandArgs &a, const CoefRows &c) {
    a.coef = c.base;
    a.row0 = c.row0;
    a.rows = c.rows;
}

const void *band_analysis_kernel(const BandClass &c, int lanes, bool chained);    // band_analysis.cu
const void *band_synthesis_kernel(const BandClass &c, int lanes, bool chained);   // band_synthesis.cu

template <bool ANALYSIS>
static const void *class_kernel(const BandClass &c, int lanes, bool chained) {
    return ANALYSIS ? band_analysis_kernel(c, lanes, chained) : band_synthesis_kernel(c, lanes, chained);
}

// Lanes per work item of the class of the shortest bands (0: the class gives every item a whole CTA).  A band of at
// most 128 coefficients has at most 16 radix-8 butterflies per stage, so 8 lanes per item keep the lanes busy: fewer
// warps for the same work, which leaves the SMs to the long-band classes running beside it.  A whole warp per item
// has the shorter critical path, which is what counts in a call with few items (a single signal, one streaming hop).
static int lanes_for(const cqt_plan &p, const BandClass &c, long long items) {
    return items >= 8ll * p.sm_count ? c.lanes_many : c.lanes_few;
}

template <bool ANALYSIS>
static cudaError_t launch_class(const cqt_plan &p, int cls, const char *name, BandArgs &a, cudaStream_t st) {
    const BandClass &c = p.cls[cls];
    if (c.n_bands == 0) return cudaSuccess;
    const long long items = (long long)c.n_bands * a.batch;
    const int lanes = lanes_for(p, c, items);
    const int per_cta = lanes ? c.threads / lanes : 1;
    const size_t smem = (size_t)c.max_elems * per_cta * sizeof(float2);
    const long long grid = (items + per_cta - 1) / per_cta;
    void *args[] = {&a};
    const void *fn = class_kernel<ANALYSIS>(c, lanes, false);
    if (!fn) return cudaErrorInvalidDeviceFunction;
    cudaError_t e = launch_kernel(fn, dim3((unsigned)grid), dim3(c.threads), args, smem, st);
    note_launch(p, name, st);
    return e;
}

const void *band_analysis_merged_kernel();    // band_analysis.cu
const void *band_synthesis_merged_kernel();   // band_synthesis.cu

// Shape of the few-items form for a batch: the bands longer than class 0's in one launch, those of them that would take
// 1024 threads each (the first segment) split into four work items in another, class 0 in one.
struct FewLaunch {
    struct Part {
        BandSegments sg{};
        int threads = 0, grid = 0;
        size_t smem = 0;
    };
    Part part;
    bool split = false;                 // bands on the split kernel
    bool chirp = false;                 // bands on the chirp-z kernel
    int short_threads = 0, short_grid = 0;
    bool short_smooth = false;          // class 0 on the kernel of 5-smooth lengths
};

// CTAs of a launch that share an SM, at most `most` (what its launch bounds allow): its shared memory decides the rest.
static long long ctas_per_sm(const cqt_plan &p, size_t smem, int most) {
    return std::min<long long>(most, (p.max_smem_optin + 1024ll) / ((long long)smem + 1024));
}

// Segments [first, last) in CTAs filled to 1 / share; returns the SMs the launch occupies, and whether CTAs hold more
// than one item.
static long long few_part(const cqt_plan &p, int64_t batch, int first, int last, int share, FewLaunch::Part &t, bool &spread) {
    t = FewLaunch::Part{};
    if (first == last) return 0;
    const MergedBands &mg = p.merged;
    t.threads = std::max(128, 1 << mg.segs[first].lg_nthr);
    t.sg.n = last - first;
    long long grid = 0;
    for (int i = first; i < last; ++i) {
        const MergedBands::Segment &s = mg.segs[i];
        const int full = std::min(t.threads >> s.lg_nthr, kMaxGroups), per = std::max(1, full / share);
        spread = spread || per > 1;
        t.sg.s[i - first] = BandSegment{(int)grid, s.first_band, s.n_bands, s.lg_nthr, per, s.elems};
        t.smem = std::max(t.smem, (size_t)per * s.elems * sizeof(float2));
        grid += ((long long)s.n_bands * batch + per - 1) / per;
        if (grid > (1 << 20)) return grid;
    }
    t.grid = (int)grid;
    const long long per_sm = ctas_per_sm(p, t.smem + kMaxGroups * sizeof(BandItem), 1024 / t.threads);
    return per_sm > 0 ? (grid + per_sm - 1) / per_sm : 1 << 20;
}

// The few-items form is taken where every CTA of the longer bands is resident at once.  A call that small is a chain of
// latencies, and side by side on streams each class adds a launch, an event and two cross-stream waits to it (round trips
// at 48 bands per octave: 4 signals of 2^13 samples 35.8 us in this form, 43.5 in the other; 398 bands of 80 bins, 4
// signals of 2^15: 37.8 and 45.3).
//
// The short class is chained behind them on a warp per item, up to 16 items per SM.  Above, neither form is the faster one
// for every plan: at 17 - 22 items per SM the chained form took 39 us where the classes took 41 (8 signals of 2^13 samples
// at 48 bands per octave) and 42 where they took 49 (398 bands of 80 bins), but 49 where they took 41 (8 signals of 2^15
// samples at 48 bands per octave); from 80 items per SM on the classes' 8 lanes per item win (63 against 77 us at 129).
//
// Up to 4 items per SM its CTAs have 64 threads, so that they lie on all SMs, above that 256.  Where the class holds direct
// sums, whose items take long, that pays (multiple-of-4 lengths, 2 signals of 2^16: 52.5 us, with 256 threads 55.8); for
// 5-smooth lengths it is within the spread of runs or a little slower (2^13 samples, 24 bands per octave, 4 signals: 38.7
// us, with 256 threads 37.2).
//
// 5-smooth lengths run on their own kernel, 8 lanes per item, up to 6 items per SM, unless bands are split (above 6144
// coefficients).  Round trips of 1 - 12 signals in 16 layouts, a warp per item on the run-time planned kernel against this one: without
// split bands 3.7 % less on average up to 4 items per SM (4 signals of 2^13 samples at 24 bands per octave 39.9 -> 34.0 us, one of 2^16
// at 24 42.6 -> 41.1, one of 2^18 at 96 50.2 -> 47.0; four of 40 calls 2 - 4.5 % slower); above 6 items per SM the two alternate.
// Single calls scatter, since launches that run at the same time share SMs as they happen to fall (2^12 samples at 24, analysis of one, two,
// three signals on the run-time planned kernel: 11.3, 12.2, 10.3 us): over 76 calls of 2^12 ... 2^17 samples round trips differ from 17 % less
// to 12 % more, 3.6 % less on average, analysis alone from 30 % less to 18 % more, 5.7 % less, synthesis alone from 25 % less to 19 % more,
// 5.7 % less (64 threads per CTA: 2.9, 4.5 and 4.9 % less).
// With split bands it costs more than it gives (36 bands per octave: one signal of 2^17 60.1 -> 69.3 us, two 61.0 -> 71.8; one of
// 2^18 at 24 55.6 -> 65.3; 2^16 at 12: one 36.8 -> 38.2, two 44.9 -> 40.1, three 43.7 -> 48.5, six 46.4 -> 46.1): probably the code,
// since the split and the merged kernel wait for instructions more than for anything else and up to 19 lengths' code then passes
// through the same caches.  256 threads per CTA at any number of items: with 64 or 128 the same layouts gain 2.9 and 3.4 % where
// 256 gain 3.7.
static bool few_shape(const cqt_plan &p, int64_t batch, FewLaunch &f) {
    const int n = (int)p.merged.segs.size();
    const int split = n && p.merged.segs[0].lg_nthr == 10 ? 1 : 0;
    if (n - split > kMaxSegments) return false;
    for (int share = 1;; share *= 2) {   // emptier CTAs while there are SMs to spread over
        FewLaunch t;
        bool spread = false;
        t.chirp = !p.chirp.recs.empty();
        t.split = split > 0;
        // launch bounds of two CTAs per SM; one sub-transform of 8,192 points gives every CTA of its launch 139 KB
        auto add = [&](long long ctas, size_t smem) {
            const long long per_sm = std::max(1ll, ctas_per_sm(p, smem, 2));
            return (ctas + per_sm - 1) / per_sm;
        };
        long long sms = t.chirp ? add(chirp_grid(p, batch, nullptr), chirp_smem(p)) : 0;
        if (t.split) sms += add(4 * (long long)p.split.recs.size() * batch, split_smem(p));
        sms += few_part(p, batch, split, n, share, t.part, spread);
        if (sms > p.sm_count) {
            if (share == 1) return false;
            break;
        }
        f = t;
        if (!spread) break;
    }
    const long long items = (long long)p.cls[0].n_bands * batch;
    if (items > 16ll * p.sm_count) return false;
    f.short_threads = items > 4ll * p.sm_count ? 256 : 64;
    f.short_smooth = has_smooth(p, true, 0) && !f.split && items <= 6ll * p.sm_count;
    f.short_grid = (int)((items * 32 + f.short_threads - 1) / f.short_threads);
    return true;
}

template <bool ANALYSIS>
static cudaError_t launch_few(const cqt_plan &p, BandArgs &a, FewLaunch &f, cudaStream_t st) {
    static const char *names[2][2] = {{"bands_to_spectrum/merged", "bands_to_spectrum/class0"},
                                      {"bands_from_spectrum/merged", "bands_from_spectrum/class0"}};
    cudaError_t e = cudaSuccess;
    const int launches = f.chirp + f.split + (f.part.grid > 0) + (f.short_grid > 0);
    a.chain = launches > 1 ? kChainHead : kAlone;
    if (f.chirp) {
        e = launch_chirp(p, ANALYSIS, a, st);
        a.chain = a.chain == kChainHead ? kChainMember : a.chain;
    }
    if (f.split && e == cudaSuccess) {
        e = launch_split(p, ANALYSIS, a, st);
        a.chain = a.chain == kChainHead ? kChainMember : a.chain;
    }
    if (f.part.grid && e == cudaSuccess) {
        FewLaunch::Part &t = f.part;
        a.items = p.merged.d_items;
        void *args[] = {&a, &t.sg};
        const void *fn = ANALYSIS ? band_analysis_merged_kernel() : band_synthesis_merged_kernel();
        e = launch_kernel(fn, dim3((unsigned)t.grid), dim3((unsigned)t.threads), args, t.smem, st);
        note_launch(p, names[ANALYSIS][0], st);
        a.chain = a.chain == kChainHead ? kChainMember : a.chain;
    }
    if (f.short_grid && e == cudaSuccess) {
        const BandClass &c = p.cls[0];
        if (f.short_smooth) return launch_smooth(p, ANALYSIS, 0, a, st);
        a.items = c.d_items;
        void *args[] = {&a};
        e = launch_kernel(class_kernel<ANALYSIS>(c, 32, true), dim3((unsigned)f.short_grid), dim3((unsigned)f.short_threads), args,
                          (size_t)c.max_elems * (f.short_threads / 32) * sizeof(float2), st);
        note_launch(p, names[ANALYSIS][1], st);
    }
    return e;
}

// Power-of-two plans: two or three launches, chained, at any batch.  Class 0 on the kernel of 5-smooth lengths, against the run-time planned
// one, 38 calls of 2^12 ... 2^17 samples, 12 - 96 bands per octave and the multi-resolution layout, 1 - 415 signals: round trips from 24 % less to
// 6 % more, 9 % less on average; analysis alone from 35 % less to 23 % more, 11 % less; synthesis alone from 37 % less to 17 % more, 7 % less.
// A call that loses in one gains elsewhere (analysis, synthesis, round trip: 9 signals of 2^14 at 36 13.6 -> 16.7, 18.3 -> 16.5, 35.0 -> 34.5
// us; 115 of 2^12 at 12 16.2 -> 11.9, 17.9 -> 20.1, 32.5 -> 34.5); neither items per SM nor share of the coefficients tells them apart.
// CTAs of 64 or 128 threads instead of 256 above 4 items per SM: round trips 4 and 1 % slower on average (from 3 % less to 23 % more, 5 %
// less to 12 % more).
template <bool ANALYSIS>
static cudaError_t launch_pow2_plan(const cqt_plan &p, BandArgs &a, cudaStream_t st) {
    const BandClass &c = p.cls[0];
    const bool longer = pow2_has(p, true), shorter = pow2_has(p, false);
    cudaError_t e = cudaSuccess;
    a.chain = longer + shorter + (c.n_bands > 0) > 1 ? kChainHead : kAlone;
    for (bool long_ones : {true, false}) {
        if (!(long_ones ? longer : shorter) || e != cudaSuccess) continue;
        e = launch_pow2(p, ANALYSIS, long_ones, a, st);
        a.chain = a.chain == kChainHead ? kChainMember : a.chain;
    }
    if (c.n_bands > 0 && e == cudaSuccess) {
        const long long items = (long long)c.n_bands * a.batch;
        const int lanes = lanes_for(p, c, items), threads = items > 4ll * p.sm_count ? c.threads : 64, per_cta = threads / lanes;
        if (has_smooth(p, ANALYSIS, 0)) return launch_smooth(p, ANALYSIS, 0, a, st, threads);
        void *args[] = {&a};
        e = launch_kernel(class_kernel<ANALYSIS>(c, lanes, true), dim3((unsigned)((items + per_cta - 1) / per_cta)), dim3((unsigned)threads), args,
                          (size_t)c.max_elems * per_cta * sizeof(float2), st);
        note_launch(p, ANALYSIS ? "bands_from_spectrum/class0" : "bands_to_spectrum/class0", st);
    }
    return e;
}

// The classes of one call are independent (disjoint outputs), and most of them alone leave SMs idle, so they run
// side by side on the caller's stream and the plan's helper streams (one stream per class when all five classes
// have bands): fork after the caller's stream, join back into it.
// Per call, each class's run time is estimated as the larger of the time of its longest work item and its work
// at this batch size over the machine's throughput; the classes go, longest first, to the stream with the least
// time so far (the longest one therefore stays on the caller's stream).  With event timing on, everything stays
// on the caller's stream.
struct ForkJoin {
    const cqt_plan &p;
    cudaStream_t st;
    bool used[cqt_plan::kHelpers] = {};
    bool serial;
    int slot[kNumClasses] = {0, 0, 0, 0, 0};
    ForkJoin(const cqt_plan &plan, cudaStream_t s, int64_t batch)
        : p(plan), st(s), serial(plan.timing || !plan.aux[cqt_plan::kHelpers - 1]) {
        if (serial) return;
        constexpr double kElementStagesPerUs = 6.7e5;   // the 4096 < M <= 13,500 class at 32 signals
        double est[kNumClasses], load[cqt_plan::kHelpers] = {};   // the last helper is kept for the two-pass bands
        int order[kNumClasses];
        for (int c = 0; c < kNumClasses; ++c) {
            order[c] = c;
            est[c] = p.cls[c].n_bands ? std::max(p.cls[c].latency_us, p.cls[c].stage_work * (double)batch / kElementStagesPerUs) : 0.0;
        }
        std::stable_sort(order, order + kNumClasses, [&](int a, int b) { return est[a] > est[b]; });
        for (int i = 0; i < kNumClasses; ++i) {
            const int c = order[i];
            if (!p.cls[c].n_bands) continue;
            int best = 0;
            for (int j = 1; j < cqt_plan::kHelpers; ++j)
                if (load[j] < load[best]) best = j;
            slot[c] = best;
            load[best] += est[c];
        }
        cudaEventRecord(p.ev_fork, st);
    }
    cudaStream_t stream_for(int cls) {
        if (serial || slot[cls] == 0 || p.cls[cls].n_bands == 0) return st;
        const int i = slot[cls] - 1;
        if (!used[i]) { cudaStreamWaitEvent(p.aux[i], p.ev_fork, 0); used[i] = true; }
        return p.aux[i];
    }
    cudaStream_t two_pass_stream() {
        if (serial) return st;
        const int i = cqt_plan::kHelpers - 1;
        if (!used[i]) { cudaStreamWaitEvent(p.aux[i], p.ev_fork, 0); used[i] = true; }
        return p.aux[i];
    }
    void join() {
        for (int i = 0; i < cqt_plan::kHelpers; ++i)
            if (used[i]) { cudaEventRecord(p.ev_join[i], p.aux[i]); cudaStreamWaitEvent(st, p.ev_join[i], 0); }
    }
};

static bool has_two_pass(const cqt_plan &p) { return !p.two_pass[0].bands.empty() || !p.two_pass[1].bands.empty(); }

// Classes of the side-by-side form that run on the kernels of 5-smooth lengths.
// Analysis: class 1 alone 51 -> 44 us (256 signals of 2^15 samples at 24 bands per octave, whole call 90 -> 78), class 2 35 -> 31
// (32 signals of 2^19).  The two stay on the run-time planned engine in calls with two-pass bands, which have few items (one
// 2^22-sample signal 214 us, on these kernels 220), and in synthesis, where their last stage (window value, predicated store per
// slot) holds the items longer: class 1 37 -> 39, class 2 35 -> 39.  Nor class 1 beside class 0 alone, whose items then come
// late: 64 hops of a stereo stream 126.7 -> 131.6 us.
// Class 4, both directions: the items of one call fill one round of the SMs, and what counts is the time of one of them: 42 -> 33 us
// analysis, 39 -> 33 synthesis (128 items of up to 23,040 coefficients).  Not beside two-pass bands, where every SM has a length of
// its own and all their code passes through the caches at once (86 items of 27 lengths, one 2^22-sample signal at 96 bands per octave:
// analysis 85.0 -> 87.2, synthesis 113.8 -> 119.8; 49 items of 28 lengths, two 2^21-sample signals at 48: 99.6 -> 104.0, 121.8 -> 137.5).
// Class 0, 8 lanes per item either way, two stages instead of three.  Analysis, 12 layouts with 2 - 512 signals: from 43 % less to 1.4 %
// more (2^14 samples, 96 bands per octave: 512 signals 152 -> 86, 32 signals 21.4 -> 21.7); where it has 7 % of the coefficients or less,
// between 4 % less and 0.6 % more, whatever the items per SM (front end of 16, 64, 128 signals: 32.9 -> 33.1, 85.9 -> 86.3, 161.8 -> 160.7).
// Synthesis where class 1 is the longest: 33 % less to 0.9 % more in five layouts; beside longer classes its narrower shared memory lets
// more of its CTAs in ahead of their long items (front end of 32 signals 55.6 -> 57.4, 64 signals of 2^16 samples 62.6 -> 63.6).
bool smooth_form(const cqt_plan &p, bool analysis, int cls) {
    if (has_two_pass(p)) return false;
    const bool longer = p.cls[2].n_bands || p.cls[3].n_bands || p.cls[4].n_bands;
    return cls == 0 ? analysis || !longer : (analysis && longer) || cls == 4;
}
static bool class_is_smooth(const cqt_plan &p, bool analysis, int cls) { return has_smooth(p, analysis, cls) && smooth_form(p, analysis, cls); }

cudaError_t launch_bands_from_spectrum(const cqt_plan &p, const float *table, const float2 *X, const CoefRows &c,
                                       float2 *scratch, int64_t batch, cudaStream_t st) {
    FewLaunch f;
    if (!has_two_pass(p) && (!p.pow2.recs.empty() || few_shape(p, batch, f))) {
        BandArgs a = make_args(p, p.cls[0], table, batch);
        a.spec = X;
        a.spec_pitch = p.lf.x_pitch;
        set_rows(a, c);
        return p.pow2.recs.empty() ? launch_few<true>(p, a, f, st) : launch_pow2_plan<true>(p, a, st);
    }
    ForkJoin fj(p, st, batch);
    if (has_two_pass(p)) {
        cudaError_t e = launch_two_pass_from_spectrum(p, table, X, c, scratch, batch, fj.two_pass_stream());
        if (e != cudaSuccess) { fj.join(); return e; }
    }
    if (!p.pow2.recs.empty()) {   // its other bands are class 0's and two-pass ones
        BandArgs a = make_args(p, p.cls[0], table, batch);
        a.spec = X;
        a.spec_pitch = p.lf.x_pitch;
        set_rows(a, c);
        cudaError_t e = launch_pow2_plan<true>(p, a, st);
        fj.join();
        return e;
    }
    if (!p.chirp.recs.empty()) {
        BandArgs a = make_args(p, p.cls[0], table, batch);
        a.spec = X;
        a.spec_pitch = p.lf.x_pitch;
        set_rows(a, c);
        cudaError_t e = launch_chirp(p, true, a, fj.two_pass_stream());
        if (e != cudaSuccess) { fj.join(); return e; }
    }
    static const char *names[kNumClasses] = {"bands_from_spectrum/class0", "bands_from_spectrum/class1",
                                              "bands_from_spectrum/class2", "bands_from_spectrum/class3",
                                              "bands_from_spectrum/class4"};
    for (int i = kNumClasses - 1; i >= 0; --i) {   // longest bands first
        BandArgs a = make_args(p, p.cls[i], table, batch);
        a.spec = X;
        a.spec_pitch = p.lf.x_pitch;
        set_rows(a, c);
        if (p.cls[i].n_bands == 0) continue;
        cudaError_t e = class_is_smooth(p, true, i) ? launch_smooth(p, true, i, a, fj.stream_for(i)) : launch_class<true>(p, i, names[i], a, fj.stream_for(i));
        if (e != cudaSuccess) { fj.join(); return e; }
    }
    fj.join();
    return cudaSuccess;
}

// Zero-fill of the bins between a band's support and its widened range (layouts with nested supports).
__global__ void __launch_bounds__(128) zero_fill_kernel(float2 *Y, long long y_pitch, const int2 *seg) {
    const int2 sg = seg[blockIdx.x];
    float2 *y = Y + (long long)blockIdx.y * y_pitch + sg.x;
    for (int i = threadIdx.x; i < sg.y; i += blockDim.x) y[i] = make_float2(0.f, 0.f);
}

cudaError_t launch_bands_to_spectrum(const cqt_plan &p, const float *table, bool fold_sidebands, const CoefRows &c,
                                     float2 *Y, float2 *scratch, int64_t batch, cudaStream_t st) {
    if (p.n_zero_seg > 0) {
        zero_fill_kernel<<<dim3((unsigned)p.n_zero_seg, (unsigned)batch), 128, 0, st>>>(Y, p.y_pitch, p.d.zero_seg);
        note_launch(p, "zero_fill", st);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    FewLaunch f;
    if (!has_two_pass(p) && (!p.pow2.recs.empty() || few_shape(p, batch, f))) {
        BandArgs a = make_args(p, p.cls[0], table, batch);
        set_rows(a, c);
        a.Y = Y;
        a.fold = fold_sidebands ? 1 : 0;
        return p.pow2.recs.empty() ? launch_few<false>(p, a, f, st) : launch_pow2_plan<false>(p, a, st);
    }
    ForkJoin fj(p, st, batch);
    if (has_two_pass(p)) {
        cudaError_t e = launch_two_pass_to_spectrum(p, table, fold_sidebands, c, Y, scratch, batch, fj.two_pass_stream());
        if (e != cudaSuccess) { fj.join(); return e; }
    }
    if (!p.pow2.recs.empty()) {   // its other bands are class 0's and two-pass ones
        BandArgs a = make_args(p, p.cls[0], table, batch);
        set_rows(a, c);
        a.Y = Y;
        a.fold = fold_sidebands ? 1 : 0;
        cudaError_t e = launch_pow2_plan<false>(p, a, st);
        fj.join();
        return e;
    }
    if (!p.chirp.recs.empty()) {
        BandArgs a = make_args(p, p.cls[0], table, batch);
        set_rows(a, c);
        a.Y = Y;
        a.fold = fold_sidebands ? 1 : 0;
        cudaError_t e = launch_chirp(p, false, a, fj.two_pass_stream());
        if (e != cudaSuccess) { fj.join(); return e; }
    }
    static const char *names[kNumClasses] = {"bands_to_spectrum/class0", "bands_to_spectrum/class1",
                                              "bands_to_spectrum/class2", "bands_to_spectrum/class3",
                                              "bands_to_spectrum/class4"};
    for (int i = kNumClasses - 1; i >= 0; --i) {
        BandArgs a = make_args(p, p.cls[i], table, batch);
        set_rows(a, c);
        a.Y = Y;
        a.fold = fold_sidebands ? 1 : 0;
        if (p.cls[i].n_bands == 0) continue;
        cudaError_t e = class_is_smooth(p, false, i) ? launch_smooth(p, false, i, a, fj.stream_for(i)) : launch_class<false>(p, i, names[i], a, fj.stream_for(i));
        if (e != cudaSuccess) { fj.join(); return e; }
    }
    fj.join();
    return cudaSuccess;
}

cudaError_t configure_band_kernels(const cqt_plan &p) {
    for (const void *fn : {band_analysis_merged_kernel(), band_synthesis_merged_kernel()}) {
        cudaError_t e = allow_dynamic_smem(fn, 0, p);
        if (e != cudaSuccess) return e;
    }
    for (int i = 0; i < kNumClasses; ++i) {
        if (p.cls[i].n_bands == 0) continue;
        for (int lanes : {p.cls[i].lanes_few, p.cls[i].lanes_many})
            for (bool chained : {false, true}) {
                if (chained && i > 0) continue;   // chains contain class 0 only
                const size_t s = (size_t)p.cls[i].max_elems * (lanes ? p.cls[i].threads / lanes : 1) * sizeof(float2);
                if (!class_kernel<true>(p.cls[i], lanes, chained)) return cudaErrorInvalidDeviceFunction;
                cudaError_t e = allow_dynamic_smem(class_kernel<true>(p.cls[i], lanes, chained), s, p);
                if (e != cudaSuccess) return e;
                e = allow_dynamic_smem(class_kernel<false>(p.cls[i], lanes, chained), s, p);
                if (e != cudaSuccess) return e;
            }
    }
    return cudaSuccess;
}

}  // namespace cqt
