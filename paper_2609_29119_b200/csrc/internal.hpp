// Internal interfaces between the plan builder, the kernel launchers and the C ABI.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "layout.hpp"
#include "plan_types.h"

namespace cqt {

constexpr int kNumClasses = 5;
// Launch shape of one band-length class.
struct BandClass {
    int threads = 0;         // threads per CTA
    int min_blocks = 1;      // CTAs per SM the kernel instantiation is compiled for (register budget)
    int lanes_few = 0, lanes_many = 0;   // > 0: several (band, signal) items per CTA, that many lanes each, in a call
                                         // with few / many items; 0: one item per CTA
    int max_radix = 16;      // largest butterfly radix in the class's plans
    bool has_generic = false; // some band has a length with a prime factor above 5 (direct-sum stage)
    int max_elems = 0;       // shared-memory elements (float2) per item
    int n_bands = 0;         // bands in the class
    double stage_work = 0.0; // element-stages of the class's transforms per signal (stream assignment)
    double latency_us = 0.0; // estimated run time of the class's longest work item alone
    BandItem *d_items = nullptr;   // records + radix plans of the class's bands, longest first
    std::vector<int32_t> work;
};

// The single-CTA bands longer than class 0's ordered for one launch of all of them (calls with few work items): bands of one
// segment get the same number of threads per item, a power of two.
struct MergedBands {
    struct Segment { int first_band, n_bands, lg_nthr, elems; };   // elems: shared-memory elements (float2) of one item
    std::vector<Segment> segs;       // most threads first
    std::vector<int32_t> work;       // band indices in launch order
    BandItem *d_items = nullptr;
};

struct ChirpBands {
    int n_bands[kChirpLengths] = {};   // per length L of the sub-transforms, longest first
    std::vector<ChirpRec> recs;        // in that order
    ChirpRec *d_recs = nullptr;
};

struct Pow2Bands {
    int n_bands[kPow2Lengths] = {};    // per length, longest first
    std::vector<Pow2Rec> recs;         // in that order
    Pow2Rec *d_recs = nullptr;
};

// Bands of one class on the kernels of 5-smooth lengths: equal lengths adjacent, longest first
struct SmoothBands {
    struct Length { int M, first_band, n_bands, per; };   // per: work items of a CTA (SmoothShape::PER)
    std::vector<Length> lengths;
    size_t smem = 0;                   // of a CTA, the largest of the lengths
    std::vector<SmoothRec> recs;
    SmoothRec *d_recs = nullptr;
};

struct SplitBands {
    std::vector<BandItem> items;     // record of the band, radix plan of a quarter of its length
    std::vector<SplitRec> recs;
    BandItem *d_items = nullptr;
    SplitRec *d_recs = nullptr;
    int max_elems = 0;               // shared-memory elements (float2) of one item
};

struct LongFft {
    int64_t Lp = 0, A = 1, B = 0;
    int fft_A = -1, fft_B = -1;   // FftPlan indices
    int tw_n = 0, log_n_c = 0, n_n = 0;           // two-level table of W_N inside the twiddle array, its entry count
    int tw_fwd_u = 0, tw_fwd_v = 0, tw_inv_u = 0, tw_inv_v = 0;   // twiddles between the passes (api.cu)
    int64_t x_pitch = 0;          // elements per signal of the half-spectrum buffer (Lp + 1 rounded up)
};

using TwoPassBand = TwoPassRec;

struct TwoPassGroup {
    std::vector<TwoPassBand> bands;
    TwoPassRec *d_recs = nullptr;
    // per tile width (kTwoPassWidths): CTAs along the tiled index and shared memory of the two passes
    int max_tiles_cols[3] = {0, 0, 0}, max_tiles_rows[3] = {0, 0, 0};
    size_t smem_cols[3] = {0, 0, 0}, smem_rows[3] = {0, 0, 0};
};

struct DevicePlan {
    std::vector<void *> allocations;   // what the pointers below lie in
    BandRec *bands = nullptr;
    FftPlan *ffts = nullptr;
    float2 *tw = nullptr;
    float *tab_analysis = nullptr;     // g / M
    float *tab_synthesis = nullptr;    // h
    float *tab_analysis_adj = nullptr; // N g / (2 M)
    float *tab_synthesis_adj = nullptr;// h w_k / N
    int32_t *cover = nullptr;          // per bin: the planes that hold it (plane_sum in long_common.cuh)
    int *dbg = nullptr;                // 8 status words of the debug-bounds build
    int2 *zero_seg = nullptr;          // (offset into one signal's weighted-bin scratch, length): bins synthesis zero-fills
};

}  // namespace cqt

struct cqt_plan {
    cqt::HostLayout lay;
    std::vector<float> g32, h32;
    std::vector<cqt::FftPlan> ffts;
    std::vector<cqt::BandRec> bands;
    int device = -1;
    int64_t N = 0;
    int64_t y_pitch = 0;               // weighted-bin scratch elements per signal (y_planes * y_plane)
    int64_t y_plane = 0;               // elements per plane (N/2 + 1 rounded up)
    int y_planes = 1;                  // largest number of bands covering one bin
    int n_zero_seg = 0;                // zero-fill segments (layouts with nested supports only)
    cqt::LongFft lf;
    cqt::BandClass cls[cqt::kNumClasses];
    cqt::MergedBands merged;
    cqt::ChirpBands chirp;
    cqt::Pow2Bands pow2;
    cqt::SmoothBands smooth[cqt::kNumClasses];   // by class
    cqt::SplitBands split;             // the bands of the first segment of `merged` when that has 1024 threads per item
    std::vector<int8_t> band_class;    // length class of every band, -1: two-pass kernels
    cqt::TwoPassGroup two_pass[2];     // [0]: both factors <= 256, [1]: larger factors
    int64_t two_pass_pitch = 0;        // scratch elements per signal for the two-pass bands
    cqt::DevicePlan d;
    int max_smem_optin = 0;
    int sm_count = 0;
    // helper streams on which the short-band classes run beside the long-band classes of the same call
    static constexpr int kHelpers = 5;   // one per band class beside the caller's stream, one for the two-pass bands
    cudaStream_t aux[kHelpers] = {};
    cudaEvent_t ev_fork = nullptr, ev_join[kHelpers] = {};
    // launch counter and optional per-kernel event timing (benchmark aid; not thread safe)
    mutable int64_t launches = 0;
    mutable bool timing = false;
    mutable std::vector<cudaEvent_t> ev;
    mutable std::vector<const char *> ev_name;
    mutable size_t ev_used = 0;
};

namespace cqt {

// the per-bin cover words of the plan are bit masks of planes (plane_sum in long_common.cuh)
inline bool cover_is_mask(const cqt_plan &p) { return p.y_planes <= 31; }

// table selectors of the band kernels
enum { TAB_ANALYSIS = 0, TAB_SYNTHESIS = 1, TAB_ANALYSIS_ADJ = 2, TAB_SYNTHESIS_ADJ = 3 };

// api.cu: called after every kernel launch (and once at the start of a call with name == nullptr)
void note_launch(const cqt_plan &p, const char *name, cudaStream_t st);

// long_fft_forward.cu, long_fft_inverse.cu
// Input of the forward long FFT taken from a stream instead of signal rows (sliced transform, slice cut fused into the
// load): row r = slice r / channels of channel r % channels; sample i of that slice is win[i] * stream sample
// first + (r / channels) * hop + i, zero before the stream's start.  Stream samples from index new_first on are in the
// caller's buffer (fresh, zeros if null), older ones in the ring (sample n at n mod ring_len).  The last slice of the
// call also stores its fresh samples of index >= keep_from in the ring, where later slices find them.
struct SliceSource {
    float *ring;
    const float *win;
    long long ring_len, first, hop;
    int channels, slices;
    const float *fresh;
    long long fresh_stride, new_first, keep_from;
};
// src != nullptr needs a plan whose long FFT runs in two passes (can_fuse_slice_cut)
cudaError_t launch_rfft_forward(const cqt_plan &p, const float *x, int64_t x_stride, int64_t batch, int64_t valid_len,
                                float2 *T, float2 *X, cudaStream_t st, const SliceSource *src = nullptr);
inline bool can_fuse_slice_cut(const cqt_plan &p) { return p.lf.A > 1; }
cudaError_t launch_rfft_inverse(const cqt_plan &p, const float2 *Y, float2 *T, float *x, int64_t x_stride,
                                int64_t batch, int64_t valid_len, cudaStream_t st);
// The dynamic shared-memory limit is a property of the kernel function, shared by every plan of the process: it is
// raised to the device maximum, not to one plan's need (a later plan needing less would otherwise lower it under an
// earlier plan, whose launches would then fail).
inline cudaError_t allow_dynamic_smem(const void *fn, size_t need, const cqt_plan &p) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, fn);
    if (e != cudaSuccess) return e;
    const long long most = (long long)p.max_smem_optin - (long long)fa.sharedSizeBytes;   // static + dynamic share the limit
    if ((long long)need > most) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

// radix of the last stage of the passes that end with the twiddles between the passes
int long_cols_last_radix(int64_t A);            // forward pass C
int long_rows_inverse_last_radix(int64_t B);    // inverse pass R'
cudaError_t configure_long_forward_kernels(const cqt_plan &p);
cudaError_t configure_long_inverse_kernels(const cqt_plan &p);
cudaError_t configure_short_fft_kernels(const cqt_plan &p);

// Launch with the programmatic-serialization attribute (see pdl_wait in engine.cuh).
inline cudaError_t launch_kernel(const void *fn, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t st) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

// The same for a kernel called with its arguments (replaces kernel<<<grid, block, smem, st>>>(args...)).
template <class... KArgs, class... Args>
inline cudaError_t launch_kernel_args(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Coefficient rows of a call: row r at base + ((row0 + r) mod rows) * coeff_count.  Plain calls have row0 = 0 and no end;
// the sliced form keeps its slices in a ring of rows, and slices that wrap around its end go through one call.
struct CoefRows {
    float2 *base;
    int row0 = 0, rows = INT32_MAX;
};
__host__ __device__ inline long long coef_row(int row0, int rows, int r) { return r < rows - row0 ? row0 + r : row0 + r - rows; }

// band.cu
// every band of the plan: the single-CTA classes and, beside them on a stream of their own, the two-pass bands
// (scratch: their rows in the workspace)
cudaError_t launch_bands_from_spectrum(const cqt_plan &p, const float *table, const float2 *X, const CoefRows &c,
                                       float2 *scratch, int64_t batch, cudaStream_t st);
cudaError_t launch_bands_to_spectrum(const cqt_plan &p, const float *table, bool fold_sidebands, const CoefRows &c,
                                     float2 *Y, float2 *scratch, int64_t batch, cudaStream_t st);
cudaError_t configure_band_kernels(const cqt_plan &p);

// band_chirp.cu
int chirp_length_index(int64_t m);     // which L serves m-point sub-transforms, -1: none
int chirp_length(int index);
cudaError_t configure_chirp_kernels(const cqt_plan &p);

// band_pow2.cu
int pow2_length_index(int64_t M);                  // place of a length in Pow2Bands::n_bands, -1: not a length of that kernel
void pow2_radices(int index, int (&r)[5]);         // its stages (1: none)
cudaError_t configure_pow2_kernels(const cqt_plan &p);

// band_smooth.cu
struct SmoothInfo { int M, per, buf, r[5]; };        // r: stages (1: none); buf: shared-memory elements (float2) of an item
bool smooth_form(const cqt_plan &p, bool analysis, int cls);   // band.cu: the side-by-side form runs the class on them
const SmoothInfo *smooth_info(int64_t M);          // null: no shape for that length
cudaError_t configure_smooth_kernels(const cqt_plan &p);

// band_split.cu
cudaError_t configure_split_kernels(const cqt_plan &p);

// band_two_pass.cu
cudaError_t launch_two_pass_from_spectrum(const cqt_plan &p, const float *table, const float2 *X, const CoefRows &c,
                                          float2 *scratch, int64_t batch, cudaStream_t st);
cudaError_t launch_two_pass_to_spectrum(const cqt_plan &p, const float *table, bool fold, const CoefRows &c, float2 *Y,
                                        float2 *scratch, int64_t batch, cudaStream_t st);
cudaError_t configure_two_pass_kernels(const cqt_plan &p);
// tile widths (columns of pass 1 / rows of pass 2 per CTA) the kernels are compiled for, widest first
constexpr int kTwoPassWidths[3] = {16, 8, 4};
size_t two_pass_smem_cols(const TwoPassBand &b, int width);
size_t two_pass_smem_rows(const TwoPassBand &b, int width);

}  // namespace cqt
