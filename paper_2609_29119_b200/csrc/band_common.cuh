// Fused band kernels.
//  bands_from_spectrum: analysis form (Eq. analysis / band-spectrum).  One work item = (band, signal):
//      gather the band's bins from the half spectrum, multiply by the window table, place bin
//      kc + d in slot d mod M, zero the other slots, M-point inverse DFT in shared memory,
//      write the coefficients in time order.
//  bands_to_spectrum: synthesis form (Eq. synthesis).  M-point forward DFT of the coefficients in
//      shared memory, multiply the support slots by the dual-window table and write them in bin
//      order to the weighted-bin row of the signal (summed later, in fixed order, by the first pass
//      of the inverse long FFT).
// The same two kernels serve the adjoints with other tables (Sec. "Adjoints for training").
// This header: what the analysis-form and the synthesis-form kernels (one translation unit each) share.
#pragma once
#include "engine.cuh"
#include "internal.hpp"

namespace cqt {

struct BandArgs {
    const BandItem *items;   // per band of the class, in launch order (longest first): record + radix plan
    const float2 *tw;
    const float *table;
    int n_work;
    int batch;
    int N;
    int max_elems;           // shared-memory elements per item
    int fold;                // synthesis form: add conj of the mirrored slot for sidebands
    const float2 *spec;      // analysis form: half spectrum rows; synthesis form: unused
    long long spec_pitch;
    float2 *coef;            // coefficients (read or written), see CoefRows
    int row0, rows;
    long long coeff_count;
    float2 *Y;               // synthesis form: weighted-bin rows
    long long y_pitch;
    long long table_len;
    int chain;               // kAlone, kChainHead, kChainMember
    int *dbg;
};

// Band kernels of one call write disjoint outputs and need nothing of one another, only the kernel before the first
// of them.  In a chain on one stream the head lets its successor start only once all of its own CTAs have seen that
// kernel finish, so a member needs no wait before it reads; it waits for its predecessor at its end instead, so that
// "the last member has finished" means all have.  No event and no second stream is involved.
//
// What a member relies on.  Order: it starts after every CTA of the head has returned from griddepcontrol.wait (the head
// issues launch_dependents after it), so after the kernel before the head has finished.  Visibility: that wait makes what
// the earlier kernel wrote visible to the head, whose CTAs run on any SM, so it is in the L2 by then; the member has no wait
// of its own that would promise it the same, and its SM's L1 may in principle hold an older copy of a line.  Members
// therefore read the spectrum and the coefficients with strong loads of device scope (ld_chained), which go to the L2.
// Nothing else that a member reads is written by a kernel: records and tables belong to the plan.  What it costs: 3 clips
// of 8,000 samples 38.2 -> 38.6 us, one signal of 2^16 51.0 -> 51.3, seven of 99,225 68.8 -> 69.1, 128 signals of the
// multi-resolution layout 231 -> 231.  Kernels that wait for themselves keep ordinary loads: with strong ones in all class
// kernels 32 clips of 441,000 samples took 427 us instead of 423 and the front end of 64 clips 198 instead of 194.
enum { kAlone = 0, kChainHead = 1, kChainMember = 2 };
__device__ __forceinline__ void chain_enter(const BandArgs &a) {
    if (a.chain != kChainHead) pdl_launch_dependents();
}
__device__ __forceinline__ void chain_begin(const BandArgs &a) {
    if (a.chain != kChainMember) pdl_wait();
    if (a.chain == kChainHead) pdl_launch_dependents();
}
__device__ __forceinline__ void chain_end(const BandArgs &a) {
    if (a.chain == kChainMember) pdl_wait();
}

// One launch for all bands of a call with few work items (band.cu decides).  The bands are ordered by the number of
// threads an item of theirs gets, a power of two; a segment is a run of bands with the same number, walked by CTAs
// cta0 .. of the grid with per_cta items each (fewer than blockDim / nthr when there are SMs to spread over: the
// remaining threads exit).
constexpr int kMaxSegments = 6;    // 32 ... 1024 threads per item
constexpr int kMaxGroups = 16;     // items per CTA (one named barrier each)
struct BandSegment {
    int cta0, first_band, n_work, lg_nthr, per_cta, elems;   // elems: shared-memory elements of one item
};
struct BandSegments {
    int n;
    BandSegment s[kMaxSegments];
};
struct MergedItem {
    int band, ch, slot, tid, nthr, smem_off;
};
__device__ __forceinline__ bool merged_item(const BandArgs &a, const BandSegments &sg, MergedItem &m) {
    BandSegment s = sg.s[0];
#pragma unroll
    for (int i = 1; i < kMaxSegments; ++i)
        if (i < sg.n && (int)blockIdx.x >= sg.s[i].cta0) s = sg.s[i];
    m.slot = (int)threadIdx.x >> s.lg_nthr;
    const int item = ((int)blockIdx.x - s.cta0) * s.per_cta + m.slot;
    if (m.slot >= s.per_cta || item >= s.n_work * a.batch) return false;   // whole groups leave together
    m.nthr = 1 << s.lg_nthr;
    m.tid = (int)threadIdx.x & (m.nthr - 1);
    const int b = item / a.batch;
    m.band = s.first_band + b;
    m.ch = item - b * a.batch;
    m.smem_off = m.slot * s.elems;
    return true;
}

// THREADS / MINB: launch bounds of the class (64 registers per thread when THREADS * MINB = 1024 ... 2048)
// LANES: 0 = the whole CTA works on one item; 32, 16, 8 = that many consecutive lanes per item (THREADS / LANES items
// per CTA): the shortest bands have fewer butterflies per stage than a warp has lanes
template <int LANES>
struct Group {
    __device__ static int tid() { return LANES ? (int)(threadIdx.x & (LANES - 1)) : (int)threadIdx.x; }
    __device__ static int nthr() { return LANES ? LANES : (int)blockDim.x; }
    __device__ static int per_cta() { return LANES ? (int)blockDim.x / (LANES ? LANES : 1) : 1; }
    __device__ static int slot() { return LANES ? (int)threadIdx.x / (LANES ? LANES : 1) : 0; }
    __device__ static int item() { return LANES ? (int)blockIdx.x * per_cta() + slot() : (int)blockIdx.x; }
};
template <int LANES>
using GroupSync = typename std::conditional<LANES == 0, BlockSync,
                                            typename std::conditional<LANES == 32, WarpSync, LaneGroupSync<(LANES ? LANES : 1)>>::type>::type;

// Loads of the spectrum and of coefficients in kernels that run both as members of a chain and waiting for themselves
template <bool CHAINED>
__device__ __forceinline__ float2 ld_spectrum(const float2 *p) { return CHAINED ? ld_chained(p) : ld_data(p); }
template <bool CHAINED>
__device__ __forceinline__ float2 ld_coefficient(const float2 *p) { return CHAINED ? ld_chained(p) : __ldcs(p); }

extern __shared__ float2 smem_band[];

// The work item's band record and radix plan are fetched together, once, into shared memory: their fields are
// read inside the stage loops, where a shared-memory copy costs a short-latency load and the global original a
// cache lookup, and one cooperative load replaces a chain of two dependent ones.
template <class Sync>
__device__ __forceinline__ void fetch_item(const BandItem &g, BandItem &s, int tid, int nthr) {
    constexpr int kWords = (int)(sizeof(BandItem) / sizeof(int));
    for (int i = tid; i < kWords; i += nthr) reinterpret_cast<int *>(&s)[i] = __ldg(reinterpret_cast<const int *>(&g) + i);
    Sync::sync(nthr);
}

// Analysis form, any band: slot m of the transform's input, i.e. tab[d] X[kc + d] with d = m or m - M, zero outside the
// support; bins outside 0..N/2 are the conjugates of their mirror bins.
// No branch around the loads, so that those of several slots are in flight together.
template <bool CHAINED>
__device__ __forceinline__ float2 slot_value(const BandRec &br, const float *__restrict__ tab,
                                             const float2 *__restrict__ X, int N, int m, int *dbg) {
    const bool lo = m <= br.d0 + br.S - 1, ok = lo || m >= br.M + br.d0;
    const int d = ok ? (lo ? m : m - br.M) : 0, k = br.kc + d, half = N >> 1;
    const bool mirrored = k < 0 || k > half;
    const int km = k < 0 ? -k : (k > half ? N - k : k);
    if (!CQT_CHK(dbg, 405, d - br.d0, br.S) || !CQT_CHK(dbg, 406, km, half + 1)) return make_float2(0.f, 0.f);
    const float g = ok ? __ldg(tab + (d - br.d0)) : 0.f;
    const float2 x = ld_spectrum<CHAINED>(X + km);
    return make_float2(g * x.x, mirrored ? -(g * x.y) : g * x.y);
}

// Synthesis form, any band: output u of slot m, times the window table, to bin kc + d of the band's plane Y (only bins
// 0..N/2 are kept).
__device__ __forceinline__ void slot_store(const BandRec &br, const float *__restrict__ tab, float2 *__restrict__ Y, int N, int m, float2 u,
                                           int *dbg = nullptr, long long limit = 1ll << 40) {
    const int last_pos = br.d0 + br.S - 1, first_neg = br.M + br.d0;
    int d;
    if (m <= last_pos) d = m;
    else if (m >= first_neg) d = m - br.M;
    else return;
    const int k = br.kc + d;
    if (k < 0 || k > (N >> 1)) return;
    const float h = __ldg(tab + (d - br.d0));
    if (CQT_CHK(dbg, 404, k, limit)) Y[k] = make_float2(h * u.x, h * u.y);
}

// band_pow2.cu: every band of more than 128 coefficients of a plan where those are all powers of two, in two launches by
// length (the first often empty)
bool pow2_has(const cqt_plan &p, bool long_ones);
cudaError_t launch_pow2(const cqt_plan &p, bool analysis, bool long_ones, const BandArgs &b, cudaStream_t st);

// band_smooth.cu: every band of class cls, where the plan and the direction have that form; threads: of a CTA, 0: the class's (only class 0 has a choice)
bool has_smooth(const cqt_plan &p, bool analysis, int cls);
cudaError_t launch_smooth(const cqt_plan &p, bool analysis, int cls, const BandArgs &b, cudaStream_t st, int threads = 0);

// band_split.cu: long bands of calls with few items
size_t split_smem(const cqt_plan &p);
cudaError_t launch_split(const cqt_plan &p, bool analysis, const BandArgs &b, cudaStream_t st);

// band_chirp.cu: bands of more than 128 coefficients whose length has a prime factor above 5
constexpr int kChirpThreads = 256;
struct ChirpSegment {
    int cta0, n_cta, first_band, n_bands;
};
int chirp_grid(const cqt_plan &p, int64_t batch, ChirpSegment *seg);
size_t chirp_smem(const cqt_plan &p);
cudaError_t launch_chirp(const cqt_plan &p, bool analysis, const BandArgs &b, cudaStream_t st);

// Kernel instantiations: (threads per CTA, CTAs per SM the registers must allow, lanes per item or 0 for the whole CTA, largest radix
// compiled in), each with and without the prime-factor paths (GEN): code a class never runs is left out, which also
// frees registers in the paths it does run.
#define CQT_KERNEL_TABLE(X) \
    X(256, 4, 8, 8) X(256, 4, 32, 8) X(128, 8, 0, 12) X(256, 4, 0, 12) X(512, 2, 0, 16) X(1024, 1, 0, 16)

}  // namespace cqt
