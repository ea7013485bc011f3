// Long bands of calls with few items, each as four work items.
//
// Bounds: latency.  A band of 24,000 coefficients on one CTA is 24 elements per thread and stage on a single SM: 31 us
// analysis, 35 us synthesis, of a 100 us round trip of seven signals whose other bands were done after 9.  One radix-4
// step, taken on load, makes four independent transforms of a quarter of the length (as in band_chirp.cu, with m = M/4),
//   X[k0 + 4 k'] = sum_n' W_m^{n' k'} y_k0[n'],   y_k0[n'] = W_M^{n' k0} sum_q W_4^{q k0} x[n' + q m],
// on four SMs, at the price of reading every input four times, from the L2.
#include "band_common.cuh"

namespace cqt {

constexpr int kSplitThreads = 512;

template <int R, int SIGN>
__device__ __forceinline__ void split_first_stage(float2 *buf, const FftPlan &fp, const float2 *tw, int tid, int nthr) {
    const int s = fp.st[0].stride, step = s + fp.pad_delta, logC = fp.logC;
    for (int b = tid; b < s; b += nthr) {
        float2 *p = buf + b;
        float re[R], im[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const float2 v = p[q * step];
            re[q] = v.x; im[q] = v.y;
        }
        if (SIGN < 0) Codelet<R>::run(re, im); else Codelet<R>::run(im, re);
        apply_twiddle_powers<R, SIGN>(tw, logC, (uint32_t)b, re, im);
#pragma unroll
        for (int q = 0; q < R; ++q) p[q * step] = make_float2(re[q], im[q]);
    }
}

template <int SIGN, class Store>
__device__ __forceinline__ void split_fft(float2 *buf, const FftPlan &fp, const float2 *tw, Store store, int *dbg, int tid, int nthr) {
    const int d = fp.nstages;
    const Tile t{buf, 1, 1, 0u, fp.M + 16, dbg};
#define X(RR) case RR: split_first_stage<RR, SIGN>(buf, fp, tw, tid, nthr); break;
    switch (fp.st[0].radix) { CQT_RADIX_CASES_ALL(X) default: break; }
#undef X
    __syncthreads();
    int n_cur = fp.st[0].stride, tmul = fp.st[0].radix;
#pragma unroll 1
    for (int j = 1; j < d - 1; ++j) {
#define X(RR) case RR: middle_stage<RR, SIGN, true, false>(t, fp, tw, j, n_cur, tmul, tid, nthr); break;
        switch (fp.st[j].radix) { CQT_RADIX_CASES_ALL(X) default: break; }
#undef X
        __syncthreads();
        n_cur = fp.st[j].stride;
        tmul *= fp.st[j].radix;
    }
#define X(RR) case RR: last_stage<RR, SIGN, true, true, false>(t, fp, store, tid, nthr); break;
    switch (fp.st[d - 1].radix) { CQT_RADIX_CASES_ALL(X) default: break; }
#undef X
}


extern __shared__ float2 smem_split[];

// items: record of the band (M coefficients) with the radix plan of length M / 4
template <bool ANALYSIS>
__global__ void __launch_bounds__(kSplitThreads, 2) split_bands_kernel(BandArgs a, const SplitRec *extra) {
    chain_enter(a);
    const int tid = threadIdx.x;
    const int k0 = blockIdx.x & 3, item = blockIdx.x >> 2, band = item / a.batch, ch = item - band * a.batch;
    __shared__ BandItem it;
    fetch_item<BlockSync>(a.items[band], it, tid, kSplitThreads);
    const BandRec br = it.br;
    const FftPlan &fp = it.fp;
    const int m = fp.M;
    float2 *buf = smem_split, *tws = buf + m + 16, *twm = tws + fp.tw_count;
    const SplitRec x = extra[band];
    stage_twiddles(tws, a.tw, fp, tid, kSplitThreads);
    for (int i = tid; i < x.n_m; i += kSplitThreads) twm[i] = __ldg(a.tw + x.tw_m + i);
    chain_begin(a);   // record, plan and tables belong to the plan; what follows touches the predecessor's output
    __syncthreads();
    const float *tab = a.table + br.tab_off;
    const float2 *X = ANALYSIS ? a.spec + (long long)ch * a.spec_pitch : nullptr;
    float2 *c = a.coef + coef_row(a.row0, a.rows, ch) * a.coeff_count + br.coeff_off;
    float2 *Y = ANALYSIS ? nullptr : a.Y + (long long)ch * a.y_pitch + br.y_off;
    const bool fold = !ANALYSIS && a.fold && br.side != 0;
    auto in = [&](int n) -> float2 {
        if constexpr (ANALYSIS) return slot_value<true>(br, tab, X, a.N, n, a.dbg);
        const float2 v = CQT_CHK(a.dbg, 601, n, br.M) ? ld_chained(c + n) : make_float2(0.f, 0.f);
        return fold ? make_float2(2.f * v.x, 0.f) : v;
    };
    constexpr float sign = ANALYSIS ? 1.f : -1.f;    // of the transform's exponent
    const int s0 = fp.st[0].stride;
    const uint32_t s0magic = fp.st[0].smagic;
    const float e2 = (k0 & 1) ? -1.f : 1.f, o2 = (k0 & 2) ? -1.f : 1.f;
#pragma unroll 4
    for (int n = tid; n < m; n += kSplitThreads) {
        const float2 x0 = in(n), x1 = in(n + m), x2 = in(n + 2 * m), x3 = in(n + 3 * m);
        const float2 e = make_float2(fmaf(e2, x2.x, x0.x), fmaf(e2, x2.y, x0.y)), o = make_float2(fmaf(e2, x3.x, x1.x), fmaf(e2, x3.y, x1.y));
        // k0 even: e +- o; k0 odd: e +- i o, plus for k0 = 1 with a positive exponent
        const float u = (k0 & 1) ? sign * o2 : o2;
        const float2 v = (k0 & 1) ? make_float2(fmaf(-u, o.y, e.x), fmaf(u, o.x, e.y)) : make_float2(fmaf(u, o.x, e.x), fmaf(u, o.y, e.y));
        float2 w = twiddle_s(twm, x.log_m_c, (uint32_t)n * (uint32_t)k0);
        if (ANALYSIS) w.y = -w.y;
        buf[fp.pad_delta ? n + (int)fastdiv((uint32_t)n, s0magic, (uint32_t)s0) : n] = cmul(v, w);
    }
    __syncthreads();
    if constexpr (ANALYSIS)
        split_fft<+1>(buf, fp, tws, [&](int n, int, float2 v) { if (CQT_CHK(a.dbg, 602, k0 + 4 * n, br.M)) c[k0 + 4 * n] = v; }, a.dbg, tid, kSplitThreads);
    else
        split_fft<-1>(buf, fp, tws, [&](int n, int, float2 v) { slot_store(br, tab, Y, a.N, k0 + 4 * n, v, a.dbg, (long long)a.y_pitch - br.y_off); }, a.dbg, tid,
                      kSplitThreads);
    chain_end(a);
}

size_t split_smem(const cqt_plan &p) { return (size_t)p.split.max_elems * sizeof(float2); }

cudaError_t launch_split(const cqt_plan &p, bool analysis, const BandArgs &b, cudaStream_t st) {
    BandArgs a = b;
    a.items = p.split.d_items;
    const SplitRec *extra = p.split.d_recs;
    void *args[] = {&a, &extra};
    const void *fn = analysis ? (const void *)split_bands_kernel<true> : (const void *)split_bands_kernel<false>;
    cudaError_t e = launch_kernel(fn, dim3((unsigned)(4 * p.split.recs.size() * b.batch)), dim3(kSplitThreads), args, split_smem(p), st);
    note_launch(p, analysis ? "bands_from_spectrum/split" : "bands_to_spectrum/split", st);
    return e;
}

cudaError_t configure_split_kernels(const cqt_plan &p) {
    if (p.split.recs.empty()) return cudaSuccess;
    cudaError_t e = allow_dynamic_smem((const void *)split_bands_kernel<true>, split_smem(p), p);
    return e != cudaSuccess ? e : allow_dynamic_smem((const void *)split_bands_kernel<false>, split_smem(p), p);
}

}  // namespace cqt
