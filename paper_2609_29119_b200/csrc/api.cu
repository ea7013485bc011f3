// Plan construction and the C ABI of the transform calls (see include/cqt.h).
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <memory>
#include <new>

#include "../../include/cqt.h"
#include "internal.hpp"
#include "table_upload.hpp"

using namespace cqt;

namespace {

const double kPi = 3.14159265358979323846;

uint32_t magic_of(uint32_t d) { return d <= 1 ? 0u : (uint32_t)(((1ull << 32) + d - 1) / d); }

// two-level table of exp(-2 pi i y / n), 0 <= y < n, appended to tw; returns offset and log2 C
int append_twiddles(std::vector<float2> &tw, int64_t n, int &logC) {
    logC = 0;
    while ((1ll << (2 * logC)) < n) ++logC;
    const int64_t C = 1ll << logC;
    const int64_t nhi = (n + C - 1) / C;
    const int off = (int)tw.size();
    for (int64_t j = 0; j < C; ++j) {
        const double ang = -2.0 * kPi * (double)(j % n) / (double)n;
        tw.push_back(make_float2((float)std::cos(ang), (float)std::sin(ang)));
    }
    for (int64_t i = 0; i < nhi; ++i) {
        const double ang = -2.0 * kPi * (double)((i * C) % n) / (double)n;
        tw.push_back(make_float2((float)std::cos(ang), (float)std::sin(ang)));
    }
    return off;
}

// Twiddle rows of the stages before the last (radices r, trailing ones: fewer stages), appended to tw: on sub-transforms of n
// points rows W_n^{p y}, y < n / r, p = 1, 2, 4, ... < r.  Returns the offset.  W_n^y is a product of two double factors
// (1e-16), rounded once: sqrt(n) sines and cosines instead of n.  Plain arrays, the rows sized ahead: the 87 lengths up to 4096 that
// have shapes take 0.22 ms, with std::polar, complex vectors and push_back 1.15 (a plan with rows for 62 lengths 4.12 and 4.35).
int append_twiddle_rows(std::vector<float2> &tw, int64_t M, const int (&r)[5]) {
    const size_t off = tw.size();
    size_t entries = 0;
    int n = (int)M;
    for (int j = 0; j < 4 && r[j + 1] > 1; ++j) {
        n /= r[j];
        for (int pw = 1; pw < r[j]; pw *= 2) entries += (size_t)n;
    }
    tw.resize(off + entries);
    float2 *out = tw.data() + off;
    std::vector<double> roots;   // W_n^i, then W_n^{i 2^lg}
    n = (int)M;
    for (int j = 0; j < 4 && r[j + 1] > 1; ++j) {
        int lg = 2;
        while ((1ll << (2 * lg)) < n) ++lg;
        const int low = (1 << lg) - 1, coarse = (n + low) >> lg;
        roots.resize((size_t)(2 * (low + 1 + coarse)));
        double *const fine = roots.data(), *const high = fine + 2 * (low + 1);
        auto fill = [&](double *to, int count, int step) {
            for (int i = 0; i < count; ++i) {
                const double angle = -2.0 * kPi * (double)(i * step) / (double)n;
                to[2 * i] = std::cos(angle);
                to[2 * i + 1] = std::sin(angle);
            }
        };
        fill(fine, low + 1, 1);
        fill(high, coarse, 1 << lg);
        for (int pw = 1; pw < r[j]; pw *= 2)
            for (int i = 0, y = 0; i < n / r[j]; ++i, y += pw) {   // y below n
                const double *u = fine + 2 * (y & low), *v = high + 2 * (y >> lg);
                *out++ = make_float2((float)(u[0] * v[0] - u[1] * v[1]), (float)(u[0] * v[1] + u[1] * v[0]));
            }
        n /= r[j];
    }
    return (int)off;
}

const int kBandRadices[] = {16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2};
const int kPow2Radices[] = {16, 8, 4, 2};

// fewest stages, then smallest largest radix; no radix above `cap`
bool best_split(int64_t m, const int *radices, int nr, int cap, std::map<int64_t, std::vector<int>> &memo, std::vector<int> &out) {
    if (m == 1) { out.clear(); return true; }
    auto it = memo.find(m);
    if (it != memo.end()) { out = it->second; return !out.empty(); }
    std::vector<int> best;
    for (int i = 0; i < nr; ++i) {
        const int r = radices[i];
        if (m % r || r > cap) continue;
        std::vector<int> sub;
        if (!best_split(m / r, radices, nr, cap, memo, sub)) continue;
        sub.push_back(r);
        std::sort(sub.begin(), sub.end(), [](int a, int b) { return a > b; });
        if (best.empty() || sub.size() < best.size() || (sub.size() == best.size() && sub[0] < best[0])) best = sub;
    }
    memo[m] = best;
    out = best;
    return !best.empty();
}

// returns false if M cannot be planned
bool make_fft_plan(int64_t M, bool pow2, std::vector<float2> &tw, FftPlan &fp, bool want_full = false, int radix_cap = 16) {
    std::memset(&fp, 0, sizeof(fp));
    fp.M = (int32_t)M;
    int64_t smooth = M, rest = 1;
    if (!pow2) {
        smooth = 1;
        int64_t m = M;
        for (int p : {2, 3, 5})
            while (m % p == 0) { m /= p; smooth *= p; }
        rest = m;
        if (rest > 4096) return false;
    }
    std::map<int64_t, std::vector<int>> memo;
    std::vector<int> radices;
    if (!best_split(smooth, pow2 ? kPow2Radices : kBandRadices, pow2 ? 4 : 11, radix_cap, memo, radices)) return false;
    if (rest > 1) { radices.insert(radices.begin(), (int)rest); fp.generic = 1; }
    if (radices.empty()) radices.push_back(1);
    if ((int)radices.size() > kMaxStages) return false;
    fp.nstages = (int32_t)radices.size();
    int64_t n_cur = M;
    for (int j = 0; j < fp.nstages; ++j) {
        fp.st[j].radix = radices[j];
        fp.st[j].stride = (int32_t)(n_cur / radices[j]);
        fp.st[j].rmagic = magic_of((uint32_t)radices[j]);
        fp.st[j].smagic = magic_of((uint32_t)fp.st[j].stride);
        const int64_t kd = j == 0 ? 1 : fp.st[0].stride / n_cur;
        fp.st[j].k1div = (int32_t)kd;
        fp.st[j].k1magic = magic_of((uint32_t)kd);
        n_cur /= radices[j];
    }
    int logC;
    fp.tw_off = append_twiddles(tw, M, logC);
    fp.logC = logC;
    fp.tw_count = (int32_t)((1ll << logC) + (M + (1ll << logC) - 1) / (1ll << logC));
    fp.pad_delta = (fp.nstages > 1 && (fp.st[0].stride % 2 == 0)) ? 1 : 0;
    fp.tw_full_off = -1;
    if (pow2 || want_full) {
        fp.tw_full_off = (int32_t)tw.size();
        for (int64_t y = 0; y < M; ++y) {
            const double ang = -2.0 * kPi * (double)y / (double)M;
            tw.push_back(make_float2((float)std::cos(ang), (float)std::sin(ang)));
        }
    }
    return true;
}

// host-side helpers for the chirp-z tables
void host_fft_pow2(std::vector<std::complex<double>> &v) {   // in-place radix-2, forward sign
    const size_t n = v.size();
    for (size_t i = 1, j = 0; i < n; ++i) {
        size_t bit = n >> 1;
        for (; j & bit; bit >>= 1) j ^= bit;
        j ^= bit;
        if (i < j) std::swap(v[i], v[j]);
    }
    for (size_t len = 2; len <= n; len <<= 1) {
        const double ang = -2.0 * kPi / (double)len;
        for (size_t i = 0; i < n; i += len)
            for (size_t k = 0; k < len / 2; ++k) {
                const std::complex<double> w = std::polar(1.0, ang * (double)k);
                const std::complex<double> u = v[i + k], t = v[i + k + len / 2] * w;
                v[i + k] = u + t;
                v[i + k + len / 2] = u - t;
            }
    }
}

// tables of a band on the chirp-z kernel (see ChirpRec): sub-transforms of m points, convolution length L
void make_chirp_tables(int64_t m, int64_t L, std::vector<float2> &tw, ChirpRec &cr) {
    cr.pre_off = (int32_t)tw.size();
    for (int64_t k0 = 0; k0 < 4; ++k0)
        for (int64_t n = 0; n < m; ++n) {
            // n k0 / (2 m) + n^2 / m in units of 1 / (2 m), periodic with 4 m
            const double ang = -kPi * (double)((n * k0 + 2 * n * n) % (4 * m)) / (double)(2 * m);
            tw.push_back(make_float2((float)std::cos(ang), (float)std::sin(ang)));
        }
    std::vector<std::complex<double>> b((size_t)L, 0.0);
    for (int64_t n = 0; n < m; ++n) {
        const std::complex<double> c = std::polar(1.0, kPi * (double)((n * n) % (2 * m)) / (double)m);   // conj chirp
        b[(size_t)n] = c;
        if (n) b[(size_t)(L - n)] = c;
    }
    host_fft_pow2(b);
    cr.filter_off = (int32_t)tw.size();
    for (const std::complex<double> &v : b) tw.push_back(make_float2((float)(v.real() / (double)L), (float)(v.imag() / (double)L)));
}

void free_device(cqt_plan *p) {
    if (p->device < 0) return;
    int cur = 0;
    cudaGetDevice(&cur);
    cudaSetDevice(p->device);
    for (void *a : p->d.allocations) cudaFree(a);
    for (cudaEvent_t e : p->ev) cudaEventDestroy(e);
    for (int i = 0; i < cqt_plan::kHelpers; ++i) {
        if (p->aux[i]) cudaStreamDestroy(p->aux[i]);
        if (p->ev_join[i]) cudaEventDestroy(p->ev_join[i]);
    }
    if (p->ev_fork) cudaEventDestroy(p->ev_fork);
    cudaSetDevice(cur);
}

struct PlanDestroy {
    void operator()(cqt_plan *p) const { cqt_plan_destroy(p); }
};
using OwnedPlan = std::unique_ptr<cqt_plan, PlanDestroy>;   // on every path out of a creating function, exceptions among them

struct RestoreDevice {
    int cur;
    ~RestoreDevice() { cudaSetDevice(cur); }
};

bool is_pow2(int64_t v) { return v > 0 && (v & (v - 1)) == 0; }

}  // namespace

extern "C" {

const char *cqt_status_string(cqt_status s) {
    switch (s) {
        case CQT_OK: return "ok";
        case CQT_ERR_INVALID_ARG: return "invalid argument";
        case CQT_ERR_UNSUPPORTED: return "unsupported size or layout";
        case CQT_ERR_BAD_LAYOUT: return "band layout is not a painless frame";
        case CQT_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
        case CQT_ERR_CUDA: return "CUDA error";
        case CQT_ERR_STATE: return "call not valid in this state";
        case CQT_ERR_DEVICE_CHECK: return "device-side check failed";
    }
    return "unknown status";
}

cqt_status cqt_plan_create(double fs, double fmin, double fmax, int bins_per_octave, int64_t L, cqt_window window,
                           cqt_plan **out) {
    cqt_plan_desc d;
    d.fs = fs; d.fmin = fmin; d.fmax = fmax; d.bins_per_octave = bins_per_octave; d.L = L;
    d.window = (int)window; d.m_policy = CQT_M_MULT4; d.min_win = 4.0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return CQT_ERR_CUDA;
    d.device = dev;
    return cqt_plan_create_ex(&d, out);
}

static cqt_status finish_plan(OwnedPlan p, int64_t N, int device, const cqt_plan_tuning &tune, cqt_plan **out);

static bool length_supported(int64_t N) { return is_pow2(N) && N >= 64 && N <= (1ll << 22); }

cqt_status cqt_plan_create_ex(const cqt_plan_desc *desc, cqt_plan **out) {
    return cqt_plan_create_tuned(desc, nullptr, out);
}

cqt_status cqt_plan_create_tuned(const cqt_plan_desc *desc, const cqt_plan_tuning *tuning, cqt_plan **out) try {
    if (!desc || !out) return CQT_ERR_INVALID_ARG;
    cqt_plan_tuning tune{};
    if (tuning) tune = *tuning;
    if (tune.max_cta_elems < 0 || tune.two_pass_min < 0) return CQT_ERR_INVALID_ARG;
    const int64_t N = desc->L;
    if (N < 0) return CQT_ERR_INVALID_ARG;
    if (!length_supported(N)) return CQT_ERR_UNSUPPORTED;
    OwnedPlan p(new cqt_plan());
    LayoutDesc ld{desc->fs, desc->fmin, desc->fmax, desc->bins_per_octave, N, desc->window, desc->m_policy,
                  desc->min_win > 0 ? desc->min_win : 4.0};
    std::string why;
    int rc = build_layout(ld, p->lay, why);
    if (rc != 0) return (cqt_status)rc;
    return finish_plan(std::move(p), N, desc->device, tune, out);
} catch (...) {   // host memory ran out
    return CQT_ERR_CUDA;
}

cqt_status cqt_plan_create_bands(const cqt_band_list_desc *desc, cqt_plan **out) try {
    if (!desc || !out || !desc->centre_hz || !desc->width_bins || desc->n_bands < 1 || desc->L < 0) return CQT_ERR_INVALID_ARG;
    const int64_t N = desc->L;
    if (!length_supported(N)) return CQT_ERR_UNSUPPORTED;
    if (desc->n_bands > 100000) return CQT_ERR_UNSUPPORTED;
    std::vector<BandSpec> specs((size_t)desc->n_bands);
    for (int64_t i = 0; i < desc->n_bands; ++i)
        specs[i] = BandSpec{desc->centre_hz[i], desc->width_bins[i], desc->group ? desc->group[i] : -1};
    OwnedPlan p(new cqt_plan());
    LayoutDesc ld{desc->fs, 0.0, 0.0, 0, N, desc->window, desc->m_policy, 4.0};
    std::string why;
    int rc = build_layout_bands(ld, specs, p->lay, why);
    if (rc != 0) return (cqt_status)rc;
    return finish_plan(std::move(p), N, desc->device, cqt_plan_tuning{}, out);
} catch (...) {
    return CQT_ERR_CUDA;
}

cqt_status cqt_multires_bands(double fs, double fmin, int64_t L, const int *octaves, const int *bins_per_octave,
                              int n_sections, double min_win, int64_t capacity, double *centre_hz, double *width_bins,
                              int32_t *group, int64_t *n_bands) try {
    if (!n_bands || capacity < 0) return CQT_ERR_INVALID_ARG;
    std::vector<BandSpec> specs;
    std::string why;
    int rc = multires_bands(fs, fmin, L, octaves, bins_per_octave, n_sections, min_win > 0 ? min_win : 4.0, specs, why);
    if (rc != 0) return (cqt_status)rc;
    *n_bands = (int64_t)specs.size();
    for (int64_t i = 0; i < std::min<int64_t>(capacity, (int64_t)specs.size()); ++i) {
        if (centre_hz) centre_hz[i] = specs[i].f;
        if (width_bins) width_bins[i] = specs[i].W;
        if (group) group[i] = specs[i].group;
    }
    return CQT_OK;
} catch (...) {
    return CQT_ERR_CUDA;
}

static cqt_status finish_plan(OwnedPlan p, int64_t N, int device, const cqt_plan_tuning &tune, cqt_plan **out) {
    p->N = N;
    const HostLayout &L = p->lay;
    p->g32.resize(L.table_len);
    p->h32.resize(L.table_len);
    for (int64_t i = 0; i < L.table_len; ++i) { p->g32[i] = (float)L.g[i]; p->h32[i] = (float)L.h[i]; }
    p->y_planes = 1;
    for (int64_t k = 0; k <= N / 2; ++k) p->y_planes = std::max(p->y_planes, (int)L.cover_n[k]);
    p->y_plane = (N / 2 + 1 + 7) / 8 * 8;
    p->y_pitch = p->y_plane * p->y_planes;

    // ---- transform-length plans and twiddles
    std::vector<float2> tw;
    std::map<int64_t, int> fft_of;
    enum { kPlanBand = 0, kPlanPow2 = 1, kPlanFull = 2 };
    auto plan_for = [&](int64_t M, int kind, int cap) -> int {
        const int64_t key = M + ((int64_t)kind << 40) + ((int64_t)cap << 44);
        auto it = fft_of.find(key);
        if (it != fft_of.end()) return it->second;
        FftPlan fp;
        if (!make_fft_plan(M, kind == kPlanPow2, tw, fp, kind == kPlanFull, cap)) return fft_of[key] = -1;
        p->ffts.push_back(fp);
        return fft_of[key] = (int)p->ffts.size() - 1;
    };
    LongFft &lf = p->lf;
    lf.Lp = N / 2;
    if (lf.Lp <= 4096) { lf.A = 1; lf.B = lf.Lp; }   // one CTA per signal: data and full twiddle table in shared memory
    else {
        int lg = 0;
        while ((1ll << lg) < lf.Lp) ++lg;
        lf.B = std::min<int64_t>(1024, 1ll << ((lg + 1) / 2));
        lf.A = lf.Lp / lf.B;
    }
    lf.fft_B = plan_for(lf.B, kPlanPow2, 16);
    lf.fft_A = lf.A > 1 ? plan_for(lf.A, kPlanPow2, 16) : lf.fft_B;
    if (lf.A > 1) {
        // twiddles between the passes, W_Lp^{i (low + q NL)} = U[low][i] V[q][i] for element q of the last-stage butterfly whose
        // lowest frequency is low: both factors rounded once from their exact value
        std::vector<std::complex<double>> fine, coarse;   // W_Lp^y and W_Lp^{2048 y}
        for (int64_t y = 0; y < 2048; ++y) fine.push_back(std::polar(1.0, -2.0 * kPi * (double)y / (double)lf.Lp));
        for (int64_t y = 0; y < (lf.Lp + 2047) / 2048; ++y) coarse.push_back(std::polar(1.0, -2.0 * kPi * (double)(2048 * y) / (double)lf.Lp));
        auto outer = [&](int64_t rows, int64_t cols, int64_t scale) {   // [row][col] = W_Lp^{scale row col}
            const int off = (int)tw.size();
            for (int64_t r = 0; r < rows; ++r)
                for (int64_t c = 0; c < cols; ++c) {
                    const int64_t y = (scale * r * c) % lf.Lp;   // product of two double factors: 1e-16, rounded once
                    const std::complex<double> w = fine[(size_t)(y & 2047)] * coarse[(size_t)(y >> 11)];
                    tw.push_back(make_float2((float)w.real(), (float)w.imag()));
                }
            return off;
        };
        const int64_t nl_cols = lf.A / long_cols_last_radix(lf.A), nl_rows = lf.B / long_rows_inverse_last_radix(lf.B);
        lf.tw_fwd_u = outer(nl_cols, lf.B, 1);
        lf.tw_fwd_v = outer(lf.A / nl_cols, lf.B, nl_cols);
        lf.tw_inv_u = outer(nl_rows, lf.A, 1);
        lf.tw_inv_v = outer(lf.B / nl_rows, lf.A, nl_rows);
    }
    lf.tw_n = append_twiddles(tw, N, lf.log_n_c);
    lf.n_n = (int)tw.size() - lf.tw_n;
    lf.x_pitch = (lf.Lp + 1 + 7) / 8 * 8;

    // Plane of every band in the weighted-bin scratch: bands of one plane share no bin.  Range starts ascend, so the lowest
    // plane that is free never exceeds the largest cover, and bins that few bands cover use the lowest planes only.
    std::vector<int> plane_of(L.bands.size());
    std::vector<int32_t> cover(N / 2 + 1, 0);
    {
        std::vector<int64_t> end((size_t)p->y_planes, -1);
        for (size_t i = 0; i < L.bands.size(); ++i) {
            const HostBand &hb = L.bands[i];
            const int64_t s = hb.kc + hb.d0 + hb.j_lo - hb.zl, e = s + hb.zl + hb.n_in - 1 + hb.zr;
            int pl = (int)(i % (size_t)p->y_planes);
            if (cover_is_mask(*p)) {
                pl = 0;
                while (pl + 1 < p->y_planes && end[(size_t)pl] >= s) ++pl;
                end[(size_t)pl] = e;
                for (int64_t k = s; k <= e; ++k) cover[(size_t)k] |= 1 << pl;
            }
            plane_of[i] = pl;
        }
        if (!cover_is_mask(*p))
            for (int64_t k = 0; k <= N / 2; ++k) cover[(size_t)k] = ((L.cover_lo[k] % p->y_planes) << 8) | L.cover_n[k];
    }

    // ---- band records
    p->bands.resize(L.bands.size());
    for (size_t i = 0; i < L.bands.size(); ++i) {
        const HostBand &hb = L.bands[i];
        BandRec &br = p->bands[i];
        br.kc = (int32_t)hb.kc; br.d0 = (int32_t)hb.d0; br.S = (int32_t)hb.S; br.M = (int32_t)hb.M;
        br.tab_off = (int32_t)hb.tab_off; br.coeff_off = (int32_t)hb.coeff_off;
        br.y_off = (int32_t)((int64_t)plane_of[i] * p->y_plane);
        br.side = hb.side;
        br.fft = -1;
    }
    // ---- launch classes by band length
    // class 0: 8 lanes per item, 32 items per CTA, or a warp per item in a call with few items.
    // class 1: a warp per item, 8 items per CTA, in every call.  With a CTA of 64 threads per item the class was bound by the
    // rate at which CTAs start (17 % of the warps active): 256 signals at 24 bands per octave 57 -> 52 us, their whole
    // analysis 102 -> 95.  Most calls with few items take the merged form instead; those with a two-pass band do not, and
    // for them the two are alike: round trip of one 2^22-sample signal at 96 bands per octave 215.7 us, with 64 threads
    // per item 215.0, of one 2^20-sample signal at 48 111.9 and 119.7, of four 2^18-sample ones at 24 88.4 and 83.7.
    // The others: one CTA per item, sized so that several CTAs share an SM (64 registers per thread) except for the longest
    // bands, which fill its shared memory.
    const int limits[kNumClasses] = {128, 1024, 4096, 13500, 1 << 30};
    {
        const int threads[kNumClasses] = {256, 256, 256, 512, 1024};
        const int minb[kNumClasses] = {4, 4, 4, 2, 1};
        for (int c = 0; c < kNumClasses; ++c) {
            p->cls[c].threads = threads[c];
            p->cls[c].min_blocks = minb[c];
            p->cls[c].lanes_few = c <= 1 ? 32 : 0;
            p->cls[c].lanes_many = c == 0 ? 8 : (c == 1 ? 32 : 0);
            p->cls[c].max_radix = c <= 1 ? 8 : (c == 2 ? 12 : 16);
        }
    }
    std::vector<int> order(L.bands.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return L.bands[a].M > L.bands[b].M; });
    int64_t smem_cap_elems = (227 * 1024) / 8;
    // test hook: a smaller cap sends shorter bands through the two-pass (huge band) kernels
    if (tune.max_cta_elems >= 64 && tune.max_cta_elems < smem_cap_elems) smem_cap_elems = tune.max_cta_elems;
    // bands above this length take the two-pass kernels (small tiles, many CTAs per SM)
    const int64_t two_pass_min = tune.two_pass_min > 0 ? std::max<int64_t>(64, tune.two_pass_min) : (1ll << 40);
    // M = A * B with plannable factors: fewest stages, then the most balanced split; 0 if there is none
    const int tp_radix_cap = 16;
    auto split_two_pass = [&](int64_t M) -> int64_t {
        int64_t bestA = 0;
        int best_cost = 1 << 30;
        for (int64_t a = 2; a * a <= M; ++a) {
            if (M % a || M / a > 1600) continue;
            FftPlan t1, t2;
            std::vector<float2> scratch_tw;
            if (!make_fft_plan(a, false, scratch_tw, t1, false, tp_radix_cap) || t1.generic) continue;
            if (!make_fft_plan(M / a, false, scratch_tw, t2, false, tp_radix_cap) || t2.generic) continue;
            const int cost = t1.nstages + t2.nstages;
            if (cost <= best_cost) { best_cost = cost; bestA = a; }
        }
        return bestA;
    };
    // shared memory per item: padded buffer + two-level twiddle table (two buffers for a direct-sum stage)
    auto band_elems = [&](int32_t b) -> int64_t {
        const FftPlan &bf = p->ffts[(size_t)p->bands[(size_t)b].fft];
        return bf.generic ? 2 * (int64_t)bf.M + bf.st[0].radix : bf.M + 16 + bf.tw_count;
    };
    auto smooth = [](int64_t m) {
        for (int f : {2, 3, 5})
            while (m % f == 0) m /= f;
        return m == 1;
    };
    p->band_class.assign(L.bands.size(), -1);
    std::vector<int> chirp_bands[kChirpLengths];
    // plans whose bands of more than 128 coefficients are all powers of two (those beyond one CTA's shared memory apart)
    auto pow2_band = [&](int64_t M) { return pow2_length_index(M) >= 0 && M <= two_pass_min && M + M / 8 + 64 <= smem_cap_elems; };
    bool all_pow2 = true;
    for (const HostBand &hb : L.bands) all_pow2 = all_pow2 && (hb.M <= limits[0] || pow2_band(hb.M) || hb.M + 16 > smem_cap_elems);
    std::vector<int> pow2_bands[kPow2Lengths];
    for (int i : order) {
        const int64_t M = L.bands[i].M;
        int c = 0;
        while (M > limits[c]) ++c;
        bool single = M <= two_pass_min;
        int64_t A2 = 0;
        if (!single) { A2 = split_two_pass(M); single = A2 == 0; }
        p->band_class[(size_t)i] = (int8_t)c;
        if (c > 0 && all_pow2 && pow2_band(M)) {
            pow2_bands[pow2_length_index(M)].push_back(i);
            continue;
        }
        if (c > 0 && !smooth(M)) {
            const int li = M % 4 == 0 ? chirp_length_index(M / 4) : -1;
            if (li < 0) return CQT_ERR_UNSUPPORTED;
            chirp_bands[li].push_back(i);
            continue;
        }
        if (single) {
            // short bands: fewer registers, more CTAs per SM
            p->bands[i].fft = plan_for(M, kPlanBand, p->cls[c].max_radix);
            if (p->bands[i].fft < 0) return CQT_ERR_UNSUPPORTED;
            const int64_t elems = band_elems(i);
            if (elems > smem_cap_elems) {   // the cap is per work item; the classes with several items per CTA are far below it
                A2 = split_two_pass(M);
                if (!A2) return CQT_ERR_UNSUPPORTED;
                single = false;
            } else {
                p->cls[c].work.push_back(i);
                p->cls[c].max_elems = (int)std::max<int64_t>(p->cls[c].max_elems, elems);
                p->cls[c].n_bands++;
                if (p->ffts[p->bands[i].fft].generic) p->cls[c].has_generic = true;
            }
        }
        if (!single) {
            p->band_class[(size_t)i] = -1;
            TwoPassBand tb{};
            tb.band = i;
            tb.A = (int32_t)A2;
            tb.B = (int32_t)(M / A2);
            tb.fft_A = plan_for(tb.A, kPlanFull, tp_radix_cap);
            tb.fft_B = plan_for(tb.B, kPlanFull, tp_radix_cap);
            int lc = 0;
            tb.tw_m = append_twiddles(tw, M, lc);
            tb.log_m_c = lc;
            tb.n_m = (int32_t)tw.size() - tb.tw_m;
            tb.scratch_off = p->two_pass_pitch;
            p->two_pass_pitch += (M + 7) / 8 * 8;
            TwoPassGroup &g = p->two_pass[(tb.A <= 256 && tb.B <= 256) ? 0 : 1];
            g.bands.push_back(tb);
            for (int wi = 0; wi < 3; ++wi) {
                const int tw_tile = kTwoPassWidths[wi];
                g.max_tiles_cols[wi] = std::max(g.max_tiles_cols[wi], (tb.B + tw_tile - 1) / tw_tile);
                g.max_tiles_rows[wi] = std::max(g.max_tiles_rows[wi], (tb.A + tw_tile - 1) / tw_tile);
                g.smem_cols[wi] = std::max(g.smem_cols[wi], two_pass_smem_cols(tb, tw_tile));
                g.smem_rows[wi] = std::max(g.smem_rows[wi], two_pass_smem_rows(tb, tw_tile));
            }
        }
    }
    for (int li = 0; li < kPow2Lengths; ++li) {
        p->pow2.n_bands[li] = (int)pow2_bands[li].size();
        if (pow2_bands[li].empty()) continue;
        int r[5];
        pow2_radices(li, r);
        const int off = append_twiddle_rows(tw, L.bands[(size_t)pow2_bands[li][0]].M, r);
        for (int b : pow2_bands[li]) {
            Pow2Rec rec{};
            rec.br = p->bands[(size_t)b];
            rec.tw_off = off;
            p->pow2.recs.push_back(rec);
        }
    }
    // classes whose lengths all have a shape of their own: records by length, longest first, and the lengths' twiddle rows
    for (int c = 0; c < kNumClasses; ++c) {
        const std::vector<int32_t> &work = p->cls[c].work;
        if (c > 0 && !smooth_form(*p, true, c) && !smooth_form(*p, false, c)) continue;
        if (!std::all_of(work.begin(), work.end(), [&](int32_t b) { return smooth_info(L.bands[(size_t)b].M) != nullptr; })) continue;
        SmoothBands &sb = p->smooth[c];
        int off = 0;
        for (int32_t b : work) {
            const int64_t M = L.bands[(size_t)b].M;
            if (sb.lengths.empty() || sb.lengths.back().M != M) {
                const SmoothInfo &si = *smooth_info(M);
                off = append_twiddle_rows(tw, M, si.r);
                sb.lengths.push_back({(int)M, (int)sb.recs.size(), 0, si.per});
                sb.smem = std::max(sb.smem, sizeof(float2) * (size_t)(si.per * si.buf));
            }
            sb.lengths.back().n_bands++;
            SmoothRec rec{};
            rec.br = p->bands[(size_t)b];
            rec.tw_off = off;
            sb.recs.push_back(rec);
        }
    }
    // every length L that occurs: one full twiddle table; bands of equal length share their tables
    for (int li = 0; li < kChirpLengths; ++li) {
        p->chirp.n_bands[li] = (int)chirp_bands[li].size();
        std::map<int64_t, ChirpRec> of_length;
        for (int b : chirp_bands[li]) {
            const int64_t M = L.bands[(size_t)b].M;
            if (!of_length.count(M)) {
                ChirpRec cr{};
                const int f = plan_for(chirp_length(li), kPlanPow2, 16);
                make_chirp_tables(M / 4, chirp_length(li), tw, cr);
                cr.tw_full_off = p->ffts[(size_t)f].tw_full_off;
                of_length[M] = cr;
            }
            ChirpRec cr = of_length[M];
            cr.br = p->bands[(size_t)b];
            p->chirp.recs.push_back(cr);
        }
    }
    // a middle class whose longest band has at most one butterfly per thread at half the threads runs narrower CTAs
    if (p->cls[2].n_bands && L.bands[(size_t)p->cls[2].work[0]].M <= 2304) { p->cls[2].threads = 128; p->cls[2].min_blocks = 8; }
    // the same bands for the one-launch form: about one radix-8 butterfly per thread and stage, so that an item's chain
    // of dependent instructions is as short as its stages allow
    {
        MergedBands &mg = p->merged;
        auto lg_threads = [&](int32_t b) {
            const FftPlan &bf = p->ffts[(size_t)p->bands[(size_t)b].fft];
            int lg = 5;
            while (lg < 10 && (3ll << lg) < bf.M / 4) ++lg;   // 1.5 * threads < points / 8
            return lg;
        };
        for (int c = kNumClasses - 1; c >= 1; --c) mg.work.insert(mg.work.end(), p->cls[c].work.begin(), p->cls[c].work.end());
        std::stable_sort(mg.work.begin(), mg.work.end(), [&](int32_t x, int32_t y) { return lg_threads(x) > lg_threads(y); });
        for (size_t i = 0; i < mg.work.size(); ++i) {
            const int lg = lg_threads(mg.work[i]);
            if (mg.segs.empty() || mg.segs.back().lg_nthr != lg) mg.segs.push_back({(int)i, 0, lg, 0});
            mg.segs.back().n_bands++;
            mg.segs.back().elems = std::max(mg.segs.back().elems, (int)band_elems(mg.work[i]));
            if (lg < 10) continue;
            // the longest ones are split into four work items instead
            BandItem item;
            const int64_t M = p->bands[(size_t)mg.work[i]].M;
            item.br = p->bands[(size_t)mg.work[i]];
            item.fp = p->ffts[(size_t)plan_for(M / 4, kPlanBand, 16)];
            SplitRec sr{};
            int lc = 0;
            sr.tw_m = append_twiddles(tw, M, lc);
            sr.log_m_c = lc;
            sr.n_m = (int32_t)tw.size() - sr.tw_m;
            p->split.items.push_back(item);
            p->split.recs.push_back(sr);
            p->split.max_elems = std::max(p->split.max_elems, (int)(M / 4) + 16 + item.fp.tw_count + sr.n_m);
        }
    }
    // estimates for the per-call assignment of classes to streams (band.cu): total work, and the time one CTA
    // needs for the longest item (microseconds per element by class, from measured kernel times)
    {
        const double us_per_elem[kNumClasses] = {0.04, 0.015, 0.004, 0.0016, 0.0016};
        for (int c = 0; c < kNumClasses; ++c) {
            BandClass &bc = p->cls[c];
            int64_t longest = 0;
            for (int32_t b : bc.work) {
                const int64_t M = p->bands[(size_t)b].M;
                bc.stage_work += (double)M * (p->ffts[(size_t)p->bands[(size_t)b].fft].nstages + 1);
                longest = std::max(longest, M);
            }
            bc.latency_us = bc.n_bands ? 5.0 + us_per_elem[c] * (double)longest : 0.0;
        }
    }
    if (device < 0) { *out = p.release(); return CQT_OK; }

    // ---- device tables
    int cur = 0;
    if (cudaGetDevice(&cur) != cudaSuccess || cudaSetDevice(device) != cudaSuccess) return CQT_ERR_CUDA;
    const RestoreDevice restore{cur};
    p->device = device;   // from here on there may be something to free on it
    std::vector<float> tA(L.table_len), tS(L.table_len), tTA(L.table_len), tSA(L.table_len);
    for (size_t i = 0; i < L.bands.size(); ++i) {
        const HostBand &hb = L.bands[i];
        for (int64_t j = 0; j < hb.S; ++j) {
            const int64_t k = hb.kc + hb.d0 + j;
            const double g = L.g[hb.tab_off + j], h = L.h[hb.tab_off + j];
            const double wk = (k == 0 || k == N / 2) ? 1.0 : 2.0;
            tA[hb.tab_off + j] = (float)(g / (double)hb.M);
            tS[hb.tab_off + j] = (float)h;
            tTA[hb.tab_off + j] = (float)((double)N * g / (2.0 * (double)hb.M));
            tSA[hb.tab_off + j] = (float)(h * wk / (double)N);
        }
    }
    cudaError_t e = cudaSuccess;
    auto chk = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
    TableUpload up([&](const void *src, size_t n, void *&dev) {
        chk(cudaMalloc(&dev, n));
        if (e != cudaSuccess) return false;
        p->d.allocations.push_back(dev);
        chk(cudaMemcpy(dev, src, n, cudaMemcpyHostToDevice));
        return e == cudaSuccess;
    });
    up.add(p->d.bands, p->bands);
    up.add(p->d.ffts, p->ffts);
    up.add(p->d.tw, tw);
    up.add(p->d.tab_analysis, tA);
    up.add(p->d.tab_synthesis, tS);
    up.add(p->d.tab_analysis_adj, tTA);
    up.add(p->d.tab_synthesis_adj, tSA);
    up.add(p->d.cover, cover);
    // nested supports: the bins of a band's widened range outside its support hold zeros in the band's plane
    std::vector<int2> zero_seg;
    for (size_t i = 0; i < L.bands.size(); ++i) {
        const HostBand &hb = L.bands[i];
        const int64_t s = hb.kc + hb.d0, en = s + hb.S - 1;
        if (hb.zl > 0) zero_seg.push_back(make_int2((int)(p->bands[i].y_off + s - hb.zl), (int)hb.zl));
        if (hb.zr > 0) zero_seg.push_back(make_int2((int)(p->bands[i].y_off + en + 1), (int)hb.zr));
    }
    p->n_zero_seg = (int)zero_seg.size();
    up.add(p->d.zero_seg, zero_seg);
    up.add(p->d.dbg, std::vector<int>(8, 0));
    auto upload_items = [&](BandItem *&dst, const std::vector<int32_t> &work) {
        // record and radix plan of every band of the class, in launch order: what a work item fetches first
        std::vector<BandItem> items(work.size());
        for (size_t i = 0; i < items.size(); ++i) {
            const int b = work[i];
            items[i].br = p->bands[(size_t)b];
            items[i].fp = p->ffts[(size_t)p->bands[(size_t)b].fft];
        }
        up.add(dst, items);
    };
    for (auto &c : p->cls) upload_items(c.d_items, c.work);
    upload_items(p->merged.d_items, p->merged.work);
    up.add(p->chirp.d_recs, p->chirp.recs);
    up.add(p->pow2.d_recs, p->pow2.recs);
    for (auto &sb : p->smooth) up.add(sb.d_recs, sb.recs);
    up.add(p->split.d_items, p->split.items);
    up.add(p->split.d_recs, p->split.recs);
    for (auto &g : p->two_pass) up.add(g.d_recs, g.bands);
    up.finish();
    // a copy from pageable memory may return when the data is staged; the first call may come on a stream that does not wait
    // for the default one
    chk(cudaStreamSynchronize(nullptr));
    chk(cudaDeviceGetAttribute(&p->sm_count, cudaDevAttrMultiProcessorCount, p->device));
    chk(cudaDeviceGetAttribute(&p->max_smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, p->device));
    // the helper streams carry the shorter classes: at the highest priority their CTAs are placed ahead of the
    // long class on the caller's stream, whatever order the launches (or the nodes of a captured graph) arrive in
    int prio_least = 0, prio_greatest = 0;
    chk(cudaDeviceGetStreamPriorityRange(&prio_least, &prio_greatest));
    for (int i = 0; i < cqt_plan::kHelpers && e == cudaSuccess; ++i) {
        chk(cudaStreamCreateWithPriority(&p->aux[i], cudaStreamNonBlocking, prio_greatest));
        chk(cudaEventCreateWithFlags(&p->ev_join[i], cudaEventDisableTiming));
    }
    chk(cudaEventCreateWithFlags(&p->ev_fork, cudaEventDisableTiming));
    if (e == cudaSuccess) chk(configure_band_kernels(*p));
    if (e == cudaSuccess) chk(configure_chirp_kernels(*p));
    if (e == cudaSuccess) chk(configure_pow2_kernels(*p));
    if (e == cudaSuccess) chk(configure_smooth_kernels(*p));
    if (e == cudaSuccess) chk(configure_split_kernels(*p));
    if (e == cudaSuccess) chk(p->lf.A == 1 ? configure_short_fft_kernels(*p) : configure_long_forward_kernels(*p));
    if (e == cudaSuccess && p->lf.A > 1) chk(configure_long_inverse_kernels(*p));
    if (e == cudaSuccess) chk(configure_two_pass_kernels(*p));
    if (e != cudaSuccess) return CQT_ERR_CUDA;
    *out = p.release();
    return CQT_OK;
}

cqt_status cqt_plan_destroy(cqt_plan *p) {
    if (!p) return CQT_OK;
    free_device(p);
    delete p;
    return CQT_OK;
}

int64_t cqt_plan_num_bands(const cqt_plan *p) { return p ? (int64_t)p->lay.bands.size() : -1; }
int64_t cqt_plan_coeff_count(const cqt_plan *p) { return p ? p->lay.coeff_count : -1; }
int64_t cqt_plan_signal_length(const cqt_plan *p) { return p ? p->N : -1; }
int64_t cqt_plan_table_length(const cqt_plan *p) { return p ? p->lay.table_len : -1; }
int cqt_plan_device(const cqt_plan *p) { return p ? p->device : -1; }

cqt_status cqt_plan_band_info(const cqt_plan *p, int64_t band, cqt_band_info *out) {
    if (!p || !out || band < 0 || band >= (int64_t)p->lay.bands.size()) return CQT_ERR_INVALID_ARG;
    const HostBand &hb = p->lay.bands[band];
    out->centre_hz = hb.centre_hz; out->centre_bin = hb.kc; out->support = hb.S; out->first_offset = hb.d0;
    out->M = hb.M; out->coeff_offset = hb.coeff_off; out->table_offset = hb.tab_off; out->is_sideband = hb.side;
    out->launch_class = p->band_class[(size_t)band];   // -1: two-pass bands belong to no single-CTA class
    return CQT_OK;
}

size_t cqt_plan_workspace_bytes(const cqt_plan *p, int64_t batch) {
    if (!p || batch <= 0) return 0;
    const int64_t t = p->lf.A > 1 ? p->lf.Lp : 0;
    const int64_t per = t + std::max<int64_t>(p->lf.x_pitch, p->y_pitch) + p->two_pass_pitch;
    return (size_t)(256 + batch * per * (int64_t)sizeof(float2));
}

cqt_status cqt_plan_tables(const cqt_plan *p, const float **g_host, const float **h_host) {
    if (!p) return CQT_ERR_INVALID_ARG;
    if (g_host) *g_host = p->g32.data();
    if (h_host) *h_host = p->h32.data();
    return CQT_OK;
}

cqt_status cqt_plan_check(const cqt_plan *p) {
    if (!p) return CQT_ERR_INVALID_ARG;
    if (p->device < 0 || !p->d.dbg) return CQT_OK;
    int w[8];
    if (cudaMemcpy(w, p->d.dbg, sizeof(w), cudaMemcpyDeviceToHost) != cudaSuccess) return CQT_ERR_CUDA;
    if (w[0] == 0) return CQT_OK;
    std::fprintf(stderr, "cqt debug check: site %d index %lld limit %lld block (%d,%d) thread %d\n", w[0],
                 ((long long)w[2] << 32) | (unsigned)w[1], ((long long)w[4] << 32) | (unsigned)w[3], w[5], w[6], w[7]);
    return CQT_ERR_DEVICE_CHECK;
}

}  // extern "C"

namespace cqt {

void note_launch(const cqt_plan &p, const char *name, cudaStream_t st) {
    if (name) ++p.launches;
    if (!p.timing) return;
    if (p.ev_used == p.ev.size()) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) return;
        p.ev.push_back(e);
        p.ev_name.push_back(nullptr);
    }
    p.ev_name[p.ev_used] = name;
    cudaEventRecord(p.ev[p.ev_used], st);
    ++p.ev_used;
}

}  // namespace cqt

extern "C" {

int64_t cqt_plan_launch_count(const cqt_plan *p) { return p ? p->launches : -1; }

cqt_status cqt_plan_set_timing(const cqt_plan *p, int enable) {
    if (!p) return CQT_ERR_INVALID_ARG;
    p->timing = enable != 0;
    p->ev_used = 0;
    return CQT_OK;
}

cqt_status cqt_plan_read_timing(const cqt_plan *p, const char **names, float *ms, int64_t capacity, int64_t *count) {
    if (!p || !count || capacity < 0 || (capacity > 0 && (!names || !ms))) return CQT_ERR_INVALID_ARG;
    int64_t n = 0;
    for (size_t i = 1; i < p->ev_used; ++i) {
        if (!p->ev_name[i]) continue;   // start-of-call marker
        if (n < capacity) {
            if (cudaEventSynchronize(p->ev[i]) != cudaSuccess) return CQT_ERR_CUDA;
            if (cudaEventElapsedTime(&ms[n], p->ev[i - 1], p->ev[i]) != cudaSuccess) return CQT_ERR_CUDA;
            names[n] = p->ev_name[i];
        }
        ++n;
    }
    *count = n;
    p->ev_used = 0;
    return CQT_OK;
}

}  // extern "C"

namespace {

struct Call {
    const cqt_plan *p;
    float2 *T, *second, *huge;   // workspace regions
    cudaStream_t st;
    int prev_dev;
};

cqt_status begin_call(const cqt_plan *p, const void *sig, int64_t stride, int64_t batch, int64_t valid_len,
                      const void *coef, void *ws, size_t ws_bytes, void *stream, Call &c) {
    if (!p || !sig || !coef) return CQT_ERR_INVALID_ARG;
    if (batch <= 0 || batch > 65535 || valid_len <= 0 || valid_len > p->N || stride < valid_len) return CQT_ERR_INVALID_ARG;
    if (p->device < 0) return CQT_ERR_STATE;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255) || ws_bytes < cqt_plan_workspace_bytes(p, batch)) return CQT_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(coef) & 7) || (reinterpret_cast<uintptr_t>(sig) & 3)) return CQT_ERR_INVALID_ARG;
    c.p = p;
    c.T = reinterpret_cast<float2 *>(ws);
    c.second = c.T + (p->lf.A > 1 ? batch * p->lf.Lp : 0);
    c.huge = c.second + batch * std::max<int64_t>(p->lf.x_pitch, p->y_pitch);
    c.st = reinterpret_cast<cudaStream_t>(stream);
    if (cudaGetDevice(&c.prev_dev) != cudaSuccess) return CQT_ERR_CUDA;
    if (c.prev_dev != p->device && cudaSetDevice(p->device) != cudaSuccess) return CQT_ERR_CUDA;
    note_launch(*p, nullptr, c.st);
    return CQT_OK;
}

cqt_status end_call(const Call &c, cudaError_t e) {
    if (c.prev_dev != c.p->device) cudaSetDevice(c.prev_dev);
    return e == cudaSuccess ? CQT_OK : CQT_ERR_CUDA;
}

cqt_status run_analysis_form(const cqt_plan *p, const float *table, const float *x, int64_t x_stride, int64_t batch,
                             int64_t valid_len, cqt_c64 *c, void *ws, size_t ws_bytes, void *stream,
                             const cqt::SliceSource *src = nullptr, int row0 = 0, int rows = INT32_MAX) {
    Call k;
    cqt_status s = begin_call(p, x, x_stride, batch, valid_len, c, ws, ws_bytes, stream, k);
    if (s != CQT_OK) return s;
    cudaError_t e = launch_rfft_forward(*p, x, x_stride, batch, valid_len, k.T, k.second, k.st, src);
    if (e == cudaSuccess) e = launch_bands_from_spectrum(*p, table, k.second, CoefRows{reinterpret_cast<float2 *>(c), row0, rows}, k.huge, batch, k.st);
    return end_call(k, e);
}

cqt_status run_synthesis_form(const cqt_plan *p, const float *table, bool fold, const cqt_c64 *c, int64_t batch,
                              int64_t valid_len, float *x, int64_t x_stride, void *ws, size_t ws_bytes, void *stream, int row0 = 0, int rows = INT32_MAX) {
    Call k;
    cqt_status s = begin_call(p, x, x_stride, batch, valid_len, c, ws, ws_bytes, stream, k);
    if (s != CQT_OK) return s;
    cudaError_t e = launch_bands_to_spectrum(*p, table, fold, CoefRows{reinterpret_cast<float2 *>(const_cast<cqt_c64 *>(c)), row0, rows}, k.second, k.huge, batch, k.st);
    if (e == cudaSuccess) e = launch_rfft_inverse(*p, k.second, k.T, x, x_stride, batch, valid_len, k.st);
    return end_call(k, e);
}

}  // namespace

namespace cqt {

// The sliced form (slicq.cu): transforms whose coefficient rows lie in a ring of `rows` rows at c, the first at row0.
// src: the slice cut fused into the load of the long FFT's first pass; else the slices are the rows of x.
cqt_status analyse_slices(const cqt_plan *p, const SliceSource *src, const float *x, int64_t batch, cqt_c64 *c, int row0, int rows, void *ws,
                          size_t ws_bytes, void *stream) {
    if (!p || (src && (!src->ring || !src->win || !can_fuse_slice_cut(*p)))) return CQT_ERR_INVALID_ARG;
    return run_analysis_form(p, p->d.tab_analysis, src ? src->ring : x, p->N, batch, p->N, c, ws, ws_bytes, stream, src, row0, rows);
}
cqt_status synthesise_slices(const cqt_plan *p, const cqt_c64 *c, int row0, int rows, int64_t batch, float *x, void *ws, size_t ws_bytes,
                             void *stream) {
    if (!p) return CQT_ERR_INVALID_ARG;
    return run_synthesis_form(p, p->d.tab_synthesis, false, c, batch, p->N, x, p->N, ws, ws_bytes, stream, row0, rows);
}

}  // namespace cqt

extern "C" {

cqt_status cqt_analyse(const cqt_plan *p, const float *x, int64_t x_stride, int64_t batch, int64_t valid_len,
                       cqt_c64 *c, void *ws, size_t ws_bytes, void *stream) {
    return run_analysis_form(p, p ? p->d.tab_analysis : nullptr, x, x_stride, batch, valid_len, c, ws, ws_bytes, stream);
}

cqt_status cqt_synthesise(const cqt_plan *p, const cqt_c64 *c, int64_t batch, int64_t valid_len, float *x,
                          int64_t x_stride, void *ws, size_t ws_bytes, void *stream) {
    return run_synthesis_form(p, p ? p->d.tab_synthesis : nullptr, false, c, batch, valid_len, x, x_stride, ws, ws_bytes, stream);
}

cqt_status cqt_analyse_adjoint(const cqt_plan *p, const cqt_c64 *c_bar, int64_t batch, int64_t valid_len, float *x_bar,
                               int64_t x_stride, void *ws, size_t ws_bytes, void *stream) {
    return run_synthesis_form(p, p ? p->d.tab_analysis_adj : nullptr, true, c_bar, batch, valid_len, x_bar, x_stride, ws, ws_bytes, stream);
}

cqt_status cqt_synthesise_adjoint(const cqt_plan *p, const float *x_bar, int64_t x_stride, int64_t batch,
                                  int64_t valid_len, cqt_c64 *c_bar, void *ws, size_t ws_bytes, void *stream) {
    return run_analysis_form(p, p ? p->d.tab_synthesis_adj : nullptr, x_bar, x_stride, batch, valid_len, c_bar, ws, ws_bytes, stream);
}

}  // extern "C"
