// The kernel of one class of 5-smooth lengths, one direction and one kind of launch (band_smooth.cuh); compiled once for each, with
// CQT_CLASS, CQT_ANALYSIS and CQT_CHAINED from the command line.
#include "band_smooth.cuh"

namespace cqt {

#define CQT_CAT_(a, b) a##b
#define CQT_CAT(a, b) CQT_CAT_(a, b)
#define CQT_SHAPES CQT_CAT(CQT_SHAPES_, CQT_CLASS)

constexpr int kThreads = smooth_threads(CQT_CLASS);

static __global__ void __launch_bounds__(kThreads, 1024 / kThreads) smooth_bands_kernel(const __grid_constant__ SmoothArgs a) {
    chain_enter(a.b);
    const int seg = smooth_segment(a);
    chain_begin(a.b);   // records and tables belong to the plan; what follows touches the predecessor's output
    switch (a.seg[seg].shape) {
#define X(M, ...) case M: smooth_units<CQT_ANALYSIS != 0, CQT_CHAINED != 0, SmoothShape<M, __VA_ARGS__>>(a, seg); break;
        CQT_SHAPES(X)
#undef X
        default: break;
    }
    chain_end(a.b);
}

template <>
const void *SmoothKernel<CQT_ANALYSIS != 0, CQT_CLASS, CQT_CHAINED != 0>::get() { return (const void *)smooth_bands_kernel; }

}  // namespace cqt
