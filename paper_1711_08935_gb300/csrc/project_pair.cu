// Projection shapes of complex128 states in FP32-pair arithmetic.
#include "project_kernels.cuh"

namespace dftu {

// The shapes selectable with dftu_set_kernel_variant: X as for the complex64 shapes (project_f32.cu).  L2 prefetch: 1 =
// the next chain, 5 = also the next band's first chain.  Tile size PTILE selects the projection's own tiling
// (single-system launches; batched launches use TILE, on which variant 1 is the default shape).
#define DFTU_PROJECT_SHAPES_PAIR(X) \
    X(1, P_PAIR, 8, 8, 8, 5, 2, 256, TILE) X(2, P_PAIR, 8, 8, 4, 5, 2, 256, PTILE) X(3, P_PAIR, 8, 8, 16, 5, 2, 256, PTILE) \
    X(4, P_PAIR, 16, 8, 16, 5, 2, 256, PTILE) X(5, P_PAIR, 8, 8, 8, 1, 2, 256, PTILE) X(6, P_PAIR, 8, 8, 4, 5, 2, 256, TILE) \
    X(7, P_PAIR, 8, 6, 8, 5, 2, 256, PTILE)
#define DFTU_PROJECT_DEFAULT_PAIR P_PAIR, 8, 8, 8, 5, 2, 256, PTILE

// The default shape, with fewer bands per CTA where the grid would not fill the GPU (balanced_groups).  Calls so
// small that single groups on the 1024-point tiles do not fill the GPU are one chain of latencies per CTA: they
// run on the 512-point tiles, and with 16 lanes per band while those too leave SMs idle.
// Isolated d shell, 21 bands (10 CTAs -> 40): 30.3 -> 14.8 us; small oxide cell, 23 bands in 4 (k, spin) (204 CTAs ->
// 368): 46.9 -> 40.4.
static cudaError_t project_pair_default(const View& v, const ProjArgs& a, cudaStream_t st, View* used) {
    const int64_t sms = sm_count(), rows = (int64_t)v.nk * v.ns, groups = (a.nbands + 31) / 32;
    if (v.nptiles * groups * rows >= 2 * sms) return run_project_default<DFTU_PROJECT_DEFAULT_PAIR>(v, a, st, used);
    if (v.ntiles * groups * rows >= sms) return run_project<P_PAIR, 8, 8, 1, 1, 2, 0, 1, 256, TILE, false, true>(v, a, st, used);
    return run_project<P_PAIR, 16, 8, 1, 1, 2, 0, 1, 256, TILE>(v, a, st, used);
}

cudaError_t project_pair(const View& v, const ProjArgs& a, int variant, cudaStream_t st, View* used) {
#define DFTU_CASE(i, POL, Q, CH, NBG, PF, MB, NT, TP) case i: return run_project<POL, Q, CH, NBG, PF, MB, 0, 1, NT, TP>(v, a, st, used);
    switch (variant) {
        DFTU_PROJECT_SHAPES_PAIR(DFTU_CASE)
        default: return project_pair_default(v, a, st, used);
    }
#undef DFTU_CASE
}

cudaError_t project_pair_batch(const BatchLaunch& b, int variant, cudaStream_t st) {
#define DFTU_CASE(i, POL, Q, CH, NBG, PF, MB, NT, TP) case i: return run_project_batch<POL, Q, CH, NBG, PF, MB, NT>(b, st);
    switch (variant) {
        DFTU_PROJECT_SHAPES_PAIR(DFTU_CASE)
        default: return run_project_batch_default<DFTU_PROJECT_DEFAULT_PAIR>(b, st);
    }
#undef DFTU_CASE
}

}  // namespace dftu
