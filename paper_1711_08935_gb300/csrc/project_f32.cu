// Projection shapes of complex64 states.
#include "project_kernels.cuh"

namespace dftu {

// The shapes selectable with dftu_set_kernel_variant, listed once for the single-system and the batched
// launches: X(variant, policy, lanes per band Q, points per chain, band groups per CTA, L2 prefetch,
// minimum blocks per SM, threads per CTA, tile size).  Variant 0 is the default case of each switch.
// P_F32B2 has two bands per lane, P_F32B2F also each product's hi and lo halves folded into one sum, P_F32 one band
// per lane.  Tile size PTILE selects the projection's own tiling (single-system launches).
#define DFTU_PROJECT_SHAPES_F32(X) \
    X(1, P_F32B2F, 16, 8, 4, 0, 3, 256, PTILE) X(2, P_F32B2F, 8, 8, 4, 0, 3, 256, TILE) X(3, P_F32B2, 8, 8, 4, 0, 2, 256, TILE) \
    X(4, P_F32B2F, 16, 8, 4, 0, 2, 256, TILE) X(5, P_F32B2F, 16, 8, 8, 0, 3, 256, TILE) \
    X(6, P_F32B2F, 16, 6, 4, 0, 3, 256, TILE) X(7, P_F32, 8, 16, 8, 0, 2, 256, TILE)
#define DFTU_PROJECT_DEFAULT_F32 P_F32B2F, 16, 8, 4, 0, 3, 256, TILE

// The default shape, with fewer bands per CTA where the grid would not fill the GPU (balanced_groups): lanes and
// tiles stay, so the order of the FP32 sums does not depend on the size of the call and batched launches give
// the same bits (their tile reduce takes each member in the form that a single call of its size takes).
cudaError_t project_f32(const View& v, const ProjArgs& a, int variant, cudaStream_t st, View* used) {
#define DFTU_CASE(i, POL, Q, CH, NBG, PF, MB, NT, TP) case i: return run_project<POL, Q, CH, NBG, PF, MB, 0, 1, NT, TP>(v, a, st, used);
    switch (variant) {
        DFTU_PROJECT_SHAPES_F32(DFTU_CASE)
        default: return run_project_default<DFTU_PROJECT_DEFAULT_F32>(v, a, st, used);
    }
#undef DFTU_CASE
}

cudaError_t project_f32_batch(const BatchLaunch& b, int variant, cudaStream_t st) {
#define DFTU_CASE(i, POL, Q, CH, NBG, PF, MB, NT, TP) case i: return run_project_batch<POL, Q, CH, NBG, PF, MB, NT>(b, st);
    switch (variant) {
        DFTU_PROJECT_SHAPES_F32(DFTU_CASE)
        default: return run_project_batch_default<DFTU_PROJECT_DEFAULT_F32>(b, st);
    }
#undef DFTU_CASE
}

}  // namespace dftu
