// The fused INT8 round, instances for tensor parts that all start at a
// multiple of kPad elements, and the choice between the two sets.
#include "aloco_int8_fused.cuh"

namespace aloco {

bool int8_fused_fits(int M, aloco_dtype dtype) {
    (void)dtype;
    return M >= 1 && M <= kFusedMax;
}

cudaError_t launch_int8_fused(const SyncArgs &a, const Int8Parts &P, aloco_dtype dtype,
                              int sm_count, int max_grid, cudaStream_t stream,
                              int *grid_out) {
    if (!int8_fused_fits(a.M, dtype)) return cudaErrorInvalidValue;
    // A part that starts off a multiple of kPad (from the vector's first
    // aligned element) puts all its blocks off 16-byte boundaries; the
    // instances that stage such blocks as windows then run.
    bool odd = false;
    for (int p = 0; a.nvec > 0 && p < P.n_parts; ++p)
        odd = odd || (P.off[p] & (kPad - 1)) != 0;
    if (odd) return launch_int8_fused_odd(a, P, dtype, sm_count, max_grid, stream, grid_out);
    return dtype == ALOCO_BF16
               ? fused_dispatch<true, false>(a, P, sm_count, max_grid, stream, grid_out)
               : fused_dispatch<false, false>(a, P, sm_count, max_grid, stream, grid_out);
}

}  // namespace aloco
