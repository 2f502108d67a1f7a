// The fused INT8 round, instances for vectors with tensor parts that start
// off a multiple of kPad elements.
#include "aloco_int8_fused.cuh"

namespace aloco {

cudaError_t launch_int8_fused_odd(const SyncArgs &a, const Int8Parts &P, aloco_dtype dtype,
                                  int sm_count, int max_grid, cudaStream_t stream,
                                  int *grid_out) {
    return dtype == ALOCO_BF16
               ? fused_dispatch<true, true>(a, P, sm_count, max_grid, stream, grid_out)
               : fused_dispatch<false, true>(a, P, sm_count, max_grid, stream, grid_out);
}

}  // namespace aloco
