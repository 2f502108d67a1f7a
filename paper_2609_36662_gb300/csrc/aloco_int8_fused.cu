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
    // instances that stage such blocks as windows then run.  With 9 to 12 bf16
    // workers those take 11-15 % longer over aligned blocks (other shapes up to
    // 9 %), so in long vectors few odd blocks go element by element instead, at two to
    // three times an aligned block's cost: from 8 turns of the grid (two CTAs
    // per SM) while they are at most a sixteenth.  Kernel us, windows and elements, 9
    // / 12 workers:
    //   turns   one odd block            1/32 odd                 1/14 odd
    //     2     46.7  53.3 / 56.7  65.9  45.8  52.9 / 57.0  66.2
    //     4     73.3  69.9 / 91.2  87.9  72.8  74.4 / 92.5  94.6
    //     8    121.5 109.5 / 159  141    122   118  / 159  153    123  125 / 159  161
    //    24    315   277   / 417  365    314   292  / 413  382    313  312 / 415  407
    const int64_t blocks = P.blk[P.n_parts];
    int64_t odd = 0;
    for (int p = 0; a.nvec > 0 && p < P.n_parts; ++p)
        if ((P.off[p] & (kPad - 1)) != 0) odd += P.blk[p + 1] - P.blk[p];
    const bool spare = dtype == ALOCO_BF16 && a.M >= 9 && a.M <= 12 &&
                       blocks >= (int64_t)16 * sm_count && odd * 16 <= blocks;
    if (odd > 0 && !spare)
        return launch_int8_fused_odd(a, P, dtype, sm_count, max_grid, stream, grid_out);
    return dtype == ALOCO_BF16
               ? fused_dispatch<true, false>(a, P, sm_count, max_grid, stream, grid_out)
               : fused_dispatch<false, false>(a, P, sm_count, max_grid, stream, grid_out);
}

}  // namespace aloco
