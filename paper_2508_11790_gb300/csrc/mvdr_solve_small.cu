// Stand-alone solve, windows of up to 16 beams, without a preconditioner.
#include "mvdr_solve_small.cuh"

namespace bs {

bs_status launch_solve_small(const bs_plan *p, int W, const double2 *R, float2 *c, int32_t *info, cudaStream_t st,
                             const float *dpre, int refine, int f64, bool dependent) {
    return launch_solve_small_t<false>(p, W, R, c, info, st, dpre, refine, f64, dependent);
}

}  // namespace bs
