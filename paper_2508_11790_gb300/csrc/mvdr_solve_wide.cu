// Stand-alone solve of windows of 17 to 32 beams.
#include "common.cuh"
#include "internal.h"
#include "solve_dev.cuh"

#include <algorithm>

namespace bs {

// Windows of 17..32 beams: one warp per pair, solved at WT = 20, 24, 28 or 32
// (padded, see solve_pair_core), one launch per size class present.  Bound by
// latency: the warp's Cholesky is a chain of shuffles and FMAs, so what counts
// is the number of warps an SM holds.  A copy of the padded matrix and an
// FP64 scratch in shared memory (35 KB per warp) held it at four: 2560 pairs
// of W = 32 took 371 us.  The matrix is read in place and the FP64 factor
// packed (8 KB): sixteen warps, 118 us, of which fetching the 11 600
// straight-line instructions of a solve was the largest stall.  Now the twenty
// warps that an SM holds at 96 registers are one CTA in lockstep: 92 us, one
// wave (sixteen in lockstep: 134 us, two waves).  Fewer pairs than that are
// spread evenly over the SMs, so that they share an SM's issue with fewer others
// (256 pairs of W = 32 53 -> 42 us, with a preconditioner 62 -> 45, 2560 pairs 54
// -> 51).
constexpr int WIDE_WARPS = 20;   // of a CTA, at most

template <int WT, bool PRE>
__global__ void __launch_bounds__(WIDE_WARPS * 32, 1)
    mvdr_solve_wide_kernel(const double2 *__restrict__ R, const int64_t *__restrict__ roff,
                           const int32_t *__restrict__ Wg, const int64_t *__restrict__ woff,
                           const float2 *__restrict__ at32, const float2 *__restrict__ atlo,
                           const double2 *__restrict__ at64, float2 *__restrict__ c, int32_t *__restrict__ info,
                           int64_t slot0, int64_t slot1, double kappa_max, int refine, int allow_f64,
                           const int32_t *__restrict__ order, const float *__restrict__ dpre) {
    extern __shared__ __align__(16) unsigned char scratch[];   // solve_scratch_bytes<32> per warp
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t at = slot0 + (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    const int64_t slot = at < slot1 ? at : slot1 - 1;
    const int64_t g = order ? (int64_t)order[slot] : slot;
    const int64_t wo = woff[g];
    solve_pair_core<WT, 32, PRE, true>(0xFFFFFFFFu, lane, Wg[g], R + roff[g], at32 + wo, atlo + wo, at64 + wo, c + wo,
                                       info + g, kappa_max, refine, allow_f64,
                                       scratch + warp * solve_scratch_bytes<32>, PRE ? dpre + wo : nullptr, at < slot1);
}

// The pairs of window sizes WT - 3 .. WT.
template <int WT>
static bs_status launch_wide_t(const bs_plan *p, const double2 *R, float2 *c, int32_t *info, cudaStream_t st,
                            const float *dpre, int refine, int f64) {
    const int64_t s0 = p->wstart[WT - 3], s1 = p->wstart[WT + 1];
    const int32_t *order = p->Wmin == p->Wmax ? nullptr : p->d_order_w;
    const int warps = (int)std::min<int64_t>(WIDE_WARPS, (s1 - s0 + p->num_sms - 1) / p->num_sms);
    const unsigned blocks = (unsigned)((s1 - s0 + warps - 1) / warps);
    constexpr int smem = WIDE_WARPS * solve_scratch_bytes<32>;
    static PerDevice attr;
    if (bs_status s = attr.get([](int *) {
            cudaError_t e = cudaFuncSetAttribute(mvdr_solve_wide_kernel<WT, true>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(mvdr_solve_wide_kernel<WT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         smem);
            return cuda_error(e, "solve (wide) attribute");
        }))
        return s;
    const auto kernel = dpre ? mvdr_solve_wide_kernel<WT, true> : mvdr_solve_wide_kernel<WT, false>;
    kernel<<<blocks, warps * 32, warps * solve_scratch_bytes<32>, st>>>(R, p->d_roff, p->d_Wg, p->d_woff, p->d_at32, p->d_atlo, p->d_at64, c,
                                               info, s0, s1, p->cfg.kappa_max, refine, f64, order, dpre);
    return check_launch("solve (wide) launch");
}

bs_status launch_solve_wide(const bs_plan *p, int W, const double2 *R, float2 *c, int32_t *info, cudaStream_t st,
                            const float *dpre, int refine, int f64) {
    switch (W) {
        case 20: return launch_wide_t<20>(p, R, c, info, st, dpre, refine, f64);
        case 24: return launch_wide_t<24>(p, R, c, info, st, dpre, refine, f64);
        case 28: return launch_wide_t<28>(p, R, c, info, st, dpre, refine, f64);
        default: return launch_wide_t<32>(p, R, c, info, st, dpre, refine, f64);
    }
}

}  // namespace bs
