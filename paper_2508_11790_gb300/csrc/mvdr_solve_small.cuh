// Kernels of the stand-alone solve for windows of up to 16 beams, compiled
// without and with the diagonal preconditioner in translation units of their
// own (mvdr_solve_small.cu, mvdr_solve_precond.cu) so that they build in
// parallel.
#pragma once
#include "common.cuh"
#include "internal.h"
#include "solve_dev.cuh"

namespace bs {

// The pairs of one window size W <= 16, solved by a kernel compiled for
// that size alone: one kernel holding the bodies of all sixteen sizes
// behind a switch stalled mostly on instruction fetch.  GW = 8 lanes per
// pair for W <= 8 (sixteen pairs per CTA), else 16 (eight pairs per CTA).
// PRE: with a preconditioner.
template <int WT, bool PRE>
__global__ void __launch_bounds__(128, 4)
    mvdr_solve_w_kernel(const double2 *R, const int64_t *__restrict__ roff,
                        const int64_t *__restrict__ woff, const float2 *__restrict__ at32,
                        const float2 *__restrict__ atlo, const double2 *__restrict__ at64, float2 *__restrict__ c,
                        int32_t *__restrict__ info, int64_t slot0, int64_t slot1, double kappa_max, int refine,
                        int allow_f64, const int32_t *__restrict__ order, const float *__restrict__ dpre) {
    wait_for_predecessor();
    constexpr int GW = (WT <= 8) ? 8 : 16;
    constexpr int PPC = 128 / GW;
    __shared__ __align__(16) unsigned char scratch[PPC][solve_scratch_bytes<GW>];
    const int grp = threadIdx.x / GW;
    const int lane = threadIdx.x % GW;
    const unsigned mask = (GW == 8) ? (0xFFu << (threadIdx.x & 24)) : ((threadIdx.x & 16) ? 0xFFFF0000u : 0x0000FFFFu);
    const int64_t slot = slot0 + (int64_t)blockIdx.x * PPC + grp;
    if (slot >= slot1) return;   // uniform over the group
    const int64_t g = order ? (int64_t)order[slot] : slot;
    const int64_t wo = woff[g];
    solve_pair_core<WT, GW, PRE>(mask, lane, WT, R + roff[g], at32 + wo, atlo + wo, at64 + wo, c + wo, info + g,
                                 kappa_max, refine, allow_f64, scratch[grp], PRE ? dpre + wo : nullptr);
}

// The pairs of window size WT: slots wstart[WT] .. wstart[WT + 1] - 1 of
// the W-grouped order (the identity when every pair has that size).
template <int WT, bool PRE>
bs_status launch_solve_w(const bs_plan *p, const double2 *R, float2 *c, int32_t *info, cudaStream_t st,
                         const float *dpre, int refine, int f64, bool dependent) {
    constexpr int PPC = 128 / ((WT <= 8) ? 8 : 16);
    const int64_t s0 = p->wstart[WT], s1 = p->wstart[WT + 1];
    if (s1 <= s0) return BS_OK;
    const int32_t *order = p->Wmin == p->Wmax ? nullptr : p->d_order_w;
    const unsigned blocks = (unsigned)((s1 - s0 + PPC - 1) / PPC);
    launch_stage(dependent, mvdr_solve_w_kernel<WT, PRE>, blocks, 128, 0, st, R, p->d_roff, p->d_woff, p->d_at32,
                 p->d_atlo, p->d_at64, c, info, s0, s1, p->cfg.kappa_max, refine, f64, order, dpre);
    return check_launch("solve (one window size) launch");
}

// The pairs of window size W of the plan.
template <bool PRE>
bs_status launch_solve_small_t(const bs_plan *p, int W, const double2 *R, float2 *c, int32_t *info, cudaStream_t st,
                               const float *dpre, int refine, int f64, bool dependent) {
#define BS_SOLVE_W(n) \
    case n: return launch_solve_w<n, PRE>(p, R, c, info, st, dpre, refine, f64, dependent);
    switch (W) {
        BS_SOLVE_W(1) BS_SOLVE_W(2) BS_SOLVE_W(3) BS_SOLVE_W(4) BS_SOLVE_W(5) BS_SOLVE_W(6) BS_SOLVE_W(7) BS_SOLVE_W(8)
        BS_SOLVE_W(9) BS_SOLVE_W(10) BS_SOLVE_W(11) BS_SOLVE_W(12) BS_SOLVE_W(13) BS_SOLVE_W(14) BS_SOLVE_W(15)
        BS_SOLVE_W(16)
    }
#undef BS_SOLVE_W
    return set_error(BS_EUNSUPPORTED, "W > 16");
}

}  // namespace bs
