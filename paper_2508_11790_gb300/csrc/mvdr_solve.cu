// Stand-alone MVDR solve (Eq. BeamCorrMVDR) of every pair from its stored
// FP64 covariance: one launch per window size present, pairs visited in
// the plan's W-grouped order.  An 8-lane group solves a pair of W <= 8, a
// half-warp one of 8 < W <= 16 (mvdr_solve_small.cuh), a warp one of
// 16 < W <= 32 (mvdr_solve_wide.cu).  The solve
// itself (FP32 Cholesky, compensated refinement, FP64 escalation) is
// solve_pair_core() in solve_dev.cuh.
#include <math.h>

#include "common.cuh"
#include "internal.h"
#include "solve_dev.cuh"

namespace bs {

// Plain FP32 per-pair solve: one thread factorises and solves its pair in
// shared memory (no refinement, no FP64), c = v / |u|^2.
__global__ void plain_solve_kernel(const double2 *__restrict__ R, const int64_t *__restrict__ roff,
                                   const int32_t *__restrict__ Wg, const int64_t *__restrict__ woff,
                                   const float2 *__restrict__ at32, float2 *__restrict__ c,
                                   int32_t *__restrict__ info) {
    __shared__ float2 Lm[WMAX_WIDE][WMAX_WIDE];
    __shared__ float2 u[WMAX_WIDE], v[WMAX_WIDE];
    const int64_t g = blockIdx.x;
    const int W = Wg[g];
    const double2 *Rg = R + roff[g];
    for (int e = threadIdx.x; e < W * W; e += blockDim.x) {
        const double2 r = Rg[e];
        Lm[e / W][e % W] = make_float2((float)r.x, (float)r.y);
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    int fail = 0;
    for (int k = 0; k < W && !fail; ++k) {
        float d = Lm[k][k].x;
        for (int m = 0; m < k; ++m) d -= Lm[k][m].x * Lm[k][m].x + Lm[k][m].y * Lm[k][m].y;
        if (!(d > 0.f)) { fail = k + 1; break; }
        d = sqrtf(d);
        Lm[k][k] = make_float2(d, 0.f);
        for (int i = k + 1; i < W; ++i) {
            float2 s = Lm[i][k];
            for (int m = 0; m < k; ++m) s = csub(s, cmulc(Lm[i][m], Lm[k][m]));
            Lm[i][k] = cscale(s, 1.f / d);
        }
    }
    if (fail) {
        for (int i = 0; i < W; ++i) c[woff[g] + i] = make_float2(nanf(""), nanf(""));
        info[g] = fail;
        return;
    }
    float nu = 0.f;
    for (int i = 0; i < W; ++i) {
        float2 s = at32[woff[g] + i];
        for (int m = 0; m < i; ++m) s = csub(s, cmul(Lm[i][m], u[m]));
        u[i] = cscale(s, 1.f / Lm[i][i].x);
        nu += u[i].x * u[i].x + u[i].y * u[i].y;
    }
    for (int i = W - 1; i >= 0; --i) {
        float2 s = u[i];
        for (int m = i + 1; m < W; ++m) s = csub(s, conjmul(Lm[m][i], v[m]));
        v[i] = cscale(s, 1.f / Lm[i][i].x);
    }
    for (int i = 0; i < W; ++i) c[woff[g] + i] = cscale(v[i], 1.f / nu);
    info[g] = 0;
}

// Fork: the first nst - 1 side streams of the plan wait for `st`.
static bs_status fork_streams(const bs_plan *p, cudaStream_t st, int nst) {
    if (nst <= 1) return BS_OK;
    cudaError_t e = cudaEventRecord(p->ev_fork, st);
    for (int k = 0; k + 1 < nst && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(p->solve_st[k], p->ev_fork, 0);
    return e == cudaSuccess ? BS_OK : cuda_error(e, "solve fork");
}
// Join: `st` waits for everything issued to those side streams.
static bs_status join_streams(const bs_plan *p, cudaStream_t st, int nst) {
    cudaError_t e = cudaSuccess;
    for (int k = 0; k + 1 < nst && e == cudaSuccess; ++k) {
        e = cudaEventRecord(p->ev_join[k], p->solve_st[k]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(st, p->ev_join[k], 0);
    }
    return e == cudaSuccess ? BS_OK : cuda_error(e, "solve join");
}
static int window_classes(const bs_plan *p) {
    int n = 0;
    for (int w = 1; w <= 16; ++w) n += p->wstart[w + 1] > p->wstart[w];
    return n;
}
static int wide_classes(const bs_plan *p) {   // of four sizes each: 17..20, .., 29..32
    int n = 0;
    for (int w = 17; w <= 29; w += 4) n += p->wstart[w + 4] > p->wstart[w];
    return n;
}

bool mvdr_solve_is_one_launch(const bs_plan *p) {
    return (p->cfg.flags & BS_FLAG_PLAIN) || wide_classes(p) + window_classes(p) == 1;
}

bool cov_solve_chains_apply(const bs_plan *p) {
    return !(p->cfg.flags & BS_FLAG_PLAIN) && p->nsmall == p->pairs && window_classes(p) > 1 &&
           window_cov_uses_warp(p);
}

bs_status launch_cov_solve_chains(const bs_plan *p, const void *ztr, double2 *R, float2 *c, int32_t *info,
                                  cudaStream_t st) {
    const int refine = (p->cfg.flags & BS_FLAG_NO_REFINE) ? 0 : 1;
    const int f64 = (p->cfg.flags & BS_FLAG_NO_FP64) ? 0 : 1;
    const int ncls = window_classes(p);
    const int nst = ncls < 1 + bs_plan::kSolveStreams ? ncls : 1 + bs_plan::kSolveStreams;
    if (bs_status s = fork_streams(p, st, nst)) return s;
    int li = 0;
    // one chain per window size (covariance of its pairs, then their solve),
    // largest windows first, chain i on stream i mod nst
    for (int W = 16; W >= 1; --W) {
        if (p->wstart[W + 1] == p->wstart[W]) continue;
        const int k = li++ % nst;
        const cudaStream_t s_ = k == 0 ? st : p->solve_st[k - 1];
        if (bs_status s = launch_window_cov_warp(p, ztr, nullptr, R, s_, p->wstart[W], p->wstart[W + 1], p->d_order_w))
            return s;
        if (bs_status s = launch_solve_small(p, W, R, c, info, s_, nullptr, refine, f64)) return s;
    }
    return join_streams(p, st, nst);
}

bs_status launch_mvdr_solve(const bs_plan *p, const double2 *R, float2 *c, int32_t *info, cudaStream_t st,
                            const float *dpre, bool dependent) {
    const int64_t G = p->pairs;
    if (p->Wmax > WMAX_WIDE) return set_error(BS_EUNSUPPORTED, "W > 32");
    if (p->cfg.flags & BS_FLAG_PLAIN) {
        plain_solve_kernel<<<(unsigned)G, 32, 0, st>>>(R, p->d_roff, p->d_Wg, p->d_woff, p->d_at32, c, info);
        return check_launch("plain solve launch");
    }
    const int refine = (p->cfg.flags & BS_FLAG_NO_REFINE) ? 0 : 1;
    const int f64 = (p->cfg.flags & BS_FLAG_NO_FP64) ? 0 : 1;
    // windows of up to 16 beams: one launch per window size present, each of
    // a kernel compiled for that size alone (above 16: for four sizes).  The
    // launches are independent (disjoint pairs): with several, they are spread
    // over `st` and the plan's side streams (forked from `st` and joined back into it; under
    // graph capture, parallel branches), so that one launch's tail overlaps
    // the others' work.
    const int nlaunch = wide_classes(p) + window_classes(p);
    dependent = dependent && nlaunch == 1;
    const int nst = nlaunch < 1 + bs_plan::kSolveStreams ? nlaunch : 1 + bs_plan::kSolveStreams;
    if (bs_status s = fork_streams(p, st, nst)) return s;
    int li = 0;   // launches issued; launch i goes to stream i mod nst
    auto next_stream = [&]() -> cudaStream_t {
        const int k = li++ % (nst > 0 ? nst : 1);
        return k == 0 ? st : p->solve_st[k - 1];
    };
    // largest windows first: the longest launches start first on their streams
    for (int W = 32; W > 16; W -= 4)
        if (p->wstart[W + 1] > p->wstart[W - 3])
            if (bs_status s = launch_solve_wide(p, W, R, c, info, next_stream(), dpre, refine, f64)) return s;
    for (int W = 16; W >= 1; --W) {
        if (p->wstart[W + 1] == p->wstart[W]) continue;
        const cudaStream_t ws = next_stream();
        if (bs_status s = dpre ? launch_solve_small_precond(p, W, R, c, info, ws, dpre, refine, f64, dependent)
                               : launch_solve_small(p, W, R, c, info, ws, dpre, refine, f64, dependent))
            return s;
    }
    return join_streams(p, st, nst);   // `st` waits for every side stream's launches
}

}  // namespace bs
