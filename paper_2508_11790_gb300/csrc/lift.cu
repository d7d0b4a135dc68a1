// Lifted correlator (Sec. III-C, Eq. AntennaEqCorr): c_hat_g = D^H S_g^T c_g,
// i.e. c_hat_g[n] = M^-1/2 sum_w c_g[w] e^{+j 2 pi m_w n / M} with
// m_w = start_g + w.  With z = e^{+j 2 pi n/M} this is
// M^-1/2 z^start (sum_w c_g[w] z^w), the sum by Horner's rule: two conjugated
// entries of the plan's M-point twiddle table per output (indices n and
// start n mod M) and no transcendental.  Its antenna-space output and its
// beam pattern are in lift_tc.cu.
//
// A CTA takes LIFT_PAIRS pairs; a thread four elements a block apart of each
// pair: z is read once, the four Horner chains share the weights' loads and
// loop, and run two to a packed FP32x2 FMA.  The scattered reads of z^start
// go to a copy of the twiddle table in shared memory, one spare slot per 16
// entries (steps of 16 and more would hit one bank): from L1 they touched
// about as many lines as lanes and alone took 25 us of the figures below.
// 8192 pairs of W = 9, N = 1024 (67 MB written): 47 us with one output per
// thread and the table in L1, 30 with two, 25 now.
#include "common.cuh"
#include "internal.h"

namespace bs {

constexpr int LIFT_PAIRS = 8;

__global__ void __launch_bounds__(256)
    lift_kernel(const float2 *__restrict__ c, const int64_t *__restrict__ woff, const int32_t *__restrict__ Wg,
                const int32_t *__restrict__ start, const float2 *__restrict__ twM, int M, int N, int64_t pairs,
                float scale, float2 *__restrict__ c_hat) {
    const int64_t g0 = (int64_t)blockIdx.x * LIFT_PAIRS;
    const int np = (int)min((int64_t)LIFT_PAIRS, pairs - g0);
    __shared__ float4 cw[LIFT_PAIRS][32];   // (re, re, im, im)
    __shared__ int Ws[LIFT_PAIRS], st[LIFT_PAIRS];
    for (int e = threadIdx.x; e < 32 * np; e += blockDim.x) {
        const int k = e >> 5, w = e & 31;
        const int W = Wg[g0 + k];
        if (w < W) {
            const float2 v = c[woff[g0 + k] + w];
            cw[k][w] = make_float4(v.x, v.x, v.y, v.y);
        }
        if (w == 0) Ws[k] = W, st[k] = start[g0 + k];
    }
    extern __shared__ float2 tw[];   // the M twiddles, padded
    for (int m = threadIdx.x; m < M; m += blockDim.x) tw[padrow(m)] = __ldg(&twM[m]);
    __syncthreads();
    const int nt = blockDim.x, n = blockIdx.y * 4 * nt + threadIdx.x;   // elements n + i nt
    if (n >= N) return;
    // z = e^{+j 2 pi n / M} of elements (n, n + nt) and (n + 2 nt, n + 3 nt)
    float2 zr[2], zi[2], nz[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float2 a = tw[padrow((n + 2 * h * nt) & (M - 1))], b = tw[padrow((n + (2 * h + 1) * nt) & (M - 1))];
        zr[h] = make_float2(a.x, b.x);
        zi[h] = make_float2(-a.y, -b.y);
        nz[h] = make_float2(a.y, b.y);
    }
    for (int k = 0; k < np; ++k) {
        const int W = Ws[k];
        const float4 top = cw[k][W - 1];
        float2 ar[2], ai[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            ar[h] = make_float2(top.x, top.y);
            ai[h] = make_float2(top.z, top.w);
        }
#pragma unroll 2
        for (int w = W - 2; w >= 0; --w) {
            const float4 b = cw[k][w];
            const float2 br = make_float2(b.x, b.y), bi = make_float2(b.z, b.w);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 re = __ffma2_rn(ar[h], zr[h], __ffma2_rn(ai[h], nz[h], br));
                ai[h] = __ffma2_rn(ar[h], zi[h], __ffma2_rn(ai[h], zr[h], bi));
                ar[h] = re;
            }
        }
        float2 *o = c_hat + (g0 + k) * N;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = n + i * nt;
            const float2 t = tw[padrow((st[k] * e) & (M - 1))];   // conjugate of z's start-th power
            const float2 a = (i & 1) ? make_float2(ar[i >> 1].y, ai[i >> 1].y) : make_float2(ar[i >> 1].x, ai[i >> 1].x);
            if (e < N) o[e] = cscale(cmulc(a, t), scale);
        }
    }
}

bs_status launch_lift(const bs_plan *p, const float2 *c, float2 *c_hat, cudaStream_t st) {
    const int N = p->cfg.N;
    if (p->pairs == 0) return BS_OK;
    if (p->Wmax > 32) return set_error(BS_EUNSUPPORTED, "W > 32");
    const int M = p->cfg.M;
    const int thr = N >= 1024 ? 256 : ((N + 3) / 4 + 31) & ~31;
    const dim3 grid((unsigned)((p->pairs + LIFT_PAIRS - 1) / LIFT_PAIRS), (N + 4 * thr - 1) / (4 * thr));
    lift_kernel<<<grid, thr, padded_len(M < 16 ? 16 : M) * sizeof(float2), st>>>(
        c, p->d_woff, p->d_Wg, p->d_start, p->d_twM, M, N, p->pairs, 1.0f / sqrtf((float)M), c_hat);
    return check_launch("lift launch");
}

}  // namespace bs
