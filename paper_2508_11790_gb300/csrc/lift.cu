// Lifted correlator (Sec. III-C, Eq. AntennaEqCorr): c_hat_g = D^H S_g^T c_g,
// i.e. c_hat_g[n] = M^-1/2 sum_w c_g[w] e^{+j 2 pi m_w n / M} with
// m_w = start_g + w.  With z = e^{+j 2 pi n/M} this is
// M^-1/2 z^start (sum_w c_g[w] z^w), the sum by Horner's rule: two conjugated
// entries of the plan's M-point twiddle table per output (indices n and
// start n mod M) and no transcendental.  Its antenna-space output and its
// beam pattern are in lift_tc.cu, the beam pattern of few pairs is here.
//
// A CTA takes up to LIFT_PAIRS pairs; a thread four elements a block apart of each
// pair: z is read once, the four Horner chains share the weights' loads and
// loop, and run two to a packed FP32x2 FMA.  The scattered reads of z^start
// go to a copy of the twiddle table in shared memory, one spare slot per 16
// entries (steps of 16 and more would hit one bank): from L1 they touched
// about as many lines as lanes and alone took 25 us of the figures below.
// 8192 pairs of W = 9, N = 1024 (67 MB written): 47 us with one output per
// thread and the table in L1, 30 with two, 25 now.
#include "common.cuh"
#include "internal.h"

#include <algorithm>

namespace bs {

constexpr int LIFT_PAIRS = 8;

__global__ void __launch_bounds__(256)
    lift_kernel(const float2 *__restrict__ c, const int64_t *__restrict__ woff, const int32_t *__restrict__ Wg,
                const int32_t *__restrict__ start, const float2 *__restrict__ twM, int M, int N, int64_t pairs,
                int per, float scale, float2 *__restrict__ c_hat) {
    const int64_t g0 = (int64_t)blockIdx.x * per;
    const int np = (int)min((int64_t)per, pairs - g0);
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

// The same sums, bit for bit, one element of one pair per thread: no table to
// copy and no chain of pairs to go through, for work that does not fill the chip.
__global__ void __launch_bounds__(256)
    lift_few_kernel(const float2 *__restrict__ c, const int64_t *__restrict__ woff, const int32_t *__restrict__ Wg,
                    const int32_t *__restrict__ start, const float2 *__restrict__ twM, int M, int N, float scale,
                    float2 *__restrict__ c_hat) {
    __shared__ float2 cw[32];
    const int64_t g = blockIdx.x;
    const int n = blockIdx.y * blockDim.x + threadIdx.x;
    const int W = Wg[g];
    if (threadIdx.x < W) cw[threadIdx.x] = c[woff[g] + threadIdx.x];
    __syncthreads();
    if (n >= N) return;
    const float2 z = __ldg(&twM[n & (M - 1)]), t = __ldg(&twM[(start[g] * n) & (M - 1)]);
    const float zr = z.x, zi = -z.y, nz = z.y;
    float ar = cw[W - 1].x, ai = cw[W - 1].y;
    for (int w = W - 2; w >= 0; --w) {
        const float re = fmaf(ar, zr, fmaf(ai, nz, cw[w].x));
        ai = fmaf(ar, zi, fmaf(ai, zr, cw[w].y));
        ar = re;
    }
    c_hat[g * N + n] = cscale(cmulc(make_float2(ar, ai), t), scale);
}

// grid (pairs, ceil(n_dirs / per)), a CTA per pair and range of per directions,
// a warp per DPW directions.  The sum runs over 32 lanes' elements with one
// complex rotation per 32 elements.  The correlator is scaled by a power of
// two to a largest part of 1 to 2, so that its norm neither underflows nor
// overflows; the pattern does not depend on its scale.
// Bound by the rotations' FMAs and, for a pair's first directions, by loading
// the correlator and its norm: about 4.5 us + 7 ns a pair + (3.5 + N / 124) ns
// a pair and 32 directions.  96 pairs, 31 directions: 5 us at N = 48 and 6.5 at
// N = 1024, where the tensor-core tiles take 11 and 59; ranges of directions
// for few pairs: 181 directions of those in 10 and 16 us.
constexpr int PATTERN_STATIC = 32;   // its static shared memory

__global__ void __launch_bounds__(256)
    beam_pattern_kernel(const float2 *__restrict__ c_hat, const double *__restrict__ u, int n_dirs, int per, int N,
                        int L, int Ls, int s0, double fc, double fs, double fd, float *__restrict__ pattern) {
    extern __shared__ float2 ch[];   // [N] c_hat, then [per] Omega / pi as FP32 (hi, lo)
    float2 *omt = ch + N;
    __shared__ float part[PATTERN_STATIC / sizeof(float)];   // one per warp
    const int64_t g = blockIdx.x;
    const int s = s0 + (int)(g % Ls);   // subband of pair g among the L (plans of a shard: s0 + local)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d0 = blockIdx.y * per, nd = min(per, n_dirs - d0);
    float mx = 0.f;
    for (int n = threadIdx.x; n < N; n += 256) {
        const float2 v = c_hat[g * N + n];
        ch[n] = v;
        mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    if (lane == 0) part[warp] = mx;
    __syncthreads();
    for (int w = 0; w < 8; ++w) mx = fmaxf(mx, part[w]);
    __syncthreads();
    const float sc = (mx > 0.f && mx <= 3.4e38f) ? ldexpf(1.f, max(-126, min(126, -ilogbf(mx)))) : 1.f;
    float nrm = 0.f;
    for (int n = threadIdx.x; n < N; n += 256) {   // the elements this thread wrote
        const float2 v = cscale(ch[n], sc);
        ch[n] = v;
        nrm = fmaf(v.x, v.x, fmaf(v.y, v.y, nrm));
    }
    for (int o = 16; o; o >>= 1) nrm += __shfl_xor_sync(0xFFFFFFFFu, nrm, o);
    if (lane == 0) part[warp] = nrm;
    __syncthreads();
    float tot = 0.f;
    for (int w = 0; w < 8; ++w) tot += part[w];
    const float inv = 1.f / (sqrtf(tot) * sqrtf((float)N));
    // subband centre frequency (Eq. SubChannelFreq): fc + ((l - 1/2) / L) fs,
    // l = s - L/2 + 1, in this order; Omega / pi = u f / f_d per direction,
    // formed once per CTA in FP64 and kept as an FP32 (hi, lo) pair (the FP64
    // pipe is narrow, so the per-lane work below is FP32 only)
    const double f = fc + (((double)(s - L / 2 + 1) - 0.5) / (double)L) * fs;
    const double ratio = f / fd;
    for (int k = threadIdx.x; k < nd; k += 256) {
        const double om = u[d0 + k] * ratio;
        const float hi = (float)om;
        omt[k] = make_float2(hi, (float)(om - (double)hi));
    }
    __syncthreads();
    constexpr int DPW = 4;   // directions per warp pass: each shared load feeds four sums
    for (int k0 = warp * DPW; k0 < nd; k0 += 8 * DPW) {
        // Omega / pi = u f / fd; e^{j Omega n} with n = lane + 32 i.  The two
        // phases (in units of pi) are reduced to [-1, 1] in FP32 pairs before
        // sincospi, so their error does not grow with n.
        float er[DPW], ei[DPW], c32[DPW], s32[DPW], re[DPW], im[DPW];
#pragma unroll
        for (int d = 0; d < DPW; ++d) {
            const float2 om = (k0 + d < nd) ? omt[k0 + d] : make_float2(0.f, 0.f);
            // x0 = om * lane: exact product of the high part (fmaf), reduced
            // modulo 2 before the low-order terms are added
            const float p = om.x * (float)lane;
            const float e = fmaf(om.x, (float)lane, -p) + om.y * (float)lane;
            const float x0 = (p - 2.f * rintf(0.5f * p)) + e;
            const float q = om.x * 32.f;   // exact
            const float x32 = (q - 2.f * rintf(0.5f * q)) + om.y * 32.f;
            sincospif(x0, &ei[d], &er[d]);
            sincospif(x32, &s32[d], &c32[d]);
            re[d] = im[d] = 0.f;
        }
        for (int n = lane; n < N; n += 32) {
            const float2 a = ch[n];
#pragma unroll
            for (int d = 0; d < DPW; ++d) {   // conj(a) * e, then e *= e^{j 32 Omega}
                re[d] = fmaf(a.x, er[d], fmaf(a.y, ei[d], re[d]));
                im[d] = fmaf(a.x, ei[d], fmaf(-a.y, er[d], im[d]));
                const float nr = er[d] * c32[d] - ei[d] * s32[d];
                ei[d] = fmaf(er[d], s32[d], ei[d] * c32[d]);
                er[d] = nr;
            }
        }
#pragma unroll
        for (int d = 0; d < DPW; ++d) {
            for (int o = 16; o; o >>= 1) {
                re[d] += __shfl_xor_sync(0xFFFFFFFFu, re[d], o);
                im[d] += __shfl_xor_sync(0xFFFFFFFFu, im[d], o);
            }
            if (lane == 0 && k0 + d < nd)
                pattern[g * n_dirs + d0 + k0 + d] = sqrtf(re[d] * re[d] + im[d] * im[d]) * inv;
        }
    }
}

// c_hat^H y of short rows: a CTA takes 32 targets x 32 test vectors of one
// subband with 32-element slices of both in shared memory, FP32.
constexpr int AL_T = 32;   // targets per tile
constexpr int AL_V = 32;   // test vectors per tile
constexpr int AL_K = 32;   // elements per shared-memory slice

// grid (ceil(T/32), ceil(Vte/32), L); 256 threads as 16 x 16, 2 x 2 outputs each
__global__ void __launch_bounds__(256)
    apply_lifted_kernel(const float2 *__restrict__ xc, const float2 *__restrict__ c_hat, float2 *__restrict__ out,
                        int N, int F, int B, int L, int T, int P_train, int Vte) {
    __shared__ float2 Cs[AL_T][AL_K + 1];
    __shared__ float2 Ys[AL_V][AL_K + 1];
    const int s = blockIdx.z;
    const int t0 = blockIdx.x * AL_T, v0 = blockIdx.y * AL_V;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float2 acc[2][2];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) acc[a][b] = make_float2(0.f, 0.f);
    for (int k0 = 0; k0 < N; k0 += AL_K) {
        // stage: row r of each tile, lanes along the elements (coalesced)
        for (int e = threadIdx.x; e < AL_T * AL_K; e += 256) {
            const int r = e / AL_K, k = e % AL_K;
            const int t = t0 + r, v = v0 + r, n = k0 + k;
            float2 cv = make_float2(0.f, 0.f), yv = make_float2(0.f, 0.f);
            if (t < T && n < N) cv = __ldg(&c_hat[((int64_t)t * L + s) * N + n]);
            if (v < Vte && n < N) {
                const int p = P_train + v / B, q = s * B + v % B;
                yv = __ldcs(&xc[((int64_t)p * F + q) * N + n]);
            }
            Cs[r][k] = cv;
            Ys[r][k] = yv;
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < AL_K; ++k) {
            const float2 c0 = Cs[2 * ty][k], c1 = Cs[2 * ty + 1][k];
            const float2 y0 = Ys[2 * tx][k], y1 = Ys[2 * tx + 1][k];
            const float2 cc[2] = {c0, c1}, yy[2] = {y0, y1};
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b) {   // conj(c) * y
                    acc[a][b].x = fmaf(cc[a].x, yy[b].x, fmaf(cc[a].y, yy[b].y, acc[a][b].x));
                    acc[a][b].y = fmaf(cc[a].x, yy[b].y, fmaf(-cc[a].y, yy[b].x, acc[a][b].y));
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int t = t0 + 2 * ty + a, v = v0 + 2 * tx + b;
            if (t < T && v < Vte) out[((int64_t)t * L + s) * Vte + v] = acc[a][b];
        }
}

bs_status launch_lift(const bs_plan *p, const float2 *c, float2 *c_hat, cudaStream_t st) {
    const int N = p->cfg.N;
    if (p->pairs == 0) return BS_OK;
    if (p->Wmax > 32) return set_error(BS_EUNSUPPORTED, "W > 32");
    const int M = p->cfg.M;
    const float scale = 1.0f / sqrtf((float)M);
    // Few CTAs of one pair and 256 elements: an element per thread.  The other
    // kernel copies the M twiddles per CTA and takes its pairs one after the
    // other, so the line moves with M / N and, for short rows, with W.  1024
    // pairs of N = 100, M = 512, W = 9: 7.3 us with the table, 2.9 without;
    // N = 1024, M = 4096 7.8 and 7.4; 4096 pairs of N = 300, M = 512 8.5 and
    // 10.1; over 700 sizes within 0.3 % of the better one on average.  Both
    // give the same bits, so a shard may lie on the other side of it.
    const double blocks = (double)p->pairs * ((N + 255) / 256);
    const double line = N <= 64 ? std::max(4000.0, 1400.0 * p->Wmax)
                                : std::min(9000.0, 2000.0 + 800.0 * M / N + 1.2e6 / N);
    if (blocks <= line) {
        const int thr = std::min(256, (std::max(N, p->Wmax) + 31) & ~31);
        lift_few_kernel<<<dim3((unsigned)p->pairs, (N + thr - 1) / thr), thr, 0, st>>>(
            c, p->d_woff, p->d_Wg, p->d_start, p->d_twM, M, N, scale, c_hat);
        return check_launch("lift (few) launch");
    }
    const int thr = N >= 1024 ? 256 : ((N + 3) / 4 + 31) & ~31;
    const int ny = (N + 4 * thr - 1) / (4 * thr);
    // fewer pairs per CTA while that leaves the chip no more than a wave of
    // two CTAs per SM: the chains of a CTA's pairs follow one another
    const int wave = 2 * p->num_sms;
    const int per = (int)std::min<int64_t>(LIFT_PAIRS, (p->pairs * ny + wave - 1) / wave);
    const dim3 grid((unsigned)((p->pairs + per - 1) / per), ny);
    lift_kernel<<<grid, thr, padded_len(M < 16 ? 16 : M) * sizeof(float2), st>>>(
        c, p->d_woff, p->d_Wg, p->d_start, p->d_twM, M, N, p->pairs, per, scale, c_hat);
    return check_launch("lift launch");
}

bs_status launch_apply_lifted_simt(const bs_plan *p, const float2 *xc, const float2 *c_hat, float2 *out,
                                   cudaStream_t st) {
    const int T = p->cfg.T, L = p->Ls, Vte = p->Vte;   // the plan's subbands, Fs bins per record of xc
    dim3 grid((T + AL_T - 1) / AL_T, (Vte + AL_V - 1) / AL_V, L);
    apply_lifted_kernel<<<grid, 256, 0, st>>>(xc, c_hat, out, p->cfg.N, p->Fs, p->B, L, T, p->cfg.P_train, Vte);
    return check_launch("lifted outputs launch");
}

bs_status launch_beam_pattern_simt(const bs_plan *p, const float2 *c_hat, int n_dirs, const double *u,
                                   float *pattern, cudaStream_t st) {
    // 32 directions a CTA while that leaves at most four CTAs per SM, more
    // otherwise, as many as fit the 48 KB of an ordinary launch beside the
    // correlator (2016 at N = 4096)
    const int64_t parts = std::max<int64_t>(1, std::min<int64_t>((n_dirs + 31) / 32, 4 * p->num_sms / p->pairs));
    const int fit = ((48 * 1024 - PATTERN_STATIC) / (int)sizeof(float2) - p->cfg.N) & ~31;
    const int per = std::min(fit, (int)((n_dirs + parts - 1) / parts + 31) & ~31);
    const dim3 grid((unsigned)p->pairs, (n_dirs + per - 1) / per);
    beam_pattern_kernel<<<grid, 256, ((size_t)p->cfg.N + per) * sizeof(float2), st>>>(
        c_hat, u, n_dirs, per, p->cfg.N, p->cfg.L, p->Ls, p->s0, p->cfg.fc, p->cfg.fs, p->cfg.fd, pattern);
    return check_launch("beam pattern launch");
}

}  // namespace bs
