// Beamspace transform and window gather (Eq. VerDFT, Eq. BeamTransform,
// Eq. OverallWindow, Eq. ApplyWindow).
//
// Every (record, bin) vector of N elements (contiguous in the channelised
// cube) is zero-padded to M points and transformed by an M-point Stockham
// FFT in shared memory; a CTA takes VPB consecutive vectors.  The windowed
// variant then writes, for every target, the W_t beams of its window
// (start_g + w mod M) straight from shared memory into the packed training
// or test window arrays; the full variant writes all M beams.  Decoding each
// (target, beam) entry once for all VPB vectors instead of once per output took
// 24 576 vectors of N = 256, M = 512 from 35 to 32 us and 16 384 of 100 targets
// of 11 beams from 64 to 44 us.
#include "beamspace_dev.cuh"
#include "internal.h"

namespace bs {

// kFull: write all M beams to out[v][m]; else gather windows (PREC = storage
// precision of the training windows).
template <int M, bool kFull, int PREC>
__global__ void __launch_bounds__(BsCfg<M>::nthr, BsCfg<M>::minb)
    beamspace_kernel(const float2 *y, int64_t nvec, int N, const float2 *__restrict__ tw,
                     float scale, float2 *__restrict__ out, GatherArgs ga, const int32_t *__restrict__ glist,
                     int sumW) {
    using RP = Radix<M>;
    constexpr int vpb = BsCfg<M>::vpb;
    constexpr int nthr = BsCfg<M>::nthr;
    constexpr int pl = BsCfg<M>::pl;
    extern __shared__ float2 sm[];
    // per-target gather entries of this CTA (uniform path), filled before the
    // FFT so that the table loads overlap the butterflies
    __shared__ long long tab_base[kTabT];
    __shared__ int tab_sw[kTabT];     // start | (W << 16)
    __shared__ int tab_n[kTabT];      // vectors of this CTA that the target's windows take (0: none)
    wait_for_predecessor();
    const int tid = threadIdx.x;
    const int64_t vid0 = (int64_t)blockIdx.x * vpb;
    int s_cta = 0, v0_cta = 0;
    bool train_cta = false;
    if constexpr (!kFull) {
        if (ga.uniform && vid0 < ga.nvec) {
            const int p = (int)((ga.vbase + vid0) >> ga.log2F);
            const int q = (int)((ga.vbase + vid0) & ((1 << ga.log2F) - 1));
            s_cta = q >> ga.log2B;
            const int i0 = q & ((1 << ga.log2B) - 1);
            train_cta = p < ga.P_train;
            v0_cta = train_cta ? (p << ga.log2B) + i0 : ((p - ga.P_train) << ga.log2B) + i0;
            const int nv = (ga.nvec - vid0 < (int64_t)vpb) ? (int)(ga.nvec - vid0) : vpb;
            for (int t = tid; t < ga.T && t < kTabT; t += nthr)
                fill_target_entry(ga, t, s_cta, v0_cta, nv, train_cta, tab_base, tab_sw, tab_n);
        }
    }

    auto gload = [&](int c, int n) -> float2 {
        const int64_t v = vid0 + c;
        if (n >= N || v >= nvec) return make_float2(0.f, 0.f);
        return __ldcs(&y[v * N + n]);
    };
    auto sload = [&](int c, int m) -> float2 { return sm[c * pl + padrow(m)]; };
    auto sstore = [&](int c, int m, float2 v) { sm[c * pl + padrow(m)] = v; };

    if constexpr (RP::npass == 1) {
        stockham_pass<M, RP::r0, 1, vpb, nthr, false, false>(tid, tw, gload, sstore);
    } else if constexpr (RP::npass == 2) {
        stockham_pass<M, RP::r0, 1, vpb, nthr, false, false>(tid, tw, gload, sstore);
        __syncthreads();
        stockham_pass<M, RP::r1, RP::r0, vpb, nthr, false, true>(tid, tw, sload, sstore);
    } else {
        stockham_pass<M, RP::r0, 1, vpb, nthr, false, false>(tid, tw, gload, sstore);
        __syncthreads();
        stockham_pass<M, RP::r1, RP::r0, vpb, nthr, false, true>(tid, tw, sload, sstore);
        __syncthreads();
        stockham_pass<M, RP::r2, RP::r0 * RP::r1, vpb, nthr, false, true>(tid, tw, sload, sstore);
    }
    __syncthreads();

    if constexpr (kFull) {
        for (int e = tid; e < vpb * M; e += nthr) {
            const int c = e / M, m = e % M;
            const int64_t v = vid0 + c;
            if (v < nvec) out[v * M + m] = cscale(sload(c, m), scale);
        }
    } else if (ga.uniform) {
        // All vpb vectors share record p and subband s (bins i0 .. i0+vpb-1):
        // a thread decodes a (target, beam w) entry once and stores it for
        // every vector (the vectors' rows of W_t are contiguous from the
        // target's base).
        if (vid0 >= ga.nvec) return;
        const int nv = (ga.nvec - vid0 < (int64_t)vpb) ? (int)(ga.nvec - vid0) : vpb;
        for (int e = tid; e < sumW; e += nthr) {
            const int packed = __ldg(&glist[e]);   // (t << 8) | w, target-major
            const int t = packed >> 8, w = packed & 255;
            long long base;
            int sw, n;
            if (t < kTabT) {
                base = tab_base[t];
                sw = tab_sw[t];
                n = tab_n[t];
            } else {
                fill_target_entry(ga, t, s_cta, v0_cta, nv, train_cta, &base, &sw, &n, 0);
            }
            const int W = sw >> 16;
            const float2 *src = sm + padrow(((sw & 0xFFFF) + w) & (M - 1));
            const long long o = base + w;
            if (train_cta) {
#pragma unroll 4
                for (int c = 0; c < n; ++c)
                    store_train<PREC>(ga.ztr, o + (long long)c * W, cscale(src[c * pl], scale), ga.store_scale);
            } else {
#pragma unroll 4
                for (int c = 0; c < n; ++c) ga.zte[o + (long long)c * W] = cscale(src[c * pl], scale);
            }
        }
    } else {
        const int Fm1 = (1 << ga.log2F) - 1, Bm1 = (1 << ga.log2B) - 1;
        for (int e = tid; e < ga.ngather; e += nthr) {
            const int packed = __ldg(&ga.gather[e]);
            const int t = packed >> 10, c = (packed >> 5) & 31, w = packed & 31;
            const int64_t g0 = (int64_t)t * ga.L;
            const int W = __ldg(&ga.Wg[g0]);
            const int64_t vid = vid0 + c;
            if (vid >= nvec) continue;
            const int p = (int)((ga.vbase + vid) >> ga.log2F);
            const int q = (int)((ga.vbase + vid) & Fm1);
            const int s = q >> ga.log2B, i = q & Bm1;
            const int64_t g = g0 + s;
            const int m = (__ldg(&ga.start[g]) + w) & (M - 1);
            const float2 val = cscale(sload(c, m), scale);
            if (p < ga.P_train) {
                const int vv = (p << ga.log2B) + i;
                if (vv < __ldg(&ga.Kg[g]))
                    store_train<PREC>(ga.ztr, __ldg(&ga.ztr_off[g]) + (int64_t)vv * W + w, val, ga.store_scale);
            } else {
                const int vv = ((p - ga.P_train) << ga.log2B) + i;
                ga.zte[__ldg(&ga.zte_off[g]) + (int64_t)vv * W + w] = val;
            }
        }
    }
}

// What the plan adds to GatherArgs for the one-shot kernel and its launch.
struct OneShotArgs {
    const int32_t *glist = nullptr;
    int sumW = 0, sms = 0;
    int64_t pred = 0;   // CTAs of the preceding stage (launch_beamspace)
};

template <int M, bool kFull, int PREC>
static bs_status launch_bs_t(const float2 *y, int64_t nvec, int N, const float2 *tw, float2 *out,
                             const GatherArgs &ga, const OneShotArgs &oa, cudaStream_t st) {
    using C = BsCfg<M>;
    static PerDevice attr;
    int per_sm = 0;
    if (bs_status s = attr.get(
            [](int *v) {
                const auto kernel = beamspace_kernel<M, kFull, PREC>;
                cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::smem);
                if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(v, kernel, C::nthr, C::smem);
                return cuda_error(e, "beamspace attribute");
            },
            &per_sm))
        return s;
    const int64_t blocks = (nvec + C::vpb - 1) / C::vpb;
    if (blocks > 0x7FFFFFFF) return set_error(BS_EUNSUPPORTED, "too many vectors");
    if (blocks == 0) return BS_OK;
    // M >= 1024: several waves gain nothing (N = 1500: 1.5 % slower)
    const bool dependent = oa.pred > 0 && (3 * oa.pred <= oa.sms || oa.pred + blocks <= oa.sms ||
                                           (M < 1024 && blocks >= 2LL * per_sm * oa.sms));
    launch_stage(dependent, beamspace_kernel<M, kFull, PREC>, (unsigned)blocks, C::nthr, C::smem, st, y, nvec, N, tw,
                 1.0f / sqrtf((float)M), out, ga, oa.glist, oa.sumW);
    return check_launch("beamspace launch");
}

template <bool kFull, int PREC>
static bs_status launch_bs(int M, const float2 *y, int64_t nvec, int N, const float2 *tw, float2 *out,
                           const GatherArgs &ga, const OneShotArgs &oa, cudaStream_t st) {
    switch (M) {
        case 16: return launch_bs_t<16, kFull, PREC>(y, nvec, N, tw, out, ga, oa, st);
        case 32: return launch_bs_t<32, kFull, PREC>(y, nvec, N, tw, out, ga, oa, st);
        case 64: return launch_bs_t<64, kFull, PREC>(y, nvec, N, tw, out, ga, oa, st);
        case 128: return launch_bs_t<128, kFull, PREC>(y, nvec, N, tw, out, ga, oa, st);
        case 256: return launch_bs_t<256, kFull, PREC>(y, nvec, N, tw, out, ga, oa, st);
        case 512: return launch_bs_t<512, kFull, PREC>(y, nvec, N, tw, out, ga, oa, st);
        case 1024: return launch_bs_t<1024, kFull, PREC>(y, nvec, N, tw, out, ga, oa, st);
        case 2048: return launch_bs_t<2048, kFull, PREC>(y, nvec, N, tw, out, ga, oa, st);
        case 4096: return launch_bs_t<4096, kFull, PREC>(y, nvec, N, tw, out, ga, oa, st);
    }
    return set_error(BS_EUNSUPPORTED, "M not supported");
}

static int ilog2(int v) {
    int r = 0;
    while ((1 << r) < v) ++r;
    return r;
}

bs_status launch_beamspace(const bs_plan *p, const float2 *xc, void *ztr, float2 *zte, cudaStream_t st, int p0,
                           int np, int64_t pred, int64_t *ctas) {
    if (np < 0) np = p->P - p0;
    GatherArgs ga;
    ga.nvec = (int64_t)np * p->Fs;   // Fs = Ls B bins per record (F without a shard)
    ga.vbase = (int64_t)p0 * p->Fs;
    xc += ga.vbase * p->cfg.N;   // the kernels index vectors of this range
    ga.log2F = ilog2(p->Fs);
    ga.log2B = ilog2(p->B);
    ga.L = p->Ls;
    ga.T = p->cfg.T;
    ga.P_train = p->cfg.P_train;
    ga.uniform = (p->B % p->vpb) == 0;
    ga.gather = p->d_gather;
    ga.gsub = reinterpret_cast<const longlong2 *>(p->d_gsub);
    ga.ngather = (int)p->gather.size();
    ga.Wg = p->d_Wg;
    ga.Kg = p->d_Kg;
    ga.start = p->d_start;
    ga.ztr_off = p->d_ztr_off;
    ga.zte_off = p->d_zte_off;
    ga.ztr = ztr;
    ga.zte = zte;
    ga.store_scale = p->cfg.store_scale;
    const OneShotArgs oa{p->d_glist, p->sumW, p->num_sms, pred};
    if (ctas) *ctas = p->num_sms;   // every kernel but the last fills the chip
    if (p->planar) return launch_beamspace2d(p, xc, ga, st);
    bool used = false;
    bs_status s = BS_OK;
    // -1: the first variant that applies, in the order tensor cores, warp per
    // transform, one-shot (0, 2 and 3 start the search there).  The
    // bulk-copy-staged kernel is slower than the one-shot kernel wherever both
    // apply and the first two do not (24 576 vectors of N = 256, M = 512, 16
    // targets: 45 against 32 us; 16 384 of N = 300, 100 targets: 148 against 44;
    // 6 144 of N = 1500, M = 2048: 48 against 39; N = 2000, M = 4096: 87 against
    // 76) and runs where it is asked for.
    const int v = p->tune_beamspace;
    if (v < 0 || v == 3) {
        s = launch_beamspace_tc(p, xc, ga, st, &used);
        if (s || used) return s;
    }
    if (v <= 0 || v == 3) {
        s = launch_beamspace_warp(p, xc, ga, st, &used);
        if (s || used) return s;
    }
    if (v == 1 || (v < 0 && (p->cfg.flags & BS_FLAG_STAGED_FFT))) {
        s = launch_beamspace_tma(p, xc, ga, st, &used);
        if (s || used) return s;
    }
    if (ctas) *ctas = (ga.nvec + p->vpb - 1) / p->vpb;
    switch (p->cfg.precision) {
        case BS_PREC_FP32: return launch_bs<false, BS_PREC_FP32>(p->cfg.M, xc, ga.nvec, p->cfg.N, p->d_twM, nullptr, ga, oa, st);
        case BS_PREC_FP16: return launch_bs<false, BS_PREC_FP16>(p->cfg.M, xc, ga.nvec, p->cfg.N, p->d_twM, nullptr, ga, oa, st);
        default: return launch_bs<false, BS_PREC_BF16>(p->cfg.M, xc, ga.nvec, p->cfg.N, p->d_twM, nullptr, ga, oa, st);
    }
}

bs_status launch_beamspace_full(const bs_plan *p, const float2 *y, int64_t nvec, float2 *yb,
                                cudaStream_t st) {
    GatherArgs ga{};
    return launch_bs<true, BS_PREC_FP32>(p->cfg.M, y, nvec, p->cfg.N, p->d_twM, yb, ga, OneShotArgs{}, st);
}

}  // namespace bs
