// Beamformer output (Sec. II-B, applied per pair to the windowed test
// vectors): out[g][v'] = c_g^H z_test[g][v'] = sum_w conj(c_g[w]) z[v'][w].
//
// One thread per output.  The windows of a warp's 32 consecutive outputs
// are one contiguous span of the test-window array (pair-major, then
// vector, then beam), so the warp first copies that span to shared memory
// with coalesced loads and each thread then reads its W_g entries there
// (per-thread loads of 8 W contiguous bytes would touch 32 sectors per
// instruction).  Memory bound (8 W + 8 bytes per output).
#include "common.cuh"
#include "internal.h"

#include <algorithm>

namespace bs {

// WM: the largest window (16, or 32 with half as many warps per CTA), so a
// warp's span of 32 outputs x W_g entries fits its shared-memory buffer.
template <int WM>
struct ApplyCfg {
    static constexpr int threads = WM <= 16 ? 256 : 128;
    static constexpr int span = 32 * WM;   // float2 per warp
};

template <int WM>
__global__ void __launch_bounds__(ApplyCfg<WM>::threads)
    apply_kernel(const float2 *z, const int64_t *__restrict__ zte_off,
                 const int32_t *__restrict__ Wg, const int64_t *__restrict__ woff,
                 const float2 *c, float2 *__restrict__ out, int64_t total, int Vte) {
    __shared__ float2 span[ApplyCfg<WM>::threads / 32][ApplyCfg<WM>::span];
    wait_for_predecessor();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t idx0 = (int64_t)blockIdx.x * blockDim.x + warp * 32;
    if (idx0 >= total) return;   // uniform per warp
    const int64_t idx = idx0 + lane;
    const bool valid = idx < total;
    const int64_t gi = valid ? idx : total - 1;   // invalid lanes repeat the last output's window
    const int64_t g = gi / Vte;
    const int v = (int)(gi - g * Vte);
    const int W = __ldg(&Wg[g]);
    const int64_t start = __ldg(&zte_off[g]) + (int64_t)v * W;
    const int64_t s0 = __shfl_sync(0xFFFFFFFFu, start, 0);
    const int64_t e31 = __shfl_sync(0xFFFFFFFFu, start + W, 31);
    const int n = (int)(e31 - s0);   // <= 32 * WM
    float2 *buf = span[warp];
    for (int e = lane; e < n; e += 32) buf[e] = __ldcs(&z[s0 + e]);
    __syncwarp();
    const float2 *zv = buf + (start - s0);
    const float2 *cg = c + __ldg(&woff[g]);
    float re = 0.f, im = 0.f;
    for (int w = 0; w < W; ++w) {
        const float2 a = zv[w];
        const float2 b = cg[w];
        // conj(b) * a
        re = fmaf(b.x, a.x, fmaf(b.y, a.y, re));
        im = fmaf(b.x, a.y, fmaf(-b.y, a.x, im));
    }
    if (valid) out[idx] = make_float2(re, im);
}

// Whole blocks of 32 test vectors (Vte a multiple of 32): a warp takes up to
// `bpw` consecutive blocks of one pair, so that the pair's fields and weights
// are read once, without the 64-bit division and per-lane offsets above, the
// spans start on 16 bytes and the next block's loads are in flight during a
// block's sums.  Figures at the launcher.
template <int WM>
__global__ void __launch_bounds__(ApplyCfg<WM>::threads)
    apply_blocks_kernel(const float2 *z, const int64_t *__restrict__ zte_off,
                        const int32_t *__restrict__ Wg, const int64_t *__restrict__ woff,
                        const float2 *c, float2 *__restrict__ out, unsigned units, unsigned upp, int nb,
                        int bpw) {
    constexpr int NW = ApplyCfg<WM>::threads / 32, NR = WM / 2;   // 16-byte loads per lane: 16 W per block
    __shared__ __align__(16) float2 span[NW][ApplyCfg<WM>::span];
    __shared__ float2 cw[NW][WM];
    wait_for_predecessor();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned unit = blockIdx.x * NW + warp;   // upp units per pair
    if (unit >= units) return;   // uniform per warp
    const unsigned g = unit / upp;
    const int b0 = (int)(unit - g * upp) * bpw, b1 = min(nb, b0 + bpw);
    const int W = __ldg(&Wg[g]);
    if (lane < W) cw[warp][lane] = c[__ldg(&woff[g]) + lane];
    const float4 *src = reinterpret_cast<const float4 *>(z + __ldg(&zte_off[g]) + (int64_t)b0 * 32 * W);
    float2 *buf = span[warp];
    float4 r[NR];
    auto fetch = [&]() {
#pragma unroll
        for (int k = 0; k < NR; ++k)
            if (lane + 32 * k < 16 * W) r[k] = __ldcs(src + lane + 32 * k);
    };
    fetch();
    float2 *o = out + (int64_t)g * nb * 32 + lane;
    for (int b = b0; b < b1; ++b) {
        __syncwarp();
#pragma unroll
        for (int k = 0; k < NR; ++k)
            if (lane + 32 * k < 16 * W) reinterpret_cast<float4 *>(buf)[lane + 32 * k] = r[k];
        src += 16 * W;
        if (b + 1 < b1) fetch();
        __syncwarp();
        const float2 *zv = buf + lane * W;
        float re = 0.f, im = 0.f;
        for (int w = 0; w < W; ++w) {
            const float2 a = zv[w], q = cw[warp][w];
            // conj(q) * a
            re = fmaf(q.x, a.x, fmaf(q.y, a.y, re));
            im = fmaf(q.x, a.y, fmaf(-q.y, a.x, im));
        }
        o[b * 32] = make_float2(re, im);
    }
}

// Blocks of one pair that a warp takes: several only where the pairs alone fill
// the GPU (64 warps an SM).
static int blocks_per_warp(const bs_plan *p) {
    return p->pairs >= 32LL * p->num_sms ? std::min(4, p->Vte / 32) : 1;
}

// Whole blocks pay where a warp takes several, or where latency counts (up to
// 20 warps an SM in all: 64 pairs of W = 9, 128 vectors 2.5 us against 3.0).
// Between, with a block per warp, they are 5 to 40 % slower than an output per
// thread for small windows (2560 pairs of W = 2, 256 vectors 8.7 us against 6.3,
// 32 768 pairs of one block 12.4 against 8.7), and windows of a multiple of 8
// beams, whose reads of shared memory conflict, need more pairs (W = 32, 5120
// pairs, 96 vectors 39 us against 36).  Both kernels give the same bits.  Over
// 660 sizes within 1 % of the better one on average.
static bool apply_by_blocks(const bs_plan *p) {
    if (blocks_per_warp(p) > 1) return p->Wmax < 16 || p->Wmax % 8 != 0 || p->pairs >= 96LL * p->num_sms;
    return p->pairs * (p->Vte / 32) <= 20LL * p->num_sms;
}

template <int WM>
static bs_status launch_apply_blocks(const bs_plan *p, const float2 *z, const float2 *c, float2 *out, cudaStream_t st,
                                     bool dependent) {
    constexpr int NW = ApplyCfg<WM>::threads / 32;
    const int nb = p->Vte / 32, bpw = blocks_per_warp(p);
    const unsigned upp = (unsigned)((nb + bpw - 1) / bpw);
    const unsigned units = (unsigned)p->pairs * upp;
    launch_stage(dependent, apply_blocks_kernel<WM>, (units + NW - 1) / NW, ApplyCfg<WM>::threads, 0, st, z, p->d_zte_off,
                 p->d_Wg, p->d_woff, c, out, units, upp, nb, bpw);
    return check_launch("apply launch");
}

bs_status launch_apply(const bs_plan *p, const float2 *zte, const float2 *c, float2 *out, cudaStream_t st,
                       bool dependent) {
    const int64_t total = p->pairs * p->Vte;
    if (total == 0) return BS_OK;
    if (p->Wmax > 32) return set_error(BS_EUNSUPPORTED, "W > 32");
    // zte_off are sums of W Vte, so with Vte a multiple of 32 every block's span
    // starts on 16 bytes if the array does.  8192 pairs of W = 9, 128 vectors:
    // 21.3 -> 19.3 us (12.5 at the copy bandwidth); 32 768 pairs of W = 3..15:
    // 67.6 -> 53.8 (46).
    if (p->Vte % 32 == 0 && (reinterpret_cast<uintptr_t>(zte) & 15) == 0 && total / 32 < (1LL << 31) && apply_by_blocks(p))
        return p->Wmax <= 16 ? launch_apply_blocks<16>(p, zte, c, out, st, dependent)
                             : launch_apply_blocks<32>(p, zte, c, out, st, dependent);
    const bool wide = p->Wmax > 16;
    const int thr = wide ? ApplyCfg<32>::threads : ApplyCfg<16>::threads;
    launch_stage(dependent, wide ? apply_kernel<32> : apply_kernel<16>, (unsigned)((total + thr - 1) / thr), thr, 0, st,
                 zte, p->d_zte_off, p->d_Wg, p->d_woff, c, out, total, p->Vte);
    return check_launch("apply launch");
}

}  // namespace bs
