// Planar-array beamspace transform and window gather (Eq. ArrayFactor,
// Eq. VerDFT, Eq. HorDFT, Eq. OverallDFT, Eq. BeamTransform, Eq.
// OverallWindow read as S_h (x) S_v, Eq. ApplyWindow).
//
// Elements n = n_x Nz + n_z, beams m = m_x Mz + m_z, window entries
// w = w_x Wz + w_z.  Planar plans are limited to N <= 1024 and M <= 2048 (the
// paper's array is 4 x 32).
//
// beamspace2d_fft_kernel: a CTA takes 4096 / M consecutive vectors.  A thread
// loads one column of Nz elements straight from memory, takes its Mz-point
// DFT in registers and writes Mz rows of the shared buffer; all 4096 / Mx rows
// then go through the Mx-point Stockham passes of the linear kernels (zero
// past Nx).  The vectors of a subband share their targets' windows, so a
// thread decodes a (target, entry) once and stores it for all of them.  Bound
// by the window stores: 20 targets of 4 x 8 beams write 5 KB per 1 KB vector.
// 24 576 vectors of 4 x 32 elements, 8 x 64 beams: 38 us (22 us at the copy
// bandwidth; 195 us with the general kernel).
//
// beamspace2d_kernel: any other shape; one warp per vector (radix-2 passes in
// shared memory, direct vertical sums, every entry decoded per vector).
#include "beamspace_dev.cuh"
#include "internal.h"

#include <type_traits>

#include <algorithm>

namespace bs {

// Targets of the current subband: window-array base of its first vector, window
// starts, and how many of its vectors store.
struct __align__(16) Tgt2d {
    long long base;
    int sxz;   // start_x | start_z << 16
    int wn;    // W | Wz << 8 | stores << 16 | training << 24
};

constexpr int kPts2d = 4096;   // points per CTA

template <int MZ>
__device__ __forceinline__ void column_dft(const float2 *__restrict__ y, int Nz, bool valid, float2 *b, int pitch) {
    float2 a[MZ];
#pragma unroll
    for (int k = 0; k < MZ; ++k) a[k] = (valid && k < Nz) ? __ldg(y + k) : make_float2(0.f, 0.f);
    RegDFT<MZ>::run(a);
#pragma unroll
    for (int k = 0; k < MZ; ++k) b[k * pitch] = a[k];
}

template <int MX>
__global__ void __launch_bounds__(256, 4)
    beamspace2d_fft_kernel(const float2 *__restrict__ y, int Nx, int Nz, int Mz, float scale, int prec, GatherArgs ga,
                           const int32_t *__restrict__ start_z, const int32_t *__restrict__ Wz,
                           const int32_t *__restrict__ glist, int sumW, const float2 *__restrict__ tw) {
    using RP = Radix<MX>;
    constexpr int rows = kPts2d / MX, pl = padded_len(MX), nthr = 256;
    __shared__ float2 b[rows * pl];
    __shared__ float2 twx[MX];
    __shared__ Tgt2d tgt[kTabT];
    const int tid = threadIdx.x;
    const int N = Nx * Nz, V = rows / Mz;   // vectors of this CTA
    const int64_t vid0 = (int64_t)blockIdx.x * V;
    for (int k = tid; k < MX; k += nthr) twx[k] = __ldg(&tw[k * Mz]);
    for (int c = tid; c < V * Nx; c += nthr) {   // columns (v, n_x)
        const int v = c / Nx, nx = c - v * Nx;
        const bool valid = vid0 + v < ga.nvec;
        const float2 *col = y + (valid ? (vid0 + v) * N + nx * Nz : 0);
        float2 *d = b + v * Mz * pl + padrow(nx);
        switch (Mz) {
            case 1: column_dft<1>(col, Nz, valid, d, pl); break;
            case 2: column_dft<2>(col, Nz, valid, d, pl); break;
            case 4: column_dft<4>(col, Nz, valid, d, pl); break;
            case 8: column_dft<8>(col, Nz, valid, d, pl); break;
            default: column_dft<16>(col, Nz, valid, d, pl); break;
        }
    }
    __syncthreads();
    auto twl = [&](int k) -> float2 { return twx[k]; };
    auto cload = [&](int r, int t) -> float2 { return t < Nx ? b[r * pl + padrow(t)] : make_float2(0.f, 0.f); };
    auto sload = [&](int r, int t) -> float2 { return b[r * pl + padrow(t)]; };
    auto sstore = [&](int r, int t, float2 v) { b[r * pl + padrow(t)] = v; };
    stockham_pass_tw<MX, RP::r0, 1, rows, nthr, false, true>(tid, twl, cload, sstore);
    __syncthreads();
    if constexpr (RP::npass >= 2) {
        stockham_pass_tw<MX, RP::r1, RP::r0, rows, nthr, false, true>(tid, twl, sload, sstore);
        __syncthreads();
    }
    if constexpr (RP::npass >= 3) {
        stockham_pass_tw<MX, RP::r2, RP::r0 * RP::r1, rows, nthr, false, true>(tid, twl, sload, sstore);
        __syncthreads();
    }

    // window stores: the vectors of one subband (a group) share their targets'
    // windows; as many groups at a time as the entry table holds (with one, 32
    // vectors of B = 1 went through 32 barriers: 21 us for 64 vectors of M = 128)
    const int Bv = min(V, 1 << ga.log2B);
    const int ng = (int)min((int64_t)(V / Bv), (ga.nvec - vid0 + Bv - 1) / Bv), gmax = kTabT / ga.T;
    auto store_groups = [&](int g0, int gn, auto single) {   // single: gn = 1, no divisions
        for (int e = tid; e < gn * ga.T; e += nthr) {
            const int k = single ? 0 : e / ga.T, t = single ? e : e - k * ga.T;
            const int64_t vec = ga.vbase + vid0 + (g0 + k) * Bv;
            const int p = (int)(vec >> ga.log2F);
            const int q = (int)(vec & ((1 << ga.log2F) - 1));
            const int s = q >> ga.log2B, i = q & ((1 << ga.log2B) - 1);
            const bool train = p < ga.P_train;
            const int v0 = train ? (p << ga.log2B) + i : ((p - ga.P_train) << ga.log2B) + i;
            const int64_t g = (int64_t)t * ga.L + s;
            const int W = __ldg(&ga.Wg[g]);
            const int n = train ? max(0, min(Bv, __ldg(&ga.Kg[g]) - v0)) : Bv;
            Tgt2d x;
            x.base = __ldg(train ? &ga.ztr_off[g] : &ga.zte_off[g]) + (long long)v0 * W;
            x.sxz = __ldg(&ga.start[g]) | (__ldg(&start_z[g]) << 16);
            x.wn = W | (__ldg(&Wz[t]) << 8) | (n << 16) | (!single && train ? 1 << 24 : 0);
            tgt[e] = x;
        }
        __syncthreads();
        const bool train0 = (ga.vbase + vid0 + g0 * Bv) >> ga.log2F < ga.P_train;
        for (int e = tid; e < gn * sumW; e += nthr) {
            const int k = single ? 0 : e / sumW;
            const int packed = __ldg(&glist[e - k * sumW]);
            const int w = packed & 255;
            const Tgt2d te = tgt[k * ga.T + (packed >> 8)];
            const int W = te.wn & 255, wz = (te.wn >> 8) & 255, n = single ? te.wn >> 16 : (te.wn >> 16) & 255;
            const bool train = single ? train0 : (te.wn >> 24) != 0;
            const int wx = w / wz;
            const int mx = ((te.sxz & 0xFFFF) + wx) & (MX - 1), mz = ((te.sxz >> 16) + w - wx * wz) & (Mz - 1);
            const float2 *src = b + ((g0 + k) * Bv * Mz + mz) * pl + padrow(mx);
            const int64_t o = te.base + w;
            auto all = [&](auto put) {
#pragma unroll 4
                for (int v = 0; v < n; ++v) put(o + (int64_t)v * W, cscale(src[v * Mz * pl], scale));
            };
            if (!train) all([&](int64_t k, float2 v) { ga.zte[k] = v; });
            else if (prec == BS_PREC_FP32) all([&](int64_t k, float2 v) { store_train<BS_PREC_FP32>(ga.ztr, k, v, 1.f); });
            else if (prec == BS_PREC_FP16) all([&](int64_t k, float2 v) { store_train<BS_PREC_FP16>(ga.ztr, k, v, ga.store_scale); });
            else all([&](int64_t k, float2 v) { store_train<BS_PREC_BF16>(ga.ztr, k, v, ga.store_scale); });
        }
        __syncthreads();   // the entries are rewritten for the next groups
    };
    if (V == Bv) store_groups(0, 1, std::true_type{});
    else
        for (int g0 = 0; g0 < ng; g0 += gmax) store_groups(g0, min(gmax, ng - g0), std::false_type{});
}

__global__ void __launch_bounds__(128)
    beamspace2d_kernel(const float2 *__restrict__ y, int Nx, int Nz, int Mx, int Mz, float scale, int prec,
                       GatherArgs ga, const int32_t *__restrict__ start_z, const int32_t *__restrict__ Wz,
                       const int32_t *__restrict__ glist, int sumW) {
    extern __shared__ float2 sm2[];
    const int N = Nx * Nz, M = Mx * Mz;
    float2 *twx = sm2;             // [Mx / 2] e^{-2 pi i k / Mx}
    float2 *twz = twx + Mx / 2;    // [Mz]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float2 *ys = twz + Mz + (size_t)warp * (N + 2 * M);   // [N]
    float2 *b0 = ys + N;                                  // [Mz][Mx]
    float2 *b1 = b0 + M;                                  // [Mz][Mx]
    for (int k = tid; k < Mx / 2; k += blockDim.x) {
        float sn, cs;
        sincospif(-2.f * (float)k / (float)Mx, &sn, &cs);
        twx[k] = make_float2(cs, sn);
    }
    for (int k = tid; k < Mz; k += blockDim.x) {
        float sn, cs;
        sincospif(-2.f * (float)k / (float)Mz, &sn, &cs);
        twz[k] = make_float2(cs, sn);
    }
    __syncthreads();
    const int64_t vid = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    if (vid >= ga.nvec) return;   // no CTA barrier below
    for (int n = lane; n < N; n += 32) ys[n] = __ldcs(&y[vid * N + n]);
    __syncwarp();
    for (int e = lane; e < M; e += 32) {   // vertical DFT of every column n_x; zero past Nx
        const int mz = e / Mx, nx = e % Mx;
        float2 acc = make_float2(0.f, 0.f);
        if (nx < Nx)
            for (int nz = 0; nz < Nz; ++nz) acc = cadd(acc, cmul(ys[nx * Nz + nz], twz[(mz * nz) & (Mz - 1)]));
        b0[e] = acc;
    }
    __syncwarp();
    // horizontal FFT of every row: radix-2 Stockham passes (sub-transform
    // size Ns = 1, 2, .., Mx/2), ping-pong between b0 and b1
    float2 *src = b0, *dst = b1;
    const int half = Mx >> 1;
    for (int Ns = 1; Ns < Mx; Ns <<= 1) {
        for (int e = lane; e < M / 2; e += 32) {
            const int row = e / half, j = e % half;
            const float2 *x = src + row * Mx;
            const int k = j & (Ns - 1);
            const float2 a = x[j];
            const float2 b = cmul(x[j + half], twx[k * (half / Ns)]);
            float2 *o = dst + row * Mx + ((j - k) << 1) + k;
            o[0] = cadd(a, b);
            o[Ns] = csub(a, b);
        }
        __syncwarp();
        float2 *t = src;
        src = dst;
        dst = t;
    }
    const float2 *yb = src;   // [Mz][Mx]: beam m = m_x Mz + m_z at m_z Mx + m_x

    // window gather: a lane per entry of the flat (target, entry) list
    const int64_t v = ga.vbase + vid;
    const int p = (int)(v >> ga.log2F);
    const int q = (int)(v & ((1 << ga.log2F) - 1));
    const int s = q >> ga.log2B, i = q & ((1 << ga.log2B) - 1);
    const bool train = p < ga.P_train;
    const int v0 = train ? (p << ga.log2B) + i : ((p - ga.P_train) << ga.log2B) + i;
    const float sc_tr = (prec == BS_PREC_FP32) ? 1.f : ga.store_scale;
    for (int e = lane; e < sumW; e += 32) {
        const int packed = __ldg(&glist[e]);
        const int t = packed >> 8, w = packed & 255;
        const int64_t g = (int64_t)t * ga.L + s;
        const int W = __ldg(&ga.Wg[g]);
        const int wz = __ldg(&Wz[t]);
        const int mx = (__ldg(&ga.start[g]) + w / wz) & (Mx - 1);
        const int mz = (__ldg(&start_z[g]) + w % wz) & (Mz - 1);
        const float2 val = cscale(yb[mz * Mx + mx], scale);
        if (!train) {
            ga.zte[__ldg(&ga.zte_off[g]) + (int64_t)v0 * W + w] = val;
        } else if (v0 < __ldg(&ga.Kg[g])) {
            const int64_t idx = __ldg(&ga.ztr_off[g]) + (int64_t)v0 * W + w;
            if (prec == BS_PREC_FP16) store_train<BS_PREC_FP16>(ga.ztr, idx, val, sc_tr);
            else if (prec == BS_PREC_BF16) store_train<BS_PREC_BF16>(ga.ztr, idx, val, sc_tr);
            else store_train<BS_PREC_FP32>(ga.ztr, idx, val, 1.f);
        }
    }
}

template <int MX>
static bs_status launch_2d_fft(const bs_plan *p, const float2 *xc, const GatherArgs &ga, cudaStream_t st) {
    const int V = kPts2d / (MX * p->Mz);
    const int64_t blocks = (ga.nvec + V - 1) / V;
    if (blocks > 0x7FFFFFFF) return set_error(BS_EUNSUPPORTED, "too many vectors");
    beamspace2d_fft_kernel<MX><<<(unsigned)blocks, 256, 0, st>>>(
        xc, p->Nx, p->Nz, p->Mz, 1.0f / sqrtf((float)(MX * p->Mz)), p->cfg.precision, ga, p->d_start_z, p->d_Wz,
        p->d_glist, p->sumW, p->d_twM);
    return check_launch("planar beamspace launch");
}

bs_status launch_beamspace2d(const bs_plan *p, const float2 *xc, const GatherArgs &ga, cudaStream_t st) {
    const int Nx = p->Nx, Nz = p->Nz, Mx = p->Mx, Mz = p->Mz;
    if (ga.nvec == 0) return BS_OK;
    // rows of 8 to 1024 beams (Stockham radices), columns of up to 16 (in
    // registers), 2 to 32 vectors per CTA, targets within the entry table.  Not
    // where a CTA's subbands take three turns of the table or more (20 targets,
    // B = 1, M = 128: 11.5 us against 7.6; 100 targets, B = 2 22 against 16; two
    // turns: 10.0 and 10.4), nor where 32 vectors a CTA leave sixteen CTAs or
    // fewer (64 vectors, 2 targets 6.3 and 5.7).
    const int V = std::max(1, kPts2d / (Mx * Mz)), groups = std::max(1, V / p->B);
    const bool turns = p->cfg.T <= kTabT && groups > 2 * (kTabT / p->cfg.T);
    if (Mx >= 8 && Mx <= 1024 && Mz <= 16 && Mx * Mz >= 128 && p->cfg.T <= kTabT && !turns &&
        !(V == 32 && ga.nvec <= 16 * V)) {
        switch (Mx) {
            case 8: return launch_2d_fft<8>(p, xc, ga, st);
            case 16: return launch_2d_fft<16>(p, xc, ga, st);
            case 32: return launch_2d_fft<32>(p, xc, ga, st);
            case 64: return launch_2d_fft<64>(p, xc, ga, st);
            case 128: return launch_2d_fft<128>(p, xc, ga, st);
            case 256: return launch_2d_fft<256>(p, xc, ga, st);
            case 512: return launch_2d_fft<512>(p, xc, ga, st);
            default: return launch_2d_fft<1024>(p, xc, ga, st);
        }
    }
    const size_t per_warp = ((size_t)Nx * Nz + 2 * (size_t)Mx * Mz) * sizeof(float2);
    const size_t tables = ((size_t)Mx / 2 + Mz) * sizeof(float2);
    // up to 4 vectors (warps) per CTA while their buffers stay within 48 KB
    int nw = (int)std::min<size_t>(4, std::max<size_t>(1, (48 * 1024 - tables) / per_warp));
    const size_t smem = tables + (size_t)nw * per_warp;
    const int64_t blocks = (ga.nvec + nw - 1) / nw;
    if (blocks > 0x7FFFFFFF) return set_error(BS_EUNSUPPORTED, "too many vectors");
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(beamspace2d_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return cuda_error(e, "planar beamspace attribute");
    }
    beamspace2d_kernel<<<(unsigned)blocks, 32 * nw, smem, st>>>(xc, Nx, Nz, Mx, Mz, 1.0f / sqrtf((float)(Mx * Mz)),
                                                              p->cfg.precision, ga, p->d_start_z, p->d_Wz,
                                                              p->d_glist, p->sumW);
    return check_launch("planar beamspace launch");
}

}  // namespace bs
