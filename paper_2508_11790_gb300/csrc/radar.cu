// Processing after the beamformer (Sec. II, Fig. 1: synthesis of the
// wideband output and standard range-Doppler processing; Sec. IV: detection
// 10 dB above the noise floor).
//
// * rows: the beamformed output of pair (t, s) at test vector r B + i is bin
//   q = s B + i of record r, FFT bin k = (q - F/2) mod F.  The matched filter
//   multiplies it by conj(P[k]) (P: the transmitted pulse's orthonormal
//   spectrum).  The synthesis IFFT runs as a forward FFT of the conjugate,
//   IFFT(Z) = conj(FFT(conj Z)) (orthonormal), so the first FFT pass reads
//   conj(Y conj(P)) = conj(Y) P straight from the outputs.
// * doppler: map[t][d][tau] = |sum_r rp[t][r][tau] e^{-j 2 pi d r / P_te}|^2
//   with rp = conj(row FFT output); thread per (t, tau), all d.  Up to 16
//   records the thread keeps its column in registers and the P_te phase
//   factors come from shared memory.
// * cfar (Sec. IV-B: a one-dimensional CFAR across the velocity bins): a
//   cluster of up to 8 CTAs per target, a thread per range cell tau: the floor
//   of cell (d, tau) is the mean of the other P_te - 1 velocity bins of range
//   cell tau (the cell under test left out), a detection is a cell above its
//   floor x 10^(thr/10) (FP32); the CTAs count the detections and reduce the
//   strongest one (smallest index on ties) through distributed shared memory.
//
// Bound by memory latency and launches (16 MB in all at 64 targets, 8 records,
// 2048 points).  There: matched filter as a pass of its own 9 us + rows 8 ->
// the rows alone; doppler a sincospi and a load per record, bin and cell (28
// us); CFAR one CTA per target (32 us).  The three launches together: 75 -> 34
// us.
#include "beamspace_dev.cuh"
#include "common.cuh"
#include "internal.h"

namespace bs {

// Matched filter and row FFT: vpb rows (t, r) of F points per CTA.
template <int F>
__global__ void __launch_bounds__(BsCfg<F>::nthr, BsCfg<F>::minb)
    rd_rows_kernel(const float2 *__restrict__ out, const float2 *__restrict__ pulse, const float2 *__restrict__ tw,
                   float scale, float2 *__restrict__ fr, int64_t rows, int L, int log2B, int P_te) {
    using RP = Radix<F>;
    constexpr int vpb = BsCfg<F>::vpb, nthr = BsCfg<F>::nthr, pl = BsCfg<F>::pl;
    extern __shared__ float2 sm[];
    const int tid = threadIdx.x;
    const int64_t row0 = (int64_t)blockIdx.x * vpb;
    // subband 0 of each row's outputs, decoded once: a division per load held
    // the loads back (2 rows of F = 64 took 10 us, gather and FFT apart 7)
    __shared__ int64_t first[vpb];
    if (tid < vpb) {
        const int64_t row = row0 + tid, t = row / P_te;
        first[tid] = row < rows ? (t * L * P_te + (row - t * P_te)) << log2B : -1;
    }
    __syncthreads();
    auto gload = [&](int c, int k) -> float2 {
        const int64_t o = first[c];
        if (o < 0) return make_float2(0.f, 0.f);
        const int q = (k + F / 2) & (F - 1);
        const float2 y = __ldg(&out[o + (((int64_t)(q >> log2B) * P_te) << log2B) + (q & ((1 << log2B) - 1))]);
        const float2 pk = __ldg(&pulse[k]);
        return make_float2(y.x * pk.x + y.y * pk.y, y.x * pk.y - y.y * pk.x);   // conj(y) pk
    };
    auto sload = [&](int c, int m) -> float2 { return sm[c * pl + padrow(m)]; };
    auto sstore = [&](int c, int m, float2 v) { sm[c * pl + padrow(m)] = v; };
    stockham_pass<F, RP::r0, 1, vpb, nthr, false, false>(tid, tw, gload, sstore);
    __syncthreads();
    if constexpr (RP::npass >= 2) {
        stockham_pass<F, RP::r1, RP::r0, vpb, nthr, false, true>(tid, tw, sload, sstore);
        __syncthreads();
    }
    if constexpr (RP::npass >= 3) {
        stockham_pass<F, RP::r2, RP::r0 * RP::r1, vpb, nthr, false, true>(tid, tw, sload, sstore);
        __syncthreads();
    }
    for (int e = tid; e < vpb * F; e += nthr) {
        const int c = e / F, m = e % F;
        if (row0 + c < rows) fr[(row0 + c) * F + m] = cscale(sload(c, m), scale);
    }
}

constexpr int RD_P = 16;   // records of the register paths

template <int PM>
__global__ void __launch_bounds__(128)
    rd_doppler_reg_kernel(const float2 *__restrict__ fr, float *__restrict__ map, int T, int P_te, int F) {
    __shared__ float2 tw[PM];
    if (threadIdx.x < P_te) {
        float sn, cs;
        sincospif(-2.f * (float)threadIdx.x / (float)P_te, &sn, &cs);
        tw[threadIdx.x] = make_float2(cs, sn);
    }
    __syncthreads();
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // (t, tau)
    if (e >= (int64_t)T * F) return;
    const int tau = (int)(e % F), t = (int)(e / F);
    const float2 *col = fr + (int64_t)t * P_te * F + tau;
    float2 v[PM];
#pragma unroll
    for (int r = 0; r < PM; ++r) v[r] = r < P_te ? __ldg(&col[(int64_t)r * F]) : make_float2(0.f, 0.f);
    for (int d = 0; d < P_te; ++d) {
        float re = 0.f, im = 0.f;
        int k = 0;   // d r mod P_te
#pragma unroll
        for (int r = 0; r < PM; ++r) {
            if (r < P_te) {
                const float2 w = tw[k];
                // conj(v) * (cs + j sn)
                re = fmaf(v[r].x, w.x, fmaf(v[r].y, w.y, re));
                im = fmaf(v[r].x, w.y, fmaf(-v[r].y, w.x, im));
            }
            k += d;
            if (k >= P_te) k -= P_te;
        }
        map[((int64_t)t * P_te + d) * F + tau] = re * re + im * im;
    }
}

__global__ void rd_doppler_kernel(const float2 *__restrict__ fr, float *__restrict__ map, int T, int P_te, int F) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // (t, tau)
    if (e >= (int64_t)T * F) return;
    const int tau = (int)(e % F), t = (int)(e / F);
    const float2 *col = fr + (int64_t)t * P_te * F + tau;
    for (int d = 0; d < P_te; ++d) {
        float re = 0.f, im = 0.f;
        for (int r = 0; r < P_te; ++r) {
            const float2 v = col[(int64_t)r * F];       // rp = conj(v)
            float sn, cs;
            sincospif(-2.f * (float)((d * r) % P_te) / (float)P_te, &sn, &cs);
            // conj(v) * (cs + j sn)
            re = fmaf(v.x, cs, fmaf(v.y, sn, re));
            im = fmaf(v.x, sn, fmaf(-v.y, cs, im));
        }
        map[((int64_t)t * P_te + d) * F + tau] = re * re + im * im;
    }
}

// Strongest detection so far; ties keep the smaller cell index.
struct Best {
    float v;
    int i;   // -1: none
};
__device__ __forceinline__ bool better(Best a, Best b) {   // a over b
    return a.i >= 0 && (b.i < 0 || a.v > b.v || (a.v == b.v && a.i < b.i));
}

// PM: the range cell's P_te <= PM bins are kept in registers (0: read again, eight
// at a time; one at a time 8 targets of 64 records, F = 256: 121 us, 83 now).
// nc CTAs (one cluster) per target.
template <int PM>
__global__ void __launch_bounds__(256) rd_cfar_kernel(const float *__restrict__ map, int P_te, int F, float ratio,
                                                      float *__restrict__ floor_out, int32_t *__restrict__ count,
                                                      uint8_t *__restrict__ mask, int32_t *__restrict__ peak, int nc) {
    const int t = blockIdx.x / nc, rank = blockIdx.x - t * nc;
    const int64_t cells = (int64_t)P_te * F;
    const float *m = map + (int64_t)t * cells;
    __shared__ Best best[8];
    __shared__ int hits[8];
    __shared__ Best cta_best;
    __shared__ int cta_hits;
    const float inv = 1.0f / (float)(P_te - 1);
    Best b{-1.0f, -1};
    int mine = 0;
    for (int tau = rank * 256 + threadIdx.x; tau < F; tau += nc * 256) {
        float v[PM ? PM : 1];
        if constexpr (PM > 0) {
#pragma unroll
            for (int e = 0; e < PM; ++e) v[e] = e < P_te ? __ldg(&m[(int64_t)e * F + tau]) : 0.f;
        }
        auto cell = [&](int d, float x, float sum) {
            const float fl = sum * inv;
            const int64_t c = (int64_t)d * F + tau;
            const bool hit = x > fl * ratio;
            floor_out[(int64_t)t * cells + c] = fl;
            if (mask) mask[(int64_t)t * cells + c] = hit ? 1 : 0;
            mine += hit;
            const Best h{x, (int)c};
            if (hit && x > -1.0f && better(h, b)) b = h;
        };
        // the sum of the other velocity bins of range cell tau, in order
        if constexpr (PM > 0) {
#pragma unroll
            for (int d = 0; d < PM; ++d) {
                float sum = 0.f;
#pragma unroll
                for (int e = 0; e < PM; ++e)
                    if (e != d && e < P_te) sum += v[e];
                if (d < P_te) cell(d, v[d], sum);
            }
        } else {
            for (int d = 0; d < P_te; ++d) {
                float sum = 0.f;
                auto add = [&](int e0, int e1) {   // eight loads in flight, added in order
                    const float *x = m + (int64_t)e0 * F + tau;
#pragma unroll 8
                    for (int e = e0; e < e1; ++e, x += F) sum += __ldg(x);
                };
                add(0, d);
                add(d + 1, P_te);
                cell(d, __ldg(&m[(int64_t)d * F + tau]), sum);
            }
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto warp_best = [&](Best x) {
        for (int o = 16; o; o >>= 1) {
            const Best y{__shfl_xor_sync(0xFFFFFFFFu, x.v, o), __shfl_xor_sync(0xFFFFFFFFu, x.i, o)};
            if (better(y, x)) x = y;
        }
        return x;
    };
    b = warp_best(b);
    mine = __reduce_add_sync(0xFFFFFFFFu, mine);
    if (lane == 0) best[warp] = b, hits[warp] = mine;
    __syncthreads();
    if (threadIdx.x == 0) {
        int n = 0;
        for (int w = 0; w < 8; ++w) {
            n += hits[w];
            if (better(best[w], b)) b = best[w];
        }
        if (nc == 1) {
            count[t] = n;
            if (peak) peak[t] = b.i;
        } else {
            cta_best = b;
            cta_hits = n;
        }
    }
    if (nc == 1) return;   // no cluster
    cluster_sync();
    if (rank == 0 && threadIdx.x == 0) {
        int n = 0;
        Best r{-1.0f, -1};
        for (int z = 0; z < nc; ++z) {
            auto remote = [&](const void *p) {
                unsigned a, x;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                             : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(z));
                asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(x) : "r"(a) : "memory");
                return x;
            };
            const Best h{__uint_as_float(remote(&cta_best.v)), (int)remote(&cta_best.i)};
            n += (int)remote(&cta_hits);
            if (better(h, r)) r = h;
        }
        count[t] = n;
        if (peak) peak[t] = r.i;
    }
    // no CTA leaves while the first may read its result
    cluster_sync();
}

template <int F>
static bs_status launch_rd_rows(const bs_plan *p, const float2 *out, const float2 *pulse, float2 *fr, int log2B,
                                cudaStream_t st) {
    using C = BsCfg<F>;
    static PerDevice attr;
    if (bs_status s = attr.get([](int *) {
            return cuda_error(cudaFuncSetAttribute(rd_rows_kernel<F>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)C::smem),
                              "range-Doppler rows attribute");
        }))
        return s;
    const int64_t rows = (int64_t)p->cfg.T * p->cfg.P_test;
    const int64_t blocks = (rows + C::vpb - 1) / C::vpb;
    if (blocks > 0x7FFFFFFF) return set_error(BS_EUNSUPPORTED, "too many rows");
    rd_rows_kernel<F><<<(unsigned)blocks, C::nthr, C::smem, st>>>(out, pulse, p->d_twF, 1.0f / sqrtf((float)F), fr, rows,
                                                                 p->cfg.L, log2B, p->cfg.P_test);
    return check_launch("range-Doppler rows launch");
}

bs_status launch_range_doppler(const bs_plan *p, const float2 *out, const float2 *pulse, float2 *work, float *map,
                               cudaStream_t st) {
    const int T = p->cfg.T, P_te = p->cfg.P_test, F = p->cfg.F;
    if (P_te == 0 || T == 0) return BS_OK;
    int log2B = 0;
    while ((1 << log2B) < p->B) ++log2B;
    bs_status s = BS_OK;
    switch (F) {   // a power of two in 16 .. 4096 (plan validation)
        case 16: s = launch_rd_rows<16>(p, out, pulse, work, log2B, st); break;
        case 32: s = launch_rd_rows<32>(p, out, pulse, work, log2B, st); break;
        case 64: s = launch_rd_rows<64>(p, out, pulse, work, log2B, st); break;
        case 128: s = launch_rd_rows<128>(p, out, pulse, work, log2B, st); break;
        case 256: s = launch_rd_rows<256>(p, out, pulse, work, log2B, st); break;
        case 512: s = launch_rd_rows<512>(p, out, pulse, work, log2B, st); break;
        case 1024: s = launch_rd_rows<1024>(p, out, pulse, work, log2B, st); break;
        case 2048: s = launch_rd_rows<2048>(p, out, pulse, work, log2B, st); break;
        default: s = launch_rd_rows<4096>(p, out, pulse, work, log2B, st); break;
    }
    if (s) return s;
    const int64_t n2 = (int64_t)T * F;
    const auto doppler = P_te <= 8 ? rd_doppler_reg_kernel<8> : P_te <= RD_P ? rd_doppler_reg_kernel<RD_P> : rd_doppler_kernel;
    doppler<<<(unsigned)((n2 + 127) / 128), 128, 0, st>>>(work, map, T, P_te, F);
    return check_launch("Doppler launch");
}

bs_status launch_cfar(const bs_plan *p, const float *map, float threshold_db, float *floor, int32_t *count,
                      uint8_t *mask, int32_t *peak, cudaStream_t st) {
    const int T = p->cfg.T;
    if (T == 0 || p->cfg.P_test == 0) return BS_OK;
    const float ratio = powf(10.f, threshold_db / 10.f);
    const int P_te = p->cfg.P_test, F = p->cfg.F;
    // CTAs per target: 256 range cells each, up to the portable cluster size and
    // to eight CTAs an SM in all (1000 targets of 3 records, F = 2048: 34 us with
    // eight each)
    int nc = 1;
    while (nc < 8 && nc * 256 < F && (int64_t)nc * T < 8LL * p->num_sms) nc *= 2;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(nc * T));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = nc;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = nc > 1 ? 1 : 0;
    const auto kernel = P_te <= 4 ? rd_cfar_kernel<4> : P_te <= 8 ? rd_cfar_kernel<8> : P_te <= RD_P ? rd_cfar_kernel<RD_P>
                        : P_te <= 32 ? rd_cfar_kernel<32> : rd_cfar_kernel<0>;
    return cuda_error(cudaLaunchKernelEx(&cfg, kernel, map, P_te, F, ratio, floor, count, mask, peak, nc), "CFAR launch");
}

}  // namespace bs
