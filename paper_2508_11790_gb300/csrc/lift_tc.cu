// Products of the lifted correlators on the tensor cores: their antenna-space
// output (Sec. III-C, below Eq. AntennaEqCorr) and their beam patterns
// (Eq. Cosine Sim).
//
// For one subband both are a complex matrix product C^H Y of the [T][N]
// correlators with N x columns: the columns are the channelised test vectors,
// or the steering vectors e^{j Omega n} of a grid of directions, which depend
// on the subband and the direction only and are generated as the operand is
// staged.  A CTA computes 64 targets by up to 128 columns (192 directions).
//
// tcgen05.mma, M = 128: rows 0-63 hold (Re c, Im c) and rows 64-127
// (-Im c, Re c) interleaved along K, so that with columns (Re y, Im y) they
// give Re and Im of conj(c) y; no row is padding when T is a multiple of 64.
// FP32 accuracy: every value is cut into three BF16 parts of 8 significant
// bits (truncated: they sum to it exactly, whatever its scale) and the six
// largest of the nine products are summed; the rest is below 2^-24 of the
// product.  The tensor core truncates its accumulator, so the leading product
// is drained every 64 elements into FP32 sums in registers; the other five
// (2^-8 of it and less) chain in an accumulator of their own.
//
// 17 warps, one CTA per SM.  Warps 0-15 stage operands and drain sums: two
// groups of eight warps take the even and the odd stages (load FP32 a turn
// ahead, split, store in the canonical K-major layout with core matrices 160
// bytes apart along K, so that the 16-byte stores of a quarter warp hit
// distinct banks), and each warp drains 32 tensor-memory lanes x a quarter of
// the columns of every chunk.  Warp 16 issues the products: per stage of 16
// elements 2 x 6, the trailing ones first, so that the drain of the last
// chunk's leading sum is hidden behind them.
//
// Measured at 64 targets, 1024 elements and 128 subbands: 128 test vectors
// 327 -> 62 us, 181 directions 598 -> 88 us; the SIMT kernels measured
// against were bound by shared-memory loads (2 x 2 register tiles, 26 TFLOP/s) and by
// one rotation per pair, element and direction.  With two leading sums drained
// two stages late and two direction tiles of 128: 76 and 122 us.  Timing copies
// with parts left out: products alone 45 us for 128 columns and 53 for 192 (98
// and 111 cycles each: both operands come from shared memory), hand-overs alone
// 19 and 25 (8 of launch, drain and store), loading, splitting and storing the
// operands alone 54 and 68.
#include "common.cuh"
#include "internal.h"
#include "tcgen05.cuh"

#include <algorithm>
#include <cmath>

namespace bs {
namespace {

constexpr int LT_T = 64;          // targets per CTA
constexpr int LT_K = 16;          // elements per stage (32 real rows of K)
constexpr int LT_CHUNK = 4;       // stages per drained chunk
constexpr int LT_STAGES = 3;
constexpr int LT_THREADS = 544;
constexpr int LT_LBO = 160, LT_SBO = 640;              // core matrices along K; 8-row groups
constexpr int LT_PART = 16 * LT_SBO;                   // one part of the 128 rows of A
constexpr int LT_OP = 3 * LT_PART;                     // A's three parts
// CC columns per CTA: 128 test vectors, or 192 directions (181 degrees in one
// tile: a product costs nearly the same for 64 to 192 columns, and the
// correlators are split once)
template <int CC>
struct LtTile {
    static constexpr int bpart = CC / 8 * LT_SBO;      // one part of the CC columns of B
    static constexpr int stage = LT_OP + 3 * bpart;
    static constexpr int misc = LT_STAGES * stage;
    static constexpr int smem = misc + 128 + 2 * LT_T * 8;
    static constexpr int pitch = CC + 1;               // output tile, float2
    static constexpr int dc = CC / 4;                  // columns drained per warp
    static_assert(LT_T * pitch * 8 <= misc, "the output tile reuses the stages");
    static_assert(smem <= 227 * 1024, "one CTA's shared memory");
    static_assert(2 * CC <= 512, "tensor memory: leading sum at column 0, trailing sum at 256");
};
constexpr uint32_t LT_COLS = 512;                      // tensor memory columns

struct LtArgs {
    const float2 *c_hat;   // [T][L][N]
    int N, L, T, cols;     // columns: test vectors or directions
    int tt, ct;            // tiles along targets and columns
    int *err;
    // output of the test vectors
    const float2 *xc;
    int F, B, P_train;
    float2 *out;           // [T][L][cols]
    // beam patterns
    const double *u;
    int Ltot, s0;
    double fc, fs, fd;
    float *pattern;        // [T][L][cols]
};

__device__ __forceinline__ uint64_t lt_desc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(LT_LBO >> 4) << 16) | ((uint64_t)(LT_SBO >> 4) << 32) |
           (1ull << 46);
}
// D (+)= A B, both operands in shared memory.  USE 0: A is read and kept in
// the collector buffer, 1: A is the buffer's, 2: for the last time, 3: A is
// read for this product alone.
template <int USE>
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, int accumulate) {
#define BS_MMA_SS(COLLECTOR)                                                                     \
    asm volatile("{\n\t.reg .pred p;\n\t"                                                       \
                 "setp.ne.b32 p, %4, 0;\n\t"                                                     \
                 "tcgen05.mma.cta_group::1.kind::f16" COLLECTOR " [%0], %1, %2, %3, p;\n\t}\n" \
                 ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory")
    if constexpr (USE == 0) BS_MMA_SS(".collector::a::fill");
    else if constexpr (USE == 1) BS_MMA_SS(".collector::a::use");
    else if constexpr (USE == 2) BS_MMA_SS(".collector::a::lastuse");
    else BS_MMA_SS("");
#undef BS_MMA_SS
}

// Four elements (eight floats) as three parts of four packed words each
// (word = real low, imaginary high).  The leading part of an infinity is that
// infinity, its trailing parts are NaN (join_parts).
__device__ __forceinline__ void split_item(const float2 (&v)[4], uint32_t (&w)[3][4]) {
    // minus the leading 8 bits of both components
    auto ntop = [](float2 x) {
        return make_float2(__uint_as_float((__float_as_uint(x.x) & 0xFFFF0000u) ^ 0x80000000u),
                           __uint_as_float((__float_as_uint(x.y) & 0xFFFF0000u) ^ 0x80000000u));
    };
    auto pack = [](float2 x) { return __byte_perm(__float_as_uint(x.x), __float_as_uint(x.y), 0x7632); };
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 x1 = __fadd2_rn(v[i], ntop(v[i]));
        const float2 x2 = __fadd2_rn(x1, ntop(x1));
        w[0][i] = pack(v[i]);
        w[1][i] = pack(x1);
        w[2][i] = pack(x2);
    }
}

// Four consecutive elements of a row from element n; zero past N.
template <bool VEC>
__device__ __forceinline__ void load_item(const float2 *row, int n, int N, bool valid, float2 (&v)[4]) {
    if constexpr (VEC) {   // N even, rows 16-byte aligned
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
            if (valid && n + 2 * h < N) q = __ldg(reinterpret_cast<const float4 *>(row + n + 2 * h));
            v[2 * h] = make_float2(q.x, q.y);
            v[2 * h + 1] = make_float2(q.z, q.w);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = (valid && n + i < N) ? __ldg(row + n + i) : make_float2(0.f, 0.f);
    }
}

// e^{j pi om x} with om = (hi, lo): the exact product of the high part is
// reduced modulo 2 before the low-order terms are added.
__device__ __forceinline__ float2 steer(float2 om, float x) {
    const float p = om.x * x;
    const float e = fmaf(om.x, x, -p) + om.y * x;
    float2 r;
    sincospif((p - 2.f * rintf(0.5f * p)) + e, &r.y, &r.x);
    return r;
}

template <bool PATTERN, bool VEC>
__global__ void __launch_bounds__(LT_THREADS, 1) lift_tc_kernel(const LtArgs a) {
    constexpr int CC = PATTERN ? 192 : 128, NI = CC / 64;   // NI: column items per thread and stage
    using TT = LtTile<CC>;
    constexpr int LT_MISC = TT::misc, LT_STAGE = TT::stage, LT_PITCH = TT::pitch, LT_C = CC;
    extern __shared__ __align__(128) unsigned char smlt[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint64_t *full = reinterpret_cast<uint64_t *>(smlt + LT_MISC);   // [LT_STAGES] stage written (the 8 warps of a group)
    uint64_t *empty = full + LT_STAGES;                              // [LT_STAGES] its products are done
    uint64_t *dfull = empty + LT_STAGES;                             // a chunk's leading sum is complete
    uint64_t *dempty = dfull + 1;                                    // it has been drained (16 warps)
    uint32_t *tslot = reinterpret_cast<uint32_t *>(dempty + 1);
    float2 *nrm = reinterpret_cast<float2 *>(smlt + LT_MISC + 128);  // [2 groups][64] ||sc c_hat||^2 of its stages, sc
    const uint32_t sbase = smem_u32(smlt);

    const int s = blockIdx.x / (a.tt * a.ct);
    const int rem = blockIdx.x - s * a.tt * a.ct;
    const int t0 = (rem / a.ct) * LT_T, v0 = (rem % a.ct) * LT_C;
    const int ncol = min(LT_C, a.cols - v0);
    const int NB = (ncol + 15) & ~15;                 // columns of the products
    const int nst = (a.N + LT_K - 1) / LT_K;
    const int nch = (nst + LT_CHUNK - 1) / LT_CHUNK;

    if (tid == 0) {
        for (int j = 0; j < LT_STAGES; ++j) {
            mbar_init(&full[j], 8);
            mbar_init(&empty[j], 1);
        }
        mbar_init(dfull, 1);
        mbar_init(dempty, 16);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 16) tmem_alloc(tslot, LT_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;

    if (warp < 16) {
        // ---- a thread of group grp stages elements 4 c .. of row (target) r
        // and of columns r and r + 64
        // (four neighbouring lanes read 128 bytes of a row)
        const int grp = warp >> 3, r = 8 * (warp & 7) + (lane >> 2), c = lane & 3;
        const uint32_t off = sbase + (uint32_t)((r >> 3) * LT_SBO + c * LT_LBO + (r & 7) * 16);
        // and drains rows 32 q + lane, columns DC h ..
        constexpr int DC = TT::dc;
        const int q = warp & 3, h = warp >> 2;
        const uint32_t dat = tmem + ((uint32_t)(32 * q) << 16) + DC * h;
        const bool mine = DC * h < NB;
        float2 acc[DC / 2];
#pragma unroll
        for (int k = 0; k < DC / 2; ++k) acc[k] = make_float2(0.f, 0.f);
        auto drain = [&](int j) -> bool {   // chunk j's leading sum
            if (!mbar_wait_bounded(dfull, (unsigned)j & 1u)) return false;
            if (mine) {
                tc_fence_after();
#pragma unroll
                for (int p = 0; p < DC / 16; ++p) {
                    float d[16];
                    tmem_ld16(dat + 16 * p, d);
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        acc[8 * p + k] = __fadd2_rn(acc[8 * p + k], make_float2(d[2 * k], d[2 * k + 1]));
                }
                tc_fence_before();
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(dempty);
            return true;
        };
        const bool tval = t0 + r < a.T;
        const float2 *crow = a.c_hat + ((int64_t)min(t0 + r, a.T - 1) * a.L + s) * a.N;
        const float2 *yrow[PATTERN ? 1 : NI];
        float2 om[PATTERN ? NI : 1], rot[PATTERN ? NI : 1];
        bool cval[NI];
#pragma unroll
        for (int b = 0; b < NI; ++b) {
            const int v = v0 + r + 64 * b;
            cval[b] = v < a.cols;
            if constexpr (PATTERN) {
                // subband centre frequency (Eq. SubChannelFreq): fc + ((l - 1/2) / L) fs,
                // l = s - L/2 + 1, in this order; Omega / pi = u f / f_d in FP64 once,
                // kept as an FP32 (hi, lo) pair (the FP64 pipe is narrow)
                const int sg = a.s0 + s;
                const double f = a.fc + (((double)(sg - a.Ltot / 2 + 1) - 0.5) / (double)a.Ltot) * a.fs;
                const double o = cval[b] ? a.u[v] * (f / a.fd) : 0.0;
                om[b].x = (float)o;
                om[b].y = (float)(o - (double)om[b].x);
                rot[b] = steer(om[b], 1.f);
            } else {
                const int vv = cval[b] ? v : 0;
                yrow[b] = a.xc + ((int64_t)(a.P_train + vv / a.B) * a.F + (int64_t)s * a.B + vv % a.B) * a.N;
            }
        }
        const int nb = (NB + 63) >> 6;   // blocks of 64 columns in use
        float nh = 0.f, nl = 0.f;   // sum of squares of this thread's part of the row, (hi, lo)
        float2 xa[4], xb[PATTERN ? 1 : NI][4];
        auto fetch = [&](int st) {
            const int n = st * LT_K + 4 * c;
            load_item<VEC>(crow, n, a.N, tval, xa);
            if constexpr (!PATTERN) {
                load_item<VEC>(yrow[0], n, a.N, cval[0], xb[0]);
                if (nb > 1) load_item<VEC>(yrow[1], n, a.N, cval[1], xb[1]);
            }
        };
        auto put = [&](uint32_t addr, uint32_t part, const uint32_t (&w)[3][4]) {
#pragma unroll
            for (int p = 0; p < 3; ++p) st_shared_v4(addr + p * part, w[p][0], w[p][1], w[p][2], w[p][3]);
        };
        auto stage = [&](int st) -> bool {
            const int b = st % LT_STAGES, use = st / LT_STAGES;
            if (use > 0 && !mbar_wait_bounded(&empty[b], (unsigned)(use - 1) & 1u)) return false;
            const uint32_t at = off + (uint32_t)(b * LT_STAGE);
            uint32_t w[3][4];
            split_item(xa, w);
            put(at, LT_PART, w);
#pragma unroll
            for (int p = 0; p < 3; ++p)
#pragma unroll
                for (int i = 0; i < 4; ++i) w[p][i] = __byte_perm(w[p][i], w[p][i], 0x1032) ^ 0x8000u;   // (-Im, Re)
            put(at + 8 * LT_SBO, LT_PART, w);   // row r + 64
            if constexpr (PATTERN) {
                float2 q = make_float2(0.f, 0.f);
#pragma unroll
                for (int i = 0; i < 4; ++i) q = __ffma2_rn(xa[i], xa[i], q);
                const float s2 = q.x + q.y;
                const float sm = nh + s2, bb = sm - nh;
                nl += (nh - (sm - bb)) + (s2 - bb);
                nh = sm;
            }
#pragma unroll
            for (int h = 0; h < NI; ++h) {
                if (h >= nb) break;
                if constexpr (PATTERN) {
                    float2 e[4];
                    e[0] = steer(om[h], (float)(st * LT_K + 4 * c));
#pragma unroll
                    for (int i = 0; i < 3; ++i) e[i + 1] = cmul(e[i], rot[h]);
                    split_item(e, w);
                } else {
                    split_item(xb[h], w);
                }
                put(at + LT_OP + h * 8 * LT_SBO, TT::bpart, w);
            }
            fence_proxy_async();   // the tensor core reads the stage through the async proxy
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[b]);
            if (st + 2 < nst) fetch(st + 2);
            return true;
        };
        if (grp < nst) fetch(grp);
        bool ok = true;
        int j = 0;   // chunks drained
        for (int st = grp; st < nst && ok; st += 2) {
            // chunk j is drained once this group has staged a part of the next
            // chunk, whose leading products wait for it (its trailing ones,
            // issued first, do not)
            if (st > LT_CHUNK * j + LT_CHUNK) ok = drain(j++);
            if (ok) ok = stage(st);
        }
        for (; j < nch && ok; ++j) ok = drain(j);
        if (ok) {   // the last chunk's barrier covers every product
            if (mine) {
                tc_fence_after();
#pragma unroll
                for (int p = 0; p < DC / 16; ++p) {
                    float d[16];
                    tmem_ld16(dat + 256 + 16 * p, d);
#pragma unroll
                    for (int k = 0; k < 8; ++k) acc[8 * p + k] = join_parts(acc[8 * p + k], make_float2(d[2 * k], d[2 * k + 1]));
                }
                const int row = 32 * q + lane;
                float *tile = reinterpret_cast<float *>(smlt) + ((row & 63) * LT_PITCH + DC * h) * 2 + (row >> 6);
#pragma unroll
                for (int k = 0; k < DC / 2; ++k) {
                    tile[4 * k] = acc[k].x;
                    tile[4 * k + 2] = acc[k].y;
                }
            }
        } else if (lane == 0) {
            atomicOr(a.err, 1);
        }
        if constexpr (PATTERN) {
            // The norm is n2 / sc^2.  Squares that left FP32's range, or come
            // near its ends, are formed again of elements scaled by a power
            // of two to a largest part of 1 to 2; a row's first elements say
            // nothing about the others, and following the largest so far
            // inside the loop took 6 to 10 of 90 us.
            float n2 = nh + nl, sc = 1.f;
            if (tval && !(n2 >= 0x1p-70f && n2 <= 0x1p96f)) {
                float m = 0.f;
                for (int st = grp; st < nst; st += 2) {
                    load_item<VEC>(crow, st * LT_K + 4 * c, a.N, true, xa);
#pragma unroll
                    for (int i = 0; i < 4; ++i) m = fmaxf(m, fmaxf(fabsf(xa[i].x), fabsf(xa[i].y)));
                }
                const int e = max(-126, min(126, (__float_as_int(m) >> 23) - 127));
                sc = __int_as_float((127 - e) << 23);
                n2 = 0.f;
                for (int st = grp; st < nst; st += 2) {
                    load_item<VEC>(crow, st * LT_K + 4 * c, a.N, true, xa);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float x = xa[i].x * sc, y = xa[i].y * sc;
                        n2 = fmaf(x, x, fmaf(y, y, n2));
                    }
                }
            }
            // the four lanes of a row, on the smallest of their scales
            if (n2 == 0.f) sc = 0x1p126f;
            float to = fminf(sc, __shfl_xor_sync(0xFFFFFFFFu, sc, 1));
            to = fminf(to, __shfl_xor_sync(0xFFFFFFFFu, to, 2));
            const float f = to * (1.f / sc);
            n2 = n2 * f * f;
            sc = to;
            n2 += __shfl_xor_sync(0xFFFFFFFFu, n2, 1);
            n2 += __shfl_xor_sync(0xFFFFFFFFu, n2, 2);
            if (c == 0) nrm[64 * grp + r] = make_float2(n2, sc);
        }
    } else {
        // ---- MMA warp
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10)            // D FP32; A, B BF16, K-major
                               | ((uint32_t)(NB >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        bool ok = true;
        for (int st = 0; st < nst && ok; ++st) {
            const int b = st % LT_STAGES, j = st / LT_CHUNK;
            ok = mbar_wait_bounded(&full[b], (unsigned)(st / LT_STAGES) & 1u);
            if (!ok) break;
            tc_fence_after();
            const uint32_t sa = sbase + b * LT_STAGE, sb = sa + LT_OP;
            if (lane == 0) {   // trailing products
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    uint64_t da[3], db[3];
#pragma unroll
                    for (int p = 0; p < 3; ++p) {
                        da[p] = lt_desc(sa + p * LT_PART + k * 2 * LT_LBO);
                        db[p] = lt_desc(sb + p * TT::bpart + k * 2 * LT_LBO);
                    }
                    mma_ss<0>(tmem + 256, da[0], db[1], idesc, st | k);
                    mma_ss<2>(tmem + 256, da[0], db[2], idesc, 1);
                    mma_ss<0>(tmem + 256, da[1], db[0], idesc, 1);
                    mma_ss<2>(tmem + 256, da[1], db[1], idesc, 1);
                    mma_ss<3>(tmem + 256, da[2], db[0], idesc, 1);
                }
            }
            __syncwarp();
            if (st % LT_CHUNK == 0 && j >= 1) ok = mbar_wait_bounded(dempty, (unsigned)(j - 1) & 1u);
            if (!ok) break;
            tc_fence_after();
            if (lane == 0) {   // leading products
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    mma_ss<3>(tmem, lt_desc(sa + k * 2 * LT_LBO), lt_desc(sb + k * 2 * LT_LBO), idesc, st % LT_CHUNK | k);
                mma_commit(&empty[b]);
                if (st % LT_CHUNK == LT_CHUNK - 1 || st + 1 == nst) mma_commit(dfull);
            }
            __syncwarp();
        }
        if (!ok && lane == 0) atomicOr(a.err, 1);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 16) tmem_dealloc(tmem, LT_COLS);
    // the tile to memory, a row of columns per target
    const float2 *tile = reinterpret_cast<const float2 *>(smlt);
    const int nt = min(LT_T, a.T - t0);
    for (int r = warp; r < nt; r += LT_THREADS / 32) {
        const int64_t o = ((int64_t)(t0 + r) * a.L + s) * a.cols + v0;
        float sc = 1.f, inv = 1.f;
        if constexpr (PATTERN) {
            const float2 n0 = nrm[r], n1 = nrm[64 + r];   // the two groups' stages
            sc = fminf(n0.y, n1.y);
            const float f0 = sc * (1.f / n0.y), f1 = sc * (1.f / n1.y);
            inv = 1.f / (sqrtf(n0.x * f0 * f0 + n1.x * f1 * f1) * sqrtf((float)a.N));
        }
        for (int k = lane; k < ncol; k += 32) {
            const float2 v = tile[r * LT_PITCH + k];
            if constexpr (PATTERN) {
                const float x = v.x * sc, y = v.y * sc;
                a.pattern[o + k] = sqrtf(x * x + y * y) * inv;
            } else {
                a.out[o + k] = v;
            }
        }
    }
}

template <bool PATTERN, bool VEC>
bs_status launch_lift_tc_t(const LtArgs &a, cudaStream_t st) {
    constexpr int smem = LtTile<PATTERN ? 192 : 128>::smem;
    static PerDevice attr;
    if (bs_status s = attr.get([](int *) {
            return cuda_error(cudaFuncSetAttribute(lift_tc_kernel<PATTERN, VEC>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                              "lifted products attribute");
        }))
        return s;
    const int64_t tiles = (int64_t)a.L * a.tt * a.ct;
    if (tiles > 0x7FFFFFFF) return set_error(BS_EUNSUPPORTED, "too many tiles");
    lift_tc_kernel<PATTERN, VEC><<<(unsigned)tiles, LT_THREADS, smem, st>>>(a);
    return check_launch("lifted products launch");
}

LtArgs lift_args(const bs_plan *p, const float2 *c_hat, int cols, int tile) {
    LtArgs a{};
    a.c_hat = c_hat;
    a.N = p->cfg.N;
    a.L = p->Ls;   // the plan's subbands
    a.T = p->cfg.T;
    a.cols = cols;
    a.tt = (a.T + LT_T - 1) / LT_T;
    a.ct = (cols + tile - 1) / tile;
    a.err = p->d_err;
    return a;
}

// Few pairs: the SIMT kernel (lift.cu).  A tile takes as long for 3 targets as
// for 64, 8 us + 51 ns an element and wave of tiles; the SIMT kernel's time
// grows with the pairs and directions from 4.5 us.  Both lines are fits within
// 10 % of 135 measured sizes (N 48 .. 1024, 48 .. 8192 pairs, 31 .. 181
// directions); at the line both take the same: 512 pairs of N = 100, 64
// directions 14.7 us each, 1024 of N = 256 23.2 and 23.3, 2048 of N = 512, 31
// directions 34.6 and 34.1.  By the whole plan's subbands, so that a shard's
// patterns are bit for bit those of the whole.
bool pattern_simt(const bs_plan *p, int n_dirs) {
    const double N = p->cfg.N, pairs = (double)p->cfg.T * p->cfg.L;
    if (p->cfg.N + (int64_t)n_dirs > 6144) return false;   // not measured beyond: the tiles
    const double tiles = (double)p->cfg.L * ((p->cfg.T + LT_T - 1) / LT_T) * ((n_dirs + 191) / 192);
    return pairs * (7.0 + (n_dirs + 31) / 32 * (3.5 + N / 124)) < (4000 + 50 * N) * std::ceil(tiles / p->num_sms);
}

// Outputs of short rows: the SIMT kernel (lift.cu).  A tensor-core tile spends
// 4 to 6 us on its start, drain and store, a SIMT tile of 32 x 32 outputs 2 us
// and 2 more per 32 elements, as long as its four times as many tiles are at
// most two waves.  N = 16, 1 to 64 targets, 16 subbands 4.0 us against 4.4 to
// 6.0; N = 64 6.3 against 7 to 8.8; N = 65 with up to a wave 8.1 and 9.0, N = 100
// 11.1 and 11.3; with 64 subbands of 64 targets x 128 vectors 7.2 and 6.1.  By
// the whole plan's subbands, so that a shard's outputs are those of the whole.
bool lifted_simt(const bs_plan *p) {
    const int N = p->cfg.N, T = p->cfg.T, L = p->cfg.L, V = p->Vte;
    if (N > 96) return false;
    const double tc = (double)L * ((T + LT_T - 1) / LT_T) * ((V + 127) / 128);
    const double simt = (double)L * ((T + 31) / 32) * ((V + 31) / 32);
    return simt <= (N <= 64 ? 2 * std::ceil(tc / p->num_sms) : 1) * p->num_sms;
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

bs_status launch_apply_lifted(const bs_plan *p, const float2 *xc, const float2 *c_hat, float2 *out,
                              cudaStream_t st) {
    if (p->Vte == 0 || p->pairs == 0) return BS_OK;
    if (lifted_simt(p)) return launch_apply_lifted_simt(p, xc, c_hat, out, st);
    LtArgs a = lift_args(p, c_hat, p->Vte, 128);
    a.xc = xc;
    a.F = p->Fs;
    a.B = p->B;
    a.P_train = p->cfg.P_train;
    a.out = out;
    const bool vec = (a.N & 1) == 0 && aligned16(xc) && aligned16(c_hat);
    return vec ? launch_lift_tc_t<false, true>(a, st) : launch_lift_tc_t<false, false>(a, st);
}

bs_status launch_beam_pattern(const bs_plan *p, const float2 *c_hat, int n_dirs, const double *u, float *pattern,
                              cudaStream_t st) {
    if (n_dirs == 0 || p->pairs == 0) return BS_OK;
    if (((size_t)p->cfg.N + n_dirs) * sizeof(float2) > 200 * 1024)
        return set_error(BS_EUNSUPPORTED, "beam pattern: N + n_dirs must be <= 25600");
    if (pattern_simt(p, n_dirs)) return launch_beam_pattern_simt(p, c_hat, n_dirs, u, pattern, st);
    LtArgs a = lift_args(p, c_hat, n_dirs, 192);
    a.u = u;
    a.Ltot = p->cfg.L;
    a.s0 = p->s0;
    a.fc = p->cfg.fc;
    a.fs = p->cfg.fs;
    a.fd = p->cfg.fd;
    a.pattern = pattern;
    const bool vec = (a.N & 1) == 0 && aligned16(c_hat);
    return vec ? launch_lift_tc_t<true, true>(a, st) : launch_lift_tc_t<true, false>(a, st);
}

}  // namespace bs
