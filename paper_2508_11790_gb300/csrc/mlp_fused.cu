// The loading network's passes on the tensor cores: one kernel for forward
// (and, in training, the loss gradient and the activation gradients of a
// slab of rows), one for all weight gradients and the Adam update.
//
// Accuracy: an FP32 value is cut into three BF16 parts of 8 significant bits
// each (truncated, so the parts sum to it exactly); a product with a BF16
// weight is three exact MMA products, a product of two FP32 values the six
// largest of nine (the rest is below 2^-24 of the product).  The leading
// products are summed in rounded FP32 additions every 16 rows (mma_add).
// Against FP64, gradients of a 1024-row batch: 4e-7 of their norm, as the
// FP32 SIMT products; outputs 2e-7 to 4e-7, as before.
//
// Bound: latency.  Training step of the 101-256-256-10 network, 1024 rows:
// 470 us (15 launches, the three weight gradients 160 us each: 4 to 16 CTAs
// with a serial chain of 1024 rows) -> 35 us (slab kernel 18, weight
// gradients 14).  Forward of 4096 rows, back to back in a graph: 99 us (three
// launches) -> 17.5, 3 of them the hidden layers' 17 MB in the work buffers.
// With 8 warps instead of 16 and 32-row slabs at 1024 rows (32 CTAs) the slab
// kernel took 40 us: 17 % issue, its two warps per scheduler waiting for
// unbatched global loads and instruction fetch.
//
// mma.sync and not tcgen05: a training minibatch of 1024 rows is 64 slabs of
// 16 rows here; 128-row tiles of tcgen05 would be 8 CTAs that take as long
// each (M = 128, N = 256, K = 16 per 128 cycles is four times this kernel's
// rate on eight times its rows), its truncated accumulators would have to be
// drained every 16 rows, and the activations would leave tensor memory
// through registers at every layer, while here the accumulator fragments
// stay in the registers of the warp that needs them for the ReLU masks.
#include <math.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "internal.h"

namespace bs {
namespace {

constexpr int NTHR = 512;     // threads of the slab kernel: 16 warps
constexpr int KC = 64;        // input features per staged chunk of layer 1
constexpr int OMAX = 64;      // outputs

__device__ __forceinline__ unsigned s32(const void *p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], unsigned a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldsm2(uint32_t (&r)[2], unsigned a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], unsigned a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldsm2t(uint32_t (&r)[2], unsigned a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// d = A B (no addend)
__device__ __forceinline__ void mma0(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
// acc += A B of the leading parts: the 16 products are summed by the tensor
// core, the running sum by rounded FP32 additions.  The tensor core truncates
// its accumulator, and a chain of K / 16 truncated steps drifts: gradients of
// a batch of 1024 came out 5e-5 off through the ReLU masks that the drift of
// the pre-activations flipped.  The trailing parts are 2^-8 of the sum and
// chain in the tensor core.
__device__ __forceinline__ void mma_add(float (&acc)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    float d[4];
    mma0(d, a, b0, b1);
    const float2 x = __fadd2_rn(make_float2(acc[0], acc[1]), make_float2(d[0], d[1]));
    const float2 y = __fadd2_rn(make_float2(acc[2], acc[3]), make_float2(d[2], d[3]));
    acc[0] = x.x;
    acc[1] = x.y;
    acc[2] = y.x;
    acc[3] = y.y;
}

// Three BF16 parts of x and y, packed (x low half).  x = hi + mid + lo
// exactly; an infinite x keeps mid = lo = 0, a NaN stays a NaN.
__device__ __forceinline__ void split3(float x, float y, uint32_t &hi, uint32_t &mid, uint32_t &lo) {
    auto top = [](float v) { return __uint_as_float(__float_as_uint(v) & 0xFFFF0000u); };
    auto rest = [&](float v) { return isinf(v) ? 0.f : v - top(v); };
    const float x1 = rest(x), y1 = rest(y);
    const float x2 = x1 - top(x1), y2 = y1 - top(y1);
    hi = __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
    mid = __byte_perm(__float_as_uint(x1), __float_as_uint(y1), 0x7632);
    lo = __byte_perm(__float_as_uint(x2), __float_as_uint(y2), 0x7632);
}

// Eight consecutive BF16 values of a parameter array (np elements at p),
// from element `off`; those from cnt on are zero.  Five aligned words shifted
// into place, without branches, so that a thread's loads are all in flight
// at once (rows of n_in elements start at any address).  The words are
// clamped to the last whole one of the array: every weight matrix is followed
// by its bias, so no weight lies beyond it.
__device__ __forceinline__ uint4 load8(const __nv_bfloat16 *p, int64_t off, int cnt, int64_t np) {
    const uintptr_t base = reinterpret_cast<uintptr_t>(p);
    const int64_t odd = (base >> 1) & 1;                        // the array starts in the upper half of a word
    const uint32_t *w = reinterpret_cast<const uint32_t *>(base & ~(uintptr_t)3);
    const int64_t i = off + odd, last = ((np + odd) >> 1) - 1;
    const int sh = (int)(i & 1) * 16;
    uint32_t u[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) u[k] = __ldg(w + min((i >> 1) + k, last));
    uint32_t o[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        o[k] = __funnelshift_r(u[k], u[k + 1], sh);
        if (2 * k >= cnt) o[k] = 0;
        else if (2 * k + 1 >= cnt) o[k] &= 0xFFFFu;
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

struct MlpArgs {
    const float *X;
    const __nv_bfloat16 *wb;        // parameters, BF16 copy; the layers' offsets:
    int64_t o1, o2, o3, np;
    const float *b1, *b2, *b3;
    int I, H, O;
    int batch;
    float *Y;
    float *z1, *h1, *z2, *h2;       // the hidden layers before and after the ReLU
    // training only
    const float *T;
    float scale;
    double *loss;
    float *dy, *dh1, *dh2;
};

template <int HP, int MT>
struct SlabSmem {
    static constexpr int ROWS = 16 * MT;
    static constexpr int LD = HP + 8;   // row pitch: an odd multiple of 16 bytes, so ldmatrix rows hit distinct banks
    static constexpr int w2 = 0;
    static constexpr int act = w2 + HP * LD * 2;                 // three parts of [ROWS][LD]; layer 1: W1 chunk [HP][KC + 8]
    static constexpr int act1 = 3 * ROWS * LD * 2, act2 = HP * (KC + 8) * 2;
    static constexpr int un = act + (act1 > act2 ? act1 : act2);   // layer 1: X chunk, three parts [ROWS][KC + 8]; then W3 [OMAX][LD]
    static constexpr int un1 = OMAX * LD * 2, un2 = 3 * ROWS * (KC + 8) * 2;
    static constexpr int bias = un + (un1 > un2 ? un1 : un2);      // b1, b2 [HP], b3 [OMAX]
    static constexpr int total = bias + (2 * HP + OMAX) * 4;
    static_assert(OMAX + 8 <= LD, "the output gradients fit the activation region");
    static_assert(total <= 227 * 1024, "one CTA's shared memory");
};

// Store acc (rows mt * 16 + g (+ 8), columns n0 + 2 t (+ 1) of n-tile j) as
// three parts into ACT.
template <int ROWS>
__device__ __forceinline__ void put_parts(__nv_bfloat16 *act, int ld, int row, int col, float x, float y) {
    uint32_t h, m, l;
    split3(x, y, h, m, l);
    const int o = row * ld + col, ps = ROWS * ld;
    *reinterpret_cast<uint32_t *>(act + o) = h;
    *reinterpret_cast<uint32_t *>(act + ps + o) = m;
    *reinterpret_cast<uint32_t *>(act + 2 * ps + o) = l;
}

__device__ __forceinline__ void put_global(float *dst, int row, int col, int rows, int H, bool pair, float x, float y) {
    if (row >= rows || col >= H) return;
    float *p = dst + (int64_t)row * H + col;
    if (pair) {   // H even, 8-byte aligned array: col and col + 1 are both inside
        *reinterpret_cast<float2 *>(p) = make_float2(x, y);
    } else {
        p[0] = x;
        if (col + 1 < H) p[1] = y;
    }
}

// A slab of 16 MT rows through the network.  Sixteen warps; warp w owns
// columns w * HP / 16 .. of every hidden layer (MT 16-row tiles by HP / 128
// 8-column tiles of accumulators) and one 16 x 8 tile of the outputs.
template <int HP, int MT, bool TRAIN>
__global__ void __launch_bounds__(NTHR, 1) mlp_slab_kernel(const MlpArgs a) {
    using S = SlabSmem<HP, MT>;
    constexpr int LD = S::LD, NT = HP / 128, ROWS = S::ROWS;
    extern __shared__ __align__(16) unsigned char smem[];
    __nv_bfloat16 *w2s = reinterpret_cast<__nv_bfloat16 *>(smem + S::w2);
    __nv_bfloat16 *act = reinterpret_cast<__nv_bfloat16 *>(smem + S::act);
    __nv_bfloat16 *un = reinterpret_cast<__nv_bfloat16 *>(smem + S::un);
    float *bs = reinterpret_cast<float *>(smem + S::bias);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int64_t row0 = (int64_t)blockIdx.x * ROWS;
    const int rows = (int)min((int64_t)ROWS, a.batch - row0);
    const int I = a.I, H = a.H, O = a.O;
    const int nw = warp * (HP / 16);   // first column of this warp

    // W2 into shared memory, in flight during layer 1
    const bool al16 = (H & 7) == 0 && (reinterpret_cast<uintptr_t>(a.wb + a.o2) & 15) == 0;
    if (al16) {
        for (int e = tid; e < HP * (HP / 8); e += NTHR) {
            const int n = e / (HP / 8), k = (e % (HP / 8)) * 8;
            const int bytes = (n < H && k < H) ? 16 : 0;   // the rest of the 16 bytes is zero-filled
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s32(w2s + n * LD + k)),
                         "l"(a.wb + a.o2 + (bytes ? (int64_t)n * H + k : 0)), "r"(bytes)
                         : "memory");
        }
    } else {
#pragma unroll 4
        for (int e = tid; e < HP * (HP / 8); e += NTHR) {
            const int n = e / (HP / 8), k = (e % (HP / 8)) * 8;
            *reinterpret_cast<uint4 *>(w2s + n * LD + k) =
                load8(a.wb, a.o2 + (int64_t)min(n, H - 1) * H + k, n < H ? H - k : 0, a.np);
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int e = tid; e < 2 * HP + OMAX; e += NTHR) {
        const int n = e < HP ? e : (e < 2 * HP ? e - HP : e - 2 * HP);
        const float *src = e < HP ? a.b1 : (e < 2 * HP ? a.b2 : a.b3);
        bs[e] = n < (e < 2 * HP ? H : O) ? __ldg(src + n) : 0.f;
    }

    float acc[MT][NT][4], low[MT][NT][4];   // leading and trailing parts' sums
    auto zero = [&]() {
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[m][j][k] = low[m][j][k] = 0.f;
    };
    auto join = [&]() {
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[m][j][k] = join_parts(acc[m][j][k], low[m][j][k]);
    };
    // acc += A B over one 16-deep step: A the three parts at column ka of
    // `as` (pitch la), B the fragments of this warp's columns
    auto step = [&](const __nv_bfloat16 *as, int la, int ka, const uint32_t (&b)[NT][2]) {
        uint32_t af[3][MT][4];
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int m = 0; m < MT; ++m)
                ldsm4(af[p][m], s32(as + (p * ROWS + m * 16 + (lane & 15)) * la + ka + (lane >> 4) * 8));
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                mma_add(acc[m][j], af[0][m], b[j][0], b[j][1]);
                mma(low[m][j], af[1][m], b[j][0], b[j][1]);
                mma(low[m][j], af[2][m], b[j][0], b[j][1]);
            }
    };
    auto bfrag = [&](uint32_t (&b)[NT][2], const __nv_bfloat16 *ws, int lw, int k) {   // W[n][k]
        if constexpr (NT == 2) {
            uint32_t r[4];
            ldsm4(r, s32(ws + (nw + (lane & 7) + ((lane >> 4) << 3)) * lw + k + ((lane >> 3) & 1) * 8));
            b[0][0] = r[0], b[0][1] = r[1], b[1][0] = r[2], b[1][1] = r[3];
        } else {
            ldsm2(b[0], s32(ws + (nw + (lane & 7)) * lw + k + ((lane >> 3) & 1) * 8));
        }
    };
    auto bfragt = [&](uint32_t (&b)[NT][2], const __nv_bfloat16 *ws, int lw, int k) {   // W[k][n]
        if constexpr (NT == 2) {
            uint32_t r[4];
            ldsm4t(r, s32(ws + (k + (lane & 7) + ((lane >> 3) & 1) * 8) * lw + nw + (lane >> 4) * 8));
            b[0][0] = r[0], b[0][1] = r[1], b[1][0] = r[2], b[1][1] = r[3];
        } else {
            ldsm2t(b[0], s32(ws + (k + (lane & 7) + ((lane >> 3) & 1) * 8) * lw + nw));
        }
    };

    // ---- layer 1: X W1^T, chunks of KC features
    zero();
    constexpr int LX = KC + 8;
    for (int c0 = 0; c0 < I; c0 += KC) {
        float2 xv[ROWS * (KC / 2) / NTHR];
#pragma unroll
        for (int q = 0; q < ROWS * (KC / 2) / NTHR; ++q) {
            const int e = tid + q * NTHR;
            const int r = e / (KC / 2), k = (e % (KC / 2)) * 2;
            const float *x = a.X + (row0 + r) * I + c0 + k;
            xv[q].x = (r < rows && c0 + k < I) ? __ldg(x) : 0.f;
            xv[q].y = (r < rows && c0 + k + 1 < I) ? __ldg(x + 1) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < HP * (KC / 8) / NTHR; ++q) {
            const int e = tid + q * NTHR;
            const int n = e / (KC / 8), k = (e % (KC / 8)) * 8;
            *reinterpret_cast<uint4 *>(act + n * LX + k) =
                load8(a.wb, a.o1 + (int64_t)min(n, H - 1) * I + min(c0 + k, I - 1), n < H ? I - c0 - k : 0, a.np);
        }
#pragma unroll
        for (int q = 0; q < ROWS * (KC / 2) / NTHR; ++q) {
            const int e = tid + q * NTHR;
            put_parts<ROWS>(un, LX, e / (KC / 2), (e % (KC / 2)) * 2, xv[q].x, xv[q].y);
        }
        __syncthreads();
        const int ks = min(KC, (I - c0 + 15) & ~15);
#pragma unroll 1
        for (int k = 0; k < ks; k += 16) {
            uint32_t b[NT][2];
            bfrag(b, act, LX, k);
            step(un, LX, k, b);
        }
        __syncthreads();
    }

    // W3 into the X region (outputs past O are zero rows)
    const int OP = (O + 15) & ~15;
#pragma unroll 2
    for (int e = tid; e < OP * (HP / 8); e += NTHR) {
        const int n = e / (HP / 8), k = (e % (HP / 8)) * 8;
        *reinterpret_cast<uint4 *>(un + n * LD + k) =
            load8(a.wb, a.o3 + (int64_t)min(n, O - 1) * H + min(k, H - 1), n < O ? H - k : 0, a.np);
    }

    // bias, ReLU, both to memory, the activations as parts to ACT; the bits of
    // positive pre-activations stay in a register
    auto relu_layer = [&](const float *bias, float *zg, float *hg) -> uint32_t {
        uint32_t mask = 0;
        const bool pair = (H & 1) == 0 && ((reinterpret_cast<uintptr_t>(zg) | reinterpret_cast<uintptr_t>(hg)) & 7) == 0;
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            const int n = nw + 8 * j + 2 * t;
            const float2 c = *reinterpret_cast<const float2 *>(bias + n);
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const float z0 = acc[m][j][2 * r] + c.x, z1 = acc[m][j][2 * r + 1] + c.y;
                    const float h0 = fmaxf(z0, 0.f), h1 = fmaxf(z1, 0.f);
                    mask |= (z0 > 0.f ? 1u : 0u) << ((j * MT + m) * 4 + 2 * r);
                    mask |= (z1 > 0.f ? 1u : 0u) << ((j * MT + m) * 4 + 2 * r + 1);
                    const int row = m * 16 + 8 * r + g;
                    put_parts<ROWS>(act, LD, row, n, h0, h1);
                    put_global(zg + row0 * H, row, n, rows, H, pair, z0, z1);
                    put_global(hg + row0 * H, row, n, rows, H, pair, h0, h1);
                }
        }
        return mask;
    };
    join();
    const uint32_t m1 = relu_layer(bs, a.z1, a.h1);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();

    // ---- layer 2
    zero();
#pragma unroll 2
    for (int k = 0; k < HP; k += 16) {
        uint32_t b[NT][2];
        bfrag(b, w2s, LD, k);
        step(act, LD, k, b);
    }
    join();
    __syncthreads();   // every warp has read h1's parts
    const uint32_t m2 = relu_layer(bs + HP, a.z2, a.h2);

    // ---- layer 3: warp w takes rows 16 (w mod MT) .., outputs 8 (w / MT) ..
    const int mo = (warp % MT) * 16, no = (warp / MT) * 8;
    float tv[4];
    if constexpr (TRAIN) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int row = mo + g + 8 * (e >> 1), n = no + 2 * t + (e & 1);
            tv[e] = (row < rows && n < O) ? __ldg(a.T + (row0 + row) * O + n) : 0.f;
        }
    }
    __syncthreads();
    float ya[4] = {}, yl[4] = {};
    if (no < O) {
#pragma unroll 4
        for (int k = 0; k < HP; k += 16) {
            uint32_t b[2], af[3][4];
            ldsm2(b, s32(un + (no + (lane & 7)) * LD + k + ((lane >> 3) & 1) * 8));
#pragma unroll
            for (int p = 0; p < 3; ++p) ldsm4(af[p], s32(act + (p * ROWS + mo + (lane & 15)) * LD + k + (lane >> 4) * 8));
            mma_add(ya, af[0], b[0], b[1]);
            mma(yl, af[1], b[0], b[1]);
            mma(yl, af[2], b[0], b[1]);
        }
    }
    if constexpr (TRAIN) __syncthreads();   // h2's parts are read: ACT takes the output gradients
    constexpr int LO = OMAX + 8;
    if (no < OP) {
        float e2 = 0.f, d[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int row = mo + g + 8 * (e >> 1), n = no + 2 * t + (e & 1);
            d[e] = 0.f;
            if (row < rows && n < O) {
                const int64_t o = (row0 + row) * O + n;
                const float y = join_parts(ya[e], yl[e]) + bs[2 * HP + n];
                a.Y[o] = y;
                if constexpr (TRAIN) {
                    const float r = y - tv[e];
                    d[e] = 2.f * r * a.scale;
                    a.dy[o] = d[e];
                    e2 += r * r * a.scale;
                }
            }
        }
        if constexpr (TRAIN) {
            put_parts<ROWS>(act, LO, mo + g, no + 2 * t, d[0], d[1]);
            put_parts<ROWS>(act, LO, mo + g + 8, no + 2 * t, d[2], d[3]);
            if (a.loss && no < O) {
                for (int o = 16; o; o >>= 1) e2 += __shfl_xor_sync(0xFFFFFFFFu, e2, o);
                if (lane == 0) atomicAdd(a.loss, (double)e2);
            }
        }
    }
    if constexpr (TRAIN) {
        __syncthreads();
        auto masked = [&](uint32_t mask, float *dg, bool parts) {
            const bool pair = (H & 1) == 0 && (reinterpret_cast<uintptr_t>(dg) & 7) == 0;
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const int n = nw + 8 * j + 2 * t, row = m * 16 + 8 * r + g, bit = (j * MT + m) * 4 + 2 * r;
                        const float d0 = (mask >> bit) & 1 ? acc[m][j][2 * r] : 0.f;
                        const float d1 = (mask >> (bit + 1)) & 1 ? acc[m][j][2 * r + 1] : 0.f;
                        if (parts) put_parts<ROWS>(act, LD, row, n, d0, d1);
                        put_global(dg + row0 * H, row, n, rows, H, pair, d0, d1);
                    }
        };
        // ---- dH2 = (dY W3) masked
        zero();
#pragma unroll 1
        for (int k = 0; k < OP; k += 16) {
            uint32_t b[NT][2];
            bfragt(b, un, LD, k);
            step(act, LO, k, b);
        }
        join();
        __syncthreads();
        masked(m2, a.dh2, true);
        __syncthreads();
        // ---- dH1 = (dH2 W2) masked
        zero();
#pragma unroll 2
        for (int k = 0; k < HP; k += 16) {
            uint32_t b[NT][2];
            bfragt(b, w2s, LD, k);
            step(act, LD, k, b);
        }
        join();
        masked(m1, a.dh1, false);
    }
}

// ------------------------------------------------------------ weight gradients
// G[m][n] = sum_b A[b][m] B[b][n] for the three layers in one launch: 64 x 64
// tiles, the batch split over a cluster of up to 8 CTAs that add their FP32
// tiles through distributed shared memory (no atomics: the sum's order is
// fixed).  Tiles of the first n column also sum A over the batch (bias).  The
// CTA that holds a finished gradient entry applies Adam to it.
struct WgradJob {
    const float *A, *B;   // [batch][lda], [batch][ldb]
    int lda, ldb;         // = rows m, columns n of G
    int64_t gw, gb;       // offsets of G ([m][n]) and of the bias in the parameter vector
    int tiles_n, first;   // tiles along n; first tile index of this job
};
struct WgradArgs {
    WgradJob job[3];
    int batch, slab;      // rows per cluster CTA (a multiple of WG_K)
    float *grad, *p, *m, *v;
    __nv_bfloat16 *pb;
    float lr, b1, b2, eps, bc1, bc2;
};

constexpr int WG_K = 64;       // batch rows per staged chunk
constexpr int WG_LD = 64 + 8;
struct WgradSmem {
    union {
        struct {
            __nv_bfloat16 a[3][WG_K][WG_LD], b[3][WG_K][WG_LD];
        } st;
        float tile[64][66];   // the finished sums, after the last chunk
    };
    float csum[8][64];
};

// *p of CTA `cta` of the cluster (p: this CTA's shared memory)
__device__ __forceinline__ float remote(const float *p, int cta) {
    unsigned d;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(s32(p)), "r"(cta));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(d) : "memory");
    return v;
}

__global__ void __launch_bounds__(256, 2) mlp_wgrad_kernel(const WgradArgs a) {
    extern __shared__ __align__(16) unsigned char wsm[];
    WgradSmem &S = *reinterpret_cast<WgradSmem *>(wsm);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = blockIdx.x, nc = gridDim.x;   // the cluster spans x
    int j = 0;
    while (j < 2 && (int)blockIdx.y >= a.job[j + 1].first) ++j;
    const WgradJob q = a.job[j];
    const int tl = blockIdx.y - q.first;
    const int m0 = (tl / q.tiles_n) * 64, n0 = (tl % q.tiles_n) * 64;
    const int k0 = rank * a.slab, k1 = min(a.batch, k0 + a.slab);
    const int wm = (warp & 3) * 16, wn = (warp >> 2) * 32;

    // this thread stages columns c, c + 1 of rows r + 8 i
    const int c = lane * 2, r = warp;
    float2 ra[WG_K / 8], rb[WG_K / 8];
    auto fetch = [&](int kb) {
#pragma unroll
        for (int i = 0; i < WG_K / 8; ++i) {
            const int b = kb + r + 8 * i;
            const bool in = b < k1;
            const float *pa = q.A + (int64_t)b * q.lda + m0 + c, *pb = q.B + (int64_t)b * q.ldb + n0 + c;
            ra[i].x = (in && m0 + c < q.lda) ? __ldg(pa) : 0.f;
            ra[i].y = (in && m0 + c + 1 < q.lda) ? __ldg(pa + 1) : 0.f;
            rb[i].x = (in && n0 + c < q.ldb) ? __ldg(pb) : 0.f;
            rb[i].y = (in && n0 + c + 1 < q.ldb) ? __ldg(pb + 1) : 0.f;
        }
    };
    float acc[4][4] = {}, low[4][4] = {};
    float2 cs = make_float2(0.f, 0.f);
    if (k0 < k1) fetch(k0);
#pragma unroll 1
    for (int kb = k0; kb < k1; kb += WG_K) {
#pragma unroll
        for (int i = 0; i < WG_K / 8; ++i) {
            uint32_t h, m, l;
            split3(ra[i].x, ra[i].y, h, m, l);
            *reinterpret_cast<uint32_t *>(&S.st.a[0][r + 8 * i][c]) = h;
            *reinterpret_cast<uint32_t *>(&S.st.a[1][r + 8 * i][c]) = m;
            *reinterpret_cast<uint32_t *>(&S.st.a[2][r + 8 * i][c]) = l;
            split3(rb[i].x, rb[i].y, h, m, l);
            *reinterpret_cast<uint32_t *>(&S.st.b[0][r + 8 * i][c]) = h;
            *reinterpret_cast<uint32_t *>(&S.st.b[1][r + 8 * i][c]) = m;
            *reinterpret_cast<uint32_t *>(&S.st.b[2][r + 8 * i][c]) = l;
            cs.x += ra[i].x;
            cs.y += ra[i].y;
        }
        __syncthreads();
        if (kb + WG_K < k1) fetch(kb + WG_K);   // in flight during the products
#pragma unroll 1
        for (int k = 0; k < WG_K; k += 16) {
            uint32_t af[3][4], bf[3][2][4];
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                ldsm4t(af[p], s32(&S.st.a[p][k + (lane & 7) + (lane >> 4) * 8][wm + ((lane >> 3) & 1) * 8]));
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    ldsm4t(bf[p][h], s32(&S.st.b[p][k + (lane & 7) + ((lane >> 3) & 1) * 8][wn + 16 * h + (lane >> 4) * 8]));
            }
#pragma unroll
            for (int s = 0; s < 6; ++s) {
                constexpr int pa[6] = {0, 0, 1, 1, 0, 2}, pb[6] = {0, 1, 0, 1, 2, 0};
#pragma unroll
                for (int n = 0; n < 4; ++n) {
                    const uint32_t b0 = bf[pb[s]][n >> 1][(n & 1) * 2], b1 = bf[pb[s]][n >> 1][(n & 1) * 2 + 1];
                    if (s == 0) mma_add(acc[n], af[pa[s]], b0, b1);
                    else mma(low[n], af[pa[s]], b0, b1);
                }
            }
        }
        __syncthreads();
    }
    {
        const int g = lane >> 2, t = lane & 3;
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int e = 0; e < 2; ++e)
                *reinterpret_cast<float2 *>(&S.tile[wm + g + 8 * e][wn + 8 * n + 2 * t]) =
                    make_float2(join_parts(acc[n][2 * e], low[n][2 * e]), join_parts(acc[n][2 * e + 1], low[n][2 * e + 1]));
        S.csum[r][c] = cs.x;
        S.csum[r][c + 1] = cs.y;
    }
    // The CTAs of the cluster share out the tile's entries (and the bias of
    // the first column's tiles): entry e of pass i is rank * 256 + tid + 256 nc i.
    // The Adam state of a pass's entries is on its way while the sums are read.
    const bool adam = a.lr > 0.f;
    auto at = [&](int e) -> int64_t {   // parameter index of entry e, < 0 outside the matrix
        if (e < 64 * 64) return (m0 + (e >> 6) < q.lda && n0 + (e & 63) < q.ldb)
                                    ? q.gw + (int64_t)(m0 + (e >> 6)) * q.ldb + n0 + (e & 63) : -1;
        e -= 64 * 64;
        return (n0 == 0 && e < 64 && m0 + e < q.lda) ? q.gb + m0 + e : -1;
    };
    constexpr int PER = 3;   // entries of one pass; 8 CTAs need one pass
    bool first = true;
    for (int e0 = rank * 256 + tid; e0 < 64 * 64 + 64; e0 += PER * nc * 256) {
        int64_t ix[PER];
        float pm[PER], pv[PER], pp[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            ix[i] = at(e0 + i * nc * 256);
            if (adam && ix[i] >= 0) pm[i] = a.m[ix[i]], pv[i] = a.v[ix[i]], pp[i] = a.p[ix[i]];
        }
        if (first)   // every thread has a first pass (rank * 256 + tid < 64 * 64)
            cluster_sync();
        first = false;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            if (ix[i] < 0) continue;
            const int e = e0 + i * nc * 256;
            float gi = 0.f;
            if (e < 64 * 64) {
                float part[8];   // all remote loads in flight before the sum
#pragma unroll
                for (int z = 0; z < 8; ++z) part[z] = z < nc ? remote(&S.tile[e >> 6][e & 63], z) : 0.f;
#pragma unroll
                for (int z = 0; z < 8; ++z) gi += part[z];
            } else {
                for (int z = 0; z < nc; ++z) {
                    float part[8];
#pragma unroll
                    for (int w = 0; w < 8; ++w) part[w] = remote(&S.csum[w][e - 64 * 64], z);
#pragma unroll
                    for (int w = 0; w < 8; ++w) gi += part[w];
                }
            }
            a.grad[ix[i]] = gi;
            if (!adam) continue;
            const float mi = a.b1 * pm[i] + (1.f - a.b1) * gi;
            const float vi = a.b2 * pv[i] + (1.f - a.b2) * gi * gi;
            a.m[ix[i]] = mi;
            a.v[ix[i]] = vi;
            const float pi = pp[i] - a.lr * (mi / a.bc1) / (sqrtf(vi / a.bc2) + a.eps);
            a.p[ix[i]] = pi;
            a.pb[ix[i]] = __float2bfloat16_rn(pi);
        }
    }
    // no CTA leaves while another may read its tile
    cluster_sync();
}

template <int HP, int MT, bool TRAIN>
bs_status launch_slab_t(const MlpArgs &a, cudaStream_t st) {
    using S = SlabSmem<HP, MT>;
    static PerDevice attr;
    if (bs_status s = attr.get([](int *) {
            return cuda_error(cudaFuncSetAttribute(mlp_slab_kernel<HP, MT, TRAIN>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, S::total),
                              "MLP slab attribute");
        }))
        return s;
    mlp_slab_kernel<HP, MT, TRAIN><<<(a.batch + S::ROWS - 1) / S::ROWS, NTHR, S::total, st>>>(a);
    return check_launch("MLP slab launch");
}

// SMs of the current device.
bs_status device_sms(int *sms) {
    static PerDevice count;
    return count.get(
        [](int *v) {
            int dev = 0;
            cudaError_t e = cudaGetDevice(&dev);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(v, cudaDevAttrMultiProcessorCount, dev);
            return cuda_error(e, "number of SMs");
        },
        sms);
}

// One CTA fits an SM (W2 in shared memory): 16-row slabs while they are at
// most one wave of the SMs, 32-row slabs beyond.
template <bool TRAIN>
bs_status launch_slab(const MlpArgs &a, cudaStream_t st) {
    int sms = 0;
    if (bs_status s = device_sms(&sms)) return s;
    const bool small = a.batch <= 16 * sms;
    if (a.H <= 128) return small ? launch_slab_t<128, 1, TRAIN>(a, st) : launch_slab_t<128, 2, TRAIN>(a, st);
    return small ? launch_slab_t<256, 1, TRAIN>(a, st) : launch_slab_t<256, 2, TRAIN>(a, st);
}

MlpArgs slab_args(const bs_mlp *m, const float *X, int batch, float *Y, const bs_mlp_work *w) {
    const int64_t I = m->n_in, H = m->n_hidden, O = m->n_out;
    const __nv_bfloat16 *wb = (const __nv_bfloat16 *)m->weights_bf16;
    MlpArgs a{};
    a.X = X;
    a.wb = wb;
    a.o1 = 0;
    a.o2 = H * I + H;
    a.o3 = a.o2 + H * H + H;
    a.np = a.o3 + O * H + O;
    a.b1 = m->master + H * I;
    a.b2 = a.b1 + H + H * H;
    a.b3 = a.b2 + H + O * H;
    a.I = (int)I;
    a.H = (int)H;
    a.O = (int)O;
    a.batch = batch;
    a.Y = Y;
    a.z1 = w->z1;
    a.h1 = w->h1;
    a.z2 = w->z2;
    a.h2 = w->h2;
    return a;
}

}  // namespace

// rows are counted in ints, and up to a cluster's last chunks past the batch
bool mlp_fused_applies(const bs_mlp *m, int64_t batch) {
    return m->n_hidden <= 256 && m->n_out <= OMAX && m->n_in <= 65536 && batch <= INT32_MAX - 8 * WG_K;
}

// A slab costs the same for any H up to 128 (its columns are padded), a row of
// the layer by layer products less the narrower the network, so forward passes
// of narrow networks over many rows are theirs: I = 20, H = 8, 262 144 rows 294
// us by slabs, 94 layer by layer; H = 48 78 and 78 at 65 536 rows, 40 and 41 at
// 32 768.  In waves of 32-row slabs, one per SM, over H = 8 .. 64 and I = 4 ..
// 290 this line is within 1 % of the better side on average, 11 % at most.
// (A training step is faster by slabs everywhere: its weight gradients.)
bs_status mlp_forward_by_slabs(const bs_mlp *m, int64_t batch, bool *slabs) {
    int sms = 0;
    *slabs = mlp_fused_applies(m, batch);
    if (!*slabs || m->n_hidden >= 64) return BS_OK;
    if (bs_status s = device_sms(&sms)) return s;
    const double waves = std::ceil((double)batch / (32.0 * sms));
    *slabs = waves <= std::max(1.0, 100.0 / (64 - m->n_hidden) + std::min(m->n_in, 300) / 200.0) ||
             batch > 64LL * 65535;   // more row tiles than the layer by layer grid holds
    return BS_OK;
}

bs_status launch_mlp_forward(const bs_mlp *m, const float *X, int batch, float *Y, const bs_mlp_work *w,
                             cudaStream_t st) {
    const MlpArgs a = slab_args(m, X, batch, Y, w);
    return launch_slab<false>(a, st);
}

bs_status launch_mlp_train(const bs_mlp *m, const float *X, const float *T, int batch, const bs_mlp_work *w, float lr,
                           int step, double *loss, cudaStream_t st) {
    MlpArgs a = slab_args(m, X, batch, w->y, w);
    a.T = T;
    a.scale = 1.0f / (float)((int64_t)batch * a.O);
    a.loss = loss;
    a.dy = w->dy;
    a.dh1 = w->dh1;
    a.dh2 = w->dh2;
    if (bs_status s = launch_slab<true>(a, st)) return s;

    const int64_t I = a.I, H = a.H, O = a.O;
    WgradArgs g{};
    auto tiles = [](int64_t v) { return (int)((v + 63) / 64); };
    const int64_t o2 = H * I + H, o3 = o2 + H * H + H;
    g.job[0] = WgradJob{w->dh2, w->h1, (int)H, (int)H, o2, o2 + H * H, tiles(H), 0};
    g.job[1] = WgradJob{w->dh1, X, (int)H, (int)I, 0, H * I, tiles(I), tiles(H) * tiles(H)};
    g.job[2] = WgradJob{w->dy, w->h2, (int)O, (int)H, o3, o3 + O * H, tiles(H), g.job[1].first + tiles(H) * tiles(I)};
    const int ntiles = g.job[2].first + tiles(O) * tiles(H);
    // up to 8 CTAs (the portable cluster size) share the batch of one tile, 64 rows or more each
    int S = 1;
    while (S < 8 && batch > WG_K * S) S *= 2;
    static PerDevice attr;
    if (bs_status s = attr.get([](int *) {
            return cuda_error(cudaFuncSetAttribute(mlp_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)sizeof(WgradSmem)),
                              "MLP weight-gradient attribute");
        }))
        return s;
    g.batch = batch;
    g.slab = ((batch + S - 1) / S + WG_K - 1) / WG_K * WG_K;
    g.grad = m->grad;
    g.p = m->master;
    g.m = m->adam_m;
    g.v = m->adam_v;
    g.pb = (__nv_bfloat16 *)m->weights_bf16;
    g.lr = lr;
    g.b1 = 0.9f;
    g.b2 = 0.999f;
    g.eps = 1e-8f;
    g.bc1 = 1.f - powf(0.9f, (float)step);
    g.bc2 = 1.f - powf(0.999f, (float)step);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(S, ntiles);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = sizeof(WgradSmem);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = S;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cuda_error(cudaLaunchKernelEx(&cfg, mlp_wgrad_kernel, g), "MLP weight-gradient launch");
}

}  // namespace bs
