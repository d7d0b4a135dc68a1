// Device helpers shared by the kernels: complex arithmetic, in-register
// power-of-two DFTs and the Stockham pass used by both FFT stages.
#pragma once
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace bs {

// Programmatic dependent launch along the pass (channelise, beamspace,
// covariance, solve, output; launch_stage() on the host): a kernel lets the
// next one's CTAs be placed while it runs, and a kernel launched that way waits
// here, before it touches memory, until its predecessor has completed.  What is
// saved is the launch and ramp-up of each stage: a pass of 64 pairs 29.8 -> 22.4 us,
// of 1024 pairs at N = 256 89 -> 81 us.  Both are no-ops in an ordinary launch;
// which stages are launched so is a question of their sizes (launch_beamspace()
// in internal.h).
// Arrays that an earlier stage of the pass writes are read by ordinary (or
// .cg / .cs) loads only, through pointers that are not const __restrict__: the
// read-only path (ld.global.nc: __ldg, or the compiler's choice for such a
// pointer) is for data that nothing writes while the kernel lives, and its life
// begins before the predecessor's ends.  The plan's tables may take it.
__device__ __forceinline__ void let_dependents_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_predecessor() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    let_dependents_launch();
}

// Barrier of the cluster, with release and acquire.  Not .aligned: it follows
// code that only some lanes of a warp run, and that form is undefined unless the
// whole warp arrives together.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Complex sums as one packed FP32x2 instruction (sm_100 and later): the same
// round-to-nearest result per component as two scalar adds, in half the
// issue slots, which the FFT kernels (issue-bound) are short of.
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
    return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
__device__ __forceinline__ float2 cscale(float2 a, float s) { return __fmul2_rn(a, make_float2(s, s)); }

// x * exp(-2 pi i e / 16); e is a compile-time constant at every call site
// (fully unrolled loops), so the switch folds to a few instructions.
__device__ __forceinline__ float2 twiddle16(int e, float2 x) {
    constexpr float C1 = 0.92387953251128674f;  // cos(pi/8)
    constexpr float S1 = 0.38268343236508978f;  // sin(pi/8)
    constexpr float H = 0.70710678118654752f;   // sqrt(1/2)
    float c, s;
    switch (e & 15) {
        case 0: return x;
        case 4: return make_float2(x.y, -x.x);
        case 8: return make_float2(-x.x, -x.y);
        case 12: return make_float2(-x.y, x.x);
        case 2: return make_float2((x.x + x.y) * H, (x.y - x.x) * H);
        case 6: return make_float2((x.y - x.x) * H, -(x.x + x.y) * H);
        case 10: return make_float2(-(x.x + x.y) * H, (x.x - x.y) * H);
        case 14: return make_float2((x.x - x.y) * H, (x.x + x.y) * H);
        case 1: c = C1; s = S1; break;
        case 3: c = S1; s = C1; break;
        case 5: c = -S1; s = C1; break;
        case 7: c = -C1; s = S1; break;
        case 9: c = -C1; s = -S1; break;
        case 11: c = -S1; s = -C1; break;
        case 13: c = S1; s = -C1; break;
        default: c = C1; s = -S1; break;  // 15
    }
    // x * (c - i s)
    return make_float2(x.x * c + x.y * s, x.y * c - x.x * s);
}

// Forward DFT of R points held in registers, natural order in and out
// (radix-2 decimation in frequency, recursion resolved at compile time).
template <int R>
struct RegDFT {
    static __device__ __forceinline__ void run(float2 *v) {
        float2 e[R / 2], o[R / 2];
#pragma unroll
        for (int k = 0; k < R / 2; ++k) {
            e[k] = cadd(v[k], v[k + R / 2]);
            o[k] = twiddle16(k * (16 / R), csub(v[k], v[k + R / 2]));
        }
        RegDFT<R / 2>::run(e);
        RegDFT<R / 2>::run(o);
#pragma unroll
        for (int k = 0; k < R / 2; ++k) {
            v[2 * k] = e[k];
            v[2 * k + 1] = o[k];
        }
    }
};
template <>
struct RegDFT<1> {
    static __device__ __forceinline__ void run(float2 *) {}
};

// Radix schedule of an n-point FFT (n = 2^k, 2..4096): passes of radix 16
// first, then one smaller pass for the remaining factor.
template <int n>
struct Radix {
    static constexpr int npass = (n <= 16) ? 1 : (n <= 256) ? 2 : 3;
    static constexpr int r0 = (n <= 16) ? n : 16;
    static constexpr int r1 = (npass < 2) ? 1 : (npass == 2 ? n / 16 : 16);
    static constexpr int r2 = (npass < 3) ? 1 : n / 256;
    static_assert(n >= 2 && n <= 4096 && (n & (n - 1)) == 0, "n must be a power of two <= 4096");
};

// w[r] = tw[r * e] for r < R (R = 2, 4, 8, 16; r * e < table length).
// Only w^1, w^4, w^8 and w^12 come from the table; the other powers are
// products of at most three table entries, which keeps their error within
// a few FP32 ulps while cutting the table loads per butterfly from R-1 to
// at most 4 (the loads of a warp hit scattered table lines).
template <int R, class Tw>
__device__ __forceinline__ void twiddle_powers(Tw tw, int e, float2 (&w)[R]) {
    w[0] = make_float2(1.f, 0.f);
    w[1] = tw(e);
    if constexpr (R >= 4) {
        w[2] = cmul(w[1], w[1]);
        w[3] = cmul(w[2], w[1]);
    }
    if constexpr (R >= 8) {
        w[4] = tw(4 * e);
#pragma unroll
        for (int r = 5; r < 8; ++r) w[r] = cmul(w[4], w[r - 4]);
    }
    if constexpr (R >= 16) {
        w[8] = tw(8 * e);
        w[12] = tw(12 * e);
#pragma unroll
        for (int r = 9; r < 12; ++r) w[r] = cmul(w[8], w[r - 8]);
#pragma unroll
        for (int r = 13; r < 16; ++r) w[r] = cmul(w[12], w[r - 12]);
    }
}

// One Stockham autosort pass (decimation in time) of an n-point FFT over a
// batch of `ncols` independent columns, processed by `nthr` threads:
//   butterfly j < n/R of column c reads a[j + r n/R] (r < R), multiplies
//   by w^(r * (j mod Ns)) with w = e^{-2 pi i/(Ns R)}, takes the R-point DFT
//   and writes b[(j/Ns) Ns R + (j mod Ns) + r Ns].
// Ns is the product of the radices of the earlier passes.  `load(c, idx)`
// and `store(c, idx, v)` address the source and destination; with
// kSyncMid the pass reads everything into registers, synchronises the CTA
// and then writes (in-place passes through shared memory).
// kColFast: butterfly id -> (column = id % ncols) else (column = id / (n/R)).
// tw(k) = e^{-2 pi i k / n}, k < n.
template <int n, int R, int Ns, int ncols, int nthr, bool kColFast, bool kSyncMid, class Tw,
          class Load, class Store>
__device__ __forceinline__ void stockham_pass_tw(int tid, Tw tw, Load load, Store store) {
    constexpr int nb = ncols * (n / R);
    static_assert(nb % nthr == 0, "butterflies must divide evenly over threads");
    constexpr int bpt = nb / nthr;
    float2 v[bpt][R];
#pragma unroll
    for (int b = 0; b < bpt; ++b) {
        const int id = tid + b * nthr;
        const int c = kColFast ? (id % ncols) : (id / (n / R));
        const int j = kColFast ? (id / ncols) : (id % (n / R));
#pragma unroll
        for (int r = 0; r < R; ++r) v[b][r] = load(c, j + r * (n / R));
        if (Ns > 1) {
            float2 w[R];
            twiddle_powers(tw, (j % Ns) * (n / (Ns * R)), w);
#pragma unroll
            for (int r = 1; r < R; ++r) v[b][r] = cmul(v[b][r], w[r]);
        }
        RegDFT<R>::run(v[b]);
    }
    if (kSyncMid) __syncthreads();
#pragma unroll
    for (int b = 0; b < bpt; ++b) {
        const int id = tid + b * nthr;
        const int c = kColFast ? (id % ncols) : (id / (n / R));
        const int j = kColFast ? (id / ncols) : (id % (n / R));
        const int k = j % Ns;
        const int base = (j / Ns) * Ns * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) store(c, base + r * Ns, v[b][r]);
    }
}

// The pass with the twiddles in global memory, tw[k] = e^{-2 pi i k / n}.
template <int n, int R, int Ns, int ncols, int nthr, bool kColFast, bool kSyncMid, class Load, class Store>
__device__ __forceinline__ void stockham_pass(int tid, const float2 *__restrict__ tw, Load load, Store store) {
    stockham_pass_tw<n, R, Ns, ncols, nthr, kColFast, kSyncMid>(
        tid, [tw](int k) { return __ldg(&tw[k]); }, load, store);
}

// The sum of a product's leading parts plus that of its trailing parts.  The
// leading parts are infinite or NaN where the values are (a quiet NaN's leading
// part is one), so an infinite leading sum is the result; the trailing parts
// hold zeros, whose products with an infinity are NaN.
__device__ __forceinline__ float join_parts(float lead, float trail) { return isinf(lead) ? lead : lead + trail; }
__device__ __forceinline__ float2 join_parts(float2 lead, float2 trail) {
    return make_float2(join_parts(lead.x, trail.x), join_parts(lead.y, trail.y));
}

// Double-float values (h + l, |l| <= ulp(h)/2): GB300's FP64 pipe is
// narrow, so the covariance epilogues assemble R in FP32 pairs and convert
// only the final value of each entry to FP64.
struct DF {
    float h, l;
};
__device__ __forceinline__ DF df_norm(float h, float l) {   // |l| small against h
    const float s = h + l;
    return DF{s, l - (s - h)};
}
__device__ __forceinline__ DF df_add(DF a, DF b) {
    const float s = a.h + b.h;
    const float bb = s - a.h;
    const float e = (a.h - (s - bb)) + (b.h - bb) + a.l + b.l;
    return df_norm(s, e);
}
__device__ __forceinline__ DF df_mul(DF a, DF b) {
    const float p = a.h * b.h;
    float e = fmaf(a.h, b.h, -p);
    e = fmaf(a.h, b.l, e);
    e = fmaf(a.l, b.h, e);
    return df_norm(p, e);
}
__device__ __forceinline__ double df_to_double(DF a) { return (double)a.h + (double)a.l; }
// host side: a double as a double-float (for kernel parameters)
inline DF df_from_double(double v) {
    const float h = (float)v;
    return DF{h, (float)(v - (double)h)};
}

// Padded shared-memory row index: one spare slot every 16 rows spreads the
// radix-16 strided accesses over the banks.
__device__ __forceinline__ int padrow(int t) { return t + (t >> 4); }
__host__ __device__ constexpr int padded_len(int n) { return n + n / 16; }

}  // namespace bs
