// reduce.cuh -- FP64 grid reductions finished by the last CTA, and the device scalar slots
// of the truncated CG / LM driver (Algorithm 1 of arXiv 2103.01767).
//
// Every CTA sums its per-thread values and stores one FP64 partial per column; after a
// __threadfence it bumps a counter, and the CTA that sees the count reach gridDim.x sums all
// partials in FP64 in a fixed order, applies a scalar update to the FP64 slots and resets the
// counter.  Nothing waits on another CTA, so no launch can hang.
#pragma once
#include <cuda_runtime.h>

namespace ptylm {

// FP64 scalar slots on the device.
enum Slot {
    S_F = 0, S_DL2 = 1,                 // forward: f, ||grad_zeta l||^2
    S_RR = 2, S_PAP = 3, S_ALPHA = 4, S_RRNEW = 5, S_BETA = 6,
    S_GG = 7,                           // ||grad f||^2
    S_DD = 8, S_DG = 9, S_DR = 10,      // step dots for the predicted reduction
    S_ER = 11, S_EI = 12, S_NO = 13, S_NR = 14,  // object-error sums
    S_RZ = 15,                          // r.z of the preconditioned CG (= r.r without preconditioner)
    S_GS = 16, S_SS = 17,               // Algorithm 2: g.s and ||s||^2
    S_FMIN = 18,                        // Poisson: sum y - y log y
    S_CG_TIMEOUT = 19,                  // set when a wait of the single-launch CG iteration gave up
    S_CG_DONE = 20, S_CG_ITERS = 21,    // device-side CG stopping: converged flag, iterations run
    S_ZERO = 23,                        // never written after the context's set-up: a skip flag that is not set
    S_COUNT = 24
};

// What the last CTA does with the column sums c[].
enum FinalOp {
    OP_STORE = 0,   // sc[dst + i] = c[i]
    OP_ALPHA = 1,   // p.Ap = c[0];  alpha = r.z / p.Ap
    OP_BETA = 2,    // beta = c[0] / r.z;  r.z = c[0];  r.r = c[1]
    OP_START = 3    // r.z = c[0];  r.r = c[1]   (CG start)
};

// Counters, one per reduction site (kernels on one stream never overlap).
// From CNT_COOP: arrivals and exits of the single-launch CG iteration, and 32 words (one
// 128-byte line) further its released round (cg_iteration.cuh).
// CNT_YBAD: flag set by the measurement copy when an entry of y is negative or not finite.
enum Counter { CNT_FWD = 0, CNT_VEC = 1, CNT_YBAD = 2, CNT_COOP = 32, CNT_COUNT = 96 };
constexpr int kCoopRelease = 32;

constexpr int kMaxReduceWidth = 4;

template <int W>
__device__ __forceinline__ void warp_sum(double (&s)[W]) {
#pragma unroll
    for (int c = 0; c < W; ++c)
        for (int off = 16; off > 0; off >>= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], off);
}

// ---- sums inside a CTA ----------------------------------------------------------------
// GB300 issues one FP64 instruction per warp and scheduler every 64-77 cycles (measured:
// DADD 65 cycles from one warp, 77 from four, 309 from sixteen; conversions the same), so an
// FP64 shuffle tree in each of 16 warps takes 1500 cycles and more.  Per-thread values are
// FP32; inside a CTA they are added as unevaluated pairs of floats whose rounding errors are
// kept exactly (Knuth's two-sum): 48 bits and more, against the 24 of what is summed.  FP64
// takes over at the CTA's total, a few instructions in one warp.
struct SumPair {
    float h, l;   // the sum h + l, |l| tiny
};
// s = a + b and its exact rounding error (0 when s is not finite, so that infinities pass)
__device__ __forceinline__ float two_sum(float a, float b, float& s) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return fabsf(s) <= 3.402823466e38f ? e : 0.0f;
}
__device__ __forceinline__ void pair_add(SumPair& a, float x) {
    float s;
    const float e = two_sum(a.h, x, s);
    a.h = s;
    a.l = __fadd_rn(a.l, e);
}
__device__ __forceinline__ SumPair pair_add(SumPair a, SumPair b) {
    float s;
    const float e = __fadd_rn(two_sum(a.h, b.h, s), __fadd_rn(a.l, b.l));
    SumPair r;
    r.l = two_sum(s, e, r.h);
    return r;
}
template <int LANES>
__device__ __forceinline__ SumPair pair_tree(SumPair v) {   // the same result in every lane of the group
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1)
        v = pair_add(v, SumPair{__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)});
    return v;
}

// FP64 totals of W per-thread pairs over the CTA (blockDim a multiple of 32, <= 512), for
// every lane of warp 0.
template <int W>
__device__ __forceinline__ void block_sum(const SumPair (&v)[W], double (&s)[W]) {
    __shared__ SumPair val[W][16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    SumPair t[W];
#pragma unroll
    for (int c = 0; c < W; ++c) t[c] = pair_tree<32>(v[c]);
    if (lane == 0)
#pragma unroll
        for (int c = 0; c < W; ++c) val[c][warp] = t[c];
    __syncthreads();
    if (warp == 0) {
        float h = 0.0f, l = 0.0f;   // lane c: column c, so that all columns convert together
#pragma unroll
        for (int c = 0; c < W; ++c) {
            const SumPair u = pair_tree<16>(lane < nw ? val[c][lane & 15] : SumPair{0.0f, 0.0f});
            if (lane == c) h = u.h, l = u.l;
        }
        const double d = (double)h + (double)l;
#pragma unroll
        for (int c = 0; c < W; ++c) s[c] = __shfl_sync(0xffffffffu, d, c);
    }
    __syncthreads();
}
template <int W>
__device__ __forceinline__ void block_sum(const float (&f)[W], double (&s)[W]) {
    SumPair v[W];
#pragma unroll
    for (int c = 0; c < W; ++c) v[c] = SumPair{f[c], 0.0f};
    block_sum<W>(v, s);
}

// ---- sums over CTAs, in FP64 -----------------------------------------------------------
// Columns c < W of the partials part[b * stride + c], b < n, summed by the whole CTA with up
// to four warps (one per scheduler) a column; thread 0 receives the result.
template <int W>
__device__ __forceinline__ void sum_partials(const double* part, int stride, int n, double (&s)[W]) {
    __shared__ double tot[W][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int per = nw >= 4 * W ? 4 : nw >= 2 * W ? 2 : 1;   // warps per column
    if (threadIdx.x < 4 * W) tot[threadIdx.x >> 2][threadIdx.x & 3] = 0.0;
    __syncthreads();
    for (int i = warp; i < W * per; i += nw) {
        const int c = i / per, q = i % per;
        double a[1] = {0.0};
        for (int b = 32 * q + lane; b < n; b += 32 * per) a[0] += __ldcg(part + (size_t)b * stride + c);
        warp_sum<1>(a);
        if (lane == 0) tot[c][q] = a[0];
    }
    __syncthreads();
    if (warp == 0) {
        double v = lane < 4 * W ? tot[lane >> 2][lane & 3] : 0.0;
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
#pragma unroll
        for (int c = 0; c < W; ++c) s[c] = __shfl_sync(0xffffffffu, v, 4 * c);
    }
}

__device__ __forceinline__ void apply_final_op(const double* c, int W, double* sc, int dst, int op) {
    switch (op) {
        case OP_STORE:
            for (int i = 0; i < W; ++i) sc[dst + i] = c[i];
            break;
        case OP_ALPHA:
            sc[S_PAP] = c[0];
            sc[S_ALPHA] = sc[S_RZ] / c[0];
            break;
        case OP_BETA:
            sc[S_RRNEW] = c[1];
            sc[S_BETA] = c[0] / sc[S_RZ];
            sc[S_RZ] = c[0];
            sc[S_RR] = c[1];
            break;
        case OP_START:
            sc[S_RZ] = c[0];
            sc[S_RR] = c[1];
            break;
    }
}

// Grid-wide FP64 reduction of W per-thread values (floats or SumPairs) finished by the last
// CTA (see header).  part: [gridDim.x][W] scratch; counter: zero on entry, zero again on
// exit; sc: slots.  Every thread of every CTA must call it exactly once.
template <int W, class V>
__device__ void grid_reduce(const V (&v)[W], double* part, unsigned* counter, double* sc, int dst, int op) {
    __shared__ bool is_last;
    double s[W];
    block_sum<W>(v, s);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int c = 0; c < W; ++c) part[blockIdx.x * W + c] = s[c];
        __threadfence();
        const unsigned prev = atomicAdd(counter, 1u);
        is_last = (prev == gridDim.x - 1);
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    sum_partials<W>(part, W, gridDim.x, s);
    if (threadIdx.x == 0) {
        apply_final_op(s, W, sc, dst, op);
        *counter = 0u;
        __threadfence();
    }
}

}  // namespace ptylm
