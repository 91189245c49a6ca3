// conv_tc.cu -- tensor-core 3x3 convolutions of the learned initialisation (see conv_tc.h).
//
// Implicit GEMM.  A tile is 16 x 8 points of an output sub-lattice (the output grid itself, or
// one parity class of it), i.e. 128 GEMM rows = 128 TMEM lanes, with up to four accumulators
// ("phases") of N columns each.  A persistent CTA per SM runs over tiles in three roles: one
// thread loads, one issues the MMAs, eight warps write the results; the accumulators are
// double buffered, so a tile's epilogue overlaps the next tile's MMAs.  The K loop runs over
// input channels, 16 per pipeline stage.  Per stage the TMA producer loads
//   * the input: boxes of (8 channels) x (9 or 10 columns) x (17 or 18 rows) from the map or its
//     parity planes.  In the canonical no-swizzle K-major layout a pixel's 8 channels are 16
//     bytes and 8 pixels a core matrix, so with 8-pixel tile rows the box row is the stride
//     between core matrices and a tap's row and column shift are a plain descriptor offset: one
//     box serves all taps.  Out-of-range coordinates fill zeros, the convolution's zero padding;
//   * the bfloat16 weights of all nine taps for those 16 channels (18 contiguous bulk copies);
// and the MMA thread issues, per (phase, tap) group and per split (hi, lo), a 128 x N x 16
// tcgen05.mma into the phase's accumulator.  Mbarrier rings (full / empty) pipeline the stages.
//
// Layer forms (s: stride-2 layer, u: upsampling layer):
//   forward s:  output (a, b) reads input (2a+u-1, 2b+v-1): the four parity planes;
//   forward u:  four phases (py, px) of the output (2a+py, 2b+px) read the low-resolution
//               input at (a + floor((py+u-1)/2), b + floor((px+v-1)/2));
//   input gradient s: four phases (qy, qx) of the input grid, (2a'+qy, 2b'+qx), collect dy at
//               (a' + e, b' + f), e, f in {0, 1}, from the taps with matching parity;
//   input gradient u: a stride-1 correlation of dy at full resolution whose 2 x 2 sums (taken
//               with warp shuffles: a warp holds four rows of the tile) give the gradient
//               of the low-resolution input.
//
// Forward pass of 225 patterns (widths 64/128/256), layers 1-5: 111, 71, 73, 145, 208 us; with
// one CTA per tile, 16-pixel tile rows, a copy of the input per column shift and operands
// moved to uniform registers MMA by MMA 179, ~100, 115, 294, ~343 us.  Layers 4 and 5 run at
// about 0.75 of the rate their MMAs allow, 1-3 are bound by their epilogues and loads.
// The weight gradient is a GEMM over pixels with MN-major operands (k_wgrad_tc).
#include "conv_tc.h"

#include <cuda.h>

#include <algorithm>
#include <cstring>

#include "tc_common.cuh"

namespace ptylm {

namespace {

using namespace tc;

constexpr int kThreads = 128;
constexpr int kEpiThreads = 256;      // epilogue: two groups of four warps, which share the 128 lanes
constexpr int kConvThreads = kEpiThreads + 64;   // ... the TMA warp, the MMA warp
constexpr int kMaxStage = 8;
constexpr int kMaxCopy = 4;
constexpr int kMaxGroup = 36;
constexpr int kSmemLimit = 232448;    // shared memory a CTA may use (static + dynamic)
constexpr int kOneCtaPerSm = 120 * 1024;  // dynamic request that leaves no room for a second CTA

enum { EPI_HIDDEN = 0, EPI_LAST = 1, EPI_BWD = 2, EPI_POOL = 3 };

struct Copy {
    int8_t row0, col;  // box start relative to the tile origin (sub-lattice units)
    int8_t par;        // parity plane of a parity-split map, -1 for a plain map
};
struct Group {
    uint8_t phase, copy, row, col, tap;
};

struct ConvArgs {
    int tiles_x, tiles_y;  // 16 x 8 (rows x columns) tiles per image
    int n_img, pgroups, n_zt;   // tiles: images x space, phase groups, column (channel) tiles
    int n_copy, split, rows, px, ksteps, N, P, n_acc, tmem_cols, n_stage;
    int a_slot;       // bytes of one (copy, chunk) box, rows * px * 16 rounded up to 128
    int a_bytes;      // A bytes of a stage: split * n_copy * 2 * a_slot
    int stage_bytes;  // a_bytes + 2 * 9 * N * 16
    int gstart[5];    // groups sorted by phase: phase p owns [gstart[p], gstart[p+1])
    Copy copy[kMaxCopy];
    Group group[kMaxGroup];
    int mode, osy, osx;
    int8_t opy[4], opx[4];
    int oH, oW, oC;  // output tensor (chunk-major pair, or FP32 planes for the last layer)
    int out_par;     // layout of (out_hi, out_lo)
    __nv_bfloat16* out_hi;
    __nv_bfloat16* out_lo;
    __nv_bfloat16* out_phi;  // optional parity-split copy of the output
    __nv_bfloat16* out_plo;
    float* out32;
    const __nv_bfloat16* wts;  // weights [9][K/8][R][8]
    int wK8, wR;
    const float* bias;
    int relu;
    const __nv_bfloat16* m_hi;
    const __nv_bfloat16* m_lo;
    int m_par;
    float* db_part;
    unsigned* err;
    unsigned spin;
};

struct ConvParams {
    CUtensorMap amap[2];  // the input tensor: hi, lo
    ConvArgs a;
    uint4 mma[2 * kMaxGroup];   // per group and split: offsets of A and B in a stage (16-byte units), column, accumulate
};

__device__ __forceinline__ unsigned char* align1024(unsigned char* p) {
    return reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// 16 channels from ch0 of pixel (y, x) into the output pair (and its parity copy)
__device__ __forceinline__ void store_out16(const ConvArgs& a, int n, int y, int x, int ch0, const float* v) {
    const int C8 = a.oC >> 3;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        store_pair8(a.out_hi, a.out_lo, chunk_at(a.out_par, C8, a.oH, a.oW, n, y, x, (ch0 >> 3) + q), v + 8 * q);
        if (a.out_phi) store_pair8(a.out_phi, a.out_plo, chunk_at(1, C8, a.oH, a.oW, n, y, x, (ch0 >> 3) + q), v + 8 * q);
    }
}

// the epilogue warps only
__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory"); }

// One tile's accumulators (at `lane_base`, this warp's TMEM lanes) through the layer's epilogue.
// Warps w and w + 4 hold the same 128 pixels and take 32 columns each of every 64; what a step
// reads from memory (the ReLU mask) is fetched before its accumulators are waited for.  With
// four warps and the mask read inside the step the input gradients of a batch of 64 took 223,
// 136, 76 and 128 us, now 138, 83, 52 and 82.
__device__ __forceinline__ void conv_epilogue(const ConvArgs& a, uint32_t lane_base, int n, int a0, int b0, int pg, int o0,
                                              size_t part, float (*red)[256]) {
    const int warp = (threadIdx.x >> 5) & 3, grp = threadIdx.x >> 7, lane = threadIdx.x & 31;
    const int r = (threadIdx.x & 127) >> 3, c = threadIdx.x & 7;
    const bool pooled = a.mode == EPI_POOL, writer = !pooled || ((r | c) & 1) == 0;
    if (a.mode >= EPI_BWD) {
        for (int i = threadIdx.x; i < 4 * 256; i += kEpiThreads) (&red[0][0])[i] = 0.0f;
        epilogue_sync();
    }
    for (int ph = 0; ph < a.P; ++ph) {
        const int phase = pg * a.P + ph;
        const int oy = a.osy * (a0 + r) + a.opy[phase], ox = a.osx * (b0 + c) + a.opx[phase];
        const int py = pooled ? (a0 + r) >> 1 : oy, px = pooled ? (b0 + c) >> 1 : ox;
        auto columns16 = [&](float (&v)[16], const uint4 (&mk)[4], int cb) {
            const int ch0 = o0 + cb;
            if (a.mode == EPI_HIDDEN) {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    v[j] += __ldg(a.bias + ch0 + j);
                    if (a.relu) v[j] = fmaxf(v[j], 0.0f);
                }
                store_out16(a, n, oy, ox, ch0, v);
            } else if (a.mode == EPI_LAST) {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (ch0 + j < a.oC)
                        a.out32[(((size_t)n * a.oC + ch0 + j) * a.oH + oy) * a.oW + ox] = v[j] + a.bias[ch0 + j];
            } else {
                if (pooled) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        v[j] += __shfl_xor_sync(0xffffffffu, v[j], 1);
                        v[j] += __shfl_xor_sync(0xffffffffu, v[j], 8);
                    }
                }
                if (writer) {
                    bool m[16];
#pragma unroll
                    for (int q = 0; q < 2; ++q) mask8(mk[2 * q], mk[2 * q + 1], m + 8 * q);
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = m[j] ? v[j] : 0.0f;
                    store_out16(a, n, py, px, ch0, v);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = 0.0f;
                }
                // column sums over the warp: each exchange halves the columns a lane carries on
                // (16 shuffles, against 80 for sixteen separate trees)
#pragma unroll
                for (int half = 8; half >= 1; half >>= 1) {
                    const bool up = lane & (2 * half);
#pragma unroll
                    for (int j = 0; j < half; ++j) {
                        const float keep = up ? v[j + half] : v[j], send = up ? v[j] : v[j + half];
                        v[j] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * half);
                    }
                }
                v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
                if (!(lane & 1)) red[warp][cb + (lane >> 1)] += v[0];
            }
        };
        for (int cb = 32 * grp; cb < a.N; cb += 64) {
            float w[2][16];
            uint4 mk[2][4];
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (cb + 16 * q < a.N) tmem_ld16_start(lane_base + (uint32_t)(ph * a.N + cb + 16 * q), w[q]);
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    mk[q][2 * h] = mk[q][2 * h + 1] = make_uint4(0, 0, 0, 0);
                    if (a.mode >= EPI_BWD && writer && cb + 16 * q < a.N) {
                        const size_t o = chunk_at(a.m_par, a.oC >> 3, a.oH, a.oW, n, py, px, ((o0 + cb) >> 3) + 2 * q + h);
                        mk[q][2 * h] = __ldg(reinterpret_cast<const uint4*>(a.m_hi + o));
                        mk[q][2 * h + 1] = __ldg(reinterpret_cast<const uint4*>(a.m_lo + o));
                    }
                }
#pragma unroll
            for (int q = 0; q < 2; ++q) tmem_ld_wait16(w[q]);
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (cb + 16 * q < a.N) columns16(w[q], mk[q], cb + 16 * q);
        }
    }
    if (a.mode >= EPI_BWD) {
        epilogue_sync();
        for (int ch = threadIdx.x; ch < a.N; ch += kEpiThreads)
            a.db_part[part * a.oC + o0 + ch] = red[0][ch] + red[1][ch] + red[2][ch] + red[3][ch];
        epilogue_sync();   // before the next tile clears red
    }
}

__global__ void __launch_bounds__(kConvThreads, 1) k_conv_tc(const __grid_constant__ ConvParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = align1024(smem_raw);
    __shared__ uint64_t full[kMaxStage], empty[kMaxStage], acc_full[2], acc_empty[2], done;
    __shared__ uint32_t tbase;
    __shared__ int abort_flag, epilogue_abort, issued, consumed;
    __shared__ float red[4][256];
    const ConvArgs& a = p.a;
    const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int per_img = a.tiles_x * a.tiles_y, n_xt = per_img * a.n_img;
    const int pg = blockIdx.y, total = n_xt * a.n_zt;   // channel tiles fastest: they share the input
    const int S = a.n_stage;

    if (warp == 0) tmem_alloc(smem_u32(&tbase), a.tmem_cols);
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            bar_init(smem_u32(&full[s]), 1);
            bar_init(smem_u32(&empty[s]), 1);
        }
        for (int s = 0; s < 2; ++s) {
            bar_init(smem_u32(&acc_full[s]), 1);
            bar_init(smem_u32(&acc_empty[s]), kEpiThreads / 32);
        }
        bar_init(smem_u32(&done), 1);
        bar_fence_init();
        abort_flag = 0;
        epilogue_abort = 0;
        issued = 0;
        consumed = 0;
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = (uint32_t)uniform((int)tbase);
    const uint32_t sbase = (uint32_t)uniform((int)smem_u32(smem));
    volatile int* aborted = &abort_flag;

    if (warp == kEpiThreads / 32) {
        if (elect_one()) {   // TMA producer
            const uint32_t abytes = (uint32_t)(a.split * a.n_copy * 2 * a.rows * a.px * 16);
            int it = 0, s = 0;
            uint32_t par = 1;   // a fresh barrier's previous phase counts as complete
            for (int t = blockIdx.x; t < total && !*aborted; t += gridDim.x) {
                const int xt = t / a.n_zt, o0 = (t - xt * a.n_zt) * a.N;
                const int n = xt / per_img, tt = xt - n * per_img, ty = tt / a.tiles_x;
                const int a0 = ty * 16, b0 = (tt - ty * a.tiles_x) * 8;
                const int nb = min(a.N, a.wR - o0);   // weight rows present (the rest is never read into D)
                // a tap's weights of the stage's two chunks are contiguous when the tile holds all rows
                const int wq = nb == a.wR && nb == a.N ? 1 : 2;
                for (int ks = 0; ks < a.ksteps; ++ks, ++it) {
                    const uint32_t st = sbase + s * a.stage_bytes, fb = smem_u32(&full[0]) + 8 * s;
                    if (!bar_wait(smem_u32(&empty[0]) + 8 * s, par, a.spin)) {
                        atomicOr(a.err, 1u);
                        abort_flag = 1;
                    }
                    if (*aborted) break;
                    bar_expect_tx(fb, abytes + 18u * (uint32_t)nb * 16u);
                    for (int sp = 0; sp < a.split; ++sp)
                        for (int j = 0; j < a.n_copy; ++j) {
                            const uint32_t dst = st + (uint32_t)((sp * a.n_copy + j) * 2 * a.a_slot);
                            const Copy cp = a.copy[j];
                            const int x = (b0 + cp.col) * 8, y = a0 + cp.row0;
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const int chunk = 2 * ks + q;
                                tma_load_4d(dst + q * a.a_slot, &p.amap[sp], x, y, cp.par < 0 ? chunk : 4 * chunk + cp.par, n, fb);
                            }
                        }
                    const uint32_t bdst = st + a.a_bytes;
                    for (int w = 0; w < 9; ++w)
                        for (int q = 0; q < wq; ++q) {
                            const __nv_bfloat16* src = a.wts + (((size_t)w * a.wK8 + 2 * ks + q) * a.wR + o0) * 8;
                            bulk_load(bdst + (uint32_t)((2 * w + q) * a.N * 16), src, (uint32_t)nb * (wq == 1 ? 32u : 16u), fb);
                        }
                    if (++s == S) s = 0, par ^= 1u;
                }
            }
            issued = it;
        }
        __syncwarp();
    } else if (warp == kEpiThreads / 32 + 1) {
        if (elect_one()) {
            // MMA issuer.  The tensor pipe takes an MMA every 44 (N <= 32), 48 (N = 64) or 64 cycles
            // (N = 128; the shared-memory reads of A and B bound the smaller N), so issuing one may
            // cost no more: the operand offsets come from a table in the kernel's parameters, in the
            // descriptors' 16-byte units, and everything they are added to is a loop counter, a
            // parameter or a block index, which stays in uniform registers (tc_common.cuh).
            const uint32_t idesc = idesc_bf16(128, a.N, 0, 0);
            const int i0 = a.gstart[pg * a.P] * a.split, i1 = a.gstart[pg * a.P + a.P] * a.split;
            int it = 0, s = 0, buf = 0;
            uint32_t par = 0, apar = 1;
            bool gone = false;
            for (int t = blockIdx.x; t < total && !gone; t += gridDim.x) {
                if (!bar_wait(smem_u32(&acc_empty[0]) + 8 * buf, apar, a.spin)) {
                    atomicOr(a.err, 64u);
                    abort_flag = 1;
                    break;
                }
                fence_after();
                const uint32_t d0 = tmem + (uint32_t)(buf * a.P * a.N);
                for (int ks = 0; ks < a.ksteps; ++ks, ++it) {
                    if (!bar_wait(smem_u32(&full[0]) + 8 * s, par, a.spin)) {
                        atomicOr(a.err, 2u);
                        abort_flag = 1;
                        gone = true;
                        break;
                    }
                    fence_after();
                    const uint32_t st = sbase + s * a.stage_bytes;
                    const uint64_t ad0 = sdesc(st, (uint32_t)a.a_slot, (uint32_t)a.px * 16u);
                    const uint64_t bd0 = sdesc(st + a.a_bytes, (uint32_t)a.N * 16u, 128u);
#pragma unroll 4
                    for (int i = i0; i < i1; ++i) {
                        const uint4 m = p.mma[i];
                        mma_bf16(d0 + m.z, ad0 + m.x, bd0 + m.y, idesc, m.w | (uint32_t)ks);
                    }
                    mma_commit(smem_u32(&empty[0]) + 8 * s);
                    if (++s == S) s = 0, par ^= 1u;
                }
                mma_commit(smem_u32(&acc_full[0]) + 8 * buf);
                if (++buf == a.n_acc) buf = 0, apar ^= 1u;
                gone = gone || *aborted;
            }
            consumed = it;
            mma_commit(smem_u32(&done));
        }
        __syncwarp();
    } else {
        int buf = 0;
        uint32_t fpar = 0;
        for (int t = blockIdx.x; t < total; t += gridDim.x) {
            const int xt = t / a.n_zt, o0 = (t - xt * a.n_zt) * a.N;
            const int n = xt / per_img, tt = xt % per_img;
            // all epilogue warps leave together (the epilogue has barriers of its own): the flag they
            // test is only written between the barrier at the end of a tile and the next one
            const bool ok = bar_wait(smem_u32(&acc_full[buf]), fpar, a.spin);
            if (!ok && lane == 0) {
                atomicOr(a.err, 4u);
                abort_flag = 1;
            }
            if (lane == 0 && *aborted) *(volatile int*)&epilogue_abort = 1;
            epilogue_sync();
            if (*(volatile int*)&epilogue_abort) break;
            fence_after();
            conv_epilogue(a, tmem + (uint32_t)(buf * a.P * a.N) + ((uint32_t)(32 * (warp & 3)) << 16), n, (tt / a.tiles_x) * 16,
                          (tt % a.tiles_x) * 8, pg, o0, (size_t)pg * n_xt + xt, red);
            fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive(smem_u32(&acc_empty[buf]));
            if (++buf == a.n_acc) buf = 0, fpar ^= 1u;
            epilogue_sync();
        }
    }
    const bool ok = bar_wait(smem_u32(&done), 0, a.spin);
    if (!ok && lane == 0) atomicOr(a.err, 4u);
    fence_after();
    __syncthreads();
    if ((*aborted || !ok) && threadIdx.x == 0) {
        // let the copies still in flight land before the CTA's shared memory is released
        for (int it = consumed; it < issued; ++it) bar_wait(smem_u32(&full[it % S]), (it / S) & 1, a.spin);
    }
    fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, a.tmem_cols);
}

// ---------------------------------------------------------------------------------------
// Weight gradient: D_t[row][col] = sum over pixels p of A_t[row][p] B_t[col][p], one TMEM
// accumulator of N columns per tap t.  One operand is the output gradient dy at the forward
// pass's output pixels (shared by all taps), the other the tap-shifted input.  Both are stored
// pixel-major with channels contiguous, i.e. MN-major operands; K is the pixel index, 16
// pixels (one row of the tile) per MMA.  The input is loaded once per (parity) plane with the
// columns the shifts reach, 18 pixels a row: in the no-swizzle layout a pixel is 16 bytes, so a
// column shift is a descriptor offset like a row shift.  An MMA of 128 rows takes the tensor
// pipe 64 cycles at N = 128, 48 at 64 and still 44 at 32, so a CTA holds as many columns as fit:
// all nine taps up to N = 56, else the three taps of one kernel row with up to 128 columns
// (nine taps of 32 columns before: layers 2-5 at batch 64 took 96, ~212, ~212 and 600 us, now
// 47, 55, 84 and 128).
// A CTA runs over a strided subset of the pixel tiles and writes its partial sums;
// k_wgrad_reduce adds them in a fixed order.  Rows beyond the real channel count read whatever
// lies next in shared memory and are discarded.

struct WgArgs {
    int tiles_x, tiles_y, phases, n_tiles, rows_px;
    int w2;           // 0: A = dy (rows = output channels), B = input; 1: swapped
    int taps;         // taps per CTA: 9, or 3 (one kernel row u = kind % 3)
    int up;
    int g_real;       // dy chunk boxes per split
    int x_real;       // input chunk boxes per plane and split
    int planes, rows, N, c_tiles, tmem_cols, n_stage;
    int g_slot, x_slot, g_bytes, x_bytes, stage_bytes;
    int n_split;      // gridDim.x
    uint32_t tap_at[3][4][9];   // kernel row (0 if all), phase, tap: offset of its input in a stage, 16-byte units
    int Co, Ci;
    float* part;
    unsigned* err;
    unsigned spin;
};

constexpr int kWgPx = 18, kWgPitch = kWgPx * 16;   // input pixels and bytes of a loaded row (8 channels)

// floor((p + t - 1) / 2) for phase p in {0, 1} and tap t: the input pixel a tap of an upsampling layer reads
__device__ __forceinline__ int tap_shift(int p, int t) { return (p + t + 1) / 2 - 1; }

struct WgParams {
    CUtensorMap gmap[2];  // dy (or its parity copy): hi, lo
    CUtensorMap xmap[2];  // the layer input: hi, lo
    WgArgs a;
};

__global__ void __launch_bounds__(kThreads, 1) k_wgrad_tc(const __grid_constant__ WgParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = align1024(smem_raw);
    __shared__ uint64_t full[kMaxStage], empty[kMaxStage], done;
    __shared__ uint32_t tbase;
    __shared__ int abort_flag, issued, consumed;
    const WgArgs& a = p.a;
    const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int split = blockIdx.x, kind = blockIdx.y * gridDim.z + blockIdx.z;
    const int S = a.n_stage;
    const int u0 = a.taps == 3 ? (int)blockIdx.z : -1;     // the kernel row, -1: all
    const int mt = blockIdx.y / a.c_tiles, nt = blockIdx.y % a.c_tiles;
    const int o0 = a.w2 ? nt * a.N : mt * 128, c0 = a.w2 ? mt * 128 : nt * a.N;
    const int per_phase = a.tiles_x * a.tiles_y;

    if (warp == 0) tmem_alloc(smem_u32(&tbase), a.tmem_cols);
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            bar_init(smem_u32(&full[s]), 1);
            bar_init(smem_u32(&empty[s]), 1);
        }
        bar_init(smem_u32(&done), 1);
        bar_fence_init();
        abort_flag = 0;
        issued = 0;
        consumed = 0;
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = (uint32_t)uniform((int)tbase);
    const uint32_t sbase = (uint32_t)uniform((int)smem_u32(smem));
    const int my_tiles = split < a.n_tiles ? (a.n_tiles - 1 - split) / a.n_split + 1 : 0;   // in each phase

    if (warp == 0) {
        if (elect_one()) {   // TMA producer
            const uint32_t bytes = (uint32_t)(2 * (a.g_real * a.g_slot + a.planes * a.x_real * a.rows * kWgPitch));
            int it = 0, s = 0;
            uint32_t par = 1;   // a fresh barrier's previous phase counts as complete
            for (int i = 0; i < a.phases * my_tiles; ++i, ++it) {
                const int ph = i / my_tiles, tile = split + (i - ph * my_tiles) * a.n_split;
                const int nimg = tile / per_phase, tt = tile - nimg * per_phase, ty = tt / a.tiles_x;
                const int a0 = ty * a.rows_px, b0 = (tt - ty * a.tiles_x) * 16;
                if (!bar_wait(smem_u32(&empty[0]) + 8 * s, par, a.spin)) {
                    atomicOr(a.err, 8u);
                    abort_flag = 1;
                    break;
                }
                if (*(volatile int*)&abort_flag) break;
                const uint32_t st = sbase + s * a.stage_bytes, fb = smem_u32(&full[0]) + 8 * s;
                // first input row: all nine taps start one row up, one kernel row at its own
                const int row0 = u0 < 0 ? a0 - 1 : a0 + (a.up ? tap_shift(ph >> 1, u0) : (u0 == 0 ? -1 : 0));
                bar_expect_tx(fb, bytes);
                for (int sp = 0; sp < 2; ++sp) {
                    for (int q = 0; q < a.g_real; ++q) {
                        const int chunk = (o0 >> 3) + q;
                        tma_load_4d(st + (uint32_t)((sp * a.g_real + q) * a.g_slot), &p.gmap[sp], b0 * 8, a0,
                                    a.up ? 4 * chunk + ph : chunk, nimg, fb);
                    }
                    for (int pl = 0; pl < a.planes; ++pl) {
                        // parity plane (qy, qx) of a stride-2 layer's input: pl = 2 qy + qx, or qx with qy = (u0 != 1)
                        const int pq = u0 < 0 ? pl : 2 * (u0 != 1) + pl;
                        const uint32_t xb = st + (uint32_t)(a.g_bytes + ((sp * a.planes + pl) * a.x_real) * a.x_slot);
                        for (int q = 0; q < a.x_real; ++q) {
                            const int chunk = (c0 >> 3) + q;
                            tma_load_4d(xb + (uint32_t)(q * a.x_slot), &p.xmap[sp], (b0 - 1) * 8, row0,
                                        a.up ? chunk : 4 * chunk + pq, nimg, fb);
                        }
                    }
                }
                if (++s == S) s = 0, par ^= 1u;
            }
            issued = it;
        }
        __syncwarp();
    } else if (warp == 1) {
        if (elect_one()) {
            // MMA issuer: as in k_conv_tc, every operand is formed from parameters, loop counters and
            // block indices
            const uint32_t idesc = idesc_bf16(128, a.N, 1, 1);
            const uint32_t xlo = (uint32_t)(a.planes * a.x_real * a.x_slot) >> 4;  // hi -> lo half
            const uint32_t glo = (uint32_t)(a.g_real * a.g_slot) >> 4;
            int it = 0, s = 0;
            uint32_t par = 0, acc0 = 0u;
            bool gone = false;
            for (int ph = 0; ph < a.phases && !gone; ++ph)
                for (int i = 0; i < my_tiles; ++i, ++it) {
                    if (!bar_wait(smem_u32(&full[0]) + 8 * s, par, a.spin)) {
                        atomicOr(a.err, 16u);
                        abort_flag = 1;
                        gone = true;
                        break;
                    }
                    fence_after();
                    const uint32_t st = sbase + s * a.stage_bytes;
                    const uint64_t gd0 = sdesc(st, 128u, (uint32_t)a.g_slot);
                    const uint64_t xd0 = sdesc(st, 128u, (uint32_t)a.x_slot);
                    for (int tap = 0; tap < a.taps; ++tap) {
                        const uint32_t d = tmem + (uint32_t)(tap * a.N);
                        uint64_t gh = gd0, xh = xd0 + a.tap_at[blockIdx.z][ph][tap];
                        uint32_t acc = acc0;
#pragma unroll 4
                        for (int k = 0; k < a.rows_px; ++k, gh += 16, xh += kWgPitch / 16) {   // a row of 16 dy pixels is 256 bytes
                            const uint64_t gl = gh + glo, xl = xh + xlo;
                            if (a.w2) {   // hi.hi, hi.lo, lo.hi
                                mma_bf16(d, xh, gh, idesc, acc);
                                mma_bf16(d, xl, gh, idesc, 1u);
                                mma_bf16(d, xh, gl, idesc, 1u);
                            } else {
                                mma_bf16(d, gh, xh, idesc, acc);
                                mma_bf16(d, gh, xl, idesc, 1u);
                                mma_bf16(d, gl, xh, idesc, 1u);
                            }
                            acc = 1u;
                        }
                    }
                    acc0 = 1u;
                    mma_commit(smem_u32(&empty[0]) + 8 * s);
                    if (++s == S) s = 0, par ^= 1u;
                }
            consumed = it;
            mma_commit(smem_u32(&done));
        }
        __syncwarp();
    }
    const bool ok = bar_wait(smem_u32(&done), 0, a.spin);
    if (!ok && lane == 0) atomicOr(a.err, 32u);
    fence_after();
    __syncthreads();
    const bool abort = *(volatile int*)&abort_flag || !ok;
    if (abort && threadIdx.x == 0)
        for (int it = consumed; it < issued; ++it) bar_wait(smem_u32(&full[it % S]), (it / S) & 1, a.spin);
    if (!abort) {
        const int row = 32 * warp + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(32 * warp) << 16);
        const size_t blk = (size_t)kind * a.n_split + split;
        for (int tap = 0; tap < a.taps; ++tap)
            for (int cb = 0; cb < a.N; cb += 16) {
                float v[16];
                tmem_ld16(lane_base + (uint32_t)(tap * a.N + cb), v);
                if (my_tiles == 0)
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = 0.0f;
                float4* dst = reinterpret_cast<float4*>(a.part + (((blk * a.taps + tap) * 128 + row) * a.N + cb));
#pragma unroll
                for (int q = 0; q < 4; ++q) dst[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, a.tmem_cols);
}

// dw[o][c][t] = sum_s part[kind][s][t][row][col] in split order; consecutive threads take
// consecutive columns (blockIdx.y = kind)
__global__ void k_wgrad_reduce(const float* __restrict__ part, int Co, int Ci, int w2, int taps, int c_tiles, int N,
                               int n_split, float* __restrict__ dw) {
    const int kind = blockIdx.y, total = taps * 128 * N;
    const int tile_kind = taps == 3 ? kind / 3 : kind, mt = tile_kind / c_tiles, nt = tile_kind % c_tiles;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const int col = i % N, row = (i / N) & 127, t = (taps == 3 ? 3 * (kind % 3) : 0) + i / (128 * N);
        const int o = w2 ? nt * N + col : mt * 128 + row, c = w2 ? mt * 128 + row : nt * N + col;
        if (o >= Co || c >= Ci) continue;
        const float* src = part + (size_t)kind * n_split * total + i;
        float s = 0.0f;
#pragma unroll 8
        for (int q = 0; q < n_split; ++q) s += src[(size_t)q * total];
        dw[((size_t)o * Ci + c) * 9 + t] = s;
    }
}

// bias gradient: slice sums of the partial rows (32 channels x 8 rows of parts per block),
// then the slices in order; both steps in a fixed order
__global__ void __launch_bounds__(256) k_bias_slices(const float* __restrict__ part, int n_part, int C, int per_slice,
                                                     float* __restrict__ tmp) {
    const int tx = threadIdx.x & 31, r = threadIdx.x >> 5;
    const int c = blockIdx.x * 32 + tx;
    const int q0 = blockIdx.y * per_slice, q1 = min(n_part, q0 + per_slice);
    float s = 0.0f;
    if (c < C)
        for (int q = q0 + r; q < q1; q += 8) s += part[(size_t)q * C + c];
    __shared__ float red[8][32];
    red[r][tx] = s;
    __syncthreads();
    if (r == 0 && c < C) {
        float t = 0.0f;
        for (int k = 0; k < 8; ++k) t += red[k][tx];
        tmp[(size_t)blockIdx.y * C + c] = t;
    }
}

__global__ void k_bias_final(const float* __restrict__ tmp, int slices, int C, float* __restrict__ db) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    float s = 0.0f;
    for (int q = 0; q < slices; ++q) s += tmp[(size_t)q * C + c];
    db[c] = s;
}

// wf[t][c/8][o][c%8] = w[o][c][t] (c < Ci_pad), wb[t][o/8][c][o%8] = w[o][c][t] (o < Co_pad)
__global__ void k_weights_tc(const float* __restrict__ w, int Co, int Ci, int Ci_pad, int Co_pad,
                             __nv_bfloat16* __restrict__ wf, __nv_bfloat16* __restrict__ wb) {
    const int total = 9 * Co * Ci_pad + 9 * Ci * Co_pad;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        if (i < 9 * Co * Ci_pad) {
            const int e = i & 7, r = i >> 3, o = r % Co, q = (r / Co) % (Ci_pad >> 3), t = r / Co / (Ci_pad >> 3);
            const int c = 8 * q + e;
            wf[i] = __float2bfloat16_rn(c < Ci ? w[((size_t)o * Ci + c) * 9 + t] : 0.0f);
        } else {
            const int j = i - 9 * Co * Ci_pad;
            const int e = j & 7, r = j >> 3, c = r % Ci, q = (r / Ci) % (Co_pad >> 3), t = r / Ci / (Co_pad >> 3);
            const int o = 8 * q + e;
            wb[j] = __float2bfloat16_rn(o < Co ? w[((size_t)o * Ci + c) * 9 + t] : 0.0f);
        }
    }
}

__global__ void k_pack_input(const float* __restrict__ X, int N, int H, int W, int par, __nv_bfloat16* __restrict__ hi,
                             __nv_bfloat16* __restrict__ lo) {
    const long HW = (long)H * W, total = (long)N * HW;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
        const int n = (int)(i / HW), y = (int)((i % HW) / W), x = (int)(i % W);
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = j < 2 ? X[((size_t)n * 2 + j) * HW + (i % HW)] : 0.0f;
        store_pair8(hi, lo, chunk_at(par, 1, H, W, n, y, x, 0), v);
    }
}

// out[n][c][y][x] = hi + lo of channel c < C_real of the pair a (any layout)
__global__ void k_unpack_act(const __nv_bfloat16* __restrict__ hi, const __nv_bfloat16* __restrict__ lo, int N, int H,
                             int W, int C8, int par, int C_real, float* __restrict__ out) {
    const long HW = (long)H * W, total = (long)N * C_real * HW;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
        const int n = (int)(i / (C_real * HW)), c = (int)((i / HW) % C_real), y = (int)((i % HW) / W), x = (int)(i % W);
        const size_t o = chunk_at(par, C8, H, W, n, y, x, c >> 3) + (c & 7);
        out[i] = __bfloat162float(hi[o]) + __bfloat162float(lo[o]);
    }
}

__global__ void __launch_bounds__(256) k_mse_tc(const float* __restrict__ out, const float* __restrict__ t,
                                                const float* __restrict__ mask, int N, int H, int W, float inv_terms,
                                                __nv_bfloat16* __restrict__ ghi, __nv_bfloat16* __restrict__ glo,
                                                __nv_bfloat16* __restrict__ gphi, __nv_bfloat16* __restrict__ gplo,
                                                float* __restrict__ db_part, double* loss) {
    double acc = 0.0;
    float d0 = 0.0f, d1 = 0.0f;
    const long HW = (long)H * W, total = (long)N * HW;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
        const int n = (int)(i / HW), p = (int)(i % HW), y = p / W, x = p % W;
        const float mk = mask[p];
        float g[8];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const long k = ((long)n * 2 + c) * HW + p;
            const float d = (out[k] - t[k]) * mk;
            acc += (double)d * d;
            g[c] = 2.0f * d * inv_terms;
        }
#pragma unroll
        for (int c = 2; c < 8; ++c) g[c] = 0.0f;
        d0 += g[0];
        d1 += g[1];
        store_pair8(ghi, glo, chunk_at(0, 1, H, W, n, y, x, 0), g);
        if (gphi) store_pair8(gphi, gplo, chunk_at(1, 1, H, W, n, y, x, 0), g);
    }
    __shared__ double rl[8];
    __shared__ float r0[8], r1[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
        d0 += __shfl_xor_sync(0xffffffffu, d0, o);
        d1 += __shfl_xor_sync(0xffffffffu, d1, o);
    }
    if ((threadIdx.x & 31) == 0) {
        rl[threadIdx.x >> 5] = acc;
        r0[threadIdx.x >> 5] = d0;
        r1[threadIdx.x >> 5] = d1;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        float s0 = 0.0f, s1 = 0.0f;
        for (int q = 0; q < 8; ++q) {
            s += rl[q];
            s0 += r0[q];
            s1 += r1[q];
        }
        atomicAdd(loss, s * inv_terms);
        db_part[blockIdx.x * 2] = s0;
        db_part[blockIdx.x * 2 + 1] = s1;
    }
}

// ---------------------------------------------------------------------------------------
// host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;
bool g_ready = false;
int g_conv_dyn = 0, g_wg_dyn = 0;   // dynamic shared memory the two kernels may request

// map of one half (hi or lo) of a chunk-major tensor; box = `px` pixels x 8 channels x `rows`
// rows of one chunk (one parity plane of a parity-split tensor: chunk coordinate 4 q + plane)
bool enc_act(CUtensorMap* m, const __nv_bfloat16* base, const Act2& t, bool parity, int rows, int px = 16) {
    const size_t es = sizeof(__nv_bfloat16);
    const int C8 = t.C / 8, H = parity ? t.H / 2 : t.H, W = parity ? t.W / 2 : t.W, planes = parity ? 4 : 1;
    cuuint64_t dims[4] = {(cuuint64_t)W * 8, (cuuint64_t)H, (cuuint64_t)C8 * planes, (cuuint64_t)t.N};
    cuuint64_t strides[3] = {(cuuint64_t)W * 8 * es, (cuuint64_t)H * W * 8 * es, (cuuint64_t)C8 * planes * H * W * 8 * es};
    cuuint32_t box[4] = {(cuuint32_t)px * 8, (cuuint32_t)rows, 1, 1}, estr[4] = {1, 1, 1, 1};
    return g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int pow2_cols(int c) {
    int r = 32;
    while (r < c) r <<= 1;
    return r;
}

// floor((p + u - 1) / 2) for p, u in {0, 1} x {0, 1, 2}
int half_shift(int p, int u) { return (p + u - 1) >= 0 ? (p + u - 1) / 2 : -1; }

struct ConvPlan {
    ConvParams prm;
    dim3 grid;
    int smem;
};

void sort_groups(ConvArgs& a, const Group* g, int ng, int phases) {
    int k = 0;
    for (int ph = 0; ph < phases; ++ph) {
        a.gstart[ph] = k;
        for (int i = 0; i < ng; ++i)
            if (g[i].phase == ph) a.group[k++] = g[i];
    }
    for (int ph = phases; ph <= 4; ++ph) a.gstart[ph] = k;
}

// stages and tile sizes for a given N; returns false when not even one stage fits
bool fit_stages(ConvArgs& a) {
    a.a_slot = (a.rows * a.px * 16 + 127) / 128 * 128;   // a TMA load's destination: 128-byte aligned
    a.a_bytes = a.split * a.n_copy * 2 * a.a_slot;
    a.stage_bytes = a.a_bytes + 2 * 9 * a.N * 16;
    a.n_stage = std::min(kMaxStage, (g_conv_dyn - 1024) / a.stage_bytes);
    return a.n_stage >= 1;
}

cudaError_t finish_plan(ConvPlan& pl, int n_img, int num_sms, int phases, int Ntot) {
    ConvArgs& a = pl.prm.a;
    // N: largest divisor of Ntot (<= 256) for which two stages fit, else one
    int best = 0;
    for (int N = std::min(256, Ntot); N >= 16; N -= 16) {
        if (Ntot % N) continue;
        a.N = N;
        if (!fit_stages(a)) continue;
        if (a.n_stage >= 2) {
            best = N;
            break;
        }
        if (!best) best = N;
    }
    if (!best) return cudaErrorInvalidConfiguration;
    a.N = best;
    fit_stages(a);
    // phases per tile: all of them if two sets of accumulators fit in TMEM and the tiles still
    // cover the SMs
    const int tiles = a.tiles_x * a.tiles_y * n_img * (Ntot / a.N);
    a.P = phases;
    while (a.P > 1 && (2 * a.P * a.N > 512 || tiles * (phases / a.P) < num_sms)) a.P >>= 1;
    a.n_acc = 2 * a.P * a.N <= 512 ? 2 : 1;
    if (a.P * a.N > 512) return cudaErrorInvalidConfiguration;
    a.tmem_cols = pow2_cols(a.n_acc * a.P * a.N);
    for (int i = 0; i < a.gstart[phases] * a.split; ++i) {
        const Group gr = a.group[i / a.split];
        const int sp = i % a.split;
        const bool first = sp == 0 && i / a.split == a.gstart[gr.phase];
        pl.prm.mma[i] = make_uint4((unsigned)((sp * a.n_copy + gr.copy) * 2 * a.a_slot + (gr.row * a.px + gr.col) * 16) >> 4,
                                   (unsigned)(gr.tap * 2 * a.N * 16) >> 4, (unsigned)(gr.phase % a.P * a.N), first ? 0u : 1u);
    }
    a.n_img = n_img;
    a.pgroups = phases / a.P;
    a.n_zt = Ntot / a.N;
    pl.grid = dim3(std::min(std::max(1, num_sms / a.pgroups), tiles), a.pgroups);
    // one CTA per SM, so that its TMEM allocation never waits
    pl.smem = std::max(a.n_stage * a.stage_bytes + 1024, kOneCtaPerSm);
    return pl.smem > g_conv_dyn ? cudaErrorInvalidConfiguration : cudaSuccess;
}

}  // namespace

cudaError_t tc_prepare() {
    if (g_ready) return cudaSuccess;
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return e != cudaSuccess ? e : cudaErrorNotSupported;
    g_encode = reinterpret_cast<EncodeTiledFn>(fn);
    int dev = 0, optin = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
    cudaFuncAttributes fa;
    if ((e = cudaFuncGetAttributes(&fa, k_conv_tc)) != cudaSuccess) return e;
    g_conv_dyn = std::min(kSmemLimit, optin - (int)fa.sharedSizeBytes);
    if ((e = cudaFuncGetAttributes(&fa, k_wgrad_tc)) != cudaSuccess) return e;
    g_wg_dyn = std::min(kSmemLimit, optin - (int)fa.sharedSizeBytes);
    if ((e = cudaFuncSetAttribute(k_conv_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, g_conv_dyn)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, g_wg_dyn)) != cudaSuccess) return e;
    g_ready = true;
    return cudaSuccess;
}

cudaError_t tc_conv_forward(const TcLayer& L, const Act2& x, const __nv_bfloat16* wf, const float* bias, const Act2* y,
                            float* y32, unsigned* err, unsigned spin, int num_sms, cudaStream_t st) {
    cudaError_t e = tc_prepare();
    if (e != cudaSuccess) return e;
    static ConvPlan pl;
    std::memset(&pl, 0, sizeof pl);
    ConvArgs& a = pl.prm.a;
    const int Ho = L.Hout();
    Group g[kMaxGroup];
    int ng = 0, phases;
    a.split = 2;
    a.ksteps = L.Ci_pad / 16;
    if (!L.up) {
        // the input is read by parity planes: it must be stored split by parity
        if (!x.par) return cudaErrorInvalidValue;
        phases = 1;
        a.tiles_y = Ho / 16;
        a.tiles_x = Ho / 8;
        a.rows = 17;
        a.px = 9;
        a.n_copy = 4;
        for (int pl4 = 0; pl4 < 4; ++pl4) a.copy[pl4] = Copy{-1, -1, (int8_t)pl4};
        for (int u = 0; u < 3; ++u)
            for (int v = 0; v < 3; ++v)
                g[ng++] = Group{0, (uint8_t)(2 * (u != 1) + (v != 1)), (uint8_t)(u == 0 ? 0 : 1), (uint8_t)(v == 0 ? 0 : 1),
                                (uint8_t)(3 * u + v)};
        a.osy = a.osx = 1;
    } else {
        phases = 4;
        a.tiles_y = L.Hin / 16;
        a.tiles_x = L.Hin / 8;
        if (x.par) return cudaErrorInvalidValue;
        a.rows = 18;
        a.px = 10;
        a.n_copy = 1;
        a.copy[0] = Copy{-1, -1, -1};
        for (int py = 0; py < 2; ++py)
            for (int px = 0; px < 2; ++px)
                for (int u = 0; u < 3; ++u)
                    for (int v = 0; v < 3; ++v)
                        g[ng++] = Group{(uint8_t)(2 * py + px), 0, (uint8_t)(half_shift(py, u) + 1),
                                        (uint8_t)(half_shift(px, v) + 1), (uint8_t)(3 * u + v)};
        a.osy = a.osx = 2;
        for (int ph = 0; ph < 4; ++ph) {
            a.opy[ph] = (int8_t)(ph >> 1);
            a.opx[ph] = (int8_t)(ph & 1);
        }
    }
    sort_groups(a, g, ng, phases);
    const bool last = y == nullptr;
    const int Ntot = (L.Co + 15) / 16 * 16;
    if ((e = finish_plan(pl, x.N, num_sms, phases, Ntot)) != cudaSuccess) return e;
    if (!enc_act(&pl.prm.amap[0], x.hi, x, x.par != 0, a.rows, a.px) || !enc_act(&pl.prm.amap[1], x.lo, x, x.par != 0, a.rows, a.px))
        return cudaErrorInvalidValue;
    a.wts = wf;
    a.wK8 = L.Ci_pad / 8;
    a.wR = L.Co;
    a.mode = last ? EPI_LAST : EPI_HIDDEN;
    a.oH = Ho;
    a.oW = Ho;
    a.oC = L.Co;
    a.out_par = last ? 0 : y->par;
    a.out_hi = last ? nullptr : y->hi;
    a.out_lo = last ? nullptr : y->lo;
    a.out_phi = last ? nullptr : y->phi;
    a.out_plo = last ? nullptr : y->plo;
    a.out32 = y32;
    a.bias = bias;
    a.relu = L.relu;
    a.err = err;
    a.spin = spin;
    k_conv_tc<<<pl.grid, kConvThreads, pl.smem, st>>>(pl.prm);
    return cudaGetLastError();
}

int tc_bias_parts(const TcLayer& L, int N, int num_sms) {
    // upper bound: one part per (tile, phase group)
    const int S = L.up ? L.Hout() : L.Hin / 2;   // sub-lattice side of the output gradient tiles
    (void)num_sms;
    return (S / 8) * (S / 16) * N * 4;
}

cudaError_t tc_conv_backward_data(const TcLayer& L, const Act2& dy, const __nv_bfloat16* wb, const Act2& act,
                                  const Act2& dx, float* db_part, int* n_part, unsigned* err, unsigned spin, int num_sms,
                                  cudaStream_t st) {
    cudaError_t e = tc_prepare();
    if (e != cudaSuccess) return e;
    static ConvPlan pl;
    std::memset(&pl, 0, sizeof pl);
    ConvArgs& a = pl.prm.a;
    Group g[kMaxGroup];
    int ng = 0, phases;
    a.split = 2;
    a.ksteps = L.Co_pad / 16;
    if (!L.up) {
        // dx on the input grid in four parity phases; dy rows a'+e, columns b'+f
        phases = 4;
        const int Sd = L.Hin / 2;
        a.tiles_y = Sd / 16;
        a.tiles_x = Sd / 8;
        a.rows = 17;
        a.px = 9;
        a.n_copy = 1;
        a.copy[0] = Copy{0, 0, -1};
        for (int qy = 0; qy < 2; ++qy)
            for (int qx = 0; qx < 2; ++qx)
                for (int u = 0; u < 3; ++u)
                    for (int v = 0; v < 3; ++v) {
                        if ((qy == 0) != (u == 1) || (qx == 0) != (v == 1)) continue;
                        const int ey = (qy == 1 && u == 0) ? 1 : 0, ex = (qx == 1 && v == 0) ? 1 : 0;
                        g[ng++] = Group{(uint8_t)(2 * qy + qx), 0, (uint8_t)ey, (uint8_t)ex, (uint8_t)(3 * u + v)};
                    }
        a.osy = a.osx = 2;
        for (int ph = 0; ph < 4; ++ph) {
            a.opy[ph] = (int8_t)(ph >> 1);
            a.opx[ph] = (int8_t)(ph & 1);
        }
        a.mode = EPI_BWD;
    } else {
        // stride-1 correlation of dy with the transposed weights, then 2 x 2 sums
        phases = 1;
        const int Sd = L.Hout();
        a.tiles_y = Sd / 16;
        a.tiles_x = Sd / 8;
        a.rows = 18;
        a.px = 10;
        a.n_copy = 1;
        a.copy[0] = Copy{-1, -1, -1};
        for (int u = 0; u < 3; ++u)
            for (int v = 0; v < 3; ++v)
                g[ng++] = Group{0, 0, (uint8_t)(2 - u), (uint8_t)(2 - v), (uint8_t)(3 * u + v)};
        a.osy = a.osx = 1;
        a.mode = EPI_POOL;
    }
    sort_groups(a, g, ng, phases);
    if (dy.par) return cudaErrorInvalidValue;   // both forms read dy by plain rows
    if ((e = finish_plan(pl, dy.N, num_sms, phases, L.Ci)) != cudaSuccess) return e;
    if (!enc_act(&pl.prm.amap[0], dy.hi, dy, false, a.rows, a.px) || !enc_act(&pl.prm.amap[1], dy.lo, dy, false, a.rows, a.px))
        return cudaErrorInvalidValue;
    a.wts = wb;
    a.wK8 = L.Co_pad / 8;
    a.wR = L.Ci;
    a.oH = L.Hin;
    a.oW = L.Hin;
    a.oC = L.Ci;
    a.out_par = dx.par;
    a.out_hi = dx.hi;
    a.out_lo = dx.lo;
    a.out_phi = dx.phi;
    a.out_plo = dx.plo;
    a.m_par = act.par;
    a.m_hi = act.hi;
    a.m_lo = act.lo;
    a.db_part = db_part;
    a.err = err;
    a.spin = spin;
    *n_part = a.tiles_x * a.tiles_y * a.n_img * a.pgroups;
    k_conv_tc<<<pl.grid, kConvThreads, pl.smem, st>>>(pl.prm);
    return cudaGetLastError();
}

namespace {

struct WgPlan {
    WgParams prm;
    dim3 grid;
    int smem;
};

cudaError_t plan_wgrad(WgPlan& pl, const TcLayer& L, const Act2* x, const Act2* dy, int n_img, int num_sms) {
    std::memset(&pl, 0, sizeof pl);
    WgArgs& a = pl.prm.a;
    a.up = L.up;
    a.Co = L.Co;
    a.Ci = L.Ci;
    // the 128 rows of an MMA go to the side that fills them
    a.w2 = L.Co <= 16 || (L.Co < 128 && L.Ci >= 128) ? 1 : 0;
    a.phases = L.up ? 4 : 1;
    const int S = L.up ? L.Hin : L.Hout();   // per-phase output sub-lattice side
    const int cols = a.w2 ? (L.Co + 15) / 16 * 16 : L.Ci_pad;
    a.N = 16;
    for (int n = 16; n <= std::min(128, cols); n += 16)
        if (cols % n == 0) a.N = n;
    a.taps = 9 * a.N <= 512 ? 9 : 3;
    a.c_tiles = cols / a.N;
    const int g_ch = a.w2 ? a.N : std::min(128, L.Co), x_ch = a.w2 ? std::min(128, L.Ci) : a.N;
    a.g_real = std::min((L.Co + 7) / 8, g_ch / 8);
    a.x_real = x_ch / 8;
    const int kinds = ((a.w2 ? L.Ci : L.Co) + 127) / 128 * a.c_tiles * (9 / a.taps);
    a.tmem_cols = pow2_cols(a.taps * a.N);
    a.planes = L.up ? 1 : a.taps == 9 ? 4 : 2;
    // pixel rows per stage: 8 if two stages fit, else 4
    const int budget = g_wg_dyn - 1024;
    for (int rp = 8; rp >= 4; rp -= 4) {
        a.rows_px = rp;
        a.rows = rp + (a.taps == 3 ? 0 : L.up ? 2 : 1);
        a.g_slot = rp * 16 * 16;
        a.x_slot = (a.rows * kWgPitch + 127) / 128 * 128;   // a TMA load's destination: 128-byte aligned
        a.g_bytes = 2 * a.g_real * a.g_slot;
        a.x_bytes = 2 * a.planes * a.x_real * a.x_slot;
        a.stage_bytes = a.g_bytes + a.x_bytes;
        // rows / columns beyond the real channels read on into the next 16 slots at most
        const int tail = 16 * std::max(a.g_slot, a.x_slot);
        a.n_stage = std::min(kMaxStage, (budget - tail) / a.stage_bytes);
        if (a.n_stage >= 2 || rp == 4) break;
    }
    if (a.n_stage < 1) return cudaErrorInvalidConfiguration;
    a.tiles_y = S / a.rows_px;
    a.tiles_x = S / 16;
    a.n_tiles = n_img * a.tiles_x * a.tiles_y;   // of one phase
    a.n_split = std::max(1, std::min(a.n_tiles, num_sms / kinds));
    if (x && dy) {
        // up layers read dy by parity planes (its parity copy), stride-2 layers by plain rows;
        // the input x of a stride-2 layer is read by parity planes, of an up layer by plain rows
        if (L.up ? (!dy->phi || x->par) : (dy->par || !x->par)) return cudaErrorInvalidValue;
        const __nv_bfloat16* ghi = L.up ? dy->phi : dy->hi;
        const __nv_bfloat16* glo = L.up ? dy->plo : dy->lo;
        if (!enc_act(&pl.prm.gmap[0], ghi, *dy, L.up != 0, a.rows_px) || !enc_act(&pl.prm.gmap[1], glo, *dy, L.up != 0, a.rows_px) ||
            !enc_act(&pl.prm.xmap[0], x->hi, *x, x->par != 0, a.rows, kWgPx) ||
            !enc_act(&pl.prm.xmap[1], x->lo, *x, x->par != 0, a.rows, kWgPx))
            return cudaErrorInvalidValue;
    }
    const int rows_u = 9 / a.taps;   // kernel rows handled apart
    for (int ur = 0; ur < rows_u; ++ur)
        for (int ph = 0; ph < a.phases; ++ph)
            for (int t = 0; t < a.taps; ++t) {
                const int u = rows_u == 3 ? ur : t / 3, v = t % 3;
                int plane, row, col;
                if (L.up) {
                    plane = 0;
                    row = rows_u == 3 ? 0 : half_shift(ph >> 1, u) + 1;
                    col = half_shift(ph & 1, v) + 1;
                } else {
                    plane = (rows_u == 3 ? 0 : 2 * (u != 1)) + (v != 1);
                    row = rows_u == 3 ? 0 : (u == 0 ? 0 : 1);
                    col = v == 0 ? 0 : 1;
                }
                a.tap_at[ur][ph][t] = (uint32_t)(a.g_bytes + plane * a.x_real * a.x_slot + row * kWgPitch + col * 16) >> 4;
            }
    pl.grid = dim3(a.n_split, kinds / rows_u, rows_u);
    pl.smem = a.n_stage * a.stage_bytes + 16 * std::max(a.g_slot, a.x_slot) + 1024;
    if (a.tmem_cols > 256) pl.smem = std::max(pl.smem, kOneCtaPerSm);
    if (pl.smem > g_wg_dyn) return cudaErrorInvalidConfiguration;
    return cudaSuccess;
}

}  // namespace

size_t tc_wgrad_workspace(const TcLayer& L, int N, int num_sms) {
    if (tc_prepare() != cudaSuccess) return 0;
    static WgPlan pl;
    if (plan_wgrad(pl, L, nullptr, nullptr, N, num_sms) != cudaSuccess) return 0;
    return (size_t)pl.grid.x * pl.grid.y * pl.grid.z * pl.prm.a.taps * 128 * pl.prm.a.N;
}

cudaError_t tc_conv_wgrad(const TcLayer& L, const Act2& x, const Act2& dy, float* ws, float* dw, unsigned* err,
                          unsigned spin, int num_sms, cudaStream_t st) {
    cudaError_t e = tc_prepare();
    if (e != cudaSuccess) return e;
    static WgPlan pl;
    if ((e = plan_wgrad(pl, L, &x, &dy, x.N, num_sms)) != cudaSuccess) return e;
    WgArgs& a = pl.prm.a;
    a.part = ws;
    a.err = err;
    a.spin = spin;
    k_wgrad_tc<<<pl.grid, kThreads, pl.smem, st>>>(pl.prm);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_wgrad_reduce<<<dim3((a.taps * 128 * a.N + 255) / 256, pl.grid.y * pl.grid.z), 256, 0, st>>>(ws, L.Co, L.Ci, a.w2, a.taps,
                                                                                    a.c_tiles, a.N, a.n_split, dw);
    return cudaGetLastError();
}

cudaError_t tc_bias_reduce(const float* part, int n_part, int C, float* tmp, float* db, cudaStream_t st) {
    if (n_part < 1 || C < 1) return cudaErrorInvalidValue;
    const int slices = std::min(kBiasSlices, n_part), per = (n_part + slices - 1) / slices;
    k_bias_slices<<<dim3((C + 31) / 32, slices), 256, 0, st>>>(part, n_part, C, per, tmp);
    k_bias_final<<<(C + 127) / 128, 128, 0, st>>>(tmp, slices, C, db);
    return cudaGetLastError();
}

cudaError_t tc_weights(const TcLayer& L, const float* w32, __nv_bfloat16* wf, __nv_bfloat16* wb, cudaStream_t st) {
    const int total = 9 * L.Co * L.Ci_pad + 9 * L.Ci * L.Co_pad;
    k_weights_tc<<<std::max(1, std::min(1024, (total + 255) / 256)), 256, 0, st>>>(w32, L.Co, L.Ci, L.Ci_pad, L.Co_pad, wf,
                                                                                  wb);
    return cudaGetLastError();
}

cudaError_t tc_pack_input(const float* X, const Act2& x0, cudaStream_t st) {
    const long total = (long)x0.N * x0.H * x0.W;
    k_pack_input<<<(int)std::min<long>(2048, (total + 255) / 256), 256, 0, st>>>(X, x0.N, x0.H, x0.W, x0.par, x0.hi, x0.lo);
    return cudaGetLastError();
}

cudaError_t tc_unpack(const Act2& a, int C_real, float* out, cudaStream_t st) {
    if (C_real < 1 || C_real > a.C) return cudaErrorInvalidValue;
    const long total = (long)a.N * C_real * a.H * a.W;
    if (total == 0) return cudaSuccess;
    const int blocks = (int)std::min<long>((total + 255) / 256, 4096);
    k_unpack_act<<<blocks, 256, 0, st>>>(a.hi, a.lo, a.N, a.H, a.W, a.C >> 3, a.par, C_real, out);
    return cudaGetLastError();
}

cudaError_t tc_mse(const float* out, const float* t, const float* mask, const Act2& g, double n_terms, float* db_part,
                   int* n_part, double* loss, cudaStream_t st) {
    if (g.par) return cudaErrorInvalidValue;
    k_mse_tc<<<kMseBlocks, 256, 0, st>>>(out, t, mask, g.N, g.H, g.W, (float)(1.0 / n_terms), g.hi, g.lo, g.phi, g.plo,
                                         db_part, loss);
    *n_part = kMseBlocks;
    return cudaGetLastError();
}

}  // namespace ptylm
