// The front of stage 1 of the Fused MoE description when the layer starts from
// bf16 hidden states: the router projection ("routing scores via a lightweight
// linear projection") and the input-side FP8 quantisation of the activations
// (one fp32 scale per token per 128 columns, scale = amax / 448).
//
// The expert indices selected from the logits are compared bit for bit, so the
// fp32 summation order of the projection is fixed: 32 partial sums, partial l
// takes the l-th pair of every run of 64 elements in increasing order with one
// fused multiply-add per element (bf16 x bf16 is exact in fp32), then five
// pairwise rounds p[l] += p[l xor d], d = 16, 8, 4, 2, 1.  That order is what a
// warp computes naturally: lane l owns partial l and the rounds are butterfly
// shuffles.  It runs on the fp32 pipes, not on the tensor cores, whose
// accumulation order is not specified.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <stdint.h>

#include "ptx.cuh"

namespace moe {

// logits[t, e] = sum_h x[t, h] * w[e, h] in the order stated above.  A warp owns MT tokens x ME experts with the K
// dimension spread over its lanes, a CTA WT x WE such warps; rows come in through a ring of S stages of KC elements
// (cp.async).  x [T, H] and w [E, H] bf16, H a multiple of KC, E a multiple of WE * ME.
//
// Large batches are bound by the fp32 pipes (2 x 7168 x 256 FLOP per token) and the issue slots around the FMAs.  The FMA
// with bf16 factors takes its words as they are, with nothing to convert and no factor to put into both halves of a pair:
// alone it runs at 25.7 TFMA/s on the chip, the packed fp32 FMA at 32.2 and at 27.3 beside the conversions for an 8 x 8 tile,
// but in this kernel it is the faster one (packed / this: 94.9 / 83.3 us at 1024 tokens; one of each per word 86.8).  ldmatrix
// hands a lane its words of four rows in one instruction.  Small batches are bound by latency and the number of warps that
// stream the 3.7 MB of weights.  Hence two shapes (us, packed fp32 FMAs / this kernel):
//   8 x 8 per warp, 2 x 2 warps   many small CTAs balance the SMs: 257 tokens 33.5 / 29.4, 1024 94.9 / 83.3, 8192 660 (16 x 8
//                                 per warp) / 627, 24.0 TFMA/s; with the bf16 FMA 16 x 8 is slower (662)
//   4 x 4, 2 x 1 warps            many loads in flight per warp: 16 tokens 11.2 / 8.9, 64 tokens 15.2 / 11.1 in rows of 512
//                                 elements, four stages (256, eight stages: 9.6 and 13.5)
// The line lies where they are equal.  us per forward from hidden states with 8 x 8 / 4 x 4, hidden 7168: without local rows 28.1 /
// 26.8 at 80 tokens, 33.7 / 32.8 at 96, 34.6 / 34.3 at 128, 34.9 / 35.0 at 144; 32 experts of 7168 x 2048 158.0 / 145.4 at 72, 202.6 / 196.7 at
// 100, 161.0 / 152.5 at 128; hidden 2048 34.1 / 33.1 at 100, 34.5 / 33.8 at 128, 37.2 / 37.8 at 200; hidden 512 26.5 / 25.7 at 100, 20.4 / 20.8
// at 200.
template <int WT, int WE, int MT, int ME, int KC, int S>
struct RouterShape {
    static constexpr int ROWS_T = WT * MT, ROWS_E = WE * ME, THREADS = WT * WE * 32, ROWS = ROWS_T + ROWS_E;
    static constexpr int SMEM_BYTES = S * ROWS * KC * 2;
    static_assert(MT % 4 == 0 && ME % 4 == 0 && KC % 64 == 0, "rows are read four at a time, in runs of 64 elements");
};
constexpr int RP_SMALL_MAX_TOKENS = 128;   // 4 x 4 up to here

template <int WT, int WE, int MT, int ME, int KC, int S>
__global__ void __launch_bounds__(WT * WE * 32)
router_logits_kernel(int T, int H, int E, const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ w,
                     float* __restrict__ logits) {
    using Shape = RouterShape<WT, WE, MT, ME, KC, S>;
    extern __shared__ __align__(128) uint8_t rp_smem[];
    constexpr int ROWS_T = Shape::ROWS_T, ROWS = Shape::ROWS, THREADS = Shape::THREADS;
    constexpr int CHUNKS_PER_ROW = KC / 8, ROW_BYTES = KC * 2;     // 16-byte chunks of one staged row
    pdl_launch_dependents();  // (quantize_rows_kernel needs nothing from here)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wt = warp / WE, we = warp % WE;
    const int t0 = blockIdx.x * ROWS_T, e0 = blockIdx.y * Shape::ROWS_E;
    const uint32_t smem0 = smem_u32(rp_smem);
    const int nkc = H / KC;

    // stage K-chunk kc of the tile's rows (tokens first, then experts); rows past T read as zero
    auto stage = [&](int kc) {
        if (kc < nkc) {
            const uint32_t dst = smem0 + (kc % S) * ROWS * ROW_BYTES;
#pragma unroll
            for (int c = tid; c < ROWS * CHUNKS_PER_ROW; c += THREADS) {
                const int r = c / CHUNKS_PER_ROW, cc = c % CHUNKS_PER_ROW;
                const __nv_bfloat16* src;
                uint32_t bytes = 16;
                if (r < ROWS_T) {
                    const int t = t0 + r;
                    if (t >= T) bytes = 0;
                    src = x + static_cast<size_t>(t < T ? t : 0) * H + kc * KC + cc * 8;
                } else {
                    src = w + static_cast<size_t>(e0 + r - ROWS_T) * H + kc * KC + cc * 8;
                }
                cp_async_16(dst + r * ROW_BYTES + cc * 16, src, bytes);
            }
        }
        cp_async_commit();
    };

    float acc[MT][ME];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < ME; ++j) acc[i][j] = 0.0f;

#pragma unroll
    for (int i = 0; i < S - 1; ++i) stage(i);
    // this lane's row addresses for ldmatrix: piece lane & 7 of row lane >> 3 of a group of four
    const uint32_t x_off = (wt * MT + (lane >> 3)) * ROW_BYTES + (lane & 7) * 16;
    const uint32_t w_off = (ROWS_T + we * ME + (lane >> 3)) * ROW_BYTES + (lane & 7) * 16;
    for (int kc = 0; kc < nkc; ++kc) {
        cp_async_wait<S - 2>();
        __syncthreads();  // the chunk has landed, and everybody has left the buffer that is refilled next
        stage(kc + S - 1);
        const uint32_t base = smem0 + (kc % S) * ROWS * ROW_BYTES;
#pragma unroll
        for (int run = 0; run < KC / 64; ++run) {
            uint32_t xr[MT];  // elements 2l, 2l+1 of the run
#pragma unroll
            for (int q = 0; q < MT / 4; ++q) {
                uint32_t r[4];
                ldmatrix_x4(base + x_off + q * 4 * ROW_BYTES + run * 128, r);
#pragma unroll
                for (int i = 0; i < 4; ++i) xr[4 * q + i] = r[i];
            }
#pragma unroll
            for (int q = 0; q < ME / 4; ++q) {
                uint32_t r[4];
                ldmatrix_x4(base + w_off + q * 4 * ROW_BYTES + run * 128, r);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
#pragma unroll
                    for (int i = 0; i < MT; ++i) acc[i][4 * q + j] = fma_bf16_lo(xr[i], r[j], acc[i][4 * q + j]);  // element 2l
#pragma unroll
                    for (int i = 0; i < MT; ++i) acc[i][4 * q + j] = fma_bf16_hi(xr[i], r[j], acc[i][4 * q + j]);  // then 2l+1
                }
            }
        }
    }

    // five pairwise rounds, after which every lane holds every logit of the warp tile; the lanes store them in turn
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < ME; ++j) {
            float v = acc[i][j];
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, d));
            const int t = t0 + wt * MT + i;
            if (lane == (i * ME + j) % 32 && t < T) logits[static_cast<size_t>(t) * E + e0 + we * ME + j] = v;
        }
}

// One warp per (token, 128-column block): amax, scale = amax / 448 (1 for an all-zero block), codes =
// e4m3(x / scale) with IEEE division, round to nearest even, saturating.  scale_layout 0: [T, H/128], 1: [H/128, T].
// Runs beside the router projection (programmatic dependent launch): it reads the same input and waits for that kernel
// only at its end, so that whoever follows finds both done.
__global__ void __launch_bounds__(256) quantize_rows_kernel(int T, int H, int scale_layout,
                                                            const __nv_bfloat16* __restrict__ x,
                                                            uint8_t* __restrict__ q, float* __restrict__ scale) {
    const int lane = threadIdx.x & 31;
    const int nb = H / 128;
    const long long nblocks = static_cast<long long>(T) * nb;
    const long long warp0 = static_cast<long long>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long nwarps = static_cast<long long>(gridDim.x) * (blockDim.x >> 5);
    for (long long blk = warp0; blk < nblocks; blk += nwarps) {
        const long long t = blk / nb;
        const int b = static_cast<int>(blk - t * nb);
        const uint2 raw = *reinterpret_cast<const uint2*>(x + t * H + b * 128 + lane * 4);
        const float v0 = __uint_as_float(raw.x << 16), v1 = __uint_as_float(raw.x & 0xffff0000u);
        const float v2 = __uint_as_float(raw.y << 16), v3 = __uint_as_float(raw.y & 0xffff0000u);
        float amax = fmaxf(fmaxf(fabsf(v0), fabsf(v1)), fmaxf(fabsf(v2), fabsf(v3)));
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, d));
        const float sc = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, 448.0f);
        const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(__fdiv_rn(v0, sc), __fdiv_rn(v1, sc)),
                                                     __NV_SATFINITE, __NV_E4M3);
        const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(__fdiv_rn(v2, sc), __fdiv_rn(v3, sc)),
                                                     __NV_SATFINITE, __NV_E4M3);
        *reinterpret_cast<uint32_t*>(q + t * H + b * 128 + lane * 4) = lo | (hi << 16);
        if (lane == 0) scale[scale_layout ? static_cast<long long>(b) * T + t : t * nb + b] = sc;
    }
    pdl_wait();
}

}  // namespace moe
