// Stage 4 of the Fused MoE description: bring the expert outputs back to token
// order, weighted by the routing weights.  The threads of a token pull its (at
// most 8) bf16 rows in routing order, accumulate in fp32 and round once to
// bf16; tokens without a local expert are written as zeros.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include "gemm.cuh"
#include "ptx.cuh"

namespace moe {

// Bound by the latency of scattered 32-byte reads (a token's rows lie in up to eight row tiles, its 16-column groups 1 KB
// apart): about 4.7 TB/s with all experts local.  So only the rows that exist are looked at, the loads of up to four of them
// are under way in a thread, the token's table entries come one token ahead, and a block holds a part of a token's columns:
// 75 registers, six blocks of four warps on an SM (at hidden 7168 the last of four parts has columns for two of its warps).  us for one block of 256 threads per token and all eight slots in turn / this form: 12.3
// / 8.2 at 257 tokens (257 rows), 16.4 / 14.4 at 1024 (1602), 43.0 / 36.9 at 4096 (6007), 131 / 115 at 8192 skewed (33838), 127
// / 110 at 4096 with 256 experts (32768).  Blocks of 448 threads 41, 122 and 118 for the last three; two or three rows under
// way 37 to 39, 115 to 118 and 110; eight rows 88, 226 and 164 (registers: few warps).
constexpr int COMBINE_BATCH = 4;         // rows of a token whose loads a thread has under way
constexpr int COMBINE_MAX_THREADS = 128;
constexpr int COMBINE_BLOCKS_PER_SM = 16;  // grid, per part of the columns

// y is the tile-blocked bf16 output of GEMM2 (see y_block_offset); each thread owns 16 columns
// (one 32-byte group) of one token, blockIdx.y says which part of the groups.
__global__ void __launch_bounds__(COMBINE_MAX_THREADS) combine_kernel(int T, int H, const int* slot_to_row, const float* topk_w,
                                                                      const uint8_t* y, __nv_bfloat16* __restrict__ out) {
    pdl_launch_dependents();
    pdl_wait();
    const int groups = H / 16, n_tiles = H / 256, lane = threadIdx.x & 31;
    // lane j < 8: row and weight of the token's j-th slot, fetched one token ahead (written by the kernels before this
    // one: coherent loads)
    int row = -1;
    float w = 0.0f;
    if (lane < 8 && static_cast<int>(blockIdx.x) < T) {
        row = __ldcg(slot_to_row + blockIdx.x * 8 + lane);
        w = __ldcg(topk_w + blockIdx.x * 8 + lane);
    }
    for (int t = blockIdx.x; t < T; t += gridDim.x) {
        const int my_row = row;
        const float my_w = w;
        const int tn = t + static_cast<int>(gridDim.x);
        if (lane < 8 && tn < T) {
            row = __ldcg(slot_to_row + static_cast<size_t>(tn) * 8 + lane);
            w = __ldcg(topk_w + static_cast<size_t>(tn) * 8 + lane);
        }
        const uint32_t local = __ballot_sync(0xffffffffu, lane < 8 && my_row >= 0);
        const int c = blockIdx.y * blockDim.x + threadIdx.x;
        const bool live = c < groups;  // (whole warps: they shuffle)
        float acc[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[i] = 0.0f;
        for (uint32_t todo = local; todo;) {
            uint32_t u[COMBINE_BATCH][8];
            float wj[COMBINE_BATCH];
#pragma unroll
            for (int k = 0; k < COMBINE_BATCH; ++k) {
                wj[k] = 0.0f;
                if (todo) {
                    const int j = __ffs(todo) - 1;
                    todo &= todo - 1;
                    const int r = __shfl_sync(0xffffffffu, my_row, j);
                    wj[k] = __shfl_sync(0xffffffffu, my_w, j);
                    if (live) ld_global_v8(y + y_block_offset(r, c, n_tiles), u[k]);
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) u[k][i] = 0u;
                }
            }
#pragma unroll
            for (int k = 0; k < COMBINE_BATCH; ++k) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    acc[2 * i] = fmaf(wj[k], __uint_as_float(u[k][i] << 16), acc[2 * i]);
                    acc[2 * i + 1] = fmaf(wj[k], __uint_as_float(u[k][i] & 0xffff0000u), acc[2 * i + 1]);
                }
            }
        }
        if (!live) continue;
        uint32_t o[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const __nv_bfloat162 p = __floats2bfloat162_rn(acc[2 * i], acc[2 * i + 1]);
            o[i] = *reinterpret_cast<const uint32_t*>(&p);
        }
        uint4* dst = reinterpret_cast<uint4*>(out + static_cast<size_t>(t) * H + c * 16);  // 16-byte aligned
        dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
        dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
    }
}

}  // namespace moe
