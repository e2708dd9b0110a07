// Stage 2 of the Fused MoE description: per-expert histogram, exclusive scan,
// stable placement of the local (token, expert) slots into expert-contiguous
// rows (experts ascending, tokens ascending inside an expert), and the gather
// of FP8 activation rows and their 128-wide scales into that order.  All
// metadata stays on the device; nothing here synchronises with the host.
//
// Row numbering: "canonical" rows are dense (expert e starts at offset[e]);
// "padded" rows start every expert on a multiple of the GEMM tile height so a
// tile never straddles two experts.
#pragma once
#include <stdint.h>

#include "limits.cuh"
#include "ptx.cuh"
#include "routing.cuh"

namespace moe {

constexpr int TILE_M = 128;              // GEMM tile height (rows)
// A list of GEMM1 tiles in `mlp_claimed`: open to all, being worked on, open to all but its own CTA.
constexpr int LIST_OPEN = 0, LIST_CLAIMED = 1, LIST_LEFT = 2;

struct PermuteMeta {
    int* block_hist;     // [nblk, E_loc] per-block counts, turned into per-block bases by the last block
    uint8_t* slot_rank;  // [T*8] rank of a local slot among the rows of its expert inside its block of tokens
    int* expert_count;   // [E_loc]
    int* expert_offset;  // [E_loc+1] canonical (unpadded) exclusive scan
    int* padded_offset;  // [E_loc+1] exclusive scan of counts rounded up to TILE_M
    int* tile_expert;    // [max_m_tiles] local expert of each row tile
    int* tile_rows;      // [max_m_tiles] valid rows in each row tile (1..TILE_M)
    int* num_m_tiles;    // [1]
    int* mlp_ready;      // [max_m_tiles] grouped_mlp_kernel's counters, zeroed with the tables: parts of GEMM1 stored,
    int* mlp_claimed;    // [mlp_grid] lists of tiles claimed, [1] GEMM2 tiles handed out
    int mlp_grid;
    int mlp_left;        // test hook: the first lists, which their own CTAs leave to the others (0 outside of tests)
    int* slot_to_row;    // [T*8] padded row of each slot, -1 when the slot's expert is not local
    int* row_to_slot;    // [T*8] canonical row -> slot id (first S entries valid)
    int* row_token;      // [row_cap] padded row -> token (valid rows only)
    int* tok_nlocal;     // [T] local slots of each token (small batches only: route_permute_kernel / _in_cta)
    // small batches only, for the fused kernel: the row tiles cut into sub-tiles of at most 32 rows
    int* st_expert;      // [max sub-tiles] local expert
    int* st_row0;        // [max sub-tiles] first padded row (a multiple of 32)
    int* st_rows;        // [max sub-tiles] valid rows (1..32)
    int* num_st;         // [1]
};
constexpr int ST_ROWS = 32;

// Row tables of all experts from their counts, by one thread block.  In: s_cnt[e] = rows of local expert e for
// e < P_MAX_LOCAL (zero past E_loc).  Out: the tables of `m`; s_cnt / s_pad hold the exclusive scans of the counts and
// of the counts rounded up to TILE_M, the totals in entry P_MAX_LOCAL.
__device__ __forceinline__ void scan_experts(int E_loc, int* s_cnt, int* s_pad, const PermuteMeta& m) {
    const int tid = threadIdx.x, lane = tid & 31;
    __syncthreads();
    if (tid < 32) {  // lane l owns entries 8l .. 8l+7
        int c[8], sc = 0, sq = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            c[i] = s_cnt[lane * 8 + i];
            sc += c[i];
            sq += (c[i] + TILE_M - 1) / TILE_M * TILE_M;
        }
        int ec = sc, eq = sq;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int vc = __shfl_up_sync(0xffffffffu, ec, d), vq = __shfl_up_sync(0xffffffffu, eq, d);
            if (lane >= d) {
                ec += vc;
                eq += vq;
            }
        }
        int bc = ec - sc, bq = eq - sq;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            s_cnt[lane * 8 + i] = bc;
            s_pad[lane * 8 + i] = bq;
            bc += c[i];
            bq += (c[i] + TILE_M - 1) / TILE_M * TILE_M;
        }
        if (lane == 31) {
            s_cnt[P_MAX_LOCAL] = ec;
            s_pad[P_MAX_LOCAL] = eq;
            *m.num_m_tiles = eq / TILE_M;
        }
    }
    __syncthreads();
    for (int e = tid; e < E_loc; e += blockDim.x) {
        const int total = s_cnt[e + 1] - s_cnt[e];
        m.expert_count[e] = total;
        m.expert_offset[e] = s_cnt[e];
        m.padded_offset[e] = s_pad[e];
        const int t0 = s_pad[e] / TILE_M;
        for (int i = 0; i * TILE_M < total; ++i) {
            m.tile_expert[t0 + i] = e;
            m.tile_rows[t0 + i] = min(TILE_M, total - i * TILE_M);
            m.mlp_ready[t0 + i] = 0;
        }
    }
    for (int v = tid; v < m.mlp_grid; v += blockDim.x) m.mlp_claimed[v] = v < m.mlp_left ? LIST_LEFT : LIST_OPEN;
    if (tid == 0) {
        m.mlp_claimed[m.mlp_grid] = 0;
        // entries past E_loc count nothing, so entry E_loc already holds the totals
        m.expert_offset[E_loc] = s_cnt[E_loc];
        m.padded_offset[E_loc] = s_pad[E_loc];
    }
}

// Routing and everything of the permutation that needs all tokens, in one launch: one warp per token routes it, its
// block counts the rows of every expert and the rank of each of its slots among them (bit w of mask[e]: the token of
// warp w routes to local expert e; the popcount below a token's bit is its stable rank), and the block that finishes
// last -- found with a ticket counter, nobody waits -- turns the blocks' counts into bases and builds the row tables.
// What is left, one sum per slot, place_gather_kernel does where it copies the rows.  Bound by latency: the routing
// of a token is a chain of about 2 us, so a block takes few tokens (8) while the blocks fit the SMs at once, and 32
// where the counts of many blocks would make the last block's pass over them long.
// This kernel and place_gather_kernel replaced five kernels (route, count, scan, place, gather; up to 512 tokens two, the
// first of which placed all rows in its last block, equal in time): 23 us instead of 34 at 1024 tokens, 30 instead of
// 39 at 4096, 305 instead of 359 at 16384 tokens with all experts local, where a row is now read once instead of
// eight times (sums of the kernels' event times).
// `ticket` must be zero at launch; the last block leaves it zero.
constexpr int RC_SMALL_MAX_TOKENS = 1024;   // 128 blocks of 8 tokens
// Blocks of 8 tokens up to RC_SMALL_MAX_TOKENS while a thread of the last block (of 256; `ep` of them, the local experts
// rounded up to a power of two, side by side) has at most 32 blocks to sum up: T x ep <= 65536.  us per forward of a small
// layer, 32 / 8 tokens per block: 129 to 256 local experts 37.2 / 32.9 at 128 tokens, 41.3 / 39.2 at 256, 41.6 / 41.2 at 300,
// 43.3 / 44.9 at 512; 65 to 128 experts 33.0 / 28.5 at 192, 37.6 / 35.1 at 512, 39.6 / 43.3 at 700; a line at 64 local
// experts, whatever the batch, made batches of 81 to 512 tokens with more of them up to 10 % slower than the one-block
// placement that was here before.
__host__ __device__ constexpr int route_count_tokens_per_block(int T, int E_loc) {
    int ep = 1;
    while (ep < E_loc) ep <<= 1;
    return T <= RC_SMALL_MAX_TOKENS && T * ep <= 65536 ? 8 : 32;
}
template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32) route_count_kernel(
    int T, int E_loc, int off, const float* __restrict__ logits, const __nv_bfloat16* __restrict__ bias, float scaling,
    int* __restrict__ topk_idx, float* __restrict__ topk_w, PermuteMeta m, int* __restrict__ ticket,
    int* __restrict__ status) {
    pdl_launch_dependents();
    pdl_wait();
    constexpr int THREADS = WARPS * 32;
    __shared__ uint32_t mask[P_MAX_LOCAL];
    __shared__ int s_part[THREADS];
    __shared__ int s_cnt[P_MAX_LOCAL + 1];
    __shared__ int s_pad[P_MAX_LOCAL + 1];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (blockIdx.x == 0 && tid == 0) *status = DEV_OK;  // first kernel of a forward: clear the fault word
    for (int e = tid; e < P_MAX_LOCAL; e += THREADS) mask[e] = 0u;
    __syncthreads();
    const int t = blockIdx.x * WARPS + warp;
    int my_e = -1;
    if (t < T) {
        float bias_f[8];
        load_bias8(bias, lane, bias_f);
        int my_idx;
        float my_w;
        route_token(t, lane, logits, bias_f, scaling, my_idx, my_w);
        if (lane < R_TOPK) {
            topk_idx[static_cast<size_t>(t) * R_TOPK + lane] = my_idx;
            topk_w[static_cast<size_t>(t) * R_TOPK + lane] = my_w;
            const int e = my_idx - off;
            if (e >= 0 && e < E_loc) {
                my_e = e;
                atomicOr(&mask[e], 1u << warp);
            }
        }
    }
    __syncthreads();
    if (my_e >= 0)
        m.slot_rank[static_cast<size_t>(t) * R_TOPK + lane] = static_cast<uint8_t>(__popc(mask[my_e] & ((1u << warp) - 1u)));
    for (int e = tid; e < E_loc; e += THREADS) m.block_hist[static_cast<size_t>(blockIdx.x) * E_loc + e] = __popc(mask[e]);
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        const int n = atomicAdd(ticket, 1);
        s_last = (n == static_cast<int>(gridDim.x) - 1);
        if (s_last) *ticket = 0;
        // A counter that did not start at zero (somebody wrote into the workspace) would leave this forward
        // without a last block and with stale tables: say so instead of returning them silently.
        if (n < 0 || n >= static_cast<int>(gridDim.x)) {
            atomicExch(status, DEV_BAD_TICKET);
            *ticket = 0;
        }
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();

    // The counts of all blocks: thread (group q, expert e) sums a contiguous range of blocks, then replaces every
    // count of its range by the number of rows of e in front of that block.
    int ep = 1;
    while (ep < E_loc) ep <<= 1;
    const int nblk = static_cast<int>(gridDim.x);
    const int groups = min(THREADS / ep, 32), per = (nblk + groups - 1) / groups;
    const int e = tid & (ep - 1), q = tid / ep;
    const bool mine = q < groups && e < E_loc;
    const int b0 = min(nblk, q * per), b1 = min(nblk, b0 + per);
    // (the first HELD counts of a range stay in registers, which is all of them up to 16384 tokens on 32 experts and 2048
    // on 256: one round trip to L2 instead of two chains of them.  With blocks of 8 tokens the next HELD do as well, and that is
    // all there can be: left to the loops behind, what remains after whole batches of loads goes one by one, 38.0
    // against 31 us per forward at 457 tokens on 65 experts.)
    constexpr int HELD = 16;
    constexpr bool ALL_HELD = WARPS == 8;
    int held2[HELD];
    const bool more = ALL_HELD && per > HELD;  // (the same for the whole block)
    int* hist = m.block_hist + static_cast<size_t>(b0) * E_loc + e;
    int held[HELD], sum = 0;
    if (mine) {
#pragma unroll
        for (int i = 0; i < HELD; ++i) held[i] = b0 + i < b1 ? __ldcg(hist + static_cast<size_t>(i) * E_loc) : 0;
#pragma unroll
        for (int i = 0; i < HELD; ++i) sum += held[i];
        if (more) {
#pragma unroll
            for (int i = 0; i < HELD; ++i) held2[i] = b0 + HELD + i < b1 ? __ldcg(hist + static_cast<size_t>(HELD + i) * E_loc) : 0;
#pragma unroll
            for (int i = 0; i < HELD; ++i) sum += held2[i];
        }
#pragma unroll 16
        for (int i = HELD; !ALL_HELD && i < b1 - b0; ++i) sum += __ldcg(hist + static_cast<size_t>(i) * E_loc);
    }
    s_part[tid] = sum;
    for (int i = tid; i < P_MAX_LOCAL; i += THREADS) s_cnt[i] = 0;
    __syncthreads();
    if (mine) {
        int base = 0;
        for (int i = 0; i < q; ++i) base += s_part[i * ep + e];
        if (q == groups - 1) s_cnt[e] = base + sum;
#pragma unroll
        for (int i = 0; i < HELD; ++i) {
            if (b0 + i < b1) hist[static_cast<size_t>(i) * E_loc] = base;
            base += held[i];
        }
        if (more) {
#pragma unroll
            for (int i = 0; i < HELD; ++i) {
                if (b0 + HELD + i < b1) hist[static_cast<size_t>(HELD + i) * E_loc] = base;
                base += held2[i];
            }
        }
#pragma unroll 16
        for (int i = HELD; !ALL_HELD && i < b1 - b0; ++i) {
            const int c = __ldcg(hist + static_cast<size_t>(i) * E_loc);
            hist[static_cast<size_t>(i) * E_loc] = base;
            base += c;
        }
    }
    scan_experts(E_loc, s_cnt, s_pad, m);
}

// One warp per token: the padded row of each of its local slots (base of its block inside the expert + rank inside the
// block), the tables that depend on it, and the copy of the token's FP8 row (H bytes) and its H/128 scales to those
// rows, read once and written up to eight times.  The scales are written transposed ([H/128, row_cap]) so the GEMM
// epilogue reads them coalesced across the rows of a tile.  Rows past an expert's count are padding and are left
// untouched (their results are never stored).  Bound by the writes: 7392 bytes per slot.
__global__ void __launch_bounds__(256) place_gather_kernel(int T, int H, int E_loc, int off, int row_cap, int tokens_per_block,
                                                           int scale_layout, const int* topk_idx,
                                                           const uint8_t* __restrict__ hidden,
                                                           const float* __restrict__ hidden_scale, PermuteMeta m,
                                                           uint8_t* __restrict__ a1, float* __restrict__ a1_scale_t,
                                                           int* __restrict__ status) {
    const int lane = threadIdx.x & 31;
    const int nwarps = gridDim.x * (blockDim.x >> 5);
    const int chunks = H / 16, nkb = H / 128;
    constexpr int BATCH = 7;  // 16-byte chunks of a row that a lane holds at a time (a row of 7168 bytes: two batches)
    pdl_wait();
    // (only now: whoever is started by this may read the row tables without waiting for this kernel)
    pdl_launch_dependents();
    for (int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < T; t += nwarps) {
        int prow = -1;
        if (lane < R_TOPK) {
            const int slot = t * R_TOPK + lane;
            const int e = __ldcg(topk_idx + slot) - off;
            if (e >= 0 && e < E_loc) {
                const int within = __ldcg(m.block_hist + static_cast<size_t>(t / tokens_per_block) * E_loc + e) + __ldcg(m.slot_rank + slot);
                prow = __ldcg(m.padded_offset + e) + within;
                if (prow < 0 || prow >= row_cap) {
                    atomicExch(status, DEV_BAD_ROW);
                    prow = -1;
                } else {
                    m.row_to_slot[__ldcg(m.expert_offset + e) + within] = slot;
                    m.row_token[prow] = t;
                }
            }
            m.slot_to_row[slot] = prow;
        }
        const uint32_t local = __ballot_sync(0xffffffffu, prow >= 0);
        if (local == 0) continue;
        const uint4* src = reinterpret_cast<const uint4*>(hidden + static_cast<size_t>(t) * H);
        for (int cb = 0; cb < chunks; cb += 32 * BATCH) {  // (the same number of rounds for all lanes: they shuffle)
            const int c0 = cb + lane;
            uint4 v[BATCH];
#pragma unroll
            for (int i = 0; i < BATCH; ++i)
                if (c0 + i * 32 < chunks) v[i] = __ldg(src + c0 + i * 32);
            for (uint32_t todo = local; todo; todo &= todo - 1) {
                const int r = __shfl_sync(0xffffffffu, prow, __ffs(todo) - 1);
                uint4* dst = reinterpret_cast<uint4*>(a1 + static_cast<size_t>(r) * H);
#pragma unroll
                for (int i = 0; i < BATCH; ++i)
                    if (c0 + i * 32 < chunks) dst[c0 + i * 32] = v[i];
            }
        }
        for (int kb = lane; kb < (nkb + 31) / 32 * 32; kb += 32) {
            const float s = kb >= nkb ? 0.0f
                            : scale_layout ? __ldg(hidden_scale + static_cast<size_t>(kb) * T + t)
                                           : __ldg(hidden_scale + static_cast<size_t>(t) * nkb + kb);
            for (uint32_t todo = local; todo; todo &= todo - 1) {
                const int r = __shfl_sync(0xffffffffu, prow, __ffs(todo) - 1);
                if (kb < nkb) a1_scale_t[static_cast<size_t>(kb) * row_cap + r] = s;
            }
        }
    }
}

// In front of the fused small-batch kernel: routing in parallel blocks (one warp per token), then the block that
// finishes last -- found with a ticket counter, nobody waits -- builds histogram, scan and placement for all
// tokens on its own (the rows are gathered by the fused kernel).  Same arithmetic and outputs as
// route_count_kernel + place_gather_kernel, plus the tables of sub-tiles.  `ticket` must be zero at launch; the last block leaves it zero
// (moe_fp8_set_workspace zeroes it once, nothing else ever writes it).
// Dynamic shared memory: E_loc * ceil(T/32) words of masks, then as many 16-bit prefix counts.
constexpr int P_TAIL_MAX_TOKENS = 256;   // the largest batch the fused kernel takes
constexpr int P_TAIL_THREADS = 256;
__host__ __device__ constexpr size_t route_permute_smem_bytes(int T, int E_loc) {
    return static_cast<size_t>(E_loc) * ((T + 31) / 32) * 6;
}
__global__ void __launch_bounds__(P_TAIL_THREADS) route_permute_kernel(
    int T, int E_loc, int off, int row_cap, const float* __restrict__ logits, const __nv_bfloat16* __restrict__ bias,
    float scaling, int* __restrict__ topk_idx, float* __restrict__ topk_w, PermuteMeta m, int* __restrict__ ticket,
    int* __restrict__ status) {
    pdl_launch_dependents();
    pdl_wait();
    extern __shared__ uint32_t dyn_smem[];
    __shared__ int s_cnt[P_MAX_LOCAL + 1];
    __shared__ int s_pad[P_MAX_LOCAL + 1];
    __shared__ int s_warp[3][P_TAIL_THREADS / 32];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31;
    if (blockIdx.x == 0 && tid == 0) *status = DEV_OK;  // first kernel of a forward: clear the fault word
    {   // stage 1: one warp per token
        const int warps_per_block = blockDim.x >> 5;
        const int nwarps = gridDim.x * warps_per_block;
        float bias_f[8];
        load_bias8(bias, lane, bias_f);
        for (int t = blockIdx.x * warps_per_block + (tid >> 5); t < T; t += nwarps) {
            int my_idx;
            float my_w;
            route_token(t, lane, logits, bias_f, scaling, my_idx, my_w);
            if (lane < R_TOPK) {
                topk_idx[static_cast<size_t>(t) * R_TOPK + lane] = my_idx;
                topk_w[static_cast<size_t>(t) * R_TOPK + lane] = my_w;
            }
        }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        const int n = atomicAdd(ticket, 1);
        s_last = (n == static_cast<int>(gridDim.x) - 1);
        if (s_last) *ticket = 0;
        // A counter that did not start at zero (somebody wrote into the workspace) would leave this forward
        // without a last block and with stale tables: say so instead of returning them silently.
        if (n < 0 || n >= static_cast<int>(gridDim.x)) {
            atomicExch(status, DEV_BAD_TICKET);
            *ticket = 0;
        }
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();

    // stage 2 for all tokens, in this block, thread t on token t and on expert t.  Bit t of mask[e] says: token t routes
    // to local expert e.
    const int W = (T + 31) / 32;
    uint32_t* mask = dyn_smem;                                             // [E_loc][W]
    uint16_t* pre = reinterpret_cast<uint16_t*>(dyn_smem + E_loc * W);     // [E_loc][W] tokens of e below word w
    const int t = tid;
    int ids[R_TOPK];
    if (t < T) {
        const int4 a = __ldcg(reinterpret_cast<const int4*>(topk_idx) + 2 * t);
        const int4 b = __ldcg(reinterpret_cast<const int4*>(topk_idx) + 2 * t + 1);
        ids[0] = a.x - off, ids[1] = a.y - off, ids[2] = a.z - off, ids[3] = a.w - off;
        ids[4] = b.x - off, ids[5] = b.y - off, ids[6] = b.z - off, ids[7] = b.w - off;
    }
    for (int i = tid; i < E_loc * W; i += blockDim.x) mask[i] = 0u;
    __syncthreads();
    if (t < T) {
#pragma unroll
        for (int j = 0; j < R_TOPK; ++j)
            if (ids[j] >= 0 && ids[j] < E_loc) atomicOr(&mask[ids[j] * W + (t >> 5)], 1u << (t & 31));
    }
    __syncthreads();
    int total = 0;
    if (tid < E_loc)
        for (int w = 0; w < W; ++w) {
            pre[tid * W + w] = static_cast<uint16_t>(total);
            total += __popc(mask[tid * W + w]);
        }
    // exclusive scans over the experts of the counts, the padded counts and the numbers of sub-tiles: inside the warps by
    // shuffles, then over the eight warps (by one thread over 256 experts: 5 us of the forward of 33 tokens)
    const int val[3] = {total, (total + TILE_M - 1) / TILE_M * TILE_M, (total + ST_ROWS - 1) / ST_ROWS};
    int inc[3] = {val[0], val[1], val[2]};
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int o = __shfl_up_sync(0xffffffffu, inc[k], d);
            if (lane >= d) inc[k] += o;
        }
    if (lane == 31)
#pragma unroll
        for (int k = 0; k < 3; ++k) s_warp[k][tid >> 5] = inc[k];
    __syncthreads();
    int base[3] = {0, 0, 0};
    for (int w = 0; w < (tid >> 5); ++w)
#pragma unroll
        for (int k = 0; k < 3; ++k) base[k] += s_warp[k][w];
    const int cnt0 = base[0] + inc[0] - val[0], pad0 = base[1] + inc[1] - val[1], st0 = base[2] + inc[2] - val[2];
    s_cnt[tid] = cnt0;
    s_pad[tid] = pad0;
    if (tid == P_MAX_LOCAL - 1) {  // experts past E_loc count nothing: these are the totals
        *m.num_m_tiles = (pad0 + val[1]) / TILE_M;
        *m.num_st = st0 + val[2];
        m.expert_offset[E_loc] = cnt0 + val[0];
        m.padded_offset[E_loc] = pad0 + val[1];
    }
    __syncthreads();
    if (tid < E_loc) {
        m.expert_count[tid] = total;
        m.expert_offset[tid] = cnt0;
        m.padded_offset[tid] = pad0;
        for (int i = 0; i * TILE_M < total; ++i) {
            m.tile_expert[pad0 / TILE_M + i] = tid;
            m.tile_rows[pad0 / TILE_M + i] = min(TILE_M, total - i * TILE_M);
        }
        for (int i = 0; i * ST_ROWS < total; ++i) {
            m.st_expert[st0 + i] = tid;
            m.st_row0[st0 + i] = pad0 + i * ST_ROWS;
            m.st_rows[st0 + i] = min(ST_ROWS, total - i * ST_ROWS);
        }
    }
    if (t < T) {
        const int word = t >> 5, bit = t & 31;
        int nlocal = 0, prows[R_TOPK];
#pragma unroll
        for (int j = 0; j < R_TOPK; ++j) {
            const int e = ids[j];
            int prow = -1;
            if (e >= 0 && e < E_loc) {
                ++nlocal;
                const int rank = pre[e * W + word] + __popc(mask[e * W + word] & ((1u << bit) - 1u));
                prow = s_pad[e] + rank;
                if (prow < 0 || prow >= row_cap) {
                    atomicExch(status, DEV_BAD_ROW);
                    prow = -1;
                } else {
                    m.row_to_slot[s_cnt[e] + rank] = t * R_TOPK + j;
                    m.row_token[prow] = t;
                }
            }
            prows[j] = prow;
        }
        reinterpret_cast<int4*>(m.slot_to_row)[2 * t] = make_int4(prows[0], prows[1], prows[2], prows[3]);
        reinterpret_cast<int4*>(m.slot_to_row)[2 * t + 1] = make_int4(prows[4], prows[5], prows[6], prows[7]);
        m.tok_nlocal[t] = nlocal;
    }
}
static_assert(P_TAIL_THREADS == P_MAX_LOCAL && P_TAIL_THREADS >= P_TAIL_MAX_TOKENS, "a thread per expert, and per token");
static_assert(TILE_M % ST_ROWS == 0, "sub-tiles do not straddle row tiles");

// Stages 1 and 2 for a batch of at most 16 tokens, computed by ONE thread block for itself: every CTA of the
// fused small-batch kernel runs this on the same inputs and writes the same tables (to the same addresses, with
// the same values), so no CTA ever waits for another one and no separate routing launch is needed.  Same
// arithmetic and outputs as route_permute_kernel.  `scratch` is RP_CTA_SCRATCH_INTS ints of shared memory;
// the block needs at least P_MAX_LOCAL threads and T warps are busy at a time.  Ends with a block barrier after
// which every thread of the block may read the tables.
// The tiles also stay in shared memory (CtaTiles): read back from global memory, each table cost the roles a round trip to
// L2 in a chain of three or four before their first loads.
constexpr int RP_CTA_MAX_TOKENS = 16;
struct CtaTiles {
    uint2 tile[RP_CTA_MAX_TOKENS * 8];  // local expert; the set of its tokens, which are its rows in order
    int count;
    uint32_t none_local;                // the set of tokens without a local expert
};
// the r-th token of a set
__device__ __forceinline__ int set_member(uint32_t set, int r) {
    for (; r > 0; --r) set &= set - 1;
    return __ffs(set) - 1;
}
constexpr int RP_CTA_SCRATCH_INTS = RP_CTA_MAX_TOKENS * 8 + P_MAX_LOCAL + 2 * (P_MAX_LOCAL + 1);
__device__ __forceinline__ void route_permute_in_cta(int* scratch, CtaTiles& tiles, int T, int E_loc, int off, int row_cap,
                                                     const float* __restrict__ logits,
                                                     const __nv_bfloat16* __restrict__ bias, float scaling,
                                                     int* topk_idx, float* topk_w, const PermuteMeta& m, int* status) {
    int* s_idx = scratch;                                                  // [T][8] selected experts
    uint32_t* mask = reinterpret_cast<uint32_t*>(scratch + RP_CTA_MAX_TOKENS * 8);   // [P_MAX_LOCAL] bit t: token t
    int* s_cnt = scratch + RP_CTA_MAX_TOKENS * 8 + P_MAX_LOCAL;            // [P_MAX_LOCAL + 1]
    int* s_pad = s_cnt + P_MAX_LOCAL + 1;                                  // [P_MAX_LOCAL + 1]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    if (tid < P_MAX_LOCAL) mask[tid] = 0u;
    if (tid == 0) tiles.none_local = 0u;
    {
        float bias_f[8];
        load_bias8(bias, lane, bias_f);
        for (int t = warp; t < T; t += nwarps) {
            int my_idx;
            float my_w;
            route_token(t, lane, logits, bias_f, scaling, my_idx, my_w);
            if (lane < R_TOPK) {
                s_idx[t * R_TOPK + lane] = my_idx;
                topk_idx[t * R_TOPK + lane] = my_idx;
                topk_w[t * R_TOPK + lane] = my_w;
            }
        }
    }
    __syncthreads();
    if (tid < T) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int e = s_idx[tid * 8 + j] - off;
            if (e >= 0 && e < E_loc) atomicOr(&mask[e], 1u << tid);
        }
    }
    __syncthreads();
    int total = 0;
    if (tid < P_MAX_LOCAL) {
        total = tid < E_loc ? __popc(mask[tid]) : 0;
        s_cnt[tid] = total;
        s_pad[tid] = (total + TILE_M - 1) / TILE_M * TILE_M;
    }
    __syncthreads();
    if (warp == 0) {  // exclusive scans of both arrays: lane l owns entries 8l .. 8l+7
        int c[8], q[8], sc = 0, sq = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            c[i] = s_cnt[lane * 8 + i];
            q[i] = s_pad[lane * 8 + i];
            sc += c[i];
            sq += q[i];
        }
        int ec = sc, eq = sq;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int vc = __shfl_up_sync(0xffffffffu, ec, d), vq = __shfl_up_sync(0xffffffffu, eq, d);
            if (lane >= d) {
                ec += vc;
                eq += vq;
            }
        }
        int bc = ec - sc, bq = eq - sq;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            s_cnt[lane * 8 + i] = bc;
            s_pad[lane * 8 + i] = bq;
            bc += c[i];
            bq += q[i];
        }
        if (lane == 31) {
            s_cnt[P_MAX_LOCAL] = ec;
            s_pad[P_MAX_LOCAL] = eq;
        }
    }
    __syncthreads();
    if (tid < E_loc) {
        m.expert_count[tid] = total;
        m.expert_offset[tid] = s_cnt[tid];
        m.padded_offset[tid] = s_pad[tid];
        // at most RP_CTA_MAX_TOKENS rows per expert: one row tile, which is also its only sub-tile
        const int t0 = s_pad[tid] / TILE_M;
        if (total > 0) {
            tiles.tile[t0] = make_uint2(tid, mask[tid]);
            m.tile_expert[t0] = tid;
            m.tile_rows[t0] = total;
            m.st_expert[t0] = tid;
            m.st_row0[t0] = s_pad[tid];
            m.st_rows[t0] = total;
        }
    }
    if (tid == 0) {  // entries past E_loc count nothing, so entry E_loc already holds the totals
        tiles.count = s_pad[E_loc] / TILE_M;
        *m.num_m_tiles = s_pad[E_loc] / TILE_M;
        *m.num_st = s_pad[E_loc] / TILE_M;
        m.expert_offset[E_loc] = s_cnt[E_loc];
        m.padded_offset[E_loc] = s_pad[E_loc];
    }
    if (tid < T) {
        int nlocal = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int e = s_idx[tid * 8 + j] - off;
            int prow = -1;
            if (e >= 0 && e < E_loc) {
                ++nlocal;
                const int rank = __popc(mask[e] & ((1u << tid) - 1u));
                prow = s_pad[e] + rank;
                if (prow < 0 || prow >= row_cap) {
                    atomicExch(status, DEV_BAD_ROW);
                    prow = -1;
                } else {
                    m.row_to_slot[s_cnt[e] + rank] = tid * 8 + j;
                    m.row_token[prow] = tid;
                }
            }
            m.slot_to_row[tid * 8 + j] = prow;
        }
        m.tok_nlocal[tid] = nlocal;
        if (nlocal == 0) atomicOr(&tiles.none_local, 1u << tid);
    }
    __syncthreads();
}

}  // namespace moe
