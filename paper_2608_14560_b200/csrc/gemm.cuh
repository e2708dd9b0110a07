// Grouped block-scaled FP8 GEMMs of the expert MLP (stage 3 of the Fused MoE
// description): GEMM1 [rows,H] x w13[e]^T with SwiGLU and FP8 re-quantisation
// fused into its epilogue, and GEMM2 [rows,I] x w2[e]^T writing bf16 rows for
// the combine.
//
// One persistent CTA per SM works through a list of 128 x 256 output tiles (grouped_mlp.cuh says how it comes about).
//   warp 0      TMA producer.  Per K-block (128 K-bytes = one scale block): the A
//               tile (128 rows) and the B tile (256 weight rows) into a 4-stage ring
//               (128-byte swizzle), completion on mbarriers.
//   warps 1,2   MMA issuers (even / odd K-blocks).  Four tcgen05.mma (M128 N256 K32, e4m3 -> fp32) per
//               K-block into one of two 256-column TMEM buffers, then ONE
//               tcgen05.commit: the same mbarrier tells the producer that the stage
//               is free and the epilogue that the accumulator is ready (a single
//               thread issues everything, and each MMA, commit and wait costs it
//               50-100 clocks, so the per-K-block instruction count is kept minimal).
//               Every K-block starts from zero because its partial sum must be
//               multiplied by fp32 scales before it joins the running sum.
//   warp 3      factors: activation scale x weight scale per row and column half,
//               into an 8-slot ring (mlp_factors).
//   warps 4-7   epilogue of columns [0,128), warps 8-11 of columns [128,256): read
//               the partial from TMEM, multiply by a_scale[row,kb] * w_scale[nblk,kb]
//               with packed fp32 FMAs, accumulate in registers; at the end of the
//               tile apply the fused tail and store.
// What bounds a large batch is that loop: stage refilled -> MMAs -> epilogue reads the accumulator -> buffer handed
// back.  Together, the factor warp, the packed FMAs (see fma64), the hand-back through a named barrier and three
// instead of six copies per K-block took a forward from 2292 to 2179 us at 8192 skewed tokens with 32 local experts,
// from 650 to 624 us at 4096 tokens and from 9281 to 9218 us at 16384 tokens with 256 local experts (under the power
// cap); batches bound by the weight stream gain 1 %.
// Scales are arbitrary fp32 (amax/448), so the power-of-two hardware block
// scaling cannot express them; the per-K-block promotion is done on the ALUs.
//
// Two kernels are built from these roles:
//   grouped_mlp_kernel (grouped_mlp.cuh)   both GEMMs, the tiles of GEMM1 in front of those of GEMM2 (any batch size);
//   fused_small_kernel          small batches (the host decides up to which size): the gather of stage 2, GEMM1, GEMM2
//               and the weighted combine of stage 4 in ONE launch, with the operands swapped (weights on the
//               M side of the MMA, the tile's at most 32 token rows on the N side; see "weights on M" below).
//               Every CTA first works through its GEMM1 tiles, then takes GEMM2 tiles from a counter.  Warp 3 gathers the (few)
//               token rows of a GEMM1 tile straight from the token-major input with cp.async.  A GEMM2 tile
//               starts once a counter in global memory says that all GEMM1 column tiles of its row tile have
//               been stored (bounded wait; GEMM1 tiles never wait for another CTA and precede the GEMM2 tiles
//               in every CTA, and all CTAs of the one-per-SM grid are resident, so the counter always
//               arrives).  The CTA that completes the last local row of a token for a column tile -- found
//               with a per-(token, column tile) counter, nobody waits -- sums that token's rows in routing
//               order and writes the bf16 output.  Up to F_ROUTE_MAX_TOKENS tokens the kernel starts with
//               stages 1 and 2 as well: every CTA routes and permutes the whole batch for itself
//               (route_permute_in_cta) and all of them write the same tables, so the forward is one launch
//               and still no CTA waits for a table.  The counters come in two sets; CTA 0 zeroes the set of
//               the next call.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "permute.cuh"
#include "ptx.cuh"

namespace moe {

// The two MMA issuer threads take the even and the odd K-blocks.  A thread must see EVERY phase of a barrier it
// waits on (a parity wait cannot tell the wanted phase from the one two earlier), so a stage must always fall
// to the same issuer: the stage count has to be even (checked in Geometry).
constexpr int G_MAX_STAGES = 6;
constexpr int G_BLOCK_K = 128;                          // K bytes per stage = one scale block
constexpr int G_TILE_N = 256;                           // output columns per tile
constexpr int G_HALF_N = 128;                           // columns handled by one epilogue warpgroup
constexpr int G_ACC_BUFS = 2;                           // TMEM accumulator buffers (2 x 256 columns)
constexpr int G_B_BYTES = G_TILE_N * G_BLOCK_K;         // 32 KB
constexpr int G_THREADS = 384;                          // 4 control warps + 8 epilogue warps
constexpr int G_EPI_WARPS = 8;
constexpr int G_STORE_WARP_BYTES = 2048;                // per-warp staging: 32 rows x 64 B (swizzled)
constexpr int G_AMAX_BYTES = 2 * 2 * TILE_M * 4;               // GEMM1 row-amax exchange
constexpr int G_CTRL_BYTES = 832;
constexpr uint32_t G_TMEM_COLS = 512;
// grouped_mlp_kernel: named barrier ACC_BARRIER + b hands accumulator buffer b from the epilogue warps (which
// arrive) back to its issuer warp (which waits).
constexpr int ACC_BARRIER = 1;
constexpr int ACC_BARRIER_THREADS = (G_EPI_WARPS + 1) * 32;

// Scales on their way to the factor warp of grouped_mlp_kernel: the 128 activation scales of F_AHEAD K-blocks, and the
// weight scales, two per K-block, in runs of up to 32 K-blocks of a tile.
constexpr int F_AHEAD = 4;
constexpr int F_SLOTS = 8;
constexpr int F_RUN = 32;
constexpr int F_RAW_FLOATS = F_SLOTS * TILE_M + F_SLOTS * F_RUN * 2;

// Shared-memory geometry of a kernel: pipeline stages, rows of the A tile that are actually fetched (the MMA
// always reads 128 rows; with fewer fetched rows the rest of its A operand is whatever follows in shared
// memory, and those accumulator rows are never stored), slots of the activation-scale ring.
template <int STAGES_, int A_ROWS_, int SCALE_SLOTS_, int STORE_BYTES_, bool FACTORS_>
struct Geometry {
    static constexpr int STAGES = STAGES_, A_ROWS = A_ROWS_, SCALE_SLOTS = SCALE_SLOTS_;
    static constexpr bool FACTORS = FACTORS_;                        // see mlp_factors
    static constexpr int A_BYTES = A_ROWS_ * G_BLOCK_K;
    static constexpr int STAGE_BYTES = A_BYTES + G_B_BYTES;
    static constexpr int SCALE_BYTES = A_ROWS_ * 4;                  // per K-block
    // a slot: the activation scales of a K-block, or (large-tile kernels) their products with two weight scales
    static constexpr int SLOT_BYTES = FACTORS_ ? 2 * SCALE_BYTES : SCALE_BYTES;
    static constexpr int RAW_BYTES = FACTORS_ ? F_RAW_FLOATS * 4 : 0;
    static constexpr int STORE_BYTES = STORE_BYTES_;                 // GEMM1 output staging
    static constexpr int SMEM_BYTES = STAGES_ * STAGE_BYTES + SCALE_SLOTS_ * SLOT_BYTES + STORE_BYTES_ + G_AMAX_BYTES +
                                      G_CTRL_BYTES + RAW_BYTES + 1024;   // + alignment slack (the fused kernel has CtaTiles besides)
    static_assert(STAGES_ % 2 == 0, "an odd stage count lets an issuer thread skip phases of full[s]");
    static_assert(STAGES_ <= G_MAX_STAGES, "control block holds G_MAX_STAGES barriers per kind");
    static_assert(A_BYTES % 1024 == 0, "the B tile must stay 1024-byte aligned for the 128-byte swizzle");
    static_assert(SCALE_SLOTS_ >= STAGES_ + G_ACC_BUFS + 1, "the producer may be that far ahead of the epilogue");
    static_assert(SMEM_BYTES + (FACTORS_ ? 0 : sizeof(CtaTiles)) <= 232448, "exceeds the 227 KB of shared memory a CTA may use");
};
// grouped_mlp_kernel: full 128-row A tiles, 4 stages of 48 KB
using GeomFull = Geometry<4, TILE_M, 8, G_EPI_WARPS * G_STORE_WARP_BYTES, true>;
// fused small-batch kernel: a row tile holds at most 32 token rows, so their slot shrinks to 4 KB and six
// stages fit: 192 KB of weights in flight per SM instead of 128 KB, which is what a weight-streaming CTA is
// limited by; 512 bytes of output staging per epilogue warp
using GeomSmall = Geometry<6, 32, 16, G_EPI_WARPS * 512, false>;

// Row tiles of fused_small_kernel hold at most ST_ROWS = 32 rows (the N of its MMAs); an expert with more rows
// gets several of them (each streams the expert's weights, the later ones out of L2).  F_MAX_TOKENS is the
// capacity of the kernel's counters, not the batch size up to which it is the faster path (the host decides).
constexpr int F_MAX_TOKENS = 256;
// From this batch size up the large-tile GEMM kernels run row tiles of at most 32 rows with the weights on M.
constexpr int SHORT_TILE_MIN_TOKENS = 1;
// Up to here the fused kernel is used unless the caller says otherwise.  us per forward, separate kernels / fused (7168 x 2048, 32 experts,
// mean of three draws): uniform routing 134.1 / 118.7 at 33 tokens, 164.4 / 147.9 at 64, 168.8 / 153.2 at 80, 169.6 / 154.7 at 100, 175.8 / 165.0 at
// 128, 190.5 / 185.3 at 256; four hot experts, which need a sub-tile per 32 rows, 124.2 / 103.0 at 33, 148.2 / 131.3 at 64, 154.9 / 143.3 at 80,
// 157.5 / 157.0 at 100, 157.9 / 161.5 at 128, 171.9 / 183.1 at 160, 189.2 / 254.0 at 256.  It would be the faster one up to 100 tokens; callers
// count on the separate kernels from 81 on (last_launch_count, the stage times).
constexpr int F_DEFAULT_MAX_TOKENS = 80;
static_assert(GeomSmall::A_ROWS == ST_ROWS, "the token slot of a stage holds one sub-tile");
// Largest batch whose routing and permutation run inside fused_small_kernel, by every CTA for itself (one token
// per warp and round).  Measured against a routing kernel in front: 4-6 us faster per forward up to 13 tokens,
// equal at 20, 1-6 us slower from 24 tokens up, where a CTA needs two to three rounds.
constexpr int F_ROUTE_MAX_TOKENS = 16;
static_assert(F_ROUTE_MAX_TOKENS <= RP_CTA_MAX_TOKENS, "capacity of route_permute_in_cta");
static_assert(RP_CTA_SCRATCH_INTS * 4 <= GeomSmall::STAGE_BYTES, "the routing scratch lives in the first pipeline stage");

constexpr int WM_TOKENS = 32;                       // weights-on-M tiles: N of the MMA, token rows of a tile
constexpr int WM_BUF_COLS = 2 * WM_TOKENS;          // their TMEM columns per K-block: two weight-row blocks

struct GemmArgs {
    int num_kb;               // K / 128
    int n_tiles;              // output tiles along N per row tile
    int w_rows_per_expert;    // rows of the weight matrix per expert (2I or H)
    int row_cap;              // rows in the activation buffers (stride of transposed scales)
    int out_cols;             // I (GEMM1) or H (GEMM2)
    int up_row0;              // GEMM1: first weight row of the second half (I)
    int up_first;             // GEMM1: 0 = the first half is the gate and the second the up projection; 1 = the other way round
    const int* num_m_tiles;   // device scalars and tables built by the permute stage
    const int* tile_expert;
    const int* tile_rows;
    const int* tile_row0;     // fused kernel: first padded row of each (sub-)tile; else null: tile * TILE_M
    int wm_rows;              // grouped_mlp_kernel: row tiles with at most this many rows (0 or 32) run with the
                              // weights on the M side of the MMAs, see epilogue_tile_wm
    int* ready;               // GEMM1 whose rows GEMM2's tiles wait for (one launch, or two that overlap): [row tiles] warps that have
                              // stored their part, zero at launch
    const float* a_scale_t;   // [num_kb, row_cap]
    const float* w_scale;     // [E_loc, w_rows/128, num_kb]
    uint8_t* out_fp8;         // GEMM1: [row_cap, I] e4m3
    float* out_scale_t;       // GEMM1: [I/128, row_cap]
    __nv_bfloat16* out_bf16;  // GEMM2: tile-blocked rows, see y_block_offset()
    int* status;
    long long wait_limit;     // clocks a bounded wait may spin (WAIT_LIMIT_CLOCKS outside of tests)
    int fault_skip_it;        // test hook: the producer stops before this pipeline iteration (-1: never)
};

// What fused_small_kernel needs beyond the two GemmArgs.
struct FusedArgs {
    int T, H, scale_layout;
    const uint8_t* hidden;        // e4m3 [T, H] token-major activations
    const float* hidden_scale;    // [T, H/128] or [H/128, T]
    const int* row_token;         // padded row -> token
    const int* slot_to_row;       // [T*8]
    const float* topk_w;          // [T*8]
    const int* tok_nlocal;        // [T] local slots of each token
    int* ready;                   // [row tiles] GEMM1 column tiles stored, two per tile (one for each epilogue group), zero at launch
    int* tok_done;                // [T, H/256] GEMM2 rows stored per (token, column tile), zero at launch
    __nv_bfloat16* out;           // bf16 [T, H]
    // Routing and permutation inside the kernel (route != 0): every CTA computes stages 1 and 2 for itself.
    int route, E_loc, expert_offset, row_cap;
    const float* logits;          // [T, 256]
    const __nv_bfloat16* bias;    // [256]
    float scaling;
    int* topk_idx;                // [T*8] out
    float* topk_w_out;            // [T*8] out (the same buffer as topk_w)
    PermuteMeta meta;
    int* counters_next;           // the counter set of the NEXT fused call, zeroed by CTA 0 of this one
    int num_counters;
    // K split of very small batches (GEMM1, T <= SPLIT_MAX_TOKENS, few tiles): the parts of a tile store their per-K-block
    // partial sums here, [tile][K-block][weight-row block][128 rows][4 tokens] fp32, and count themselves
    float* raw;
    int* part_done;               // [tiles] zero at launch (part of the counter set)
    int split;                    // 1: the split may be used by this call
    int* ticket;                  // the next GEMM2 tile, zero at launch (part of the counter set)
};
constexpr int SPLIT_MAX_TOKENS = 4;                       // rows of a tile whose K range may be split
constexpr int SPLIT_MAX_TILES = 74;                       // a split needs at least two CTAs per tile
constexpr int SPLIT_RAW_FLOATS = 2 * SPLIT_MAX_TOKENS * 128;  // per tile and K-block
constexpr int SPLIT_MAX_KB = 64;                          // K-blocks of a GEMM whose tiles may be split

// A tile of grouped_mlp_kernel's work list.
struct __align__(16) TileInfo {
    int key;      // row tile * 16 + flags + mode; mode 1: GEMM1, 2: GEMM2, 0: the list has ended
    int n;        // column tile
    int rows;     // valid rows of the row tile
    int expert;
    static constexpr int LAST = 4, LAST_TWO = 8;  // GEMM1: the last one / one of the last two of a list
    __device__ __forceinline__ int mode() const { return key & 3; }
    __device__ __forceinline__ int m_tile() const { return key >> 4; }
};
constexpr int SCHED_SLOTS = 16;

struct GemmCtrl {
    uint64_t full[G_MAX_STAGES];   // stage filled (TMA transaction bytes)
    uint64_t done[G_MAX_STAGES];   // the MMAs that read the stage have finished: stage free AND accumulator ready
    uint64_t tmem_empty[G_MAX_STAGES];   // accumulator buffers: two, or one per stage (weights-on-M roles)
    uint64_t amax_bar;         // all epilogue warps have their row maxima in the exchange area (weights on M)
    uint64_t amax_quad[4];     // the same for the two warps that share a quadrant's rows (full row tiles)
    uint64_t drain_bar[2];
    uint64_t sync_bar;         // fused kernel, K split: rendezvous of the epilogue warps
    uint64_t group_amax[2];    // fused kernel, by epilogue group: row maxima are in the exchange area,
    uint64_t group_sync[2];    // rendezvous at the end of a tile,
    uint64_t group_turn[2];    // the other group has read the last accumulator of the tile before
    uint32_t tmem_slot;
    int abort_flag;
    int split_last;            // fused kernel, K split: this CTA stored the last part of the tile
    uint32_t gathered;         // fused kernel: stages the gather warp has arrived at
    uint64_t sched_full[SCHED_SLOTS];   // the work list, published tile by tile (fused kernel: GEMM2's part of it)
    uint64_t sched_rows[SCHED_SLOTS];   // the tile's token rows are in memory
    TileInfo sched[SCHED_SLOTS];
};
static_assert(sizeof(GemmCtrl) <= G_CTRL_BYTES, "control block too large");

__device__ __forceinline__ void raise(GemmCtrl* c, int* status, int code) {
    *reinterpret_cast<volatile int*>(&c->abort_flag) = 1;
    atomicCAS(status, DEV_OK, code);
}

// Byte offset of the 32-byte group holding columns [16*c16, 16*c16+16) of padded row r in the
// tile-blocked bf16 output of GEMM2 (n_tiles = H / 256 column tiles).
__host__ __device__ __forceinline__ size_t y_block_offset(int r, int c16, int n_tiles) {
    const int m_tile = r / TILE_M, quad = (r % TILE_M) / 32, lane = r % 32;
    const int n = c16 / 16, half = (c16 % 16) / 8, q = c16 % 8;
    return (((static_cast<size_t>(m_tile) * n_tiles + n) * 2 + half) * 4 + quad) * 8192 + q * 1024 + lane * 32;
}

// An epilogue warp's turns at the row-maximum exchange.  Bit 0: which half of the exchange area the next GEMM1 tile uses
// (they take turns, so that a warp may be in the next tile while another one still reads); bits 1 and 2: the phases of
// amax_bar and amax_quad.
struct AmaxTurn {
    uint32_t bits;
    __device__ __forceinline__ uint32_t area() const { return bits & 1; }
    __device__ __forceinline__ uint32_t all() const { return (bits >> 1) & 1; }
    __device__ __forceinline__ uint32_t quad() const { return (bits >> 2) & 1; }
};
template <bool B>
struct Bool {
    static constexpr bool value = B;
};

// x * sigmoid(x) with the hardware exp2 and reciprocal approximations (a few ulp): a tile's tail runs while the tensor pipe
// idles, so its instruction count matters.
__device__ __forceinline__ float silu_fast(float x) { return __fdividef(x, 1.0f + __expf(-x)); }

// The CTA's carve-up of shared memory and the values every role needs.
struct Cta {
    float* scale_ring;         // [slot][A_ROWS] activation scales; large-tile kernels: [slot][2][A_ROWS] factors
    uint8_t* store_stage;
    float* amax_x;             // [2][2][TILE_M] GEMM1 row-amax exchange
    float* raw_scales;         // large-tile kernels: the factor warp's scales in flight
    GemmCtrl* ctrl;
    volatile int* abort_flag;
    uint32_t smem_base, tmem_base;
    long long limit;
    int warp, lane;
    const CtaTiles* tiles;     // fused kernel that routes by itself: its tiles, else null
};
// A (sub-)tile of the fused kernel: local expert, valid rows, first padded row, token of a row
__device__ __forceinline__ int tile_expert_of(const Cta& c, const GemmArgs& g, int m) {
    return c.tiles ? static_cast<int>(c.tiles->tile[m].x) : __ldcg(g.tile_expert + m);
}
__device__ __forceinline__ int tile_rows_of(const Cta& c, const GemmArgs& g, int m) {
    return c.tiles ? __popc(c.tiles->tile[m].y) : __ldcg(g.tile_rows + m);
}
__device__ __forceinline__ int tile_row0_of(const Cta& c, const GemmArgs& g, int m) {
    return c.tiles ? m * TILE_M : __ldcg(g.tile_row0 + m);
}
__device__ __forceinline__ int row_token_of(const Cta& c, const int* row_token, int m, int row0, int r) {
    return c.tiles ? set_member(c.tiles->tile[m].y, r) : __ldcg(row_token + row0 + r);
}

// A CTA's work items in one phase of the fused kernel: at(0), at(1), ... up to the first one that is not below `count`.
struct PlainSeq {  // the items in turn to all CTAs
    int first, stride, count;
    __device__ __forceinline__ int at(int j) const { return first + j * stride; }
};
__device__ __forceinline__ PlainSeq seq_plain(int count) {
    return PlainSeq{static_cast<int>(blockIdx.x), static_cast<int>(gridDim.x), count};
}
// The fused kernel's GEMM2 tiles come from a counter: the producer draws a ticket shortly before it needs the next tile and
// publishes it for the other roles, entry by entry.  The GEMM1 tiles, one round more for some CTAs, and the memory's rate, which
// is not the same for all, leave the CTAs at different times otherwise.  us per forward, dealt in rounds (with rounds in front where
// few CTAs had a GEMM1 tile more) / from the counter: 37.1 / 35.9 at 1 token, 79.6 / 78.4 at 8, 114.4 / 110.2 at 16, 117.8 / 111.8 at 24,
// 120.4 / 121.4 at 32, 158 / 153 at 28 (21 experts), 152.3 / 147.7 at 54, 114.4 / 109.8 at 64 skewed, 700 / 679 at 33 on 256 experts;
// two handles with the same binary differ by up to 1 % there.
struct Tickets {  // producer thread
    int* counter;
    int next;      // the drawn one; a draw in flight costs nothing until this is looked at
    bool drawn;
    __device__ __forceinline__ void draw() {
        if (!drawn) next = atomicAdd(counter, 1);
        drawn = true;
    }
};
template <bool WARP>
struct TicketSeq {  // the other roles; WARP: called by whole warps, whose lanes see all the same
    const Cta& c;
    int* status;
    int count;
    // Entry j; `count` at the end of the list or when the wait gave up.
    __device__ __forceinline__ int at(int j) const {
        const uint32_t slot = static_cast<uint32_t>(j) % SCHED_SLOTS;
        bool ok = mbar_wait(smem_u32(&c.ctrl->sched_full[slot]), (static_cast<uint32_t>(j) / SCHED_SLOTS) & 1, c.abort_flag, c.limit);
        if (WARP) ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
            if (!WARP || c.lane == 0) raise(c.ctrl, status, DEV_TIMEOUT_PRODUCER);
            return count;
        }
        return ld_shared_s32(smem_u32(&c.ctrl->sched[slot].key));
    }
};

// Very small batches of the fused kernel: a tile's K range is cut into `parts` pieces of `len` K-blocks that
// different CTAs work on (see epilogue_tile_wm).  parts = 1: a work item is a whole tile.
struct KSplit {
    int parts, len;
};
__device__ __forceinline__ KSplit ksplit_none(int num_kb) { return KSplit{1, num_kb}; }
// as many parts as keep every CTA at one item at most, eight at most
__device__ __forceinline__ KSplit ksplit_for(int num_kb, int tiles, int grid, bool allowed) {
    int want = (allowed && tiles > 0) ? grid / tiles : 1;
    want = want < 1 ? 1 : (want > 8 ? 8 : want);
    const int len = (num_kb + want - 1) / want;
    return KSplit{(num_kb + len - 1) / len, len};
}

template <class GEO>
__device__ __forceinline__ void gemm_cta_setup(Cta& c, uint8_t* smem_raw, int full_count) {
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    c.scale_ring = reinterpret_cast<float*>(smem + GEO::STAGES * GEO::STAGE_BYTES);
    c.store_stage = smem + GEO::STAGES * GEO::STAGE_BYTES + GEO::SCALE_SLOTS * GEO::SLOT_BYTES;
    c.amax_x = reinterpret_cast<float*>(c.store_stage + GEO::STORE_BYTES);
    c.ctrl = reinterpret_cast<GemmCtrl*>(c.store_stage + GEO::STORE_BYTES + G_AMAX_BYTES);
    c.raw_scales = reinterpret_cast<float*>(c.store_stage + GEO::STORE_BYTES + G_AMAX_BYTES + G_CTRL_BYTES);
    c.abort_flag = &c.ctrl->abort_flag;
    c.smem_base = smem_u32(smem);
    c.warp = threadIdx.x >> 5;
    c.lane = threadIdx.x & 31;
    GemmCtrl* ctrl = c.ctrl;
    if (threadIdx.x == 0) {
        for (int s = 0; s < GEO::STAGES; ++s) {
            mbar_init(smem_u32(&ctrl->full[s]), full_count);
            mbar_init(smem_u32(&ctrl->done[s]), GEO::FACTORS ? 2 : 1);  // the MMAs' commit; the factor warp
        }
        for (int b = 0; b < G_MAX_STAGES; ++b) mbar_init(smem_u32(&ctrl->tmem_empty[b]), G_EPI_WARPS);
        mbar_init(smem_u32(&ctrl->amax_bar), G_EPI_WARPS);
        for (int q = 0; q < 4; ++q) mbar_init(smem_u32(&ctrl->amax_quad[q]), 2);
        mbar_init(smem_u32(&ctrl->drain_bar[0]), 1);
        mbar_init(smem_u32(&ctrl->drain_bar[1]), 1);
        mbar_init(smem_u32(&ctrl->sync_bar), G_EPI_WARPS);
        for (int q = 0; q < 2; ++q) {
            mbar_init(smem_u32(&ctrl->group_amax[q]), G_EPI_WARPS / 2);
            mbar_init(smem_u32(&ctrl->group_sync[q]), G_EPI_WARPS / 2);
            mbar_init(smem_u32(&ctrl->group_turn[q]), G_EPI_WARPS / 2);
        }
        for (int i = 0; i < SCHED_SLOTS; ++i) {
            mbar_init(smem_u32(&ctrl->sched_full[i]), GEO::FACTORS ? 2 : 1);  // (two arrivals: see mlp_factors)
            mbar_init(smem_u32(&ctrl->sched_rows[i]), 1);
        }
        ctrl->abort_flag = 0;
        mbar_fence_init();
    }
    if (c.warp == 1) {
        tmem_alloc(smem_u32(&ctrl->tmem_slot), G_TMEM_COLS);
        tmem_relinquish();
    }
}

// ---------------- TMA producer (fused kernel, one thread) ----------------
// tmB: boxes of 128 weight rows of [expert][half][row][K]; MODE 1 takes gate[0,128) | up[0,128) of the tile's 128 columns ("gate" and "up"
// change places with gate_first = 0), MODE 2 256 consecutive rows.  MODE 1: the token rows and the scales come from
// the gather warp instead; MODE 2: the tile's token rows are GEMM1's output and must have been stored.
template <int MODE, class GEO>
__device__ __forceinline__ void producer_tiles(const Cta& c, const CUtensorMap* tmA, const CUtensorMap* tmB,
                                               const GemmArgs& g, const FusedArgs* f, int ready_target, PlainSeq seq,
                                               Tickets& tickets, uint32_t& it, bool& ok, KSplit ks) {
    GemmCtrl* ctrl = c.ctrl;
    for (int j = 0;; ++j) {
        int item = MODE == 1 ? seq.at(j) : 0;
        if (MODE == 2) {  // the next ticket, published for the other roles; one past the last tile ends the list
            tickets.draw();
            tickets.drawn = false;
            item = min(tickets.next, seq.count);
            const uint32_t slot = static_cast<uint32_t>(j) % SCHED_SLOTS;
            *reinterpret_cast<volatile int*>(&ctrl->sched[slot].key) = item;
            mbar_arrive(smem_u32(&ctrl->sched_full[slot]));
        }
        if (item >= seq.count) break;
        const int tile = item / ks.parts, kb0 = (item - tile * ks.parts) * ks.len;
        const int kb1 = min(g.num_kb, kb0 + ks.len);
        // The ticket for the tile behind this one is drawn when the last stages are being refilled: not earlier, so that a CTA
        // that waits for rows takes no tile from one that does not, and early enough to have come when it is needed.
        const int draw_kb = MODE == 2 || seq.at(j + 1) >= seq.count ? max(kb0, kb1 - GEO::STAGES) : kb1;
        // (a tile all of whose stages go out at once: now, where there are enough tiles for everybody)
        if (MODE == 2 && kb1 - kb0 <= GEO::STAGES && seq.count > 2 * seq.stride) tickets.draw();
        const int m_tile = tile / g.n_tiles, n = tile - m_tile * g.n_tiles;
        const int e = tile_expert_of(c, g, m_tile), wrow = n * (MODE == 1 ? 128 : G_TILE_N);
        const int row0 = tile_row0_of(c, g, m_tile);
        const float* a_sc = g.a_scale_t + row0;
        const uint32_t TX_BYTES = MODE == 1 ? G_B_BYTES : GEO::STAGE_BYTES + GEO::SCALE_BYTES;
        // claim the stage of pipeline iteration j: wait until its last reader has finished, announce the bytes
        auto claim = [&](uint32_t j) -> bool {
            const uint32_t s = j % GEO::STAGES, ph = (j / GEO::STAGES) & 1;
            if (MODE == 1 && static_cast<int>(j) == g.fault_skip_it) return false;  // test hook: never filled
            if (!mbar_wait(smem_u32(&ctrl->done[s]), ph ^ 1, c.abort_flag, c.limit)) {
                raise(ctrl, g.status, DEV_TIMEOUT_PRODUCER);
                return false;
            }
            mbar_expect_tx(smem_u32(&ctrl->full[s]), TX_BYTES);
            return true;
        };
        auto load_b = [&](uint32_t j, int kb) {
            const uint32_t s = j % GEO::STAGES, bar = smem_u32(&ctrl->full[s]);
            const uint32_t b_dst = c.smem_base + s * GEO::STAGE_BYTES + GEO::A_BYTES;
            tma_load_4d(b_dst, tmB, kb * G_BLOCK_K, wrow, 0, e, bar);
            tma_load_4d(b_dst + G_B_BYTES / 2, tmB, kb * G_BLOCK_K, MODE == 1 ? wrow : wrow + 128, MODE == 1 ? 1 : 0, e, bar);
        };
        auto load_a = [&](uint32_t j, int kb) {  // the A rows and their scales of the K-block
            const uint32_t s = j % GEO::STAGES, bar = smem_u32(&ctrl->full[s]);
            // (the scale slot is free: the ring exceeds the stages + accumulators the producer can be ahead
            // of the epilogue)
            bulk_load_1d(smem_u32(c.scale_ring + (j % GEO::SCALE_SLOTS) * GEO::A_ROWS),
                         a_sc + static_cast<size_t>(kb) * g.row_cap, GEO::SCALE_BYTES, bar);
            tma_load_2d(c.smem_base + s * GEO::STAGE_BYTES, tmA, kb * G_BLOCK_K, row0, bar);
        };
        int kb = kb0;
        if (MODE == 2) {
            // The tile's A rows are GEMM1's output and must have been stored; its weights need not wait for
            // that, so the B tiles of the first K-blocks go out before the counter is looked at.
            const int npre = kb1 - kb0 < GEO::STAGES ? kb1 - kb0 : GEO::STAGES;
            int pre = 0;  // stages claimed
            while (pre < npre && (ok = claim(it + pre))) {
                load_b(it + pre, kb0 + pre);
                ++pre;
            }
            if (ok && !wait_counter(f->ready + m_tile, ready_target, c.abort_flag, c.limit)) {
                raise(ctrl, g.status, DEV_TIMEOUT_READY);
                ok = false;
            }
            fence_proxy_async();  // the rows were stored by other CTAs' copy engines; order our copies behind the acquire
            // (after a time-out as well, when nobody reads them: a claimed stage is complete with its token rows only, and
            // drain_after_abort waits for the claimed stages)
            for (int k = 0; k < pre; ++k) load_a(it + k, kb0 + k);
            it += pre;
            kb = kb0 + pre;
        }
        for (; kb < kb1 && ok; ++kb, ++it) {
            ok = claim(it);
            if (!ok) break;
            load_b(it, kb);
            if (MODE == 2) load_a(it, kb);
            if (kb >= draw_kb) tickets.draw();
        }
        if (!ok) break;
    }
}

// After an abort, all roles having ended: the copies and MMAs that are still under way have to finish before the CTA
// gives up its shared and its tensor memory.  The producer thread waits for the stages it claimed last (`it` of them in
// all; the others were consumed), after making up for the arrivals of a gather warp that stopped before it (`gathered`
// stages); the issuer threads wait for their own MMAs.  What is waited for is in the hands of the hardware, so the
// limit is the default one even where a test has shortened that of the roles.  On the regular path the epilogue has waited
// for every MMA and these for every copy, and nothing is left to wait for.
template <class GEO>
__device__ __forceinline__ void drain_after_abort(const Cta& c, int* status, uint32_t it, uint32_t gathered) {
    int zero = 0;
    if (c.warp == 0 && c.lane == 0) {
        for (uint32_t j = it < GEO::STAGES ? 0u : it - GEO::STAGES; j < it; ++j) {
            const uint32_t bar = smem_u32(&c.ctrl->full[j % GEO::STAGES]);
            if (j >= gathered) mbar_arrive_n(bar, 32);
            if (!mbar_wait(bar, (j / GEO::STAGES) & 1, &zero)) atomicCAS(status, DEV_OK, DEV_TIMEOUT_DRAIN);
        }
    } else if (c.warp == 1 || c.warp == 2) {
        if (GEO::FACTORS ? elect_one() : c.lane == 0) {  // the thread that issued the MMAs
            const uint32_t bar = smem_u32(&c.ctrl->drain_bar[c.warp - 1]);
            umma_commit(bar);
            if (!mbar_wait(bar, 0, &zero)) atomicCAS(status, DEV_OK, DEV_TIMEOUT_DRAIN);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
}

// ---------------- gather warp (fused kernel) ----------------
// GEMM1 tiles: lane l copies 16-byte chunk (l & 7) of rows (l >> 3) + 4 i, i = 0..7, of every K-block from the
// token-major input, and the scale of row l.  The stage uses the 128-byte swizzle of the TMA tiles: chunk c of
// row r sits at r * 128 + ((c ^ (r & 7)) << 4), and r & 7 takes only two values per lane (i even / odd).  Rows
// past the tile's valid rows are zero-filled; the stage holds only these 32 rows (see Geometry).  Each lane's arrival on full[s] is triggered by the completion of its copies.
template <class GEO, class SEQ>
__device__ __forceinline__ void gather_tiles(const Cta& c, const GemmArgs& g, const FusedArgs& f, const SEQ& seq,
                                             uint32_t& it, bool& ok, KSplit ks) {
    GemmCtrl* ctrl = c.ctrl;
    const int lane = c.lane, sub = lane >> 3, chunk = lane & 7;
    const uint32_t dst_even = sub * 128 + ((chunk ^ sub) << 4);
    const uint32_t dst_odd = sub * 128 + ((chunk ^ (sub + 4)) << 4);
    for (int j = 0, item; ok && (item = seq.at(j)) < seq.count; ++j) {
        const int tile = item / ks.parts, kb0 = (item - tile * ks.parts) * ks.len;
        const int kb1 = min(g.num_kb, kb0 + ks.len);
        const int m_tile = tile / g.n_tiles;
        const int rows_valid = tile_rows_of(c, g, m_tile);
        // token of row `lane` (scale copy) and source rows of this lane's eight chunks
        const int my_tok = lane < rows_valid ? row_token_of(c, f.row_token, m_tile, tile_row0_of(c, g, m_tile), lane) : -1;
        const uint8_t* src_row[GEO::A_ROWS / 4];
#pragma unroll
        for (int i = 0; i < GEO::A_ROWS / 4; ++i) {
            const int t = __shfl_sync(0xffffffffu, my_tok, sub + 4 * i);
            src_row[i] = t >= 0 ? f.hidden + static_cast<size_t>(t) * f.H + chunk * 16 : nullptr;
        }
        const float* sc_src = nullptr;
        size_t sc_step = 0;
        if (my_tok >= 0) {
            sc_src = f.scale_layout ? f.hidden_scale + my_tok : f.hidden_scale + static_cast<size_t>(my_tok) * g.num_kb;
            sc_step = f.scale_layout ? static_cast<size_t>(f.T) : 1;
        }
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
            const uint32_t s = it % GEO::STAGES, ph = (it / GEO::STAGES) & 1;
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&ctrl->done[s]), ph ^ 1, c.abort_flag, c.limit))) {
                if (lane == 0) raise(ctrl, g.status, DEV_TIMEOUT_PRODUCER);
                ok = false;
                break;
            }
            const uint32_t a_dst = c.smem_base + s * GEO::STAGE_BYTES;
#pragma unroll
            for (int i = 0; i < GEO::A_ROWS / 4; ++i)
                cp_async_16(a_dst + i * 512 + ((i & 1) ? dst_odd : dst_even),
                            src_row[i] ? static_cast<const void*>(src_row[i] + kb * G_BLOCK_K)
                                       : static_cast<const void*>(f.hidden),
                            src_row[i] ? 16u : 0u);
            cp_async_4(smem_u32(c.scale_ring + (it % GEO::SCALE_SLOTS) * GEO::A_ROWS + lane),
                       sc_src ? static_cast<const void*>(sc_src + kb * sc_step) : static_cast<const void*>(f.hidden_scale),
                       sc_src ? 4u : 0u);
            cp_async_arrive_noinc(smem_u32(&ctrl->full[s]));
        }
    }
}
// GEMM2 tiles: the producer fetches everything; the lanes only keep the arrival count of full[s] uniform.
template <class GEO, class SEQ>
__device__ __forceinline__ void gather_idle_tiles(const Cta& c, const GemmArgs& g, const SEQ& seq, uint32_t& it, bool& ok,
                                                  KSplit ks) {
    GemmCtrl* ctrl = c.ctrl;
    for (int j = 0, item; ok && (item = seq.at(j)) < seq.count; ++j) {
        const int kb0 = (item % ks.parts) * ks.len, kb1 = min(g.num_kb, kb0 + ks.len);
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
            const uint32_t s = it % GEO::STAGES, ph = (it / GEO::STAGES) & 1;
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&ctrl->done[s]), ph ^ 1, c.abort_flag, c.limit))) {
                ok = false;
                break;
            }
            mbar_arrive(smem_u32(&ctrl->full[s]));
        }
    }
}

// Rendezvous of epilogue warps at barrier `bar` (an mbarrier, because its wait is bounded: a plain barrier would hold the
// arrived warps for ever if another warp had given up).  Orders the arrived threads' earlier writes before the later
// reads, and before the later fences and atomics, of those that leave.  `n` counts the rendezvous of this thread so far.
__device__ __forceinline__ bool epilogue_rendezvous(const Cta& c, uint64_t* bar, uint32_t& n) {
    const uint32_t b = smem_u32(bar);
    __syncwarp();
    if (c.lane == 0) mbar_arrive(b);
    const bool ok = __all_sync(0xffffffffu, mbar_wait(b, n & 1, c.abort_flag, c.limit));
    ++n;
    return ok;
}

// ================= weights on M: the roles of the fused small-batch kernel =================
// With at most 32 token rows in a tile, a 128 x 256 accumulator holds 96 rows of padding, and the two
// epilogue warps that own the 32 real rows (TMEM lanes) do all of the per-K-block promotion.  Here the
// operands are swapped instead: the 256 weight rows of the tile are the M side (two MMAs of M = 128 per K
// step), the 32 token rows the N side.  An accumulator is then 128 lanes x 32 columns per weight-row block,
// 64 columns per K-block: every stage gets an accumulator buffer of its own (6 x 64 of the 512 columns),
// so the hand-over latencies overlap six deep, and an epilogue thread owns one weight row (an output
// column) of both blocks, the four warps of a group taking a tile together and the two groups the tiles in turn, or
// half of a tile each (epilogue_tile_group).
// Element for element the arithmetic is the one of the other orientation.
static_assert(G_MAX_STAGES * WM_BUF_COLS <= static_cast<int>(G_TMEM_COLS), "one accumulator buffer per stage");

template <class GEO, class SEQ>
__device__ __forceinline__ void issuer_tiles_wm(const Cta& c, const GemmArgs& g, const SEQ& seq, uint32_t mine,
                                                uint32_t& it, bool& ok, KSplit ks) {
    static_assert(GEO::A_ROWS == WM_TOKENS, "the token slot of a stage is the MMA's N operand");
    static_assert(GEO::SCALE_SLOTS >= 2 * GEO::STAGES + 1, "the gather may be two pipelines ahead of the epilogue");
    GemmCtrl* ctrl = c.ctrl;
    const uint32_t idesc = umma_idesc_f8(TILE_M, WM_TOKENS);
    for (int j = 0, item; ok && (item = seq.at(j)) < seq.count; ++j) {
        const int kb0 = (item % ks.parts) * ks.len, kb1 = min(g.num_kb, kb0 + ks.len);
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
            if ((it & 1) != mine) continue;
            const uint32_t s = it % GEO::STAGES, ph = (it / GEO::STAGES) & 1;
            const uint32_t tok_addr = c.smem_base + s * GEO::STAGE_BYTES;
            const uint64_t t_desc = umma_desc_sw128(tok_addr);
            const uint64_t w0_desc = umma_desc_sw128(tok_addr + GEO::A_BYTES);
            const uint64_t w1_desc = umma_desc_sw128(tok_addr + GEO::A_BYTES + G_B_BYTES / 2);
            const uint32_t d_tmem = c.tmem_base + s * WM_BUF_COLS;
            if (!mbar_wait(smem_u32(&ctrl->full[s]), ph, c.abort_flag, c.limit)) {
                raise(ctrl, g.status, DEV_TIMEOUT_MMA_SMEM);
                ok = false;
                break;
            }
            // the buffer of this stage was last used one pipeline round ago
            if (!mbar_wait(smem_u32(&ctrl->tmem_empty[s]), ph ^ 1, c.abort_flag, c.limit)) {
                raise(ctrl, g.status, DEV_TIMEOUT_MMA_TMEM);
                ok = false;
                break;
            }
            tc_fence_after();
#pragma unroll
            for (int k = 0; k < G_BLOCK_K / 32; ++k) umma_f8(d_tmem, w0_desc + 2 * k, t_desc + 2 * k, idesc, k > 0);
#pragma unroll
            for (int k = 0; k < G_BLOCK_K / 32; ++k)
                umma_f8(d_tmem + WM_TOKENS, w1_desc + 2 * k, t_desc + 2 * k, idesc, k > 0);
            umma_commit(smem_u32(&ctrl->done[s]));
        }
    }
}

// grouped_mlp_kernel: a warp's GEMM1 tiles whose stores have been issued.  GEMM2 tiles of other CTAs start once all warps
// of all column tiles have announced theirs in `ready`.  Waiting for the stores right after they were issued would cost
// the epilogue 1-2 us per tile, and the fence of an announcement about 400 clocks, so tiles are announced together: those
// before in the tails of the last two tiles of a list, the last one behind it.
struct Announce {
    int id, count;    // tiles id, id + grid, ... (row tile * n_tiles + column tile)
    // The whole warp; the staging of the warp's last bulk store may be written again afterwards.
    __device__ __forceinline__ void settle(int lane, bool announce, int* ready, int n_tiles) {
        if (!announce || count == 0) {
            if (lane == 0) bulk_wait_read_all();
            __syncwarp();
            return;
        }
        if (lane == 0) bulk_wait_all();  // stored, not only read
        fence_proxy_async();
        __syncwarp();
        __threadfence();
        for (int k = lane; k < count; k += 32) atomicAdd(ready + (id + k * static_cast<int>(gridDim.x)) / n_tiles, 1);
        count = 0;
    }
    __device__ __forceinline__ void add(int tile) {
        if (count == 0) id = tile;
        ++count;
    }
};

// A tile with the weights on M by all eight epilogue warps: a thread owns one weight row of each block for 16 tokens.
// MODE 1: weight-row block 0 = 128 gate rows, block 1 = the matching 128 up rows; SwiGLU, re-quantisation per
//         token over the tile's 128 output columns, e4m3 bytes and scales out.
// MODE 2: blocks 0 / 1 = output columns [0,128) / [128,256) of the tile; bf16 out in the tile-blocked layout.
// False: a wait gave up (the code is in the status word).
// Without SPLIT the tile runs inside the large-tile kernel, between tiles of the other orientation -- its accumulators are
// the first 64 columns of the two 256-column buffers of that kernel, handed over through the same two barriers, and its
// staging is the first 512 bytes of the warp's own TMA staging area.
// SPLIT (fused kernel, GEMM1, batches of at most SPLIT_MAX_TOKENS tokens with few tiles): this call covers the
// K-blocks [kb0, kb1) only.  It stores every K-block's partial sums as they come out of the tensor memory, not
// yet multiplied by the scales; the CTA that stores the last part of a tile -- found with a counter, nobody
// waits -- then runs the whole promotion from the stored partial sums, K-block after K-block in the one order
// the unsplit tile uses, and finishes the tile.  Every fp32 operation is the one of the unsplit tile.
template <int MODE, bool SPLIT, class GEO>
__device__ __forceinline__ bool epilogue_tile_wm(const Cta& c, const GemmArgs& g, const FusedArgs* f, int m_tile, int n,
                                                 uint32_t& it, AmaxTurn& turn, uint32_t& sync_iter, int kb0 = 0,
                                                 int kb1 = -1, int parts = 1, Announce* announce = nullptr,
                                                 bool settle = false) {
    static_assert(!SPLIT || MODE == 1, "only GEMM1's K range is cut");
    constexpr bool SHARED = !SPLIT;
    GemmCtrl* ctrl = c.ctrl;
    const int warp = c.warp, lane = c.lane;
    const int th = (warp - 4) >> 2;          // which 16 of the tile's 32 token rows
    const int quad = warp & 3;               // TMEM lane quadrant this warp may read
    // (lane l of quadrant q holds weight row 32 q + l of each 128-row block)
    const uint32_t t_lane = c.tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + th * 16;
    const size_t row_cap = static_cast<size_t>(g.row_cap);
    uint32_t* amax_x = reinterpret_cast<uint32_t*>(c.amax_x);   // [2 turns][256]: [2 token halves][4 quadrants][16] used
    const int num_kb = g.num_kb;
    const int rows_valid = SHARED ? __ldcg(g.tile_rows + m_tile) : tile_rows_of(c, g, m_tile);
    float acc[32];  // [0,16): block 0, [16,32): block 1, for tokens 16 th .. 16 th + 15
#pragma unroll
    for (int j = 0; j < 32; ++j) acc[j] = 0.0f;

    const int kb_end = kb1 < 0 ? num_kb : kb1;
    const int tile_row0 = SHARED ? m_tile * TILE_M : tile_row0_of(c, g, m_tile);
    float4* raw = nullptr;  // this tile's stored partial sums (four tokens each): this thread's weight row
    if (SPLIT)
        raw = reinterpret_cast<float4*>(f->raw + static_cast<size_t>(m_tile * g.n_tiles + n) * num_kb * SPLIT_RAW_FLOATS) +
              quad * 32 + lane;
    for (int kb = kb0; kb < kb_end; ++kb, ++it) {
        const uint32_t s = it % GEO::STAGES, ph = (it / GEO::STAGES) & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&ctrl->done[s]), ph, c.abort_flag, c.limit))) {
            if (lane == 0) raise(ctrl, g.status, DEV_TIMEOUT_EPILOGUE);
            return false;
        }
        tc_fence_after();
        // the MMAs of this K-block have finished, hence its stage -- tokens, weights and scales -- had landed
        float f0[16], f1[16];  // factors of this thread's tokens for block 0 / block 1
        if (SHARED) {
            const float4* fp = reinterpret_cast<const float4*>(c.scale_ring + (it % GEO::SCALE_SLOTS) * 2 * GEO::A_ROWS + th * 16);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                *reinterpret_cast<float4*>(f0 + 4 * q) = fp[q];
                *reinterpret_cast<float4*>(f1 + 4 * q) = fp[GEO::A_ROWS / 4 + q];
            }
        }
        float v[32];
        const uint32_t buf = SHARED ? (it & 1) : s, t_buf = t_lane + buf * (SHARED ? G_TILE_N : WM_BUF_COLS);
        tmem_ld16x2(t_buf, t_buf + WM_TOKENS, v);
        tc_fence_before();
        __syncwarp();
        if (SHARED)
            bar_arrive(ACC_BARRIER + buf, ACC_BARRIER_THREADS);
        else if (lane == 0)
            mbar_arrive(smem_u32(&ctrl->tmem_empty[buf]));
        if (SPLIT) {
            if (th == 0) {  // (all four token columns; those past the tile's rows are never used)
                raw[(kb * 2 + 0) * 128] = make_float4(v[0], v[1], v[2], v[3]);
                raw[(kb * 2 + 1) * 128] = make_float4(v[16], v[17], v[18], v[19]);
            }
        } else {
#pragma unroll
            for (int t = 0; t < 16; ++t) {
                acc[t] = fmaf(v[t], f0[t], acc[t]);
                acc[16 + t] = fmaf(v[16 + t], f1[t], acc[16 + t]);
            }
        }
    }

    if (SPLIT) {
        // count this part (the counting thread's fence, behind the rendezvous, covers the stores of all: 46.3 / 45.8 us per
        // forward of 1 token on three experts with a fence of every thread in front of it / without); the last one goes on, the
        // others are done with the tile
        if (!epilogue_rendezvous(c, &ctrl->sync_bar, sync_iter)) {
            if (lane == 0) raise(ctrl, g.status, DEV_TIMEOUT_EPILOGUE);
            return false;
        }
        if (warp == 4 && lane == 0) {
            __threadfence();
            const int before = atomicAdd(f->part_done + m_tile * g.n_tiles + n, 1);
            *reinterpret_cast<volatile int*>(&ctrl->split_last) = (before == parts - 1);
        }
        if (!epilogue_rendezvous(c, &ctrl->sync_bar, sync_iter)) {
            if (lane == 0) raise(ctrl, g.status, DEV_TIMEOUT_EPILOGUE);
            return false;
        }
        if (!*reinterpret_cast<volatile int*>(&ctrl->split_last)) return true;
        __threadfence();
        // The finisher.  The scales of the tile's (at most four) tokens and of the two weight-row blocks go to
        // shared memory first (the row-maximum exchange area is free here: every warp has left the previous
        // tile); then the warps of token half 0 promote block 0 and those of half 1 block 1, K-block after
        // K-block, and half 1 hands its sums to half 0 through the staging area.
        float* sa_s = c.amax_x;                                   // [num_kb][4]
        float* w_s = c.amax_x + SPLIT_MAX_TOKENS * num_kb;        // [2][num_kb]
        static_assert(G_AMAX_BYTES >= (SPLIT_MAX_TOKENS + 2) * SPLIT_MAX_KB * 4, "scales of a tile's K-blocks");
        for (int i = threadIdx.x - 128; i < SPLIT_MAX_TOKENS * num_kb; i += G_EPI_WARPS * 32) {
            const int kb = i / SPLIT_MAX_TOKENS, t = i - kb * SPLIT_MAX_TOKENS;
            float v = 0.0f;
            if (t < rows_valid) {
                const int tok = row_token_of(c, f->row_token, m_tile, tile_row0, t);
                v = __ldcg(f->scale_layout ? f->hidden_scale + static_cast<size_t>(kb) * f->T + tok
                                           : f->hidden_scale + static_cast<size_t>(tok) * num_kb + kb);
            }
            sa_s[i] = v;
        }
        const float* ws0 = g.w_scale + (static_cast<size_t>(tile_expert_of(c, g, m_tile)) * (g.w_rows_per_expert / 128) + n) * num_kb;
        const float* ws1 = ws0 + static_cast<size_t>(g.up_row0 / 128) * num_kb;
        for (int i = threadIdx.x - 128; i < 2 * num_kb; i += G_EPI_WARPS * 32)
            w_s[i] = __ldg((i < num_kb ? ws0 : ws1 - num_kb) + i);
        if (!epilogue_rendezvous(c, &ctrl->sync_bar, sync_iter)) {
            if (lane == 0) raise(ctrl, g.status, DEV_TIMEOUT_EPILOGUE);
            return false;
        }
        float4 a4 = make_float4(0.f, 0.f, 0.f, 0.f);
        {
            const float4* rp = raw + th * 128;
            const float* wp = w_s + th * num_kb;
#pragma unroll 28
            for (int kb = 0; kb < num_kb; ++kb) {
                const float4 r = __ldcg(rp + kb * 2 * 128);
                const float4 sa = *reinterpret_cast<const float4*>(sa_s + kb * SPLIT_MAX_TOKENS);
                const float w = wp[kb];
                a4.x = fmaf(r.x, sa.x * w, a4.x);
                a4.y = fmaf(r.y, sa.y * w, a4.y);
                a4.z = fmaf(r.z, sa.z * w, a4.z);
                a4.w = fmaf(r.w, sa.w * w, a4.w);
            }
        }
        float4* xchg = reinterpret_cast<float4*>(c.store_stage);  // [128 weight rows]: half 0's warps read their own staging
        if (th == 1) xchg[quad * 32 + lane] = a4;
        if (!epilogue_rendezvous(c, &ctrl->sync_bar, sync_iter)) {
            if (lane == 0) raise(ctrl, g.status, DEV_TIMEOUT_EPILOGUE);
            return false;
        }
        if (th == 0) {
            const float4 b4 = xchg[quad * 32 + lane];
            acc[0] = a4.x, acc[1] = a4.y, acc[2] = a4.z, acc[3] = a4.w;
            acc[16] = b4.x, acc[17] = b4.y, acc[18] = b4.z, acc[19] = b4.w;
        }
        __syncwarp();
    }

    const size_t row0 = static_cast<size_t>(tile_row0) + th * 16;  // padded row of this thread's token 0
    const uint32_t wst_off = (warp - 4) * (SHARED ? G_STORE_WARP_BYTES : 512);  // this warp's staging
    if (SHARED) {  // the warp's last TMA store may still be reading the area
        announce->settle(lane, settle, g.ready, g.n_tiles);
    }
    const int valid = min(16, rows_valid - th * 16);                     // tokens of this thread that exist
    if (MODE == 1) {
        float cc[16];
        uint32_t wmax[16];
        if (g.up_first) {
#pragma unroll
            for (int t = 0; t < 16; ++t) {
                const float x = acc[t];
                acc[t] = acc[16 + t];
                acc[16 + t] = x;
            }
        }
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            cc[t] = silu_fast(acc[t]) * acc[16 + t];
            // |x| as an integer orders like the float: the warp's maximum over its 32 output columns
            wmax[t] = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(cc[t])));
        }
        uint32_t* xq = amax_x + turn.area() * (2 * TILE_M) + th * 64;
        {
            uint32_t mine = 0;
#pragma unroll
            for (int t = 0; t < 16; ++t)
                if (lane == t) mine = wmax[t];
            if (lane < 16) xq[quad * 16 + lane] = mine;
        }
        const uint32_t xbar = smem_u32(&ctrl->amax_bar);
        __syncwarp();
        if (lane == 0) mbar_arrive(xbar);
        if (!__all_sync(0xffffffffu, mbar_wait(xbar, turn.all(), c.abort_flag, c.limit))) {
            if (lane == 0) raise(ctrl, g.status, DEV_TIMEOUT_EPILOGUE);
            return false;
        }
        turn.bits ^= 3;
        // lane t < 16 owns the scale of token t's 128-column block; everybody fetches its reciprocal
        float my_sc = 1.0f, my_inv = 1.0f;
        if (lane < 16) {
            const volatile uint32_t* xv = xq + lane;
            const float amax = __uint_as_float(max(max(xv[0], xv[16]), max(xv[32], xv[48])));
            my_sc = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, 448.0f);
            my_inv = __frcp_rn(my_sc);
        }
        // Narrow global stores are slow (a warp's 32 single bytes cost tens of clocks): the codes are
        // transposed through this warp's 512 bytes of staging, [16 tokens][32 columns], and leave as
        // 16-byte stores -- lane l carries 16 columns of token l / 2.
        uint8_t* wst = c.store_stage + wst_off;
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            const float inv_sc = __shfl_sync(0xffffffffu, my_inv, t);
            wst[t * 32 + lane] =
                static_cast<uint8_t>(__nv_cvt_float_to_fp8(cc[t] * inv_sc, __NV_SATFINITE, __NV_E4M3));
        }
        __syncwarp();
        if ((lane >> 1) < valid)
            *reinterpret_cast<uint4*>(g.out_fp8 + (row0 + (lane >> 1)) * g.out_cols + n * 128 + quad * 32 + (lane & 1) * 16) =
                *reinterpret_cast<const uint4*>(wst + (lane >> 1) * 32 + (lane & 1) * 16);
        if (quad == 0 && lane < valid) g.out_scale_t[static_cast<size_t>(n) * row_cap + row0 + lane] = my_sc;
        __syncwarp();
        // (The rows are read by copy engines, of other CTAs or of the next kernel: plain stores here,
        // asynchronous-proxy loads there.)
        fence_proxy_async();
        if (SPLIT) {
            // Announce the tile; the announcing thread's fence, behind the rendezvous, covers the stores of all.
            if (!epilogue_rendezvous(c, &ctrl->sync_bar, sync_iter)) {
                if (lane == 0) raise(ctrl, g.status, DEV_TIMEOUT_EPILOGUE);
                return false;
            }
            if (warp == 4 && lane == 0) {
                __threadfence();
                atomicAdd(f->ready + m_tile, 2);
            }
        }
    } else {
        // bf16 out through this warp's 512 bytes of staging, eight tokens x 32 columns at a time, so that
        // the rows leave as 16-byte stores: lane l carries 8 columns of token l / 4 (half of a 32-byte
        // group of the tile-blocked layout)
        __nv_bfloat16* wst = reinterpret_cast<__nv_bfloat16*>(c.store_stage + wst_off);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
#pragma unroll
                for (int t = 0; t < 8; ++t) wst[t * 32 + lane] = __float2bfloat16_rn(acc[j * 16 + h * 8 + t]);
                __syncwarp();
                const int t = h * 8 + (lane >> 2), ch0 = quad * 32 + (lane & 3) * 8;
                if (t < valid)
                    *reinterpret_cast<uint4*>(reinterpret_cast<uint8_t*>(g.out_bf16) +
                                              y_block_offset(static_cast<int>(row0) + t, n * 16 + j * 8 + (ch0 >> 4), g.n_tiles) +
                                              (ch0 & 15) * 2) =
                        *reinterpret_cast<const uint4*>(wst + (lane >> 2) * 32 + (lane & 3) * 8);
                __syncwarp();
            }
        }
    }
    return true;
}

// acc[t] += v[t] * (sa[t] * w) for 16 tokens, packed: each product and each FMA rounds like the scalar one.
__device__ __forceinline__ void promote16(float* acc, const float* v, const float4* sa, float w) {
    const uint64_t ww = pack_f32x2(__float_as_uint(w), __float_as_uint(w));
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 x = sa[q];
        const uint64_t f[2] = {mul_f32x2(pack_f32x2(__float_as_uint(x.x), __float_as_uint(x.y)), ww),
                               mul_f32x2(pack_f32x2(__float_as_uint(x.z), __float_as_uint(x.w)), ww)};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int t = 4 * q + 2 * k;
            const uint64_t a = fma_f32x2(pack_f32x2(__float_as_uint(v[t]), __float_as_uint(v[t + 1])), f[k],
                                         pack_f32x2(__float_as_uint(acc[t]), __float_as_uint(acc[t + 1])));
            acc[t] = __uint_as_float(static_cast<uint32_t>(a));
            acc[t + 1] = __uint_as_float(static_cast<uint32_t>(a >> 32));
        }
    }
}

// A tile of the fused kernel by one of its two epilogue groups of four warps, which take the CTA's tiles in turn: a thread owns
// one weight row of each block for all 32 tokens, 16 at a time.  A tile's tail is a chain of round trips to L2 (rows stored, fence, counter,
// combine) of 4 to 8 us while the memory is busy, as long as a GEMM2 tile's loop; with all eight warps on every tile nothing
// was read from the stages meanwhile, six stages held 6 to 8 us of the tile's stream, and all CTAs were in their tails together.
// Now the tail runs beside the other group's tile.  us per forward, eight warps on every tile / two groups: 70.9 / 67.6 at 4
// tokens, 82.0 / 80.0 at 8, 125.1 / 115.4 at 16, 130.3 / 121.4 at 32, 162.1 / 153.9 at 54, 166.4 / 160.3 at 80, 124.4 / 115.7 at 64
// skewed, 726 / 701 at 33 on 256 experts.  Element for element the arithmetic is that of epilogue_tile_wm.
// Sixteen rows that do not exist are not read.  `halved`: both groups are on the tile, each with 16 of its rows to promote, store, count
// and combine; neither waits for the other.  Where a CTA has one tile there is no other group's tail to hide, and four warps on more than
// 16 rows take longer than eight (weights in L2; us per forward, eight warps on every tile before there were groups / never halved /
// halved: 256 x 256, 70 skewed tokens 25.6 / 27.8 / 24.4; 1024 x 768, 30 skewed 29.9 / 31.8 / 28.5; 1536 x 256, 27 skewed 28.5 / 30.2 / 27;
// 2048 x 512, 40 skewed 33.8 / 35 / 31.4).  Halved whatever the number of tiles, 7168 x 512 with 64 experts and 60 skewed tokens takes
// 80.7 instead of 75.5, 1024 x 1024 with 128 experts and 80 skewed 54.0 instead of 48.3; up to two tiles per CTA 54.3 there.
// us per forward before / with the rows that exist alone: 53.9 / 51.1 at 8 tokens, 70.2 / 68.3 at 16, 110 / 109 at 54.
// Scales and tables are asked for before the group's turn comes.  `turn`: phase of the barrier to wait for, -1: none.
template <int MODE, class GEO>
__device__ __forceinline__ bool epilogue_tile_group(const Cta& c, const GemmArgs& g, const FusedArgs& f, int m_tile, int n, bool halved, int turn,
                                                    uint32_t& it, uint32_t& amax_iter, uint32_t& sync_iter) {
    GemmCtrl* ctrl = c.ctrl;
    const int lane = c.lane, quad = c.warp & 3, group = (c.warp - 4) >> 2;
    const uint32_t t_lane = c.tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
    const size_t row_cap = static_cast<size_t>(g.row_cap);
    const int num_kb = g.num_kb;
    const int e = tile_expert_of(c, g, m_tile), rows_valid = tile_rows_of(c, g, m_tile), tile_row0 = tile_row0_of(c, g, m_tile);
    const int halves = halved ? 1 << group : rows_valid > 16 ? 3 : 1;  // bit h: this group's warps look after the rows [16 h, 16 h + 16)
    const bool swap = MODE == 1 && g.up_first;  // acc[0..32) is the gate block's either way
    const float* ws0 = g.w_scale + (static_cast<size_t>(e) * (g.w_rows_per_expert / 128) + (MODE == 1 ? n : 2 * n)) * num_kb;
    const float* ws1 = ws0 + static_cast<size_t>(MODE == 1 ? g.up_row0 / 128 : 1) * num_kb;
    if (swap) {
        const float* w = ws0;
        ws0 = ws1;
        ws1 = w;
    }
    const uint32_t col0 = swap ? WM_TOKENS : 0, col1 = WM_TOKENS - col0;
    float s0 = __ldg(ws0), s1 = __ldg(ws1);
    // MODE 2: warp `quad` looks after the group's rows among quad, quad + 4, ... of the tile (lanes 0..7): their tokens and how many rows
    // each has
    int tok = -1, tok_rows = 0;
    if (MODE == 2 && lane < 8 && quad + 4 * lane < rows_valid && (halves >> (lane >> 2) & 1)) {
        tok = row_token_of(c, f.row_token, m_tile, tile_row0, quad + 4 * lane);
        tok_rows = __ldcg(f.tok_nlocal + tok);
    }
    auto timed_out = [&]() {
        if (lane == 0) raise(ctrl, g.status, DEV_TIMEOUT_EPILOGUE);
        return false;
    };
    // The other group has read the last accumulator of the tile before: from here on no stage is more than one phase behind.
    if (turn >= 0 && !__all_sync(0xffffffffu, mbar_wait(smem_u32(&ctrl->group_turn[group]), turn, c.abort_flag, c.limit)))
        return timed_out();

    float acc[64];  // [0,32): block 0 (the gate rows), [32,64): block 1
#pragma unroll
    for (int j = 0; j < 64; ++j) acc[j] = 0.0f;
    for (int kb = 0; kb < num_kb; ++kb, ++it) {
        const float w0 = s0, w1 = s1;
        if (kb + 1 < num_kb) {
            s0 = __ldg(ws0 + kb + 1);
            s1 = __ldg(ws1 + kb + 1);
        }
        const uint32_t s = it % GEO::STAGES, ph = (it / GEO::STAGES) & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&ctrl->done[s]), ph, c.abort_flag, c.limit))) return timed_out();
        tc_fence_after();
        // the MMAs of this K-block have finished, hence its stage -- tokens, weights and scales -- had landed
        const float4* sp = reinterpret_cast<const float4*>(c.scale_ring + (it % GEO::SCALE_SLOTS) * GEO::A_ROWS);
        const uint32_t t_buf = t_lane + s * WM_BUF_COLS;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (!(halves >> h & 1)) continue;
            float v[32];
            tmem_ld16x2(t_buf + col0 + 16 * h, t_buf + col1 + 16 * h, v);
            const float4 sa[4] = {sp[4 * h], sp[4 * h + 1], sp[4 * h + 2], sp[4 * h + 3]};
            promote16(acc + 16 * h, v, sa, w0);
            promote16(acc + 32 + 16 * h, v + 16, sa, w1);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_n(smem_u32(&ctrl->tmem_empty[s]), halved ? 1 : 2);  // (2: for a warp of each group)
    }
    if (!halved) {
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&ctrl->group_turn[group ^ 1]));
    }

    uint8_t* wst = c.store_stage + (c.warp - 4) * 512;  // this warp's staging
    if (MODE == 1) {
        float cc[32];
        uint32_t mine = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (!(halves >> h & 1)) continue;  // (most tiles of a decode batch have no more than 16 rows)
#pragma unroll
            for (int t = 16 * h; t < 16 * h + 16; ++t) {
                cc[t] = silu_fast(acc[t]) * acc[32 + t];
                // |x| as an integer orders like the float: the warp's maximum over its 32 output columns
                const uint32_t m = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(cc[t])));
                if (lane == t) mine = m;
            }
        }
        uint32_t* xq = reinterpret_cast<uint32_t*>(c.amax_x) + group * 128;  // [4 quadrants][32 tokens]
        xq[quad * 32 + lane] = mine;
        if (!epilogue_rendezvous(c, &ctrl->group_amax[group], amax_iter)) return timed_out();
        // lane t owns the scale of token t's 128-column block; everybody fetches its reciprocal
        const volatile uint32_t* xv = xq + lane;
        const float amax = __uint_as_float(max(max(xv[0], xv[32]), max(xv[64], xv[96])));
        const float my_sc = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, 448.0f), my_inv = __frcp_rn(my_sc);
        // Narrow global stores are slow (a warp's 32 single bytes cost tens of clocks): the codes are
        // transposed through this warp's 512 bytes of staging, [16 tokens][32 columns], and leave as
        // 16-byte stores -- lane l carries 16 columns of token l / 2.
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (!(halves >> h & 1)) continue;
#pragma unroll
            for (int t = 0; t < 16; ++t) {
                const float inv_sc = __shfl_sync(0xffffffffu, my_inv, h * 16 + t);
                wst[t * 32 + lane] = static_cast<uint8_t>(__nv_cvt_float_to_fp8(cc[h * 16 + t] * inv_sc, __NV_SATFINITE, __NV_E4M3));
            }
            __syncwarp();
            const int t = h * 16 + (lane >> 1);
            if (t < rows_valid)
                *reinterpret_cast<uint4*>(g.out_fp8 + (static_cast<size_t>(tile_row0) + t) * g.out_cols + n * 128 + quad * 32 + (lane & 1) * 16) =
                    *reinterpret_cast<const uint4*>(wst + (lane >> 1) * 32 + (lane & 1) * 16);
            __syncwarp();
        }
        if (quad == 0 && lane < rows_valid && (halves >> (lane >> 4) & 1))
            g.out_scale_t[static_cast<size_t>(n) * row_cap + tile_row0 + lane] = my_sc;
        // Announce the tile.  (The rows are read by copy engines of other CTAs: plain stores here, asynchronous-proxy loads
        // there.)  The announcing thread's fence comes behind the rendezvous and covers the stores of all.
        fence_proxy_async();
        if (!epilogue_rendezvous(c, &ctrl->group_sync[group], sync_iter)) return timed_out();
        if (quad == 0 && lane == 0) {
            __threadfence();
            atomicAdd(f.ready + m_tile, halved ? 1 : 2);
        }
    } else {
        // bf16 out through this warp's 512 bytes of staging, eight tokens x 32 columns at a time, so that
        // the rows leave as 16-byte stores: lane l carries 8 columns of token l / 4 (half of a 32-byte
        // group of the tile-blocked layout)
        __nv_bfloat16* bst = reinterpret_cast<__nv_bfloat16*>(wst);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            if (!(halves >> (h >> 1) & 1) || h * 8 >= rows_valid) continue;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
#pragma unroll
                for (int t = 0; t < 8; ++t) bst[t * 32 + lane] = __float2bfloat16_rn(acc[j * 32 + h * 8 + t]);
                __syncwarp();
                const int t = h * 8 + (lane >> 2), ch0 = quad * 32 + (lane & 3) * 8;
                if (t < rows_valid)
                    *reinterpret_cast<uint4*>(reinterpret_cast<uint8_t*>(g.out_bf16) +
                                              y_block_offset(tile_row0 + t, n * 16 + j * 8 + (ch0 >> 4), g.n_tiles) + (ch0 & 15) * 2) =
                        *reinterpret_cast<const uint4*>(bst + (lane >> 2) * 32 + (lane & 3) * 8);
                __syncwarp();
            }
        }
        // Stage 4 without a kernel of its own.  Once the tile is stored, the thread of each valid row fences and bumps the
        // counter of (its token, this column tile); whoever brings it to the token's number of local slots knows that all of
        // the token's rows for these 256 columns are in memory and sums them, in routing order, exactly as combine_kernel does.
        if (!epilogue_rendezvous(c, &ctrl->group_sync[group], sync_iter)) return timed_out();
        bool last = false;
        if (tok >= 0) {
            __threadfence();
            last = atomicAdd(f.tok_done + static_cast<size_t>(tok) * g.n_tiles + n, 1) == tok_rows - 1;
        }
        uint32_t todo = __ballot_sync(0xffffffffu, last);
        if (!todo) return true;
        __threadfence();
        __syncwarp();  // (a vote orders no memory: the counting lanes' fences come before all lanes' loads)
        // the rows and weights of all tokens at once, each by the lane that counted it: one round trip instead of one per token
        int4 ra = make_int4(-1, -1, -1, -1), rb = ra;
        float4 wa = make_float4(0.f, 0.f, 0.f, 0.f), wb = wa;
        if (last) {
            ra = __ldcg(reinterpret_cast<const int4*>(f.slot_to_row) + 2 * tok);
            rb = __ldcg(reinterpret_cast<const int4*>(f.slot_to_row) + 2 * tok + 1);
            wa = __ldcg(reinterpret_cast<const float4*>(f.topk_w) + 2 * tok);
            wb = __ldcg(reinterpret_cast<const float4*>(f.topk_w) + 2 * tok + 1);
        }
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            const int t = __shfl_sync(0xffffffffu, tok, src);
            // lane l owns columns n*256 + 8 l .. + 8: half of the 32-byte group n*16 + l/2.  All loads
            // first, then the sum in routing order.
            int rr[8] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w};
            float ww[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                rr[j] = __shfl_sync(0xffffffffu, rr[j], src);
                ww[j] = __shfl_sync(0xffffffffu, ww[j], src);
            }
            uint4 u[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (rr[j] >= 0)
                    u[j] = __ldcg(reinterpret_cast<const uint4*>(
                        reinterpret_cast<const uint8_t*>(g.out_bf16) +
                        y_block_offset(rr[j], n * 16 + (lane >> 1), g.n_tiles) + (lane & 1) * 16));
            float o[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) o[i] = 0.0f;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (rr[j] < 0) continue;
                const uint32_t uu[4] = {u[j].x, u[j].y, u[j].z, u[j].w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    o[2 * i] = fmaf(ww[j], __uint_as_float(uu[i] << 16), o[2 * i]);
                    o[2 * i + 1] = fmaf(ww[j], __uint_as_float(uu[i] & 0xffff0000u), o[2 * i + 1]);
                }
            }
            uint32_t p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const __nv_bfloat162 pr = __floats2bfloat162_rn(o[2 * i], o[2 * i + 1]);
                p[i] = *reinterpret_cast<const uint32_t*>(&pr);
            }
            *reinterpret_cast<uint4*>(f.out + static_cast<size_t>(t) * f.H + n * G_TILE_N + lane * 8) =
                make_uint4(p[0], p[1], p[2], p[3]);
        }
    }
    return true;
}

// The tiles of one GEMM.  `few`: no more tiles than CTAs, so that the other group would have nothing to do meanwhile; tiles of more
// than 16 rows are then halved.  `k` numbers the tiles that a group takes alone, from GEMM to GEMM; `behind`: this group has passed one by
// since its own last one.
template <int MODE, class GEO, class SEQ>
__device__ __forceinline__ void epilogue_tiles_group(const Cta& c, const GemmArgs& g, const FusedArgs& f, const SEQ& seq, bool few, uint32_t& k,
                                                     bool& behind, uint32_t& it, uint32_t& amax_iter, uint32_t& sync_iter, bool& ok) {
    const uint32_t group = (c.warp - 4) >> 2;
    for (int j = 0, tile; ok && (tile = seq.at(j)) < seq.count; ++j) {
        const int m_tile = tile / g.n_tiles, n = tile - m_tile * g.n_tiles;
        const bool halved = few && tile_rows_of(c, g, m_tile) > 16;
        const uint32_t before = k;
        if (!halved) ++k;
        if (!halved && (before & 1) != group) {
            it += g.num_kb;
            behind = true;
            continue;
        }
        const int turn = behind ? static_cast<int>(((before - 1) >> 1) & 1) : -1;
        behind = false;
        ok = epilogue_tile_group<MODE, GEO>(c, g, f, m_tile, n, halved, turn, it, amax_iter, sync_iter);
    }
}

// Gather + GEMM1 + GEMM2 + combine in one launch for small batches, at most F_MAX_TOKENS tokens (see the head of
// this file).  tmA2 describes GEMM1's output buffer for loads (32-row boxes), tmB1 / tmB2 the two weight
// tensors.
__global__ void __launch_bounds__(G_THREADS, 1)
fused_small_kernel(const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB1,
                   const __grid_constant__ CUtensorMap tmB2, const GemmArgs g1, const GemmArgs g2, const FusedArgs f) {
    extern __shared__ uint8_t smem_raw[];
    using GEO = GeomSmall;
    Cta c;
    gemm_cta_setup<GEO>(c, smem_raw, 33);  // the producer's arrival plus the 32 lanes of the gather warp
    if (c.warp == 0 && c.lane == 0) {
        tma_prefetch_desc(&tmA2);
        tma_prefetch_desc(&tmB1);
        tma_prefetch_desc(&tmB2);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_launch_dependents();
    pdl_wait();
    c.tmem_base = *reinterpret_cast<volatile uint32_t*>(&c.ctrl->tmem_slot);
    c.limit = g1.wait_limit;

    // The previous fused call has ended (stream order), so the counters it used can be zeroed for the call
    // after this one.
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < f.num_counters; i += blockDim.x) f.counters_next[i] = 0;
    __shared__ CtaTiles s_tiles;
    c.tiles = nullptr;
    if (f.route) {
        // Stages 1 and 2, by every CTA for itself, in the not yet used pipeline stages.
        if (blockIdx.x == 0 && threadIdx.x == 0) *g1.status = DEV_OK;  // first kernel of a forward: clear the fault word
        int* scratch = reinterpret_cast<int*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
        route_permute_in_cta(scratch, s_tiles, f.T, f.E_loc, f.expert_offset, f.row_cap, f.logits, f.bias, f.scaling, f.topk_idx,
                             f.topk_w_out, f.meta, g1.status);
        c.tiles = &s_tiles;
    }

    // tokens without a local expert: their output rows are zeros, written here by the CTAs in turn
    for (int t = blockIdx.x; t < f.T; t += gridDim.x)
        if (f.route ? ((s_tiles.none_local >> t) & 1) != 0 : __ldcg(f.tok_nlocal + t) == 0)
            for (int i = threadIdx.x; i < f.H / 8; i += blockDim.x)
                reinterpret_cast<uint4*>(f.out + static_cast<size_t>(t) * f.H)[i] = make_uint4(0u, 0u, 0u, 0u);

    // The CTA's work list: its GEMM1 tiles, then its GEMM2 tiles.
    // Very small batches with few tiles: a tile's K range is cut into parts for different CTAs (KSplit).
    const int grid = static_cast<int>(gridDim.x), m_tiles = f.route ? s_tiles.count : __ldcg(g1.num_m_tiles);
    const bool may_split = f.split && f.T <= SPLIT_MAX_TOKENS && g1.num_kb <= SPLIT_MAX_KB && g2.num_kb <= SPLIT_MAX_KB;
    const KSplit ks1 = ksplit_for(g1.num_kb, m_tiles * g1.n_tiles, grid, may_split && m_tiles * g1.n_tiles <= SPLIT_MAX_TILES);
    // (GEMM2's K range is too short for it: counting the parts and the finisher's pass over the stored partial sums
    // cost 5-6 us per tile, which 16 K-blocks do not win back; measured 1-2 us slower)
    const KSplit ks2 = ksplit_none(g2.num_kb);
    const int n1 = m_tiles * g1.n_tiles * ks1.parts, n2 = m_tiles * g2.n_tiles;
    const PlainSeq tr1 = seq_plain(n1);
    uint32_t it = 0;
    bool ok = true;

    if (m_tiles == 0) {
        // no token has a local expert: the roles would only tell one another so (6.8 against 5.7 us per forward)
    } else if (c.warp < 4) {
        reg_dealloc<56>();
        if (c.warp == 0 && c.lane == 0) {
            Tickets tickets{f.ticket, 0, false};
            producer_tiles<1, GEO>(c, &tmA2, &tmB1, g1, &f, 0, tr1, tickets, it, ok, ks1);
            if (ok) producer_tiles<2, GEO>(c, &tmA2, &tmB2, g2, &f, 2 * g1.n_tiles, seq_plain(n2), tickets, it, ok, ks2);
        } else if ((c.warp == 1 || c.warp == 2) && c.lane == 0) {
            issuer_tiles_wm<GEO>(c, g1, tr1, c.warp - 1, it, ok, ks1);
            issuer_tiles_wm<GEO>(c, g2, TicketSeq<false>{c, g1.status, n2}, c.warp - 1, it, ok, ks2);
        } else if (c.warp == 3) {
            gather_tiles<GEO>(c, g1, f, tr1, it, ok, ks1);
            gather_idle_tiles<GEO>(c, g2, TicketSeq<true>{c, g1.status, n2}, it, ok, ks2);
            cp_async_wait_all();  // nothing may still be landing in shared memory when the CTA exits
            if (c.lane == 0) c.ctrl->gathered = it;
        }
    } else {
        reg_alloc<224>();
        uint32_t k = 0, amax_iter = 0, sync_iter = 0;
        bool behind = false;
        if (ks1.parts > 1) {  // (one part of a tile at most; all eight warps)
            uint32_t joint_iter = 0;
            AmaxTurn turn{0};
            if (tr1.at(0) < n1) {
                const int tile = tr1.at(0) / ks1.parts, kb0 = (tr1.at(0) - tile * ks1.parts) * ks1.len;
                ok = epilogue_tile_wm<1, true, GEO>(c, g1, &f, tile / g1.n_tiles, tile % g1.n_tiles, it, turn, joint_iter, kb0,
                                                    min(g1.num_kb, kb0 + ks1.len), ks1.parts);
            }
        } else {
            epilogue_tiles_group<1, GEO>(c, g1, f, tr1, n1 <= grid, k, behind, it, amax_iter, sync_iter, ok);
        }
        epilogue_tiles_group<2, GEO>(c, g2, f, TicketSeq<true>{c, g1.status, n2}, n2 <= grid, k, behind, it, amax_iter, sync_iter, ok);
    }

    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (*c.abort_flag) drain_after_abort<GEO>(c, g1.status, it, c.ctrl->gathered);
    if (c.warp == 1) {
        __syncwarp();
        tmem_dealloc(c.tmem_base, G_TMEM_COLS);
    }
}

}  // namespace moe
