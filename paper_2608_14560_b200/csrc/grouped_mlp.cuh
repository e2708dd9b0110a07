// The expert MLP (stage 3 of the Fused MoE description) of batches beyond the fused kernel's range: GEMM1 with SwiGLU and
// re-quantisation and GEMM2, in one launch.  Roles and their loop: see gemm.cuh.
//
// Every CTA has a list of tiles, GEMM1's first: CTA b takes GEMM1 tiles b, b + grid, ... and then GEMM2 tiles from a counter
// until there are none (the first one is dealt where tiles are few, see mlp_first_tile_dealt).  A GEMM2 tile starts once GEMM1's column tiles of its row tile have been announced (bounded wait).  So that no CTA ever depends on one that has not started -- two such kernels may share the
// GPU from different streams --, a CTA claims its list of GEMM1 tiles when it starts, and before its first GEMM2 tile it
// works through the lists nobody has claimed: every GEMM1 tile it may then wait for is in the hands of a running CTA.
// Fixed lists for GEMM1, not a counter that hands out tiles: neighbouring tiles share operands, and CTAs that read the same lines
// at the same time get them out of L2 faster (loads-only kernel: 26 against 17 TB/s).  Tiles handed out in order of
// arrival took GEMM1 of 8192 skewed tokens from 1226 to 1331 us.  For GEMM2 the counter is the better way, or an equal one: row
// tiles differ in time and CTAs in their share of the memory's rate, and dealt in rounds, with up to three rounds in front
// for the CTAs with one GEMM1 tile less, the last CTA ended 12 us (6 %) behind the middle one at 257 tokens, now 5.  us per forward
// dealt / counter: 194.0 / 193.4 at 100 tokens, 139.9 / 137.0 at 150 skewed, 205.7 / 202.2 at 257, 204.7 / 202.0 at 400, 223.1 /
// 221.5 at 901, 251.5 / 248.8 at 1500, 436.5 / 433.4 at 4096, 1589 / 1591 at 8192 skewed; on 256 experts 1184 / 1178 at 300, 1405 /
// 1394 at 1000, 4006 / 4001 at 8192 (runs too short for the power cap, under which 8192 skewed tokens take 2100).
// What the common list is for: a launch per GEMM leaves most SMs idle in its last, partly filled wave.  With 24 active
// experts (257 tokens) GEMM1 is 384 tiles of 56 K-blocks, 2.6 waves, and GEMM2 672 tiles of 16, 4.5 waves: 248 K-block
// times per launch pair against 218 in one list.  Measured per forward, two launches against one, this kernel on both
// sides (the first 32 experts, uniform routing, runs too short for the power cap): 187 -> 170 us at 257 tokens, 208 -> 193
// at 512, 212 -> 197 at 901, 261 -> 238 at 2048, 351 -> 338 at 4096.  In long runs two launches are better where a list is
// long (see MLP_JOINT_MAX_SLOTS) and the CTAs, in step after a launch, drift apart.
#pragma once
#include "gemm.cuh"

namespace moe {

// Batches of more than MLP_SPLIT_MAX_TOKENS tokens and at most MLP_JOINT_MAX_SLOTS expected local slots (tokens x 8 x
// the local share of the experts) run both GEMMs in one launch, the others in one each.  us per forward, one launch
// against two: 248 / 256 at 1109 slots, 417 / 429 at 4171, 1435 / 1439 at 4096 with 256 experts, 1055 / 1065 at 16872
// skewed, 1116 / 1125 at 16167, 2194 / 2201 at 16384 with 256 experts, 3170 / 3159 at 32768, 8913 / 8626 at 131072.
// The last figure sets the line: under the power cap, which short runs do not reach (there one launch stays ahead: 2908 / 2987
// at 32768 slots, 5066 / 5169 at 65536), the largest batches lose 3 %.
// Two launches overlap up to MLP_SPLIT_MAX_TOKENS tokens: a CTA of the second one starts on an SM that has finished its GEMM1 tiles, all
// CTAs of the first one run by then (they allow the second launch when they start), and its tiles wait for the announcements
// of their rows like those of the one launch.  us per forward, one launch after the
// other / overlapping: 191.4 / 179.3 at 81 tokens, 195.9 / 184.5 at 128, 196.5 / 182.6 at 160, 208.5 / 205.1 at 200, 208.9 / 205.1 at
// 256; skewed 138.0 / 128.4 at 81, 175.6 / 159.2 at 200; on 256 experts 1187 / 1172 at 256.
// The lower line is not set by speed: callers count on two GEMM launches up to 256 tokens (last_launch_count, the stage
// times of the two GEMMs).
constexpr int MLP_SPLIT_MAX_TOKENS = 256;
constexpr int MLP_JOINT_MAX_SLOTS = 16384;

// GEMM2 tiles that are dealt, one to every CTA (all or none); the later ones come from the counter.  With the counter alone a CTA
// that waits for its first rows has already drawn a second tile, and where there are not many of them others have none.  Dealt
// in one launch where there is no tile of GEMM1 or of GEMM2 for every CTA; in a launch of its own where there is no GEMM2 tile for
// every CTA and a tile is longer than the ring of stages: short ones are better off on the CTAs that start first.  us per forward
// from the counter / with one dealt: 7168 x 2048, 8 experts, 300 tokens 66.6 / 60.9, 3 experts, 600 tokens 72.8 / 66.9; 2048 x 2048,
// 16 experts, 200 skewed 54.9 / 50.4; 512 x 2048, 64 experts, 100 tokens 53.2 / 49.5; 2048 x 1024, 16 experts, 400 tokens 38.4 / 35.0;
// 768 x 768, 32 experts, 256 skewed 31.8 / 29.3.  Beyond the lines: 1024 x 1024, 64 experts, 114 tokens 48.8 / 50.6; 512 x 512, 100
// experts, 92 tokens 30.9 / 32.3; 7168 x 2048, 32 experts, 901 tokens 194.3 / 195.1.
__device__ __forceinline__ bool mlp_first_tile_dealt(bool joint, int m_tiles, const GemmArgs& g1, const GemmArgs& g2, int grid) {
    const bool few1 = m_tiles * g1.n_tiles <= grid, few2 = m_tiles * g2.n_tiles <= grid;
    return joint ? few1 || few2 : few2 && g2.num_kb > GeomFull::STAGES;
}

constexpr int MLP_MAX_GRID = 1023;   // lists that `claimed` has room for
struct MlpArgs {
    GemmArgs g1, g2;
    int phases;          // bit 0: GEMM1's tiles, bit 1: GEMM2's
    int by_row;          // a GEMM2 tile waits for the announcements of its rows: both GEMMs in one launch, or in two that overlap
    int* claimed;        // [grid] the lists of GEMM1 tiles, LIST_OPEN (or LIST_LEFT) at launch (both GEMMs only), and
                         // the next GEMM2 tile behind the dealt ones, zero at launch
};

__device__ __forceinline__ TileInfo read_tile(const Cta& c, uint32_t i) {  // an entry that has been waited for
    const int4 v = ld_shared_v4(smem_u32(&c.ctrl->sched[i % SCHED_SLOTS]));
    return TileInfo{v.x, v.y, v.z, v.w};
}
// Entry i of the CTA's work list, as the factor warp published it.  A role that gave up here while the others went on
// would leave them at a named barrier, whose wait has no limit (see mlp_issuer), so this wait has to outlast every chain of
// waits in front of an entry or the list's end, and its limit is not the one that a test may shorten: with that, a role that
// looked for its first entry before it was published could take the list for empty.
constexpr long long SCHED_LIMIT_CLOCKS = 16 * WAIT_LIMIT_CLOCKS;
__device__ __forceinline__ TileInfo next_tile(const Cta& c, uint32_t i) {
    int zero = 0;
    const uint32_t slot = i % SCHED_SLOTS;
    if (!mbar_wait(smem_u32(&c.ctrl->sched_full[slot]), (i / SCHED_SLOTS) & 1, &zero, SCHED_LIMIT_CLOCKS)) return TileInfo{};
    return read_tile(c, i);
}
// The same by a whole warp: all lanes see the entry or none does.
__device__ __forceinline__ TileInfo next_tile_warp(const Cta& c, uint32_t i) {
    TileInfo t = next_tile(c, i);
    if (!__all_sync(0xffffffffu, t.mode() != 0)) t.key = 0;
    return t;
}

// ---------------- TMA producer (one thread) ----------------
// One copy for the token rows and two for the 256 weight rows of a K-block: a copy instruction costs this thread
// about 85 clocks, which is part of the time a stage needs to be refilled (500 clocks with the weight rows as four
// copies and the scales as another one); boxes of 256 rows move at 52 bytes per clock and SM out of L2, boxes of 128
// rows at 67 (measured with a loads-only kernel).
// Weight rows of a stage, N side of the MMAs: GEMM1 gate[0,64) | up[0,64) | gate[64,128) | up[64,128) of the tile's 128
// columns (tmB1n), GEMM2 256 consecutive rows (tmB2); M side (short row tiles): GEMM1 gate[0,128) | up[0,128) (tmB1m).
// All three maps see the weights as [expert][half][row][K]; a stage takes two boxes of 128 rows.
// Refilling a freed stage is part of the loop that bounds a large batch, so this thread waits for nothing in global
// memory: with the ticket and the table entries of the next tile fetched here, a GEMM1 tile took 1 us longer.
// Returns the number of stages it has claimed.
template <class GEO>
__device__ __forceinline__ uint32_t mlp_producer(const Cta& c, const CUtensorMap* tmA1, const CUtensorMap* tmA1s,
                                             const CUtensorMap* tmB1n, const CUtensorMap* tmB1m, const CUtensorMap* tmA2,
                                             const CUtensorMap* tmA2s, const CUtensorMap* tmB2, const MlpArgs& a) {
    GemmCtrl* ctrl = c.ctrl;
    uint32_t it = 0;
    bool ok = true, waited = a.phases == 2 && a.by_row;  // waited: the kernels before this one have finished (or need not have)
    for (uint32_t i = 0; ok; ++i) {
        const TileInfo cur = next_tile(c, i);
        if (cur.mode() == 0) break;
        const bool m1 = cur.mode() == 1;
        const int num_kb = m1 ? a.g1.num_kb : a.g2.num_kb;
        const bool wm = cur.rows <= a.g1.wm_rows;  // a short row tile: 32 token rows fetched, weights for the M side
        const CUtensorMap* tA = m1 ? (wm ? tmA1s : tmA1) : (wm ? tmA2s : tmA2);
        const CUtensorMap* tB = m1 ? (wm ? tmB1m : tmB1n) : tmB2;
        // the two boxes of weight rows: (row, half)
        const int y0 = cur.n * (m1 ? 128 : G_TILE_N), y1 = y0 + (m1 ? (wm ? 0 : 64) : 128), z1 = (m1 && wm) ? 1 : 0;
        const int e = cur.expert, row0 = cur.m_tile() * TILE_M;
        const uint32_t tx = wm ? WM_TOKENS * G_BLOCK_K + G_B_BYTES : GEO::STAGE_BYTES;
        const int skip_it = m1 ? a.g1.fault_skip_it : -1;
        // claim the stage of pipeline iteration j: wait until its last reader has finished, announce the bytes
        auto claim = [&](uint32_t j) -> bool {
            const uint32_t s = j % GEO::STAGES, ph = (j / GEO::STAGES) & 1;
            if (static_cast<int>(j) == skip_it) return false;  // test hook: never filled
            if (!mbar_wait(smem_u32(&ctrl->done[s]), ph ^ 1, c.abort_flag, c.limit)) {
                raise(ctrl, a.g1.status, DEV_TIMEOUT_PRODUCER);
                return false;
            }
            mbar_expect_tx(smem_u32(&ctrl->full[s]), tx);
            return true;
        };
        auto load_b = [&](uint32_t j, int kb) {
            const uint32_t s = j % GEO::STAGES, bar = smem_u32(&ctrl->full[s]);
            const uint32_t dst = c.smem_base + s * GEO::STAGE_BYTES + GEO::A_BYTES;
            tma_load_4d(dst, tB, kb * G_BLOCK_K, y0, 0, e, bar);
            tma_load_4d(dst + G_B_BYTES / 2, tB, kb * G_BLOCK_K, y1, z1, e, bar);
        };
        auto load_a = [&](uint32_t j, int kb) {
            const uint32_t s = j % GEO::STAGES;
            tma_load_2d(c.smem_base + s * GEO::STAGE_BYTES, tA, kb * G_BLOCK_K, row0, smem_u32(&ctrl->full[s]));
        };
        const uint32_t rows_bar = smem_u32(&ctrl->sched_rows[i % SCHED_SLOTS]), rows_ph = (i / SCHED_SLOTS) & 1;
        const bool must_wait = !m1 && a.by_row;
        bool rows_there = !must_wait || mbar_test(rows_bar, rows_ph);
        int kb = 0;
        if (!waited || !rows_there) {
            // The token rows may not be there yet, the weights are: those of the first stages go out at once.
            const int npre = num_kb < GEO::STAGES ? num_kb : GEO::STAGES;
            while (kb < npre && (ok = claim(it + kb))) {
                load_b(it + kb, kb);
                ++kb;
            }
            if (!waited) {
                pdl_wait();
                waited = true;
            }
            if (ok && !rows_there) {  // (8: longer than the factor warp's wait for the same rows)
                ok = mbar_wait(rows_bar, rows_ph, c.abort_flag, 8 * c.limit);
                if (!ok) raise(ctrl, a.g1.status, DEV_TIMEOUT_READY);
            }
            fence_proxy_async();
            // (after a time-out as well, when nobody reads them: a claimed stage is complete with its token rows only, and
            // drain_after_abort waits for the claimed stages)
            for (int k = 0; k < kb; ++k) load_a(it + k, k);
            it += kb;
        } else if (must_wait) {
            fence_proxy_async();  // stored by other CTAs' copy engines; order our copies behind the barrier
        }
        for (; kb < num_kb && ok; ++kb, ++it) {
            ok = claim(it);
            if (!ok) break;
            load_b(it, kb);  // (first: it may have to come from HBM, the token rows are in L2)
            load_a(it, kb);
        }
    }
    if (!waited) pdl_wait();
    return it;
}

// ---------------- MMA issuers (two warps) ----------------
// Two warps share the issue work: `mine` = 0 takes the even K-blocks (TMEM buffer 0), 1 the odd ones (buffer 1).  A
// commit only tracks the MMAs of its own thread, so while one thread pays for its commit and waits the other keeps
// the tensor pipe fed.
// An accumulator buffer comes back through a named barrier that the eight epilogue warps arrive at and the issuer
// warp waits on, once per K-block (see ACC_BARRIER): the hand-over is part of the loop that bounds the kernel, and
// through an mbarrier it cost 0.4-0.9 % of a large batch.  Such a wait has no limit of its own, so no role may ever
// miss its turn: after an abort the issuers and the epilogue warps go on to the end of the published list with the
// barriers alone (the waits on mbarriers stay bounded, and the factor warp always publishes an end).
template <class GEO>
__device__ __forceinline__ void mlp_issuer(const Cta& c, const MlpArgs& a, uint32_t mine) {
    GemmCtrl* ctrl = c.ctrl;
    const uint32_t idesc = umma_idesc_f8(TILE_M, G_TILE_N), idesc_wm = umma_idesc_f8(TILE_M, WM_TOKENS);
    // Lanes that wait for the stages: the one that issues the MMAs in any case (a shuffle from another one orders no memory).  All of
    // them, without a branch around the wait, are 1 to 1.5 % faster up to MLP_JOINT_MAX_SLOTS (us per forward one lane / all: 185.0 / 182.2
    // at 257 tokens, 223.8 / 221.5 at 901, 415.9 / 411.6 at 4096, equal at 8192 skewed); beyond, at the power cap, 32 polling lanes cost
    // more than they save (7440 / 7545 at 16384 tokens on 256 experts).
    const bool waits = a.by_row || elect_one();
    uint32_t it = 0;
    bool ok = true;
    for (uint32_t i = 0;; ++i) {
        const TileInfo t = next_tile_warp(c, i);
        if (t.mode() == 0) break;
        // a short row tile: the stage's weight rows are the M side (two blocks of 128), its 32 token rows the N
        // side; the accumulator is the first 64 columns of the buffer
        const bool wm = t.rows <= a.g1.wm_rows;
        const int num_kb = t.mode() == 1 ? a.g1.num_kb : a.g2.num_kb;
        for (int kb = 0; kb < num_kb; ++kb, ++it) {
            if ((it & 1) != mine) continue;
            const uint32_t s = it % GEO::STAGES, ph = (it / GEO::STAGES) & 1;
            // The stage has normally landed long before the accumulator is handed back, so that
            // wait comes first and only the hand-over itself is left on the critical path.
            const uint32_t a_addr = c.smem_base + s * GEO::STAGE_BYTES;
            const uint64_t a_desc = umma_desc_sw128(a_addr);  // 128 rows from here, fetched or not
            const uint64_t b_desc = umma_desc_sw128(a_addr + GEO::A_BYTES);
            const uint32_t d_tmem = c.tmem_base + mine * G_TILE_N;
            if (ok) {
                if (waits) ok = mbar_wait(smem_u32(&ctrl->full[s]), ph, c.abort_flag, c.limit);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok && c.lane == 0) raise(ctrl, a.g1.status, DEV_TIMEOUT_MMA_SMEM);
            }
            if (it >= G_ACC_BUFS) bar_sync(ACC_BARRIER + mine, ACC_BARRIER_THREADS);
            if (!ok) continue;
            tc_fence_after();
            // (by a lane chosen by its number, eight MMAs of a short tile took 850 clocks to issue, now 690)
            if (elect_one()) {
                if (wm) {
                    const uint64_t w1_desc = umma_desc_sw128(a_addr + GEO::A_BYTES + G_B_BYTES / 2);
#pragma unroll
                    for (int k = 0; k < G_BLOCK_K / 32; ++k) umma_f8(d_tmem, b_desc + 2 * k, a_desc + 2 * k, idesc_wm, k > 0);
#pragma unroll
                    for (int k = 0; k < G_BLOCK_K / 32; ++k)
                        umma_f8(d_tmem + WM_TOKENS, w1_desc + 2 * k, a_desc + 2 * k, idesc_wm, k > 0);
                } else {
#pragma unroll
                    for (int k = 0; k < G_BLOCK_K / 32; ++k)  // 32 K-bytes per instruction: +2 in 16-B units
                        umma_f8(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, k > 0);
                }
                umma_commit(smem_u32(&ctrl->done[s]));
            }
            __syncwarp();
        }
    }
    if (it > mine) bar_sync(ACC_BARRIER + mine, ACC_BARRIER_THREADS);  // the buffer's last hand-over
}

// ---------------- factor warp, which is also the tile scheduler ----------------
// Factors: multiplies the activation scales of every K-block with the two weight scales of the tile's 256 columns, so
// that an epilogue thread finds its factor with one shared-memory load: [slot][2][row].  With the weight scales fetched
// from global memory by the epilogue threads themselves, and the products formed there, an epilogue warp spent
// about 500 of its 1240 clocks per K-block between handing a buffer back and being ready for the next one.  The
// warp's arrival is the second one on done[s]: whoever sees that barrier finds the factors complete.  Like the
// producer it claims a stage by waiting for the previous phase of done[s]; the slot it then writes was read by the
// epilogue eight K-blocks ago (done of four K-blocks ago implies that the accumulator of six ago was handed back).
// The scales come in F_AHEAD K-blocks ahead, across the ends of tiles: with loads that started anew at every tile the
// warp's first arrival was late by the latency of three dependent loads, 3 % of a batch of 257 tokens.  It does not
// look from a GEMM1 tile into a GEMM2 tile, whose scales may not be there before this CTA's GEMM1 tiles are done.
// Scheduling: when the fetch of scales enters a tile, the next one is published; its table entries go straight from the
// tables into the ring, the publishing arrival triggered by their copies.  Nothing in that waits for another role, so
// the producer, which may need a tile as soon as this warp's writes (F_AHEAD = STAGES K-blocks behind its fetches) have
// passed the tile before it, is always served.  The rows of a GEMM2 tile are awaited here too, F_AHEAD K-blocks before
// they are needed.
template <class GEO>
__device__ __forceinline__ void mlp_factors(const Cta& c, const MlpArgs& a) {
    static_assert(GEO::FACTORS && GEO::A_ROWS == 128, "a lane looks after four rows");
    static_assert(GEO::SCALE_SLOTS >= GEO::STAGES + G_ACC_BUFS + 1, "slots still read by the epilogue");
    static_assert(F_AHEAD < F_SLOTS && F_AHEAD <= GEO::STAGES, "a slot is refilled after it was read; see above");
    GemmCtrl* ctrl = c.ctrl;
    const int lane = c.lane;
    const int ready_target = a.g1.n_tiles * G_EPI_WARPS;
    const int m_tiles = __ldcg(a.g1.num_m_tiles);
    const int n1 = (a.phases & 1) ? m_tiles * a.g1.n_tiles : 0, n12 = n1 + ((a.phases & 2) ? m_tiles * a.g2.n_tiles : 0);
    const int grid = static_cast<int>(gridDim.x);
    // GEMM1: tiles id1, id1 + grid, ... ; GEMM2: the dealt one, if any, then whichever is next when this CTA needs one (a ticket,
    // drawn when it enters the tile before).
    int id1 = static_cast<int>(blockIdx.x);
    int drawn = -1, dealt = 0;  // GEMM2: the dealt tile (a ticket that has been drawn already); the number of dealt tiles
    if (mlp_first_tile_dealt(a.phases == 3, m_tiles, a.g1, a.g2, grid)) {
        const int late = n1 % grid;  // CTAs with one GEMM1 tile more: they come last
        drawn = id1 < late ? id1 + grid - late : id1 - late;
        dealt = grid;
    }
    if (a.phases == 3) {
        int was = LIST_OPEN;
        if (lane == 0) was = atomicCAS(a.claimed + blockIdx.x, LIST_OPEN, LIST_CLAIMED);
        if (__shfl_sync(0xffffffffu, was, 0) != LIST_OPEN) id1 = n1;  // (somebody else works on it, or will)
    }
    uint32_t published = 0;
    int last_key = 1;
    auto publish = [&](bool end) {  // the next tile of the list, or its end
        if (a.phases == 3 && id1 >= n1 && !end && (last_key & 3) == 1) {
            // the end of a list of GEMM1 tiles: go on with one that nobody has claimed, if there is any
            for (int v0 = 0; v0 < grid && id1 >= n1; v0 += 32) {
                const int v = v0 + lane;
                const bool other = v < grid && v < n1 && v != static_cast<int>(blockIdx.x);
                uint32_t open = __ballot_sync(0xffffffffu, other && __ldcg(a.claimed + v) != LIST_CLAIMED);
                while (open && id1 >= n1) {
                    const int u = v0 + __ffs(open) - 1;
                    open &= open - 1;
                    int was = LIST_CLAIMED;
                    if (lane == 0) was = atomicExch(a.claimed + u, LIST_CLAIMED);
                    if (__shfl_sync(0xffffffffu, was, 0) != LIST_CLAIMED) id1 = u;
                }
            }
        }
        int id = n12;
        if (id1 < n1) {
            id = id1;
            id1 += grid;
        } else if ((a.phases & 2) && !end) {
            int ticket = drawn;
            if (lane == 0 && drawn < 0) ticket = dealt + atomicAdd(a.claimed + grid, 1);
            drawn = -1;
            id = n1 + __shfl_sync(0xffffffffu, ticket, 0);
        }
        const bool live = !end && id < n12;
        const bool first = id < n1;
        const int k = first ? id : id - n1, nt = first ? a.g1.n_tiles : a.g2.n_tiles, m = k / nt;
        last_key = !live ? 0 : !first ? m * 16 + 2
                   : m * 16 + 1 + (id + grid >= n1 ? TileInfo::LAST : 0) + (id + 2 * grid >= n1 ? TileInfo::LAST_TWO : 0);
        if (lane == 0) {
            const uint32_t slot = published % SCHED_SLOTS, bar = smem_u32(&ctrl->sched_full[slot]);
            TileInfo* p = &ctrl->sched[slot];
            if (live) {
                *reinterpret_cast<volatile int*>(&p->n) = k - m * nt;
                cp_async_4(smem_u32(&p->rows), a.g1.tile_rows + m, 4);
                cp_async_4(smem_u32(&p->expert), a.g1.tile_expert + m, 4);
            }
            *reinterpret_cast<volatile int*>(&p->key) = last_key;
            cp_async_arrive_noinc(bar);  // once the copies have landed
            mbar_arrive(bar);            // (orders the plain stores)
        }
        ++published;
    };
    publish(false);
    if (a.phases != 2 || !a.by_row) pdl_wait();
    // The fetch cursor: K-blocks fetched, tile, K-block in it, K-blocks left of the run.  Past the last tile of a GEMM it
    // goes on fetching the last K-block's scales, which nobody reads, so that the regular step has no branch for it.
    uint32_t fit = 0, fi = 0, frun = 0;
    int fkb = 0, fleft = 0, fnum = 0;
    const float* as = nullptr;
    const float* ws = nullptr;
    ptrdiff_t as_step = 0;
    const uint32_t raw = smem_u32(c.raw_scales) + lane * 16, raw_w = smem_u32(c.raw_scales + F_SLOTS * TILE_M);
    auto enter = [&](int mode) -> bool {  // the next run, perhaps of the next tile
        if (fkb == fnum) {
            const TileInfo t = next_tile_warp(c, fi);
            if (t.mode() != mode) {
                as -= as_step;
                as_step = 0;
                fleft = 1 << 30;
                return true;
            }
            const bool m1 = mode == 1;
            const int n_tile = t.n, blocks = m1 ? 2 * a.g1.out_cols / 128 : a.g2.out_cols / 128;
            fnum = m1 ? a.g1.num_kb : a.g2.num_kb;
            fkb = 0;
            as = (m1 ? a.g1.a_scale_t : a.g2.a_scale_t) + static_cast<size_t>(t.m_tile()) * TILE_M + lane * 4;
            as_step = a.g1.row_cap;
            ws = (m1 ? a.g1.w_scale : a.g2.w_scale) +
                 (static_cast<size_t>(t.expert) * blocks + (m1 ? n_tile : 2 * n_tile)) * fnum;
            publish(false);
            bool there = true;
            if (lane == 0) {
                // (Four limits, so that this warp is not the first to give up when another CTA's roles wait in vain: the
                // status word then says which wait it was.  The bound on the whole is one limit all the same: meanwhile
                // this warp holds back its arrivals on done[], and the other roles of the CTA, once they wait for those,
                // give up after one, which ends this wait as well.  Rows that never come are thus reported as the time-out
                // of whichever role that is.)
                if (!m1 && a.by_row)
                    there = wait_counter(a.g1.ready + t.m_tile(), ready_target, c.abort_flag, 4 * c.limit);
                if (there) mbar_arrive(smem_u32(&ctrl->sched_rows[fi % SCHED_SLOTS]));
            }
            there = __shfl_sync(0xffffffffu, there, 0);
            __syncwarp();  // a shuffle orders no memory: lane 0 has seen the rows announced, all lanes fetch their scales
            if (!there) {
                if (lane == 0) raise(ctrl, a.g1.status, DEV_TIMEOUT_READY);
                return false;
            }
            ++fi;
        }
        fleft = min(F_RUN, fnum - fkb);
        if (lane < fleft) {  // weight scales of K-block fkb + lane: the tile's first and second 128 weight rows
            const float* w0 = ws + fkb + lane;
            const size_t second = static_cast<size_t>(mode == 1 ? a.g1.out_cols / 128 : 1) * fnum;
            const uint32_t dst = raw_w + ((frun % F_SLOTS) * F_RUN + lane) * 8;
            cp_async_4(dst, w0, 4);
            cp_async_4(dst + 4, w0 + second, 4);
        }
        ++frun;
        fkb += fleft;
        return true;
    };
    auto fetch = [&](int mode) -> bool {
        if (fleft == 0 && !enter(mode)) return false;
        --fleft;
        cp_async_16(raw + (fit % F_SLOTS) * (TILE_M * 4), as, 16);
        as += as_step;
        ++fit;
        cp_async_commit();
        return true;
    };
    uint32_t it = 0, i = 0, run = 0;  // K-blocks, tiles and runs written
    bool ok = true;
    while (ok) {
        TileInfo t = next_tile_warp(c, i);
        if (t.mode() == 0) break;
        const int mode = t.mode();  // the tiles of one GEMM
        const int num_kb = mode == 1 ? a.g1.num_kb : a.g2.num_kb;
        cp_async_wait_all();  // (the fetches past the end of the GEMM before)
        __syncwarp();
        fit = it;
        fkb = fnum = fleft = 0;
        for (int k = 0; k < F_AHEAD && ok; ++k) ok = fetch(mode);
        while (ok && t.mode() == mode) {
            for (int kb = 0; kb < num_kb; ++kb, ++it) {
                const uint32_t s = it % GEO::STAGES;
                cp_async_wait<F_AHEAD - 1>();
                __syncwarp();
                if (kb % F_RUN == 0) ++run;
                const int4 xi = ld_shared_v4(raw + (it % F_SLOTS) * (TILE_M * 4));
                const uint32_t w_addr = raw_w + (((run - 1) % F_SLOTS) * F_RUN + kb % F_RUN) * 8;
                const float w0 = ld_shared_f32(w_addr), w1 = ld_shared_f32(w_addr + 4);
                const float4 x = make_float4(__int_as_float(xi.x), __int_as_float(xi.y), __int_as_float(xi.z), __int_as_float(xi.w));
                ok = fetch(mode);
                if (!ok) break;
                if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&ctrl->done[s]), ((it / GEO::STAGES) & 1) ^ 1, c.abort_flag, c.limit))) {
                    if (lane == 0) raise(ctrl, a.g1.status, DEV_TIMEOUT_PRODUCER);
                    ok = false;
                    break;
                }
                float* dst = c.scale_ring + (it % GEO::SCALE_SLOTS) * 2 * GEO::A_ROWS + lane * 4;
                *reinterpret_cast<float4*>(dst) = make_float4(x.x * w0, x.y * w0, x.z * w0, x.w * w0);
                *reinterpret_cast<float4*>(dst + GEO::A_ROWS) = make_float4(x.x * w1, x.y * w1, x.z * w1, x.w * w1);
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctrl->done[s]));
            }
            if (ok) t = next_tile_warp(c, ++i);
        }
    }
    // after an abort the list ends here for every role
    if (!ok && last_key != 0) publish(true);
    cp_async_wait_all();  // nothing may still be landing in shared memory when the CTA exits
}

// acc[0..64) += v * f with packed fp32 FMAs: one instruction, two independent round-to-nearest FMAs, the bits of the
// scalar form.  Beside scalar FMAs the MMA issuers, which share the schedulers with the epilogue warps, needed 955
// clocks per K-block in a probe of this loop, beside packed ones 672 (602 beside an epilogue without FMAs).
template <bool FIRST>
__device__ __forceinline__ void fma64(float* acc, const float (&v)[64], float f) {
    const uint64_t p = pack_f32x2(__float_as_uint(f), __float_as_uint(f));
#pragma unroll
    for (int j = 0; j < 64; j += 2) {
        const uint64_t a = fma_f32x2(pack_f32x2(__float_as_uint(v[j]), __float_as_uint(v[j + 1])), p,
                                     FIRST ? 0ull : pack_f32x2(__float_as_uint(acc[j]), __float_as_uint(acc[j + 1])));
        acc[j] = __uint_as_float(static_cast<uint32_t>(a));
        acc[j + 1] = __uint_as_float(static_cast<uint32_t>(a >> 32));
    }
}

// ---------------- epilogue warps ----------------
// bf16 rows out in a tile-blocked layout: block (row tile, column tile, half, quadrant) holds a warp's 32 rows x 128
// columns as [8 column groups][32 rows][16 bf16], so every warp store instruction writes 1 KB of contiguous memory (32
// bytes per lane).  `p` is where the first of four groups goes.
__device__ __forceinline__ void store_rows64(uint8_t* p, const float* acc) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const __nv_bfloat162 pr = __floats2bfloat162_rn(acc[q * 16 + 2 * i], acc[q * 16 + 2 * i + 1]);
            w[i] = *reinterpret_cast<const uint32_t*>(&pr);
        }
        st_global_v8(p + q * 1024, w);
    }
}

// GEMM1: gate/up projection + SwiGLU + re-quantisation; tmOut describes the e4m3 output [row_cap, I] for 64-byte x
// 32-row TMA stores.  GEMM2: down projection, bf16 rows out in the tile-blocked layout.  One full row tile, entry i of the
// list; false: a wait gave up (the code is in the status word) and `it` stands at the K-block whose buffer was not handed
// back.  Otherwise `t` is the next entry.
// The MMAs run two K-blocks ahead and then wait for this function to come round, so what lies between the last K-block of
// a tile and the first of the next is lost beyond about 1700 clocks (it was 5600 of GEMM1's 51 000 and 1800 of GEMM2's
// 14 600).  Hence no clearing of the sums, an exchange of maxima between the two warps concerned and not among all eight,
// the next entry read beside it (GEMM2: not behind all of the stores, which hold up every later access to shared memory),
// and the halves of the weights taken in the order gate, up instead of changing places behind the loop.
// The loop has 192 of its 224 registers in its two arrays: what it does not need, the tile's entry for one, is fetched again
// behind it.  Spilling decides here: forms with 110 to 380 bytes of spilled registers were 2 to 8 % slower, tiles of the other
// orientation included; this one stores 12 bytes and loads 28.
// us of the GEMM launches before / this form: 8192 skewed tokens on 32 experts 1536 / 1432, 4096 tokens 399 / 387, 8192 tokens
// on 256 experts 3926 / 3674.  What is left of the tails is 1 % (the SwiGLU left out altogether: 1416, 382).
template <int MODE, class GEO>
__device__ __forceinline__ bool mlp_epilogue_tile(const Cta& c, const CUtensorMap* tmOut, const GemmArgs& g, uint32_t i,
                                                  TileInfo& t, uint32_t& it, AmaxTurn& turn, Announce& announce) {
    static_assert(GEO::A_ROWS == TILE_M && GEO::STORE_BYTES == G_EPI_WARPS * G_STORE_WARP_BYTES, "full row tiles");
    GemmCtrl* ctrl = c.ctrl;
    const int warp = c.warp, lane = c.lane;
    const int widx = warp - 4;
    const int half = widx >> 2;              // which 128-column half of the tile
    const int quad = warp & 3;               // TMEM lane quadrant this warp may read
    const int r_in_tile = quad * 32 + lane;  // accumulator row == TMEM lane
    // GEMM1: of this warpgroup's 128 columns, one half of 64 are gate columns (they go to acc[0..64)) and the other the
    // matching up columns, each with its own factor; GEMM2: one factor
    const uint32_t swap = MODE == 1 && g.up_first ? 1 : 0;
    const uint32_t t_lane = c.tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + half * G_HALF_N + swap * 64;
    const uint32_t factors = smem_u32(c.scale_ring + r_in_tile + (MODE == 1 ? swap : half) * GEO::A_ROWS);
    const uint32_t second = 64 - swap * 128, second_f = (GEO::A_ROWS - swap * 2 * GEO::A_ROWS) * 4;
    float acc[128];

    // One K-block; the first one starts the sums (nothing has to be cleared between two tiles).
    auto k_block = [&](auto first) -> bool {
        constexpr bool FIRST = decltype(first)::value;
        const uint32_t s = it % GEO::STAGES, ph = (it / GEO::STAGES) & 1, buf = it & 1;
        // Every lane polls (a single polling lane plus a broadcast was measured 2.5 % slower); the vote
        // keeps the warp converged when a wait gives up: either all lanes go on or none does.
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&ctrl->done[s]), ph, c.abort_flag, c.limit))) {
            if (lane == 0) raise(ctrl, g.status, DEV_TIMEOUT_EPILOGUE);
            return false;
        }
        tc_fence_after();
        const uint32_t col = t_lane + buf * G_TILE_N;
        float v[64];
        tmem_ld32_issue(col, v);
        tmem_ld32_issue(col + 32, v + 32);
        const uint32_t slot = factors + (it % GEO::SCALE_SLOTS) * 2 * GEO::A_ROWS * 4;
        const float f0 = ld_shared_f32(slot), f1 = MODE == 1 ? ld_shared_f32(slot + second_f) : f0;
        tmem_wait_ld(v);
        fma64<FIRST>(acc, v, f0);
        tmem_ld32_issue(col + second, v);
        tmem_ld32_issue(col + second + 32, v + 32);
        tmem_wait_ld(v);
        tc_fence_before();
        bar_arrive(ACC_BARRIER + buf, ACC_BARRIER_THREADS);
        fma64<FIRST>(acc + 64, v, f1);
        ++it;
        return true;
    };
    const uint32_t end = it + g.num_kb;
    if (!k_block(Bool<true>{})) return false;
    while (it != end)
        if (!k_block(Bool<false>{})) return false;

    t = read_tile(c, i);
    const int m_tile = t.m_tile(), n = t.n, rows_valid = t.rows;
    if (MODE == 2) {
        uint8_t* blk = reinterpret_cast<uint8_t*>(g.out_bf16) +
                       (((static_cast<size_t>(m_tile) * g.n_tiles + n) * 2 + half) * 4 + quad) * 8192 + lane * 32;
        if (quad * 32 < rows_valid) store_rows64(blk, acc);
        t = next_tile_warp(c, i + 1);  // (not behind all of the stores)
        if (quad * 32 < rows_valid) store_rows64(blk + 4096, acc + 64);
        return true;
    }
    const size_t row_cap = static_cast<size_t>(g.row_cap);
    const size_t row = static_cast<size_t>(m_tile) * TILE_M + r_in_tile;
    uint8_t* stage = c.store_stage + widx * G_STORE_WARP_BYTES;  // staging of this warp's GEMM1 rows
    // The staging area of this warp was handed to the TMA engine at the end of the previous tile; by now (a whole tile
    // later) that copy has long landed, so this wait does not stall.
    announce.settle(lane, t.key & TileInfo::LAST_TWO, g.ready, g.n_tiles);
    const int sw = (lane >> 1) & 3;  // 64-byte swizzle: 16-byte chunk index ^= bits 7..8 of the address
    // SwiGLU on this thread's 64 columns, then the row's 128-wide amax across the two halves
    float cc[64];
    float amax = 0.0f;
#pragma unroll
    for (int j = 0; j < 64; ++j) {
        cc[j] = silu_fast(acc[j]) * acc[64 + j];
        amax = fmaxf(amax, fabsf(cc[j]));
    }
    // The two warps of these 32 rows exchange their maxima.
    float* ax = c.amax_x + turn.area() * 2 * TILE_M;
    ax[half * TILE_M + r_in_tile] = amax;
    const uint32_t xbar = smem_u32(&ctrl->amax_quad[quad]);
    __syncwarp();
    if (lane == 0) mbar_arrive(xbar);
    t = next_tile_warp(c, i + 1);
    if (!__all_sync(0xffffffffu, mbar_wait(xbar, turn.quad(), c.abort_flag, c.limit))) {
        if (lane == 0) raise(ctrl, g.status, DEV_TIMEOUT_EPILOGUE);
        return false;
    }
    turn.bits ^= 5;
    amax = fmaxf(amax, *reinterpret_cast<volatile float*>(&ax[(half ^ 1) * TILE_M + r_in_tile]));
    const float sc = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, 448.0f);
    const float inv_sc = __frcp_rn(sc);
    if (quad * 32 < rows_valid) {
        // e4m3 rows out: 32 rows x 64 bytes per warp, staged with the 64-byte swizzle, one TMA store
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = q * 16 + k * 4;
                const uint32_t lo = __nv_cvt_float2_to_fp8x2(
                    make_float2(cc[j] * inv_sc, cc[j + 1] * inv_sc), __NV_SATFINITE, __NV_E4M3);
                const uint32_t hi = __nv_cvt_float2_to_fp8x2(
                    make_float2(cc[j + 2] * inv_sc, cc[j + 3] * inv_sc), __NV_SATFINITE, __NV_E4M3);
                w[k] = lo | (hi << 16);
            }
            *reinterpret_cast<uint4*>(stage + lane * 64 + ((q ^ sw) << 4)) =
                make_uint4(w[0], w[1], w[2], w[3]);
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
            tma_store_2d(tmOut, smem_u32(stage), n * 128 + half * 64, m_tile * TILE_M + quad * 32);
            bulk_commit_group();
        }
        if (half == 0 && r_in_tile < rows_valid)
            g.out_scale_t[static_cast<size_t>(n) * row_cap + row] = sc;
    }
    return true;
}

template <class GEO>
__device__ __forceinline__ void mlp_epilogue(const Cta& c, const CUtensorMap* tmOut, const MlpArgs& a) {
    uint32_t it = 0, unused = 0;
    AmaxTurn turn{0};
    bool ok = true;
    Announce announce{0, 0};
    TileInfo t = next_tile_warp(c, 0);
    for (uint32_t i = 0; t.mode() != 0; ++i) {
        const uint32_t end = it + (t.mode() == 1 ? a.g1.num_kb : a.g2.num_kb);
        const bool wm = t.rows <= a.g1.wm_rows;
        const int tile = t.m_tile() * a.g1.n_tiles + t.n;  // (GEMM1)
        const bool last = t.key & TileInfo::LAST;
        if (ok) {
            if (t.mode() == 1) {
                ok = wm ? epilogue_tile_wm<1, false, GEO>(c, a.g1, nullptr, t.m_tile(), t.n, it, turn, unused, 0, -1, 1,
                                                                &announce, t.key & TileInfo::LAST_TWO)
                        : mlp_epilogue_tile<1, GEO>(c, tmOut, a.g1, i, t, it, turn, announce);
                if (ok) {
                    if (a.by_row) announce.add(tile);
                    if (last) announce.settle(c.lane, true, a.g1.ready, a.g1.n_tiles);  // somebody may be waiting for it
                }
            } else {
                ok = wm ? epilogue_tile_wm<2, false, GEO>(c, a.g2, nullptr, t.m_tile(), t.n, it, turn, unused, 0, -1, 1,
                                                                &announce, false)
                        : mlp_epilogue_tile<2, GEO>(c, tmOut, a.g2, i, t, it, turn, announce);
            }
        }
        // After an abort: the hand-overs this warp still owes, waiting for the issuer so that no turn is taken twice.
        for (; it < end; ++it) bar_sync(ACC_BARRIER + (it & 1), ACC_BARRIER_THREADS);
        if (!ok || wm) t = next_tile_warp(c, i + 1);
    }
    if (c.lane == 0) bulk_wait_all();
}

// tmA*s: 32-row boxes of the same buffers for short row tiles.
__global__ void __launch_bounds__(G_THREADS, 1)
grouped_mlp_kernel(const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmA1s,
                   const __grid_constant__ CUtensorMap tmB1n, const __grid_constant__ CUtensorMap tmB1m,
                   const __grid_constant__ CUtensorMap tmOut, const __grid_constant__ CUtensorMap tmA2,
                   const __grid_constant__ CUtensorMap tmA2s, const __grid_constant__ CUtensorMap tmB2, const __grid_constant__ MlpArgs a) {
    extern __shared__ uint8_t smem_raw[];
    using GEO = GeomFull;
    Cta c;
    gemm_cta_setup<GEO>(c, smem_raw, 1);
    if (c.warp == 0 && c.lane == 0) {
        tma_prefetch_desc(&tmA1);
        tma_prefetch_desc(&tmB1n);
        tma_prefetch_desc(&tmB1m);
        tma_prefetch_desc(&tmB2);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // Everything above touched only this CTA's shared and tensor memory; activations and scales were written by the
    // kernels before this one (warps 0 and 3 wait for them by themselves: weights and tile tables are there already,
    // see place_gather_kernel).
    pdl_launch_dependents();
    const bool overlaps = a.phases == 2 && a.by_row;  // with the GEMM1 launch before it, see MLP_SPLIT_MAX_TOKENS
    if (c.warp != 0 && c.warp != 3 && !overlaps) pdl_wait();
    c.tmem_base = *reinterpret_cast<volatile uint32_t*>(&c.ctrl->tmem_slot);
    c.limit = a.g1.wait_limit;
    uint32_t claimed = 0;

    if (c.warp < 4) {
        reg_dealloc<56>();
        if (c.warp == 0) {
            if (c.lane == 0) claimed = mlp_producer<GEO>(c, &tmA1, &tmA1s, &tmB1n, &tmB1m, &tmA2, &tmA2s, &tmB2, a);
        } else if (c.warp == 3) {
            mlp_factors<GEO>(c, a);
        } else {
            mlp_issuer<GEO>(c, a, c.warp - 1);
        }
    } else {
        reg_alloc<224>();
        mlp_epilogue<GEO>(c, &tmOut, a);
    }

    __syncwarp();
    if (overlaps) pdl_wait();  // (so that whoever follows finds GEMM1's launch finished as well)
    tc_fence_before();
    __syncthreads();
    if (*c.abort_flag) drain_after_abort<GEO>(c, a.g1.status, claimed, claimed);
    if (c.warp == 1) {
        __syncwarp();
        tmem_dealloc(c.tmem_base, G_TMEM_COLS);
    }
}

}  // namespace moe
