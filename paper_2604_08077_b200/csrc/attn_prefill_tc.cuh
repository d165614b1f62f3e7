// K4: gathered flash-style attention on the 5th-generation tensor cores (Eq. 3; un-permute of
// Algorithm 1 fused into the epilogue).
//
// Two CTAs of a cluster (cta_group::2) work on one "pair tile": 256 consecutive cube-major query rows of one query head,
// 128 rows in either CTA's TMEM, the K / V^T tiles split between the CTAs' shared memories.  The kernel is persistent: a
// cluster draws pair tile after pair tile, longest first, and the roles of a CTA (512 threads) go through them side by side,
// coupled by barriers alone, so that plan, loads and first scores of the next pair tile overlap the end of the present one:
//   warps 0-11  softmax, three warpgroups that take the key steps in turn (thread = query row = TMEM lane)
//   warp  12    TMA producer of K
//   warp  13    MMA issuer (CTA 0): S = Q K^T (operands in shared memory), O += P V (P in TMEM); CTA 1: passes on that its Q is there
//   warp  14    TMA producer of V^T
//   warp  15    planner: the list of visited key blocks, the Q tile and the score bounds of the next pair tile
// Key blocks (64 cube-major positions) are visited in pairs (128 keys per step).  A block is
// needed if any row of the pair tile selected a cube inside it or if it overlaps the tile's local
// range (own cubes / text prefix).  Each softmax thread masks its own row: one selection bit per
// (row, cube) for blocks before the local range, the exact per-key rule inside it.
//
// Who waits for whom, so that nobody waits in a circle.  The issuer never waits for a pair tile that it has not begun while a
// product of an earlier one is still to be issued.  For the plan of pair tile k, in either CTA, waits for the softmax warps of
// k - 2 to have finished (k - 1, where long block lists leave one slot), and their rows, where no reference is fixed in
// advance, wait with the rescaling in step g for the product of step g - 1 to have completed.  Were the issuer to wait for k with
// products of k - 1 outstanding, CTA 1 could wait for those products and the issuer for CTA 1 (its Q of k is loaded behind its plan
// of k).  With every product up to k - 1 issued all softmax warps get to the end of k - 1: scores have been issued ahead of
// the products, K / V^T loads wait for scores and products only, an epilogue for the last product, the sums of its own pair tile and the
// output rows of the one before; so plan, Q and first scores of k follow.  Inside a begun pair tile the issuer waits for K, V^T
// (loaded behind plans that both CTAs have: CTA 1 reports its Q behind its plan), for weights (the softmax of scores issued before, in
// the order of the steps) and for the epilogue before the first product.
//
// TMEM (512 columns): three tiles of 128 columns for S (fp32) -- P (bf16 pairs) overwrites the first 64 -- and D columns
// for O.  What bounds a step is the chain S -> softmax -> P -> O, S of one such tile, 3100 to 3800 cycles.  With two tiles (and two
// O, 256 rows of one CTA) it took 3180 cycles for both, 2048 of them tensor core; three tiles leave two steps in the softmax while
// one is on the tensor core: 1260 a step of 128 rows, 1024 of them tensor core.  O fits beside three tiles only because a CTA holds
// 128 rows; that K / V^T traffic does not double by it is what the CTA pair is for.  The persistent form hides 7000 cycles of
// set-up and 3000 of epilogue a pair tile (12 % at 16384 tokens); beyond some ten thousand tokens the board's power limit
// bounds the kernel: it executes 1340 TFLOP/s at 1.5 GHz, cuBLAS over seconds 1436.  Measured, 28 heads, 64-token cubes, p 0.9:
// 1.65 -> 1.51 ms at 16384 tokens, 25.2 -> 23.2 at 65536; 256-token cubes, cohesive queries: 0.87 -> 0.79; dense, 16 heads of 64, 8192 tokens:
// 0.238 -> 0.213.  Two softmax warpgroups instead of three: 5 % slower.
#pragma once
#include "tc_common.cuh"

namespace adaspark {

constexpr int kSoftmaxGroups = 3;                      // warpgroups that take the key steps in turn
constexpr int kTcThreads = (kSoftmaxGroups + 1) * 128;
constexpr int kSoftmaxRegs = 144;     // per-thread registers of the softmax warpgroups after setmaxnreg
constexpr int kHelperRegs = 80;       // ... of the other warpgroup
// setmaxnreg only moves registers inside what the CTA got at launch: 512 threads x 128 registers (the
// compile-time bound of __launch_bounds__(512, 1)).  A request beyond that blocks forever.
static_assert(kSoftmaxGroups * 128 * kSoftmaxRegs + 128 * kHelperRegs <= kTcThreads * 128, "setmaxnreg must stay inside the CTA's launch allocation");
constexpr int kPairRows = 256;
constexpr int kScoreBufs = 3;         // score / weight tiles in TMEM
static_assert(kScoreBufs == kSoftmaxGroups, "a warpgroup owns a tile");
constexpr int kRefSlots = 4;          // a warpgroup is at most three steps behind the others: slots of the running reference
// Reference of a row's softmax fixed in advance: the bound B of its scores (log2 units; every score lies in [-B, B]), up to this B.
// Every weight 2^(s - B) is at least 2^-2B = 2^-96: nothing underflows, and 30 binades remain above the smallest normal fp32 for
// the products with V.  Not beyond: the largest weights of a row, 1 or a power of two near it on the running maximum, are any numbers with
// a fixed reference and lose up to 2^-9 each in bf16.  References up to B = 88 (96 - B) and in later chunks gained 8 % on a chunk, but
// their error against 64 bits was up to 5 % larger (sharp queries, p 0.95: 0.00226 -> 0.00234; a chunk 0.00232 -> 0.00235).
constexpr float kFixedRefMax = 48.f;
// |q|^2, largest |k|^2 of the head: infinite, not in advance
__device__ __forceinline__ float fixed_reference(float q2, float k2, float scale_log2) {
    const float bound = sqrtf(q2 * k2) * scale_log2 * 1.01f + 0.01f;     // 1 % for the rounding of the norms and of s
    return bound <= kFixedRefMax ? bound : INFINITY;
}
constexpr int kFmaExpEvery = 2;       // of every 4 kFmaExpEvery exponentials one is a cubic on the FMA pipe (one in four: no faster, four times the error)
constexpr int kMaxKeyBlocks = 32768;  // key blocks per sequence (2M positions): a number and a flag fit 16 bits
constexpr uint32_t kPartialBlock = 0x8000u;   // flag of a listed block: some of its slots hold no token (ragged grid)
// Lists of up to this many key blocks (147456 positions) are kept twice, for the present and the next pair tile; a longer one once,
// in the place of the last K / V^T tiles.
constexpr int kBlockListShort = 2304;
__host__ __device__ constexpr int max_kv_stages(int D) { return D == 64 ? 6 : 3; }   // K and V^T tiles in flight
// ... of a call whose sequences have n_blocks key blocks
__host__ __device__ constexpr int kv_stages(int D, int n_blocks) {
    return n_blocks <= kBlockListShort ? max_kv_stages(D) : max_kv_stages(D) - (2 * n_blocks + 256 * D - 1) / (256 * D);
}
static_assert(kv_stages(64, kMaxKeyBlocks) >= 1 && kv_stages(128, kMaxKeyBlocks) >= 1, "room for the longest list");

// Does the key block lie (in part) in a cube that holds fewer tokens than slots?
__device__ __forceinline__ bool block_partial(const Geom& g, int kb) {
    for (int pos = kb * kBlockTok; pos < min((kb + 1) * kBlockTok, g.S_v); pos += min(g.C, kBlockTok))
        if (cube_tokens_held(g, pos >> g.c_shift) != g.C) return true;
    return false;
}

template <int D>
struct TcAttnSmem {
    __nv_bfloat16 q[2][D / 64][128][64];              // [pair tile & 1][d panel][row][64 d]
    __nv_bfloat16 kv[2 * max_kv_stages(D)][64 * D];   // a K tile ([d panel][key of this CTA's block][64 d]) or a V^T tile
                                                      // ([block][this CTA's half of d][64 keys]) each
    unsigned char out[128][2 * D + 16];               // output rows (16 bytes of padding spread the banks)
    float ref[kRefSlots][128];                        // running reference of a row after a step
    float part_l[2][kSoftmaxGroups][128], part_m[2][kSoftmaxGroups][128];   // sums and references of the warpgroups
    float fixed[4][128];                              // reference of a row fixed in advance, infinite if it is not
    uint64_t q_full[2], q_peer[2], q_empty[2], k_full[max_kv_stages(D)], k_empty[max_kv_stages(D)], v_full[max_kv_stages(D)], v_empty[max_kv_stages(D)];
    uint64_t s_full[kScoreBufs], p_full[kScoreBufs], ref_done[kRefSlots][4], o_full, o_free;
    uint64_t plan_full[2], plan_empty[2], bound_full[4], part_full[2], part_free[2], out_free;
    int plan_blocks[2], plan_item[2];                 // visited key blocks; pair tile, -1: no more
    uint64_t item_full[4];                            // (CTA 1) CTA 0 has drawn the pair tile
    int next_item[4];
    uint32_t tmem_base;
    int abort_flag;
    uint16_t list[2][kBlockListShort];                // the visited key blocks in order
};

template <int D>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTcThreads, 1) attn_prefill_tc_kernel(
    Geom g, const __grid_constant__ CUtensorMap tmQ, const __nv_bfloat16* __restrict__ q, const __grid_constant__ CUtensorMap tmK,
    const __grid_constant__ CUtensorMap tmV, const uint32_t* tile_mask, const uint32_t* tile_union, const uint32_t* slot_valid,
    const uint32_t* pair_mode, int n_pairs_cap, float2* ml_local, const uint32_t* key_norm2_bits, __nv_bfloat16* out,
    uint32_t* next_pair_tile, unsigned long long* executed_blocks, uint32_t* max_tile_blocks, int32_t* status) {
    extern __shared__ unsigned char tc_smem_raw[];
    TcAttnSmem<D>& sm = *reinterpret_cast<TcAttnSmem<D>*>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr int kPanels = D / 64;
    constexpr int kQKSteps = D / 16;                            // k-steps of S = Q K^T
    constexpr uint32_t kIdescS = tc::make_idesc_bf16(256, 128);  // S tile: 256 rows (128 per CTA) x 128 keys
    constexpr uint32_t kIdescO = tc::make_idesc_bf16(256, D);    // O tile: 256 rows x D
    constexpr uint32_t kTileBytes = 64 * D * 2;                  // a CTA's share of the K or V^T tile of a step
    constexpr int kKWarp = kSoftmaxGroups * 4, kMmaWarp = kKWarp + 1, kVWarp = kKWarp + 2, kPlanWarp = kKWarp + 3;
    constexpr uint32_t kOCol = kScoreBufs * 128;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)(blockIdx.x & 1u), n_clusters = (int)(gridDim.x >> 1);
    const int n_hb = g.Hq * g.B, n_pairs = (g.S + kPairRows - 1) / kPairRows;
    const int n_items = (n_pairs - g.pos_begin / kPairRows) * n_hb;
    const int n_stages = kv_stages(D, g.n_kv_blocks_cap);
    const bool long_list = g.n_kv_blocks_cap > kBlockListShort;
    // pair tile number k of this cluster: pair-major, the late (long) pairs of every head and batch entry first
    struct Item { int pair, b, h, gk; };
    auto item_at = [&](int i) -> Item {
        Item it;
        const int p = i / n_hb, hb = i - p * n_hb;
        it.pair = n_pairs - 1 - p;
        it.b = hb / g.Hq;
        it.h = hb - it.b * g.Hq;
        it.gk = it.h / g.G;
        return it;
    };
    // slot of pair tile k's block list and phase of its barriers
    auto plan_slot = [&](int k) -> int { return long_list ? 0 : k & 1; };
    auto plan_phase = [&](int k) -> uint32_t { return (uint32_t)(long_list ? k & 1 : (k >> 1) & 1); };
    auto list_at = [&](int slot) -> uint16_t* { return long_list ? reinterpret_cast<uint16_t*>(&sm.kv[2 * n_stages][0]) : sm.list[slot]; };

    // ---------------------------------------------------------------- set-up
    launch_dependents();
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&sm.q_full[i], 1);
            tc::mbar_init(&sm.q_peer[i], 1);
            tc::mbar_init(&sm.q_empty[i], 1);
            tc::mbar_init(&sm.plan_full[i], 1);
            tc::mbar_init(&sm.plan_empty[i], 3 + kSoftmaxGroups * 4);
            tc::mbar_init(&sm.part_full[i], (kSoftmaxGroups - 1) * 4);
            tc::mbar_init(&sm.part_free[i], 4);
        }
        for (int i = 0; i < max_kv_stages(D); ++i) {
            tc::mbar_init(&sm.k_full[i], 1);
            tc::mbar_init(&sm.k_empty[i], 1);
            tc::mbar_init(&sm.v_full[i], 1);
            tc::mbar_init(&sm.v_empty[i], 1);
        }
        for (int i = 0; i < kScoreBufs; ++i) {
            tc::mbar_init(&sm.s_full[i], 1);
            tc::mbar_init(&sm.p_full[i], 8);                    // a warp of either CTA each
        }
        for (int i = 0; i < 4; ++i) {
            tc::mbar_init(&sm.bound_full[i], 1);
            tc::mbar_init(&sm.item_full[i], 1);
            for (int w = 0; w < 4; ++w) tc::mbar_init(&sm.ref_done[i][w], 1);
        }
        tc::mbar_init(&sm.o_full, 1);
        tc::mbar_init(&sm.o_free, 8);
        tc::mbar_init(&sm.out_free, 4);
        sm.abort_flag = 0;
        tc::fence_barrier_init();
        tc::prefetch_tensormap(&tmQ);
        tc::prefetch_tensormap(&tmK);
        tc::prefetch_tensormap(&tmV);
    }
    __syncwarp();
    wait_for_previous_kernel();
    // (not before the wait: a CTA of the previous kernel that is still to allocate would wait for this one)
    if (warp == kMmaWarp) tc::tmem_alloc_pair<512>(&sm.tmem_base);
    tc::tc_fence_before_sync();
    cluster_sync();                                              // barriers and TMEM of both CTAs
    tc::tc_fence_after_sync();
    const uint32_t tbase = sm.tmem_base;
    volatile int* abort_flag = &sm.abort_flag;

    if (warp >= kKWarp) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kHelperRegs));
    if (warp == kPlanWarp) {
        // ------------------------------------------------------------ planner
        unsigned long long blocks_sum = 0;
        uint32_t blocks_max = 0;
        bool ok = true;
        // The first pair tile is the cluster's own number, the second is dealt backwards, so that the longest first one is joined by the
        // shortest second (drawn when all clusters begin, one ahead, it would be the longest: 1536 tokens, 16 heads of 64, 71 for 67 us;
        // 512 + 40 tokens, 28 heads, 34.2 for 31.1), the others are drawn from a counter by CTA 0, one ahead.  (Dealt out in
        // turn: 0.89 for 0.82 ms with 256-token cubes, whose unions differ, 1.65 for 1.55 with equal ones.)
        int i = (int)(blockIdx.x >> 1);
        for (int k = 0; ok; ++k) {
            const int slot = plan_slot(k);
            if (k > 0) {
                if (rank == 0) i = __shfl_sync(0xffffffffu, i, 0);
                else {
                    if (!(ok = tc::mbar_wait(&sm.item_full[(k - 1) & 3], ((k - 1) >> 2) & 1, abort_flag))) break;
                    asm volatile("fence.acq_rel.cluster;\n" ::: "memory");
                    i = *(volatile int*)&sm.next_item[(k - 1) & 3];
                }
            }
            int drawn = n_items;
            if (rank == 0 && lane == 0 && i < n_items)
                drawn = k == 0 ? 2 * n_clusters - 1 - i : 2 * n_clusters + (int)atomicAdd(next_pair_tile, 1u);
            if (!(ok = tc::mbar_wait(&sm.plan_empty[slot], plan_phase(k) ^ 1u, abort_flag))) break;
            if (i >= n_items) {
                if (lane == 0) {
                    sm.plan_item[slot] = -1;
                    tc::mbar_arrive(&sm.plan_full[slot]);
                }
                break;
            }
            const int item = i;
            const Item it = item_at(item);
            const int pair_pos0 = it.pair * kPairRows, tile_pos0 = pair_pos0 + rank * 128;
            const int pair_end = min(pair_pos0 + kPairRows, g.S);       // exclusive
            // key blocks that can matter: up to the pair's own end, and for a pair with video rows also the blocks
            // of the text prefix (attended by every video row)
            const int prefix_blk0 = g.S_v / kBlockTok, prefix_blk1 = (g.S_v + g.n_prefix + kBlockTok - 1) / kBlockTok;
            const bool sees_prefix = g.n_prefix > 0 && pair_pos0 < g.S_v;
            const int n_blk_own = (pair_end + kBlockTok - 1) / kBlockTok;
            const int n_blk = sees_prefix ? max(n_blk_own, prefix_blk1) : n_blk_own;
            const int first_local_blk = pair_first_local_blk(g, pair_pos0);
            // A pair whose selected cubes go through the query-gather kernels (attn_gather.cuh) visits only its local
            // range and the text prefix here and leaves (reference exponent, sum) of every row for the merge.
            const bool gathered = pair_mode != nullptr && pair_mode[(size_t)(it.b * g.Hq + it.h) * n_pairs_cap + it.pair] != 0u;
            // The Q tile does not wait for the plan.  It comes straight from the caller's tensor [B, S_io, Hq, D]: the video
            // rows of a tile are whole boxes of a cube's window (or the cubes themselves, below 128 tokens) in the
            // (head x d, x, y, t, batch) view of that tensor, which one 5-D TMA load per box and 64-element panel turns into
            // cube-major rows (a coordinate beyond the grid reads zeros: the empty slots of a boundary cube); text rows and
            // the slots beyond the sequence, a few tiles per head, are copied by the warp's lanes.
            const int qs = k & 1;
            if (!(ok = tc::mbar_wait(&sm.q_empty[qs], ((k >> 1) & 1) ^ 1, abort_flag))) break;
            unsigned char* qt = reinterpret_cast<unsigned char*>(&sm.q[qs][0][0][0]);
            const int rpb = min(g.C, 128);                            // rows per box
            const int n_vid = max(0, min(tile_pos0 + 128, g.S_v) - tile_pos0);  // video slots of the tile (a multiple of rpb or of C)
            for (int idx = lane; idx < (128 - n_vid) * (D / 8); idx += 32) {
                const int row = n_vid + idx / (D / 8), c = idx % (D / 8);
                const int pos = tile_pos0 + row;
                unsigned char* dst = qt + (c >> 3) * (128 * 128) + sw128(row, c & 7);
                if (pos < g.S) cp_async_16(dst, q + (io_row(g, it.b, pos) * g.Hq + it.h) * D + c * 8);
                else *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
            }
            // all copies under way at once (a load and a store at a time: 3 to 6 us of a call of a few thousand tokens with text)
            cp_async_commit();
            cp_async_wait<0>();
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // the copied rows are read by the tensor core
            __syncwarp();
            if (lane == 0) {
                if (n_vid) tc::mbar_arrive_expect_tx(&sm.q_full[qs], (uint32_t)n_vid * D * 2);
                else tc::mbar_arrive(&sm.q_full[qs]);
                for (int r = 0; r < n_vid; r += rpb) {
                    const int pos = tile_pos0 + r;
                    const int c = pos >> g.c_shift, r0 = pos & (g.C - 1);
                    int cx, cy, cb, tt;
                    g.div_nW.divmod(c, tt, cx);
                    g.div_nH.divmod(tt, cb, cy);
                    const int x = cx * g.cw + (r0 & (g.cw - 1));
                    const int y = cy * g.ch + ((r0 >> g.cw_shift) & (g.ch - 1));
                    const int fr = cb * g.ct + (r0 >> (g.cw_shift + g.ch_shift)) - g.frame_begin;
                    for (int p = 0; p < kPanels; ++p)
                        tc::tma_load_5d(&sm.q[qs][p][r][0], &tmQ, it.h * D + p * 64, x, y, fr, it.b, &sm.q_full[qs]);
                }
            }
            __syncwarp();
            // The visited blocks, a lane per word of 32: a block is visited if any of the pair's 256 rows selected a cube in it
            // (OR of the two tiles' union words, written by the selection kernel) or the local range or the prefix needs it.
            uint16_t* list = list_at(slot);
            const uint32_t* un0 = tile_union + ((size_t)(it.b * g.Hq + it.h) * g.n_tiles_cap + it.pair * 2) * g.n_words;
            const uint32_t* un1 = it.pair * 2 + 1 < g.n_tiles ? un0 + g.n_words : un0;
            int n_needed = 0;
            for (int w32 = 0; w32 * 32 < n_blk; w32 += 32) {
                const int wi = w32 + lane, kb0 = wi * 32;
                uint32_t bits = 0;
                if (!gathered && kb0 < first_local_blk) {
                    if (g.c_shift >= 6) {                           // 32 blocks are 32 >> (c_shift - 6) cubes of one word
                        const int sh = g.c_shift - 6, c0 = kb0 >> sh;
                        const uint32_t u = (un0[c0 >> 5] | un1[c0 >> 5]) >> (c0 & 31);
                        if (sh == 0) bits = u;
                        else
                            for (int x = 0; x < 32; ++x) bits |= ((u >> (x >> sh)) & 1u) << x;
                    } else {                                        // 32 blocks are the cubes of 2 (32 tokens) or 4 words
                        const int per = 6 - g.c_shift, n_w = 1 << per;   // n_w cubes per block
                        for (int x = 0; x < n_w; ++x) {
                            const int w = wi * n_w + x;
                            const uint32_t u = w < g.n_words ? (un0[w] | un1[w]) : 0u;
                            const int n_b = 32 >> per;              // blocks of this word
                            for (int y = 0; y < n_b; ++y)
                                if ((u >> (y << per)) & ((1u << n_w) - 1u)) bits |= 1u << (x * n_b + y);
                        }
                    }
                    if (first_local_blk - kb0 < 32) bits &= (1u << (first_local_blk - kb0)) - 1u;
                }
                // blocks [lo, hi) of the word
                auto range = [&](int lo, int hi) -> uint32_t {
                    lo = min(max(lo - kb0, 0), 32);
                    hi = min(max(hi - kb0, 0), 32);
                    return hi > lo ? (0xffffffffu >> (32 - (hi - lo))) << lo : 0u;
                };
                bits |= range(first_local_blk, n_blk_own);
                if (sees_prefix) bits |= range(prefix_blk0, n_blk);
                for (uint32_t words = __ballot_sync(0xffffffffu, bits != 0u); words; words &= words - 1u) {
                    const int x = __ffs(words) - 1;
                    const uint32_t bw = __shfl_sync(0xffffffffu, bits, x);
                    if ((bw >> lane) & 1u) {
                        const int kb = (w32 + x) * 32 + lane;
                        list[n_needed + __popc(bw & ((1u << lane) - 1u))] = (uint16_t)((uint32_t)kb | (g.ragged && block_partial(g, kb) ? kPartialBlock : 0u));
                    }
                    n_needed += __popc(bw);
                }
            }
            __syncwarp();
            if (lane == 0) {
                if (n_needed & 1) list[n_needed] = list[n_needed - 1];   // odd count: the last block once more, masked
                sm.plan_blocks[slot] = n_needed;
                sm.plan_item[slot] = item;
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&sm.plan_full[slot]);
            if (rank == 0) {                                      // (CTA 1 has read what the slot held: it has worked on pair tile k - 2)
                if (lane == 0) {
                    asm volatile("st.shared::cluster.u32 [%0], %1;\n" ::"r"(cluster_address(&sm.next_item[k & 3], 1)), "r"(drawn) : "memory");
                    tc::mbar_arrive_release_cluster(cluster_address(&sm.item_full[k & 3], 1));
                }
                i = drawn;
            }
            blocks_sum += (unsigned long long)(2 * n_needed);
            blocks_max = max(blocks_max, (uint32_t)n_needed);
            // Bound of a row's scores: |s| <= |q| |k| for every key; the largest key norm of the head comes from the re-layout
            // kernel (none when not every attended key went through this call's re-layout).
            {
                if (!(ok = tc::mbar_wait(&sm.q_full[qs], (k >> 1) & 1, abort_flag))) break;
                const float k2 = key_norm2_bits != nullptr ? __uint_as_float(key_norm2_bits[it.b * g.Hkv + it.gk]) : INFINITY;
#pragma unroll 1
                for (int row = lane; row < 128; row += 32) {
                    unsigned long long qq[2] = {0ull, 0ull};
#pragma unroll
                    for (int c = 0; c < D / 8; ++c) {
                        const uint4 qv = *reinterpret_cast<const uint4*>(qt + (c >> 3) * (128 * 128) + sw128(row, c & 7));
                        const uint32_t w[4] = {qv.x, qv.y, qv.z, qv.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const unsigned long long x2 = pack_f32x2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u));
                            qq[e & 1] = fma_f32x2(x2, x2, qq[e & 1]);
                        }
                    }
                    float qa, qb;
                    unpack_f32x2(add_f32x2(qq[0], qq[1]), qa, qb);
                    sm.fixed[k & 3][row] = fixed_reference(qa + qb, k2, g.scale_log2);
                }
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&sm.bound_full[k & 3]);
            }
        }
        if (rank == 0 && lane == 0 && ok) {
            atomicAdd(executed_blocks, blocks_sum);
            atomicMax(max_tile_blocks, blocks_max);
        }
    } else if (warp == kKWarp || warp == kVWarp) {
        // ------------------------------------------------------------ TMA producers, one of K and one of V^T
        // CTA r fetches block r of a step's two K blocks and half r of d of both V^T blocks: its share of the B operands.
        // Both CTAs' loads complete on the barriers of CTA 0, whose warp issues the MMAs.
        const bool is_v = warp == kVWarp;
        if (tc::elect_one()) {
            uint64_t* const full = is_v ? sm.v_full : sm.k_full;
            uint64_t* const empty = is_v ? sm.v_empty : sm.k_empty;
            const uint32_t bar0 = cluster_address(full, 0);
            int st = 0, ph = 1;                                   // stage and phase of the next tile
            bool ok = true;
            for (int k = 0; ok; ++k) {
                const int slot = plan_slot(k);
                if (!(ok = tc::mbar_wait(&sm.plan_full[slot], plan_phase(k), abort_flag))) break;
                if (sm.plan_item[slot] < 0) break;
                const Item it = item_at(sm.plan_item[slot]);
                const int row0 = is_v ? (it.b * g.Hkv + it.gk) * g.n_kv_blocks_cap * D + rank * (D / 2) : (it.b * g.Hkv + it.gk) * g.S_cap;
                const uint32_t* steps = reinterpret_cast<const uint32_t*>(list_at(slot));
                const int n_steps = (sm.plan_blocks[slot] + 1) / 2;
                for (int j = 0; j < n_steps; ++j) {
                    const uint32_t blk = steps[j];
                    const int kb_a = (int)(blk & 0x7fffu), kb_b = (int)((blk >> 16) & 0x7fffu);
                    if (!(ok = tc::mbar_wait(&empty[st], ph, abort_flag))) break;
                    if (rank == 0) tc::mbar_arrive_expect_tx(&full[st], 2 * kTileBytes);
                    if (is_v) {
                        tc::tma_load_2d_pair(&sm.kv[n_stages + st][0], &tmV, 0, row0 + kb_a * D, bar0 + st * 8);
                        tc::tma_load_2d_pair(&sm.kv[n_stages + st][(D / 2) * 64], &tmV, 0, row0 + kb_b * D, bar0 + st * 8);
                    } else {
                        for (int p = 0; p < kPanels; ++p)
                            tc::tma_load_2d_pair(&sm.kv[st][p * 64 * 64], &tmK, p * 64, row0 + (rank ? kb_b : kb_a) * kBlockTok, bar0 + st * 8);
                    }
                    if (++st == n_stages) { st = 0; ph ^= 1; }
                }
                tc::mbar_arrive(&sm.plan_empty[slot]);
            }
        }
    } else if (warp == kMmaWarp && rank == 1) {
        // ------------------------------------------------------------ CTA 1: Q is there, said to the issuing warp of CTA 0
        if (lane == 0) {
            for (int k = 0;; ++k) {
                if (!tc::mbar_wait(&sm.plan_full[plan_slot(k)], plan_phase(k), abort_flag) || sm.plan_item[plan_slot(k)] < 0) break;
                if (!tc::mbar_wait(&sm.q_full[k & 1], (k >> 1) & 1, abort_flag)) break;
                asm volatile("fence.acq_rel.cluster;\n" ::: "memory");
                tc::mbar_arrive_cluster(cluster_address(&sm.q_peer[k & 1], 0));
                tc::mbar_arrive(&sm.plan_empty[plan_slot(k)]);
            }
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------ MMA issuer
        // One elected thread runs the whole loop with warp-uniform operands: 64 cycles per 256x128x16 MMA, the tensor core's own
        // (an election before every batch, with the whole warp waiting on the barriers in between: 74).  The scores run three
        // steps ahead of the products with V, over the end of a pair tile as well.
        constexpr uint32_t kKStep = 32 >> 4;                                        // 16 elements of a 128-byte row
        constexpr uint32_t kQPanelStep = (128 * 128) >> 4, kKPanelStep = (64 * 128) >> 4, kVBlockStep = ((D / 2) * 128) >> 4;
        constexpr uint32_t kQSlotStep = (uint32_t)sizeof(sm.q[0]) >> 4, kStageStep = (uint32_t)sizeof(sm.kv[0]) >> 4;
        const uint32_t q_lo0 = __shfl_sync(0xffffffffu, tc::smem_desc_lo_sw128(smem_u32(&sm.q[0][0][0][0])), 0);
        const uint32_t k_lo0 = __shfl_sync(0xffffffffu, tc::smem_desc_lo_sw128(smem_u32(&sm.kv[0][0])), 0);
        const uint32_t v_lo0 = __shfl_sync(0xffffffffu, tc::smem_desc_lo_sw128(smem_u32(&sm.kv[n_stages][0])), 0);
        const uint32_t tb = __shfl_sync(0xffffffffu, tbase, 0);
        if (tc::elect_one()) {
            bool ok = true;
            // scores: pair tile ks, steps left in it, score tile, K stage
            bool ended = false;
            int ks = -1, s_left = 0, sbuf = 0, kst = 0, kph = 0, ahead = 0;
            int n_steps0 = 0, n_steps1 = 0, n_steps2 = 0;         // steps of pair tiles ks, ks - 1, ks - 2
            // S of the next step, if there is one.  While products are left to issue (must = false) the next pair tile is begun only
            // when its plan and both CTAs' Q tiles are there, and is not waited for: its plan, in either CTA, may wait for steps
            // whose rows wait for these products (see the file's header).
            auto next_scores = [&](bool must) -> bool {
                if (s_left == 0) {
                    if (ended) return false;
                    const int kn = ks + 1, slot = plan_slot(kn);
                    auto there = [&](uint64_t* bar, uint32_t phase) -> bool { return must ? (ok = tc::mbar_wait(bar, phase, abort_flag)) : tc::mbar_test(bar, phase); };
                    if (!there(&sm.plan_full[slot], plan_phase(kn))) return false;
                    if ((ended = sm.plan_item[slot] < 0)) return false;
                    if (!there(&sm.q_full[kn & 1], (kn >> 1) & 1) || !there(&sm.q_peer[kn & 1], (kn >> 1) & 1)) return false;
                    ks = kn;
                    n_steps2 = n_steps1;
                    n_steps1 = n_steps0;
                    s_left = n_steps0 = (sm.plan_blocks[slot] + 1) / 2;
                    tc::mbar_arrive(&sm.plan_empty[slot]);
                }
                if (!(ok = tc::mbar_wait(&sm.k_full[kst], kph, abort_flag))) return false;
                tc::tc_fence_after_sync();
                const uint32_t qa = q_lo0 + (ks & 1) * kQSlotStep, kb = k_lo0 + kst * kStageStep, dst = tb + sbuf * 128;
#pragma unroll
                for (int x = 0; x < kQKSteps; ++x)
                    tc::umma_ss_pair(dst, tc::smem_desc_from_halves(qa + (x >> 2) * kQPanelStep + (x & 3) * kKStep, tc::kSmemDescHiSw128),
                                     tc::smem_desc_from_halves(kb + (x >> 2) * kKPanelStep + (x & 3) * kKStep, tc::kSmemDescHiSw128), kIdescS, x > 0);
                tc::umma_commit_pair(&sm.s_full[sbuf]);
                tc::umma_commit_pair(&sm.k_empty[kst]);
                if (--s_left == 0) tc::umma_commit_pair(&sm.q_empty[ks & 1]);
                if (++sbuf == kScoreBufs) sbuf = 0;
                if (++kst == n_stages) { kst = 0; kph ^= 1; }
                ++ahead;
                return true;
            };
            int buf = 0, buf_ph = 0, vst = 0, vph = 0;            // score tile and V^T stage of the next product
            for (int k = 0; ok; ++k) {
                int steps = 1;
                for (int j = 0; j < steps; ++j) {
                    while (ahead < kScoreBufs && next_scores(ahead == 0)) {}
                    if (!ok || ahead == 0) { ok = false; break; }  // no more
                    if (j == 0) steps = ks == k ? n_steps0 : ks == k + 1 ? n_steps1 : n_steps2;
                    if (!(ok = tc::mbar_wait(&sm.v_full[vst], vph, abort_flag))) break;
                    if (j == 0 && k > 0 && !(ok = tc::mbar_wait(&sm.o_free, (k - 1) & 1, abort_flag))) break;   // O of the pair tile before has been read
                    if (!(ok = tc::mbar_wait(&sm.p_full[buf], buf_ph, abort_flag))) break;
                    tc::tc_fence_after_sync();
                    const uint32_t vb = v_lo0 + vst * kStageStep, src = tb + buf * 128;
#pragma unroll
                    for (int x = 0; x < 8; ++x)                    // O (+)= P V
                        tc::umma_ts_pair(tb + kOCol, src + x * 8,
                                         tc::smem_desc_from_halves(vb + (x >> 2) * kVBlockStep + (x & 3) * kKStep, tc::kSmemDescHiSw128), kIdescO, x > 0 || j > 0);
                    tc::umma_commit_pair(&sm.v_empty[vst]);
                    if (j == steps - 1) tc::umma_commit_pair(&sm.o_full);
                    if (++vst == n_stages) { vst = 0; vph ^= 1; }
                    if (++buf == kScoreBufs) { buf = 0; buf_ph ^= 1; }
                    --ahead;
                }
            }
        }
    } else if (warp < kKWarp) {
        // ------------------------------------------------------------ softmax warps
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(kSoftmaxRegs));
        const int wg = warp >> 2, quad = warp & 3;                // this warpgroup takes every third step of the cluster and owns a score tile
        const int row = quad * 32 + lane;                         // row inside the tile = TMEM lane
        const uint32_t lane_addr = tbase + ((uint32_t)(quad * 32) << 16);
        const uint32_t s_addr = lane_addr + wg * 128;
        const float scale_log2 = g.scale_log2;
        const uint32_t p_bar = cluster_address(&sm.p_full[wg], 0), o_free_bar = cluster_address(&sm.o_free, 0);
        const int cube_shift = max(g.c_shift - 6, 0);             // log2(key blocks per cube), cubes of 64 tokens and more
        bool ok = true;
        int g0 = 0;                                               // steps of the pair tiles before this one
        uint32_t s_ph = 0;                                        // phase of the warpgroup's score tile
        // The rows of an epilogue leave shared memory while this warpgroup goes on; it says so after the steps of its next pair tile
        // (waiting for it at once held the next step up: 128 copies of a row each; ragged grid 743 -> 737 us).
        bool out_pending = false;
        auto release_out = [&]() {
            if (out_pending) {
                asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&sm.out_free);
                out_pending = false;
            }
        };
        for (int k = 0;; ++k) {
            const int slot = plan_slot(k);
            if (!(ok = tc::mbar_wait(&sm.plan_full[slot], plan_phase(k), abort_flag))) break;
            const int item = sm.plan_item[slot];
            if (item < 0) break;
            const Item it = item_at(item);
            const int tile_pos0 = it.pair * kPairRows + rank * 128, pr = tile_pos0 + row;   // cube-major position of the row
            const int first_local_blk = pair_first_local_blk(g, it.pair * kPairRows);
            // selection words of the row
            const uint32_t* my_mask = it.pair * 2 + rank < g.n_tiles ? tile_mask + mask_index(g, it.b, it.h, it.pair * 2 + rank, 0, row) : nullptr;
            auto load_word = [&](int w) -> uint32_t { return my_mask != nullptr && w < g.n_words ? my_mask[(size_t)w * kTileRows] : 0u; };
            int cached_w = -1;                                    // selection word in use, and the next one requested ahead
            uint32_t cached_word = 0, next_word = load_word(0);
            auto get_word = [&](int w) -> uint32_t {
                if (w != cached_w) {                              // (the same for all rows)
                    cached_word = w == cached_w + 1 ? next_word : load_word(w);
                    cached_w = w;
                    next_word = load_word(w + 1);
                }
                return cached_word;
            };
            // before the local range a block's keys are visible in whole cubes: a bit per 16 keys, from one word of the row
            auto cube_bits = [&](int kb) -> uint32_t {            // 4 bits
                if (g.c_shift >= 6) {
                    const int cube = kb >> cube_shift;
                    return ((get_word(cube >> 5) >> (cube & 31)) & 1u) ? 0xfu : 0u;
                }
                const int cube = (kb * kBlockTok) >> g.c_shift;
                const uint32_t bits = get_word(cube >> 5) >> (cube & 31);
                return g.c_shift == 5 ? ((bits & 1u) ? 3u : 0u) | ((bits & 2u) ? 0xcu : 0u) : bits & 0xfu;
            };
            const uint32_t* steps_list = reinterpret_cast<const uint32_t*>(list_at(slot));
            const int n_steps = (sm.plan_blocks[slot] + 1) / 2;   // >= 1: the local range is never empty
            const int j0 = (wg + kSoftmaxGroups - g0 % kSoftmaxGroups) % kSoftmaxGroups;   // first step of this warpgroup
            const bool last_wg = (g0 + n_steps - 1) % kSoftmaxGroups == wg;               // ... and does it take the last one?
            float m_ref = -INFINITY, l_sum = 0.f;
            // With a reference fixed in advance the row needs no maximum and no rescaling of O.  The rows of the warp take
            // this path together; otherwise the running maximum below decides.
            bool fixed_ref = false;
            if (j0 < n_steps) {
                if (!(ok = tc::mbar_wait(&sm.bound_full[k & 3], (k >> 2) & 1, abort_flag))) break;
                const float fixed = sm.fixed[k & 3][row];
                fixed_ref = __all_sync(0xffffffffu, fixed < INFINITY);
                if (fixed_ref) m_ref = fixed;
            }
            uint32_t blk_next = j0 < n_steps ? steps_list[j0] : 0u;
            for (int j = j0; j < n_steps; j += kSoftmaxGroups) {
                const int kb_a = (int)(blk_next & 0x7fffu), kb_b = (int)((blk_next >> 16) & 0x7fffu);   // the same: no second block
                const uint32_t partial = blk_next & (kPartialBlock | (kPartialBlock << 16));
                if (j + kSoftmaxGroups < n_steps) blk_next = steps_list[j + kSoftmaxGroups];
                // ---- visibility of the 128 keys of this step for this row: a bit per 16 keys, or one per key
                const bool by_cube = partial == 0u && kb_a != kb_b && kb_b < first_local_blk;
                uint32_t groups = 0, amask[4];
                if (by_cube) {
                    groups = cube_bits(kb_a);
                    groups |= cube_bits(kb_b) << 4;
                } else {
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        const int kb = hf ? kb_b : kb_a;
                        const int pk0 = kb * kBlockTok;
                        uint32_t m0 = 0, m1 = 0;
                        if (hf == 1 && kb_a == kb_b) {
                            // odd count: nothing visible
                        } else if (kb < first_local_blk) {
                            const uint32_t bits = cube_bits(kb);
                            m0 = ((bits & 1u) ? 0x0000ffffu : 0u) | ((bits & 2u) ? 0xffff0000u : 0u);
                            m1 = ((bits & 4u) ? 0x0000ffffu : 0u) | ((bits & 8u) ? 0xffff0000u : 0u);
                        } else {
                            // local range: every aligned group of 16 keys lies in one cube or in the text
                            // (C >= 16 and S_v is a multiple of C), so the rule of Eq. 3 is closed-form per group
                            const uint32_t word = pk0 < g.S_v ? get_word((pk0 >> g.c_shift) >> 5) : 0u;
                            uint32_t gm[4];
        #pragma unroll
                            for (int q4 = 0; q4 < 4; ++q4) {
                                const int pg = pk0 + q4 * 16;
                                // keys pg..pr; a video row sees the text prefix (slots S_v .. S_v + n_prefix) in full
                                const int n_causal = (pg >= g.S_v && pr < g.S_v) ? min(max(g.S_v + g.n_prefix - pg, 0), 16)
                                                                                 : min(max(pr - pg + 1, 0), 16);
                                const uint32_t causal = (1u << n_causal) - 1u;
                                const int ck = pg >> g.c_shift;
                                const bool own = pg >= g.S_v || (pr < g.S_v && ck == (pr >> g.c_shift));
                                const uint32_t picked = (pg < g.S_v && ((word >> (ck & 31)) & 1u)) ? 0xffffu : 0u;
                                gm[q4] = own ? causal : picked;
                            }
                            m0 = gm[0] | (gm[1] << 16);
                            m1 = gm[2] | (gm[3] << 16);
                        }
                        if (partial != 0u && pk0 < g.S_v && !(hf == 1 && kb_a == kb_b)) {   // empty slots of boundary cubes are never attended
                            m0 &= slot_valid[2 * kb];
                            m1 &= slot_valid[2 * kb + 1];
                        }
                        amask[hf * 2] = m0;
                        amask[hf * 2 + 1] = m1;
                    }
                }
                const int gs = g0 + j, rs = gs & (kRefSlots - 1);
                if (!(ok = tc::mbar_wait(&sm.s_full[wg], s_ph, abort_flag))) break;
                s_ph ^= 1u;
                tc::tc_fence_after_sync();
                bool rescale = false;                                     // some row of the warp moves its reference: O is scaled by its factor
                float factor = 1.f;
                if (!fixed_ref) {
                    // ---- row maximum over the visible keys; the reference moves through the warpgroups step by step
                    float mx = -INFINITY;
                    auto fold = [&](const uint32_t (&s)[32], int c) {
                        float a0 = -INFINITY, a1 = -INFINITY;
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            a0 = fmax3(a0, __uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1]));
                            a1 = fmax3(a1, __uint_as_float(s[16 + 2 * i]), __uint_as_float(s[17 + 2 * i]));
                        }
                        mx = fmax3(mx, (groups >> (2 * c)) & 1u ? a0 : -INFINITY, (groups >> (2 * c)) & 2u ? a1 : -INFINITY);
                    };
                    if (by_cube) {
                        uint32_t s0[32], s1[32];                          // the next chunk is requested before the present one is looked at
                        tc::tmem_ld_32x32(s_addr, s0);
                        tc::tmem_wait_ld_for(s0);
                        tc::tmem_ld_32x32(s_addr + 32, s1);
                        fold(s0, 0);
                        tc::tmem_wait_ld_for(s1);
                        tc::tmem_ld_32x32(s_addr + 64, s0);
                        fold(s1, 1);
                        tc::tmem_wait_ld_for(s0);
                        tc::tmem_ld_32x32(s_addr + 96, s1);
                        fold(s0, 2);
                        tc::tmem_wait_ld_for(s1);
                        fold(s1, 3);
                    } else {
#pragma unroll 1
                        for (int c = 0; c < 4; ++c) {
                            uint32_t s[32];
                            tc::tmem_ld_32x32(s_addr + c * 32, s);
                            tc::tmem_wait_ld_for(s);
                            const uint32_t am = c < 2 ? (c == 0 ? amask[0] : amask[1]) : (c == 2 ? amask[2] : amask[3]);
                            float a0 = -INFINITY, a1 = -INFINITY;
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                a0 = fmaxf(a0, ((am >> (2 * i)) & 1u) ? __uint_as_float(s[2 * i]) : -INFINITY);
                                a1 = fmaxf(a1, ((am >> (2 * i + 1)) & 1u) ? __uint_as_float(s[2 * i + 1]) : -INFINITY);
                            }
                            mx = fmax3(mx, a0, a1);
                        }
                    }
                    const float mx_x = mx * scale_log2;                   // scale > 0: max commutes with it
                    float m_prev = -INFINITY;
                    if (gs > 0 && !(ok = tc::mbar_wait(&sm.ref_done[(gs - 1) & (kRefSlots - 1)][quad], ((gs - 1) / kRefSlots) & 1, abort_flag))) break;
                    if (j > 0) m_prev = sm.ref[(gs - 1) & (kRefSlots - 1)][row];
                    // ---- lazy rescale: move the reference only when it grows by more than 2^8
                    const bool need = mx_x > m_prev + 8.f;                 // also true on the first visible key
                    const float m_new = need ? mx_x : m_prev;
                    sm.ref[rs][row] = m_new;
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&sm.ref_done[rs][quad]);
                    rescale = j > 0 && __any_sync(0xffffffffu, need);
                    if (need) factor = fast_exp2(m_prev - mx_x);          // 0 when nothing was visible before
                    // this warpgroup's sum is relative to the reference of its previous step
                    l_sum = m_ref == -INFINITY ? 0.f : l_sum * fast_exp2(m_ref - m_new);
                    m_ref = m_new;
                } else if (lane == 0) {
                    tc::mbar_arrive(&sm.ref_done[rs][quad]);              // (every step counts, so that the phases agree)
                }
                // ---- P = 2^(s*scale - m_ref) on visible keys, 0 elsewhere; bf16 pairs over the scores, 32 keys at a time.
                // The scale-subtract and the row sums use the packed fp32x2 instructions: 10 instead of 14 instructions per
                // four keys.
                const float neg_ref = -m_ref;                          // finite whenever a key is visible
                unsigned long long psA = 0ull, psB = 0ull;             // two packed pairs of partial row sums
                const unsigned long long scale2 = pack_f32x2(scale_log2, scale_log2);
                if (by_cube) {
                    auto emit = [&](const uint32_t (&s)[32], int c) {
                        uint32_t pk[16];
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            const float addend = (groups >> (2 * c + hf)) & 1u ? neg_ref : -INFINITY;   // 2^(-inf) = 0 hides the 16 keys
                            const unsigned long long add2 = pack_f32x2(addend, addend);
#pragma unroll
                            for (int i = 4 * hf; i < 4 * hf + 4; ++i) {
                                const unsigned long long x01 = fma_f32x2(pack_f32x2(__uint_as_float(s[4 * i]), __uint_as_float(s[4 * i + 1])), scale2, add2);
                                const unsigned long long x23 = fma_f32x2(pack_f32x2(__uint_as_float(s[4 * i + 2]), __uint_as_float(s[4 * i + 3])), scale2, add2);
                                float x0, x1, x2, x3;
                                unpack_f32x2(x01, x0, x1);
                                unpack_f32x2(x23, x2, x3);
                                const float p0 = fast_exp2(x0), p1 = fast_exp2(x1), p2 = fast_exp2(x2), p3 = (i % kFmaExpEvery) == kFmaExpEvery - 1 ? fma_exp2(x3) : fast_exp2(x3);
                                psA = add_f32x2(psA, pack_f32x2(p0, p1));
                                psB = add_f32x2(psB, pack_f32x2(p2, p3));
                                pk[2 * i] = pack_bf16x2(p0, p1);
                                pk[2 * i + 1] = pack_bf16x2(p2, p3);
                            }
                        }
                        tc::tmem_st_32x16(s_addr + c * 16, pk);
                    };
                    uint32_t s0[32];
                    // the scores of the next chunk are requested before the present one is worked on; chunk c of P (columns
                    // [16 c, 16 c + 16)) lies over scores that are in registers by then
                    uint32_t s1[32];
                    tc::tmem_ld_32x32(s_addr, s0);
                    tc::tmem_wait_ld_for(s0);
                    tc::tmem_ld_32x32(s_addr + 32, s1);
                    emit(s0, 0);
                    tc::tmem_wait_ld_for(s1);
                    tc::tmem_ld_32x32(s_addr + 64, s0);
                    emit(s1, 1);
                    tc::tmem_wait_ld_for(s0);
                    tc::tmem_ld_32x32(s_addr + 96, s1);
                    emit(s0, 2);
                    tc::tmem_wait_ld_for(s1);
                    emit(s1, 3);
                } else {
#pragma unroll 1
                    for (int c = 0; c < 4; ++c) {
                        uint32_t s[32], pk[16];
                        const uint32_t am = c < 2 ? (c == 0 ? amask[0] : amask[1]) : (c == 2 ? amask[2] : amask[3]);
                        tc::tmem_ld_32x32(s_addr + c * 32, s);
                        tc::tmem_wait_ld_for(s);
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const unsigned long long add2 = pack_f32x2((am >> (2 * i)) & 1u ? neg_ref : -INFINITY, (am >> (2 * i + 1)) & 1u ? neg_ref : -INFINITY);
                            float x0, x1;
                            unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), scale2, add2), x0, x1);
                            const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
                            psA = add_f32x2(psA, pack_f32x2(p0, p1));
                            pk[i] = pack_bf16x2(p0, p1);
                        }
                        tc::tmem_st_32x16(s_addr + c * 16, pk);
                    }
                }
                if (rescale) {
                    // O holds the products of all steps up to the last one, and no later one starts before this step's weights are
                    // reported: it is scaled behind them, so that the last product may complete meanwhile (before them, and with the
                    // maximum taken one chunk at a time: 2.47 for 2.16 ms with sharp queries, 16384 tokens, 28 heads, sigma 3, p 0.95)
                    if (!(ok = tc::mbar_wait(&sm.v_empty[(gs - 1) % n_stages], ((gs - 1) / n_stages) & 1, abort_flag))) break;
                    tc::tc_fence_after_sync();
#pragma unroll 1
                    for (int c = 0; c < D / 32; c += 2) {
                        uint32_t o0[32], o1[32];
                        tc::tmem_ld_32x32(lane_addr + kOCol + c * 32, o0);
                        tc::tmem_wait_ld_for(o0);
                        tc::tmem_ld_32x32(lane_addr + kOCol + c * 32 + 32, o1);
#pragma unroll
                        for (int e = 0; e < 32; ++e) o0[e] = __float_as_uint(__uint_as_float(o0[e]) * factor);
                        tc::tmem_st_32x32(lane_addr + kOCol + c * 32, o0);
                        tc::tmem_wait_ld_for(o1);
#pragma unroll
                        for (int e = 0; e < 32; ++e) o1[e] = __float_as_uint(__uint_as_float(o1[e]) * factor);
                        tc::tmem_st_32x32(lane_addr + kOCol + c * 32 + 32, o1);
                    }
                }
                tc::tmem_wait_st();
                tc::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive_cluster(p_bar);
                float a0, a1, b0, b1;
                unpack_f32x2(psA, a0, a1);
                unpack_f32x2(psB, b0, b1);
                l_sum += (a0 + a1) + (b0 + b1);
            }
            if (!ok) break;
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&sm.plan_empty[slot]);
            // ---- the sums of the three warpgroups meet in the one that took the last step; the others go on to the next pair tile
            release_out();
            const int ps = k & 1, p_ph = (k >> 1) & 1;
            if (!last_wg) {
                if (!(ok = tc::mbar_wait(&sm.part_free[ps], p_ph ^ 1, abort_flag))) break;
                sm.part_l[ps][wg][row] = l_sum;
                sm.part_m[ps][wg][row] = m_ref;
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&sm.part_full[ps]);
            } else {
                // ---- epilogue: O / l -> bf16 at the raster position of the row
                if (!(ok = tc::mbar_wait(&sm.part_full[ps], p_ph, abort_flag))) break;
                float l_fin = 0.f;                                // the reference only grows: the last step's is the largest
#pragma unroll
                for (int r = 0; r < kSoftmaxGroups; ++r) {        // in the order of the steps, whichever warpgroup took the first
                    int w = g0 % kSoftmaxGroups + r;
                    w = w >= kSoftmaxGroups ? w - kSoftmaxGroups : w;
                    const float l = w == wg ? l_sum : sm.part_l[ps][w][row], m = w == wg ? m_ref : sm.part_m[ps][w][row];
                    if (l != 0.f) l_fin += l * fast_exp2(m - m_ref);
                }
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&sm.part_free[ps]);
                const float inv = l_fin > 0.f ? 1.f / l_fin : 0.f;
                // The row goes through shared memory to its raster position as ONE 2*D-byte bulk copy: scattered 16-byte stores
                // of 32 different rows per instruction touch twice as many sectors (measured 1.7 % slower).
                if (k > 0 && !(ok = tc::mbar_wait(&sm.out_free, (k - 1) & 1, abort_flag))) break;
                if (!(ok = tc::mbar_wait(&sm.o_full, k & 1, abort_flag))) break;
                tc::tc_fence_after_sync();
                unsigned char* srow = sm.out[row];
#pragma unroll 1
                for (int c = 0; c < D / 32; ++c) {
                    uint32_t o[32];
                    tc::tmem_ld_32x32(lane_addr + kOCol + c * 32, o);
                    tc::tmem_wait_ld_for(o);
                    if (c == D / 32 - 1) {
                        tc::tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive_cluster(o_free_bar);
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        uint4 val;
                        val.x = pack_bf16x2(__uint_as_float(o[8 * e + 0]) * inv, __uint_as_float(o[8 * e + 1]) * inv);
                        val.y = pack_bf16x2(__uint_as_float(o[8 * e + 2]) * inv, __uint_as_float(o[8 * e + 3]) * inv);
                        val.z = pack_bf16x2(__uint_as_float(o[8 * e + 4]) * inv, __uint_as_float(o[8 * e + 5]) * inv);
                        val.w = pack_bf16x2(__uint_as_float(o[8 * e + 6]) * inv, __uint_as_float(o[8 * e + 7]) * inv);
                        *reinterpret_cast<uint4*>(srow + (c * 4 + e) * 16) = val;
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                if (slot_live(g, pr)) {
                    if (pair_mode != nullptr && pair_mode[(size_t)(it.b * g.Hq + it.h) * n_pairs_cap + it.pair] != 0u)
                        ml_local[(size_t)(it.b * g.Hq + it.h) * g.S_cap + pr] = make_float2(m_ref, l_fin);
                    __nv_bfloat16* dst = out + (io_row(g, it.b, pr) * g.Hq + it.h) * D;
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst), "r"(smem_u32(srow)), "n"(2 * D) : "memory");
                }
                asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
                out_pending = true;
            }
            g0 += n_steps;
        }
        release_out();
    }
    // ---------------------------------------------------------------- teardown
    __syncwarp();
    tc::tc_fence_before_sync();
    cluster_sync();                                              // nothing of the other CTA reaches this one any more
    if (tid == 0 && sm.abort_flag) atomicExch(status, 6);        // a bounded wait expired
    if (warp == kMmaWarp) tc::tmem_dealloc_pair<512>(tbase);
}

}  // namespace adaspark
