// K4c: attention of calls in which whole cubes of 128 tokens and more may be gathered (attn_gather.cuh).
//
// The kernel of attn_prefill_tc.cuh (CTA pairs, roles, TMEM, barriers: see there) in two forms:
//   attn_cubes_tc_kernel<D, false>  pair tiles.  A gathered pair visits its local range alone; its rows' outputs leave in fp32 for the
//                                   merge (their sums are held in 32 bits on the union path too), with their references
//   attn_cubes_tc_kernel<D, true>   gathered rows: a "pair tile" is an item of up to 256 rows of one (batch, kv head) that selected one
//                                   cube, its keys are the cube's, all of them visible.  The softmax warps copy the rows of Q two items
//                                   ahead; what leaves is the normalised partial output (fp32) and (reference exponent, sum) of
//                                   every entry.  Items are short (C / 128 steps), so what bounds it are the steps between items: 5500
//                                   to 7000 cycles for one of two steps, 2100 of them tensor core
// It is a source of its own because it costs the other kernel registers: both in one template ran 16384 tokens 1.5 %, ragged grids
// 2 % slower (softmax warps of 144 registers, which spill either way).  What a call of 256-token cubes gains by it: 24576 tokens,
// 16 heads, p 0.7 2.15 -> 1.78 ms; 65536, 28 heads 25.5 -> 17.1.
#pragma once
#include "attn_prefill_tc.cuh"

namespace adaspark {

template <int D, bool kGathered>
struct CubesSmem {
    static constexpr int kQSlots = kGathered ? 3 : 2, kStages = max_kv_stages(D) - (kGathered ? 1 : 0);
    __nv_bfloat16 q[kQSlots][D / 64][128][64];        // [pair tile % kQSlots][d panel][row][64 d]
    __nv_bfloat16 kv[2 * kStages][64 * D];            // a K tile ([d panel][key of this CTA's block][64 d]) or a V^T tile
                                                      // ([block][this CTA's half of d][64 keys]) each
    unsigned char out[128][2 * D + 16];               // output rows (16 bytes of padding spread the banks)
    float ref[kRefSlots][128];                        // running reference of a row after a step
    float part_l[2][kSoftmaxGroups][128], part_m[2][kSoftmaxGroups][128];   // sums and references of the warpgroups
    float fixed[4][128];                              // reference of a row fixed in advance, infinite if it is not
    uint64_t q_full[kQSlots], q_peer[kQSlots], q_empty[kQSlots], k_full[kStages], k_empty[kStages], v_full[kStages], v_empty[kStages];
    uint64_t s_full[kScoreBufs], p_full[kScoreBufs], ref_done[kRefSlots][4], o_full[4], o_free;
    // (A warpgroup may be three gathered items of one step ahead of another: what it waits for must not be two uses of a barrier
    // away, which its phase could not tell from none.)
    uint64_t plan_full[4], plan_empty[4], bound_full[4], part_full[2], part_free[2], out_free[4];
    int plan_blocks[4], plan_item[4];                 // visited key blocks; pair tile, -1: no more
    uint4 plan_rows[4];                               // gathered: (batch, kv head), first entry, entries
    uint32_t entries[kGathered ? 4 : 1][128];         // ... and the entries of this CTA's rows
    uint64_t item_full[8];                            // (CTA 1) CTA 0 has drawn the pair tile
    int next_item[8];
    uint32_t tmem_base;
    int abort_flag;
    uint16_t list[2][kBlockListShort];                // the visited key blocks in order
};

// Buffers of the query-gather path for this kernel.
struct GatherTiles {
    const uint4* items;          // (column, first entry, entries, 0)
    const uint32_t* ctrl;        // [0] 0: none, [1] items
    const uint32_t* entries;     // token of the call's tensors | head in group << 21
    float* part_o;               // [entries][D]; (not gathered: the local range of the rows of gathered pairs, [place][256][D])
    const uint32_t* pair_place;  // (not gathered) of a gathered pair, in the order of that buffer
    float2* part_ml;
    int n_cols;                  // columns (cubes) of a list set
};
constexpr uint32_t kEntryPosMask = 0x1fffffu;   // 21 bits of token index (a sequence holds at most 2^21 rows)

template <int D, bool kGathered>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTcThreads, 1) attn_cubes_tc_kernel(
    Geom g, const __grid_constant__ CUtensorMap tmQ, const __nv_bfloat16* __restrict__ q, const __grid_constant__ CUtensorMap tmK,
    const __grid_constant__ CUtensorMap tmV, const uint32_t* tile_mask, const uint32_t* tile_union, const uint32_t* slot_valid,
    const uint32_t* pair_mode, int n_pairs_cap, float2* ml_local, const GatherTiles gt, float* row_ref, const uint32_t* key_norm2_bits,
    __nv_bfloat16* out, uint32_t* next_pair_tile, unsigned long long* executed_blocks, uint32_t* max_tile_blocks, int32_t* status) {
    extern __shared__ unsigned char tc_smem_raw[];
    using Smem = CubesSmem<D, kGathered>;
    Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~(uintptr_t)1023);
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
    const int n_stages = kGathered ? Smem::kStages : kv_stages(D, g.n_kv_blocks_cap);
    const bool long_list = !kGathered && g.n_kv_blocks_cap > kBlockListShort;
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
    // slot of pair tile k's plan and phase of its barriers: two block lists, one if they are long, four of the few blocks of a cube
    auto plan_slot = [&](int k) -> int { return kGathered ? k & 3 : long_list ? 0 : k & 1; };
    auto plan_phase = [&](int k) -> uint32_t { return (uint32_t)((kGathered ? k >> 2 : long_list ? k : k >> 1) & 1); };
    auto list_at = [&](int slot) -> uint16_t* {
        return kGathered ? sm.list[0] + slot * 16 : long_list ? reinterpret_cast<uint16_t*>(&sm.kv[2 * n_stages][0]) : sm.list[slot];
    };

    // slot of its Q tile
    auto q_slot = [&](int k) -> int { return kGathered ? k % 3 : k & 1; };
    auto q_phase = [&](int k) -> uint32_t { return (uint32_t)((kGathered ? k / 3 : k >> 1) & 1); };

    // ---------------------------------------------------------------- set-up
    if (!kGathered) launch_dependents();                        // (the merge: its CTAs start when this grid ends, see its launch)
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&sm.part_full[i], (kSoftmaxGroups - 1) * 4);
            tc::mbar_init(&sm.part_free[i], 4);
        }
        for (int i = 0; i < Smem::kQSlots; ++i) {
            tc::mbar_init(&sm.q_full[i], kGathered ? kSoftmaxGroups * 4 : 1);
            tc::mbar_init(&sm.q_peer[i], 1);
            tc::mbar_init(&sm.q_empty[i], 1);
        }
        for (int i = 0; i < Smem::kStages; ++i) {
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
            tc::mbar_init(&sm.plan_full[i], 1);
            tc::mbar_init(&sm.plan_empty[i], 3 + kSoftmaxGroups * 4);
            tc::mbar_init(&sm.bound_full[i], 1);
            tc::mbar_init(&sm.o_full[i], 1);
            tc::mbar_init(&sm.out_free[i], 4);
            tc::mbar_init(&sm.item_full[i], 1);
            tc::mbar_init(&sm.item_full[4 + i], 1);
            for (int w = 0; w < 4; ++w) tc::mbar_init(&sm.ref_done[i][w], 1);
        }
        tc::mbar_init(&sm.o_free, 8);
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
    const int n_items = kGathered ? (gt.ctrl[0] ? (int)gt.ctrl[1] : 0) : (n_pairs - g.pos_begin / kPairRows) * n_hb;

    if (warp >= kKWarp) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kHelperRegs));
    if (warp == kPlanWarp) {
        // ------------------------------------------------------------ planner
        unsigned long long blocks_sum = 0;
        uint32_t blocks_max = 0;
        bool ok = true;
        auto bounds = [&](int k, int bkv, float* row_ref_at, int row_pos0) -> bool {
            if constexpr (kGathered) {                            // the references that the rows' local range was given
                const uint4 d = sm.plan_rows[plan_slot(k)];
                const size_t base = (size_t)(bkv / g.Hkv) * g.S_io * g.Hq + (bkv % g.Hkv) * g.G;
                float ref[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const uint32_t e = sm.entries[k & 3][x * 32 + lane];
                    ref[x] = rank * 128 + x * 32 + lane < (int)d.z ? row_ref[base + (size_t)(e & kEntryPosMask) * g.Hq + ((e >> 21) & 15u)] : 0.f;
                }
#pragma unroll
                for (int x = 0; x < 4; ++x) sm.fixed[k & 3][x * 32 + lane] = ref[x];
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&sm.bound_full[k & 3]);
                return true;
            }
            // Bound of a row's scores: |s| <= |q| |k| for every key; the largest key norm of the head comes from the re-layout
            // kernel (none when not every attended key went through this call's re-layout).
            const int qs = q_slot(k);
            const unsigned char* qt = reinterpret_cast<const unsigned char*>(&sm.q[qs][0][0][0]);
            {
                if (!tc::mbar_wait(&sm.q_full[qs], q_phase(k), abort_flag)) return false;
                const float k2 = key_norm2_bits != nullptr ? __uint_as_float(key_norm2_bits[bkv]) : INFINITY;
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
            if (!kGathered && row_ref_at != nullptr) {                          // for the gathered cubes of these rows
#pragma unroll 1
                for (int row = lane; row < 128; row += 32)
                    if (slot_live(g, row_pos0 + row)) row_ref_at[io_row(g, bkv / g.Hkv, row_pos0 + row) * g.Hq] = sm.fixed[k & 3][row];
            }
            return true;
        };
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
                    if (!(ok = tc::mbar_wait(&sm.item_full[(k - 1) & 7], ((k - 1) >> 3) & 1, abort_flag))) break;
                    asm volatile("fence.acq_rel.cluster;\n" ::: "memory");
                    i = *(volatile int*)&sm.next_item[(k - 1) & 7];
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
            const int item = i, qs = q_slot(k);
            uint16_t* list = list_at(slot);
            unsigned char* qt = reinterpret_cast<unsigned char*>(&sm.q[qs][0][0][0]);
            int n_needed = 0, bkv, row_pos0 = 0;                  // visited key blocks; (batch, kv head)
            float* row_ref_at = nullptr;                          // references of the rows of a pair whose cubes are gathered whole
            if constexpr (kGathered) {
                const uint4 d = gt.items[item];
                uint32_t ent[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) ent[x] = rank * 128 + x * 32 + lane < (int)d.z ? gt.entries[d.y + (uint32_t)(rank * 128 + x * 32 + lane)] : 0u;
                bkv = (int)(d.x / (uint32_t)gt.n_cols) % (g.B * g.Hkv);
                n_needed = g.C / kBlockTok;                       // (even)
                const int kb0 = (int)(d.x % (uint32_t)gt.n_cols) * n_needed;
                for (int x = lane; x < n_needed; x += 32)
                    list[x] = (uint16_t)((uint32_t)(kb0 + x) | (g.ragged && block_partial(g, kb0 + x) ? kPartialBlock : 0u));
                if (lane == 0) sm.plan_rows[slot] = make_uint4((uint32_t)bkv, d.y, d.z, 0u);
                if (rank == 0 && lane == 0 && drawn < n_items) prefetch_l1(gt.items + drawn);
#pragma unroll
                for (int x = 0; x < 4; ++x) sm.entries[slot][x * 32 + lane] = ent[x];
            } else {
                const Item it = item_at(item);
                bkv = it.b * g.Hkv + it.gk;
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
                row_pos0 = tile_pos0;
                const bool gathered = pair_mode != nullptr && pair_mode[(size_t)(it.b * g.Hq + it.h) * n_pairs_cap + it.pair] != 0u;
                if (gathered) row_ref_at = row_ref + it.h;
                // The Q tile does not wait for the plan.  It comes straight from the caller's tensor [B, S_io, Hq, D]: the video
                // rows of a tile are whole boxes of a cube's window (or the cubes themselves, below 128 tokens) in the
                // (head x d, x, y, t, batch) view of that tensor, which one 5-D TMA load per box and 64-element panel turns into
                // cube-major rows (a coordinate beyond the grid reads zeros: the empty slots of a boundary cube); text rows and
                // the slots beyond the sequence, a few tiles per head, are copied by the warp's lanes.
                if (!(ok = tc::mbar_wait(&sm.q_empty[qs], q_phase(k) ^ 1u, abort_flag))) break;
                const int rpb = min(g.C, 128);                            // rows per box
                const int n_vid = max(0, min(tile_pos0 + 128, g.S_v) - tile_pos0);  // video slots of the tile (a multiple of rpb or of C)
                for (int idx = lane; idx < (128 - n_vid) * (D / 8); idx += 32) {
                    const int row = n_vid + idx / (D / 8), c = idx % (D / 8);
                    const int pos = tile_pos0 + row;
                    unsigned char* dst = qt + (c >> 3) * (128 * 128) + sw128(row, c & 7);
                    if (pos < g.S) cp_async_16(dst, q + (io_row(g, it.b, pos) * g.Hq + it.h) * D + c * 8);
                    else *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
                }
                // all copies under way at once
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
                const uint32_t* un0 = tile_union + ((size_t)(it.b * g.Hq + it.h) * g.n_tiles_cap + it.pair * 2) * g.n_words;
                const uint32_t* un1 = it.pair * 2 + 1 < g.n_tiles ? un0 + g.n_words : un0;
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
            }
            __syncwarp();
            if (lane == 0) {
                if (n_needed & 1) list[n_needed] = list[n_needed - 1];   // odd count: the last block once more, masked
                sm.plan_blocks[slot] = n_needed;
                sm.plan_item[slot] = item;
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&sm.plan_full[slot]);
            if (rank == 0) {                                      // (CTA 1 has read what the slot held: it has worked on pair tile k - 4)
                if (lane == 0) {
                    asm volatile("st.shared::cluster.u32 [%0], %1;\n" ::"r"(cluster_address(&sm.next_item[k & 7], 1)), "r"(drawn) : "memory");
                    tc::mbar_arrive_release_cluster(cluster_address(&sm.item_full[k & 7], 1));
                }
                i = drawn;
            }
            blocks_sum += (unsigned long long)(2 * n_needed);
            blocks_max = max(blocks_max, (uint32_t)n_needed);
            if (!(ok = bounds(k, bkv, row_ref_at, row_pos0))) break;
        }
        if (rank == 0 && lane == 0 && ok) {
            atomicAdd(executed_blocks, blocks_sum);
            if (!kGathered) atomicMax(max_tile_blocks, blocks_max);
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
                int bkv;
                if constexpr (kGathered) {
                    bkv = (int)sm.plan_rows[slot].x;
                } else {
                    const Item it = item_at(sm.plan_item[slot]);
                    bkv = it.b * g.Hkv + it.gk;
                }
                const int row0 = is_v ? bkv * g.n_kv_blocks_cap * D + rank * (D / 2) : bkv * g.S_cap;
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
                if (!tc::mbar_wait(&sm.q_full[q_slot(k)], q_phase(k), abort_flag)) break;
                asm volatile("fence.acq_rel.cluster;\n" ::: "memory");
                tc::mbar_arrive_cluster(cluster_address(&sm.q_peer[q_slot(k)], 0));
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
            // whose rows wait for these products (see the header of attn_prefill_tc.cuh).
            auto next_scores = [&](bool must) -> bool {
                if (s_left == 0) {
                    if (ended) return false;
                    const int kn = ks + 1, slot = plan_slot(kn);
                    auto there = [&](uint64_t* bar, uint32_t phase) -> bool { return must ? (ok = tc::mbar_wait(bar, phase, abort_flag)) : tc::mbar_test(bar, phase); };
                    if (!there(&sm.plan_full[slot], plan_phase(kn))) return false;
                    if ((ended = sm.plan_item[slot] < 0)) return false;
                    if (!there(&sm.q_full[q_slot(kn)], q_phase(kn)) || !there(&sm.q_peer[q_slot(kn)], q_phase(kn))) return false;
                    ks = kn;
                    n_steps2 = n_steps1;
                    n_steps1 = n_steps0;
                    s_left = n_steps0 = (sm.plan_blocks[slot] + 1) / 2;
                    tc::mbar_arrive(&sm.plan_empty[slot]);
                }
                if (!(ok = tc::mbar_wait(&sm.k_full[kst], kph, abort_flag))) return false;
                tc::tc_fence_after_sync();
                const uint32_t qa = q_lo0 + q_slot(ks) * kQSlotStep, kb = k_lo0 + kst * kStageStep, dst = tb + sbuf * 128;
#pragma unroll
                for (int x = 0; x < kQKSteps; ++x)
                    tc::umma_ss_pair(dst, tc::smem_desc_from_halves(qa + (x >> 2) * kQPanelStep + (x & 3) * kKStep, tc::kSmemDescHiSw128),
                                     tc::smem_desc_from_halves(kb + (x >> 2) * kKPanelStep + (x & 3) * kKStep, tc::kSmemDescHiSw128), kIdescS, x > 0);
                tc::umma_commit_pair(&sm.s_full[sbuf]);
                tc::umma_commit_pair(&sm.k_empty[kst]);
                if (--s_left == 0) tc::umma_commit_pair(&sm.q_empty[q_slot(ks)]);
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
                    if (j == steps - 1) tc::umma_commit_pair(&sm.o_full[k & 3]);
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
        // Gathered rows of Q: the softmax warps copy them, two items ahead (a warp of its own took 7000 cycles an item).  A row is
        // 2 D bytes; consecutive lanes copy consecutive 16-byte pieces, so that an instruction covers whole rows.
        int n_fetched = 0;                                        // items whose rows have been requested; the last one's end
        bool more_items = kGathered;
        auto fetch = [&]() -> bool {
            constexpr int kPieces = D / 8, kRowsPerPass = 32 / kPieces, kWarps = kSoftmaxGroups * 4, kTurns = (128 / kRowsPerPass + kWarps - 1) / kWarps;
            if (more_items) {
                const int k = n_fetched, slot = plan_slot(k);
                if (!tc::mbar_wait(&sm.plan_full[slot], plan_phase(k), abort_flag)) return false;
                if (sm.plan_item[slot] < 0) {
                    more_items = false;
                } else {
                    const uint4 d = sm.plan_rows[slot];
                    const int piece = lane % kPieces, rsub = lane / kPieces, n = min(max((int)d.z - rank * 128, 0), 128);
                    const int b = (int)d.x / g.Hkv, head0 = ((int)d.x - b * g.Hkv) * g.G;
                    uint32_t ent[kTurns];
#pragma unroll
                    for (int t = 0; t < kTurns; ++t) {
                        const int r = (t * kWarps + warp) * kRowsPerPass + rsub;
                        ent[t] = r < n ? sm.entries[slot][r] : 0u;
                    }
                    if (!tc::mbar_wait(&sm.q_empty[q_slot(k)], q_phase(k) ^ 1u, abort_flag)) return false;
                    unsigned char* qbase = reinterpret_cast<unsigned char*>(&sm.q[q_slot(k)][0][0][0]) + (piece >> 3) * (128 * 128);
                    const __nv_bfloat16* src0 = q + ((size_t)b * g.S_io * g.Hq + head0) * D + piece * 8;
#pragma unroll
                    for (int t = 0; t < kTurns; ++t) {
                        const int r = (t * kWarps + warp) * kRowsPerPass + rsub;
                        unsigned char* dst = qbase + sw128(r, piece & 7);
                        if (r < n) cp_async_16(dst, src0 + ((size_t)(ent[t] & kEntryPosMask) * g.Hq + ((ent[t] >> 21) & 15u)) * D);
                        else if (r < 128) *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
                    }
                    ++n_fetched;
                }
            }
            cp_async_commit();
            return true;
        };
        auto landed = [&](int k) {                                // this warp's share of item k's rows
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&sm.q_full[q_slot(k)]);
        };
        if constexpr (kGathered) {
            ok = fetch() && fetch();
            cp_async_wait<0>();
            if (n_fetched > 0) landed(0);
            if (n_fetched > 1) landed(1);
        }
        // The rows of an epilogue leave shared memory while this warpgroup goes on; it says so after the steps of its next pair tile
        // (waiting for it at once held the next step up for thousands of cycles: 128 copies of a row each).
        int out_pending = -1;                                     // the pair tile whose rows those are
        auto release_out = [&]() {
            if (out_pending >= 0) {
                asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&sm.out_free[out_pending & 3]);
                out_pending = -1;
            }
        };
        for (int k = 0; ok; ++k) {
            const int slot = plan_slot(k);
            if (!(ok = tc::mbar_wait(&sm.plan_full[slot], plan_phase(k), abort_flag))) break;
            const int item = sm.plan_item[slot];
            if (item < 0) break;
            if constexpr (kGathered) {
                if (!(ok = fetch())) break;                       // item k + 2
            }
            const Item it = kGathered ? Item{0, 0, 0, 0} : item_at(item);
            const int tile_pos0 = it.pair * kPairRows + rank * 128, pr = tile_pos0 + row;   // cube-major position of the row
            const int first_local_blk = pair_first_local_blk(g, it.pair * kPairRows);
            // selection words of the row
            const uint32_t* my_mask = !kGathered && it.pair * 2 + rank < g.n_tiles ? tile_mask + mask_index(g, it.b, it.h, it.pair * 2 + rank, 0, row) : nullptr;
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
            const uint4 rows = kGathered ? sm.plan_rows[slot] : make_uint4(0u, 0u, 0u, 0u);
            const uint32_t* steps_list = reinterpret_cast<const uint32_t*>(list_at(slot));
            const int n_steps = (sm.plan_blocks[slot] + 1) / 2;   // >= 1: the local range is never empty
            const int j0 = (wg + kSoftmaxGroups - g0 % kSoftmaxGroups) % kSoftmaxGroups;   // first step of this warpgroup
            const bool last_wg = (g0 + n_steps - 1) % kSoftmaxGroups == wg;               // ... and does it take the last one?
            float m_ref = -INFINITY, l_sum = 0.f;
            // With a reference fixed in advance the row needs no maximum and no rescaling of O.  The rows of the warp take this
            // path together; otherwise the running maximum below decides (gathered: for the rows without one, so that no row
            // depends on its neighbours in the list, which come in any order).
            bool fixed_ref = false, own_fixed = false;
            if (j0 < n_steps) {
                if (!(ok = tc::mbar_wait(&sm.bound_full[k & 3], (k >> 2) & 1, abort_flag))) break;
                const float fixed = sm.fixed[k & 3][row];
                own_fixed = fixed < INFINITY;
                fixed_ref = __all_sync(0xffffffffu, own_fixed);
                if (kGathered ? own_fixed : fixed_ref) m_ref = fixed;
            }
            uint32_t blk_next = j0 < n_steps ? steps_list[j0] : 0u;
            for (int j = j0; j < n_steps; j += kSoftmaxGroups) {
                const int kb_a = (int)(blk_next & 0x7fffu), kb_b = (int)((blk_next >> 16) & 0x7fffu);   // the same: no second block
                const uint32_t partial = blk_next & (kPartialBlock | (kPartialBlock << 16));
                if (j + kSoftmaxGroups < n_steps) blk_next = steps_list[j + kSoftmaxGroups];
                // ---- visibility of the 128 keys of this step for this row: a bit per 16 keys, or one per key
                const bool by_cube = partial == 0u && (kGathered || (kb_a != kb_b && kb_b < first_local_blk));
                uint32_t groups = 0, amask[4];
                if (by_cube) {
                    if constexpr (kGathered) groups = 0xffu;
                    else {
                        groups = cube_bits(kb_a);                 // (in this order: the words of a row are walked forwards)
                        groups |= cube_bits(kb_b) << 4;
                    }
                } else {
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        const int kb = hf ? kb_b : kb_a;
                        const int pk0 = kb * kBlockTok;
                        uint32_t m0 = 0, m1 = 0;
                        if (kGathered) {
                            m0 = m1 = 0xffffffffu;                // the rows selected the cube
                        } else if (hf == 1 && kb_a == kb_b) {
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
                        if (partial != 0u && pk0 < g.S_v && (kGathered || !(hf == 1 && kb_a == kb_b))) {   // empty slots of boundary cubes are never attended
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
                    if (!kGathered && by_cube) {
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
                            if (by_cube) { fold(s, c); continue; }
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
                    float m_prev = kGathered && own_fixed ? m_ref : -INFINITY;
                    if (gs > 0 && !(ok = tc::mbar_wait(&sm.ref_done[(gs - 1) & (kRefSlots - 1)][quad], ((gs - 1) / kRefSlots) & 1, abort_flag))) break;
                    if (j > 0) m_prev = sm.ref[(gs - 1) & (kRefSlots - 1)][row];
                    // ---- lazy rescale: move the reference only when it grows by more than 2^8
                    const bool need = !(kGathered && own_fixed) && mx_x > m_prev + 8.f;                 // also true on the first visible key
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
                    // reported: it is scaled behind them, so that the last product may complete meanwhile
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
            release_out();
            if constexpr (kGathered) {
                cp_async_wait<0>();
                if (k + 2 < n_fetched) landed(k + 2);
            }
            // ---- the sums of the three warpgroups meet in the one that took the last step; the others go on to the next pair tile.
            // Of gathered items, which are short and all of the same length, only those that took a step have a part (one without
            // may still be in the epilogue before); with one step there is nothing to meet.
            const int ps = k & 1, p_ph = (k >> 1) & 1;
            if (!last_wg && (!kGathered || j0 < n_steps)) {
                if (!(ok = tc::mbar_wait(&sm.part_free[ps], p_ph ^ 1, abort_flag))) break;
                sm.part_l[ps][wg][row] = l_sum;
                sm.part_m[ps][wg][row] = m_ref;
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&sm.part_full[ps]);
            } else if (!kGathered || last_wg) {
                // ---- epilogue: O / l -> bf16 at the raster position of the row
                const bool alone = kGathered && n_steps == 1;
                if (kGathered && n_steps == 2 && lane == 0) tc::mbar_arrive(&sm.part_full[ps]);   // for the one without a step
                if (!alone && !(ok = tc::mbar_wait(&sm.part_full[ps], p_ph, abort_flag))) break;
                float l_fin = 0.f;                                // the reference only grows: the last step's is the largest
#pragma unroll
                for (int r = 0; r < kSoftmaxGroups; ++r) {        // in the order of the steps, whichever warpgroup took the first
                    int w = g0 % kSoftmaxGroups + r;
                    w = w >= kSoftmaxGroups ? w - kSoftmaxGroups : w;
                    const float l = w == wg ? l_sum : sm.part_l[ps][w][row], m = w == wg ? m_ref : sm.part_m[ps][w][row];
                    if ((!kGathered || r < n_steps) && l != 0.f) l_fin += l * fast_exp2(m - m_ref);
                }
                __syncwarp();
                if (!alone && lane == 0) tc::mbar_arrive(&sm.part_free[ps]);
                const float inv = l_fin > 0.f ? 1.f / l_fin : 0.f;
                // The row goes through shared memory to its raster position as ONE 2*D-byte bulk copy: scattered 16-byte stores
                // of 32 different rows per instruction touch twice as many sectors (measured 1.7 % slower).
                if (k > 0 && !(ok = tc::mbar_wait(&sm.out_free[(k - 1) & 3], ((k - 1) >> 2) & 1, abort_flag))) break;
                if (!(ok = tc::mbar_wait(&sm.o_full[k & 3], (k >> 2) & 1, abort_flag))) break;
                tc::tc_fence_after_sync();
                unsigned char* srow = sm.out[row];
                // The rows of a warp as one contiguous piece of fp32 partial results: 64 columns at a time through shared memory, written by
                // the warp in whole lines and past the caches' regular lines (read once, by the merge).
                auto store_partials = [&](float* dst, int n_rows) {
                    constexpr int kCols = D == 128 ? 64 : 32;     // what a row of the staging holds in fp32
#pragma unroll 1
                    for (int c0 = 0; c0 < D; c0 += kCols) {
#pragma unroll
                        for (int c = 0; c < kCols; c += 32) {
                            uint32_t o[32];
                            tc::tmem_ld_32x32(lane_addr + kOCol + c0 + c, o);
                            tc::tmem_wait_ld_for(o);
                            if (c0 + c == D - 32) {
                                tc::tc_fence_before_sync();
                                __syncwarp();
                                if (lane == 0) tc::mbar_arrive_cluster(o_free_bar);
                            }
#pragma unroll
                            for (int e = 0; e < 8; ++e)
                                *reinterpret_cast<float4*>(srow + (c + 4 * e) * 4) = make_float4(__uint_as_float(o[4 * e]) * inv, __uint_as_float(o[4 * e + 1]) * inv,
                                                                                                __uint_as_float(o[4 * e + 2]) * inv, __uint_as_float(o[4 * e + 3]) * inv);
                        }
                        __syncwarp();
#pragma unroll 4
                        for (int x = lane; x < n_rows * (kCols / 4); x += 32) {
                            const int r = x / (kCols / 4), p = x % (kCols / 4);
                            __stcs(reinterpret_cast<float4*>(dst + (size_t)r * D + c0) + p, *reinterpret_cast<const float4*>(&sm.out[quad * 32 + r][p * 16]));
                        }
                        __syncwarp();
                    }
                    if (lane == 0) tc::mbar_arrive(&sm.out_free[k & 3]);
                };
                const size_t pair_slot = (size_t)(it.b * g.Hq + it.h) * n_pairs_cap + it.pair;
                const bool gathered = !kGathered && pair_mode != nullptr && pair_mode[pair_slot] != 0u;
                if constexpr (kGathered) {
                    const int r0 = rank * 128 + quad * 32, n_rows = min(max((int)rows.z - r0, 0), 32);
                    if (lane < n_rows) __stcs(gt.part_ml + rows.y + r0 + lane, make_float2(m_ref, l_fin));
                    store_partials(gt.part_o + (size_t)(rows.y + r0) * D, n_rows);
                } else if (gathered) {               // the local range of rows whose cubes are gathered whole
                    if (slot_live(g, pr)) ml_local[(size_t)(it.b * g.Hq + it.h) * g.S_cap + pr] = make_float2(m_ref, l_fin);
                    const size_t at = (size_t)gt.pair_place[pair_slot] * kPairRows + rank * 128 + quad * 32;
                    store_partials(gt.part_o + at * D, min(max(g.S_cap - (tile_pos0 + quad * 32), 0), 32));
                } else {
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
                        const size_t at = io_row(g, it.b, pr) * g.Hq + it.h;
                        __nv_bfloat16* dst = out + at * D;
                        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst), "r"(smem_u32(srow)), "n"(2 * D) : "memory");
                    }
                    asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
                    out_pending = k;
                }
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
