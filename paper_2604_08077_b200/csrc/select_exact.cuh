// K3, fp64 path: cube scoring (Eq. 1) and nucleus selection (Eq. 2) of single query rows on the
// CUDA cores, one CTA per row.  Every product bf16 x fp32 is exact in fp64 and the sums are fp64, so
// this path has no input-range assumption.  It serves
//   - the rows the tensor-core path (score_tc.cuh, select_nucleus.cuh) hands over: rows whose exponents are outside
//     its validated range, rows whose boundary is nearer than it can tell, rows with more equal scores at the boundary
//     than it can list (list mode: row ids from the workspace, count read on the device);
//   - every row, as the independent cross-check path of the library (all mode).
// Per row: eight lanes share a mean key (a whole line per load: a lane per key, 512 bytes apart, made every
// load touch 32 lines) and the CTA's 16 groups of lanes share the candidates, 32 at a time with the next 32 on their way; scores go to shared memory, warp 0 finds the
// boundary key in place with the radix routine of select_radix.cuh, ballots of all warps emit the row's words, and the
// words are OR-ed into the tile's union.  A list is usually short (one row in a thousand), so what counts is the
// latency of one row (a warp per row, a lane per key: 41 us for a round of 244).  What bounds the scores is the
// conversion of fp32 to fp64 (16 a clock and SM): the query's are made once and kept.  (Made anew for every key, and no key loaded
// ahead, 32 scores of a row took 2300 cycles, alone or with four CTAs on the SM, three
// quarters of a row's time.  Kernel, us, before / now: 30 rows of up to 128 candidates 17 / 9.6, 176 of 256 27 / 12.8, 542 of 768
// 70 / 34, 3245 of 1024 356 / 183, 19912 of 2048 4100 / 2340.)
#pragma once
#include "common.cuh"
#include "select_radix.cuh"

namespace adaspark {

constexpr int kExactWarps = 4;
constexpr int kExactCandCap = 256;

// rows: nullptr = all mode (row id runs over [0, n_ids)); else list mode, n_ids is ignored and
// *n_list rows are taken from rows[].  Row id = ((b*Hq + h)*n_tiles_cap + tile)*128 + r.
// dynamic shared memory: N_ld doubles.
template <int D>
__global__ void __launch_bounds__(kExactWarps * 32, 4) select_exact_kernel(
    Geom g, const __nv_bfloat16* __restrict__ q, const float* cube_keys, const int32_t* rows, const uint32_t* n_list,
    long long n_ids, uint32_t* tile_mask, uint32_t* tile_union, uint32_t* sel_bitmap, int32_t* sel_count) {
    extern __shared__ __align__(16) double exact_scores[];
    __shared__ __align__(16) unsigned long long hist[kSelHistWords + kExactCandCap];
    __shared__ unsigned long long boundary;
    __shared__ int row_total;
    launch_dependents();
    wait_for_previous_kernel();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t = lane & 7;
    const long long total = rows ? (long long)*n_list : n_ids;
    unsigned long long* keys = reinterpret_cast<unsigned long long*>(exact_scores);
    const bool all = g.top_k <= 0 && !(g.top_p < 1.0);

    for (long long idx = blockIdx.x; idx < total; idx += gridDim.x) {
        const long long id = rows ? (long long)rows[idx] : idx;
        const int r = (int)(id & (kTileRows - 1));
        const int gt_cap = (int)(id >> 7);
        const int bh = gt_cap / g.n_tiles_cap, tile = gt_cap - bh * g.n_tiles_cap;
        if (tile >= g.n_tiles || tile < g.tile_begin) continue;
        int b, h;
        g.div_Hq.divmod(bh, b, h);
        const int gk = h / g.G;
        const int pos = tile * kTileRows + r;
        const bool live = slot_live(g, pos);
        const int n = live ? n_candidates(g, pos) : 0;
        const int raster = live ? pos_to_io(g, pos) - g.pos_begin : 0;   // row of the call's tensors
        if (threadIdx.x == 0) row_total = 0;
        if (!all && n > 0) {
            // ---- scores: s[j] = scale * <q, kbar_j> in fp64; lane t of eight holds elements 32 i + 4 t .. +3
            constexpr int kPieces = D / 32, kAtOnce = 2;         // 16-byte pieces of a key per lane; keys of a lane
            const __nv_bfloat16* qsrc = q + (((size_t)b * g.S_io + raster) * g.Hq + h) * D;
            const float* kbase = cube_keys + (size_t)(b * g.Hkv + gk) * g.N * D + 4 * t;
            auto load_keys = [&](int j0, float4 (&kv)[kAtOnce][kPieces]) {
#pragma unroll
                for (int x = 0; x < kAtOnce; ++x) {
                    const float* kr = kbase + (size_t)min(j0 + 4 * x + (lane >> 3), n - 1) * D;
#pragma unroll
                    for (int i = 0; i < kPieces; ++i) kv[x][i] = *reinterpret_cast<const float4*>(kr + 32 * i);
                }
            };
            double qv[D / 8];
            auto score_keys = [&](int j0, const float4 (&kv)[kAtOnce][kPieces]) {
                double sum[kAtOnce];
#pragma unroll
                for (int x = 0; x < kAtOnce; ++x) {
                    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
#pragma unroll
                    for (int i = 0; i < kPieces; ++i) {
                        a0 = fma(qv[4 * i + 0], (double)kv[x][i].x, a0);
                        a1 = fma(qv[4 * i + 1], (double)kv[x][i].y, a1);
                        a2 = fma(qv[4 * i + 2], (double)kv[x][i].z, a2);
                        a3 = fma(qv[4 * i + 3], (double)kv[x][i].w, a3);
                    }
                    sum[x] = (a0 + a1) + (a2 + a3);
                }
#pragma unroll
                for (int o = 1; o < 8; o <<= 1)
#pragma unroll
                    for (int x = 0; x < kAtOnce; ++x) sum[x] += __shfl_xor_sync(0xffffffffu, sum[x], o);
#pragma unroll
                for (int x = 0; x < kAtOnce; ++x) {
                    const int j = j0 + 4 * x + (lane >> 3);
                    if (t == x && j < n) exact_scores[j] = sum[x] * g.scale_d;
                }
            };
            constexpr int kStep = kExactWarps * 4 * kAtOnce;
            float4 ka[kAtOnce][kPieces], kb[kAtOnce][kPieces];
            int j0 = warp * 4 * kAtOnce;
            load_keys(j0, ka);                                   // (keys beyond the last candidate: that one once more)
#pragma unroll
            for (int i = 0; i < kPieces; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) qv[4 * i + e] = (double)__bfloat162float(qsrc[32 * i + 4 * t + e]);
            for (; j0 < n; j0 += 2 * kStep) {
                load_keys(j0 + kStep, kb);
                score_keys(j0, ka);
                if (j0 + kStep >= n) break;
                load_keys(j0 + 2 * kStep, ka);
                score_keys(j0 + kStep, kb);
            }
            __syncthreads();
            if (warp == 0) {
                const unsigned long long bd = nucleus_boundary_radix<32, true>(exact_scores, n, g.top_p, g.top_k, keys, hist,
                                                                               hist + kSelHistWords, kExactCandCap, lane);
                if (lane == 0) boundary = bd;
            }
        } else if (threadIdx.x == 0) {
            boundary = 0ull;                             // every candidate is selected
        }
        __syncthreads();
        const unsigned long long bd = boundary;
        // ---- the row's words
        const bool extra = live && (sel_bitmap != nullptr || sel_count != nullptr);
        int count = 0;
        for (int w = warp; w < g.n_words; w += kExactWarps) {
            const int j = w * 32 + lane;
            const bool on = j < n && (all || keys[j] >= bd);
            const uint32_t word = __ballot_sync(0xffffffffu, on);
            count += __popc(word);
            if (lane == 0) {
                tile_mask[mask_index(g, b, h, tile, w, r)] = word;
                if (word) atomicOr(tile_union + (size_t)gt_cap * g.n_words + w, word);
                if (sel_bitmap && extra) sel_bitmap[((size_t)(b * g.Hq + h) * g.S_io + raster) * g.n_words + w] = word;
            }
        }
        if (lane == 0 && count) atomicAdd(&row_total, count);
        __syncthreads();                                 // the scores are free for the next row
        if (sel_count && threadIdx.x == 0 && extra) sel_count[(size_t)(b * g.Hq + h) * g.S_io + raster] = row_total;
    }
}

}  // namespace adaspark
