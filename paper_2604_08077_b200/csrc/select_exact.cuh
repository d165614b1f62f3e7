// K3, fp64 path: cube scoring (Eq. 1) and nucleus selection (Eq. 2) of single query rows on the
// CUDA cores, one CTA per row.  Every product bf16 x fp32 is exact in fp64 and the sums are fp64, so
// this path has no input-range assumption.  It serves
//   - the rows the tensor-core path (score_tc.cuh, select_nucleus.cuh) hands over: rows whose exponents are outside
//     its validated range, rows whose boundary is nearer than it can tell, rows with more equal scores at the boundary
//     than it can list (list mode: row ids from the workspace, count read on the device);
//   - every row, as the independent cross-check path of the library (all mode).
// Per row: four lanes share a mean key (64 consecutive bytes per load: a lane per key, 512 bytes apart, made every
// load touch 32 lines) and the CTA's 32 quads share the candidates; scores go to shared memory, warp 0 finds the
// boundary key in place with the radix routine of select_radix.cuh, ballots of all warps emit the row's words, and the
// words are OR-ed into the tile's union.  A list is usually short (one row in a thousand), so what counts is the
// latency of one row: 13 us for a dozen rows (a warp per row, a lane per key: 41 us for a round of 244).
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
__global__ void __launch_bounds__(kExactWarps * 32) select_exact_kernel(
    Geom g, const __nv_bfloat16* __restrict__ q, const float* cube_keys, const int32_t* rows, const uint32_t* n_list,
    long long n_ids, uint32_t* tile_mask, uint32_t* tile_union, uint32_t* sel_bitmap, int32_t* sel_count) {
    extern __shared__ __align__(16) double exact_scores[];
    __shared__ __align__(16) unsigned long long hist[kSelHistWords + kExactCandCap];
    __shared__ unsigned long long boundary;
    __shared__ int row_total;
    launch_dependents();
    wait_for_previous_kernel();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t = lane & 3;
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
            // ---- scores: s[j] = scale * <q, kbar_j> in fp64; lane t of a quad holds elements 16 i + 4 t .. +3
            const __nv_bfloat16* qsrc = q + (((size_t)b * g.S_io + raster) * g.Hq + h) * D;
            float qv[D / 4];
#pragma unroll
            for (int i = 0; i < D / 16; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) qv[4 * i + e] = __bfloat162float(qsrc[16 * i + 4 * t + e]);
            const float* kbase = cube_keys + (size_t)(b * g.Hkv + gk) * g.N * D + 4 * t;
            for (int j0 = warp * 8; j0 < n; j0 += kExactWarps * 8) {
                const int j = j0 + (lane >> 2);
                const float* kr = kbase + (size_t)min(j, n - 1) * D;
                float4 kv[D / 16];
#pragma unroll
                for (int i = 0; i < D / 16; ++i) kv[i] = *reinterpret_cast<const float4*>(kr + 16 * i);
                double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
#pragma unroll
                for (int i = 0; i < D / 16; ++i) {
                    a0 = fma((double)qv[4 * i + 0], (double)kv[i].x, a0);
                    a1 = fma((double)qv[4 * i + 1], (double)kv[i].y, a1);
                    a2 = fma((double)qv[4 * i + 2], (double)kv[i].z, a2);
                    a3 = fma((double)qv[4 * i + 3], (double)kv[i].w, a3);
                }
                double sum = (a0 + a1) + (a2 + a3);
                sum += __shfl_xor_sync(0xffffffffu, sum, 1);
                sum += __shfl_xor_sync(0xffffffffu, sum, 2);
                if (t == 0 && j < n) exact_scores[j] = sum * g.scale_d;
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
