// K5 / K7: decode step = one new text token per sequence (text-token rule after Eq. 3).
//
//   decode_select_plan_kernel  per (b, kv head), a cluster of eight CTAs: appends the new token's K / V to the
//                              cube-major caches, then Eq. 1 scores of all heads of the GQA group against
//                              the N cube keys (fp64 tensor op, the cube keys are read once per
//                              group), Eq. 2 per head, then the list of 64-key blocks to visit =
//                              blocks holding a cube selected by any head of the group + text blocks
//   decode_combine_kernel      log-sum-exp merge of the split-KV partials
// The split-KV attention kernel itself is in decode_splitkv.cuh.  The three kernels of a step are launched so that
// each starts while the one before still runs (programmatic dependent launch): it sets itself up and waits.
#pragma once
#include "common.cuh"
#include "select_radix.cuh"

namespace adaspark {

// Appends the new token's K / V of one (batch, kv head) to the cube-major caches at text slot
// text_len[b] (the V cache holds every 64-position block transposed).  A text_len outside
// [0, n_text_max] writes nothing (the caller reports status 1).  Called by all threads of a CTA.
__device__ __forceinline__ void decode_append(const Geom& g, int b, int gk, const __nv_bfloat16* k_new,
                                              const __nv_bfloat16* v_new, __nv_bfloat16* k_cube, __nv_bfloat16* v_cube,
                                              const int32_t* text_len) {
    const int tl = text_len[b];
    if (tl < 0 || tl > g.n_text) return;             // g.n_text = n_text_max of the partition
    const int pos = g.S_v + tl, blk = pos / kBlockTok, tok = pos % kBlockTok;
    for (int d = threadIdx.x; d < g.D; d += blockDim.x) {
        const size_t src = ((size_t)b * g.Hkv + gk) * g.D + d;
        k_cube[((size_t)(b * g.Hkv + gk) * g.S_cap + pos) * g.D + d] = k_new[src];
        v_cube[(((size_t)(b * g.Hkv + gk) * g.n_kv_blocks_cap + blk) * g.D + d) * kBlockTok + tok] = v_new[src];
    }
}

constexpr int kDecodeCandCap = 256;
// CTAs of a cluster = CTAs per (batch, kv head).  The cubes are dealt to them for the scores, the heads for the
// selection.  One CTA per (batch, kv head) left most of the chip idle (4 .. 64 CTAs): 14.6 us for one sequence of 256
// cubes and 70 us for 16 sequences of 2048.
constexpr int kPlanCtas = 8;
constexpr int kPlanWarps = 4;            // at 128 registers a thread four CTAs fit an SM: 16 x 4 clusters run at once
__host__ __device__ inline int decode_head_slots(int G) { return (G + kPlanCtas - 1) / kPlanCtas; }   // heads per CTA
// dynamic smem of decode_select_plan_kernel: per head slot N_ld scores + histogram + candidates (8 bytes each), and
// the group's union of selection words
__host__ __device__ inline size_t decode_select_smem_bytes(int N_ld, int G, int n_words) {
    return (size_t)decode_head_slots(G) * ((size_t)N_ld + kSelHistWords + kDecodeCandCap) * 8 + (size_t)n_words * 4;
}

// grid (8, Hkv, B) in clusters of 8, 128 threads.
// items[(b*Hkv+gk) * n_kv_blocks_cap + i] = index of the i-th block to visit.  header: 256 bytes, set to zero.
template <int D>
__global__ void __cluster_dims__(kPlanCtas, 1, 1) __launch_bounds__(kPlanWarps * 32, 4) decode_select_plan_kernel(
    Geom g, const __nv_bfloat16* q_new, const __nv_bfloat16* k_new, const __nv_bfloat16* v_new, __nv_bfloat16* k_cube,
    __nv_bfloat16* v_cube, const float* cube_keys, const int32_t* text_len, uint32_t* dec_bitmap, uint32_t* sel_bitmap,
    int32_t* items, int32_t* n_items, uint32_t* header) {
    extern __shared__ __align__(16) double dsp_smem[];
    const int rank = blockIdx.x, gk = blockIdx.y, b = blockIdx.z;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int slots = decode_head_slots(g.G);
    double* logit = dsp_smem;                                              // [slots][N_ld]: head slot * 8 + rank
    unsigned long long* sel_scratch = reinterpret_cast<unsigned long long*>(dsp_smem + (size_t)slots * g.N_ld);   // [slots][hist + cand]
    uint32_t* bm = reinterpret_cast<uint32_t*>(sel_scratch + (size_t)slots * (kSelHistWords + kDecodeCandCap));   // [n_words] (rank 0)
    for (int w = threadIdx.x; w < g.n_words; w += blockDim.x) bm[w] = 0u;
    cluster_sync();                                                        // every CTA of the cluster runs: its memory may be written
    // Launched to overlap whatever comes before it in the stream, which may have made the inputs (none of them __restrict__).
    // Only then the next kernel: what it reads before its own wait is finished too.  (Plain launches: one sequence of 256 cubes 28.5
    // instead of 27.3 us a step, smaller ones 20.5 / 17.3, 24.2 / 22.3, 17.0 / 16.0; nothing where the caches are large.)
    wait_for_previous_kernel();
    launch_dependents();
    if (rank == kPlanCtas - 1 && k_new != nullptr) decode_append(g, b, gk, k_new, v_new, k_cube, v_cube, text_len);   // read by the next kernel
    if (rank == kPlanCtas - 2 && gk == 0 && b == 0 && threadIdx.x < 64) header[threadIdx.x] = 0u;   // the next kernels write it
    const float* kbase = cube_keys + (size_t)(b * g.Hkv + gk) * g.N * D;
    const int rq = lane >> 2, kq = lane & 3;

    const bool all = g.top_k <= 0 && !(g.top_p < 1.0);
    for (int h0 = 0; !all && h0 < g.G; h0 += 8) {
        // ---- scores: <q_(h0+r), kbar_j> of this CTA's share of the cubes.  The head-dim index is permuted
        // the same way for both operands so that each lane reads 4 consecutive elements:
        // k-step 4*S + s' uses d = 16*S + 4*kq + s'.
        float a[D / 4];
        const bool live = h0 + rq < g.G;
        {
            const __nv_bfloat16* qsrc = q_new + ((size_t)b * g.Hq + gk * g.G + (live ? h0 + rq : 0)) * D;
#pragma unroll
            for (int S = 0; S < D / 16; ++S)
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    a[4 * S + s] = live ? __bfloat162float(qsrc[16 * S + 4 * kq + s]) : 0.f;
        }
        // head h0 + r belongs to CTA r of the cluster: its score goes to that CTA's shared memory
        const uint32_t row = cluster_address(logit + (size_t)(h0 / 8) * g.N_ld, rq);
        // Groups of 8 cubes, dealt to all warps of the cluster; the mean keys stream from HBM: the loads of the next
        // group are issued before the tensor ops of this one.
        auto load_keys = [&](int c0, float4 (&kv)[D / 16]) {
            const int cube = c0 + rq;
            const float* ksrc = kbase + (size_t)(cube < g.N ? cube : 0) * D + 4 * kq;
#pragma unroll
            for (int S = 0; S < D / 16; ++S)
                kv[S] = cube < g.N ? *reinterpret_cast<const float4*>(ksrc + 16 * S) : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        auto score_keys = [&](int c0, const float4 (&kv)[D / 16]) {
            double acc[2] = {0.0, 0.0}, acc2[2] = {0.0, 0.0};              // two chains of tensor ops
#pragma unroll
            for (int S = 0; S < D / 16; ++S) {
                mma_f64_884(acc, (double)a[4 * S + 0], (double)kv[S].x);
                mma_f64_884(acc2, (double)a[4 * S + 1], (double)kv[S].y);
                mma_f64_884(acc, (double)a[4 * S + 2], (double)kv[S].z);
                mma_f64_884(acc2, (double)a[4 * S + 3], (double)kv[S].w);
            }
            // C fragment: row = lane/4, columns 2*(lane%4) + {0,1}
            if (live)
                asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};\n" ::"r"(row + (uint32_t)(c0 + 2 * kq) * 8u),
                             "d"((acc[0] + acc2[0]) * g.scale_d), "d"((acc[1] + acc2[1]) * g.scale_d)
                             : "memory");
        };
        {
            constexpr int kStep = kPlanCtas * kPlanWarps * 8;              // cubes per round of the cluster
            float4 kv_a[D / 16], kv_b[D / 16];
            int c0 = (rank * kPlanWarps + warp) * 8;
            if (c0 < g.N_ld) load_keys(c0, kv_a);
            for (; c0 < g.N_ld; c0 += 2 * kStep) {
                if (c0 + kStep < g.N_ld) load_keys(c0 + kStep, kv_b);
                score_keys(c0, kv_a);
                if (c0 + kStep < g.N_ld) {
                    if (c0 + 2 * kStep < g.N_ld) load_keys(c0 + 2 * kStep, kv_a);
                    score_keys(c0 + kStep, kv_b);
                }
            }
        }
    }
    cluster_sync();
    // ---- Eq. 2: warp s of this CTA takes head 8 s + rank
    if (warp < slots && warp * kPlanCtas + rank < g.G) {
        const int h = gk * g.G + warp * kPlanCtas + rank;
        double* row = logit + (size_t)warp * g.N_ld;
        unsigned long long* keys = reinterpret_cast<unsigned long long*>(row);
        const int n = g.N;
        unsigned long long bd = 0ull;
        if (!all) {
            unsigned long long* hist = sel_scratch + (size_t)warp * (kSelHistWords + kDecodeCandCap);
            bd = nucleus_boundary_radix<32, true>(row, n, g.top_p, g.top_k, keys, hist, hist + kSelHistWords, kDecodeCandCap, lane);
        }
        const uint32_t bm0 = cluster_address(bm, 0);
        for (int w = 0; w < g.n_words; ++w) {
            const int j = w * 32 + lane;
            const bool on = j < n && (all || keys[j] >= bd);
            const uint32_t word = __ballot_sync(0xffffffffu, on);
            if (lane == 0) {
                dec_bitmap[((size_t)b * g.Hq + h) * g.n_words + w] = word;
                if (sel_bitmap) sel_bitmap[((size_t)b * g.Hq + h) * g.n_words + w] = word;
                asm volatile("red.shared::cluster.or.b32 [%0], %1;\n" ::"r"(bm0 + 4u * w), "r"(word) : "memory");
            }
        }
    }
    cluster_sync();
    if (rank != 0) return;

    // ---- plan: blocks that hold a selected cube of any head of the group, plus the text blocks
    // (bm holds the union of the group's selections)
    // every warp takes a contiguous run of blocks: count, prefix over the warps, then write
    __shared__ int plan_cnt[kPlanWarps];
    const int tl = text_len[b];
    const int last_pos = g.S_v + tl;                     // position of the new token
    int n_blk = 0;
    if (tl >= 0 && tl <= g.n_text) n_blk = last_pos / kBlockTok + 1;
    const int per_warp = ((n_blk + kPlanWarps - 1) / kPlanWarps + 31) / 32 * 32;
    const int kb_lo = warp * per_warp, kb_hi = min(kb_lo + per_warp, n_blk);
    auto block_needed = [&](int kb) -> bool {
        if (kb >= kb_hi) return false;
        bool need = kb * kBlockTok + kBlockTok - 1 >= g.S_v;   // holds text positions
        if (kb * kBlockTok < g.S_v) {
            int c_lo = (kb * kBlockTok) >> g.c_shift;
            int c_hi = min((kb * kBlockTok + kBlockTok - 1) >> g.c_shift, g.N - 1);
            uint32_t span = c_hi - c_lo + 1;
            uint32_t bits = (span >= 32 ? 0xffffffffu : ((1u << span) - 1u)) << (c_lo & 31);
            if (bm[c_lo >> 5] & bits) need = true;
        }
        return need;
    };
    int mine = 0;
    for (int kb0 = kb_lo; kb0 < kb_hi; kb0 += 32) mine += __popc(__ballot_sync(0xffffffffu, block_needed(kb0 + lane)));
    if (lane == 0) plan_cnt[warp] = mine;
    __syncthreads();
    int count = 0, total = 0;
    for (int i = 0; i < kPlanWarps; ++i) {
        if (i < warp) count += plan_cnt[i];
        total += plan_cnt[i];
    }
    int32_t* dst = items + (size_t)(b * g.Hkv + gk) * g.n_kv_blocks_cap;
    for (int kb0 = kb_lo; kb0 < kb_hi; kb0 += 32) {
        const int kb = kb0 + lane;
        const bool need = block_needed(kb);
        const uint32_t ball = __ballot_sync(0xffffffffu, need);
        if (need) dst[count + __popc(ball & ((1u << lane) - 1u))] = kb;
        count += __popc(ball);
    }
    if (threadIdx.x == 0) n_items[b * g.Hkv + gk] = total;
}

// grid (Hq, B), 512 threads.  partial[((b*Hkv+gk)*n_splits + split)*G + row] = {m, l, o[D]}, n_splits <= 64.  512 / D
// groups of threads share the splits, and all loads of a thread are issued before the weights are needed: one round
// trip to the L2.  (A thread that walked the 64 splits by itself took 15.7 us.)  CTA (0, 0) also fills in the header:
// total_blocks = sum of n_items, status 1 if a text_len lies outside [0, n_text_max].
template <int D>
__global__ void __launch_bounds__(512) decode_combine_kernel(Geom g, int n_splits, const float* partial,
                                                             const int32_t* __restrict__ text_len,
                                                             const int32_t* n_items,
                                                             unsigned long long* __restrict__ total_blocks,
                                                             int32_t* __restrict__ status, __nv_bfloat16* __restrict__ out) {
    constexpr int kGroups = 512 / D, kPer = 64 / kGroups, kRowF = D + 2;
    __shared__ float weight[64];
    __shared__ float l_all;
    __shared__ float red[kGroups][D];
    const int h = blockIdx.x, b = blockIdx.y, d = threadIdx.x & (D - 1), grp = threadIdx.x / D;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gk = h / g.G, row = h - gk * g.G;
    launch_dependents();                                                   // the first kernel of the next step sets itself up meanwhile
    wait_for_previous_kernel();
    const float* base = partial + ((size_t)(b * g.Hkv + gk) * n_splits * g.G + row) * kRowF;
    const size_t stride = (size_t)g.G * kRowF;
    float o[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int s = grp + i * kGroups;
        o[i] = s < n_splits ? base[s * stride + 2 + d] : 0.f;
    }
    if (warp == 0) {
        float m[2], l[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int s = lane + 32 * i;
            m[i] = s < n_splits ? base[s * stride] : -INFINITY;
            l[i] = s < n_splits ? base[s * stride + 1] : 0.f;
        }
        float mx = fmaxf(m[0], m[1]), sum = 0.f;
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, k));
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float w = m[i] == -INFINITY ? 0.f : exp2f(m[i] - mx);
            weight[lane + 32 * i] = w;
            sum += l[i] * w;
        }
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, k);
        if (lane == 0) l_all = sum;
    } else if (warp == 1 && h == 0 && b == 0) {
        unsigned long long total = 0ull;
        bool bad = false;
        for (int i = lane; i < g.B * g.Hkv; i += 32) total += (unsigned long long)n_items[i];
        for (int i = lane; i < g.B; i += 32) bad = bad || text_len[i] < 0 || text_len[i] > g.n_text;
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) total += __shfl_xor_sync(0xffffffffu, total, k);
        bad = __any_sync(0xffffffffu, bad);
        if (lane == 0) {
            *total_blocks = total;
            if (bad) atomicCAS(status, 0, 1);
        }
    }
    __syncthreads();
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < kPer; ++i) acc = fmaf(o[i], weight[grp + i * kGroups], acc);
    red[grp][d] = acc;
    __syncthreads();
    if (grp == 0) {
#pragma unroll
        for (int i = 1; i < kGroups; ++i) acc += red[i][d];
        out[((size_t)b * g.Hq + h) * D + d] = __float2bfloat16(l_all > 0.f ? acc / l_all : 0.f);
    }
}

}  // namespace adaspark
