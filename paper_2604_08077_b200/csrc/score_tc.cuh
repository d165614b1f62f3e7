// K3a: cube scores (Eq. 1) of query tiles on the int8 tensor cores, as 32-bit fixed point.
//
// The selection must follow an fp64 evaluation of Eqs. 1-2 (rows may differ only inside a 1e-6 probability
// margin), so plain bf16/fp32 tensor-core arithmetic is not accurate enough.  Every query row q and every mean
// key k, less the head's first mean key k_0, are written in fixed point,
//     x = 2^(e - 29) * (d0*2^24 + d1*2^16 + d2*2^8 + d3),   digits d_i signed bytes in [-128, 127],
// with e the exponent of the largest element of the query row (e_q) or of all differences k_j - k_0 of the
// (batch, kv head) (E_K).  What all keys of a head share (a bias) moves all scores of a row alike and has no part in its
// selection, but would cost the fp32 scores their low bits.  Cube 0 is a candidate of every row that has one: no score is
// larger than the row's spread.  tcgen05.mma of kind::i8 multiplies the digit planes with exact int32
// accumulation,  S_L = sum_{a+b=L} Q_a . K_b  (10 digit pairs, levels L = 0..3, four TMEM
// accumulators), and
//     q . (k_j - k_0) = 2^(e_q + E_K - 34) * V_j,      V_j = S_0*2^24 + S_1*2^16 + S_2*2^8 + S_3   (an int64),
// up to the dropped levels >= 4 and the rounding of elements far below the row maximum.  Because the
// key exponent is shared by the whole head, all scores of a row are the SAME positive factor
// f = 2^(e_q + E_K - 34) * scale times an integer.
//
// What leaves the kernel per (row, cube) is the score in log2 units as fp32, s_j = W_j * (f 2^sh log2 e) with
// W_j = V_j >> sh an int32: sh is the row's own shift, the smallest for which |q| max|k_j - k_0| (Cauchy-Schwarz over the
// head) proves that no score overflows (on the benchmark inputs sh = 8: one unit of W is 1e-8 in the
// scaled logit, below the 2e-8 that the dropped levels leave), and the largest and smallest score of every row.  The
// selection kernel (select_nucleus.cuh) reads them from the workspace and decides every row whose boundary is clearer than
// fp32 can be wrong.  A launch covers as many query tiles as the workspace has room for, mostly those of the whole call; where it has
// less, the two kernels alternate over the call.
//
// Rows whose exponents are so large that the fixed-point error could reach the margin (f > kMaxScorePerUnit) are
// marked (NaN scores) and go to the fp64 kernel of select_exact.cuh.
//
// Roles (896 threads, one persistent CTA per SM, work item = one 128-row query tile, long tiles first):
//   warps 0-15   epilogue: warp w reads TMEM lane quarter w % 4, columns 16*(w/4) .. +15 of every column tile,
//                folds the four levels into s and stores a 32 x 16 box through shared memory with TMA.  (With eight
//                warps the epilogue was the limit: a warp's chain of loads and conversions is latency-bound)
//   warps 16-23  slicers (two threads per row, half a row each, held in registers between the sweep for the largest
//                exponent and the slicing): digit planes of the next tile's queries, two buffers.  With one thread per
//                row that read its row twice the slicers took 13 k cycles per tile and the tensor core waited
//   warp 24      TMA producer: key digit planes of one column tile (4 x 8 KB), 2 slots
//   warps 25-26  issue the tcgen05.mma stream (10 digit pairs x D/32 of 128x64x32 per column tile, half each)
//                into double-buffered accumulator sets (2 x 4 levels x 64 columns = all 512 TMEM columns);
//                each warp runs converged and issues through one elected lane
//   warp 27      clears the union words of the tile
#pragma once
#include "tc_common.cuh"

namespace adaspark {

constexpr int kScoreThreads = 896;
constexpr int kEpilogueWarps = 16;
constexpr int kRangeParts = 4;          // partial score ranges per row: one per column group of the epilogue
constexpr int kScoreTcCols = 64;         // cubes per column tile
constexpr int kDigitRowBytes = 128;      // bytes per row of a digit plane
// Largest score per unit of V (f) that is decided from these scores: 2^(7 - 34) / sqrt(64), i.e. exponents up to
// e_q + E_K = 7 at the default scale of head_dim 64: with twice the largest mean key as the largest difference, mean keys up
// to the size that was decided when the scores were not relative to k_0.  (The fixed-point error grows with f, and with it
// the share of rows that are too near to call.)
constexpr double kMaxScorePerUnit = 0.125 / 134217728.0;
// Units of V that the digits leave open in a score's distance from another's: the dropped levels and the rounding of the
// elements.  Against 64-bit products, over normal, uniform, heavy-tailed and constant queries and keys, each 512 rows x 512
// keys: rms 180 (D = 64) and 255 (D = 128), at most 1021 and 2065.
template <int D>
constexpr float kFixedErr = 16.f * D;
constexpr int kMaxRowShift = 16;         // |V| < D * 2^36 = 2^43 by construction, so a shift of 12 always suffices

// The four signed base-256 digits of v = round(x * 2^(29 - e)) (|v| <= 2^30), packed in one word:
// byte 3 = d0 (most significant) ... byte 0 = d3.  Adding 0x80 to every byte position turns the
// balanced digits into the plain unsigned bytes of v + 0x80808080, so two integer operations give
// all four.
__device__ __forceinline__ uint32_t packed_digits(int v) {
    const uint32_t u = (uint32_t)v + 0x80808080u;
    return u ^ 0x80808080u;
}
__device__ __forceinline__ float digit_scale(int e) {             // 2^(29 - e), exact for e >= -97
    return __int_as_float((156 - e) << 23);
}
__device__ __forceinline__ int row_exponent_from_field(int biased) {   // 8-bit exponent field of the row maximum
    return biased == 0 ? 0 : max(biased - 127, -90);               // rows smaller than 2^-90 keep fewer digits
}
// The digits of four elements by plane: plane[p] holds digit p (p = 0 most significant) of element i in byte i, a
// transposition of the 4 x 4 bytes.
__device__ __forceinline__ void digit_planes(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t (&plane)[4]) {
    const uint32_t a = __byte_perm(w0, w1, 0x5140), b = __byte_perm(w2, w3, 0x5140);
    const uint32_t c = __byte_perm(w0, w1, 0x7362), d = __byte_perm(w2, w3, 0x7362);
    plane[3] = __byte_perm(a, b, 0x5410);
    plane[2] = __byte_perm(a, b, 0x7632);
    plane[1] = __byte_perm(c, d, 0x5410);
    plane[0] = __byte_perm(c, d, 0x7632);
}
// V >> sh = S_0 2^(24-sh) + S_1 2^(16-sh) + ((S_2 2^8 + S_3) >> sh) for sh <= 16; m0 = 2^(24-sh), m1 = 2^(16-sh).  The sum
// fits 32 bits, its terms need not (S_0 and S_1 may cancel), so they are added as unsigned words, which wrap.
// |S_2 2^8 + S_3| < 2^31.
__host__ __device__ __forceinline__ int32_t shifted_levels(int32_t s0, int32_t s1, int32_t s2, int32_t s3, uint32_t m0, uint32_t m1, int sh) {
    const int32_t low = s2 * 256 + s3;
    return (int32_t)((uint32_t)s0 * m0 + ((uint32_t)s1 * m1 + (uint32_t)(low >> sh)));
}
__device__ __forceinline__ int head_exponent(uint32_t max_bits) { return row_exponent_from_field((int)((max_bits >> 23) & 0xffu)); }

// Digit planes of the mean keys less the head's first: planes[p][(b*Hkv+gk)*N_ld + cube][128 bytes] (int8, zero beyond D),
// all cubes of a (batch, kv head) in the fixed point of that head's exponent; rows >= N inside the padded leading
// dimension are zero-filled.  A cluster of 8 CTAs per (batch, kv head) first finds the largest |element| (exchanged through distributed shared memory, float bits: non-negative floats order like their bit patterns), then
// slices (the differences in fp64, rounded once to the fixed point), and leaves the largest |element| in head_max_bits and the
// largest norm times 2^(29 - E_K) in head_norm (of the scaled values: no size of input over- or underflows the squares).  grid (8, B*Hkv), 256 threads.
// (One kernel for all: two cost a launch more, 3 us of a short call.)
// key_hash[(b*Hkv+gk)*N_ld + cube]: 64 bits of the mean key's own bits.  Equal keys have equal words; that two different
// keys share one is left to chance (2^-64), and asked only of keys whose scores are too near to tell apart.
constexpr int kSliceCtas = 8;
__device__ __forceinline__ unsigned long long hash_multiplier(uint32_t i) {      // an odd word per element (splitmix64)
    unsigned long long z = (i + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return (z ^ (z >> 31)) | 1ull;
}
__global__ void __cluster_dims__(kSliceCtas, 1, 1) __launch_bounds__(256) slice_keys_kernel(
    Geom g, const float* cube_keys, uint32_t* head_max_bits, float* head_norm, unsigned char* planes, unsigned long long* key_hash) {
    __shared__ uint32_t head[2];
    launch_dependents();
    const int rank = blockIdx.x, bh = blockIdx.y, lane = threadIdx.x & 31;
    if (threadIdx.x < 2) head[threadIdx.x] = 0u;
    const unsigned long long hm[4] = {hash_multiplier(lane * 4), hash_multiplier(lane * 4 + 1), hash_multiplier(lane * 4 + 2), hash_multiplier(lane * 4 + 3)};
    cluster_sync();                                           // every CTA of the cluster runs: its memory may be written
    wait_for_previous_kernel();
    const float4* src = reinterpret_cast<const float4*>(cube_keys + (size_t)bh * g.N * g.D);
    const int n4 = g.N_live * (g.D / 4);                      // the cubes present so far
    uint32_t mx = 0;
    const float4 a = src[threadIdx.x & (g.D / 4 - 1)];        // of cube 0, the thread's elements in both loops (D / 4 divides 256)
#pragma unroll 4
    for (int i = rank * 256 + threadIdx.x; i < n4; i += kSliceCtas * 256) {
        const float4 x = src[i];
        mx = max(max(mx, __float_as_uint(fabsf(x.x - a.x))), max(__float_as_uint(fabsf(x.y - a.y)),
                 max(__float_as_uint(fabsf(x.z - a.z)), __float_as_uint(fabsf(x.w - a.w)))));
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane < kSliceCtas) asm volatile("red.shared::cluster.max.u32 [%0], %1;\n" ::"r"(cluster_address(head, lane)), "r"(mx) : "memory");
    cluster_sync();
    const uint32_t max_bits = head[0];
    const double mult = (double)digit_scale(head_exponent(max_bits));
    const size_t plane_stride = (size_t)g.B * g.Hkv * g.N_ld * kDigitRowBytes;
    float norm2 = 0.f;
#pragma unroll 2
    for (int cube = rank * 8 + (threadIdx.x >> 5); cube < g.N_ld; cube += kSliceCtas * 8) {
        float4 x = a;
        if (cube < g.N_live && lane * 4 < g.D) x = src[(size_t)cube * (g.D / 4) + lane];
        unsigned long long hash = __float_as_uint(x.x) * hm[0] + __float_as_uint(x.y) * hm[1] + __float_as_uint(x.z) * hm[2] + __float_as_uint(x.w) * hm[3];
        const double y0 = ((double)x.x - (double)a.x) * mult, y1 = ((double)x.y - (double)a.y) * mult;
        const double y2 = ((double)x.z - (double)a.z) * mult, y3 = ((double)x.w - (double)a.w) * mult;
        float n2 = fmaf((float)y0, (float)y0, fmaf((float)y1, (float)y1, fmaf((float)y2, (float)y2, (float)y3 * (float)y3)));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            n2 += __shfl_xor_sync(0xffffffffu, n2, o);
            hash += __shfl_xor_sync(0xffffffffu, hash, o);
        }
        norm2 = fmaxf(norm2, n2);
        if (lane == 0) key_hash[(size_t)bh * g.N_ld + cube] = hash;
        uint32_t plane[4];
        digit_planes(packed_digits(__double2int_rn(y0)), packed_digits(__double2int_rn(y1)), packed_digits(__double2int_rn(y2)),
                     packed_digits(__double2int_rn(y3)), plane);
        unsigned char* dst = planes + ((size_t)bh * g.N_ld + cube) * kDigitRowBytes + lane * 4;
#pragma unroll
        for (int p = 0; p < 4; ++p) *reinterpret_cast<uint32_t*>(dst + p * plane_stride) = plane[p];
    }
    if (lane == 0) asm volatile("red.shared::cluster.max.u32 [%0], %1;\n" ::"r"(cluster_address(head + 1, 0)), "r"(__float_as_uint(norm2)) : "memory");
    cluster_sync();
    if (rank == 0 && threadIdx.x == 0) { head_max_bits[bh] = max_bits; head_norm[bh] = sqrtf(__uint_as_float(head[1])); }
}

template <int D>
struct ScoreSmem {
    unsigned char qd[2][4][128][kDigitRowBytes];                   // digit planes of two Q tiles, UMMA layout (128-B swizzle)
    unsigned char kring[2][4][kScoreTcCols][kDigitRowBytes];       // key digit planes of a column tile, two slots
    float stage[kEpilogueWarps][32][16];                           // per epilogue warp: 32 rows x 16 scores, 64-B swizzle
    uint8_t row_shift[2][128];                                     // sh of each row of the tile (by buffer)
    float row_scale[2][128];                                       // score in log2 units per unit of W; NaN: not decided here
    uint64_t q_sliced[2], qd_free[2], k_full[2], acc_full[2], acc_free[2];
    uint32_t tmem_base;
    int abort_flag;
};

// Work item `it` of the call: long (late) tiles first.
struct ScoreItem {
    int b, h, gk, tile, n_ct;
};
__device__ __forceinline__ ScoreItem score_item(const Geom& g, int it) {
    ScoreItem w;
    const int n_hb = g.B * g.Hq;
    const int lvl = it / n_hb, hb = it - lvl * n_hb;
    w.tile = g.n_tiles - 1 - lvl;
    g.div_Hq.divmod(hb, w.b, w.h);
    w.gk = w.h / g.G;
    w.n_ct = (tile_max_candidates(g, w.tile) + kScoreTcCols - 1) / kScoreTcCols;
    return w;
}

// Ranges of a row of the items it, it + step, .. whose scores have not been computed (a wait has expired; the call's status says so).  The
// selection kernel goes by a range without bounds of its own, and the workspace holds anything: with a lower end of -inf it leaves the
// row to the fp64 kernel, which needs no scores, whatever the row's other parts are.
__host__ __device__ inline void abandon_ranges(float2* row_range, int it, int n_items, int step, int row, int part) {
    for (; it < n_items; it += step) row_range[kRangeParts * ((size_t)it * kTileRows + row) + part] = make_float2(-INFINITY, -INFINITY);
}

// Scores of the items [item0, item0 + n_items): row r of item item0 + i goes to row 128 * i + r of the scratch
// matrix that tmS describes (fp32 [rows][N_ld]; columns beyond the tile's last candidate are not written), the
// largest and smallest score of its candidates to row_range[4 * (128 * i + r) + part], part = which 16 of every 64
// columns, and what the fixed point leaves open in its scores to row_err[128 * i + r].  q: the call's queries [B, S_io, Hq, D].  tile_union words of the items are
// set to zero for the selection kernel.
template <int D>
__global__ void __launch_bounds__(kScoreThreads, 1) score_tc_kernel(
    Geom g, int item0, int n_items, const __nv_bfloat16* __restrict__ q, const __grid_constant__ CUtensorMap tmK,
    const __grid_constant__ CUtensorMap tmS, const uint32_t* head_max_bits, const float* head_norm,
    float2* row_range, float* row_err, uint32_t* tile_union, int32_t* status) {
    extern __shared__ unsigned char score_raw[];
    ScoreSmem<D>& sm = *reinterpret_cast<ScoreSmem<D>*>((reinterpret_cast<uintptr_t>(score_raw) + 1023) & ~(uintptr_t)1023);
    constexpr uint32_t kIdesc = tc::make_idesc_s8(128, kScoreTcCols);
    constexpr uint32_t kPlaneBytes = kScoreTcCols * kDigitRowBytes;
    constexpr int kSlicerWarp0 = kEpilogueWarps, kProducerWarp = 24, kMmaWarp = 25, kClearWarp = 27;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&sm.q_sliced[i], 8);                // one arrival per slicer warp
            tc::mbar_init(&sm.qd_free[i], 2 + kEpilogueWarps);   // a commit per MMA-issuing warp, an arrival per epilogue warp
            tc::mbar_init(&sm.k_full[i], 1);
            tc::mbar_init(&sm.acc_full[i], 2);
            tc::mbar_init(&sm.acc_free[i], kEpilogueWarps);   // one arrival per epilogue warp
        }
        sm.abort_flag = 0;
        tc::fence_barrier_init();
    }
    launch_dependents();
    wait_for_previous_kernel();
    if (warp == kProducerWarp) {
        tc::tmem_alloc<512>(&sm.tmem_base);
        if (lane == 0) {
            tc::prefetch_tensormap(&tmK);
            tc::prefetch_tensormap(&tmS);
        }
    }
    tc::tc_fence_before_sync();
    __syncthreads();
    tc::tc_fence_after_sync();
    const uint32_t tbase = sm.tmem_base;
    volatile int* abort_flag = &sm.abort_flag;

    if (warp == kProducerWarp) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            const int n_rows = g.B * g.Hkv * g.N_ld;
            int c = 0;                                            // running job counter of this CTA
            bool ok = true;
            for (int it = blockIdx.x; ok && it < n_items; it += gridDim.x) {
                const ScoreItem w = score_item(g, item0 + it);
                const int k_row0 = (w.b * g.Hkv + w.gk) * g.N_ld;
                for (int ct = 0; ok && ct < w.n_ct; ++ct, ++c) {
                    const int s = c & 1, use = c >> 1;
                    if (use > 0 && !(ok = tc::mbar_wait(&sm.acc_full[s], (use - 1) & 1, abort_flag))) break;   // the slot's last reader has finished
                    tc::mbar_arrive_expect_tx(&sm.k_full[s], 4 * kPlaneBytes);
                    for (int pl = 0; pl < 4; ++pl)
                        tc::tma_load_2d(&sm.kring[s][pl][0][0], &tmK, 0, pl * n_rows + k_row0 + ct * kScoreTcCols, &sm.k_full[s]);
                }
            }
        }
    } else if (warp == kMmaWarp || warp == kMmaWarp + 1) {
        // ------------------------------------------------------------ MMA issuers
        // Two warps issue the stream (one thread gets a 128x64x32 MMA accepted every ~90 cycles, the tensor core
        // would take them faster): issuer 0 owns the accumulators of levels 0 and 3, issuer 1 those of levels 1
        // and 2 (five digit pairs each, no accumulator shared); a job is ready when both have committed.
        const int issuer = warp - kMmaWarp;
        constexpr uint32_t kQPlaneStep = (uint32_t)sizeof(sm.qd[0][0]) >> 4, kKPlaneStep = (uint32_t)sizeof(sm.kring[0][0]) >> 4;
        constexpr uint32_t kQBufStep = (uint32_t)sizeof(sm.qd[0]) >> 4, kSlotStep = (uint32_t)sizeof(sm.kring[0]) >> 4, kKStep = 32 >> 4;
        const uint32_t q_lo0 = __shfl_sync(0xffffffffu, tc::smem_desc_lo_sw128(smem_u32(&sm.qd[0][0][0][0])), 0);
        const uint32_t k_lo0 = __shfl_sync(0xffffffffu, tc::smem_desc_lo_sw128(smem_u32(&sm.kring[0][0][0][0])), 0);
        const uint32_t tb = __shfl_sync(0xffffffffu, tbase, 0);
        bool ok = true;
        int c = 0, n_done = 0;
        for (int it = blockIdx.x; ok && it < n_items; it += gridDim.x) {
            const ScoreItem w = score_item(g, item0 + it);
            if (w.n_ct == 0) continue;
            const int qb = n_done & 1;
            if (!(ok = tc::mbar_wait_warp(&sm.q_sliced[qb], (n_done >> 1) & 1, abort_flag))) break;
            const uint32_t qa0 = q_lo0 + qb * kQBufStep;
            for (int ct = 0; ok && ct < w.n_ct; ++ct, ++c) {
                const int s = c & 1, use = c >> 1;
                if (use > 0 && !(ok = tc::mbar_wait_warp(&sm.acc_free[s], (use - 1) & 1, abort_flag))) break;
                if (!(ok = tc::mbar_wait_warp(&sm.k_full[s], use & 1, abort_flag))) break;
                tc::tc_fence_after_sync();
                const uint32_t kb0 = k_lo0 + s * kSlotStep;
                // level L = a + (L - a): plane a of the queries, plane L - a of the keys
                if (tc::elect_one()) {
#pragma unroll
                    for (int L = 0; L < 4; ++L) {
                        if (((L == 0 || L == 3) ? 0 : 1) != issuer) continue;
#pragma unroll
                        for (int a = 0; a <= L; ++a)
#pragma unroll
                            for (int ks = 0; ks < D / 32; ++ks)
                                tc::umma_ss_i8(tb + s * 256 + L * kScoreTcCols,
                                               tc::smem_desc_from_halves(qa0 + a * kQPlaneStep + ks * kKStep, tc::kSmemDescHiSw128),
                                               tc::smem_desc_from_halves(kb0 + (L - a) * kKPlaneStep + ks * kKStep, tc::kSmemDescHiSw128),
                                               kIdesc, !(a == 0 && ks == 0));
                    }
                    tc::umma_commit(&sm.acc_full[s]);             // accumulators ready; the key slot may be reloaded
                }
                __syncwarp();
            }
            if (ok && tc::elect_one()) tc::umma_commit(&sm.qd_free[qb]);   // the digit planes may be overwritten (both issuers)
            __syncwarp();
            ++n_done;
        }
    } else if (warp >= kSlicerWarp0 && warp < kProducerWarp) {
        // ------------------------------------------------------------ slicers (two neighbouring threads per row)
        const int r = (tid - kSlicerWarp0 * 32) >> 1, part = tid & 1;
        bool ok = true;
        int n_done = 0;
        for (int it = blockIdx.x; ok && it < n_items; it += gridDim.x) {
            const ScoreItem w = score_item(g, item0 + it);
            if (w.n_ct == 0) continue;
            const int qb = n_done & 1;
            const int pos = w.tile * kTileRows + r;
            // the row is read where the caller left it (sequence order): no cube-major copy of Q exists
            uint4 v[D / 16];                                      // chunks 2 c + part: the two threads share every 32-byte sector
            if (slot_live(g, pos)) {
                const uint4* src = reinterpret_cast<const uint4*>(q + (io_row(g, w.b, pos) * g.Hq + w.h) * D);
#pragma unroll
                for (int c = 0; c < D / 16; ++c) v[c] = __ldg(src + 2 * c + part);
            } else {
#pragma unroll
                for (int c = 0; c < D / 16; ++c) v[c] = make_uint4(0u, 0u, 0u, 0u);
            }
            uint32_t mx2 = 0;                                     // largest magnitudes of the even and the odd elements
#pragma unroll
            for (int c = 0; c < D / 16; ++c)
                mx2 = __vmaxu2(__vmaxu2(__vmaxu2(mx2, v[c].x & 0x7fff7fffu), v[c].y & 0x7fff7fffu),
                               __vmaxu2(v[c].z & 0x7fff7fffu, v[c].w & 0x7fff7fffu));
            uint32_t mxbits = max(mx2 & 0xffffu, mx2 >> 16);
            mxbits = max(mxbits, __shfl_xor_sync(0xffffffffu, mxbits, 1));
            const int e_q = row_exponent_from_field((int)(mxbits >> 7));
            const float mult = digit_scale(e_q);
            // the tile before the last is done with this buffer: its MMAs with the planes, its epilogue with the constants
            if (n_done >= 2 && !(ok = tc::mbar_wait(&sm.qd_free[qb], ((n_done >> 1) - 1) & 1, abort_flag))) break;
            unsigned char* dst = &sm.qd[qb][0][0][0];
            float q2 = 0.f;                                       // |q|^2 2^(2 (29 - e_q))
#pragma unroll
            for (int c = 0; c < D / 16; ++c) {                    // 8 elements = half a 16-byte chunk of every plane
                const uint32_t wd[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
                uint32_t pw[2][4];                                // [4 elements][plane]
#pragma unroll
                for (int q2w = 0; q2w < 2; ++q2w) {
                    const uint32_t wa = wd[2 * q2w], wb = wd[2 * q2w + 1];
                    const float y0 = __uint_as_float(wa << 16) * mult, y1 = __uint_as_float(wa & 0xffff0000u) * mult;
                    const float y2 = __uint_as_float(wb << 16) * mult, y3 = __uint_as_float(wb & 0xffff0000u) * mult;
                    q2 = fmaf(y0, y0, fmaf(y1, y1, fmaf(y2, y2, fmaf(y3, y3, q2))));
                    digit_planes(packed_digits(__float2int_rn(y0)), packed_digits(__float2int_rn(y1)), packed_digits(__float2int_rn(y2)),
                                 packed_digits(__float2int_rn(y3)), pw[q2w]);
                }
                const int off = sw128(r, c) + 8 * part;           // elements 16 c + 8 part .. +7 of the plane row
#pragma unroll
                for (int pl = 0; pl < 4; ++pl)
                    *reinterpret_cast<uint2*>(dst + (size_t)pl * sizeof(sm.qd[0][0]) + off) = make_uint2(pw[0][pl], pw[1][pl]);
            }
            // ---- the row's constants
            q2 += __shfl_xor_sync(0xffffffffu, q2, 1);
            if (part == 0) {
                const int bh = w.b * g.Hkv + w.gk;
                const int e_sum = e_q + head_exponent(head_max_bits[bh]);
                const double f = __hiloint2double((1023 + e_sum - 34) << 20, 0) * g.scale_d;   // score per unit of V
                // |V| <= |q| max|k_j - k_0| 2^(34 - e_sum), 1 % covers the rounding of the norms, 2^26 the digits' own rounding
                const float vmax = sqrtf(q2) * head_norm[bh] * (1.01f / 16777216.f) + 67108864.f;
                int sh = max((int)(__float_as_uint(vmax) >> 23) - 127 + 1 - 31, 0);            // vmax < 2^(31 + sh)
                const bool give_up = !(f <= kMaxScorePerUnit) || sh > kMaxRowShift;            // also non-finite rows
                sh = min(sh, kMaxRowShift);
                row_err[(size_t)it * kTileRows + r] = (float)(f * 1.4426950408889634) * (kFixedErr<D> + (float)(1 << sh));   // and one unit of W
                sm.row_shift[qb][r] = (uint8_t)sh;
                sm.row_scale[qb][r] = give_up ? __int_as_float(0x7fffffff)
                                              : (float)(f * __hiloint2double((1023 + sh) << 20, 0) * 1.4426950408889634);
            }
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // digit planes visible to the tensor core
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&sm.q_sliced[qb]);
            ++n_done;
        }
    } else if (warp < kSlicerWarp0) {
        // ------------------------------------------------------------ epilogue
        const int quarter = warp & 3, part = warp >> 2;
        const uint32_t lane_addr = tbase + ((uint32_t)(quarter * 32) << 16) + part * 16;
        unsigned char* stage = reinterpret_cast<unsigned char*>(&sm.stage[warp][0][0]) + lane * 64;
        const int swz = (lane >> 1) & 3;                              // 64-byte swizzle: chunk ^ (row / 2) % 4
        bool ok = true;
        int c = 0, n_done = 0, it = blockIdx.x;
        for (; it < n_items; it += gridDim.x) {
            const ScoreItem w = score_item(g, item0 + it);
            if (w.n_ct == 0) continue;
            const int qb = n_done & 1;
            const int pos = w.tile * kTileRows + quarter * 32 + lane;
            const int n = slot_live(g, pos) ? n_candidates(g, pos) : 0;
            const int n_warp = __reduce_max_sync(0xffffffffu, n);
            if (!(ok = tc::mbar_wait(&sm.q_sliced[qb], (n_done >> 1) & 1, abort_flag))) break;   // the row's constants are there
            const int sh = sm.row_shift[qb][quarter * 32 + lane];
            const float per_w = sm.row_scale[qb][quarter * 32 + lane];
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&sm.qd_free[qb]);
            const uint32_t m1 = 1u << (16 - sh), m0 = m1 << 8;
            float top = -INFINITY, low = INFINITY;
            for (int ct = 0; ct < w.n_ct; ++ct, ++c) {
                const int s = c & 1;
                if (!(ok = tc::mbar_wait(&sm.acc_full[s], (c >> 1) & 1, abort_flag))) break;
                tc::tc_fence_after_sync();
                const int col0 = ct * kScoreTcCols + part * 16;
                if (col0 < n_warp) {                                  // the box holds a candidate of one of the warp's rows
                    const bool whole = __all_sync(0xffffffffu, col0 + 16 <= n);       // no column beyond a row's candidates
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        uint32_t lv[4][8];
#pragma unroll
                        for (int L = 0; L < 4; ++L) tc::tmem_ld_32x8(lane_addr + s * 256 + L * kScoreTcCols + hf * 8, lv[L]);
                        tc::tmem_wait_ld();
                        if (hf == 0) {
                            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");   // the last box has left
                            __syncwarp();
                        } else {                                      // last read of this accumulator set
                            tc::tc_fence_before_sync();
                            __syncwarp();
                            if (lane == 0) tc::mbar_arrive(&sm.acc_free[s]);
                        }
#pragma unroll
                        for (int c4 = 0; c4 < 2; ++c4) {
                            float sv[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const int e = 4 * c4 + i;
                                sv[i] = (float)shifted_levels((int)lv[0][e], (int)lv[1][e], (int)lv[2][e], (int)lv[3][e], m0, m1, sh) * per_w;
                            }
                            *reinterpret_cast<float4*>(stage + (((hf * 2 + c4) ^ swz) << 4)) = make_float4(sv[0], sv[1], sv[2], sv[3]);
                            if (whole) {
                                top = fmax3(fmax3(top, sv[0], sv[1]), sv[2], sv[3]);
                                low = fmin3(fmin3(low, sv[0], sv[1]), sv[2], sv[3]);
                            } else {
#pragma unroll
                                for (int i = 0; i < 4; ++i)
                                    if (col0 + hf * 8 + c4 * 4 + i < n) { top = fmaxf(top, sv[i]); low = fminf(low, sv[i]); }
                            }
                        }
                    }
                    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        tc::tma_store_2d(&tmS, &sm.stage[warp][0][0], col0, it * kTileRows + quarter * 32);
                        asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
                    }
                } else {
                    tc::tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&sm.acc_free[s]);
                }
            }
            if (!ok) break;
            row_range[kRangeParts * ((size_t)it * kTileRows + quarter * 32 + lane) + part] = make_float2(top, low);
            ++n_done;
        }
        if (!ok) abandon_ranges(row_range, it, n_items, gridDim.x, quarter * 32 + lane, part);
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");   // every box is in global memory
    } else if (warp == kClearWarp) {
        for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
            const ScoreItem w = score_item(g, item0 + it);
            uint32_t* dst = tile_union + ((size_t)(w.b * g.Hq + w.h) * g.n_tiles_cap + w.tile) * g.n_words;
            for (int i = lane; i < g.n_words; i += 32) dst[i] = 0u;
        }
    }
    // ---------------------------------------------------------------- teardown
    tc::tc_fence_before_sync();
    __syncthreads();
    if (tid == 0 && sm.abort_flag) atomicExch(status, 6);
    if (warp == kProducerWarp) tc::tmem_dealloc<512>(tbase);
}

}  // namespace adaspark
