// K3b: nucleus selection (Eq. 2) from the scores of score_tc.cuh, G lanes of a warp per query row.
//
// Scores s_j are in log2 units; the order is descending score, then ascending cube index, the mass of a cube is
// 2^(s_j - max).  A row's scores stay in registers (kK per lane) and are swept twice:
//   sweep 1  masses are added to the row's total Z and, quantised, to a histogram over the distance from the maximum
//            in shared memory (16 G buckets from the largest score to the smallest): the bucket in which the cumulative
//            mass crosses p Z is found from it
//   sweep 2  cubes before that bucket are selected (one bit each, collected from the sign of a subtraction) and their
//            exact mass is summed; the few cubes inside it (widened by kGuard at both ends) are listed, and each
//            learns the cumulative mass up to it: it is selected if the mass before it has not reached p Z
// A bucket with more than kSelectCand cubes is split by further histograms over its cubes alone (rare, slow path).
// Top-K (kCount): the same with every mass = 1 and a target of min(top_k, candidates).
//
// From p = 1/2 on everything runs from the other end (kTail): the order is ascending, the target (1 - p) Z, "before" is what
// is rejected, and a cube is rejected if the mass up to and including it does not exceed the target.  Masses, sums and their
// errors are then those of the 1 - p that is left out.
//
// Everything here is fp32, so a row is decided here only if its boundary is clear of what fp32 can be off by, and
// handed to the fp64 kernel (list in the workspace) otherwise:
//   - a cumulative mass within eps of the target.  With R the row's spread, S its largest |score| (relative to cube 0's: at
//     most R) and rho what the fixed point leaves open in a score, one unit of W included (row_err), a score's distance from
//     the maximum is off by rho + 2 (R + S) 2^-24 (R: the roundings of the factor of W and of the difference, S: of W and of the
//     product) and a mass by e = ln 2 times that plus 2^-22 (ex2.approx).  Masses off by e, of whatever signs, move a share q by at most
//     2 q (1 - q) e; a sum in which no term passes through more than a additions is off by a 2^-24.  With q the smaller of p and
//     1 - p:  eps = q Z (2 (1 - q) e + (additions of Z, of the base and of the list + 2) 2^-24).
//   - a last selected cube and a first rejected one, listed or not, that lie less than 2 rho + 4 |s| 2^-24 apart and are not
//     copies of one cube.  (For the unlisted ones the edge of the first bucket stands, and what finer buckets leave out.)
// That is one row in 10^4 to 10^3 on the benchmark inputs, and no more with p nearer to 1 (sums up to p Z and an eps in
// proportion to Z left 0.7 / 2.1 / 5.5 % undecided at p = 0.99 / 0.999 / 0.9999, 65536 tokens).  With them go the rows the score
// kernel marked, and rows with more equal scores at the boundary than the list holds.
//
// What bounds it: instruction issue at few candidates (about 20 instructions per score of a lane in the two sweeps and 900
// per pass of 32 / G rows beside them; 1390 per pass with 128 to 256 candidates, issue slots 63 % used, 1000 with fewer, 80 %),
// the stream of scores from memory at many (4 bytes per pair).  Sharing a warp among
// 32 / G rows spreads the second figure over several rows; the per-cube work is spread over the pipes (the bits come
// from funnel shifts of signs, the mass before the bucket from a saturating multiply, the exponential from the MUFU unit,
// the rest from packed fp32 pairs), because the integer / comparison pipe issues at half the rate of the fp32 pipe.
// Measured, scoring and selection together, 28 heads, against one kernel that recomputed the scores in every pass: 0.78 ->
// 0.354 ms at 16384 tokens and 256 cubes, 13.6 -> 4.4 at 65536 and 1024, 59.5 -> 25.3 at 131072 and 2048, half static.
#pragma once
#include <cmath>
#include <cstring>

#include "score_tc.cuh"

namespace adaspark {

constexpr int kSelectThreads = 256;
constexpr int kSelectRows = 8;           // consecutive rows of a warp: its mask words fill 32-byte sectors
constexpr int kSelectWarps = kSelectThreads / 32;
constexpr int kSelectCand = 32;          // cubes of the crossing bucket a row may list
constexpr int kMaxHistLevels = 8;        // histograms of a row before it is handed to the fp64 kernel
constexpr float kUlp = 5.9604645e-8f;    // 2^-24: the largest relative error of a rounding
constexpr float kGuard = 1e-3f;          // of a bucket
constexpr int kSumSteps = 8;             // steps of a lane (2 additions each) whose masses are summed before they join the rest
enum SelectRule { kHead, kTail, kCount };                 // Top-p from the front and from the other end, Top-K

// What a row is decided by (the same for all rows of a launch).
struct SelectTarget {
    double share;      // the target, of Z
    float eps_mass;    // 1.01 x 2 q (1 - q): eps per Z and error of a mass
    float eps_add;     // 1.01 q 2^-24: and per addition
    float unit;        // masses are counted in 1 / unit
    float q_unit;      // 2^-149 unit: a mass times it has the bits of mass x unit, rounded, up to 2^24 (a subnormal or the first binade)
};
// capacity: the scores that the kernel's shape holds.  2^head_bits: all of them, of mass 1, fit 32 bits.  From the tail the
// sums need to fit up to the target only (what comes after it may wrap), and with p near 1 the masses that matter are small:
// the target, at most q x capacity, stays below 2^31 units and, where single masses pass 2^24 units, below those.  A mass of
// more than 2^24 units is counted as less, but as more than the target.  A histogram that misleads costs a row its decision,
// no more.
inline SelectTarget select_target(SelectRule rule, double top_p, int capacity, int head_bits) {
    SelectTarget t;
    t.share = rule == kCount ? 0.0 : rule == kTail ? 1.0 - top_p : top_p;
    int bits = rule == kCount ? 0 : head_bits;
    if (rule == kTail) {
        const int il = std::ilogb(t.share * capacity), linear = 30 - il < 24 ? 30 - il : 24;
        bits = 23 - il > linear ? 23 - il : linear;
    }
    t.eps_mass = (float)(2.02 * t.share * (1.0 - t.share));
    t.eps_add = (float)(1.01 * t.share) * kUlp;
    t.unit = std::ldexp(1.f, bits);
    const uint32_t q_bits = bits < 23 ? 1u << bits : (uint32_t)(bits - 22) << 23;      // (by its bits: the host may flush subnormals)
    std::memcpy(&t.q_unit, &q_bits, 4);
    return t;
}

// Lanes per row grow with the candidate count, and the buckets with the lanes: a bucket holds at most about 5 of 256
// cubes (G = 8), 512 (16) or 1024 (32) with normally distributed scores.
// Shared memory of one warp; its mask words [n_words][8 rows] follow those of all warps.
template <int G, int kK>
struct SelectWarpSmem {
    float rows[32 / G][G * kK];                           // scores of the rows of a pass
    float4 range[32 / G][2];                              // partial ranges of the rows of a pass
    uint32_t hist[512];                                   // [bucket][row of the warp]
    float4 cand[32 / G][kSelectCand];                     // score, mass, cube
    float err[2][32 / G];                                 // row_err of this pass and of the next
    int32_t count[32 / G];
};
__host__ __device__ inline size_t select_smem_bytes(size_t warp_bytes, int n_words) {
    return kSelectWarps * (warp_bytes + (size_t)n_words * kSelectRows * 4);
}

__device__ __forceinline__ float sat_fma(float a, float b, float c) {     // min(max(a b + c, 0), 1)
    return __saturatef(fmaf(a, b, c));
}

// One warp per 8 rows of a tile, warps work on their own: 2 CTAs per item, items [first, ..) of those that the scores were
// computed for.  scores / row_range / row_err: what score_tc_kernel left for the items [item0, ..).
// tile_mask as mask_index() describes; tile_union (cleared) receives the OR of each word over the tile's rows;
// fallback_rows[0 .. *fallback_count) receives ((b*Hq+h)*n_tiles_cap + tile)*128 + r of the rows left to the fp64
// kernel.  G * kK >= the largest candidate count of these items.
template <int G, int kK, int kResident, SelectRule kRule>
__global__ void __launch_bounds__(kSelectThreads, kResident) select_nucleus_kernel(
    Geom g, SelectTarget rule, int item0, int first, const float* scores, const float4* row_range, const float* row_err, uint32_t* tile_mask, uint32_t* tile_union,
    const unsigned long long* key_hash, uint32_t* sel_bitmap, int32_t* sel_count, int32_t* fallback_rows, uint32_t* fallback_count) {
    extern __shared__ __align__(16) unsigned char select_raw[];
    constexpr int R = 32 / G, kBuckets = 16 * G, kSteps = kK / 4;          // rows per warp; steps of 4 columns per lane
    constexpr int kMasks = (kK + 31) / 32;                                 // bit words per lane
    constexpr bool kByCount = kRule == kCount, tail = kRule == kTail;
    constexpr int kBlocks = (kSteps + kSumSteps - 1) / kSumSteps;
    constexpr int kAdds = kK / 2 / kBlocks + kBlocks + (G == 8 ? 3 : G == 16 ? 4 : 5);    // a mass passes through, in a row's sum
    constexpr uint32_t kFull = 0xffffffffu;
    constexpr float kMagic = 8388608.f;                                    // 2^23: low mantissa bits = the integer part
    constexpr uint32_t kMagicBits = 0x4B000000u;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int s = lane & (G - 1), row_w = lane / G;                        // lane inside the row's group, row of the warp
    const int item = first + (blockIdx.x >> 1), row0 = ((blockIdx.x & 1) * kSelectWarps + warp) * kSelectRows;   // first row of the warp
    const ScoreItem w = score_item(g, item0 + item);
    const size_t gt_cap = (size_t)(w.b * g.Hq + w.h) * g.n_tiles_cap + w.tile;
    const int n_words_live = min(2 * w.n_ct, g.n_words);                   // words that can hold a candidate
    SelectWarpSmem<G, kK>& sm = reinterpret_cast<SelectWarpSmem<G, kK>*>(select_raw)[warp];
    uint32_t* words = reinterpret_cast<uint32_t*>(select_raw + kSelectWarps * sizeof(SelectWarpSmem<G, kK>)) + (size_t)warp * g.n_words * kSelectRows;
    uint32_t* hist = sm.hist;
#pragma unroll
    for (int u = 0; u < 4; ++u) reinterpret_cast<uint4*>(hist)[lane + 32 * u] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = lane; i < n_words_live * kSelectRows; i += 32) words[i] = 0u;
    __syncwarp();
    launch_dependents();
    wait_for_previous_kernel();

    constexpr float a_add0 = tail ? (float)(kBuckets - 1) : 0.f;
    auto group_sum = [&](float x) -> float {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
        return x;
    };
    auto group_any = [&](bool p) -> bool {
        const uint32_t m = __ballot_sync(kFull, p);
        return ((G == 32 ? m : (m >> (row_w * G)) & ((1u << (G & 31)) - 1u))) != 0u;
    };
    // The scores of a pass come through shared memory, requested while the pass before is still being decided (a warp
    // that loaded them when it needed them spent half of its time waiting, with 32 warps on the SM).
    auto candidates = [&](int pass) -> int {
        const int pos = w.tile * kTileRows + row0 + pass * R + row_w;
        return slot_live(g, pos) ? n_candidates(g, pos) : 0;
    };
    auto request = [&](int pass, int n) {
        const size_t srow = (size_t)item * kTileRows + row0 + pass * R + row_w;
        const float* src = scores + srow * g.N_ld + 4 * s;
        float* dst = &sm.rows[row_w][4 * s];
#pragma unroll
        for (int c = 0; c < kSteps; ++c)
            if (c * 4 * G + 4 * s < n) cp_async_16(dst + c * 4 * G, src + c * 4 * G);
        if (s < 2 && n > 0) cp_async_16(&sm.range[row_w][s], row_range + 2 * srow + s);
        if (s == 2 && n > 0) cp_async_4(&sm.err[pass & 1][row_w], row_err + srow);
        cp_async_commit();
    };
    int n_next = candidates(0);
    request(0, n_next);
#pragma unroll 1
    for (int pass = 0; pass < kSelectRows / R; ++pass) {
        const int rl = pass * R + row_w, r = row0 + rl;
        const int n = n_next;
        const int n_most = __reduce_max_sync(kFull, n), n_least = __reduce_min_sync(kFull, n);
        cp_async_wait<0>();
        __syncwarp();
        n_next = pass + 1 < kSelectRows / R ? candidates(pass + 1) : 0;
        if (n_most == 0) {
            request(pass + 1, n_next);
            continue;
        }
        // ---- the row's scores (column 4 G c + 4 s + i in v[4 c + i]), largest and smallest
        const float* row_scores = sm.rows[row_w];
        float v[kK];
#pragma unroll
        for (int c = 0; c < kSteps; ++c) {
            float4 x = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            if (c * 4 * G < n_most) {
                const int col = c * 4 * G + 4 * s;
                if (col < n) x = *reinterpret_cast<const float4*>(row_scores + col);
                if ((c + 1) * 4 * G > n_least) {                           // the end of a row's candidates
                    if (col + 1 >= n) x.y = -INFINITY;
                    if (col + 2 >= n) x.z = -INFINITY;
                    if (col + 3 >= n) x.w = -INFINITY;
                }
            }
            v[4 * c] = x.x; v[4 * c + 1] = x.y; v[4 * c + 2] = x.z; v[4 * c + 3] = x.w;
        }
        float top = 0.f, low = 0.f;
        if (n > 0) {
            const float4 ra = sm.range[row_w][0], rb = sm.range[row_w][1];
            top = fmaxf(fmaxf(ra.x, ra.z), fmaxf(rb.x, rb.z));
            low = fminf(fminf(ra.y, ra.w), fminf(rb.y, rb.w));
        }
        bool give_up = n > 0 && !(top > -INFINITY && low > -INFINITY);     // marked by the score kernel
        if (give_up) {
            top = low = 0.f;
#pragma unroll
            for (int e = 0; e < kK; ++e) v[e] = -INFINITY;
        }
        const int n_whole = __any_sync(kFull, give_up) ? 0 : n_least;      // columns below are scores in every row of the warp
        // mass of a score at d = s - max
        auto mass = [&](float d) -> float { return kByCount ? (d > -INFINITY ? 1.f : 0.f) : fast_exp2(d); };

        // ---- sweep 1: Z and the histogram over u = (max - s) * per_unit, or from the other end, bucket = round(u): the
        // buckets span the row
        const float per_unit = fminf((float)(kBuckets - 1) / (top - low), 1e18f);
        float a_mul = tail ? per_unit : -per_unit, a_add = a_add0;         // u = d * a_mul + a_add
        float z = 0.f;
        uint32_t* my_hist = hist + row_w;
        const uint32_t hist_addr = smem_u32(my_hist) - kMagicBits * (4u * R);   // plus 4 R times the bits of 2^23 + bucket
        auto add_to_bucket = [&](uint32_t bucket_bits, uint32_t q) {
            asm volatile("red.shared.add.u32 [%0], %1;\n" ::"r"(hist_addr + bucket_bits * (4u * R)), "r"(q) : "memory");
        };
        {
            unsigned long long z2 = 0ull, zs2 = 0ull;                      // of all steps, of the last few
            const unsigned long long neg_top2 = pack_f32x2(-top, -top), a_mul2 = pack_f32x2(a_mul, a_mul);
            const unsigned long long magic2 = pack_f32x2(kMagic + a_add0, kMagic + a_add0), q_unit2 = pack_f32x2(rule.q_unit, rule.q_unit);
#pragma unroll
            for (int c = 0; c < kSteps; ++c) {
                if ((c + 1) * 4 * G <= n_whole) {
#pragma unroll
                    for (int i = 0; i < 4; i += 2) {
                        const unsigned long long d2 = add_f32x2(pack_f32x2(v[4 * c + i], v[4 * c + i + 1]), neg_top2);
                        float d0, d1, b0, b1;
                        unpack_f32x2(d2, d0, d1);
                        v[4 * c + i] = d0;
                        v[4 * c + i + 1] = d1;
                        unpack_f32x2(fma_f32x2(d2, a_mul2, magic2), b0, b1);
                        if (kByCount) {
                            z += 2.f;
                            add_to_bucket(__float_as_uint(b0), 1u);
                            add_to_bucket(__float_as_uint(b1), 1u);
                        } else {
                            const unsigned long long m2 = pack_f32x2(mass(d0), mass(d1));
                            zs2 = add_f32x2(zs2, m2);
                            float q0, q1;
                            unpack_f32x2(mul_f32x2(m2, q_unit2), q0, q1);
                            add_to_bucket(__float_as_uint(b0), __float_as_uint(q0));
                            add_to_bucket(__float_as_uint(b1), __float_as_uint(q1));
                        }
                    }
                } else if (c * 4 * G < n_most) {                           // some columns hold no candidate (-inf: no mass)
#pragma unroll
                    for (int i = 0; i < 4; i += 2) {
                        float m[2];
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            const float d = v[4 * c + i + k] - top;
                            v[4 * c + i + k] = d;
                            m[k] = mass(d);
                            const float u01 = sat_fma(d, a_mul * (1.f / (kBuckets - 1)), tail ? 1.f : 0.f);
                            add_to_bucket(__float_as_uint(fmaf(u01, (float)(kBuckets - 1), kMagic)), __float_as_uint(m[k] * rule.q_unit));
                        }
                        zs2 = add_f32x2(zs2, pack_f32x2(m[0], m[1]));
                    }
                }
                if (c % kSumSteps == kSumSteps - 1 || c == kSteps - 1) {
                    z2 = c < kSumSteps ? zs2 : add_f32x2(z2, zs2);
                    zs2 = 0ull;
                }
            }
            float z0, z1;
            unpack_f32x2(z2, z0, z1);
            z += z0 + z1;
        }
        z = group_sum(z);
        const float target = kByCount ? fminf(z, (float)g.top_k) : (float)((double)z * rule.share);
        float base = 0.f;                                                  // mass before the bucket
        float to_edge = 0.f;                                               // u + this = 0: the edge of the first bucket on the rejected side
        float beyond = -INFINITY;                                          // my largest rejected score of that bucket that is not listed
        int adds = 2 * kAdds + 2;
        uint32_t before[kMasks], inside[kMasks];                           // per lane: bit e = its e-th score
#pragma unroll
        for (int k = 0; k < kMasks; ++k) { before[k] = 0u; inside[k] = 0u; }
        bool unsure = false;
        bool active = n > 0 && !give_up;                                   // the row still narrows its interval
        int n_cand = 0;
#pragma unroll 1
        for (int level = 0;; ++level) {
            __syncwarp();
            // ---- the bucket in which the cumulative (quantised) mass crosses the target: first the lane whose 16
            // buckets hold it, then the bucket (read in an order of its own by each lane: no bank is met twice)
            uint32_t sum = 0u;
#pragma unroll
            for (int u = 0; u < 16; ++u) sum += my_hist[(s * 16 + (u ^ (s & 15))) * R];
            uint32_t incl = sum;
#pragma unroll
            for (int o = 1; o < G; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, incl, o, G);
                if (s >= o) incl += t;
            }
            const uint32_t thr = max((uint32_t)fmaxf((target - base) * rule.unit, 0.f), 1u);
            uint32_t over = __ballot_sync(kFull, incl >= thr);
            if (G < 32) over = (over >> (row_w * G)) & ((1u << (G & 31)) - 1u);
            const int own = over ? __ffs(over) - 1 : G - 1;
            const uint32_t cum = __shfl_sync(kFull, incl - sum, own, G);
            constexpr int kPer = 16 / (G < 16 ? G : 16);                   // buckets per lane in the second step
            uint32_t part[kPer], psum = 0u;
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                part[u] = s * kPer < 16 ? my_hist[(own * 16 + (s & 15) * kPer + u) * R] : 0u;
                psum += part[u];
            }
            uint32_t pincl = psum;
#pragma unroll
            for (int o = 1; o < (G < 16 ? G : 16); o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, pincl, o, G);
                if (s >= o) pincl += t;
            }
            over = __ballot_sync(kFull, s * kPer < 16 && cum + pincl >= thr);
            if (G < 32) over = (over >> (row_w * G)) & ((1u << (G & 31)) - 1u);
            const int own2 = over ? __ffs(over) - 1 : (G < 16 ? G : 16) - 1;
            int cb = s * kPer;
            if (kPer == 2 && cum + (pincl - psum) + part[0] < thr) ++cb;
            cb = __shfl_sync(kFull, cb, own2, G) + own * 16;
            __syncwarp();
#pragma unroll
            for (int u = 0; u < 4; ++u) reinterpret_cast<uint4*>(hist)[lane + 32 * u] = make_uint4(0u, 0u, 0u, 0u);
            // ---- sweep 2: before / inside the bucket [cb - 1/2, cb + 1/2], widened by the guard
            const float lo_u = (float)cb - (0.5f + kGuard);
            const float hi_u = (float)cb + (0.5f + kGuard);
            float add = 0.f;
            n_cand = 0;
            if (level == 0) {
                const unsigned long long a_mul2 = pack_f32x2(a_mul, a_mul), lo2 = pack_f32x2(a_add0 - lo_u, a_add0 - lo_u);
                const unsigned long long width2 = pack_f32x2(lo_u - hi_u, lo_u - hi_u);
                unsigned long long add2 = 0ull, adds2 = 0ull;              // of all steps, of the last few
#pragma unroll
                for (int c = kSteps - 1; c >= 0; --c) {
                    if (c * 4 * G < n_most) {
#pragma unroll
                        for (int i = 2; i >= 0; i -= 2) {
                            const float d0 = v[4 * c + i], d1 = v[4 * c + i + 1];
                            const int k = (4 * c + i) >> 5;
                            const unsigned long long u2 = fma_f32x2(pack_f32x2(d0, d1), a_mul2, lo2);
                            float ua0, ua1, ub0, ub1;
                            unpack_f32x2(u2, ua0, ua1);
                            unpack_f32x2(add_f32x2(u2, width2), ub0, ub1);
                            before[k] = __funnelshift_l(__float_as_uint(ua1), before[k], 1);
                            before[k] = __funnelshift_l(__float_as_uint(ua0), before[k], 1);
                            inside[k] = __funnelshift_l(__float_as_uint(ub1), inside[k], 1);
                            inside[k] = __funnelshift_l(__float_as_uint(ub0), inside[k], 1);
                            // the mass of what lies before: times 2^100 and clamped, the distance is 1 before and 0 else
                            adds2 = fma_f32x2(pack_f32x2(mass(d0), mass(d1)),
                                              pack_f32x2(__saturatef(ua0 * -1.2676506e30f), __saturatef(ua1 * -1.2676506e30f)), adds2);
                        }
                    }
                    if (c % kSumSteps == 0) {
                        add2 = c + kSumSteps >= kSteps ? adds2 : add_f32x2(add2, adds2);
                        adds2 = 0ull;
                    }
                }
                float add0, add1;
                unpack_f32x2(add2, add0, add1);
                add = add0 + add1;
#pragma unroll
                for (int k = 0; k < kMasks; ++k) inside[k] &= ~before[k];
            } else {
                int n_add = 0;
                for (int k = 0; k < kMasks; ++k) {
                    uint32_t bits = active ? inside[k] : 0u;
                    while (bits) {
                        const int e = __ffs(bits) - 1;
                        bits &= bits - 1u;
                        const float x = row_scores[((k * 32 + e) >> 2) * 4 * G + 4 * s + (e & 3)], d = x - top;
                        const float u = fmaf(d, a_mul, a_add);
                        if (u < lo_u) { before[k] |= 1u << e; inside[k] &= ~(1u << e); add += mass(d); ++n_add; }
                        else if (!(u < hi_u)) inside[k] &= ~(1u << e);
                        else continue;
                        if (tail ? u < lo_u : !(u < lo_u)) beyond = fmaxf(beyond, x);
                    }
                }
                adds += __reduce_max_sync(kFull, n_add) + 6;               // (the lane's, its group's and the base's)
            }
#pragma unroll
            for (int k = 0; k < kMasks; ++k) n_cand += __popc(inside[k]);
            add = group_sum(add);
            if (G == 32) {
                n_cand = __reduce_add_sync(kFull, n_cand);
            } else {
#pragma unroll
                for (int o = G / 2; o > 0; o >>= 1) n_cand += __shfl_xor_sync(kFull, n_cand, o);
            }
            if (active) {
                base += add;
                if (level == 0) to_edge = a_add - (tail ? lo_u : hi_u);
            }
            if (n_cand <= kSelectCand) active = false;
            if (active && level + 1 == kMaxHistLevels) { give_up = true; active = false; }
            if (!__any_sync(kFull, active)) break;
            // ---- rare: split the bucket of the rows that hold too many cubes in it
            constexpr float fine = (float)(kBuckets - 1) / (1.f + 2.f * kGuard);
            if (active) {
                a_add = (a_add - lo_u) * fine;
                a_mul = a_mul * fine;
                if (!(fabsf(a_mul) < 1e30f)) { give_up = true; active = false; }
            }
            for (int k = 0; k < kMasks; ++k) {
                uint32_t bits = active ? inside[k] : 0u;
                while (bits) {
                    const int e = __ffs(bits) - 1;
                    bits &= bits - 1u;
                    const float d = row_scores[((k * 32 + e) >> 2) * 4 * G + 4 * s + (e & 3)] - top;
                    const float u01 = sat_fma(d, a_mul * (1.f / (kBuckets - 1)), a_add * (1.f / (kBuckets - 1)));
                    const uint32_t b = __float_as_uint(fmaf(u01, (float)(kBuckets - 1), kMagic)) - kMagicBits;
                    atomicAdd(&my_hist[b * R], __float_as_uint(mass(d) * rule.q_unit));
                }
            }
            __syncwarp();
        }
        // ---- list the cubes inside the bucket
        const bool decide = n > 0 && !give_up;
        const int n_list = decide ? n_cand : 0;
        const int n_list_most = __reduce_max_sync(kFull, n_list);
        if (s == 0) sm.count[row_w] = 0;
        for (int i = n_list + s; i < n_list_most; i += G) sm.cand[row_w][i] = make_float4(-INFINITY, 0.f, 0.f, 0.f);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < kMasks; ++k) {
            uint32_t bits = decide ? inside[k] : 0u;
            int slot = bits ? atomicAdd(&sm.count[row_w], __popc(bits)) : 0;
            while (bits) {
                const int e = __ffs(bits) - 1;
                bits &= bits - 1u;
                const int j = ((k * 32 + e) >> 2) * 4 * G + 4 * s + (e & 3);
                const float x = row_scores[j];
                sm.cand[row_w][slot++] = make_float4(x, mass(x - top), __int_as_float(j), 0.f);
            }
        }
        __syncwarp();
        request(pass + 1, n_next);                                         // the rows' scores are no longer read
        // ---- the words of what lies before the bucket, or else of what is neither before nor inside it: lane s holds nibble
        // s & 7 of words (s >> 3) + c G / 8
#pragma unroll
        for (int k = 0; k < kMasks; ++k) {
            uint32_t t = tail ? before[k] | inside[k] : before[k];         // nibble c: columns of step 8 k + c
            // transpose the 8 x 8 nibbles of 8 neighbouring lanes: lane c then holds word c
            uint32_t o = __shfl_xor_sync(kFull, t, 4);
            t = (s & 4) ? ((t & 0xffff0000u) | (o >> 16)) : ((t & 0x0000ffffu) | (o << 16));
            o = __shfl_xor_sync(kFull, t, 2);
            t = (s & 2) ? ((t & 0xff00ff00u) | ((o >> 8) & 0x00ff00ffu)) : ((t & 0x00ff00ffu) | ((o << 8) & 0xff00ff00u));
            o = __shfl_xor_sync(kFull, t, 1);
            t = (s & 1) ? ((t & 0xf0f0f0f0u) | ((o >> 4) & 0x0f0f0f0fu)) : ((t & 0x0f0f0f0fu) | ((o << 4) & 0xf0f0f0f0u));
            const int wd = (8 * k + (s & 7)) * (G / 8) + (s >> 3);
            if (tail) {
                t = ~t & __funnelshift_lc(0xffffffffu, 0u, max(n - wd * 32, 0));   // of the row's candidates in the word
            }
            if (wd < n_words_live && decide) words[wd * kSelectRows + rl] = t;
        }
        __syncwarp();
        // ---- each listed cube: the mass before it and with it
        const float err = n > 0 ? sm.err[pass & 1][row_w] : 0.f;
        const float mass_err = fmaf(0.6931472f, fmaf(2.f * kUlp, (top - low) + fmaxf(top, -low), err), 4.f * kUlp);
        const float eps = kByCount ? 0.f : z * fmaf(rule.eps_mass, mass_err, rule.eps_add * (float)(adds + n_list));
        float last = INFINITY, next = -INFINITY;                           // lowest selected, highest rejected score of my cubes
        bool reached = false;
        for (int i0 = 0; i0 < n_list_most; i0 += G) {
            const int i = i0 + s;
            const bool mine = i < n_list;
            const float4 me = sm.cand[row_w][min(i, n_list_most - 1)];
            const int ji = __float_as_int(me.z);
            float acc = base;                                              // and the listed cubes before mine
            for (int k = 0; k < n_list_most; ++k) {
                const float4 ck = sm.cand[row_w][k];
                const bool earlier = tail ? ck.x < me.x || (ck.x == me.x && __float_as_int(ck.z) > ji)
                                          : ck.x > me.x || (ck.x == me.x && __float_as_int(ck.z) < ji);
                if (earlier) acc += ck.y;
            }
            if (mine) {
                if (tail ? acc + me.y > target : acc < target) {
                    atomicOr(&words[(ji >> 5) * kSelectRows + rl], 1u << (ji & 31));
                    last = fminf(last, me.x);
                } else {
                    next = fmaxf(next, me.x);
                }
                reached = reached || (tail ? acc + me.y > target : acc + me.y >= target);
                if (!kByCount) unsure = unsure || fabsf(acc - target) <= eps || fabsf(acc + me.y - target) <= eps;
            }
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
            last = fminf(last, __shfl_xor_sync(kFull, last, o));
            next = fmaxf(next, __shfl_xor_sync(kFull, next, o));
        }
        const float gap = fmaf(4.f * kUlp, fabsf(last), 2.f * err);
        // an unlisted cube lies beyond the edge (u is off by a small part of the guard) or has been looked at
        unsure = unsure || (n_list < n && fabsf(fmaf(last - top, tail ? per_unit : -per_unit, to_edge)) <= fmaf(gap, per_unit, 0.5f * kGuard));
        if (__any_sync(kFull, beyond > -INFINITY)) {
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) beyond = fmaxf(beyond, __shfl_xor_sync(kFull, beyond, o));
            unsure = unsure || last - beyond <= gap;
        }
        bool tied = last < INFINITY && last - next <= gap;                 // (a row without a listed cube that is selected is unsure)
        if (__any_sync(kFull, tied)) {
            // The boundary runs through cubes whose order these scores cannot tell.  If they are copies of one cube (frames
            // that repeat: the mean keys are equal bit by bit) their scores are equal in fp64 too and the index orders them.
            // (All such rows went to the fp64 kernel: every frame twice, 65536 tokens, 57.8 instead of 4.3 ms of selection.)
            const unsigned long long* hash = key_hash + (size_t)(w.b * g.Hkv + w.gk) * g.N_ld;
            unsigned long long h_min = ~0ull, h_max = 0ull;
            for (int i = s; i < n_list; i += G) {
                const float4 me = sm.cand[row_w][i];
                if (last - me.x <= gap && me.x - next <= gap) {
                    const unsigned long long hj = hash[__float_as_int(me.z)];
                    h_min = min(h_min, hj);
                    h_max = max(h_max, hj);
                }
            }
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) {
                h_min = min(h_min, __shfl_xor_sync(kFull, h_min, o));
                h_max = max(h_max, __shfl_xor_sync(kFull, h_max, o));
            }
            tied = tied && h_min != h_max;
        }
        unsure = unsure || tied || !(last < INFINITY);
        const bool any_unsure = group_any(unsure), any_reached = group_any(reached);   // both by all lanes
        unsure = any_unsure || !any_reached || !(tail ? base <= target : base < target);
        if (n > 0 && (give_up || unsure)) {
            for (int wd = s; wd < n_words_live; wd += G) words[wd * kSelectRows + rl] = 0u;
            if (s == 0) fallback_rows[atomicAdd(fallback_count, 1u)] = (int32_t)(gt_cap * kTileRows + r);
        }
        __syncwarp();
    }
    // ---- mask words (32-byte sectors of 8 rows), union words, the caller's copies
    for (int i0 = 0; i0 < g.n_words * 2; i0 += 32) {
        const int wd = (i0 + lane) >> 1, c4 = lane & 1;
        const uint4 val = wd < n_words_live ? *reinterpret_cast<const uint4*>(&words[wd * kSelectRows + c4 * 4]) : make_uint4(0u, 0u, 0u, 0u);
        if (wd < g.n_words)
            *reinterpret_cast<uint4*>(tile_mask + (gt_cap * g.n_words + wd) * kTileRows + row0 + c4 * 4) = val;
        uint32_t u = (val.x | val.y) | (val.z | val.w);                    // OR over the two lanes of the word
        u |= __shfl_xor_sync(kFull, u, 1);
        if (c4 == 0 && u) atomicOr(tile_union + gt_cap * g.n_words + wd, u);
    }
    if (sel_bitmap != nullptr || sel_count != nullptr) {
        for (int rl = 0; rl < kSelectRows; ++rl) {
            const int pos = w.tile * kTileRows + row0 + rl;
            if (!slot_live(g, pos)) continue;
            const size_t raster_row = (size_t)(w.b * g.Hq + w.h) * g.S_io + (pos_to_io(g, pos) - g.pos_begin);
            int cnt = 0;
            for (int wd = lane; wd < g.n_words; wd += 32) {
                const uint32_t word = wd < n_words_live ? words[wd * kSelectRows + rl] : 0u;
                cnt += __popc(word);
                if (sel_bitmap) sel_bitmap[raster_row * g.n_words + wd] = word;
            }
            cnt = __reduce_add_sync(kFull, cnt);
            if (sel_count && lane == 0) sel_count[raster_row] = cnt;
        }
    }
}

// p >= 1 without Top-K: every candidate cube is selected (Eq. 2 with p = 1).  grid (tiles of the call, Hq, B),
// 128 threads = rows of the tile.
__global__ void __launch_bounds__(128) select_all_kernel(Geom g, uint32_t* tile_mask, uint32_t* tile_union,
                                                         uint32_t* sel_bitmap, int32_t* sel_count) {
    launch_dependents();
    wait_for_previous_kernel();
    const int tile = blockIdx.x + g.tile_begin, h = blockIdx.y, b = blockIdx.z, r = threadIdx.x;
    const int pos = tile * kTileRows + r;
    const bool live = slot_live(g, pos);
    const int n = live ? n_candidates(g, pos) : 0;
    const size_t gt_cap = (size_t)(b * g.Hq + h) * g.n_tiles_cap + tile;
    const size_t raster_row = live ? (size_t)(b * g.Hq + h) * g.S_io + (pos_to_io(g, pos) - g.pos_begin) : 0;
    const int n_max = tile_max_candidates(g, tile);
    for (int w = 0; w < g.n_words; ++w) {
        const int rem = n - w * 32;
        const uint32_t word = rem >= 32 ? 0xffffffffu : (rem > 0 ? (1u << rem) - 1u : 0u);
        tile_mask[(gt_cap * g.n_words + w) * kTileRows + r] = word;
        if (sel_bitmap && live) sel_bitmap[raster_row * g.n_words + w] = word;
        if (r == 0) {
            const int remx = n_max - w * 32;
            tile_union[gt_cap * g.n_words + w] = remx >= 32 ? 0xffffffffu : (remx > 0 ? (1u << remx) - 1u : 0u);
        }
    }
    if (sel_count && live) sel_count[raster_row] = n;
}

}  // namespace adaspark
