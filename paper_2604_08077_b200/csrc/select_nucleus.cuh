// K3b: nucleus selection (Eq. 2) from the scores of score_tc.cuh, R query rows at a time per warp.
//
// Scores s_j are in log2 units; the order is descending score, then ascending cube index, the mass of a cube is
// 2^(s_j - max).  A row's scores lie in shared memory and are swept twice by its 32 / R lanes:
//   sweep 1  masses are added to the row's total Z and, quantised, to a histogram over the distance from the maximum
//            in shared memory (from the largest score to the smallest): the bucket in which the cumulative
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
// That is one row in 10^4 to 10^3 on the benchmark inputs (the more cubes, the smaller the masses at the boundary: 0.8 % with 4096 cubes),
// and no more with p nearer to 1 (sums up to p Z and an eps in
// proportion to Z left 0.7 / 2.1 / 5.5 % undecided at p = 0.99 / 0.999 / 0.9999, 65536 tokens).  With them go the rows the score
// kernel marked, and rows with more equal scores at the boundary than the list holds.
//
// What bounds it: latency and instruction issue.  An SM holds 16 or 17 warps (24 in the shape for 128 candidates, 9 in that for 4096), as many
// as the scores of their rows leave room for, and issues in 58 to 70 % of the cycles (42 % with 9 warps): 18 to 20 instructions per score of
// a lane in the two sweeps and 820 to 1100 per pass of R rows beside them (ncu; 77 a row for 64 candidates, 843 for 730).  Lane = row + R x (which
// of the row's lanes): the histogram [bucket][row] is met by neighbouring lanes in different banks, the bits of 8 columns are a
// byte of the mask words without an exchange, and what is done per row (boundary, list, order of the list) is done for R rows at
// once.  (With the lanes side by side on 1 to 4 rows per pass and the scores in registers, 1000 to 1400 instructions a pass, shuffles
// for every row sum and nibbles transposed between lanes: selection kernels alone, us, before / now: 64 candidates 105 / 53, 128 to
// 256 120 / 86 (28 heads, 16384 tokens), 1024 1683 / 1263 (65536 tokens), 2048 13470 / 8950 (131072, half static); with scores and
// fp64 rows, 4096 cubes of 65536 tokens 23.1 / 16.3 ms.)  The per-cube work
// is spread over the pipes: the bits come from funnel shifts of signs, the mass before the bucket from a saturating multiply, the
// exponential from the MUFU unit, the rest from packed fp32 pairs, because the integer / comparison pipe issues at half the
// rate of the fp32 pipe.
// Rows per pass: twice as many (half as many warps on the SM) 72 / 121 / 1442 / 13973 us for the figures above; CTAs of 4 warps that
// share 8 or 16 rows and meet at barriers 136 / 124 / 1494 / 12280; scores read from global memory in both sweeps instead of staged
// 76 / 137 / 1822.  Buckets: half as many 1240 at 1024 candidates but 2910 for 2600 with static frames, whose scores lie in clumps.
#pragma once
#include <cmath>
#include <cstring>

#include "score_tc.cuh"

namespace adaspark {

constexpr int kSelectCand = 32;          // cubes of the crossing bucket a row may list
constexpr int kMaxHistLevels = 8;        // histograms of a row before it is handed to the fp64 kernel
constexpr float kUlp = 5.9604645e-8f;    // 2^-24: the largest relative error of a rounding
constexpr float kGuard = 1e-3f;          // of a bucket
constexpr int kSumIters = 4;             // chunks of a thread (4 additions each) whose masses are summed before they join the rest
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

// Shared memory of a warp on R rows of up to kCols scores.  (Normally distributed, the fullest bucket holds some 2 of 64 and 128 scores, 5 of 256
// to 1024, 11 of 2048 and 23 of 4096: the list's 32 places are near in the largest shape, which therefore splits buckets more often.)  The padding of a row keeps the 16-byte loads of 8 neighbouring
// lanes (8 rows, or with fewer rows several chunks of each, see `swap`) in 8 different bank groups.
template <int R, int kCols, int kBuckets>
struct SelectSmem {
    static constexpr int kOut = R < 8 ? 8 : R;            // rows whose mask words leave together: whole 32-byte sectors
    float rows[R][kCols + (R == 4 || R == 2 ? 8 : 4)];
    union {
        uint32_t hist[kBuckets][R];
        float4 cand[kSelectCand][R];                      // score, mass, cube; once the histogram has been read
    };
    uint32_t words[kCols / 32][kOut];
};

__device__ __forceinline__ float sat_fma(float a, float b, float c) {     // min(max(a b + c, 0), 1)
    return __saturatef(fmaf(a, b, c));
}

// One warp per CTA and `warp_rows` rows (8, 16 or 32, at least R): 128 / warp_rows CTAs per item, items [first, ..) of those that
// the scores were computed for.  scores / row_range / row_err: what score_tc_kernel left for the items [item0, ..).
// tile_mask as mask_index() describes; tile_union (cleared) receives the OR of each word over the tile's rows;
// fallback_rows[0 .. *fallback_count) receives ((b*Hq+h)*n_tiles_cap + tile)*128 + r of the rows left to the fp64
// kernel.  kCols >= the largest candidate count of these items.
template <int R, int kCols, int kBuckets, SelectRule kRule>
__global__ void __launch_bounds__(32) select_nucleus_kernel(
    Geom g, SelectTarget rule, int item0, int first, int warp_rows, const float* scores, const float4* row_range, const float* row_err, uint32_t* tile_mask,
    uint32_t* tile_union, const unsigned long long* key_hash, uint32_t* sel_bitmap, int32_t* sel_count, int32_t* fallback_rows, uint32_t* fallback_count) {
    extern __shared__ __align__(16) unsigned char select_raw[];
    constexpr int U = 32 / R;                                              // lanes of a row
    constexpr int kIter = kCols / (8 * U), kMasks = (kIter + 3) / 4;       // chunks of 8 columns per lane; bit words
    constexpr bool kByCount = kRule == kCount, tail = kRule == kTail;
    constexpr int kLaneSteps = R == 32 ? 0 : R == 16 ? 1 : R == 8 ? 2 : R == 4 ? 3 : R == 2 ? 4 : 5;     // additions that join the lanes of a row
    constexpr int kBlocks = (kIter + kSumIters - 1) / kSumIters;
    constexpr int kAdds = (kIter < kSumIters ? 4 * kIter : 4 * kSumIters) + kBlocks + 2 + kLaneSteps;    // a mass passes through, in a row's sum (at least 8 + those of the lanes)
    constexpr uint32_t kFull = 0xffffffffu;
    constexpr uint32_t kRowLanes = R == 32 ? 1u : R == 16 ? 0x10001u : R == 8 ? 0x01010101u : R == 4 ? 0x11111111u : R == 2 ? 0x55555555u : kFull;   // of row 0
    constexpr float kMagic = 8388608.f;                                    // 2^23: low mantissa bits = the integer part
    constexpr uint32_t kMagicBits = 0x4B000000u;
    static_assert(kIter * 8 * U == kCols && kCols % 64 == 0 && kIter >= 2, "shape");
    using Smem = SelectSmem<R, kCols, kBuckets>;
    constexpr int kOut = Smem::kOut;
    const int lane = threadIdx.x, row = lane % R, u = lane / R;            // row of the pass, which of its lanes
    const int per_item = kTileRows / warp_rows;
    const int item = first + blockIdx.x / per_item, row_begin = (blockIdx.x % per_item) * warp_rows;
    const ScoreItem w = score_item(g, item0 + item);
    const size_t gt_cap = (size_t)(w.b * g.Hq + w.h) * g.n_tiles_cap + w.tile;
    const int n_words_live = min(2 * w.n_ct, g.n_words);                   // words that can hold a candidate
    Smem& sm = *reinterpret_cast<Smem*>(select_raw);
    uint32_t* hist = &sm.hist[0][0];
    auto clear_hist = [&]() {
#pragma unroll 8
        for (int i = lane; i < kBuckets * R / 4; i += 32) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    };
    clear_hist();
    launch_dependents();
    wait_for_previous_kernel();

    constexpr float a_add0 = tail ? (float)(kBuckets - 1) : 0.f;
    // Scores and range of a pass, requested as soon as those of the pass before are no longer read.  All rows of the pass are
    // copied up to the largest candidate count among them (what a row does not have is not looked at).
    float4 ra, rb;
    float err_next;
    auto request = [&](int r0) -> int {
        const int pos = w.tile * kTileRows + r0 + row;
        const int n = slot_live(g, pos) ? n_candidates(g, pos) : 0;
        const int n4 = (__reduce_max_sync(kFull, n) + 3) >> 2;
        constexpr int kLanes = kCols / 4 < 32 ? kCols / 4 : 32, kRowsAtOnce = 32 / kLanes;
        const size_t srow0 = (size_t)item * kTileRows + r0;
        const float* src = scores + (srow0 + lane / kLanes) * g.N_ld;
        float* dst = sm.rows[lane / kLanes];
#pragma unroll 1
        for (int c = lane % kLanes; c < n4; c += kLanes) {
#pragma unroll
            for (int r = 0; r < R; r += kRowsAtOnce) cp_async_16(dst + r * (sizeof(sm.rows[0]) / 4) + 4 * c, src + (size_t)r * g.N_ld + 4 * c);
        }
        cp_async_commit();
        ra = row_range[2 * (srow0 + row)];
        rb = row_range[2 * (srow0 + row) + 1];
        err_next = row_err[srow0 + row];
        return n;
    };
    int n_next = request(row_begin);
#pragma unroll 1
    for (int r0 = row_begin; r0 < row_begin + warp_rows; r0 += R) {
        const int ro = r0 % kOut + row;                                    // the row's place among those that leave together
        const int n = n_next;
        float top = fmaxf(fmaxf(ra.x, ra.z), fmaxf(rb.x, rb.z)), low = fminf(fminf(ra.y, ra.w), fminf(rb.y, rb.w));
        const float err = n > 0 ? err_next : 0.f;
        bool give_up = n > 0 && !(top > -INFINITY && low > -INFINITY);     // marked by the score kernel, or its scores are missing
        const bool act = n > 0 && !give_up;
        if (!act) top = low = 0.f;
        cp_async_wait<0>();
        if (R >= 8 || r0 % kOut == 0)
            for (int i = lane; i < n_words_live * (kOut / 4); i += 32) reinterpret_cast<uint4*>(&sm.words[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        n_next = 0;
        if (__any_sync(kFull, n > 0)) {
            const float* my_row = sm.rows[row];
            auto mass = [&](float d) -> float { return kByCount ? 1.f : fast_exp2(d); };   // of a score at d = s - max
            const int own = act ? max((n / 8 - u + U - 1) / U, 0) : 0;     // my whole chunks: columns 8 (U i + u) .. +7
            const bool part = act && (n & 7) != 0 && u == (n / 8) % U;     // and the row's last columns
            // With fewer than 8 rows a load of 8 lanes meets several chunks of a row: half of the lanes read the second
            // 16 bytes of theirs first (column e of a lane's chunk is then column e ^ 4).
            const int swap = R == 4 || R == 2 ? (u & 1) * 4 : R == 1 ? (u & 4) : 0;
            const float* mine = my_row + 8 * u;
            auto load_chunk = [&](int i, unsigned long long (&x2)[4]) {
                const float4 x0 = *reinterpret_cast<const float4*>(mine + i * (8 * U) + swap), x1 = *reinterpret_cast<const float4*>(mine + i * (8 * U) + (swap ^ 4));
                x2[0] = pack_f32x2(x0.x, x0.y);
                x2[1] = pack_f32x2(x0.z, x0.w);
                x2[2] = pack_f32x2(x1.x, x1.y);
                x2[3] = pack_f32x2(x1.z, x1.w);
            };
            // ---- sweep 1: Z and the histogram over u = (max - s) * per_unit, or from the other end, bucket = round(u): the
            // buckets span the row
            const float per_unit = fminf((float)(kBuckets - 1) / (top - low), 1e18f);
            float a_mul = tail ? per_unit : -per_unit, a_add = a_add0;     // u = d * a_mul + a_add
            uint32_t* my_hist = hist + row;
            const uint32_t hist_addr = smem_u32(my_hist) - kMagicBits * (4u * R);   // plus 4 R times the bits of 2^23 + bucket
            auto add_to_bucket = [&](uint32_t bucket_bits, uint32_t q) {
                asm volatile("red.shared.add.u32 [%0], %1;\n" ::"r"(hist_addr + bucket_bits * (4u * R)), "r"(q) : "memory");
            };
            auto row_sum = [&](float x) -> float {
#pragma unroll
                for (int o = 16; o >= R; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
                return x;
            };
            const unsigned long long neg_top2 = pack_f32x2(-top, -top), a_mul2 = pack_f32x2(a_mul, a_mul);
            float z = 0.f;
            {
                unsigned long long z2 = 0ull;
                const unsigned long long magic2 = pack_f32x2(kMagic + a_add0, kMagic + a_add0), q_unit2 = pack_f32x2(rule.q_unit, rule.q_unit);
#pragma unroll 1
                for (int i0 = 0; i0 < own; i0 += kSumIters) {
                    unsigned long long zs2 = 0ull;                         // of the last few chunks
#pragma unroll
                    for (int q = 0; q < kSumIters; ++q) {
                        if (q >= kIter || i0 + q >= own) break;
                        unsigned long long x2[4];
                        load_chunk(i0 + q, x2);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const unsigned long long d2 = add_f32x2(x2[k], neg_top2);
                            float d0, d1, b0, b1;
                            unpack_f32x2(d2, d0, d1);
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
                    }
                    z2 = add_f32x2(z2, zs2);
                }
                float z0, z1, zp = 0.f;
                if (part) {
#pragma unroll 1
                    for (int j = n & ~7; j < n; ++j) {
                        const float d = my_row[j] - top, m = mass(d);
                        zp += m;
                        add_to_bucket(__float_as_uint(fmaf(d, a_mul, kMagic + a_add0)), kByCount ? 1u : __float_as_uint(m * rule.q_unit));
                    }
                }
                unpack_f32x2(z2, z0, z1);
                z += z0 + z1;
                z += zp;
            }
            __syncwarp();
            z = row_sum(z);
            const float target = kByCount ? fminf(z, (float)g.top_k) : (float)((double)z * rule.share);
            float base = 0.f;                                              // mass before the bucket
            uint32_t inside[kMasks];                                       // bit 8 i + e: column e of my i-th chunk
#pragma unroll
            for (int k = 0; k < kMasks; ++k) inside[k] = 0u;
            auto column = [&](int k, int e) -> int { return ((4 * k + (e >> 3)) * U + u) * 8 + ((e & 7) ^ swap); };
            auto of_row = [&](uint32_t ballot) -> uint32_t { return (ballot >> row) & kRowLanes; };
            // The bucket in which the cumulative (quantised) mass crosses the target.  A lane sums the buckets of its part of the
            // row (in an order of its own: no bank is met twice), the one that finds the target in it looks where.
            auto find_bucket = [&]() -> int {
                constexpr int kSeg = kBuckets / U, kGroup = R <= 2 ? 16 : 8, kGroups = kSeg / kGroup;
                uint32_t group[kGroups], sum = 0u;
                const uint32_t* seg = my_hist + u * (kSeg * R);
#pragma unroll
                for (int i = 0; i < kGroups; ++i) {
                    group[i] = 0u;
#pragma unroll
                    for (int k = 0; k < kGroup; ++k) group[i] += seg[(i * kGroup + (k ^ (u & (kGroup - 1)))) * R];
                    sum += group[i];
                }
                uint32_t incl = sum;
#pragma unroll
                for (int o = R; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(kFull, incl, o);
                    if (lane >= o) incl += t;
                }
                const uint32_t thr = max((uint32_t)fmaxf((target - base) * rule.unit, 0.f), 1u);
                const uint32_t over = of_row(__ballot_sync(kFull, incl >= thr));
                const int finder = over ? __ffs(over) - 1 + row : 32 - R + row;
                int at = kBuckets - 1;
                if (lane == finder && over) {
                    uint32_t cum = incl - sum;
                    at = 0;
#pragma unroll
                    for (int i = 0; i < kGroups - 1; ++i)
                        if (at == i * kGroup && cum + group[i] < thr) { cum += group[i]; at += kGroup; }
                    uint32_t h[kGroup];
#pragma unroll
                    for (int k = 0; k < kGroup; ++k) h[k] = seg[(at + k) * R];
                    int step = 0;
#pragma unroll
                    for (int k = 0; k < kGroup - 1; ++k) {
                        cum += h[k];
                        if (step == k && cum < thr) ++step;
                    }
                    at += step + u * kSeg;
                }
                __syncwarp();
                return __shfl_sync(kFull, at, finder);
            };
            // ---- sweep 2: before / inside the bucket [cb - 1/2, cb + 1/2], widened by the guard; what is before, or else what
            // is neither before nor inside, goes to the row's mask words
            int cb = find_bucket();
            float lo_u = (float)cb - (0.5f + kGuard), hi_u = (float)cb + (0.5f + kGuard);
            const float to_edge = a_add0 - (tail ? lo_u : hi_u);           // u + this = 0: the edge of the first bucket on the rejected side
            uint8_t* my_words = reinterpret_cast<uint8_t*>(&sm.words[0][ro]);
            auto word_byte = [&](int chunk) -> uint8_t* { return my_words + (chunk >> 2) * (4 * kOut) + (chunk & 3); };
            {
                const unsigned long long lo2 = pack_f32x2(a_add0 - lo_u, a_add0 - lo_u), width2 = pack_f32x2(lo_u - hi_u, lo_u - hi_u);
                unsigned long long add2 = 0ull;
#pragma unroll
                for (int k = 0; k < kMasks; ++k) {
                    unsigned long long adds2 = 0ull;                       // of the last few chunks
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int i = 4 * k + q;
                        if (i >= kIter) continue;
                        if (i < own) {
                            unsigned long long x2[4];
                            load_chunk(i, x2);
                            uint32_t bits = 0u, in = 0u;
#pragma unroll
                            for (int p = 3; p >= 0; --p) {
                                const unsigned long long d2 = add_f32x2(x2[p], neg_top2), u2 = fma_f32x2(d2, a_mul2, lo2);
                                float d0, d1, ua0, ua1, ub0, ub1;
                                unpack_f32x2(d2, d0, d1);
                                unpack_f32x2(u2, ua0, ua1);
                                unpack_f32x2(add_f32x2(u2, width2), ub0, ub1);
                                bits = __funnelshift_l(__float_as_uint(ua1), bits, 1);
                                bits = __funnelshift_l(__float_as_uint(ua0), bits, 1);
                                in = __funnelshift_l(__float_as_uint(ub1), in, 1);
                                in = __funnelshift_l(__float_as_uint(ub0), in, 1);
                                // the mass of what lies before: times 2^100 and clamped, the distance is 1 before and 0 else
                                adds2 = fma_f32x2(pack_f32x2(mass(d0), mass(d1)),
                                                  pack_f32x2(__saturatef(ua0 * -1.2676506e30f), __saturatef(ua1 * -1.2676506e30f)), adds2);
                            }
                            inside[k] |= (in & ~bits) << (8 * q);
                            bits = tail ? ~(bits | in) & 0xffu : bits;
                            if (R < 8) bits = (bits >> swap) | (bits << swap);
                            *word_byte(i * U + u) = (uint8_t)bits;
                        }
                    }
                    add2 = add_f32x2(add2, adds2);
                }
                float add0, add1, addp = 0.f;
                if (part) {
                    uint32_t bits = 0u, in = 0u;                           // by column
#pragma unroll 1
                    for (int j = n & ~7; j < n; ++j) {
                        const float d = my_row[j] - top, uj = fmaf(d, a_mul, a_add0 - lo_u);
                        const uint32_t bit = 1u << (j & 7);
                        if (uj < 0.f) { bits |= bit; addp += mass(d); }
                        else if (uj + (lo_u - hi_u) < 0.f) in |= bit;
                    }
                    *word_byte(n >> 3) = (uint8_t)(tail ? ~(bits | in) & ((1u << (n & 7)) - 1u) : bits);
                    if (R < 8) in = ((in >> swap) | (in << swap)) & 0xffu;
#pragma unroll
                    for (int k = 0; k < kMasks; ++k)
                        if (k == own >> 2) inside[k] |= in << (8 * (own & 3));
                }
                unpack_f32x2(add2, add0, add1);
                float add = add0 + add1;
                add += addp;
                base = row_sum(add);
            }
            // my place in the row's list, and how long it is
            int slot, n_cand;
            auto count_inside = [&]() {
                int mine_in = 0;
#pragma unroll
                for (int k = 0; k < kMasks; ++k) mine_in += __popc(inside[k]);
                int incl = mine_in;
#pragma unroll
                for (int o = R; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(kFull, incl, o);
                    if (lane >= o) incl += t;
                }
                slot = incl - mine_in;
                n_cand = __shfl_sync(kFull, incl, 32 - R + row);
            };
            count_inside();
            int adds = 2 * kAdds + 2;
            float beyond = -INFINITY;                                      // my largest rejected score of that bucket that is not listed
            bool active = act && n_cand > kSelectCand;
            if (__any_sync(kFull, active)) {
                // ---- rare: split the bucket of the rows that hold too many cubes in it
                constexpr float fine = (float)(kBuckets - 1) / (1.f + 2.f * kGuard);
#pragma unroll 1
                for (int level = 1;; ++level) {
                    if (active) {
                        a_add = (a_add - lo_u) * fine;
                        a_mul = a_mul * fine;
                        if (level == kMaxHistLevels || !(fabsf(a_mul) < 1e30f)) { give_up = true; active = false; }
                    }
                    if (!__any_sync(kFull, active)) break;
                    clear_hist();
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < kMasks; ++k) {
                        uint32_t bits = active ? inside[k] : 0u;
                        while (bits) {
                            const float d = my_row[column(k, __ffs(bits) - 1)] - top;
                            bits &= bits - 1u;
                            const float u01 = sat_fma(d, a_mul * (1.f / (kBuckets - 1)), a_add * (1.f / (kBuckets - 1)));
                            add_to_bucket(__float_as_uint(fmaf(u01, (float)(kBuckets - 1), kMagic)), kByCount ? 1u : __float_as_uint(mass(d) * rule.q_unit));
                        }
                    }
                    __syncwarp();
                    cb = find_bucket();
                    float add = 0.f;
                    int n_add = 0;
                    if (active) {
                        lo_u = (float)cb - (0.5f + kGuard);
                        hi_u = (float)cb + (0.5f + kGuard);
#pragma unroll
                        for (int k = 0; k < kMasks; ++k) {
                            uint32_t bits = inside[k];
                            while (bits) {
                                const int e = __ffs(bits) - 1, j = column(k, e);
                                bits &= bits - 1u;
                                const float x = my_row[j], d = x - top, uj = fmaf(d, a_mul, a_add);
                                const bool bef = uj < lo_u;
                                if (!bef && uj < hi_u) continue;
                                inside[k] &= ~(1u << e);
                                if (bef) { add += mass(d); ++n_add; }
                                if (bef == tail) beyond = fmaxf(beyond, x);                // rejected, or else selected
                                else atomicOr(&sm.words[j >> 5][ro], 1u << (j & 31));
                            }
                        }
                    }
                    adds += __reduce_max_sync(kFull, n_add) + 6;           // (the lane's, its row's and the base's)
                    base += row_sum(add);
                    count_inside();
                    if (n_cand <= kSelectCand) active = false;
                }
#pragma unroll
                for (int o = 16; o >= R; o >>= 1) beyond = fmaxf(beyond, __shfl_xor_sync(kFull, beyond, o));
            }
            // ---- list the cubes inside the bucket
            const bool decide = act && !give_up;
            const int n_list = decide ? n_cand : 0;
            const int n_list_most = __reduce_max_sync(kFull, n_list);
            __syncwarp();
            for (int i = n_list + u; i < n_list_most; i += U) sm.cand[i][row] = make_float4(-INFINITY, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < kMasks; ++k) {
                uint32_t bits = decide ? inside[k] : 0u;
                while (bits) {
                    const int j = column(k, __ffs(bits) - 1);
                    bits &= bits - 1u;
                    const float x = my_row[j];
                    sm.cand[slot++][row] = make_float4(x, mass(x - top), __int_as_float(j), 0.f);
                }
            }
            __syncwarp();
            if (r0 + R < row_begin + warp_rows) n_next = request(r0 + R);  // the rows' scores are no longer read
            // ---- each listed cube: the mass before it and with it
            const float mass_err = fmaf(0.6931472f, fmaf(2.f * kUlp, (top - low) + fmaxf(top, -low), err), 4.f * kUlp);
            const float eps = kByCount ? 0.f : z * fmaf(rule.eps_mass, mass_err, rule.eps_add * (float)(adds + n_list));
            float last = INFINITY, next = -INFINITY;                       // lowest selected, highest rejected score of my cubes
            bool reached = false, unsure = false;
            for (int i0 = 0; i0 < n_list_most; i0 += U) {
                const int i = i0 + u;
                const float4 me = sm.cand[min(i, n_list_most - 1)][row];
                const int ji = __float_as_int(me.z);
                float acc = base;                                          // and the listed cubes before mine
#pragma unroll 4
                for (int k = 0; k < n_list_most; ++k) {
                    const float4 ck = sm.cand[k][row];
                    const bool earlier = tail ? ck.x < me.x || (ck.x == me.x && __float_as_int(ck.z) > ji)
                                              : ck.x > me.x || (ck.x == me.x && __float_as_int(ck.z) < ji);
                    if (earlier) acc += ck.y;
                }
                if (i < n_list) {
                    if (tail ? acc + me.y > target : acc < target) {
                        atomicOr(&sm.words[ji >> 5][ro], 1u << (ji & 31));
                        last = fminf(last, me.x);
                    } else {
                        next = fmaxf(next, me.x);
                    }
                    reached = reached || (tail ? acc + me.y > target : acc + me.y >= target);
                    if (!kByCount) unsure = unsure || fabsf(acc - target) <= eps || fabsf(acc + me.y - target) <= eps;
                }
            }
#pragma unroll
            for (int o = 16; o >= R; o >>= 1) {
                last = fminf(last, __shfl_xor_sync(kFull, last, o));
                next = fmaxf(next, __shfl_xor_sync(kFull, next, o));
            }
            const float gap = fmaf(4.f * kUlp, fabsf(last), 2.f * err);
            // an unlisted cube lies beyond the edge (u is off by a small part of the guard) or has been looked at
            unsure = unsure || (n_list < n && fabsf(fmaf(last - top, tail ? per_unit : -per_unit, to_edge)) <= fmaf(gap, per_unit, 0.5f * kGuard));
            unsure = unsure || (beyond > -INFINITY && last - beyond <= gap);
            bool tied = last < INFINITY && last - next <= gap;             // (a row without a listed cube that is selected is unsure)
            if (__any_sync(kFull, tied)) {
                // The boundary runs through cubes whose order these scores cannot tell.  If they are copies of one cube (frames
                // that repeat: the mean keys are equal bit by bit) their scores are equal in fp64 too and the index orders them.
                // (All such rows went to the fp64 kernel: every frame twice, 65536 tokens, 57.8 instead of 4.3 ms of selection.)
                const unsigned long long* hash = key_hash + (size_t)(w.b * g.Hkv + w.gk) * g.N_ld;
                unsigned long long h_min = ~0ull, h_max = 0ull;
                for (int i = u; i < n_list; i += U) {
                    const float4 me = sm.cand[i][row];
                    if (last - me.x <= gap && me.x - next <= gap) {
                        const unsigned long long hj = hash[__float_as_int(me.z)];
                        h_min = min(h_min, hj);
                        h_max = max(h_max, hj);
                    }
                }
#pragma unroll
                for (int o = 16; o >= R; o >>= 1) {
                    h_min = min(h_min, __shfl_xor_sync(kFull, h_min, o));
                    h_max = max(h_max, __shfl_xor_sync(kFull, h_max, o));
                }
                tied = tied && h_min != h_max;
            }
            unsure = unsure || tied || !(last < INFINITY);
            const uint32_t any_unsure = of_row(__ballot_sync(kFull, unsure)), any_reached = of_row(__ballot_sync(kFull, reached));   // both by all lanes
            unsure = any_unsure != 0u || any_reached == 0u || !(tail ? base <= target : base < target);
            __syncwarp();                                                  // bits of the row's other lanes have arrived: none follows the zeros
            if (n > 0 && (give_up || unsure)) {
                for (int wd = u; wd < n_words_live; wd += U) sm.words[wd][ro] = 0u;
                if (u == 0) fallback_rows[atomicAdd(fallback_count, 1u)] = (int32_t)(gt_cap * kTileRows + r0 + row);
            }
            __syncwarp();
            clear_hist();
        } else if (r0 + R < row_begin + warp_rows) {
            n_next = request(r0 + R);
        }
        __syncwarp();
        // ---- mask words (whole 32-byte sectors), union words, the caller's copies
        if (R < 8 && (r0 + R) % kOut != 0) continue;
        const int out0 = r0 / kOut * kOut;
        constexpr int kParts = kOut / 4;                                   // 16-byte parts of a word's rows
        for (int i0 = 0; i0 < g.n_words * kParts; i0 += 32) {
            const int wd = (i0 + lane) / kParts, c4 = lane % kParts;
            const uint4 val = wd < n_words_live ? *reinterpret_cast<const uint4*>(&sm.words[wd][c4 * 4]) : make_uint4(0u, 0u, 0u, 0u);
            if (wd < g.n_words)
                *reinterpret_cast<uint4*>(tile_mask + (gt_cap * g.n_words + wd) * kTileRows + out0 + c4 * 4) = val;
            uint32_t un = (val.x | val.y) | (val.z | val.w);               // OR over the lanes of the word
#pragma unroll
            for (int o = kParts / 2; o > 0; o >>= 1) un |= __shfl_xor_sync(kFull, un, o);
            if (c4 == 0 && un) atomicOr(tile_union + gt_cap * g.n_words + wd, un);
        }
        if (sel_bitmap != nullptr || sel_count != nullptr) {
            for (int r = 0; r < kOut; ++r) {
                const int pos = w.tile * kTileRows + out0 + r;
                if (!slot_live(g, pos)) continue;
                const size_t raster_row = (size_t)(w.b * g.Hq + w.h) * g.S_io + (pos_to_io(g, pos) - g.pos_begin);
                int cnt = 0;
                for (int wd = lane; wd < g.n_words; wd += 32) {
                    const uint32_t word = wd < n_words_live ? sm.words[wd][r] : 0u;
                    cnt += __popc(word);
                    if (sel_bitmap) sel_bitmap[raster_row * g.n_words + wd] = word;
                }
                cnt = __reduce_add_sync(kFull, cnt);
                if (sel_count && lane == 0) sel_count[raster_row] = cnt;
            }
        }
        __syncwarp();
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
