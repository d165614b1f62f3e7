"""Host-side check of how the score kernel folds the four level sums of a digit product into one 32-bit integer
(score_tc.cuh, shifted_levels).

The result fits 32 bits, the terms it is summed from need not: the routine is read out of the source, compiled for the
host with overflow of signed integers trapped, and compared with 64-bit arithmetic."""
import os
import re
import subprocess

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_08077_b200", "csrc", "score_tc.cuh")

PROGRAM = r"""
#include <cstdint>
#include <cstdio>
#include <random>
%s
int main() {
    std::mt19937_64 rng(7);
    auto pick = [&](long long bound) { return (long long)(rng() %% (unsigned long long)(2 * bound + 1)) - bound; };
    const long long tile = 128ll * 128 * 128;             // largest |sum of one digit pair| over 128 elements
    int large_terms = 0;
    for (int sh = 0; sh <= 16; ++sh) {
        for (int i = 0; i < 20000; ++i) {
            // a wanted result anywhere in the 32 bits, and level sums that give it: S_0 makes up for what S_1 .. S_3 add
            const bool corner = i < 64;
            const long long s1 = corner ? (i & 1 ? 2 * tile : -2 * tile) : pick(2 * tile);
            const long long s2 = corner ? (i & 2 ? 3 * tile : -3 * tile) : pick(3 * tile);
            const long long s3 = corner ? (i & 4 ? 4 * tile : -4 * tile) : pick(4 * tile);
            const long long want = pick((1ll << 31) - (1ll << 25)) * (1ll << sh);
            const long long s0 = (want - s1 * 65536 - (s2 * 256 + s3)) / (1ll << 24);
            const long long v = s0 * (1ll << 24) + s1 * 65536 + s2 * 256 + s3;
            if (s0 > tile || s0 < -tile || (v >> sh) > INT32_MAX || (v >> sh) < INT32_MIN) continue;
            const long long term = s1 * (1ll << (16 - sh));
            large_terms += term > INT32_MAX || term < INT32_MIN;
            const uint32_t m1 = 1u << (16 - sh), m0 = m1 << 8;
            if (shifted_levels((int32_t)s0, (int32_t)s1, (int32_t)s2, (int32_t)s3, m0, m1, sh) != (int32_t)(v >> sh)) return 1;
        }
    }
    std::printf("%%d\n", large_terms);
    return 0;
}
"""


def test_levels_fold_without_signed_overflow(tmp_path):
    text = open(SRC).read()
    body = re.search(r"int32_t shifted_levels\(.*?\n\}\n", text, re.S).group(0)
    prog = tmp_path / "levels.cpp"
    prog.write_text(PROGRAM % body)
    exe = str(tmp_path / "levels")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=signed-integer-overflow", "-fsanitize-undefined-trap-on-error", str(prog), "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0, res.returncode
    assert int(res.stdout) > 1000                         # terms beyond 32 bits were among the cases
