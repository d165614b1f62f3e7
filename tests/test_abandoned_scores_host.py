"""Host-side check of what the score kernel leaves for query tiles that it did not finish because a wait expired (score_tc.cuh,
abandon_ranges), and of how the selection kernel reads it (select_nucleus.cuh).

The selection takes a score's bucket from the row's range without a bound, so a row whose range and scores are whatever the workspace
held must not be decided.  The routine and the lines that read a range are taken out of the sources and compiled for the host; no wait is
made to expire on a GPU."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_08077_b200", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
#define __host__
#define __device__
struct float2 { float x, y; };
struct float4 { float x, y, z, w; };
float2 make_float2(float x, float y) { return {x, y}; }
constexpr int kTileRows = 128;
%s
%s
bool decided(float4 ra, float4 rb, int n) {
    %s
    %s
    return n > 0 && !give_up;
}
int main() {
    std::mt19937 rng(3);
    const int n_items = 11, step = 4;
    for (int first = 0; first < step; ++first)                       // a CTA's items: first, first + step, ..
        for (int from = first; from < n_items + step; from += step)  // the first one it did not finish
            for (int missing = 1; missing < 1 << kRangeParts; ++missing) {
                std::vector<float2> range(kRangeParts * n_items * kTileRows + 1);
                for (auto& x : range) {                              // what was there before: any order, any finite value
                    x.x = std::ldexp((float)(int)rng(), (int)(rng() %% 60) - 40);
                    x.y = std::ldexp((float)(int)rng(), (int)(rng() %% 60) - 40);
                }
                const auto before = range;
                for (int part = 0; part < kRangeParts; ++part)
                    if (missing >> part & 1)
                        for (int row = 0; row < kTileRows; ++row) abandon_ranges(range.data(), from, n_items, step, row, part);
                for (int it = 0; it < n_items; ++it) {
                    const bool mine = it >= from && (it - first) %% step == 0;
                    for (int row = 0; row < kTileRows; ++row) {
                        const float2* p = &range[kRangeParts * (it * kTileRows + row)];
                        const float4 ra = {p[0].x, p[0].y, p[1].x, p[1].y}, rb = {p[2].x, p[2].y, p[3].x, p[3].y};
                        if (mine && decided(ra, rb, 5)) return 1;
                        if (!mine && !decided(ra, rb, 5)) return 2;
                    }
                }
                for (size_t i = 0; i < range.size(); ++i) {
                    const int it = (int)(i / (kRangeParts * kTileRows)), part = (int)(i %% kRangeParts);
                    const bool marked = it < n_items && it >= from && (it - first) %% step == 0 && (missing >> part & 1);
                    if (!marked && (range[i].x != before[i].x || range[i].y != before[i].y)) return 3;
                }
            }
    std::printf("ok\n");
    return 0;
}
"""


def test_rows_without_scores_are_not_decided(tmp_path):
    score = open(os.path.join(CSRC, "score_tc.cuh")).read()
    select = open(os.path.join(CSRC, "select_nucleus.cuh")).read()
    parts = re.search(r"constexpr int kRangeParts = 4;", score).group(0)
    body = re.search(r"__host__ __device__ inline void abandon_ranges\(.*?\n\}\n", score, re.S).group(0)
    fold = re.search(r"float top = fmaxf\(.*?;", select).group(0)
    rule = re.search(r"bool give_up = .*?;", select).group(0)
    # an epilogue warp leaves its items only through a break, and marks from the item that it left on
    epilogue = score[score.index("// ------------------------------------------------------------ epilogue"):]
    epilogue = epilogue[:epilogue.index("} else if (warp == kClearWarp)")]
    assert re.search(r"if \(!ok\) break;\n\s*row_range\[", epilogue)
    assert re.search(r"\n        \}\n        if \(!ok\) abandon_ranges\(row_range, it, n_items, gridDim\.x, quarter \* 32 \+ lane, part\);", epilogue)
    prog = tmp_path / "ranges.cpp"
    prog.write_text(PROGRAM % (parts, body, fold, rule))
    exe = str(tmp_path / "ranges")
    subprocess.run(["g++", "-std=c++17", "-O1", str(prog), "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0 and res.stdout == "ok\n", (res.returncode, res.stdout)
