"""Order and streams of the score launches of the general sequence
(swgb_internal.h): launches on one stream run one after another, so the row
counts that the long reads of a batch take must not share one."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include "swgb_internal.h"
using namespace swgb;
int main()
{
    int used[kScoreStreams] = {};
    for (int mode = 0; mode < N_VMODES; ++mode)
        for (int a = 0; a < N_SCORE_ROWS; ++a) {
            const int s = score_variant_stream(a * N_VMODES + mode);
            if (s < 0 || s >= kScoreStreams) { printf("stream %d\n", s); return 1; }
            ++used[s];
            for (int b = a + 1; b < N_SCORE_ROWS && b < a + (mode == MODE_I16S ? 2 : 4); ++b)
                if (mode != MODE_I16 && s == score_variant_stream(b * N_VMODES + mode)) {
                    printf("mode %d: %d and %d rows on stream %d\n", mode, score_rows_at(a), score_rows_at(b), s);
                    return 1;
                }
        }
    bool seen[N_SCORE_VARIANTS] = {};
    for (int q = 0; q < N_SCORE_VARIANTS; ++q) {
        const int v = score_launch_order(q);
        if (v < 0 || v >= N_SCORE_VARIANTS || seen[v]) { printf("launch %d: variant %d\n", q, v); return 1; }
        seen[v] = true;
    }
    for (int s = 0; s < kScoreStreams; ++s)
        if (!used[s]) { printf("stream %d is not used\n", s); return 1; }
    return 0;
}
"""


def test_long_reads_row_counts_run_side_by_side(tmp_path):
    src = tmp_path / "streams.cpp"
    src.write_text(SRC)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_1304_0681_gb300", "csrc"),
                           "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include", str(src), "-o",
                           str(tmp_path / "streams")])
    r = subprocess.run([str(tmp_path / "streams")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
