"""The bound on the checkpoint pool (ck_class_units in swgb_internal.h) must
cover what the score pass's tasks take, for any batch and task order."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <algorithm>
#include <cstdio>
#include <random>
#include <vector>
#include "swgb_internal.h"
using namespace swgb;
int main()
{
    std::mt19937_64 rng(5);
    auto uni = [&](int64_t lo, int64_t hi) { return lo + (int64_t)(rng() % (uint64_t)(hi - lo + 1)); };
    const int rows_of[] = {8, 16, 20, 25, 32, 50};
    for (int it = 0; it < 4000; ++it) {
        const int R = rows_of[uni(0, 5)];
        const int m_hi = it % 3 ? uni(1, 400) : uni(1, 8192), m_lo = std::max(1, m_hi - 127);
        const int lanes = std::min(32, (m_hi + R - 1) / R), per_warp = 2 * (32 / lanes);
        const int n_hi = it % 5 ? uni(1, 3000) : uni(8000, 200000);
        const int cnt = (int)uni(1, 400);
        std::vector<std::pair<int, int>> p(cnt);
        int64_t sum = 0;
        int mm = 0, mn = 0;
        for (auto &q : p) {
            q = {(int)uni(m_lo, m_hi), (int)uni(1, n_hi)};
            sum += q.second;
            mm = std::max(mm, q.first);
            mn = std::max(mn, q.second);
        }
        // falling buckets of 32, the last one open, any order inside a bucket
        std::shuffle(p.begin(), p.end(), rng);
        std::stable_sort(p.begin(), p.end(), [](auto &a, auto &b) {
            return std::min((a.second - 1) >> 5, N_NBUCKET - 1) > std::min((b.second - 1) >> 5, N_NBUCKET - 1);
        });
        for (int shift = 0; shift < 4; ++shift) {
            const int ck = ck_block_rows(R) << shift;
            if (ck % R) { printf("block of %d rows at R = %d\n", ck, R); return 1; }
            int64_t used = 0;
            for (int b = 0; b < cnt; b += per_warp) {
                int mw = 0, nw = 0;
                for (int i = b; i < std::min(cnt, b + per_warp); ++i) {
                    mw = std::max(mw, p[i].first);
                    nw = std::max(nw, p[i].second);
                }
                used += (int64_t)(32 / lanes) * ((mw - 1) / ck) * ((nw + 1) / 2 + lanes - 1);
            }
            const int64_t bound = ck_class_units(cnt, sum, mm, mn, lanes, ck);
            if (used > bound) {
                printf("used %lld of %lld: R %d lanes %d cnt %d\n", (long long)used, (long long)bound, R, lanes, cnt);
                return 1;
            }
        }
        if (ck_class_units(cnt, sum, mm, mn, lanes, mm)) { printf("a block of the whole read takes units\n"); return 1; }
    }
    return 0;
}
"""


def test_units_cover_the_tasks(tmp_path):
    src = tmp_path / "ck.cpp"
    src.write_text(SRC)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1304_0681_gb300", "csrc"),
                           "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include", str(src), "-o",
                           str(tmp_path / "ck")])
    r = subprocess.run([str(tmp_path / "ck")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
