"""How much scratch a call takes (csrc/sw_budgets.h, compiled with the host
compiler): with less memory than it would like a call takes what there is, down
to a size that serves any batch more slowly; a plan takes what its classes can use."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _run(tmp_path, main):
    src = tmp_path / "budgets.cpp"
    src.write_text('#include <cstdio>\n#include "sw_budgets.h"\nusing namespace swgb;\n' + main)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_1304_0681_gb300", "csrc"),
                           "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include", str(src), "-o",
                           str(tmp_path / "budgets")])
    r = subprocess.run([str(tmp_path / "budgets")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_a_call_takes_what_a_full_card_has(tmp_path):
    _run(tmp_path, r"""
int main()
{
    const size_t MB = 1 << 20;
    for (size_t least : {64 * MB, 3200 * MB})
        for (size_t want : {256 * MB, 3200 * MB, 16000 * MB})
            for (size_t room = 0; room <= 17000 * MB && want >= least; room += 37 * MB) {
                int tries = 0;
                const size_t got = alloc_between(want, least, [&](size_t b) { ++tries; return b <= room; });
                const bool ok = room < least ? got == 0 : got >= least && got <= room && (got == want || 2 * got > room || got == least);
                if (!ok || tries > 10) {
                    printf("want %zu least %zu room %zu: got %zu in %d tries\n", want / MB, least / MB, room / MB, got / MB, tries);
                    return 1;
                }
            }
    return 0;
}
""")


PLAN = r"""
#include <random>
static ClassInfo ci;
static void add(int m, int n, int cnt, int64_t sum_n)
{
    const int c = score_mode_for(5L * std::min(m, n), SW_SCORE_AUTO) * N_MCLASS + mclass_of(m);
    ci.count[c] = cnt;
    ci.max_m[c] = m;
    ci.max_n[c] = n;
    ci.sum_n[c] = sum_n;
}
static PlanParams params()
{
    PlanParams pp{};
    pp.sc = Scoring{5, -4, -10, -1};
    pp.allow16 = 1;
    for (int &w : pp.score_warps) w = 1216;
    for (int &w : pp.tb_warps) w = 2432;
    return pp;
}
"""


def test_a_plan_takes_what_its_pairs_can_use(tmp_path):
    _run(tmp_path, PLAN + r"""
int main()
{
    const struct { int m, n, cnt; int64_t most; } shapes[] = {
        {100, 150, 64, 4 << 20}, {150, 250, 500, 32 << 20}, {100, 200, 16384, 512 << 20}, {4000, 4100, 200, 1 << 30}};
    for (auto &q : shapes) {
        ci = ClassInfo{};
        add(q.m, q.n, q.cnt, (int64_t)q.cnt * q.n);
        int64_t bnd, tb;
        plan_budgets(ci, params(), true, bnd, tb);
        if (tb > q.most) { printf("%d x %d x %d: %lld bytes\n", q.cnt, q.m, q.n, (long long)tb); return 1; }
    }
    return 0;
}
""")


def test_a_plan_holds_a_slot_for_every_busy_warp(tmp_path):
    """Whatever the bands of an execution come out as (up to 16 GB) -- any split of the classes
    over the three parts, any window up to the widest -- the launches' slots and
    the checkpoints fit the plan's scratch."""
    _run(tmp_path, PLAN + r"""
int main()
{
    std::mt19937_64 rng(3);
    auto uni = [&](int64_t lo, int64_t hi) { return lo + (int64_t)(rng() % (uint64_t)(hi - lo + 1)); };
    const int rows_of[] = {8, 16, 20, 25, 32, 50};
    for (int it = 0; it < 3000; ++it) {
        ci = ClassInfo{};
        const int classes = (int)uni(1, 6);
        for (int k = 0; k < classes; ++k) {
            const int m = (int)(it % 2 ? uni(1, 400) : uni(1, 4000)), n = (int)uni(1, it % 3 ? 400 : 4000);
            const int cnt = (int)uni(1, it % 5 == 0 ? 3 : it % 5 == 1 ? 300 : it % 5 == 2 ? 5000 : 60000);
            add(m, n, cnt, uni(cnt, (int64_t)cnt * n));
        }
        const PlanParams pp = params();
        int64_t bnd, tb;
        plan_budgets(ci, pp, true, bnd, tb);
        if (tb > kTbCapMax) continue;  // past the bounds blocks double and warps wait
        // an execution: parts of every class, then lanes, slots and tasks as the planner counts them
        int64_t n16[kTbParts] = {}, parts[N_CLASS][kTbParts] = {}, all = 0, ck = 0;
        for (int c = N_MCLASS; c < N_CLASS; ++c) {
            const int64_t cnt = ci.count[c], mn = ci.max_n[c];
            if (!cnt) continue;
            parts[c][0] = mn > kTbWide ? uni(0, cnt) : 0;
            parts[c][1] = mn > kTbMid ? uni(0, cnt - parts[c][0]) : 0;
            parts[c][2] = cnt - parts[c][0] - parts[c][1];
            for (int p = 0; p < 2; ++p) n16[p] += parts[c][p];
            all += cnt;
            const int R = rows_of[uni(0, 5)], lanes = std::min(32, (ci.max_m[c] + R - 1) / R);
            ck += 16 * ck_class_units(cnt, (int64_t)ci.sum_n[c], ci.max_m[c], (int)mn, lanes, ck_block_rows(R));
        }
        for (int one = 0; one < 2; ++one) {
            int64_t slot[N_TB_VARIANTS] = {}, tasks[N_TB_VARIANTS] = {};
            for (int c = N_MCLASS; c < N_CLASS; ++c)
                for (int p = 0; p < kTbParts; ++p) {
                    if (!parts[c][p]) continue;
                    const int hi = p == 0 ? ci.max_n[c] : std::min(ci.max_n[c], p == 1 ? kTbWide : kTbMid);
                    const int lo = p == 0 ? kTbWide + 1 : p == 1 ? kTbMid + 1 : 1;
                    const int lanes = tb_part_lanes(one, p, all, p < 2 ? n16[p] : all, ci.count[c], ci.max_m[c], 2432);
                    TbPartPlan t{};
                    const int64_t s = tb_part_shape(c / N_MCLASS, true, ck_block_rows(rows_of[uni(0, 5)]), ci.max_m[c],
                                                    1, (int)uni(lo, hi), p, pp.sc, lanes, t);
                    const int v = tb_launch_first(t.variant);
                    slot[v] = std::max(slot[v], (s + 63) & ~(int64_t)63);
                    tasks[v] += (parts[c][p] * lanes + 63) / 64;
                }
            int64_t need = ck;
            for (int v = 0; v < N_TB_VARIANTS; ++v) need += 4 * slot[v] * std::min<int64_t>(2432, tasks[v]);
            if (need > tb || 4 * ck > 3 * tb) {
                printf("iteration %d: needs %lld (%lld of checkpoints) of %lld\n", it, (long long)need, (long long)ck, (long long)tb);
                return 1;
            }
        }
    }
    return 0;
}
""")
