"""How much scratch a call takes (csrc/sw_budgets.h, compiled with the host
compiler): with less memory than it would like a call takes what there is, down
to a size that serves any batch more slowly."""
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
