"""The rule of block tasks (swgb_internal.h): which classes may run as block
tasks, on both sides of the limits on their number and on their boundary rows,
and the rows a plan takes for them."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include "swgb_internal.h"
using namespace swgb;
static int bad = 0;
static void expect(long got, long want, const char *what)
{
    if (got != want) { printf("%s: %ld, not %ld\n", what, got, want); ++bad; }
}
int main()
{
    ClassInfo ci{};
    auto set = [&](int mode, int m, int n, int cnt) {
        const int c = mode * N_MCLASS + mclass_of(m);
        ci.count[c] = cnt;
        ci.max_m[c] = m;
        ci.max_n[c] = n;
    };
    set(MODE_I16W, 512, 9000, 4000);
    set(MODE_I32, 7000, 9000, 100);
    expect(block_task_bytes(ci, 304), 0, "reads of 512 bases and int32 classes");
    set(MODE_I16W, 513, 600, 607);
    expect(block_task_bytes(ci, 304), 16L * 600 * 304, "304 tasks");
    set(MODE_I16W, 700, 800, 1);
    expect(block_task_bytes(ci, 304), 0, "305 tasks");
    expect(block_task_bytes(ci, 305), 16L * (600 * 304 + 800), "305 tasks of 305");
    set(MODE_I16W, 2000, 1048575, 6);
    expect(block_task_bytes(ci, 400), 16L * (600 * 304 + 800 + 3 * 1048575L), "within the rows' limit");
    set(MODE_I16W, 2000, 1048575, 8);
    expect(block_task_bytes(ci, 400), kPipeBytes, "past the rows' limit");
    return bad != 0;
}
"""


def test_both_limits(tmp_path):
    src = tmp_path / "blocks.cpp"
    src.write_text(SRC)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_1304_0681_gb300", "csrc"),
                           "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include", str(src), "-o",
                           str(tmp_path / "blocks")])
    r = subprocess.run([str(tmp_path / "blocks")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
