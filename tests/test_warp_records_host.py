"""A warp keeps what its loops need in a record in shared memory, reached
through a volatile pointer.  Lanes that store different values to one shared
word leave open which value stays, so every store to a record's field has to be
one lane's: in a block or statement under `if (lane == 0)`, or in next_index(),
which holds such a store.  (A class or part index that fails to move on would
keep a persistent kernel looping for ever, so this is read from the source.)"""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_1304_0681_gb300", "csrc", "*.cu*")))
GUARD = re.compile(r"if \((lane|threadIdx\.x) == 0\)\s*$")


def _text(path):
    with open(path) as f:
        s = f.read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", lambda m: re.sub(r"[^\n]", " ", m.group()), s, flags=re.S)


def _guarded(text, at):
    """Whether the statement at `at` stands under a one-lane guard."""
    if GUARD.search(text[:at].rstrip()):
        return True
    depth = 0
    for i in range(at - 1, -1, -1):
        if text[i] == "}":
            depth += 1
        elif text[i] == "{":
            if depth == 0 and GUARD.search(text[:i].rstrip()):
                return True
            depth -= depth > 0
    return False


def _unguarded(text):
    out = []
    for record in set(re.findall(r"volatile \w+ \*const (\w+) =", text)):
        # a for statement's last part is no statement of its own, so it counts as unguarded
        for m in re.finditer(rf"\b{record}->\w+ =[^=]", text):
            if not _guarded(text, m.start()):
                out.append(f"line {text.count(chr(10), 0, m.start()) + 1}: {m.group()}")
    return out


def test_the_check_sees_a_store_of_every_lane():
    head = "volatile Ctx *const cc = &s[0];\n"
    assert _unguarded(head + "for (; a; cc->ci = cc->ci + (lane == 0 ? 1 : 0)) {}")
    assert _unguarded(head + "if (lane == 0) { x = 1; }\ncc->ci = 2;")
    assert not _unguarded(head + "if (lane == 0) cc->ci = 2;")
    assert not _unguarded(head + "if (lane == 0) {\n x = 1; if (y) { z = 1; }\n cc->ci = 2;\n}")


def test_one_lane_stores_to_a_warps_record():
    bad = {os.path.basename(p): _unguarded(_text(p)) for p in SOURCES}
    assert not {k: v for k, v in bad.items() if v}
    records = [p for p in SOURCES if re.search(r"volatile \w+ \*const \w+ =", _text(p))]
    assert len(records) >= 2    # the score and the traceback kernels
