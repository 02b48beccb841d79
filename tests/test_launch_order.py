"""Order of waits in the kernels' sources (no GPU).

Programmatic dependent launches: a kernel that calls pdl_entry calls it
first and unconditionally.  Only a grid's own wait makes earlier kernels' writes
visible to it, so nothing may be read ahead of it, and a kernel whose trigger
came ahead of its wait would let its successor start too early."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2607_28069_gb300", "csrc")


def test_kernels_wait_before_anything_else():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\bpdl_entry\(\)", text):
            start = max(text.rfind("__global__", 0, m.start()), text.rfind("__device__", 0, m.start()))
            before = text[text.index("{", start) + 1:m.start()]
            ahead = [s.strip() for s in before.split(";") if s.strip()]
            assert all(re.match(r"(constexpr|using|static_assert)\b", s) for s in ahead), (path, ahead)
            seen += 1
    assert seen >= 6


def test_waits_on_the_way_out_look_at_no_abort_flag():
    """An aborted CTA waits for its copies and MMAs in flight before it exits; a
    wait that takes the abort flag, which is set by then, gives up at once."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = open(path).read()
        for m in re.finditer(r"if \([^{;]*\*abort_flag\)|// aborted:|if \(r0 < row_end && n > 0 && lane == 0\)", text):
            for wait in re.findall(r"\bmbar_wait\w*\([^;]*;", text[m.end():m.end() + 500].split("\n  }\n")[0]):
                assert wait.startswith("mbar_wait_no_flag("), (path, wait)
