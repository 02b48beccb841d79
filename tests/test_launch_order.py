"""Programmatic dependent launches (no GPU): a kernel that calls pdl_entry calls it
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
