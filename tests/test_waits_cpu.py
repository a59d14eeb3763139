"""Rules of the kernels' bounded waits, read off the sources: a wait that a
warp-wide tensor-memory access depends on has one answer for the warp."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2602_14975_gb300", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_split_contraction_waits_by_the_warp():
    """One lane's own wait only drains the MMAs after a time-out; everywhere
    else the answer is the warp's, since drain() reads tensor memory with it."""
    src = source("gemm_split.cu")
    alone = [src[:m.start()].rsplit("\n", 1)[-1] + src[m.start():].split("\n", 1)[0]
             for m in re.finditer(r"\bmbar_wait\(", src)]
    assert len(alone) == 1 and "issued - ST" in alone[0], alone
    assert src.index("if (tid == 0) {\n            set_error") < src.index("mbar_wait(")
    assert re.search(r"auto wait = \[&\]\(int c\) \{ return warp_wait\(", src)


def test_warp_wait_is_uniform():
    src = source("ptx.cuh")
    body = src[src.index("bool warp_wait("):]
    assert "__all_sync(0xffffffffu, mbar_wait(bar, parity))" in body[:body.index("}")]
