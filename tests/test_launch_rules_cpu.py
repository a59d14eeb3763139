"""Rules of the launches that may begin before the stream's previous kernel has
ended, read off the sources: every kernel launched that way waits for its
predecessor before anything else."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2602_14975_gb300", "csrc")


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        yield os.path.basename(path), re.sub(r"//[^\n]*", "", open(path).read())


def test_every_early_launched_kernel_begins_with_the_wait():
    launched, waits = set(), set()
    for _, src in sources():
        for m in re.finditer(r"\blaunch_dep(?:_if)?\(", src):
            k = re.search(r"\bk_\w+", src[m.end():m.end() + 200])
            if k:
                launched.add(k.group(0))
        launched |= set(re.findall(r"first_launch<[^;]*?\((k_\w+)", src))
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", src):
            body = src[src.index("{", m.end()):]
            if re.match(r"\{\s*dep_entry\(", body):
                waits.add(m.group(1))
    assert len(launched) >= 20
    assert launched <= waits, launched - waits
    # and nothing that waits is launched in a way that would never let it overlap
    assert waits <= launched, waits - launched


def test_wait_comes_with_every_entry():
    text = open(os.path.join(CSRC, "launch.cuh")).read()
    body = text[text.index("void dep_entry("):]
    body = body[:body.index("\n}")]
    assert "griddepcontrol.wait" in body and "if (early)" in body
    assert body.index("launch_dependents") < body.index("griddepcontrol.wait")
