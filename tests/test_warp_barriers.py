"""Barriers that take whole warps are reached by whole warps.

`bar.sync`, `bar.red` and the `.aligned` forms of the cluster barrier and of
the tensor-memory allocation are undefined unless all threads of a warp
execute them together, and unlike every other wait of the library they have
no time limit.  Code before them diverges (one lane arrives on an mbarrier or
issues copies, ragged tiles store under a condition), so each of them has to
bring its warp together itself: `__syncwarp()` right before the instruction,
in the same block.  Read from the sources; no GPU needed."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1708_07515_gb300", "csrc")
WARP_WIDE = re.compile(r"(?<!m)\b(bar\.(sync|red|arrive)|barrier\.(cluster\.)?(arrive|wait|sync|red)|tcgen05\.alloc)")


def _code(path):
    text = open(path).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def _unguarded(text):
    """(all, unguarded) inline-assembly statements holding a warp-wide barrier."""
    found, bad = [], []
    for m in re.finditer(r"\basm\s*(?:volatile)?\s*\(", text):
        stmt = text[m.start():text.index(";\n", m.end()) if ";\n" in text[m.end():] else len(text)]
        body = stmt[:stmt.find('" :') if '" :' in stmt else len(stmt)]
        if not WARP_WIDE.search(body):
            continue
        found.append(stmt)
        before = text[text.rindex("{", 0, m.start()):m.start()]
        if "__syncwarp();" not in before:
            bad.append(" ".join(stmt.split()))
    return found, bad


@pytest.mark.parametrize("src", ["{ asm volatile(\"bar.sync 1, %0;\" ::\"n\"(8) : \"memory\");\n }",
                                 "{ if (lane == 0) arrive();\n asm volatile(\"barrier.cluster.arrive.aligned;\" ::: "
                                 "\"memory\");\n }"])
def test_the_check_sees_an_unguarded_barrier(src):
    found, bad = _unguarded(src)
    assert len(found) == 1 and len(bad) == 1
    assert _unguarded(src.replace("asm", "__syncwarp();\n asm"))[1] == []


def test_mbarrier_instructions_are_not_warp_wide():
    assert _unguarded("{ asm volatile(\"mbarrier.arrive.shared::cta.b64 _, [%0];\" ::\"r\"(a) : \"memory\");\n }") == ([], [])


def test_every_warp_wide_barrier_brings_its_warp_together():
    total = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        found, bad = _unguarded(_code(path))
        total += len(found)
        assert not bad, f"{os.path.basename(path)}: {bad}"
    assert total >= 4   # the cluster and named barriers of the backprojection, the learned decimation's
