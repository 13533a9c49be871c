"""The inline assembly of csrc/ states its effects: what its constraints leave out the compiler may assume not to happen."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1501_01405_gb300", "csrc")
# statements that order memory accesses, or make or take data of another thread or unit
ORDERING = re.compile(r"mbarrier|barrier\.cta|bar\.sync|fence|cp\.async|tcgen05|ld\.shared::cluster")


def statements():
    """(file, line, template, constraint text) of every asm statement."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = open(path).read()
        for m in re.finditer(r"\basm\b(?:\s+volatile)?\s*\(", src):
            at, depth, text = m.end(), 1, False
            while depth:
                c = src[at]
                if text:
                    at += c == "\\"
                    text = c != '"'
                else:
                    text = c == '"'
                    depth += (c == "(") - (c == ")")
                at += 1
            body = src[m.end():at - 1]
            head = re.match(r'(?:\s*"(?:[^"\\]|\\.)*")+', body)
            template = "".join(re.findall(r'"((?:[^"\\]|\\.)*)"', head.group(0))).replace("\\n", "\n").replace("\\t", " ")
            out.append((os.path.basename(path), src.count("\n", 0, m.start()) + 1, template, body[head.end():],
                        "volatile" in m.group(0)))
    return out


def test_statements_are_found():
    files = {s[0] for s in statements()}
    assert {"tc.cuh", "common.cuh", "queues.cu", "pi.cu", "forest_fire.cu", "mlp.cu"} <= files


@pytest.mark.parametrize("stmt", [s for s in statements() if ORDERING.search(s[2])], ids=lambda s: "%s:%d" % s[:2])
def test_ordering_statements_clobber_memory(stmt):
    """A wait, fence, barrier or asynchronous copy without the memory clobber leaves the compiler free to move
    ordinary loads and stores across it."""
    _, _, _, constraints, volatile = stmt
    assert volatile and '"memory"' in constraints


@pytest.mark.parametrize("stmt", [s for s in statements() if "tcgen05.ld" in s[2]], ids=lambda s: "%s:%d" % s[:2])
def test_tensor_memory_loads_hold_their_wait(stmt):
    """The registers of a tensor-memory load may be read after its wait only: one statement."""
    assert "tcgen05.wait::ld" in stmt[2]
