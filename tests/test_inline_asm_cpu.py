"""The inline assembly of csrc/ states its effects: what its constraints leave out the compiler may assume not to happen."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1501_01405_gb300", "csrc")
# statements that order memory accesses, or take data that another thread or unit made
ORDERING = re.compile(r"mbarrier|barrier\.cta|bar\.sync|fence|cp\.async|tcgen05|\bld\.(?!param)")


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


def constraints_of(text):
    """Constraint strings of the outputs and of the inputs."""
    parts, depth, word = [[]], 0, False
    for m in re.finditer(r'"([^"]*)"|([():])', re.sub(r"::", ": :", text)):
        if m.group(2) == "(":
            depth += 1
        elif m.group(2) == ")":
            depth -= 1
        elif m.group(2) == ":" and depth == 0:
            parts.append([])
        elif m.group(1) is not None and depth == 0:
            parts[-1].append(m.group(1))
    parts += [[], [], []]
    return parts[1], parts[2]


def early_writes(template, n_out):
    """Outputs %k that an instruction writes while a later one still reads an input (an operand from n_out on): the
    input's register may be the output's."""
    found = []
    ins = [i.strip() for i in template.replace("{\n", " ").replace("\n}", " ").split(";")]
    ins = [i for i in ins if i and not i.startswith(".reg")]
    for at, one in enumerate(ins):
        one = re.sub(r"^@!?\w+\s+", "", one)
        op, _, args = one.partition(" ")
        if op.split(".")[0] in ("st", "bar", "barrier", "mbarrier", "fence") or op.startswith(("tcgen05", "cp.")):
            continue
        dest = re.findall(r"%(\d+)", args.split("}")[0] if args.lstrip().startswith("{") else args.split(",")[0])
        later = {int(k) for i in ins[at + 1:] for k in re.findall(r"(?<!%)%(\d+)", i)}
        found += [int(k) for k in dest if int(k) < n_out and any(x >= n_out for x in later)]
    return found


def test_early_writes_are_seen():
    assert early_writes("add.cc.u32 %0, %0, %3; addc.u32 %1, %1, %4;", 3) == [0]
    assert early_writes("{\n .reg .u32 a;\n add.cc.u32 a, %0, %2;\n addc.u32 %1, %1, %3;\n mov.u32 %0, a;\n}", 2) == []


@pytest.mark.parametrize("stmt", statements(), ids=lambda s: "%s:%d" % s[:2])
def test_no_output_is_written_before_an_input_is_read(stmt):
    outputs, _ = constraints_of(stmt[3])
    assert early_writes(stmt[2], len(outputs)) == []
