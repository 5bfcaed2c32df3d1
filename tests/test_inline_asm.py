"""Inline assembly of several instructions: an output that is written before the last
read of an input is marked early-clobber, else the compiler may give both the same
register."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1302_7203_gb300", "csrc")


def statements(text):
    """(template, output constraints, number of inputs) of each asm statement."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"\basm\s*(?:volatile)?\s*\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0) if text[i] in "()" else 0
            i += 1
        body = text[m.end():i - 1]
        # the template's string literals, then the sections behind single colons
        lit = re.match(r'\s*(?:"(?:[^"\\]|\\.)*"\s*)+', body)
        template = "".join(re.findall(r'"((?:[^"\\]|\\.)*)"', lit.group(0)))
        sections = re.split(r"(?<!:):(?!:)", body[lit.end():].replace("::", ": :"))
        outs = re.findall(r'"([^"]*)"', sections[1]) if len(sections) > 1 else []
        ins = re.findall(r'"([^"]*)"', sections[2]) if len(sections) > 2 else []
        yield template, outs, len(ins)


def early_writes(template, outs, nins):
    """Outputs without & that are written before the last read of an input."""
    ins = [re.findall(r"%(\d+)", s) for s in template.split(";") if "%" in s]
    first = {}
    last_read = -1
    for at, ops in enumerate(ins):
        ops = [int(x) for x in ops]
        if ops and ops[0] < len(outs):
            first.setdefault(ops[0], at)
        if any(len(outs) <= x < len(outs) + nins for x in ops):
            last_read = at
    return [k for k, at in first.items() if at < last_read and "&" not in outs[k]]


def test_early_writes_are_seen():
    assert early_writes("mul.lo.u32 %0, %2, %3; mad.hi.u32 %1, %2, %3, %0;", ["=r", "=r"], 2) == [0]
    assert early_writes("mul.lo.u32 %0, %2, %3; mad.hi.u32 %1, %2, %3, %0;", ["=&r", "=r"], 2) == []


def test_outputs_written_early_are_marked():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for template, outs, nins in statements(open(path).read()):
            seen += 1
            bad = early_writes(template, outs, nins)
            assert not bad, f"{os.path.basename(path)}: {template!r} writes %{bad[0]} early"
    assert seen >= 10
