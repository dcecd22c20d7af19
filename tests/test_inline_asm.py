"""Inline assembly of several instructions: an output written before a later instruction reads an input must be
an early clobber ("=&"), else the compiler may give both the same register.
"""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_1111_6288_gb300" / "csrc"
ASM = re.compile(r"\basm(?: volatile)?\s*\(((?:\s*\"(?:[^\"\\]|\\.)*\")+)\s*:(.*?)\);", re.S)


def blocks():
    for path in sorted(CSRC.glob("*.cu")) + sorted(CSRC.glob("*.h")):
        for m in ASM.finditer(path.read_text()):
            template = "".join(re.findall(r"\"((?:[^\"\\]|\\.)*)\"", m.group(1)))
            outputs = re.findall(r"\"([=+]&?\w)\"", m.group(2).split(":")[0])
            yield path.name, template.replace("\\n", " ").replace("\\t", " "), outputs


def overwritten_early(template, outputs):
    """Outputs that an instruction names before a later one names an input, without an early clobber."""
    seen, bad = set(), set()
    for instruction in template.split(";"):
        named = {int(k) for k in re.findall(r"%(\d+)", instruction)}
        if any(k >= len(outputs) for k in named):
            bad |= {k for k in seen if "&" not in outputs[k] and "+" not in outputs[k]}
        seen |= {k for k in named if k < len(outputs)}
    return sorted(bad)


def test_the_rule_sees_a_planted_mistake():
    assert overwritten_early("ld %0, [%2]; ld %1, [%3];", ["=r", "=r"]) == [0]
    assert overwritten_early("ld %0, [%2]; ld %1, [%3];", ["=&r", "=r"]) == []
    assert overwritten_early("try p, [%1], %2; selp %0, 1, 0, p;", ["=r"]) == []


def test_early_clobbers():
    found = list(blocks())
    assert sum(bool(outputs) for _, _, outputs in found) >= 4
    bad = [(name, template[:60]) for name, template, outputs in found if overwritten_early(template, outputs)]
    assert not bad, bad
