"""Inline PTX whose effect depends on where it stands (warp-wide operations, memory) is
volatile: the compiler may merge or move any other asm statement as a function of its inputs."""
from __future__ import annotations

import glob
import os
import re

import paper_2202_13976_gb300._build as b


def _statements():
    for path in sorted(glob.glob(os.path.join(b.CSRC, "*.cu")) + glob.glob(os.path.join(b.CSRC, "*.cuh"))):
        text = open(path).read()
        for m in re.finditer(r"\basm\b(\s+volatile\b)?\s*\(\s*\"([^\"]*)\"", text):
            yield os.path.basename(path), text[: m.start()].count("\n") + 1, bool(m.group(1)), m.group(2)


def test_the_statements_are_found():
    assert len(list(_statements())) >= 8


def test_position_dependent_asm_is_volatile():
    ordered = re.compile(r"\.sync\b|\b(ld|st|red|atom)\.")
    bad = [(f, line, code) for f, line, vol, code in _statements() if ordered.search(code) and not vol]
    assert not bad
