"""Which thread issues to the tensor core.  A commit covers what its own thread has issued, and no result tells when it is another
thread's, so the sources are read."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_19178_b200", "csrc")


def code_of(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


SOURCES = [f for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))) if "tcgen05.mma" in code_of(f)]


def conditions(lines):
    """(line, conditions of the `if`s that it stands under) for every line."""
    blocks, single = [], None  # of the open braces: the condition they belong to, or None; that of an `if` without braces
    for line in lines:
        m = re.match(r"\s*(?:\} else )?if (?:constexpr )?\((.*)\)\s*(\{?)([^{]*)$", line)
        cond = m.group(1) if m else None
        yield line, [c for c in blocks + [single, cond] if c]
        single = cond if m and not m.group(2) and not m.group(3).strip() else None
        for ch in line:
            if ch == "{":
                blocks.append(cond)
                cond = None
            elif ch == "}" and blocks:
                blocks.pop()


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_products_and_commits_stand_under_the_elected_thread(path):
    code = code_of(path)
    wrappers = {re.findall(r"void (\w+)\(", code[:m.start()])[-1] for m in re.finditer(r"tcgen05\.(?:mma|commit)\.", code)}
    code = re.sub(r'"(?:[^"\\\n]|\\.)*"', '""', code)  # (the braces of strings are no blocks)
    calls = [(line.strip(), conds) for line, conds in conditions(code.split("\n"))
             if re.search(r"\b(?:%s)\(" % "|".join(wrappers), line) and "void " not in line]
    assert len(wrappers) >= 2 and len(calls) >= 5
    for line, conds in calls:
        assert any("elect_one()" in c for c in conds) and not any("lane" in c for c in conds), (line, conds)
