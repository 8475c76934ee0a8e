"""Rules of the kernels' inline PTX that no run can show, read from the sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0904_1826_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def _asm_statements(text):
    """The string parts of every asm statement, joined."""
    for m in re.finditer(r"\basm\s+volatile\s*\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield "".join(re.findall(r'"((?:[^"\\]|\\.)*)"', text[m.end():i]))


@pytest.mark.parametrize("path", [p for p in SOURCES if "tcgen05.commit" in open(p).read()], ids=os.path.basename)
def test_products_and_their_commits_have_one_issuing_thread(path):
    """tcgen05.commit tracks the products that its own thread issued.  Where an
    election picks the thread of the products, the same election has to pick
    that of the commit: which lane it is, is not specified."""
    text = open(path).read()
    asm = list(_asm_statements(text))
    mma = [a for a in asm if "tcgen05.mma" in a]
    commit = [a for a in asm if "tcgen05.commit" in a]
    assert mma and commit
    elected = ["elect.sync" in a for a in mma]
    assert len(set(elected)) == 1
    assert all(("elect.sync" in a) == elected[0] for a in commit)
    if elected[0]:   # the whole warp arrives at each commit: no lane's branch around it
        assert not re.search(r"if \([^)]*\blane\b[^)]*\)\s*(\{[^{}]*)?mma_commit\(", text)
