"""Every wait in a decode kernel is bounded, and a CTA whose wait ran out still leaves in order: its warps go on to the CTA's barriers.
That holds only if the lanes of a warp agree on what a wait said before they part ways over it.  Provoking the case needs a kernel that
hangs for the length of the bound, so the sources are read instead: a wait by all lanes that decides where they go is voted on, a wait by
one lane is handed to the others, and the softmax and gather roles only collect theirs."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_37626_b200", "csrc")
KERNELS = sorted(os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "splash_decode_umma*.cu")))


def statements(text):
    """(line number, indentation, statement) with continuation lines joined."""
    out, lines, i = [], text.split("\n"), 0
    while i < len(lines):
        line, at = lines[i].split("//")[0].rstrip(), i + 1
        while (line.count("(") > line.count(")") or line.endswith(("&&", "||"))) and i + 1 < len(lines):
            i += 1
            line += " " + lines[i].split("//")[0].strip()
        if line.strip():
            out.append((at, len(line) - len(line.lstrip()), line.strip()))
        i += 1
    return out


def by_one_lane(rows, k):
    """Is statement k inside a branch of a single lane?"""
    indent = rows[k][1]
    if "lane == 0" in rows[k][2].split("mbar_wait")[0]:
        return True
    for at, ind, s in reversed(rows[:k]):
        if ind < indent:
            if re.search(r"lane == 0|elected\)", s):
                return True
            indent = ind
    return False


@pytest.mark.parametrize("name", KERNELS)
def test_lanes_agree_on_a_wait_before_they_part(name):
    rows = statements(open(os.path.join(CSRC, name)).read())
    seen = 0
    for k, (at, ind, s) in enumerate(rows):
        if "mbar_wait" not in s or "ok &=" in s or "gather_tiles<" in s:       # (the gather: below)
            continue
        seen += 1
        if by_one_lane(rows, k) or s.startswith("mbar_wait"):                  # (or nobody asks what it said)
            continue
        assert "ok = " in s, f"{name}:{at}: a wait by all lanes whose answer is not voted on: {s}"
        # the next statements up to the vote use the answer for nothing but another wait
        for at2, _, s2 in rows[k + 1:]:
            if "__all_sync(0xffffffffu, ok)" in s2:
                break
            assert re.match(r"(if \(ok && \w+ == 0\) )?ok = .*mbar_wait", s2), \
                f"{name}:{at}: lanes may part at line {at2} before they have agreed: {s2}"
    assert seen > 0


def test_the_gather_walks_on():
    # its waits are passed in by the kernels; whatever they say, its lanes stay in step
    body = open(os.path.join(CSRC, "splash_gather.cuh")).read().split("gather_tiles(")[1]
    assert len(re.findall(r"wait_(?:stage|qk)\(\(?[^&;{]*\);", body)) == 2
    assert not re.search(r"(?:if \([^\n]*!|= |return )wait_(?:stage|qk)\(", body)
