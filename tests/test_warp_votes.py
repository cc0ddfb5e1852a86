"""Warp votes and shuffles in the kernels' sources, checked by reading (CPU): none may stand under
a condition on a shared-memory word that another warp writes meanwhile (a ring slot's tag, a
buffer's ready count).  Lanes can see such a word change at different moments, and those that
take the branch would then vote with the full mask against lanes that are somewhere else, which is
undefined and can hang.  Running the kernels cannot show it: the lanes mostly agree."""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_2405_03594_gb300", "csrc", "*.cu*")))
POLLED = re.compile(r"\btag\s*\[|\*\s*tag\b|\bready\s*\[")
COLLECTIVE = re.compile(r"\b__(?:any|all|ballot|shfl\w*|reduce\w*|match\w*)_sync\s*\(|\b__syncwarp\s*\(|\bbar_sync\s*\(")


def code_of(text):
    return re.sub(r"/\*.*?\*/|//[^\n]*", "", text, flags=re.S)


def _closing(s, i, pair):
    """Index of the bracket that closes s[i]."""
    depth = 0
    for j in range(i, len(s)):
        depth += (s[j] == pair[0]) - (s[j] == pair[1])
        if depth == 0:
            return j
    raise AssertionError("unbalanced source")


def divergent_votes(text):
    """(condition, statement) of every if or while on a polled word that holds a collective."""
    s = code_of(text)
    found = []
    for m in re.finditer(r"\b(?:if|while)\s*(?:constexpr\s*)?\(", s):
        end = _closing(s, m.end() - 1, "()")
        cond = s[m.end():end]
        if not POLLED.search(cond):
            continue
        body_at = end + 1 + len(s[end + 1:]) - len(s[end + 1:].lstrip())
        body = s[body_at:_closing(s, body_at, "{}") + 1] if s[body_at] == "{" else s[body_at:s.index(";", body_at) + 1]
        # a vote within the condition itself is reached by only some lanes after && or ||
        if COLLECTIVE.search(body) or re.search(r"(?:&&|\|\|).*", cond, flags=re.S) and COLLECTIVE.search(cond):
            found.append((" ".join(cond.split()), " ".join(body.split())))
    return found


@pytest.mark.parametrize("path", SOURCES, ids=[os.path.basename(p) for p in SOURCES])
def test_no_vote_under_a_polled_condition(path):
    with open(path) as f:
        assert divergent_votes(f.read()) == []


def test_the_check_finds_such_votes():
    assert divergent_votes("if (!dead && tag[s] != n) {\n while (tag[s] != n) {}\n dead = __any_sync(~0u, dead); }")
    assert divergent_votes("while (ready[b] != k) __syncwarp();")
    assert not divergent_votes("if (tag[s] != n) { spin(); }  // then __any_sync(\nok = __all_sync(~0u, ok);")


def test_the_polling_helper_holds_none():
    with open(os.path.join(ROOT, "paper_2405_03594_gb300", "csrc", "sp_internal.cuh")) as f:
        s = code_of(f.read())
    at = s.index("{", s.index("bool wait_claimed("))
    body = s[at:_closing(s, at, "{}")]
    assert POLLED.search(body) and not COLLECTIVE.search(body)
