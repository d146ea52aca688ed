"""Warp collectives with a full mask (shuffles, votes and the functions that hold them) may not
stand in an arm of a conditional that differs between the lanes of a warp: the lanes of the two arms
would name each other from two different calls.  Read off the sources: in an arm of ``c ? a : b`` a
collective is allowed where c is the same for the whole warp, a template constant or one of
UNIFORM."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2401_11882_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))
INTRINSIC = r"__(?:shfl|any|all|ballot|match|reduce)\w*_sync|__syncwarp"
# template parameters and constants (MODE, SAVED, KO, Eval::FLOORS, FLOOR_VJP ...), and
# conditions that are the same in all lanes (j: an unrolled loop's; use_graph: the host's)
CONSTANT = re.compile(r"^[!\s]*(?:\w+::)?[A-Z][A-Z0-9_]*(?:\s*[=!<>&|]+\s*[\w:!]+)*$")
UNIFORM = {"j < K", "use_graph"}


def _text(path):
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
    return re.sub(r"^\s*#[^\n]*", "", text, flags=re.M)


def _close(text, i):
    """Index of the bracket that closes the one at i."""
    pairs, depth = {"(": ")", "{": "}", "[": "]"}, 0
    for j in range(i, len(text)):
        if text[j] in pairs:
            depth += 1
        elif text[j] in pairs.values():
            depth -= 1
            if depth == 0:
                return j
    raise ValueError("unbalanced source")


def _functions(text):
    """(name, body) of every function and lambda definition."""
    for m in re.finditer(r"\b(\w+)\s*(?:=\s*\[[^\]]*\]\s*)?\(", text):
        end = _close(text, m.end() - 1)
        tail = re.match(r"\s*(?:const|mutable|->[\w\s<>:]+)*\s*\{", text[end + 1:])
        if tail and m.group(1) not in ("if", "for", "while", "switch"):
            b = end + 1 + tail.end() - 1
            yield m.group(1), text[b:_close(text, b) + 1]


def collectives(texts):
    """Names of the intrinsics' callers, direct or not, as one pattern."""
    names = set()
    while True:
        call = re.compile(r"\b(?:%s)\s*(?:<[^;(){}]*>)?\s*\(" %
                          "|".join([INTRINSIC] + sorted(map(re.escape, names))))
        more = {n for t in texts for n, body in _functions(t) if call.search(body)} - names
        more.discard("operator")
        if not more:
            return call
        names |= more


def _arms(text, q):
    """(condition, both arms) of the conditional expression whose ? is at q."""
    depth, i = 0, q
    while i > 0:
        c = text[i - 1]
        if c in ")]}":
            depth += 1
        elif c in "([{":
            if depth == 0:
                break
            depth -= 1
        elif depth == 0 and (c in ",;?" or (c == "=" and text[i - 2] not in "=!<>" and text[i] != "=")
                             or (c == ":" and text[i - 2] != ":" and text[i] != ":")):
            break
        i -= 1
    cond = re.sub(r"^\s*return\b", "", text[i:q])
    depth, j = 0, q + 1
    while j < len(text):
        c = text[j]
        if c in "([{":
            depth += 1
        elif c in ")]}":
            if depth == 0:
                break
            depth -= 1
        elif depth == 0 and c in ",;":
            break
        j += 1
    return " ".join(cond.split()), text[q + 1:j]


def divergent(text, call):
    """The conditionals of a source whose arms hold a collective under a per-lane condition."""
    out = []
    for m in re.finditer(r"\?", text):
        cond, arms = _arms(text, m.start())
        if call.search(arms) and cond not in UNIFORM and not CONSTANT.match(cond):
            out.append(f"{cond} ? {' '.join(arms.split())}")
    return out


def test_the_reader_finds_a_shuffle_under_a_lane_s_condition():
    texts = ["""
      template <int K> float at(float v, int r) { return __shfl_sync(0xffffffffu, v, r); }
      float two(float v) { return at<2>(v, 1); }
      float f(bool have, float v) { const float a = have ? two(v) : (two(v), 0.f); return a; }
      float g(bool have, float v) { const float a = two(v); return have ? a : 0.f; }
      float h(float v) { return FLOORS ? two(v) : 0.f; }
    """]
    assert divergent(texts[0], collectives(texts)) == ["have ? two(v) : (two(v), 0.f)"]


@pytest.fixture(scope="module")
def call():
    return collectives([_text(p) for p in SOURCES])


@pytest.mark.parametrize("name", [os.path.basename(p) for p in SOURCES])
def test_no_collective_in_an_arm_that_differs_between_lanes(call, name):
    assert divergent(_text(os.path.join(CSRC, name)), call) == []
