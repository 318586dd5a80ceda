"""Kernels that are launched while the one before them still runs (after_previous): what they read may be written until
their wait is over, so neither they nor the functions that they call may promise the compiler unchanging data."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1608_04658_gb300", "csrc")
PROMISE = re.compile(r"__restrict__|__ldg\b|ld\.global\.nc")


def _matching(text, i, step, up, down):
    """Index of the bracket that closes the one at i, walking by step."""
    depth = 0
    while True:
        depth += (text[i] == up) - (text[i] == down)
        if depth == 0:
            return i
        i += step


def _functions(text):
    """(name, signature and body) of every device function that the text defines."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
    for m in re.finditer(r"__global__|__device__", text):
        stop = re.compile(r"[{;]").search(text, m.end())
        if stop is None or text[stop.start()] == ";":
            continue
        head = text[m.start():stop.start()]
        if ")" not in head:
            continue
        p = _matching(head, head.rindex(")"), -1, ")", "(")
        name = re.search(r"(\w+)\s*(<[^<>]*>)?\s*$", head[:p])
        if name:
            yield name.group(1), text[m.start():_matching(text, stop.start(), 1, "{", "}") + 1]


def test_early_kernels_make_no_promise_of_unchanging_data():
    bodies = {}
    for f in glob.glob(os.path.join(CSRC, "*.cu*")):
        for name, text in _functions(open(f).read()):
            bodies.setdefault(name, []).append(text)
    early = [n for n, t in bodies.items() if n.endswith("_kernel") and any("after_previous()" in x for x in t)]
    assert len(early) >= 9, early
    seen, todo = set(), list(early)
    while todo:
        n = todo.pop()
        if n in seen:
            continue
        seen.add(n)
        for text in bodies[n]:
            todo += [w for w in set(re.findall(r"\w+", text)) if w in bodies]
    assert {"stage", "gather_pair", "gather_global", "node_links"} <= seen
    assert not sorted(n for n in seen if any(PROMISE.search(x) for x in bodies[n]))
