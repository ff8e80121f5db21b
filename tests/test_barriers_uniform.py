"""__syncthreads() has to be reached by every thread of the CTA at the same
place: two copies of a loop with barriers, one per kind of warp, are undefined
even where both arrive as often.  Read from the source: in the Gram kernel the
lambda that holds the slices' barriers is called where only conditions that
are the same in the whole CTA decide, never under one on a thread's or a
warp's index."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1008_1371_gb300", "csrc")
# what differs between the threads of a CTA in k_gram
PER_THREAD = re.compile(r"\b(tid|tx|ty|xw|ec|lr|lc|threadIdx)\b")


def _body(src, head):
    at = src.index(head)
    i = src.index("{", at)
    return src[i:_close(src, i) + 1]


def _close(src, i):
    depth = 0
    for k in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[k], 0)
        if depth == 0:
            return k
    raise AssertionError("unbalanced braces")


def _with_barriers(body):
    """Names of the lambdas that reach a barrier, directly or through another."""
    lam = {m.group(1): body[m.end() - 1:_close(body, m.end() - 1) + 1]
           for m in re.finditer(r"auto (\w+) = \[&\]\([^)]*\) \{", body)}
    reach = {n for n, t in lam.items() if "__syncthreads" in t}
    while True:
        more = {n for n, t in lam.items() if n not in reach and any(re.search(r"\b%s\(" % r, t) for r in reach)}
        if not more:
            return reach
        reach |= more


def test_gram_barriers_under_uniform_conditions():
    with open(os.path.join(CSRC, "blocked.cu")) as f:
        body = _body(f.read(), "k_gram(const double")
    names = _with_barriers(body)
    assert "slices" in names
    calls = [m for n in names for m in re.finditer(r"^[ \t]*(.*)\b%s\(" % n, body, re.M)]
    assert calls
    for m in calls:
        prefix = m.group(1)
        assert not PER_THREAD.search(prefix) and not prefix.startswith("else"), m.group(0)
        # the blocks around the call
        for h in re.finditer(r"(if|for|while) \(([^{;]*)\) \{", body[:m.start()]):
            if _close(body, h.end() - 1) > m.start():
                assert not PER_THREAD.search(h.group(2)), h.group(0)
