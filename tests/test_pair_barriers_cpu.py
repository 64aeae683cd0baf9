"""Two warps that meet at a named barrier inside a loop of bounded waits have to
leave that loop together: a warp that left alone would strand its partner at
the barrier for good.  Read from the sources (a failing wait is not provoked on
the GPU): pairs meet only through pair_vote(), loops that contain one are left
only on its outcome, and a wait's outcome is the same for all lanes."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_16590_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _block(text, start):
    """The braces' content that opens at or after `start`."""
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i : j + 1]
    raise AssertionError("unbalanced braces")


def _check_loop(body):
    for m in re.finditer(r"\b(break|return)\b", body):
        line = body[body.rfind("\n", 0, m.start()) + 1 : body.index("\n", m.start())]
        assert "pair_vote(" in line, line
    for m in re.finditer(r"\b(LWAIT|mbar_wait<\w+>)\(", body):
        assert re.search(r"(warp_ok\(|WARP_)$", body[: m.start()]), body[m.start() - 40 : m.end() + 40]


@pytest.mark.parametrize("name", ["linear.cu"])
def test_no_pair_waits_for_a_warp_that_left(name):
    text = _source(name)
    assert not re.search(r"bar\.sync[^;]*\b64;", text)
    loops = [_block(text, m.end()) for m in re.finditer(r"for \(int G = grp, n = 0;[^{]*", text)]
    assert len(loops) == 2 and sum(b.count("pair_vote(") for b in loops) == text.count("pair_vote(") == 3
    for body in loops:
        _check_loop(body)


def test_d128_forward_walks_its_barriers():
    """The d = 128 forward's math warps: a warp that leaves an item early goes
    through the barriers that its partner may still be at, then both vote."""
    text = _source("sm103_fwd.cu")
    start = text.index("for (int w = blockIdx.x; w < n_items; w += gridDim.x)")
    items = _block(text, start)
    after = re.sub(r"\s+", " ", text[start + items.__len__() :])
    # barriers of an item: one per block (in softmax_block, before any of its waits), one vote
    assert items.count("pair_vote(") == 1 and "pair_sync" not in items and "pair_exchange" not in items
    block = _block(text, text.index("bool softmax_block("))
    assert block.count("pair_exchange(") == 1 and "mbar_wait" not in block[: block.index("pair_exchange(")]
    # G counts the block barriers passed; Gend is known before the first wait
    assert items.index("Gend = G + tbk.NB;") < items.index("mbar_wait")
    assert re.search(r"if \(!ok\) \{\s*\+\+G;\s*break;", items[items.index("softmax_block") :])
    assert "if (!ok) { for (; G < Gend; ++G) pair_sync(quad); pair_vote(quad + 1, false); }" in after
